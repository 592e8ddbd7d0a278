"""Params reach the C struct by value and type: a field of a type that ctypes
refuses (a float, a NumPy integer) is refused whether or not an equal value of
the right type was used before, in either order; a Params of another class
brings its own c()."""
import numpy as np
import pytest

import paper_2509_26436_gb300 as Q
from paper_2509_26436_gb300 import build as B


@pytest.fixture(scope="module", autouse=True)
def _library():
    B.build()


@pytest.mark.parametrize("field,good", [("group_q", 64), ("group_s", 8), ("mode", 1), ("flag_bits", 4), ("code_bits", 16)])
@pytest.mark.parametrize("bad", [float, np.float32])
def test_refused_after_an_equal_value_was_taken(field, good, bad):
    def size(v):
        return Q.linear_workspace_size(16, 64, 64, Q.Params(**{field: v}))

    for _ in range(2):
        with pytest.raises(TypeError):
            size(bad(good))
        assert size(good) > 0
    with pytest.raises(TypeError):
        Q.linear_launch_count(16, 64, 64, Q.Params(**{field: bad(good)}))


def test_integer_types_are_treated_alike_before_and_after():
    def outcome():
        try:
            return Q.linear_workspace_size(16, 64, 64, Q.Params(group_s=np.int64(32)))
        except TypeError:
            return TypeError

    first = outcome()
    assert Q.linear_workspace_size(16, 64, 64, Q.Params(group_s=32)) > 0
    assert outcome() == first


def test_other_classes_bring_their_own_struct():
    class Fixed(Q.Params):
        __hash__ = None

        def c(self):
            return Q._native.QuartzParams(64, 16, 1, 8, 8)

    asym = Q.linear_workspace_size(16, 64, 64, Q.Params(mode=1))
    assert Q.linear_workspace_size(16, 64, 64, Fixed()) == asym != Q.linear_workspace_size(16, 64, 64)
