"""launch_pdl_cluster launches with programmatic stream serialization as
launch_pdl does: every kernel passed to it starts with griddep_wait() too
(see test_launch_invariants.py)."""
import re

from test_launch_invariants import SOURCES, _kernel_body_start


def test_every_cluster_kernel_waits_first():
    texts = {p.name: p.read_text() for p in SOURCES}
    names = {m.group(1) for t in texts.values()
             for m in re.finditer(r"launch_pdl_cluster\(\s*([A-Za-z_][A-Za-z_0-9]*)", t)}
    assert names, "no launch_pdl_cluster call found"
    for name in names:
        found = [t for t in texts.values() if _kernel_body_start(t, name) is not None]
        assert found, f"the definition of {name} was not found"
        for t in found:
            assert _kernel_body_start(t, name) == "griddep_wait()", name
