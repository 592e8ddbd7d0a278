"""Per-row scales: the plan of test_split_plan.py is taken where it spares the
busiest CTA enough 64-wide stages (linear.cu: row_split_pays).  The saving that
the host computes in closed form is restated here and compared with the work
lists: whole tiles against the plan's CTAs."""
import itertools
import re

import pytest
from test_launch_invariants import CSRC
from test_split_plan import GROUPS, SMS, TILES, grid_size, tail_split, work_item, work_items

MIN_ROW_SAVING = 32
MIN_ROW_RANGE_SAVING = 48


def saving(T, sms, G, tail, split, ls):
    P = min(T, sms)
    whole = -(-T // P) * G
    return whole - ((T - tail) // P * G + (ls if ls > 0 else -(-G // split)))


def busiest(T, sms, G, tail, split, ls):
    P = grid_size(T, sms, tail, split, ls)
    most = 0
    for c in range(P):
        items = (work_item(c, P, T, G, tail, split, ls, k) for k in range(work_items(c, P, T, G, tail, split, ls)))
        most = max(most, sum(g1 - g0 for _, g0, g1, _, _ in items))
    return most


@pytest.mark.parametrize("sms", SMS)
def test_saving_is_what_the_work_lists_spare(sms):
    for T, G in itertools.product(TILES, GROUPS):
        tail, split, ls = tail_split(T, sms, G)
        if split > 1:
            s = saving(T, sms, G, tail, split, ls)
            assert s == busiest(T, sms, G, 0, 1, 0) - busiest(T, sms, G, tail, split, ls), (T, sms, G)


def test_thresholds_and_forms_at_152_sms():
    text = (CSRC / "linear.cu").read_text()
    for name, value in (("kMinRowSaving", MIN_ROW_SAVING), ("kMinRowRangeSaving", MIN_ROW_RANGE_SAVING)):
        assert re.search(rf"constexpr int {name} = {value};", text)

    def cut(M, N, K):
        T, G = -(-M // 128) * -(-N // 256), K // 64
        tail, split, ls = tail_split(T, 152, G)
        return split > 1 and saving(T, 152, G, tail, split, ls) >= (MIN_ROW_RANGE_SAVING if ls else MIN_ROW_SAVING)

    # the shapes of test_gpu_row_split.py
    for shape in ((2048, 1280, 11520), (1999, 1272, 11584), (2560, 3072, 8192), (1790, 3064, 3072), (1000, 1304, 4160),
                  (1, 8, 12288)):
        assert cut(*shape)
    for shape in ((2560, 3072, 5120), (256, 320, 1152), (130, 264, 64)):
        assert not cut(*shape)
