"""Which degree bins a tune() result leaves open (CPU): only those whose open form
in such a batch is the one that won; every other bin keeps its tuned shape."""
import re

import pytest

from paper_2507_02164_gb300 import autotune, build

SMS = 152
WON = {"lanes": 1, "block": 256, "ctas_per_sm": 0, "polish_warps": 4, "ms": 1.0, "open": {"ms": 0.8, "best_ms": 1.0, "faster": True},
       "one_role": {"lanes": 1, "block": 64, "ctas_per_sm": 3, "ms": 1.1}}


def _open(mode, polish, n, faster=True):
    entry = dict(WON, open=dict(WON["open"], faster=faster), polish_warps=4 if mode == "mixed" else 0)
    res = {"degrees": {str(d): dict(entry) for d in range(1, 13)}, "mode": mode, "polish": polish, "sms": SMS}
    t = autotune.uneven_tuning(res, n)
    shapes = zip(t.block, t.ctas_per_sm, t.lanes, t.polish_warps)
    open_ = set()
    for d, shape in enumerate(shapes):
        if not any(shape):
            open_.add(d)
        elif mode == "mixed" and d <= 8:
            assert shape == (256, 0, 1, 4)  # the warp-specialised shape that the bins have
        else:
            assert shape == (64, 3, 1, 0)
    return open_ - {0, 13, 14, 15}


@pytest.mark.parametrize("polish,degrees,line", [("fp64", set(range(4, 13)), 6144), ("df", set(range(7, 12)), 9216)])
def test_open_only_where_the_bins_have_the_form(polish, degrees, line):
    assert _open("mixed", polish, line * SMS) == degrees
    assert _open("mixed", polish, line * SMS, faster=False) == set()
    assert _open("mixed", polish, line * SMS - 1) == set()  # no split bin in a smaller batch
    assert _open("mixed", polish, None) == set()


def test_plain_bins_are_never_left_open():
    """The pool solver that wins large uniform plain batches has no bins."""
    assert _open("plain", "fp64", 1 << 22) == set()


def test_the_lines_are_the_librarys():
    src = open(build.CSRC + "/rd_uneven.cu").read()
    df, fp64 = map(int, re.search(r"polish_mode == RD_POLISH_DF \? (\d+) : (\d+)\) \* rd_sm_count_cached", src).groups())
    lo_df, lo, hi_df = map(int, re.search(r"first = df \? (\d+) : (\d+), last = df \? (\d+) : UNEVEN_MAX_DEG", src).groups())
    assert autotune.UNEVEN_SPLIT == {"fp64": (range(lo, 13), fp64), "df": (range(lo_df, hi_df + 1), df)}
