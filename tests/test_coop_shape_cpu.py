"""The rule that gives a CG loop to the cooperative kernel: a launch's CTAs, at
most one per SM, must hold all rows in their shared memory (224 KB) and in the
bit masks of their threads (two rounds of rows).  Restated here for every kernel,
row count and number of SMs, from the sizes of the kernels."""
import ctypes

import pytest

LENGTHS = [(lm, lp) for lm in (8, 9, 10) for lp in (9, 10, 11)]


@pytest.fixture(scope="module")
def coop_ctas(bem_mod):
    f = getattr(bem_mod.load_library(), "_ZN3bem9coop_ctasEiiii")  # bem::coop_ctas(int, int, int, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 4
    return f


def geometry(lm, lp):
    """Rows and columns that a CTA transforms at a time."""
    threads = 1024 if lp == 11 else 512 if lp == 10 or lm == 10 else 256
    return min(8, threads // ((1 << lm) // 8)), min(8, threads // ((1 << lp) // 8))


def rows_fit(lm, lp, rows, nb):
    """(the bit masks hold a CTA's rows, its shared memory at least, at most)."""
    m = 1 << lm
    per_round, columns = geometry(lm, lp)
    share = 2 * max(1, -(-rows // (2 * nb)))
    fields = 16 * share * m  # p, g, t and one more, FP32
    # the transforms' workspace without its pads, which add less than a sixteenth
    work = 8 * max(per_round * m, columns * (1 << lp))
    return share <= min(16, 2 * per_round), fields + work, fields + work + work // 16 + 2048


@pytest.mark.parametrize("lm,lp", LENGTHS)
def test_rows_fit_where_the_loop_is_taken(coop_ctas, lm, lp):
    taken = 0
    for nsm in (1, 2, 7, 20, 38, 64, 76, 100, 120, 127, 128, 140, 152, 300):
        for rows in sorted({1, 2, 3, 64, 255, 256, 257, 500, 777, 1023, 1 << (lp - 1)}):
            if rows > 1 << (lp - 1):
                continue
            nb = coop_ctas(lm, lp, rows, nsm)
            assert 0 <= nb <= min(nsm, 256)
            full = min(nsm, 256, -(-((1 << lm) + 1) // geometry(lm, lp)[1]))
            masks, least, most = rows_fit(lm, lp, rows, full)
            if nb:
                taken += 1
                assert nb == full and masks and least <= 224 * 1024
            else:
                assert not masks or most > 224 * 1024
    assert taken


@pytest.mark.parametrize("lm,lp", LENGTHS)
def test_whole_device_takes_every_row_count(coop_ctas, lm, lp):
    assert all(coop_ctas(lm, lp, rows, 152) > 0 for rows in range(1, (1 << (lp - 1)) + 1))


def test_few_sms_leave_the_loop_to_the_passes(coop_ctas):
    assert coop_ctas(10, 11, 1024, 152) == 152
    assert coop_ctas(10, 11, 1024, 100) == 0  # 12 rows of 1024 points a CTA: 260 KB
    assert coop_ctas(10, 11, 600, 100) == 100


@pytest.mark.parametrize("lm,lp", [(7, 9), (8, 8), (11, 11), (10, 12), (4, 5)])
def test_other_lengths_have_no_kernel(coop_ctas, lm, lp):
    assert coop_ctas(lm, lp, 16, 152) == 0
