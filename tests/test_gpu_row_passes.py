"""The first Polonsky-Keer and fixed-set iterations by the separate passes, in every
row length and on both sides of the staged passes' condition (rows of a multiple of
16 elements), FP32 against FP64: both follow the same iteration, so that a few of
them differ by FP32 rounding only -- 1e-5 of the largest pressure for the fixed set
(as test_gpu_fixed_set_passes.py), 1e-4 for the overlap steps of Polonsky-Keer, which
divide by small differences.  And long FP64 rows, whose passes spill registers,
against the same grid transposed, whose rows are short."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

COLUMNS = [20, 32, 49, 63, 97, 99, 103, 110, 112, 119, 125, 127, 130, 192, 251, 400, 510, 1003]


def run(bem_mod, nx, ny, precision, iters, seed, fixed, timed=True):
    r = np.random.Generator(np.random.PCG64(seed))
    dx = 1.0 / max(nx, ny)
    S = np.ones((ny, nx), dtype=np.uint8)
    S[1:-1, 1:-1] = r.random((ny - 2, nx - 2)) < 0.5
    h, d = 0.01 * r.random((ny, nx)), 0.005
    p = np.empty((ny, nx))
    with bem_mod.Handle(nx, ny, dx, dx, 0.3, 0.3) as hd:
        kw = dict(precision=precision, tol=1e-30, max_iter=iters, time_passes=timed, check=False)
        if fixed:
            hd.sweep_from(h, [d], np.zeros((ny, nx)), S, dgamma=1e9, final_pressure=p, **kw)
        else:
            hd.solve(h, d, pressure_out=p, **kw)
    return p


@pytest.mark.parametrize("nx", COLUMNS)
@pytest.mark.parametrize("ny", [33, 60])
@pytest.mark.parametrize("fixed,tol", [(True, 1e-5), (False, 1e-4)])
def test_first_iterations(bem_mod, cuda_ok, nx, ny, fixed, tol):
    for iters in (1, 2, 4):
        a, b = (run(bem_mod, nx, ny, prec, iters, 3, fixed) for prec in ("fp32", "fp64"))
        assert np.abs(a - b).max() <= tol * np.abs(b).max()


@pytest.mark.parametrize("nx,ny", [(1100, 40), (2040, 33), (2100, 40), (4001, 24)])
@pytest.mark.parametrize("fixed", [True, False])
def test_long_fp64_rows_against_the_transpose(bem_mod, cuda_ok, nx, ny, fixed):
    """The problem of the transposed profile and set, its pressures transposed back: the same
    iteration with the roles of row and column passes exchanged (1e-9 after four iterations)."""
    r = np.random.Generator(np.random.PCG64(8))
    dx = 1.0 / nx
    S = (r.random((ny, nx)) < 0.5).astype(np.uint8)
    S[0] = S[-1] = 1
    S[:, 0] = S[:, -1] = 1
    h, d = 0.01 * r.random((ny, nx)), 0.005
    out = []
    for a, b, hh, ss in ((nx, ny, h, S), (ny, nx, np.ascontiguousarray(h.T), np.ascontiguousarray(S.T))):
        p = np.empty((b, a))
        kw = dict(precision="fp64", tol=1e-30, max_iter=4, check=False)
        with bem_mod.Handle(a, b, dx, dx, 0.3, 0.3) as hd:
            if fixed:
                hd.sweep_from(hh, [d], np.zeros((b, a)), ss, dgamma=1e9, final_pressure=p, **kw)
            else:
                hd.solve(hh, d, pressure_out=p, **kw)
        out.append(p)
    assert np.abs(out[0] - out[1].T).max() <= 1e-9 * np.abs(out[0]).max()
