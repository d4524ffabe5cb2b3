"""The first iterations of the fixed-set CG by the separate FP32 passes on grids
whose rows take the unstaged kernels (columns not a multiple of 16), against the
same iterations in FP64: both follow the same CG, so a few iterations differ by
FP32 rounding only (1e-5 of the largest pressure)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(60, 60), (98, 40), (100, 100), (100, 300), (126, 60), (250, 100), (500, 40),
                                   (1001, 64), (2001, 33)])
@pytest.mark.parametrize("iters", [2, 4])
def test_fixed_set_iterations(bem_mod, cuda_ok, nx, ny, iters):
    r = np.random.Generator(np.random.PCG64(1))
    dx = 1.0 / max(nx, ny)
    S = np.ones((ny, nx), dtype=np.uint8)
    S[1:-1, 1:-1] = r.random((ny - 2, nx - 2)) < 0.5
    h, d = 0.01 * r.random((ny, nx)), 0.005
    p = {}
    with bem_mod.Handle(nx, ny, dx, dx, 0.3, 0.3) as hd:
        for prec in ("fp64", "fp32"):
            p[prec] = np.empty((ny, nx))
            hd.sweep_from(h, [d], np.zeros((ny, nx)), S, dgamma=1e9, final_pressure=p[prec], precision=prec,
                          tol=1e-30, max_iter=iters, time_passes=True, check=False)
    assert np.abs(p["fp32"] - p["fp64"]).max() <= 1e-5 * np.abs(p["fp64"]).max()
