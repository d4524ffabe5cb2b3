"""The FP64 row passes of 2048 and 4096 points (grids of 1025 to 4096 columns),
built for two CTAs per SM, in every mode of the two CG loops: the first
iterations against the oracle's.  A transform's error is about 2^-52 log2(points),
5e-15 of its field; a few CG steps amplify it by no more than the ratio of the
residual's to the step's transforms, some hundreds: 1e-11 of the largest pressure."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(1025, 9), (1100, 33), (2048, 8), (2049, 5), (4095, 12), (4096, 16)]


@pytest.fixture(scope="module")
def problem(bem_mod, oracle_mod):
    made = {}

    def get(nx, ny):
        if (nx, ny) not in made:
            r = np.random.Generator(np.random.PCG64(nx))
            S = np.ones((ny, nx), dtype=np.uint8)
            S[1:-1, 1:-1] = r.random((ny - 2, nx - 2)) < 0.5
            h = 0.01 * r.random((ny, nx))
            hd = bem_mod.Handle(nx, ny, 1.0 / nx, 1.0 / nx, 0.3, 0.3)
            conv = oracle_mod.FFTConvolver(hd.influence_table()[:ny + 1, :nx + 1], ny, nx)
            made[nx, ny] = hd, h, S, oracle_mod.compliance(0.3, 0.3), conv
        return made[nx, ny]

    yield get
    for v in made.values():
        v[0].close()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("iters", [1, 4])
def test_fixed_set_iterations(bem_mod, oracle_mod, cuda_ok, problem, nx, ny, iters):
    hd, h, S, A, conv = problem(nx, ny)
    p = np.empty((ny, nx))
    hd.sweep_from(h, [0.005], np.zeros((ny, nx)), S, dgamma=1e9, final_pressure=p, precision="fp64", tol=1e-30,
                  max_iter=iters, check=False)
    ref = oracle_mod.fixed_set_cg(A, conv, h - 0.005, S, np.zeros((ny, nx)), tol=0.0, max_iter=iters).p
    assert np.abs(p - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("iters", [1, 4])
def test_polonsky_keer_iterations(bem_mod, oracle_mod, cuda_ok, problem, nx, ny, iters):
    hd, h, S, A, conv = problem(nx, ny)
    p = np.empty((ny, nx))
    hd.solve(h, 0.02, pressure_out=p, precision="fp64", tol=1e-30, max_iter=iters, check=False)
    ref = oracle_mod.pk_solve(A, conv, h, 0.02, tol=0.0, max_iter=iters).p
    assert np.abs(p - ref).max() <= 1e-11 * np.abs(ref).max()
