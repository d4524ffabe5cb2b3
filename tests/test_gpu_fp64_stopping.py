"""The end of an FP64 Polonsky-Keer solve: it goes on until two consecutive
iterations are below the tolerance, but the first one makes it converged -- at the
iteration cap, and where no second one follows it within 32 iterations."""
import numpy as np
import pytest

import paper_1612_08395_gb300.inputs as I

pytestmark = pytest.mark.gpu

N = 32


@pytest.fixture(scope="module")
def history(bem_mod, cuda_ok):
    """eps of iterations 1..240 (each from a solve that the cap ends there: repeated
    FP64 solves are bitwise the same, and the tolerance is out of reach)."""
    with bem_mod.Handle(N, N, 1.0 / N, 1.0 / N, -0.5, 0.3) as h:
        eps = []
        for m in range(1, 241):
            r, rc = h.solve(I.paraboloid(N), 0.02, precision="fp64", tol=1e-300, max_iter=m, check=False)
            if r.iterations < m or rc != bem_mod.BEM_ENOCONV:
                break
            eps.append(r.final_eps)
    return np.array(eps)


def dips(eps):
    """(iteration, tolerance) such that this iteration is the first below the tolerance
    and the next one is above it, the later in the solve the better."""
    out = []
    for i in range(1, len(eps) - 1):
        best = eps[:i].min()
        tol = 0.5 * (eps[i] + min(best, eps[i + 1]))
        if eps[i] < 0.9 * min(best, eps[i + 1]):
            out.append((i + 1, tol))
    return out


def solve(bem_mod, tol, max_iter):
    with bem_mod.Handle(N, N, 1.0 / N, 1.0 / N, -0.5, 0.3) as h:
        return h.solve(I.paraboloid(N), 0.02, precision="fp64", tol=tol, max_iter=max_iter, check=False)


@pytest.mark.parametrize("later", [0, 1])
def test_small_step_at_the_cap_is_converged(bem_mod, cuda_ok, history, later):
    cases = dips(history)
    assert cases
    for it, tol in (cases[0], cases[len(cases) // 2], cases[-1]):
        r, rc = solve(bem_mod, tol, it + later)
        assert rc == bem_mod.BEM_OK and r.status == bem_mod.BEM_OK
        assert r.iterations == it + later and r.final_eps < tol and r.stalled == 0
        r, rc = solve(bem_mod, tol, it - 1)
        assert rc == bem_mod.BEM_ENOCONV and r.iterations == it - 1


def test_solve_ends_soon_after_its_first_small_step(bem_mod, cuda_ok, history):
    for it, tol in dips(history):
        r, rc = solve(bem_mod, tol, 20000)
        assert rc == bem_mod.BEM_OK and r.stalled == 0 and r.final_eps < tol
        assert it < r.iterations <= it + 32
