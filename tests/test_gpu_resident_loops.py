"""CG loops that run as one launch -- inside one thread-block cluster (grids of at
most 256 x 256) or as one cooperative launch (transforms up to 2048 points) --
against the same solves by the separate passes (which pass timing keeps), at the
edges of their ranges: the smallest grid, rows that do not fill the cluster, odd
and rectangular sizes, whole grids and contact boxes, an empty contact, and the
iteration cap.

Plain FP32 solves of both routes stop at the same tolerance of the same iteration
but sum in another order, so they may stop some iterations apart: their pressures
agree to the solver tolerance times the conditioning, as plain FP32 results do
(3e-4); refined ones agree to the refinement's 1e-9."""
import numpy as np
import pytest

import paper_1612_08395_gb300.inputs as I

pytestmark = pytest.mark.gpu

# nx, ny, k: both sides on the cluster's range, rows below a cluster's sixteen,
# 256 x 256 (cooperative outside the server), elongated, and above 256
GRIDS = [(8, 8, 0.5), (16, 16, 0.0), (30, 17, 0.3), (33, 100, -0.2), (128, 16, 0.4), (16, 250, 0.4), (130, 130, 0.2),
         (255, 64, -0.3), (256, 256, 0.1), (250, 300, 0.3), (512, 130, 0.0), (514, 514, 0.3)]


def relL2(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def profile(nx, ny, dx, kind):
    r = I.radius_grid(nx, ny, dx)
    if kind == "punch":  # contact box of nearly the whole grid
        return np.where(r <= 0.48 * min(nx, ny) * dx, 0.0, I.EXCLUDED)
    return r * r / 2.0


@pytest.mark.parametrize("nx,ny,k", GRIDS)
@pytest.mark.parametrize("kind", ["punch", "paraboloid"])
def test_nonadhesive_matches_passes(bem_mod, cuda_ok, nx, ny, k, kind):
    dx = 1.0 / max(nx, ny)
    h = profile(nx, ny, dx, kind)
    d = 0.3 * min(nx, ny) ** 2 * dx * dx / 8.0
    with bem_mod.Handle(nx, ny, dx, dx, k, 0.3) as hd:
        for prec, tol in (("fp32", 3e-4), ("fp32_refine", 1e-9)):
            p, q = np.empty((ny, nx)), np.empty((ny, nx))
            a, rc_a = hd.solve(h, d, pressure_out=p, precision=prec)
            b, rc_b = hd.solve(h, d, pressure_out=q, precision=prec, time_passes=True)
            assert rc_a == rc_b == bem_mod.BEM_OK
            assert relL2(p, q) <= tol
            if prec == "fp32_refine":
                assert a.contact_count == b.contact_count > 0


@pytest.mark.parametrize("nx,ny,k", [g for g in GRIDS if g[0] >= 16])
def test_pull_off_matches_passes(bem_mod, cuda_ok, nx, ny, k):
    dx = 1.0 / max(nx, ny)
    h = profile(nx, ny, dx, "paraboloid")
    d0 = 0.3 * min(nx, ny) ** 2 * dx * dx / 8.0
    ds = d0 * np.linspace(1.0, 0.0, 5)
    with bem_mod.Handle(nx, ny, dx, dx, k, 0.3) as hd:
        p, q = np.empty((ny, nx)), np.empty((ny, nx))
        a, _ = hd.sweep(h, ds, dgamma=1e-3 * d0, final_pressure=p, precision="fp32_refine")
        Sa = hd.contact_set()
        b, _ = hd.sweep(h, ds, dgamma=1e-3 * d0, final_pressure=q, precision="fp32_refine", time_passes=True)
        Sb = hd.contact_set()
    assert [r.contact_count for r in a] == [r.contact_count for r in b]
    assert [r.detach_rounds for r in a] == [r.detach_rounds for r in b]
    assert np.array_equal(Sa, Sb)
    fmax = max(abs(r.force) for r in b)
    assert max(abs(x.force - y.force) for x, y in zip(a, b)) <= 1e-9 * fmax
    if np.linalg.norm(q) > 0:
        assert relL2(p, q) <= 1e-9


@pytest.mark.parametrize("n", [40, 200, 600])
def test_ends(bem_mod, cuda_ok, n):
    """No contact at all; the iteration cap; NaN in the profile; and the handle afterwards."""
    h = I.paraboloid(n)
    with bem_mod.Handle(n, n, 1.0 / n, 1.0 / n, 0.2, 0.3) as hd:
        p = np.empty((n, n))
        ref, _ = hd.solve(h, 0.02, pressure_out=p, precision="fp32")
        res, rc = hd.solve(h + 1.0, 0.02, pressure_out=p, precision="fp32")
        assert rc == bem_mod.BEM_OK and res.contact_count == 0 and not p.any()
        res, rc = hd.solve(h, 0.02, pressure_out=p, precision="fp32", tol=1e-14, max_iter=5)
        assert rc == bem_mod.BEM_ENOCONV and res.iterations == 5
        bad = h.copy()
        bad[n // 2, n // 2] = np.nan
        res, rc = hd.solve(bad, 0.02, pressure_out=p, precision="fp32", check=False)
        assert rc == bem_mod.BEM_ENUMERIC or np.isfinite(p).all()
        again, rc = hd.solve(h, 0.02, pressure_out=p, precision="fp32")
        assert rc == bem_mod.BEM_OK and again.force == ref.force and again.iterations == ref.iterations
