"""A job alone in the server gives, bitwise, the results of the same sweep on a
handle of its own: at the sizes whose CG loops run inside a cluster, as a cooperative
launch and as passes, in both FP32 modes and FP64.  Several of them together agree
to rounding."""
import numpy as np
import pytest

import paper_1612_08395_gb300.inputs as I

pytestmark = pytest.mark.gpu

# cluster; cooperative (whole grid and contact box); odd rows, passes
SIZES = [100, 256, 300, 514, 601, 1000]
MIX_TOL = {"fp64": 1e-10, "fp32_refine": 1e-9, "fp32": 3e-4}


def job(n, precision, adhesive):
    r = I.radius_grid(n, n, 1.0 / n)
    h = np.where(r <= 0.47, 2e-3 * r * r, I.EXCLUDED)
    return {"args": (n, n, 1.0 / n, 1.0 / n, 0.3, 0.3), "h": h, "d": [0.01, 0.006] if adhesive else [0.01],
            "dgamma": 1e-5 if adhesive else 0.0, "precision": precision, "p": np.empty((n, n))}


def submit(s, j):
    return s.submit(*j["args"], j["h"], j["d"], dgamma=j["dgamma"], final_pressure=j["p"], precision=j["precision"])


def facts(results):
    return [(r.force, r.iterations, r.contact_count, r.detach_rounds, r.status, r.stalled, r.final_eps) for r in results]


@pytest.mark.parametrize("precision,adhesive", [("fp32", False), ("fp32", True), ("fp32_refine", True), ("fp64", False)])
@pytest.mark.parametrize("n", SIZES)
def test_job_alone_is_its_own_handle(bem_mod, cuda_ok, n, precision, adhesive):
    j = job(n, precision, adhesive)
    p = np.empty((n, n))
    with bem_mod.Handle(*j["args"]) as h:
        res, rc = h.sweep(j["h"], j["d"], dgamma=j["dgamma"], final_pressure=p, precision=precision)
    with bem_mod.Server(nworkers=4, hbm_budget_bytes=8 << 30) as s:
        submit(s, j)
        c, = s.drain()
    assert c["status"] == rc == bem_mod.BEM_OK and res[-1].contact_count > 0
    assert facts(c["results"]) == facts(res)
    assert np.array_equal(j["p"], p)


@pytest.mark.parametrize("precision", ["fp32", "fp32_refine"])
def test_mix_agrees_with_own_handles(bem_mod, cuda_ok, precision):
    # (plain FP32: a held set may differ by an element at its edge)
    jobs = [job(n, precision, a) for n in SIZES for a in ((False, True) if precision == "fp32_refine" else (False, False))]
    alone = []
    for j in jobs:
        p = np.empty_like(j["p"])
        with bem_mod.Handle(*j["args"]) as h:
            res, rc = h.sweep(j["h"], j["d"], dgamma=j["dgamma"], final_pressure=p, precision=precision)
        alone.append((res, rc, p))
    with bem_mod.Server(nworkers=6, hbm_budget_bytes=16 << 30) as s:
        tags = [submit(s, j) for j in jobs]
        done = {c["tag"]: c for c in s.drain()}
    for t, j, (res, rc, p) in zip(tags, jobs, alone):
        c = done[t]
        assert c["status"] == rc == bem_mod.BEM_OK
        if precision == "fp32_refine":
            assert [r.contact_count for r in c["results"]] == [r.contact_count for r in res]
        assert np.linalg.norm(j["p"] - p) <= MIX_TOL[precision] * np.linalg.norm(p)
