"""Which CG loops run as one launch, and what happens where one launch is not enough.

Routing: the number of kernels a solve launches tells the loop's form -- a few for a
loop inside a cluster or a cooperative launch, three or six an iteration for the
separate passes (which pass timing keeps).  Loops of several launches: a debug build
bounds a launch to three iterations on request; the next launch takes the state up
from memory, so that the results are bitwise those of the unsplit loop -- alone,
batched in the server, and handed to the passes half way (to the refinement's
tolerance: the passes add in another order)."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_1612_08395_gb300.inputs as I

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def punch(nx, ny, dx):
    return np.where(I.radius_grid(nx, ny, dx) <= 0.48 * min(nx, ny) * dx, 0.0, I.EXCLUDED)


# one launch: clusters up to 256 x 256, cooperative from 256 x 256 to 1024 x 1024 (even rows)
@pytest.mark.parametrize("nx,ny", [(8, 8), (30, 17), (128, 16), (16, 250), (130, 130), (255, 255), (256, 256), (200, 512),
                                   (512, 130), (514, 514), (1000, 600), (1024, 1024)])
def test_loops_that_are_one_launch(bem_mod, cuda_ok, nx, ny):
    dx = 1.0 / max(nx, ny)
    with bem_mod.Handle(nx, ny, dx, dx, 0.3, 0.3) as h:
        def launches(**kw):
            n = h.info().kernel_launches
            r, rc = h.solve(punch(nx, ny, dx), 0.01, precision="fp32", **kw)
            assert rc == bem_mod.BEM_OK
            return h.info().kernel_launches - n, r.iterations
        launches()  # sub-grids are set up on first use
        n, its = launches()
        assert its >= 3 and n <= 16, (n, its)
        n, its = launches(time_passes=True)
        assert n >= 6 * its, (n, its)


@pytest.mark.parametrize("nx,ny,precision", [(300, 301, "fp32"), (2048, 1100, "fp32"), (64, 64, "fp64"), (300, 300, "fp64")])
def test_loops_that_are_passes(bem_mod, cuda_ok, nx, ny, precision):
    dx = 1.0 / max(nx, ny)
    with bem_mod.Handle(nx, ny, dx, dx, 0.3, 0.3) as h:
        n = h.info().kernel_launches
        r, rc = h.solve(punch(nx, ny, dx), 0.01, precision=precision)
        assert rc == bem_mod.BEM_OK and h.info().kernel_launches - n >= 6 * r.iterations


@pytest.mark.parametrize("n", [40, 200, 600])
def test_nan_height_is_no_contact(bem_mod, cuda_ok, n):
    """An element whose height is NaN is never below the depth: no pressure there, by every route."""
    h = I.paraboloid(n)
    h[n // 2, n // 2] = np.nan
    with bem_mod.Handle(n, n, 1.0 / n, 1.0 / n, 0.2, 0.3) as hd:
        out = []
        for kw in ({"precision": "fp32"}, {"precision": "fp32", "time_passes": True}, {"precision": "fp64"}):
            p = np.empty((n, n))
            r, rc = hd.solve(h, 0.02, pressure_out=p, check=False, **kw)
            assert rc == bem_mod.BEM_OK and np.isfinite(p).all() and p[n // 2, n // 2] == 0.0
            out.append((p, r.contact_count))
    for p, count in out[:2]:
        assert abs(count - out[2][1]) <= max(2, 0.002 * out[2][1])
        assert np.linalg.norm(p - out[2][0]) <= 3e-4 * np.linalg.norm(out[2][0])


CASE = r"""
import json, os, sys
import numpy as np
sys.path.insert(0, %r)
from paper_1612_08395_gb300 import build
build.build(debug_checks=True)
import paper_1612_08395_gb300.bem as bem
import paper_1612_08395_gb300.inputs as I
def env(iters=0, inject=0):
    for k, v in (("BEM_LOOP_ITERS", iters), ("BEM_INJECT_WAIT_TIMEOUT", inject)):
        os.environ.pop(k, None)
        if v: os.environ[k] = str(v)
out = []
for nx, ny in ((40, 40), (30, 17), (130, 200), (255, 255), (256, 256), (300, 514), (1000, 600)):
    dx = 1.0 / max(nx, ny)
    r = I.radius_grid(nx, ny, dx)
    h = np.where(r <= 0.48 * min(nx, ny) * dx, 1e-3 * r * r, I.EXCLUDED)
    with bem.Handle(nx, ny, dx, dx, 0.3, 0.3) as hd:
        for what, prec in (("solve", "fp32"), ("solve", "fp32_refine"), ("pull-off", "fp32"), ("pull-off", "fp32_refine")):
            runs = []
            for iters, inject in ((0, 0), (3, 0), (1, 0), (3, 3)):
                if inject and prec == "fp32": continue
                env(iters, inject)
                p = np.empty((ny, nx))
                if what == "solve":
                    res, rc = hd.solve(h, 0.01, pressure_out=p, precision=prec); res = [res]
                else:
                    res, rc = hd.sweep(h, [0.01, 0.004, 0.001], dgamma=1e-5, final_pressure=p, precision=prec)
                runs.append((p, rc, [(x.force, x.iterations, x.contact_count, x.detach_rounds, x.stalled) for x in res]))
            env()
            a = runs[0]
            rec = {"case": [nx, ny, what, prec], "rc": [x[1] for x in runs],
                   "bitwise": [bool(np.array_equal(a[0], x[0])) and a[2] == x[2] for x in runs[1:3]]}
            if len(runs) > 3:
                b = runs[3]
                rec["err"] = float(np.linalg.norm(a[0] - b[0]) / max(np.linalg.norm(a[0]), 1e-300))
                rec["counts"] = [x[2] for x in a[2]] == [x[2] for x in b[2]]
            out.append(rec)
# the same job several times at once in the server, whose loops share cluster launches (240: or,
# while a job happens to be the only one in flight, run as cooperative ones)
served = []
for iters in (0, 3):
    env(iters)
    jobs, ps = [], []
    with bem.Server(nworkers=4, hbm_budget_bytes=8 << 30) as s:
        for n in (100, 100, 120, 120, 240, 240):
            h = np.where(I.radius_grid(n, n, 1.0 / n) <= 0.45, 0.0, I.EXCLUDED)
            p = np.empty((n, n)); ps.append(p)
            s.submit(n, n, 1.0 / n, 1.0 / n, 0.3, 0.3, h, [0.01, 0.004], dgamma=1e-5, final_pressure=p, precision="fp32_refine")
        done = s.drain()
    served.append([p.copy() for p in ps])
env()
a, b = served
print(json.dumps({"runs": out, "bitwise": [bool(np.array_equal(x, y)) for x, y in zip(a[:4] + a[0:1] + a[2:3], b[:4] + a[1:2] + a[3:4])],
                  "rounding": [float(np.linalg.norm(x - y) / np.linalg.norm(y)) for x, y in zip(a[4:] + a[4:5], b[4:] + a[5:6])]}))
"""


@pytest.fixture(scope="module")
def split(cuda_ok, tmp_path_factory):
    env = dict(os.environ, BEM_DEBUG_CHECKS="1")
    for k in ("BEM_LOOP_ITERS", "BEM_INJECT_WAIT_TIMEOUT"):
        env.pop(k, None)
    r = subprocess.run([sys.executable, "-c", CASE % ROOT], capture_output=True, text=True, env=env, timeout=900,
                       cwd=str(tmp_path_factory.mktemp("split")))
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_split_loops_are_bitwise_the_unsplit(split):
    for r in split["runs"]:
        assert all(rc == 0 for rc in r["rc"]) and all(r["bitwise"]), r


def test_loop_handed_to_the_passes_half_way(split):
    for r in split["runs"]:
        if "err" in r:
            assert r["counts"] and r["err"] <= 1e-9, r


def test_split_loops_in_the_server(split):
    assert all(split["bitwise"]) and max(split["rounding"]) <= 1e-9
