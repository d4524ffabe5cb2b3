"""The cooperative CG loop when its launch is refused, or not all of its CTAs become
resident (another stream's kernel may hold some back): in a debug build the launch
is refused or one CTA stays away on request, the others give the gathering up after
a tenth of a second, and the loop runs as passes with the result of a solve that
always does.  And a CTA that stays
away from a later barrier: the bounded waits run out, the call returns
BEM_ETIMEOUT, and the handle recovers."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASE = r"""
import json, os, sys, time
import numpy as np
sys.path.insert(0, %r)
from paper_1612_08395_gb300 import build
build.build(debug_checks=True)
import paper_1612_08395_gb300.bem as bem
import paper_1612_08395_gb300.inputs as I
out = []
def inject(v):
    for k in ("BEM_INJECT_WAIT_TIMEOUT", "BEM_INJECT_COOP_REFUSED"):
        os.environ.pop(k, None)
    if v: os.environ["BEM_INJECT_COOP_REFUSED" if v == "refused" else "BEM_INJECT_WAIT_TIMEOUT"] = "1" if v == "refused" else str(v)
for nx, ny, box in ((256, 256, False), (300, 514, False), (1000, 600, False), (514, 514, True)):
    dx = 1.0 / max(nx, ny)
    r = I.radius_grid(nx, ny, dx)
    h = r * r / 2.0 if box else np.where(r <= 0.48 * min(nx, ny) * dx, 1e-3 * r * r, I.EXCLUDED)
    d0 = 0.3 * min(nx, ny) ** 2 * dx * dx / 8.0 if box else 0.01
    with bem.Handle(nx, ny, dx, dx, 0.3, 0.3) as hd:
        hd.solve(h, d0, precision="fp32_refine")  # sub-grids are set up on first use
        for what in ("solve", "pull-off"):
            runs = {}
            for name, v, timed in (("coop", 0, False), ("held back", 2, False), ("refused", "refused", False),
                                   ("passes", 0, True)):
                inject(v)
                p = np.empty((ny, nx))
                before = hd.info().kernel_launches
                if what == "solve":
                    res, rc = hd.solve(h, d0, pressure_out=p, precision="fp32_refine", time_passes=timed)
                    res = [res]
                else:
                    res, rc = hd.sweep(h, [d0, 0.6 * d0, 0.2 * d0], dgamma=1e-3 * d0, final_pressure=p,
                                       precision="fp32_refine", time_passes=timed)
                runs[name] = (p, rc, [x.contact_count for x in res], [x.detach_rounds for x in res],
                              int(hd.info().kernel_launches - before))
            inject(0)
            ref = runs["passes"][0]
            n = max(float(np.linalg.norm(ref)), 1e-300)
            for name in ("coop", "held back", "refused"):
                p, rc, cnt, rounds, launches = runs[name]
                out.append({"case": [nx, ny, box, what, name], "rc": rc, "err": float(np.linalg.norm(p - ref)) / n,
                            "counts": cnt == runs["passes"][2], "rounds": rounds == runs["passes"][3],
                            "launches": launches, "passes": runs["passes"][4]})
n = 256
h = np.where(I.radius_grid(n, n, 1.0 / n) <= 0.48, 0.0, I.EXCLUDED)
with bem.Handle(n, n, 1.0 / n, 1.0 / n, 0.5, 0.3) as hd:
    a, _ = hd.solve(h, 0.01, precision="fp32")
    inject(1)
    t0 = time.time()
    _, rc = hd.solve(h, 0.01, precision="fp32", check=False)
    wait, msg = time.time() - t0, bem.load_library().bem_last_error().decode()
    inject(0)
    b, _ = hd.solve(h, 0.01, precision="fp32")
print(json.dumps({"runs": out, "rc": rc, "wait": wait, "msg": msg, "force": [a.force, b.force]}))
"""


@pytest.fixture(scope="module")
def result(cuda_ok, tmp_path_factory):
    env = dict(os.environ, BEM_DEBUG_CHECKS="1")
    env.pop("BEM_INJECT_WAIT_TIMEOUT", None)
    r = subprocess.run([sys.executable, "-c", CASE % ROOT], capture_output=True, text=True, env=env, timeout=900,
                       cwd=str(tmp_path_factory.mktemp("gather")))
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_loop_held_back_runs_as_passes(result):
    for r in result["runs"]:
        assert r["rc"] == 0 and r["counts"] and r["rounds"], r
        assert r["err"] <= 1e-9, r
        # the cooperative loop is a launch where the passes are three or six an iteration
        if r["case"][4] == "coop":
            assert r["launches"] < 0.5 * r["passes"], r
        else:
            assert r["launches"] > 0.5 * r["passes"], r


def test_later_wait_runs_out_and_handle_recovers(result):
    assert result["rc"] == -5 and "gave up waiting" in result["msg"]
    assert result["wait"] < 30.0
    assert result["force"][0] == result["force"][1]
