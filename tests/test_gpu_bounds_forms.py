"""The bounds-check build (see test_gpu_bounds.py) over the forms of the
kernels that the small cases there do not reach: the projection's lane form
with empty slots, with 1 to 16 lanes per sequence and with one table per joint,
its long form above 80 steps, both standalone forms with ragged counts; the
ball-task suite on both layouts; several contacts at once, with the solve of
a lone one in both placements; a batch with projected samples.  Results match
the oracle and no check fails."""
import json
import subprocess
import sys

import pytest

from tests.test_gpu_bounds import ROOT

pytestmark = pytest.mark.gpu

CHILD = r'''
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
import oracle
from paper_2511_21264_gb300 import native, scenes
native.LIB_PATH = native.BOUNDS_LIB_PATH
import ctypes as C
import torch
L = native.lib()
word, checked = C.c_uint(), C.c_int()

def take():
    assert L.mppi_debug_bounds(C.byref(word), C.byref(checked)) == 0
    return int(word.value)

take()
out = {"checked": int(checked.value), "words": {}, "qp_err": {}, "step_err": {}}
f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
T = lambda a: torch.tensor(np.ascontiguousarray(np.asarray(a, np.float32)), device="cuda")
B = [-0.25, 0.25, -1.0, 1.0, -10.0, 10.0, -300.0, 300.0]
rng = np.random.default_rng(3)
# standalone: lanes 1..16 (few and many sequences), empty slots, the long form with 64 and 32 threads
for n, H in ((1, 1), (131, 5), (3, 17), (131, 27), (5000, 27), (20000, 16), (40000, 33), (131, 49), (70, 79), (131, 80),
             (131, 81), (70, 100), (33, 256)):
    vt = (0.2 + 0.3 * rng.normal(size=(n, H))).astype(np.float32)
    q, qd = (rng.uniform(-0.2, 0.2, n).astype(np.float32) for _ in range(2))
    v = torch.full((n, H), np.nan, device="cuda")
    native.qp_project(T(vt), np.array(B), T(q), T(qd), 0.01, iters=4, v_out=v)
    v = v.cpu().numpy().astype(np.float64)
    assert np.isfinite(v).all()
    for i in {0, n // 2, n - 1}:
        ref = oracle.qp_project(vt[i], B, q[i], qd[i], float(np.float32(0.01)), 1.0, 4)[0]
        err = float(np.max(np.abs(v[i] - ref) - 1e-4 * np.abs(ref)))
        out["qp_err"][f"{n}x{H}"] = max(err, out["qp_err"].get(f"{n}x{H}", -1.0))
    out["words"][f"project_{n}x{H}"] = take()
# drawn and projected, one table for all joints and one each
for cfg in (1, 3):
    sc = scenes.config(cfg)
    gm = native.Model(sc.to_blob())
    for K, H in ((5, 9), (37, 27), (900, 32), (37, 41), (5, 80), (5, 100)):
        for free in (False, True):
            b = scenes.projection_bounds(sc).astype(np.float32)
            if free:
                b[1, 0:2] = b[2, 4:6] = [-np.inf, np.inf]
            c = native.Controller(gm, K, H, sc.lam, sc.sigma_vec(), 5)
            c.set_projection(b, iters=3)
            u = torch.zeros((H, sc.nu), device="cuda")
            c.step(T(sc.x0), u, u)
            assert c.sync() == 0
            out["words"][f"cfg{cfg}_qp_{K}x{H}_{free}"] = take()
# the ball-task suite
for cfg, phase in ((1, 0), (3, 0), (3, 1)):
    sc = scenes.config(cfg)
    c = native.Controller(native.Model(sc.to_blob()), 5, 6, 20.0, sc.sigma_vec(), 5)
    c.set_task_cost(scenes.ball_task(sc, phase))
    for lps in (32, 16):
        c.set_layout(lps, 0)
        u = torch.zeros((6, sc.nu), device="cuda")
        c.step(T(sc.x0), u, u)
        assert c.sync() == 0
        out["words"][f"task_{cfg}_{phase}_{lps}"] = take()
# contacts of every kind, explicit steps and sampled ones
from tests.test_gpu_contact_counts import states
for cfg in (1, 2):
    n = 60
    sc, om, X, U, kinds = states(cfg, n, 40 + cfg)
    gm = native.Model(sc.to_blob())
    c = native.Controller(gm, n, 1, sc.lam, sc.sigma_vec(), 3)
    for lps in (32, 16, 8) if cfg == 1 else (32, 16):
        c.set_layout(lps, 0)
        x = T(X)
        c.sim_step(x, T(U))
        assert c.sync() == 0
        g = x.cpu().numpy()
        e = max(np.abs(g[i] - r).max() / max(1.0, np.abs(r).max())
                for i, r in ((i, om.step(X[i], U[i])[0]) for i in range(n)))
        out["step_err"][f"cfg{cfg}_{lps}"] = float(e)
        out["words"][f"contacts_{cfg}_{lps}"] = take()
    c = native.Controller(gm, 4, 3, sc.lam, sc.sigma_vec(), 3)
    for i in range(0, n, 6):
        for lps, place in ((32, 0), (32, 1), (16, 1)):
            c.set_layout(lps, place)
            u = torch.zeros((3, sc.nu), device="cuda")
            c.step(T(X[i]), u, u)
            assert c.sync() == 0
    out["words"][f"sampled_contacts_{cfg}"] = take()
# a batch with projected samples and elites
sc = scenes.config(3)
m = native.Model(sc.to_blob())
b = native.Batch([(m, 6, 9, sc.lam, sc.sigma_vec(), 1), (m, 9, 33, sc.lam, sc.sigma_vec(), 2)])
b.set_update(-1, 3, 0.7, True, 1e-6)
b.set_projection(np.stack([scenes.projection_bounds(sc)] * 2), iters=3)
us = [torch.zeros((h, sc.nu), device="cuda") for h in (9, 33)]
b.step([T(sc.x0)] * 2, us)
assert b.sync()[0] == 0
out["words"]["batch_qp"] = take()
print(json.dumps(out))
'''


def test_every_form_runs_clean_in_the_bounds_check_build():
    from paper_2511_21264_gb300 import native
    native.build(bounds=True)
    p = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT", repr(ROOT), 1)], capture_output=True, text=True,
                       timeout=900, cwd=ROOT)
    assert p.returncode == 0, p.stderr[-3000:]
    res = json.loads(p.stdout.strip().splitlines()[-1])
    assert res["checked"] == 1
    assert {k: w for k, w in res["words"].items() if w} == {}
    assert all(e <= 2e-4 for e in res["qp_err"].values()), res["qp_err"]      # the projection's parity bound
    assert all(e <= 1e-4 for e in res["step_err"].values()), res["step_err"]  # the single-step parity bound
