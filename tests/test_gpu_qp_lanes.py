"""The projection's lane form at the edges of its shapes: horizons around the
steps per lane, with empty slots, one step per lane, around 32 (where the
band factor's rounding enters) and 80 (where the long form takes over), few
and many sequences (1 to 16 lanes each, ragged tails); and joints with
different free row groups (one table each).

Tolerance: |v_gpu - v_oracle| <= 2e-4 + 1e-4 |v|, the bound of the projection's
other parity tests; an FP32 emulation of the lane form stays within 2e-6 of
the oracle up to 32 steps, and the FP32 band factor that longer horizons share
with the long form moves an element by less than 1e-4."""
import numpy as np
import pytest

import oracle
from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
BOUNDS = [-0.25, 0.25, -1.0, 1.0, -10.0, 10.0, -300.0, 300.0]


def _t(a):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, np.float32)), device=DEV)


@pytest.mark.parametrize("n", [1, 131, 5000])
@pytest.mark.parametrize("H", [1, 2, 3, 5, 7, 15, 16, 17, 27, 31, 32, 33, 49, 63, 64, 65, 79, 80, 81])
def test_lane_form_matches_oracle(n, H):
    from paper_2511_21264_gb300 import native
    rng = np.random.default_rng(1000 * H + n)
    vt = (0.2 + 0.3 * rng.normal(size=(n, H))).astype(np.float32)
    q, qd = (rng.uniform(-0.2, 0.2, n).astype(np.float32) for _ in range(2))
    out = torch.full((n, H), np.nan, device=DEV)
    native.qp_project(_t(vt), np.array(BOUNDS), _t(q), _t(qd), 0.01, iters=20, v_out=out)
    v = out.cpu().numpy().astype(np.float64)
    pick = sorted({0, 1, n // 2, n - 2, n - 1} & set(range(n)))
    for i in pick:
        ref = oracle.qp_project(vt[i], BOUNDS, q[i], qd[i], float(np.float32(0.01)), 1.0, 20)[0]
        assert np.max(np.abs(v[i] - ref) - 1e-4 * np.abs(ref)) <= 2e-4, i
    assert np.isfinite(v).all()


@pytest.mark.parametrize("H", [9, 32, 41, 100])
def test_joints_with_different_free_groups(H):
    from paper_2511_21264_gb300 import native
    K = 37
    sc = scenes.config(1)
    b = scenes.projection_bounds(sc).astype(np.float32).astype(np.float64)
    b[1, 0:2] = b[2, 4:6] = b[3, 6:8] = b[4, 2:4] = [-np.inf, np.inf]
    key = scenes.controller_key(4, H)
    ctl = native.Controller(native.Model(sc.to_blob()), K, H, 1.0, sc.sigma_vec(), key)
    ctl.set_projection(b, iters=15)
    x = np.asarray(sc.x0, np.float32)
    u, U = torch.zeros((H, sc.nu), device=DEV), torch.empty((H, K, sc.nu), device=DEV)
    ctl.step(_t(x), u)
    assert ctl.sync() == 0
    got = ctl.samples(U).cpu().numpy().astype(np.float64)
    raw = oracle.noise(key, 0, K, H, sc.nu, sc.sigma_vec().astype(np.float32).astype(np.float64))
    for k in (0, 1, K // 2, K - 1):
        for j in range(sc.nu):
            ref = oracle.qp_project(raw[k, :, j], b[j], x[j], x[sc.nq + j], sc.dt, 1.0, 15)[0]
            assert np.max(np.abs(got[:, k, j] - ref) - 1e-4 * np.abs(ref)) <= 2e-4, (k, j)
