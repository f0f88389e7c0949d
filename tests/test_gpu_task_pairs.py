"""The ball-task suite's screened collision pairs: on 16 and 32 lanes per
sample (same bits), over horizons long enough for the bounds of skipped pairs
to run down, with slow and fast arms, small and large barrier rates (gamma = 0
skips nothing) and a collision weight that makes the barrier and penetration
terms the largest part of the cost; against the oracle, which tests every
pair, within the suite's bound 1e-3 |c| + 1e-3.  A ragged sample count, and the
default shape of a large controller."""
import numpy as np
import pytest

import oracle
from paper_2511_21264_gb300 import scenes
from tests.test_gpu_task import _cases, _f32, _t

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("cfg,phase,gamma,H,v", [(1, 0, 0.2, 24, 2.0), (2, 0, 0.05, 24, 1.0), (3, 0, 0.2, 16, 0.5),
                                                  (3, 1, 0.6, 16, 2.0), (3, 1, 0.0, 4, 0.5)])
def test_screened_pairs_match_oracle(cfg, phase, gamma, H, v):
    from paper_2511_21264_gb300 import native
    K = 33
    sc = scenes.config(cfg)
    blob = sc.to_blob()
    om = oracle.Model(blob)
    task = _f32(scenes.ball_task(sc, phase=phase, gamma=gamma, w_c=20.0))
    X, U, ref = _cases(sc, om, task, K, H, 300 + cfg, v_spread=v)
    ctl = native.Controller(native.Model(blob), K, H, sc.lam, sc.sigma_vec(), 3)
    ctl.set_task_cost(task)
    got = []
    for lps in (32, 16):
        ctl.set_layout(lps, 0)
        costs = torch.empty(K, device=DEV)
        ctl.rollout_batch(_t(X), _t(U), costs)
        assert ctl.sync() == 0
        got.append(costs.cpu().numpy())
    np.testing.assert_array_equal(got[0], got[1])
    err = np.abs(got[0] - ref) - (1e-3 * np.abs(ref) + 1e-3)
    assert err.max() <= 0.0, (err.argmax(), got[0][err.argmax()], ref[err.argmax()])


def test_large_controller_runs_the_suite_on_16_lanes_with_the_same_bits():
    from paper_2511_21264_gb300 import native
    sc = scenes.config(3)
    K, H = 2500, 6
    ctl = native.Controller(native.Model(sc.to_blob()), K, H, 20.0, sc.sigma_vec(), 3)
    assert ctl.get_layout()[0] == 16
    ctl.set_task_cost(scenes.ball_task(sc, phase=1))
    outs = []
    for lps, spc in ((16, 0), (16, 32), (32, 0), (32, 3)):
        ctl.set_launch(0)
        ctl.set_layout(lps, 0)
        ctl.set_launch(spc)
        ctl.set_iteration(0)
        u = torch.zeros((H, sc.nu), device=DEV)
        ctl.step(_t(sc.x0), u)
        assert ctl.sync() == 0
        outs.append(u.cpu().numpy())
    for o in outs[1:]:
        np.testing.assert_array_equal(o, outs[0])
