"""Single simulator steps over every kind of contact set the solver tells
apart: the ball in the air, on the floor alone (closed form), on a box alone,
on the floor and a box (ball rows only), against links (1, 2, 3 and more
contacts, the Gauss-Seidel sweeps with the blocks in registers and in shared
memory), and links on boxes.  Same bits in every layout, and within the
single-step parity bound 1e-4 max(1, |x|) of the FP64 oracle."""
import collections
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _scene(cfg):
    sc = scenes.config(cfg)
    ball = sc.x0[sc.nu:sc.nu + 3]
    # two slabs near the ball
    bc = np.array([ball + [0.0, 0.16, 0.0], ball + ([0.05, -0.17, 0.1] if cfg == 1 else [0.0, -0.35, 0.05])])
    # (beside the planar arms: a row across their plane has no joint to act on)
    bh = np.array([[0.2, 0.05, 0.06], [0.1, 0.05 if cfg == 1 else 0.1, 0.04]])
    return dataclasses.replace(sc, boxes_c=bc, boxes_h=bh)


def states(cfg, n, seed):
    sc = _scene(cfg)
    om = oracle.Model(sc.to_blob())
    rng = np.random.default_rng(seed)
    kinds, out = collections.Counter(), []
    U = rng.normal(0.0, 0.4, (n, sc.nu)).astype(np.float32).astype(np.float64)
    while len(out) < n:
        x = scenes.random_states(sc, 1, int(rng.integers(1 << 30)), q_spread=0.25 if cfg == 1 else 0.1, v_spread=0.3)[0]
        fk = om.fk(x[:sc.nq])
        pick = rng.integers(4)
        if pick == 0:      # near the floor, sometimes above it
            x[sc.nu:sc.nu + 3] += rng.uniform([-0.3, -0.5, -0.01], [0.3, 0.0, 0.05])
        elif pick == 1:    # at a link
            a, i = rng.integers(2), rng.integers(sc.n_a)
            x[sc.nu:sc.nu + 3] = fk["a1"][a, i] + rng.uniform(-0.09, 0.09, 3)
        elif pick == 2:    # at a box
            b = rng.integers(2)
            side = np.where(rng.random(3) < 0.5, -1.0, 1.0) * rng.uniform(0.5, 1.0, 3)
            x[sc.nu:sc.nu + 3] = sc.boxes_c[b] + side * (sc.boxes_h[b] + 0.6 * sc.ball_r)
        else:              # between the hands, at its start
            x[sc.nu:sc.nu + 3] += rng.uniform(-0.05, 0.05, 3)
        x = x.astype(np.float32).astype(np.float64)
        if x[sc.nu + 2] < sc.ball_r - 0.05 or om.min_abs_dist(x) < 1e-4:
            continue
        cons = om.step(x, U[len(out)], want_contacts=True)[3]
        if any(c["dist"] < -0.06 for c in cons):
            continue
        links = sum(c["bodyB"] >= 0 or c["bodyA"] < sc.nu for c in cons)
        kind = ("air" if not cons else
                f"ball x{len(cons)}" + (" floor" if cons[0]["box"] < 0 else " box") if links == 0 else
                f"links {min(len(cons), 4)}")
        kinds[kind] += 1
        out.append(x)
    return sc, om, np.array(out), U, kinds


@pytest.mark.parametrize("cfg", [1, 2])
def test_single_steps_over_contact_sets(cfg):
    from paper_2511_21264_gb300 import native
    n = 300
    sc, om, X, U, kinds = states(cfg, n, 17 + cfg)
    for kind in ("air", "ball x1 floor", "ball x1 box", "ball x2 floor", "links 1", "links 2", "links 3"):
        assert kinds[kind] >= 2, kinds
    assert sum(v for k, v in kinds.items() if k.endswith("4")) >= 2 or cfg == 1, kinds
    ctl = native.Controller(native.Model(sc.to_blob()), n, 1, sc.lam, sc.sigma_vec(), 3)
    outs = []
    for lps in (32, 16, 8) if cfg == 1 else (32, 16):
        for place in (0, 1):
            ctl.set_layout(lps, place)
            x = torch.tensor(X.astype(np.float32), device=DEV)
            ctl.sim_step(x, torch.tensor(U.astype(np.float32), device=DEV))
            assert ctl.sync() == 0
            outs.append(x.cpu().numpy())
    for o in outs[1:]:
        np.testing.assert_array_equal(o, outs[0])
    for i in range(n):
        ref = om.step(X[i], U[i])[0]
        assert np.abs(outs[0][i] - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max()), i
