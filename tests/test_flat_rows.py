"""Contacts with a row that no joint moves: planar arms on boxes in their
plane, where the tangent across the plane has a zero Delassus diagonal.  That
row takes no impulse and the others are solved as always."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2511_21264_gb300 import scenes


def _scene(**kw):
    sc = scenes.config(1)
    om = oracle.Model(sc.to_blob())
    fk = om.fk(np.asarray(sc.x0, float)[:sc.nq])
    # a slab under either hand
    c = [fk["a1"][0, 2] + [-0.05, 0.0, -0.07], fk["a1"][1, 2] + [0.05, 0.0, -0.08]]
    h = [[0.06, 0.3, 0.05], [0.05, 0.02, 0.05]]
    return dataclasses.replace(sc, boxes_c=np.array(c), boxes_h=np.array(h), **kw)


def _states(sc, n, seed):
    """States with a link on a box, away from a change of the contact set."""
    om = oracle.Model(sc.to_blob())
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(60 * n):
        x = scenes.random_states(sc, 1, int(rng.integers(1 << 30)), q_spread=0.15, v_spread=0.5)[0]
        x = x.astype(np.float32).astype(np.float64)
        if om.min_abs_dist(x) < 1e-4:
            continue
        cons = om.step(x, np.zeros(sc.nu), want_contacts=True)[3]
        if any(c["bodyA"] < sc.nu and c["bodyA"] >= 0 for c in cons) and all(c["dist"] > -0.04 for c in cons):
            out.append(x)
            if len(out) == n:
                break
    assert len(out) == n
    return om, np.array(out)


def _point_velocity(sc, om, x, qd, link, p):
    """Velocity of the point p of a link for joint velocities qd."""
    fk, a, i = om.fk(x[:sc.nq]), link // sc.n_a, link % sc.n_a
    return sum(np.cross(fk["z"][a, j], p - fk["o"][a, j]) * qd[a * sc.n_a + j] for j in range(i + 1))


def test_oracle_solves_the_rows_that_move():
    # without regularisation (impedance 1) and friction, the only contact of an
    # arm is one row: exact after one sweep, so a pushing contact ends at its
    # reference velocity along the normal to FP64 rounding (1e-9)
    sc = _scene(impedance=1.0, mu=0.0)
    om, X = _states(sc, 40, 5)
    pushed = 0
    for x in X:
        xn, _, lam, cons = om.step(x, np.zeros(sc.nu), want_contacts=True)
        assert np.isfinite(xn).all()
        arms = [(k, c) for k, c in enumerate(cons) if 0 <= c["bodyA"] < sc.nu]
        for k, c in arms:
            assert lam[3 * k] >= 0.0
            v = _point_velocity(sc, om, x, xn[sc.nq:sc.nq + sc.nu], c["bodyA"], c["p"])
            assert v[1] == 0.0  # the arms stay in their plane
            alone = sum(b["bodyA"] // sc.n_a == c["bodyA"] // sc.n_a for _, b in arms) == 1 and c["bodyB"] < 0
            if alone and lam[3 * k] > 0.0:
                assert abs(c["n"] @ v - sc.erp / sc.dt * -c["dist"]) <= 1e-9
                pushed += 1
    assert pushed >= 5


@pytest.mark.gpu
def test_kernels_match_the_oracle():
    torch = pytest.importorskip("torch")
    from paper_2511_21264_gb300 import native
    sc = _scene()
    n = 120
    om, X = _states(sc, n, 11)
    U = np.random.default_rng(2).normal(0.0, 0.4, (n, sc.nu)).astype(np.float32).astype(np.float64)
    ctl = native.Controller(native.Model(sc.to_blob()), n, 1, sc.lam, sc.sigma_vec(), 3)
    outs = []
    for lps in (32, 16, 8):
        ctl.set_layout(lps, 0)
        x = torch.tensor(X.astype(np.float32), device="cuda:0")
        ctl.sim_step(x, torch.tensor(U.astype(np.float32), device="cuda:0"))
        assert ctl.sync() == 0
        outs.append(x.cpu().numpy())
    np.testing.assert_array_equal(outs[0], outs[1])
    np.testing.assert_array_equal(outs[0], outs[2])
    for i in range(n):  # the single-step parity bound
        ref = om.step(X[i], U[i])[0]
        assert np.abs(outs[0][i] - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max()), i
