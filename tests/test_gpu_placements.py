"""Both placements of the lone ball contact's solve over every kind of contact
set, through Controller.step, whose sampling kernels honour the placement
(explicit steps do not): the ball in the air, alone on the floor (closed form)
or on a box, on both, and against links.  Same bits in every layout and
placement, and the update within the parity bound 1e-3 of the FP64 oracle's."""
import numpy as np
import pytest

from tests.test_gpu_contact_counts import states

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


def _kind(cons, nu):
    links = sum(c["bodyB"] >= 0 or 0 <= c["bodyA"] < nu for c in cons)
    if links or not cons:
        return f"links {min(links, 2)}"
    return f"ball x{len(cons)}" + (" floor" if cons[0]["box"] < 0 else " box")


@pytest.mark.parametrize("cfg", [1, 2])
def test_placements_give_the_same_update(cfg):
    from paper_2511_21264_gb300 import native
    K, H, seed = 16, 2, 9
    sc, om, X, _, _ = states(cfg, 300, 70 + cfg)
    seen = {}
    for x in X:
        kind = _kind(om.step(x, np.zeros(sc.nu), want_contacts=True)[3], sc.nu)
        seen.setdefault(kind, [])
        if len(seen[kind]) < 4:
            seen[kind].append(x)
    for kind in ("ball x1 floor", "ball x1 box", "ball x2 floor", "links 0", "links 1"):
        assert seen.get(kind), kind
    ctl = native.Controller(native.Model(sc.to_blob()), K, H, 1.0, sc.sigma_vec(), seed)
    for kind, xs in seen.items():
        for x in xs:
            outs = []
            for lps in (32, 16, 8) if cfg == 1 else (32, 16):
                for place in (0, 1):
                    ctl.set_layout(lps, place)
                    ctl.set_iteration(0)
                    u = torch.zeros((H, sc.nu), device=DEV)
                    ctl.step(torch.tensor(x.astype(np.float32), device=DEV), u)
                    assert ctl.sync() == 0
                    outs.append(u.cpu().numpy())
            for o in outs[1:]:
                np.testing.assert_array_equal(o, outs[0], err_msg=kind)
            ref = om.mppi_iteration(x, np.zeros((H, sc.nu)), K, 1.0, sc.sigma_vec(), seed, 0)
            assert np.abs(outs[0] - ref["u_nom"]).max() <= 1e-3, kind
