"""A sequence's projection in calls of different sizes: the lanes that share a
sequence are chosen from the number of sequences and the horizon, and order its
sums.  An FP32 emulation of the lane form with 1 to 16 lanes differs by at most
4.9e-7 of the 2-norm (H = 16 to 80); the bound is four times that.  Above 80
steps one thread holds a sequence, whatever the number: the same bits."""
import numpy as np
import pytest

from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"
BOUNDS = np.array([-1.0, 1.0, -3.14, 3.14, -10.0, 10.0, -300.0, 300.0], np.float32)


def _close(a, b, H):
    if H > 80:
        return torch.equal(a, b)
    return float((a.double() - b.double()).norm() / b.double().norm()) <= 2e-6


@pytest.mark.parametrize("H", [7, 16, 27, 32, 33, 64, 80, 81, 128])
def test_a_part_of_the_sequences_alone(H):
    from paper_2511_21264_gb300 import native
    n, m = 20000, 40
    g = torch.Generator(DEV).manual_seed(H)
    v = 0.5 * torch.randn(n, 1, device=DEV, generator=g) + 0.2 * torch.randn(n, H, device=DEV, generator=g)
    q, qd = (0.3 * (2 * torch.rand(n, device=DEV, generator=g) - 1) for _ in range(2))
    whole = native.qp_project(v, BOUNDS, q, qd, 0.01, v_out=torch.empty_like(v))
    at = n - m
    part = native.qp_project(v[at:].contiguous(), BOUNDS, q[at:].contiguous(), qd[at:].contiguous(), 0.01)
    assert _close(part, whole[at:], H)


@pytest.mark.parametrize("H", [16, 32, 64, 100])
def test_the_first_samples_of_a_larger_controller(H):
    from paper_2511_21264_gb300 import native
    sc = scenes.config(1)
    m = native.Model(sc.to_blob())
    out = []
    for K in (40, 3000):
        ctl = native.Controller(m, K, H, 1.0, sc.sigma_vec(), 11)
        ctl.set_projection(scenes.projection_bounds(sc))
        ctl.step(torch.tensor(m.home(), device=DEV), torch.zeros((H, sc.nu), device=DEV))
        U = ctl.samples(torch.empty((H, K, sc.nu), device=DEV))
        assert ctl.sync() == 0
        out.append(U[:, :40].clone())
    assert _close(out[0], out[1], H)
