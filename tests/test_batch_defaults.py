"""A new batch's default layout and shape over the sample counts where the rule
changes: the instances' results stay bitwise those of single controllers."""
import pytest

from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("cfg,K,layout", [(2, 600, (32, 4)), (2, 609, (16, 2)), (3, 2500, (16, 16)), (1, 1200, (32, 4)),
                                          (1, 2500, (16, 16))])
def test_default_layout_keeps_single_controller_bits(tmp_path, monkeypatch, cfg, K, layout):
    monkeypatch.setenv("MPPI_TUNE_FILE", str(tmp_path / "none.txt"))
    from paper_2511_21264_gb300 import native
    sc = scenes.config(cfg)
    H = 5
    m = native.Model(sc.to_blob())
    b = native.Batch([(m, K, H, 1.0, sc.sigma_vec(), 5), (m, K + 3, H, 1.0, sc.sigma_vec(), 6)])
    assert (b.get_layout()[0], b.get_launch()[0]) == layout
    x = torch.tensor(m.home(), device=DEV)
    us = [torch.zeros((H, sc.nu), device=DEV) for _ in range(2)]
    for _ in range(2):
        b.step([x, x], us)
    assert b.sync()[0] == 0
    for k, (n, key) in enumerate(((K, 5), (K + 3, 6))):
        ctl = native.Controller(m, n, H, 1.0, sc.sigma_vec(), key)
        u = torch.zeros((H, sc.nu), device=DEV)
        for _ in range(2):
            ctl.step(x, u)
        assert ctl.sync() == 0
        assert torch.equal(u, us[k])
