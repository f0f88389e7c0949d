"""A new batch's samples per CTA are the library's choice until the caller sets
them: every layout that the header names is accepted after creation, whatever
the default shape is (16 samples on 16 lanes do not fit the 256 threads of a
CTA on 32), with the same bits; a shape that the caller set is kept."""
import pytest

from paper_2511_21264_gb300 import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("cfg,K", [(3, 2500), (1, 2500), (2, 700), (1, 40)])
def test_every_layout_after_creation(tmp_path, monkeypatch, cfg, K):
    monkeypatch.setenv("MPPI_TUNE_FILE", str(tmp_path / "none.txt"))
    from paper_2511_21264_gb300 import native
    sc = scenes.config(cfg)
    H = 4
    m = native.Model(sc.to_blob())
    x = torch.tensor(m.home(), device=DEV)
    b = native.Batch([(m, K, H, 1.0, sc.sigma_vec(), 5), (m, K + 3, H, 1.0, sc.sigma_vec(), 6)])
    first = (*b.get_layout(), b.get_launch()[0])
    outs = []
    for lps, place in ([first[:2]] + [(l, p) for l in (32, 16) + ((8,) if cfg == 1 else ()) for p in (0, 1)]
                       + [first[:2]]):
        b.set_layout(lps, place)
        b.set_iteration(-1, 0)
        us = [torch.zeros((H, sc.nu), device=DEV) for _ in range(2)]
        b.step([x, x], us)
        assert b.sync()[0] == 0
        assert b.get_layout() == (lps, place)
        outs.append(torch.stack(us))
    assert (*b.get_layout(), b.get_launch()[0]) == first  # back where it began
    assert all(torch.equal(o, outs[0]) for o in outs)
    # another order alone leaves the shape to the library; the caller's shape stays
    b.set_launch(first[2], 0)
    b.set_layout(32, 0)
    assert b.get_launch() == (4, 0)
    b.set_launch(4, 1)
    b.set_layout(32, 1)
    assert b.get_launch()[0] == 4


@pytest.mark.parametrize("cfg,H,spc", [(3, 64, 16), (3, 100, 14), (3, 146, 14), (3, 147, 16), (1, 100, 16)])
def test_default_shape_keeps_two_ctas_on_an_sm(tmp_path, monkeypatch, cfg, H, spc):
    # 6720 bytes a sample of the 7-link arms, 2608 the model, 1 KB reserved and,
    # up to 2048 values, the staged nominal sequence: two CTAs of 16 samples fit
    # an SM's 228 KB up to H = 99, two of 14 up to 146
    monkeypatch.setenv("MPPI_TUNE_FILE", str(tmp_path / "none.txt"))
    from paper_2511_21264_gb300 import native
    sc = scenes.config(cfg)
    K = 1300
    m = native.Model(sc.to_blob())
    b = native.Batch([(m, K, H, 1.0, sc.sigma_vec(), s) for s in range(4)])
    assert (b.get_layout()[0], b.get_launch()[0]) == (16, spc)
    x, us = torch.tensor(m.home(), device=DEV), [torch.zeros((H, sc.nu), device=DEV) for _ in range(4)]
    b.step([x] * 4, us)
    assert b.sync()[0] == 0
    ctl = native.Controller(m, K, H, 1.0, sc.sigma_vec(), 2)
    u = torch.zeros((H, sc.nu), device=DEV)
    ctl.step(x, u)
    assert ctl.sync() == 0 and torch.equal(u, us[2])
