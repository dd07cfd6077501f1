"""Spacings that are different doubles but the same float: their inverse squares
round to different floats, and the row-owning solver has to use each for its
direction as the diagonal sweeps do."""
import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dz,dx", [(10.0, 10.0000004), (10.0000004, 10.0), (39.999999, 40.0)])
def test_spacings_that_round_together(dz, dx, monkeypatch):
    assert np.float32(dz) == np.float32(dx)
    assert np.float32(1 / (dz * dz)) != np.float32(1 / (dx * dx))
    nz, nx = 97, 120
    vel = torch.from_numpy(inputs.layered_faulted(nz, nx, dz, dx, seed=3, water_depth=40.0)
                           .astype(np.float32)[None]).cuda()
    got = []
    with rtm.Context(0) as ctx:
        for tile in (None, "2x2"):
            if tile:
                monkeypatch.setenv("RTM_EIK_TILE", tile)
            else:
                monkeypatch.delenv("RTM_EIK_TILE", raising=False)
            for storage in ("shared", "offchip"):
                f = torch.zeros((1, 2, nz, nx), device="cuda")
                it = ctx.eikonal(vel, dz, dx, [0, 60], [5, 100], fields=f, storage=storage)
                got.append((f, it))
    for f, it in got[1:]:
        assert torch.equal(f.view(torch.int32), got[0][0].view(torch.int32)) and it == got[0][1]
