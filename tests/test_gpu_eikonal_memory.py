"""The traveltime solver's scratch: problems in groups of samples and chunks of
sources where all of them would take more than its 2 GB, and in smaller ones
where the device has less left; the results are the same bits."""
import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _models(n, nz, nx):
    return torch.from_numpy(np.stack([inputs.layered_faulted(nz, nx, 40.0, 40.0, seed=s + 1,
                                                             water_depth=80.0)
                                      for s in range(n)]).astype(np.float32)).cuda()


def _solve(ctx, vel, nsrc, fields=False):
    n, nz, nx = vel.shape
    t = torch.zeros((n, nsrc, nx), device="cuda")
    f = torch.zeros((n, nsrc, nz, nx), device="cuda") if fields else None
    six = np.linspace(0, nx - 1, nsrc).astype(np.int32)
    it = ctx.eikonal(vel, 40.0, 40.0, np.arange(nsrc, dtype=np.int32) % nz, six,
                     np.zeros(nx, np.int32), np.arange(nx, dtype=np.int32), times=t, fields=f)
    return t, f, it


# padded copies of 10 MB a problem: chunks of one sample's sources; groups of samples
@pytest.mark.parametrize("nsample,nsrc", [(1, 230), (5, 60)])
def test_groups_and_chunks(nsample, nsrc, monkeypatch):
    vel = _models(nsample, 700, 700)
    with rtm.Context(0) as ctx:
        monkeypatch.delenv("RTM_EIK_TILE", raising=False)
        t, f, it = _solve(ctx, vel, nsrc, fields=True)
        monkeypatch.setenv("RTM_EIK_TILE", "2x2")
        t2, f2, it2 = _solve(ctx, vel, nsrc, fields=True)
    assert torch.equal(t, t2) and torch.equal(f, f2) and it == it2


def test_a_nearly_full_device():
    # 64 x 34 problems want 1 GB; the bare fields would be 326 MB
    vel = _models(8, 88, 426).repeat(8, 1, 1)
    with rtm.Context(0) as ctx:
        want, _, it = _solve(ctx, vel, 34)
    with rtm.Context(0) as ctx:
        _solve(ctx, vel[:1], 34)
        _solve(ctx, vel[:1], 300)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8, device="cuda")
        try:
            got, _, it2 = _solve(ctx, vel, 34)
        finally:
            del hog
            torch.cuda.empty_cache()
    assert torch.equal(got, want) and it2 == it


def test_a_nearly_full_device_and_a_tall_grid():
    # 1600 problems of 1500 x 40 go to the diagonal sweeps, whose fields are 384 MB; with
    # less left they come in groups to the row-owning solver
    vel = _models(1, 1500, 40)
    with rtm.Context(0) as ctx:
        want, _, it = _solve(ctx, vel, 1600)
    with rtm.Context(0) as ctx:
        _solve(ctx, vel, 2)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device="cuda")
        try:
            got, _, it2 = _solve(ctx, vel, 1600)
        finally:
            del hog
            torch.cuda.empty_cache()
    assert torch.equal(got, want) and it2 == it
