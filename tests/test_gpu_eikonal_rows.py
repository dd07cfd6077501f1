"""The row-owning traveltime solver against the diagonal one (RTM_EIK_TILE
selects it): both run the sequential sweeps' updates, so fields, panels and
iteration counts are equal bit for bit, in either storage."""
import os

import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(ctx, vel, dz, dx, siz, six, storage, tile=None, max_iter=0):
    nz, nx = vel.shape[1:]
    old = os.environ.pop("RTM_EIK_TILE", None)
    if tile:
        os.environ["RTM_EIK_TILE"] = tile
    try:
        f = torch.zeros((vel.shape[0], len(siz), nz, nx), dtype=torch.float32, device="cuda")
        t = torch.zeros((vel.shape[0], len(siz), nx), dtype=torch.float32, device="cuda")
        rec = np.arange(nx, dtype=np.int32)
        it = ctx.eikonal(torch.from_numpy(vel).cuda(), dz, dx, siz, six, np.full(nx, nz - 1, np.int32),
                         rec, times=t, fields=f, storage=storage, max_iter=max_iter)
        return f.cpu().numpy().view(np.uint32), t.cpu().numpy().view(np.uint32), it
    finally:
        os.environ.pop("RTM_EIK_TILE", None)
        if old is not None:
            os.environ["RTM_EIK_TILE"] = old


# rows per lane 1 to 4 and their edges, a lane with one row, several warps (a
# last warp of one lane), columns that end inside a tile, spacings that differ
@pytest.mark.parametrize("nz,nx,dz,dx", [(1, 1, 10.0, 10.0), (1, 9, 10.0, 10.0), (7, 3, 10.0, 12.0),
                                         (32, 5, 10.0, 10.0), (33, 64, 10.0, 10.0), (64, 67, 10.0, 9.0),
                                         (65, 30, 10.0, 10.0), (97, 41, 10.0, 10.0),
                                         (128, 130, 10.0, 10.0), (129, 70, 10.0, 11.0),
                                         (260, 33, 10.0, 10.0), (385, 58, 10.0, 10.0)])
def test_rows_equal_the_diagonal_sweeps(nz, nx, dz, dx):
    vel = np.stack([inputs.layered_faulted(nz, nx, dz, dx, seed=s, water_depth=40.0)
                    for s in (3, 4)]).astype(np.float32)
    vel *= (1.0 + 0.2 * inputs.normal(8, vel.size).clip(-2, 2).reshape(vel.shape)).astype(np.float32)
    siz = np.array([0, nz - 1, nz // 2, nz // 3], np.int32)
    six = np.array([nx // 2, 0, nx - 1, nx // 3], np.int32)
    with rtm.Context(0) as ctx:
        want = _solve(ctx, vel, dz, dx, siz, six, "offchip", tile="2x2")
        for storage in ("auto", "shared", "offchip"):
            got = _solve(ctx, vel, dz, dx, siz, six, storage)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), storage
            assert got[2] == want[2], storage


@pytest.mark.parametrize("cap", [1, 2, 3])
def test_cap_gives_the_same_answer(cap):
    # stopped at a cap (or converged just below it), both solvers say the same
    nz, nx = 50, 61
    vel = inputs.layered_faulted(nz, nx, 10.0, 10.0, seed=9)[None].astype(np.float32)

    def answer(ctx, tile):
        try:
            return _solve(ctx, vel, 10.0, 10.0, [nz - 1], [nx - 1], "auto", tile=tile, max_iter=cap)[2]
        except rtm.RTMError as e:
            return e.code

    with rtm.Context(0) as ctx:
        assert answer(ctx, None) == answer(ctx, "2x2")
