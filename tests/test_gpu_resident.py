"""Phases with the grid on chip (k_resident, forced by RTM_RESIDENT=C,R) against
the single-step kernel: the same arithmetic in the same order, so traces,
images, Born data and checkpointed images are equal bit for bit for every
cluster size and rows per thread, snapshot format, odd counts of steps, sponge
widths that are not multiples of 4, dx != dz, and receivers in any pattern."""
import os

import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ENV = ("RTM_RESIDENT", "RTM_STEP_KERNEL")


class _Env:
    def __init__(self, **env):
        self.env = env

    def __enter__(self):
        self.old = {k: os.environ.pop(k, None) for k in ENV}
        os.environ.update(self.env)
        self.ctx = rtm.Context(0)
        return self.ctx

    def __exit__(self, *a):
        self.ctx.close()
        for k in ENV:
            os.environ.pop(k, None)
            if self.old[k] is not None:
                os.environ[k] = self.old[k]


def _everything(ctx, s, vel, seis, refl):
    keep = rtm._Keep()
    acq = rtm.make_acq(keep, s.src_ix, s.src_iz, s.rec_ix, s.rec_iz, s.wavelet.astype(np.float32))
    g = rtm.make_grid(*s.grid_tuple())
    v, d, m = (torch.from_numpy(a).cuda() for a in (vel, seis, refl))
    out = []
    t = torch.zeros((s.nshot, s.nt, s.nrec), dtype=torch.float32, device="cuda")
    out.append(ctx.model(g, v, acq, -1, t).clone())
    for isnap, snap, cp in ((4, rtm.SNAP_F32, 0), (3, rtm.SNAP_F32, 0), (1, rtm.SNAP_F16, 0),
                            (2, rtm.SNAP_F16, 0), (3, rtm.SNAP_BF16, 0), (4, rtm.SNAP_F32, 40),
                            (3, rtm.SNAP_F16, 10), (999, rtm.SNAP_F32, 0)):
        img = torch.zeros((s.nz, s.nx), dtype=torch.float32, device="cuda")
        out.append(ctx.migrate(g, v, acq, d, rtm.Opts(isnap, snap, 1e-6, 1, cp), img).clone())
    for isnap, snap in ((4, rtm.SNAP_F32), (3, rtm.SNAP_F16)):
        t = torch.zeros_like(t)
        out.append(ctx.born(g, v, acq, m, rtm.Opts(isnap, snap, 1e-6, 0), t).clone())
    torch.cuda.synchronize()
    return [o.cpu().numpy() for o in out]


def _survey(nx, nz, nb, dx, dz, nt, receivers):
    v = inputs.layered_faulted(nz, nx, dx, dz, seed=5, water_depth=0.2 * nz * dz)
    src_ix = np.array([0, nx // 2, nx - 1], np.int32)
    src_iz = np.array([min(1, nz - 1), nz // 2, nz - 1], np.int32)
    if receivers == "row":
        rec_ix, rec_iz = np.arange(nx), np.full(nx, min(1, nz - 1))
    elif receivers == "reversed":  # the order of the table is not the order of the cells
        rec_ix, rec_iz = np.arange(nx)[::-1], np.full(nx, nz - 1)
    else:  # scattered over neighbouring rows, some strips with one receiver, some with none
        cells = np.unique((inputs.uniform(3, 90) * (nx * min(nz, 12))).astype(np.int64))
        rec_ix, rec_iz = cells % nx, cells // nx
    return inputs.Survey(nx, nz, nb, dx, dz, 1e-3, nt, v.astype(np.float32), src_ix, src_iz,
                         np.ascontiguousarray(rec_ix, np.int32), np.ascontiguousarray(rec_iz, np.int32),
                         inputs.ricker(20.0, 1e-3, nt))


# cluster size and rows a thread: one block, rows that do not divide a block's,
# a last block with fewer than 4 rows or none, every register variant
@pytest.mark.parametrize("nx,nz,nb,dz,nt,receivers,shapes", [
    (30, 20, 8, 10.0, 61, "row", ("1", "2,4", "4,3")),
    (61, 33, 5, 10.0, 83, "scattered", ("1,4", "2,3", "2,5", "4,2", "8,1", "8,4")),
    (118, 77, 13, 10.0, 120, "row", ("8,2", "8,6", "16,1", "16,3", "4,6")),
    (90, 47, 20, 12.0, 101, "reversed", ("16,1", "16,4", "4,3", "2,6")),
    (5, 69, 0, 10.0, 57, "scattered", ("16,1", "8,2", "2,5")),
    (201, 101, 20, 10.0, 90, "row", ("16", "8", "4")),
    (470, 90, 20, 10.0, 40, "row", ("8,5", "8,6", "16,4")),
])
def test_resident_phases_equal_single_steps(nx, nz, nb, dz, nt, receivers, shapes):
    s = _survey(nx, nz, nb, 10.0, dz, nt, receivers)
    seis = (inputs.normal(9, 3 * nt * s.nrec).reshape(3, nt, s.nrec) * 1e-3).astype(np.float32)
    refl = (inputs.normal(4, nx * nz).reshape(nz, nx) * 0.05).astype(np.float32)
    with _Env(RTM_STEP_KERNEL="1") as ctx:
        want = _everything(ctx, s, s.vel, seis, refl)
    with _Env() as ctx:  # the library's own choice
        for k, (a, b) in enumerate(zip(_everything(ctx, s, s.vel, seis, refl), want)):
            assert np.array_equal(a, b), ("default", k)
    for shape in shapes:
        with _Env(RTM_RESIDENT=shape) as ctx:
            before = ctx.stats()["launches"]
            got = _everything(ctx, s, s.vel, seis, refl)
            launches = ctx.stats()["launches"] - before
        # the tile kernels would take nt / 2 launches or more for one modelling alone
        assert launches < 6 * nt, (shape, launches)
        for k, (a, b) in enumerate(zip(got, want)):
            assert np.array_equal(a, b), (shape, k)


def test_many_items_take_rounds_of_clusters():
    # more items than clusters run at once, several samples, one shot's data each
    nx, nz, nt = 118, 77, 64
    s = _survey(nx, nz, 13, 10.0, 10.0, nt, "row")
    vels = np.stack([inputs.perturb(s.vel.astype(np.float64), 10.0, 10.0, 70 + i, water_depth=100.0)
                     for i in range(40)]).astype(np.float32)
    seis = (inputs.normal(9, 3 * nt * s.nrec).reshape(3, nt, s.nrec) * 1e-3).astype(np.float32)

    def images(ctx):
        keep = rtm._Keep()
        acq = rtm.make_acq(keep, s.src_ix, s.src_iz, s.rec_ix, s.rec_iz, s.wavelet.astype(np.float32))
        out = torch.zeros((40, nz, nx), dtype=torch.float32, device="cuda")
        ctx.migrate_ensemble(rtm.make_grid(*s.grid_tuple()), torch.from_numpy(vels).cuda(), acq,
                             torch.from_numpy(seis).cuda(), rtm.Opts(2, rtm.SNAP_F16, 1e-6, 1), out)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    with _Env(RTM_STEP_KERNEL="2") as ctx:
        want = images(ctx)
    for shape in ("16", "4", "2"):
        with _Env(RTM_RESIDENT=shape) as ctx:
            assert np.array_equal(images(ctx), want), shape
