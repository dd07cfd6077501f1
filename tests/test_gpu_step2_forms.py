"""The forms of the two-step kernel that the library dispatches by the launch's
size, each forced: tiles of 16, 24 and 32 rows, as programmatic dependents of the
launch before and without (16 and 24 rows wait for d and c behind the Laplacians).
Modelling, migration in every snapshot format, checkpointed migration and Born
modelling are bitwise those of the single-step kernel, also with phases captured
into graphs and with host seismograms uploaded behind the forward phase; so are
the library's own choices with and without phases on chip."""
import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm
from test_gpu_resident import _everything, _survey

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = [dict(RTM_STEP_KERNEL="4", RTM_TILE_Z=z, RTM_PDL=p) for z in ("16", "24", "32") for p in "01"]
FORMS += [dict(RTM_STEP_KERNEL="4", RTM_TILE_Z="16", RTM_IMAGE_INPUT="1", RTM_PDL=p) for p in "01"]
FORMS += [dict(RTM_RESIDENT="0"), dict(RTM_RESIDENT="0", RTM_PDL="0"), dict()]


def _context(monkeypatch, env):
    for k in ("RTM_STEP_KERNEL", "RTM_TILE_Z", "RTM_PDL", "RTM_IMAGE_INPUT", "RTM_RESIDENT",
              "RTM_GRAPHS"):
        monkeypatch.delenv(k, raising=False)
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    return rtm.Context(0)


# several tiles a side, the last of them with one row of the grid (73 = 3 x 24 + 1 =
# 4 x 16 + 9), dx != dz, a grid of one tile
@pytest.mark.parametrize("nx,nz,nb,dz,nt,receivers", [
    (250, 90, 13, 10.0, 61, "row"), (250, 47, 13, 10.0, 60, "scattered"),
    (130, 86, 9, 12.0, 61, "reversed"), (40, 11, 2, 10.0, 41, "row")])
def test_forms_bitwise(nx, nz, nb, dz, nt, receivers, monkeypatch):
    s = _survey(nx, nz, nb, 10.0, dz, nt, receivers)
    seis = (inputs.normal(9, 3 * nt * s.nrec).reshape(3, nt, s.nrec) * 1e-3).astype(np.float32)
    refl = (inputs.normal(4, nx * nz).reshape(nz, nx) * 0.05).astype(np.float32)
    with _context(monkeypatch, dict(RTM_STEP_KERNEL="1")) as ctx:
        want = _everything(ctx, s, s.vel, seis, refl)
    for env in FORMS:
        with _context(monkeypatch, env) as ctx:
            got = _everything(ctx, s, s.vel, seis, refl)
        for k, (a, b) in enumerate(zip(got, want)):
            assert np.array_equal(a, b), (env, k)


def test_graphs_and_host_seismograms_bitwise(monkeypatch):
    nx, nz, nt = 250, 90, 80
    s = _survey(nx, nz, 13, 10.0, 10.0, nt, "row")
    seis = (inputs.normal(9, 3 * nt * nx).reshape(3, nt, nx) * 1e-3).astype(np.float32)
    keep = rtm._Keep()
    acq = rtm.make_acq(keep, s.src_ix, s.src_iz, s.rec_ix, s.rec_iz, s.wavelet.astype(np.float32))
    g = rtm.make_grid(*s.grid_tuple())
    v, d = torch.from_numpy(s.vel).cuda(), torch.from_numpy(seis).cuda()
    pinned = torch.from_numpy(seis).pin_memory()
    side = torch.cuda.Stream()

    def images(ctx, host, stream):
        out = []
        for isnap, snap, cp in ((4, rtm.SNAP_F32, 0), (2, rtm.SNAP_F16, 0), (4, rtm.SNAP_F32, 24)):
            opts = rtm.Opts(isnap, snap, 1e-6, 1, cp)
            with torch.cuda.stream(stream):
                if host:
                    img = np.zeros((nz, nx), np.float32)
                    ctx.migrate(g, s.vel, acq, pinned, opts, img)
                else:
                    img = torch.zeros((nz, nx), device="cuda")
                    ctx.migrate(g, v, acq, d, opts, img)
            torch.cuda.synchronize()
            out.append(img if host else img.cpu().numpy())
        return out

    with _context(monkeypatch, dict(RTM_STEP_KERNEL="1")) as ctx:
        want = images(ctx, False, torch.cuda.default_stream())
    for env in FORMS:
        for graphs in "01":
            with _context(monkeypatch, dict(env, RTM_GRAPHS=graphs)) as ctx:
                ctx.set_batch(2)  # two batches
                for host in (False, True):
                    for stream in (torch.cuda.default_stream(), side):
                        side.wait_stream(torch.cuda.default_stream())
                        ctx.stats(reset=True)
                        got = images(ctx, host, stream)
                        captured = ctx.stats()["graph_launches"]
                        assert (captured > 0) == (graphs == "1"), (env, graphs, host, captured)
                        for k, (a, b) in enumerate(zip(got, want)):
                            assert np.array_equal(a, b), (env, graphs, host, stream, k)


def test_repeated_receivers_bitwise(monkeypatch):
    """Receivers that share a cell: every kernel records them alike and injects all
    of them (with equal data, so that the order of the additions does not show)."""
    nx, nz, nt = 118, 77, 60
    s = _survey(nx, nz, 13, 10.0, 10.0, nt, "row")
    rec = np.r_[np.arange(nx), np.arange(0, nx, 3), np.arange(0, nx, 3), [5, 5, 5, 5, nx - 1]]
    s = inputs.Survey(nx, nz, 13, 10.0, 10.0, 1e-3, nt, s.vel, s.src_ix, s.src_iz,
                      np.ascontiguousarray(rec, np.int32), np.full(len(rec), 1, np.int32), s.wavelet)
    trace = (inputs.normal(9, 3 * nt * nx).reshape(3, nt, nx) * 1e-3).astype(np.float32)
    seis = np.ascontiguousarray(trace[:, :, rec])
    refl = (inputs.normal(4, nx * nz).reshape(nz, nx) * 0.05).astype(np.float32)
    with _context(monkeypatch, dict(RTM_STEP_KERNEL="1")) as ctx:
        want = _everything(ctx, s, s.vel, seis, refl)
    assert np.array_equal(want[0][:, :, :nx][:, :, rec], want[0])
    forms = FORMS + [dict(RTM_STEP_KERNEL=k) for k in "23"]
    forms += [dict(RTM_RESIDENT=c) for c in ("16,1", "8,2", "4,5", "8,6")]
    for env in forms:
        with _context(monkeypatch, env) as ctx:
            got = _everything(ctx, s, s.vel, seis, refl)
        for k, (a, b) in enumerate(zip(got, want)):
            assert np.array_equal(a, b), (env, k)
