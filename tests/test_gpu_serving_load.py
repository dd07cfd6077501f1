"""Requests that run side by side are launched for the device they share, not each
as if it were alone: no slower than with the two-step kernel of fixed tiles, and the
images are the same bits."""
import time

import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _serve(monkeypatch, kernel, nx, nz, nshot, nreq, nt=300):
    monkeypatch.delenv("RTM_STEP_KERNEL", raising=False)
    if kernel:
        monkeypatch.setenv("RTM_STEP_KERNEL", kernel)
    keep = rtm._Keep()
    sx = np.linspace(3, nx - 4, nshot).astype(np.int32)
    acq = rtm.make_acq(keep, sx, np.full(nshot, 1, np.int32), np.arange(nx, dtype=np.int32),
                       np.full(nx, 1, np.int32), inputs.ricker(18.0, 1e-3, nt).astype(np.float32))
    grid = rtm.make_grid(nx, nz, 20, 10.0, 10.0, 1e-3, nt)
    vel = torch.full((nz, nx), 2000.0, device="cuda")
    seis = torch.from_numpy((inputs.normal(9, nshot * nt * nx).reshape(nshot, nt, nx) * 1e-3)
                            .astype(np.float32)).cuda()
    images = torch.zeros((nreq, nz, nx), device="cuda")
    torch.cuda.synchronize()  # the request loop's streams do not wait for this one
    best = np.inf
    with rtm.Context(0, budget_bytes=64 << 30) as ctx:
        reqs = [rtm.Request(grid, vel.data_ptr(), acq, seis.data_ptr(),
                            rtm.Opts(4, rtm.SNAP_F16, 1e-6, 1, 0), images[k].data_ptr())
                for k in range(nreq)]
        for _ in range(7):
            a = time.perf_counter()
            for t in [ctx.submit(r) for r in reqs]:
                assert ctx.poll(t, 60000)[0] == rtm.REQ_DONE
            best = min(best, time.perf_counter() - a)
        torch.cuda.synchronize()
    return best, images


@pytest.mark.parametrize("nx,nz,nshot,nreq", [(401, 111, 12, 8), (851, 176, 4, 4), (201, 101, 2, 6)])
def test_requests_side_by_side(nx, nz, nshot, nreq, monkeypatch):
    fixed, a = _serve(monkeypatch, "2", nx, nz, nshot, nreq)
    default, b = _serve(monkeypatch, None, nx, nz, nshot, nreq)
    assert torch.equal(a, b)
    assert default < 1.12 * fixed, (default, fixed)  # (1.19 and 1.22 when planned alone)
