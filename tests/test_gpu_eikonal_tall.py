"""Many problems of a tall grid: whole calls cost about what the diagonal sweeps
cost (the row-owning warps' padded copies of such a grid are 50 times its
nodes), and the results are the same bits."""
import time

import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_many_tall_problems_do_not_stream_their_padding(monkeypatch):
    nz, nx, nsrc = 1500, 40, 1600
    vel = inputs.layered_faulted(nz, nx, 40.0, 40.0, seed=1, water_depth=80.0)[None].astype(np.float32)
    v = torch.from_numpy(vel).cuda()
    t = torch.zeros((1, nsrc, nx), device="cuda")
    six, siz = np.arange(nsrc, dtype=np.int32) % nx, np.arange(nsrc, dtype=np.int32) % 7
    rec, top = np.arange(nx, dtype=np.int32), np.zeros(nx, np.int32)
    best, got = {}, {}
    with rtm.Context(0) as ctx:
        for name in ("default", "2x2"):
            if name == "default":
                monkeypatch.delenv("RTM_EIK_TILE", raising=False)
            else:
                monkeypatch.setenv("RTM_EIK_TILE", name)
            best[name] = np.inf
            for _ in range(3):
                torch.cuda.synchronize()
                a = time.perf_counter()
                it = ctx.eikonal(v, 40.0, 40.0, siz, six, top, rec, times=t)
                best[name] = min(best[name], time.perf_counter() - a)
            got[name] = (t.cpu().numpy().view(np.uint32), it)
    assert np.array_equal(got["default"][0], got["2x2"][0]) and got["default"][1] == got["2x2"][1]
    assert best["default"] < 2.5 * best["2x2"], best  # (it took 5 times as long)
