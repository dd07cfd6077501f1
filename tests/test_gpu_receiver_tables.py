"""Receiver sets other than one row: a grid that no cluster of blocks holds does not
pay for the tables of the phases on chip, and phases run on chip only where their
receivers do not make that the slower form."""
import time

import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _model_time(monkeypatch, resident, nx, nz, nt, rec_ix, rec_iz, nshot=1, reps=7):
    """Shortest host time of a modelling call, and its traces."""
    monkeypatch.delenv("RTM_RESIDENT", raising=False)
    if resident is not None:
        monkeypatch.setenv("RTM_RESIDENT", resident)
    keep = rtm._Keep()
    sx = np.linspace(3, nx - 4, nshot).astype(np.int32)
    acq = rtm.make_acq(keep, sx, np.full(nshot, 1, np.int32), np.ascontiguousarray(rec_ix, np.int32),
                       np.ascontiguousarray(rec_iz, np.int32),
                       inputs.ricker(18.0, 1e-3, nt).astype(np.float32))
    grid = rtm.make_grid(nx, nz, 20, 10.0, 10.0, 1e-3, nt)
    v = torch.full((nz, nx), 2000.0, device="cuda")
    out = torch.zeros((nshot, nt, len(rec_ix)), device="cuda")
    best = np.inf
    with rtm.Context(0) as ctx:
        for _ in range(reps):
            torch.cuda.synchronize()
            a = time.perf_counter()
            ctx.model(grid, v, acq, -1, out)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - a)
    return best, out


def test_tables_of_a_grid_off_chip(monkeypatch):
    nx, nz, rows = 1201, 501, 500
    rec_ix, rec_iz = np.tile(np.arange(nx), rows), np.repeat(np.arange(rows), nx)
    want, a = _model_time(monkeypatch, "0", nx, nz, 4, rec_ix, rec_iz)
    got, b = _model_time(monkeypatch, None, nx, nz, 4, rec_ix, rec_iz)
    assert torch.equal(a, b)
    assert got < 1.25 * want, (got, want)  # (22 ms against 14)


@pytest.mark.parametrize("what", ["row", "ten rows", "well", "four wells", "every cell"])
def test_receivers_that_suit_the_tiles_better(what, monkeypatch):
    # 30 items: a row is faster on chip, the others with tiles
    nx, nz = 301, 151
    cells = {"row": [(i, 1) for i in range(nx)], "ten rows": [(i, k) for k in range(10) for i in range(nx)],
             "well": [(nx // 2, k) for k in range(nz)],
             "four wells": [(i, k) for i in (5, 50, 70, nx - 3) for k in range(nz)],
             "every cell": [(i, k) for k in range(nz) for i in range(nx)]}[what]
    rec_ix, rec_iz = np.array(cells, np.int64).T
    tiles, a = _model_time(monkeypatch, "0", nx, nz, 200, rec_ix, rec_iz, nshot=30, reps=5)
    default, b = _model_time(monkeypatch, None, nx, nz, 200, rec_ix, rec_iz, nshot=30, reps=5)
    assert torch.equal(a, b)
    assert default < 1.15 * tiles, (default, tiles)
    if what == "row":
        assert default < 0.9 * tiles, (default, tiles)
