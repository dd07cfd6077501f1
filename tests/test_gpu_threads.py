"""Contexts in several host threads whose calls run the same kernels with
different amounts of shared memory: no thread's launch depends on what another
thread's last one needed."""
import threading

import numpy as np
import pytest

from paper_2001_06444_gb300 import rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _race(big, small, calls):
    """`big` (context, call) repeated in one thread while `small` runs in another."""
    done, errors = threading.Event(), []

    def loop(make, until):
        try:
            with rtm.Context(0) as ctx, torch.cuda.stream(torch.cuda.Stream()):
                call = make(ctx)
                k = 0
                while not until(k):
                    call()
                    k += 1
        except Exception as e:  # noqa: BLE001 - reported below, whatever it is
            errors.append(e)
        finally:
            done.set()

    threads = [threading.Thread(target=loop, args=(big, lambda k: k >= calls or errors)),
               threading.Thread(target=loop, args=(small, lambda k: done.is_set()))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def _eikonal(nx):
    def make(ctx):
        vel = torch.full((1, 96, nx), 2000.0, device="cuda")
        t = torch.zeros((1, 1, 4), device="cuda")
        rec = np.arange(4, dtype=np.int32)
        torch.cuda.current_stream().synchronize()
        return lambda: ctx.eikonal(vel, 10.0, 10.0, [0], [1], np.zeros(4, np.int32), rec, times=t,
                                   storage="shared")
    return make


@pytest.mark.parametrize("tile", [None, "2x2"])
def test_traveltimes_of_two_grids(tile, monkeypatch):
    monkeypatch.delenv("RTM_EIK_TILE", raising=False)
    if tile:
        monkeypatch.setenv("RTM_EIK_TILE", tile)
    # fields of 92 KB and of 9 KB, the same kernel
    _race(_eikonal(240), _eikonal(24), 1500)


def test_statistics_of_two_ensembles():
    def make(n):
        def inner(ctx):
            x = torch.randn((n, 8), device="cuda")
            out = [torch.zeros(8, dtype=t, device="cuda")
                   for t in (torch.float64, torch.float64, torch.float32, torch.float32)]
            torch.cuda.current_stream().synchronize()
            return lambda: ctx.ensemble_stats(x, *out)
        return inner

    _race(make(20000), make(13000), 300)  # columns of 128 KB and of 64 KB
