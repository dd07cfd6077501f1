"""The autotuner against the library's own rule (phases on chip, else kernel 4 with
the tile that suits the launch): the rule is a candidate, it is kept unless
something is clearly faster, it goes by each later call's own size, and where
phases run on chip no kernel is chosen by timing the same code several times.
RTM_TRACE=1 prints how each call launches; a child process reads it."""
import json
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LINE = re.compile(r"rtm-trace (\w+) .*launches: on chip (\d), kernel (\d), rows (\d+), "
                  r"dependent (-?\d), items (\d+)")

CHILD = """
import json, sys
import numpy as np, torch
from paper_2001_06444_gb300 import inputs, rtm
nx, nz, nshot, nt, nsample = map(int, sys.argv[1:6])
v = inputs.layered_faulted(nz, nx, 10.0, 10.0, seed=61, water_depth=80.0).astype(np.float32)
src = np.linspace(5, nx - 6, nshot).astype(np.int32)
keep = rtm._Keep()
rec = np.arange(nx, dtype=np.int32)
acq = rtm.make_acq(keep, src, np.full(nshot, 1, np.int32), rec, np.full(nx, 1, np.int32),
                   inputs.ricker(18.0, 1e-3, nt).astype(np.float32))
grid = rtm.make_grid(nx, nz, 20, 10.0, 10.0, 1e-3, nt)
opts = rtm.Opts(4, rtm.SNAP_F32, 1e-6, 1)
seis = torch.from_numpy((inputs.normal(5, nshot * nt * nx).reshape(nshot, nt, nx) * 1e-3)
                        .astype(np.float32)).cuda()
one = torch.from_numpy(v).cuda()
many = one[None].repeat(nsample, 1, 1).contiguous()
got = []
with rtm.Context(0) as ctx:
    for tuned in (0, 1):
        if tuned:
            choice = ctx.autotune(grid, acq, opts, trial_steps=nt)
            print("rtm-trace tuned", file=sys.stderr, flush=True)
        a = torch.zeros((nz, nx), device="cuda")
        b = torch.zeros((nsample, nz, nx), device="cuda")
        ctx.migrate(grid, one, acq, seis, opts, a)
        ctx.migrate_ensemble(grid, many, acq, seis, opts, b)
        torch.cuda.synchronize()
        got.append((a.cpu().numpy(), b.cpu().numpy()))
assert all(np.array_equal(x, y) for x, y in zip(*got))
print(json.dumps(choice))
"""


def _run(nx, nz, nshot, nt, nsample, **env):
    """(choice, lines of the trials, lines of the two calls before and after tuning)"""
    clean = {k: v for k, v in os.environ.items() if not k.startswith("RTM_") or k == "RTM_DEBUG"}
    r = subprocess.run([sys.executable, "-c", CHILD, *map(str, (nx, nz, nshot, nt, nsample))],
                       cwd=ROOT, env=dict(clean, RTM_TRACE="1", **env), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    lines = [(m[1], *map(int, m.groups()[1:])) for m in map(LINE.match, r.stderr.splitlines()) if m]
    trials = [x[1:] for x in lines if x[0] == "rtm_autotune"]
    calls = [x[1:] for x in lines if x[0] != "rtm_autotune"]
    assert len(calls) == 4 and trials
    return json.loads(r.stdout.splitlines()[-1]), trials, calls[:2], calls[2:]


def test_a_launch_that_suits_16_rows():
    # one item of 851 x 176: 16 rows 2.55 us a step, 24 rows 2.85
    choice, trials, before, after = _run(851, 176, 1, 300, 12)
    assert (0, 4, 16) in {t[:3] for t in trials}
    assert (choice["step_kernel"], choice["tile_z"], choice["max_items"]) == (4, 16, 0)
    assert before[0][1:3] == (4, 16)
    # and its 12 samples are launched by their own size, as without tuning
    assert before[1][2] != 16 and after == before


def test_phases_on_chip_are_not_told_apart_by_kernel():
    choice, trials, before, after = _run(190, 72, 3, 330, 4)
    assert all(t[0] == 1 for t in trials), trials
    assert len({t[4] for t in trials}) <= 2 and len(trials) <= 12  # 2 graphs x 2 caps x 3 runs
    assert choice["max_items"] == 0
    assert after == before


@pytest.mark.parametrize("pdl", [0, 1])
def test_dependent_launches_stay_as_asked(pdl):
    # RTM_PDL holds in the trials and after tuning
    _, trials, before, after = _run(851, 176, 2, 120, 6, RTM_PDL=str(pdl))
    lines = [t for t in trials + before + after if t[1] == 4]
    assert len(lines) >= 6 and all(t[3] == pdl for t in lines), lines
