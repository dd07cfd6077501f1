"""RTM_EIK_SHARED holds for every grid whose field fits shared memory, the ones
that only fit without the row-owning solver's padding included: no off-chip work
fields are taken for them, and the results are those of the other storages."""
import numpy as np
import pytest

from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# of 231,424 bytes: 230 x 240 and 150 x 380 (padded: more than a CTA has), and the
# largest square with and without padding
@pytest.mark.parametrize("nz,nx", [(230, 240), (150, 380), (240, 241), (180, 180)])
def test_shared_storage_takes_no_work_fields(nz, nx):
    nsrc = 400
    vel = torch.from_numpy(inputs.layered_faulted(nz, nx, 40.0, 40.0, seed=2, water_depth=80.0)
                           .astype(np.float32)[None]).cuda()
    siz, six = np.arange(nsrc, dtype=np.int32) % nz, np.arange(nsrc, dtype=np.int32) % nx
    rec, top = np.arange(nx, dtype=np.int32), np.zeros(nx, np.int32)
    got = {}
    for storage in ("shared", "offchip"):
        t = torch.zeros((1, nsrc, nx), device="cuda")
        with rtm.Context(0) as ctx:
            # (the kernels are loaded before memory is counted)
            ctx.eikonal(vel, 40.0, 40.0, siz[:1], six[:1], top, rec, times=t[:, :1], storage=storage)
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            it = ctx.eikonal(vel, 40.0, 40.0, siz, six, top, rec, times=t, storage=storage)
            torch.cuda.synchronize()
            taken = free - torch.cuda.mem_get_info()[0]
        got[storage] = (t.cpu().numpy().view(np.uint32), it)
        # two copies of every problem's field alone are more than 4 nz nx bytes each
        if storage == "shared":
            assert taken < nsrc * nz * nx * 4 // 2, (storage, taken)
    assert np.array_equal(got["shared"][0], got["offchip"][0]) and got["shared"][1] == got["offchip"][1]
