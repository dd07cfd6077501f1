"""Decoding by windows of 1024 blocks and encoding a chunk a warp, at the sizes
where they can go wrong: one block short of, at and past the edges of a chunk (32
blocks), an encoder tile (128), a window and a segment (4096), block rows that
end inside a window, windows without a nonzero block.  Streams and decoded
arrays are the oracle's, byte for byte."""
import numpy as np
import pytest

import oracle
from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = rtm.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n0,n1", [(4, 4 * n) for n in (31, 32, 33, 127, 128, 129, 1023, 1024, 1025,
                                                        4095, 4096, 4097)]
                         + [(128, 128), (130, 129), (41, 4099), (2051, 9), (5 * 4, 1021)])
@pytest.mark.parametrize("tol", [1e-3, 0.0])
def test_edges_of_windows(ctx, n0, n1, tol):
    x = (inputs.normal(3, 2 * n0 * n1).reshape(2, n0, n1) * 2.0).astype(np.float32)
    x[1] = 0.0  # no block kept ...
    x[1, -1, -1] = 5.0  # ... but the last
    x[0, :, : n1 // 3] = 0.0
    d = torch.from_numpy(x).cuda()
    out, stride, sizes = ctx.compress(d, tol)
    y = torch.full_like(d, 7.0)
    ctx.decompress(out, stride, 2, n0, n1, y)
    blob, y = out.cpu().numpy(), y.cpu().numpy()
    for i in range(2):
        want = oracle.codec_compress(x[i], tol)
        assert blob[i * stride:i * stride + sizes[i]].tobytes() == want, i
        ref = oracle.codec_decompress(want, n0, n1)
        assert np.array_equal(y[i].view(np.uint32), ref.view(np.uint32)), i
