"""Decoding of large groups (1024 segments of 4096 blocks and more) by whole
segments: the same values as decoding a few arrays at a time by windows, for
segments of several, partly empty and clipped windows, both modes in one call, on
either side of the line; and the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2001_06444_gb300 import inputs, rtm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 260 x 301: 4940 blocks, two segments; 9 x 13: one segment of 12 blocks; 1 x 16385:
# a segment and one block
@pytest.mark.parametrize("n0,n1,count", [(260, 301, 513), (9, 13, 1023), (9, 13, 1024), (1, 16385, 512)])
def test_segments_decode_as_windows(n0, n1, count):
    kinds = 5
    x = (inputs.normal(3, kinds * n0 * n1).reshape(kinds, n0, n1) * 2.0).astype(np.float32)
    x[0, :, : n1 // 3] = 0.0      # the left third is empty
    x[1] = 0.0                    # everything is ...
    x[1, -1, -1] = 5.0            # ... but the last value
    x[2, : n0 // 2] = 0.0         # the first windows are
    x[3] = 0.0
    with rtm.Context(0) as ctx:
        d = torch.from_numpy(x).cuda()
        a, stride, _ = ctx.compress(d, 1e-3)
        b, stride_b, _ = ctx.compress(d, 0.0)
        assert stride == stride_b
        streams = torch.stack([a.view(kinds, stride), b.view(kinds, stride)])
        want = torch.full((2, kinds, n0, n1), 7.0, device="cuda")
        for m in range(2):
            ctx.decompress(streams[m].contiguous().view(-1), stride, kinds, n0, n1, want[m])
        pick = (torch.arange(count, device="cuda") * 7) % (2 * kinds)
        big = streams.view(2 * kinds, stride)[pick].contiguous()
        y = torch.full((count, n0, n1), 7.0, device="cuda")
        ctx.decompress(big.view(-1), stride, count, n0, n1, y)
        assert torch.equal(y.view(torch.int32), want.view(2 * kinds, n0, n1)[pick].view(torch.int32))
        for m, tol in enumerate((1e-3, 0.0)):
            for k in (0, 1):
                ref = oracle.codec_decompress(oracle.codec_compress(x[k], tol), n0, n1)
                assert np.array_equal(want[m, k].cpu().numpy().view(np.uint32), ref.view(np.uint32)), (m, k)


def test_damaged_stream_in_a_large_group_is_named():
    n0, n1, count = 9, 13, 1100
    x = inputs.normal(5, n0 * n1).reshape(1, n0, n1).astype(np.float32)
    with rtm.Context(0) as ctx:
        a, stride, sizes = ctx.compress(torch.from_numpy(x).cuda(), 1e-3)
        big = a.view(1, stride).expand(count, stride).contiguous()
        y = torch.zeros((count, n0, n1), device="cuda")
        ctx.decompress(big.view(-1), stride, count, n0, n1, y)
        good = y.clone()
        big[700, 64 + 16:int(sizes[0])] = 255  # its bits, behind the header and the index
        with pytest.raises(rtm.RTMError) as e:
            ctx.decompress(big.view(-1), stride, count, n0, n1, y)
        assert e.value.code == rtm.RTM_ERR_ARG and "stream 700" in str(e.value)
        keep = torch.arange(count, device="cuda") != 700
        assert torch.equal(y[keep], good[keep])
