"""Integer segmented sums as a stream, the segment left open at the end of a tile in which more segments end
than the CTA's lanes look at together (248): its start is written once, by the warp that holds it."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# `ends` segments that end in a tile, at its start, in its middle or at its end, then one that goes on into the
# next tiles: on both sides of the 248, of the 279 up to which another warp holds the open one, and of all 8 warps
@pytest.mark.parametrize("ends", [246, 247, 248, 249, 250, 260, 278, 279, 280, 310, 400, 495, 496, 497, 1240, 1241])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_open_segment_after_many_that_end(ends, dtype):
    tile = 16384 // dtype.itemsize
    ln = []
    for k in range(90):                              # three tiles each
        lead = (0, tile // 2 - ends, tile - 2 * ends - 7)[k % 3]
        lead = max(0, min(lead, tile - ends - 1))
        ones = np.ones(ends, np.int64)
        ones[:: 1 + k % 7] = k % 2                   # empty ones among them
        n = [lead, *ones.tolist()] if lead else ones.tolist()
        ln += n + [3 * tile - sum(n)]
    ln += [1 << 21]
    ln = np.asarray(ln, np.int64)
    off = np.concatenate([[0], np.cumsum(ln)])
    n, S = int(off[-1]), len(ln)
    assert n > 1 << 20 and n >= 17 * S
    x = synth.rng(ends).integers(-1000, 1001, size=n)
    ref = np.concatenate([[0], np.cumsum(x * x + 1)])
    t, o = torch.from_numpy(x).to(DEV).to(dtype), torch.from_numpy(off).to(DEV)
    for _ in range(5):
        got = api.accel_segreduce(api.RED_ADD, api.MAP_SQ_PLUS_ONE, t, o, torch.int64).cpu().numpy()
        assert np.array_equal(got, ref[off[1:]] - ref[off[:-1]])
