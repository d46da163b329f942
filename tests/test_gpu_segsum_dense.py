"""Integer segmented sums as a stream where hundreds to thousands of segments end in one tile of 16 KB (many tiny
segments side by side among long ones): both ways of looking up their boundaries, exact."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _check(ln, dtype):
    off = np.concatenate([[0], np.cumsum(ln)])
    n, S = int(off[-1]), len(ln)
    assert n > 1 << 20 and n >= 17 * S
    x = synth.rng(n).integers(-(1 << 31), 1 << 31, size=n).astype(np.int64)
    t, o = torch.from_numpy(x).to(DEV).to(dtype), torch.from_numpy(off).to(DEV)
    for mp, v in ((api.MAP_SQ_PLUS_ONE, x * x + 1), (api.MAP_SCALE, 7 * x)):
        P = np.concatenate([np.zeros(1, np.uint64), np.cumsum(v.view(np.uint64))])
        ref = (P[off[1:]] - P[off[:-1]]).view(np.int64)
        got = api.accel_segreduce(api.RED_ADD, mp, t, o, torch.int64, scalar=7.0).cpu().numpy()
        assert np.array_equal(got, ref)


# segments that end in a tile: around 248 + 496, where the way changes; as many as a tile of either type has
# elements; more than a round of all warps (992); with empty ones, more than fit a tile, and with 8,192 of them
@pytest.mark.parametrize("ends", [743, 744, 745, 746, 991, 992, 993, 1240, 1488, 2046, 2047, 2048])
@pytest.mark.parametrize("empty", [0, 1, 3, 9000])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_tiny_segments_in_a_tile(ends, empty, dtype):
    tile = 16384 // dtype.itemsize
    ln = []
    for k in range(24):
        lead = (0, tile - ends, (tile - ends) // 2)[k % 3]          # at the tile's start, end, middle
        ones = np.ones(ends, np.int64)
        if 0 < empty < 10:
            ones = np.repeat(ones, 1 + empty)
            ones[np.arange(len(ones)) % (1 + empty) != k % (1 + empty)] = 0
        elif empty:
            ones = np.insert(ones, [ends // 3] * (empty if k < 3 else 0), 0)
        n = ([lead] if lead else []) + ones.tolist()
        ln += n + [4 * tile - int(np.sum(n))]
    tail = 17 * (len(ln) + 1) + (1 << 20) + 5
    _check(np.asarray(ln + [tail], np.int64), dtype)


# whole ranges of tiny segments, from the first element and to the last, ragged at the end
@pytest.mark.parametrize("kind", ["first", "last", "middle"])
@pytest.mark.parametrize("size", [1, 2, 3, 5])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_ranges_of_tiny_segments(kind, size, dtype):
    tiny = np.full(60_000, size, np.int64)
    tiny[::7] = 0
    tiny[:5] = 0
    rest = np.full(9_000, 400, np.int64)
    ln = {"first": [tiny, rest], "last": [rest, tiny, [1]], "middle": [rest[:4000], tiny, rest[4000:]]}[kind]
    _check(np.concatenate([np.asarray(v, np.int64) for v in ln]), dtype)
