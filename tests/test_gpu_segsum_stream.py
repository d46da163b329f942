"""Integer segmented sums of more than 2^20 elements in segments of 16 on average and more (the stream):
segments across tiles, ranges and the whole array, runs of empty and of one-element segments, ragged ends;
every integer type and map, exact."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _lengths(kind, S, N):
    g = synth.rng(S + N)
    if kind == "uniform":
        x = g.integers(0, 2 * N // S + 1, size=S)
    elif kind == "one-element segments, then long ones":
        x = np.ones(S, dtype=np.int64)
        x[S // 2:] = (N - S // 2) // (S - S // 2)
    elif kind == "empty, one segment, empty":
        x = np.zeros(S, dtype=np.int64)
        x[S // 2] = N
    elif kind == "empty ones inside a tile":
        x = np.full(S, 0, dtype=np.int64)
        x[::S // 8] = N // 8
        x[1::S // 8] = 3
    elif kind == "tile by tile":                      # ends on the tiles' ends of 4-byte and 8-byte elements
        x = np.full(S, 2048, dtype=np.int64)
    return x


@pytest.mark.parametrize("kind,S,N", [("uniform", 9000, 3_000_003), ("uniform", 1100, 1_060_001), ("uniform", 130_000, 2_200_000),
                                      ("one-element segments, then long ones", 60_000, 2_000_000),
                                      ("empty, one segment, empty", 70_000, 1_500_001), ("empty, one segment, empty", 1, 40_000_013),
                                      ("empty ones inside a tile", 80_000, 5_000_000), ("tile by tile", 1000, 0)])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_sums_are_exact(kind, S, N, dtype):
    ln = _lengths(kind, S, N)
    off = np.concatenate([[0], np.cumsum(ln)])
    n = int(off[-1])
    assert n > 1 << 20 and n >= 16 * S
    x = synth.rng(n).integers(-(1 << 31), 1 << 31, size=n).astype(np.int32)
    t = torch.from_numpy(x).to(DEV).to(dtype)
    o = torch.from_numpy(off).to(DEV)
    y = x.astype(np.int64)
    for mp, v in [(api.MAP_SQ_PLUS_ONE, y * y + 1), (api.MAP_IDENTITY, y), (api.MAP_NEG, -y), (api.MAP_ABS, np.abs(y)),
                  (api.MAP_SCALE, 7 * y)]:
        P = np.concatenate([np.zeros(1, np.uint64), np.cumsum(v.view(np.uint64))])   # modulo 2^64, like the sums
        ref = (P[off[1:]] - P[off[:-1]]).view(np.int64)
        for out in (torch.int64, torch.int32):
            got = api.accel_segreduce(api.RED_ADD, mp, t, o, out, scalar=7.0).cpu().numpy()
            assert np.array_equal(got, ref if out == torch.int64 else ref.astype(np.int32))
