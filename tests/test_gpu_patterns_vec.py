"""map, loop and reduce by 16-byte vectors: sizes around the vectors and the unrolled rounds, inputs and
outputs that start anywhere, in place."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
# fewer elements than a vector, around one round and around kFlight rounds of 1,216 blocks of 256 threads
SIZES = [1, 3, 17, 70_001, 311_296 * 4 + 5, 311_296 * 16 + 3]
TYPES = [torch.int32, torch.int64, torch.float32, torch.float64]


def _map(op, x, out, y=None):
    L = api.L
    L.check("accel_map", L.load().accel_map(op, api._dt(x), api._ptr(x), api._ptr(y), api._dt(out), api._ptr(out), x.numel(),
                                            0.0, api._stream()))


def _values(n, dtype, skip):
    x = synth.rng(n).integers(-1000, 1000, size=n + skip)
    return torch.from_numpy(x).to(DEV).to(dtype)[skip:]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("a,b,o", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (3, 2, 1)])
def test_map(n, a, b, o):
    for tin in TYPES:
        for tout in TYPES:
            if tin.is_floating_point and not tout.is_floating_point:
                continue
            x, y = _values(n, tin, a), _values(n, tin, b)
            out = torch.full((n + o + 1,), 77, dtype=tout, device=DEV)
            _map(api.MAP_SQ_PLUS_ONE, x, out[o:o + n])
            # whole numbers below 2^24: exact in every type
            assert torch.equal(out[o:o + n], (x * x + 1).to(tout)) and out[o + n] == 77 and (o == 0 or out[o - 1] == 77)
            _map(api.MAP_ADD2, x, out[o:o + n], y)
            assert torch.equal(out[o:o + n], (x + y).to(tout)) and out[o + n] == 77


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("a,b", [(0, 0), (1, 0), (0, 2), (3, 3)])
def test_loop_and_reduce(n, a, b):
    for t in TYPES:
        x, y = _values(n, t, a).clone() if a == 0 else _values(n, t, a), _values(n, t, b)
        want = x + 3 * y
        api.accel_loop(api.LOOP_AXPY, x, y, 3.0)
        assert torch.equal(x, want)
        api.accel_loop(api.LOOP_SCALE, x, x if a == b else y, 2.0)
        assert torch.equal(x, 2 * (want if a == b else y))
        assert api.accel_reduce(api.RED_MAX, y).item() == y.max().item()
        assert api.accel_reduce(api.RED_MIN, y).item() == y.min().item()
        total = api.accel_reduce(api.RED_ADD, y).item()
        if t.is_floating_point:     # sums of n whole numbers below 1,000 in any order, in the type's precision
            u = 2.0 ** -24 if t == torch.float32 else 2.0 ** -53
            assert abs(total - y.double().sum().item()) <= n * u * y.double().abs().sum().item()
        else:
            assert total == y.sum().item()
