"""The all-pairs kernel that evaluates each pair of bodies once: sizes around its blocks of 1,024 and 512
bodies, bodies of zero mass and at the same place, the same result on every call."""
import numpy as np
import pytest
import torch

from oracle import pairwise as opair
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _soa(b):
    return [torch.from_numpy(b["aos"][:, k].copy()).to(DEV) for k in range(4)]


@pytest.mark.parametrize("n", [24576, 24577, 25087, 25088, 25089, 26113, 30000])
def test_matches_the_oracle(n):
    assert api.L.load().pairwise_mapreduce_workspace_size(api.L.PAIR_GRAVITY_SOFTENED, n) > 0
    b = synth.bodies(n, n)
    b["aos"][n // 2, 3] = 0.0                       # a test particle
    b["aos"][7, :3] = b["aos"][n - 1, :3]           # two bodies at one place, in different blocks
    x, y, z, m = _soa(b)
    a = torch.stack(api.pairwise_mapreduce(x, y, z, m, 1e-2), 1)
    assert torch.equal(a, torch.stack(api.pairwise_mapreduce(x, y, z, m, 1e-2), 1))
    idx = sorted({0, 7, 511, 512, 1023, 1024, 1535, 1536, n // 2, n - 513, n - 512, n - 2, n - 1} | set(range(0, n, 997)))
    pos, mass = b["aos"][:, :3], b["aos"][:, 3]
    ref = opair.accel(pos, mass, 1e-2, idx)
    # FP32 terms of a few roundings each, sums in any order: well inside 1e-4 of the net force or, where that
    # cancels, of the terms' scale
    scale = np.maximum(np.linalg.norm(ref, axis=1), opair.term_scale(pos, mass, 1e-2, idx))
    err = np.linalg.norm(a.cpu().numpy().astype(np.float64)[idx] - ref, axis=1)
    assert np.all(err <= 1e-4 * scale)


def test_too_little_scratch_is_as_good():
    n = 24600
    x, y, z, m = _soa(synth.bodies(3, n))
    lib, L = api.L.load(), api.L
    want = torch.stack(api.pairwise_mapreduce(x, y, z, m, 1e-2))
    need = lib.pairwise_mapreduce_workspace_size(L.PAIR_GRAVITY_SOFTENED, n)
    ws = torch.empty(need, dtype=torch.uint8, device=DEV)
    for w, size in [(None, 0), (ws, need - 1)]:
        out = [torch.empty(n, device=DEV) for _ in range(3)]
        L.check("pairwise_mapreduce", lib.pairwise_mapreduce_ws(
            L.PAIR_GRAVITY_SOFTENED, *(api._ptr(t) for t in (x, y, z, m)), n, 1e-2, *(api._ptr(t) for t in out),
            api._ptr(w), size, api._stream()))
        got = torch.stack(out)
        # other orders of 24,600 additions
        assert torch.all((got - want).norm(dim=0) <= 1e-4 * want.norm(dim=0) + 1e-2)
