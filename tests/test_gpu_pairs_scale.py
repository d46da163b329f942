"""All pairs at scales where the inverse cube of a distance leaves FP32's range but the acceleration does not
(metres and kilograms), with and without scratch space."""
import numpy as np
import pytest
import torch

from oracle import pairwise as opair
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# distances up to 1.7 edge: on both sides of 2^40, where the kernel changes its form; and a softening length
# past it
@pytest.mark.parametrize("edge,mass,eps", [(1e12, 1e25, 1e9), (1.2e12, 1e25, 1e9), (1e14, 2e30, 1e11), (3e15, 2e30, 1e12),
                                           (2e17, 2e34, 1e15), (1e3, 2e30, 1e14), (1e-9, 1e-12, 1e-12)])
def test_large_and_small_units(edge, mass, eps):
    n = 24600
    b = synth.bodies(11, n)
    aos = (b["aos"] * np.array([edge, edge, edge, mass])).astype(np.float32)
    x, y, z, m = (torch.from_numpy(aos[:, k].copy()).to(DEV) for k in range(4))
    idx = list(range(0, n, 499))
    pos, w = aos[:, :3].astype(np.float64), aos[:, 3].astype(np.float64)
    ref = opair.accel(pos, w, eps, idx)
    # the criterion of the tests at unit scale
    scale = np.maximum(np.linalg.norm(ref, axis=1), opair.term_scale(pos, w, eps, idx))
    lib, L = api.L.load(), api.L
    need = lib.pairwise_mapreduce_workspace_size(L.PAIR_GRAVITY_SOFTENED, n)
    assert need > 0
    ws = torch.empty(need, dtype=torch.uint8, device=DEV)
    for scratch, size in [(ws, need), (None, 0)]:
        out = [torch.empty(n, device=DEV) for _ in range(3)]
        L.check("pairwise_mapreduce", lib.pairwise_mapreduce_ws(
            L.PAIR_GRAVITY_SOFTENED, *(api._ptr(t) for t in (x, y, z, m)), n, eps, *(api._ptr(t) for t in out),
            api._ptr(scratch), size, api._stream()))
        a = torch.stack(out, 1).cpu().numpy().astype(np.float64)[idx]
        assert np.all(np.linalg.norm(a - ref, axis=1) <= 1e-4 * scale), size
