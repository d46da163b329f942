"""The pair histogram's table rows: edge lists with one edge an octave of 1 - cos, one a half octave, and
neither; separations down to the resolution of FP32; coordinates that are not unit vectors, infinite or
not numbers; counters that have to be emptied on the way.  Counts are exact."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
F = np.float32


def _gpu(A, e, B=None):
    tb = torch.from_numpy(B).to(DEV) if B is not None else None
    return api.accel_pair_histogram(torch.from_numpy(A).to(DEV), e, tb).cpu().numpy()


def _ref(A, e, B=None):
    with np.errstate(invalid="ignore", over="ignore"):
        P, Q = A, (A if B is None else B)
        d = (P[:, None, 0] * Q[None, :, 0] + P[:, None, 1] * Q[None, :, 1]) + P[:, None, 2] * Q[None, :, 2]
        b = (e[None, None, :] >= d[:, :, None]).sum(-1)
    if B is None:
        b = b[np.triu_indices(len(A), 1)]
    return np.bincount(b.ravel(), minlength=len(e) + 1)


EDGES = {
    "octaves": (1 - 2.0 * 4.0 ** -np.arange(9, -1, -1.0)).astype(F),
    "log angles": synth.angle_edges(20, 1.0, 10000.0),
    "half octaves": synth.angle_edges(30, 2.0, 6000.0),
    "close together": np.linspace(0.9, -0.9, 31).astype(F),
    "next to each other": np.array([1.0, 1 - 2.0 ** -24, 1 - 2.0 ** -23, 0.5, 0.25, -1.0], dtype=F),
    "beyond the sphere": np.array([np.inf, 3.0, 1.0, 0.0, -1.0, -3.0, -np.inf], dtype=F),
    "one": np.array([0.3], dtype=F),
}


@pytest.mark.parametrize("name", list(EDGES))
# whole tiles, ragged ones, fewer points than a tile of either side
@pytest.mark.parametrize("NA,NB", [(1030, None), (512, 512), (600, 264), (5, 1200)])
def test_edges_and_tiles(name, NA, NB):
    e = EDGES[name]
    A = synth.sphere_points(NA, NA)
    A[1::3] = A[0] + (A[1::3] * F(2.0) ** -np.arange(2, 2 + len(A[1::3]))[:, None].clip(2, 14)).astype(F)   # near A[0]
    B = None if NB is None else np.concatenate([A[:NB], synth.sphere_points(NB + 1, max(0, NB - NA))])
    assert np.array_equal(_gpu(A, e, B), _ref(A, e, B))


@pytest.mark.parametrize("name", list(EDGES))
def test_other_coordinates(name):
    e = EDGES[name]
    A = (synth.sphere_points(7, 520) * synth.rng(8).uniform(0.0, 3.0, size=(520, 1))).astype(F)
    A[3], A[100], A[400], A[401] = np.nan, np.inf, -np.inf, 0.0
    h, ref = _gpu(A, e), _ref(A, e)
    assert np.array_equal(h, ref)


def test_counters_are_emptied_in_time():
    # every pair in one bin, many tiles a block
    A = np.tile(np.array([[0, 0, 1]], dtype=F), (1 << 16, 1))
    B = np.tile(np.array([[0, 0.6, 0.8]], dtype=F), (1 << 18, 1))
    h = _gpu(A, EDGES["log angles"], B)
    k = int((EDGES["log angles"] >= F(0.8)).sum())
    assert h[k] == A.shape[0] * B.shape[0] and h.sum() == h[k]
