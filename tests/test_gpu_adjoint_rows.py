"""The adjoint with every alpha kept: padded state counts, windows of symbols, uneven slots, offsets
that start inside the observations; and the checkpointed form, which a smaller workspace selects."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import _lib, api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, S, lo, hi, seed):
    p = synth.hmm_workload(seed, K, M, S, "uniform", lo, hi)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p["obs"]).to(DEV), torch.from_numpy(p["offsets"]).to(DEV)]
    return p, logs, args


def _sizes(args, max_T):
    lib = _lib.load()
    m = api._model(*args[:3])
    S, n = args[4].numel() - 1, args[3].numel()
    return (lib.hmm_adjoint_workspace_size(C.byref(m), S, n, max_T),
            lib.hmm_adjoint_min_workspace_size(C.byref(m), S, n, max_T))


def _close(g, r):
    # the adjoint's stated criterion: 1e-4 of the entry plus 1e-6 of its row's total
    g, r = g.cpu().numpy().astype(np.float64), np.asarray(r)
    assert np.all(np.abs(g - r) <= 1e-4 * np.abs(r) + 1e-6 * np.abs(r).sum(-1, keepdims=True))


# K on both sides of the padded sizes; M across one and several windows of 64 symbols; more sequences
# than the 8 slots of every cluster (S = 2500), fewer than one cluster's, and one- and two-step ones
@pytest.mark.parametrize("K,M,S,lo,hi", [(1, 3, 5, 1, 9), (3, 64, 11, 1, 40), (63, 65, 9, 2, 70), (65, 5, 30, 1, 50),
                                         (128, 300, 7, 10, 90), (129, 9, 6, 1, 60), (256, 130, 9, 1, 40),
                                         (64, 7, 2500, 1, 9), (256, 6, 1300, 1, 6), (100, 20, 1, 777, 777)])
def test_rows_form_matches_oracle_and_checkpoints(K, M, S, lo, hi):
    p, logs, args = _inputs(K, M, S, lo, hi, K + 5 * S)
    w = torch.from_numpy(synth.rng(S).uniform(0.0, 2.0, size=S)).to(DEV)
    max_T = int(p["lengths"].max())
    full, small = _sizes(args, max_T)
    got = api.hmm_adjoint(*args, weights=w, max_T=max_T)
    ll, *ref = ohmm.gradients_batch(p, weights=w.cpu().numpy(), params=ohmm.params_from_f32_logs(logs))
    for g, r in zip(got, ref):
        _close(g, r)
    assert np.all(np.abs(got[3].cpu().numpy() - ll) <= 1e-5 * np.abs(ll))
    again = api.hmm_adjoint(*args, weights=w, max_T=max_T)
    assert all(torch.equal(a, b) for a, b in zip(got, again))
    if small < full:
        cp = api.hmm_adjoint(*args, weights=w, max_T=max_T, ws=torch.empty(small, dtype=torch.uint8, device=DEV))
        for g, r in zip(cp, ref):
            _close(g, r)
        # both forms sum in FP32 in other orders: logL differs by a few roundings a step
        assert torch.all((cp[3] - got[3]).abs() <= 1e-6 * got[3].abs())


@pytest.mark.parametrize("K", [37, 256])
def test_offsets_that_start_inside_the_observations(K):
    # sequences 5 .. 14 of 20 by a slice of the offsets: the symbols before and after belong to nobody
    p, logs, args = _inputs(K, 12, 20, 3, 80, K)
    max_T = int(p["lengths"].max())
    part = api.hmm_adjoint(*args[:4], args[4][5:16].contiguous(), max_T=max_T)
    a, b = int(p["offsets"][5]), int(p["offsets"][15])
    alone = api.hmm_adjoint(*args[:3], args[3][a:b].contiguous(), (args[4][5:16] - a).contiguous(), max_T=max_T)
    assert torch.equal(part[3], alone[3])
    for x, y in zip(part[:3], alone[:3]):
        # the rows of the products are cut at other places (their number enters the cut)
        assert torch.all((x - y).abs() <= 1e-5 * y.abs() + 1e-7 * y.abs().sum())


@pytest.mark.parametrize("K", [64, 200])
def test_saved_state_of_the_checkpointed_form(K):
    # a workspace of the smaller size carries the checkpointed state from the forward to the backward
    p, logs, args = _inputs(K, 16, 30, 20, 200, 2 * K)
    max_T = int(p["lengths"].max())
    full, small = _sizes(args, max_T)
    if small >= full:
        pytest.skip("every alpha takes less memory than the checkpoints")
    lib = _lib.load()
    m = api._model(*args[:3])
    ws = torch.empty(small, dtype=torch.uint8, device=DEV)
    S, n = 30, args[3].numel()
    ll = torch.empty(S, dtype=torch.float64, device=DEV)
    _lib.check("hmm_adjoint_forward", lib.hmm_adjoint_forward(C.byref(m), args[3].data_ptr(), args[4].data_ptr(), S, n,
                                                              max_T, ll.data_ptr(), ws.data_ptr(), small, api._stream()))
    saved = api.AdjointSaved(ws, S, n, max_T)
    got = api.hmm_adjoint_backward(*args, saved)
    one = api.hmm_adjoint(*args, max_T=max_T, ws=torch.empty(small, dtype=torch.uint8, device=DEV))
    assert torch.equal(ll, one[3]) and all(torch.equal(a, b) for a, b in zip(got, one))
