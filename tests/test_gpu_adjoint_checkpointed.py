"""The checkpointed adjoint, which a workspace of the smaller size selects (memory is short, or the rows of every
step would take more than 32 GiB): what its streams, plans and saved state are tested for, and its log-likelihoods
against those of the form that keeps every alpha."""
import ctypes as C
import threading

import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import _lib, api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, S, lo, hi, seed, kind="uniform"):
    p = synth.hmm_workload(seed, K, M, S, kind, lo, hi)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")]
    return p, logs, args, int(p["lengths"].max())


def _small(args, max_T):
    """A fresh workspace of the smaller size."""
    lib, m = _lib.load(), api._model(*args[:3])
    S, n = args[4].numel() - 1, args[3].numel()
    small = lib.hmm_adjoint_min_workspace_size(C.byref(m), S, n, max_T)
    assert small < lib.hmm_adjoint_workspace_size(C.byref(m), S, n, max_T)
    return torch.empty(small, dtype=torch.uint8, device=DEV)


def _adjoint(args, max_T, weights=None, ws=None):
    return api.hmm_adjoint(*args, weights=weights, max_T=max_T, ws=_small(args, max_T) if ws is None else ws)


def _weights(seed, S):
    return torch.from_numpy(synth.rng(seed).uniform(0.5, 2.0, size=S)).to(DEV)


# K = 64, 128 and 256 take the cluster pairs, others the streaming kernels
@pytest.mark.parametrize("K,M,S,lo,hi", [(64, 8, 200, 150, 400), (128, 16, 100, 100, 500), (256, 64, 200, 300, 700),
                                         (100, 9, 30, 200, 500)])
def test_repeated_calls_are_bit_identical(K, M, S, lo, hi):
    p, logs, args, max_T = _inputs(K, M, S, lo, hi, K + 3 * S)
    w = _weights(3, S)
    ref = None
    for rep in range(4):
        ws = _small(args, max_T).fill_(17 * rep)              # stale contents differ
        g = [t.clone() for t in _adjoint(args, max_T, w, ws)]
        ref = ref or g
        assert all(torch.equal(a, b) for a, b in zip(g, ref))
    _, *want = ohmm.gradients_batch(p, weights=w.cpu().numpy(), params=ohmm.params_from_f32_logs(logs))
    for a, b in zip(ref, want):
        a, b = a.cpu().numpy().astype(np.float64), np.asarray(b)
        assert np.all(np.abs(a - b) <= 1e-4 * np.abs(b) + 1e-6 * np.abs(b).sum(-1, keepdims=True))


@pytest.mark.parametrize("budget", [40, 8])
def test_sm_budget_gives_identical_results(budget):
    p, logs, args, max_T = _inputs(256, 64, 200, 200, 700, 77)
    w = _weights(7, 200)
    ref = [t.clone() for t in _adjoint(args, max_T, w)]
    try:
        api.set_sm_budget(budget)
        got = _adjoint(args, max_T, w)
        ll, saved = api.hmm_adjoint_forward(*args, max_T=max_T, ws=_small(args, max_T))
    finally:
        api.set_sm_budget(0)
    two = api.hmm_adjoint_backward(*args, saved, weights=w)
    for a, b, c in zip(got, ref, (*two, ll)):
        assert torch.equal(a, b) and torch.equal(c, b)


@pytest.mark.parametrize("K,M,S,lo,hi", [(64, 8, 200, 150, 400), (256, 64, 200, 300, 700), (100, 9, 30, 200, 500)])
def test_captured_in_a_cuda_graph_replays_bit_identical(K, M, S, lo, hi):
    p, logs, args, max_T = _inputs(K, M, S, lo, hi, K + 5 * S)
    w, ws = _weights(9, S), _small(args, max_T)
    ref = [t.clone() for t in _adjoint(args, max_T, w, ws)]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        _adjoint(args, max_T, w, ws)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = _adjoint(args, max_T, w, ws)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, ref))


def test_orders_with_the_callers_stream():
    p, logs, args, max_T = _inputs(128, 16, 120, 150, 400, 606)
    w_ref = _weights(12, 120)
    ref = [t.clone() for t in _adjoint(args, max_T, w_ref)]
    ws = _small(args, max_T)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    big = torch.randn(4096, 4096, device=DEV)
    w = torch.zeros(120, dtype=torch.float64, device=DEV)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(4):
            big = big @ big / 64.0                            # keeps the stream busy for a while
        w.copy_(w_ref)
        got = [t.clone() for t in _adjoint(args, max_T, w, ws)]
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, ref))


def test_from_two_host_threads_at_once():
    cases = [_inputs(K, M, S, 200, 450, 700 + K)[2:] for K, M, S in ((64, 8, 150), (256, 64, 150))]
    ref = [[t.clone() for t in _adjoint(*c)] for c in cases]
    spaces = [_small(*c) for c in cases]
    torch.cuda.synchronize()
    out, errs = [None, None], []

    def run(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(3):
                    g = _adjoint(*cases[i], ws=spaces[i])
                out[i] = [t.clone() for t in g]
            s.synchronize()
        except Exception as e:                                # surfaced below
            errs.append(e)

    th = [threading.Thread(target=run, args=(i,)) for i in range(2)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    assert not errs, errs
    for got, r in zip(out, ref):
        assert all(torch.equal(a, b) for a, b in zip(got, r))


@pytest.mark.parametrize("K,M", [(64, 8), (37, 5)])
def test_max_T_too_small_is_reported(K, M):
    p, logs, args, max_T = _inputs(K, M, 40, 150, 400, 21 + K)
    ws = _small(args, max_T)
    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    api.set_device_status(word)
    try:
        _adjoint(args, 4, ws=_small(args, 4))                 # segments of 2 steps: every sequence is too long
        with pytest.raises(_lib.AccelError) as e:
            api.sync_status(word)
        assert e.value.status == 2 and "max_T" in str(e.value)
        got = _adjoint(args, max_T, ws=ws)
        api.sync_status(word)
    finally:
        api.set_device_status(None)
    _, *want = ohmm.gradients_batch(p, params=ohmm.params_from_f32_logs(logs))
    for a, b in zip(got, want):
        assert np.linalg.norm(a.cpu().numpy() - b) <= 1e-4 * np.linalg.norm(b)


# both forms add a step's products in the same order: the same bits, in long sequences and in short ones of few
# symbols, where another order shows most; K = 64, 128 and 256 (eight parts of the rows) and others (the rows in
# order) on both sides of the padded sizes
@pytest.mark.parametrize("K", [64, 128, 256, 5, 33, 63, 65, 100, 127, 129, 200, 255])
@pytest.mark.parametrize("M,S,lo,hi", [(2, 600, 8, 60), (40, 60, 300, 500)])
def test_both_forms_give_the_same_log_likelihoods(K, M, S, lo, hi):
    for seed in range(3):
        p, logs, args, max_T = _inputs(K, M, S, lo, hi, 31 * K + seed)
        lib, m, n = _lib.load(), api._model(*args[:3]), args[3].numel()
        full = lib.hmm_adjoint_workspace_size(C.byref(m), S, n, max_T)
        # (the smaller size is that of the checkpoints only where they take less: a larger total_T's is more)
        one = api.hmm_adjoint(*args, max_T=max_T, ws=torch.empty(full, dtype=torch.uint8, device=DEV))[3]
        pad = torch.zeros(4 * n + 400_000, dtype=torch.int32, device=DEV)
        pad[:n] = args[3]
        long = [*args[:3], pad, args[4]]
        two = _adjoint(long, max_T)[3]
        assert torch.equal(one, two)
