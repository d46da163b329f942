"""The adjoint's choice of workspace on a GPU: the checkpointed form where memory is short, through the autograd
function and a given workspace; a workspace that asks the driver inside a graph capture."""
import ctypes as C

import pytest
import torch

from paper_2211_00621_gb300 import _lib, api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, S, lo, hi):
    p = synth.hmm_workload(K, K, M, S, "uniform", lo, hi)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")]
    return args, int(p["lengths"].max())


def test_autograd_and_given_workspaces_where_memory_is_short(monkeypatch):
    args, max_T = _inputs(256, 16, 400, 200, 500)
    lib, m, S, n = _lib.load(), api._model(*args[:3]), 400, args[3].numel()
    full = lib.hmm_adjoint_workspace_size(C.byref(m), S, n, max_T)
    small = lib.hmm_adjoint_min_workspace_size(C.byref(m), S, n, max_T)
    assert small < full and full > api._ADJ_ANY
    _, kept = api.hmm_adjoint_forward(*args, max_T=max_T)
    assert kept.ws.numel() == full
    want = api.hmm_adjoint(*args, max_T=max_T, ws=torch.empty(small, dtype=torch.uint8, device=DEV))
    ll, saved = api.hmm_adjoint_forward(*args, max_T=max_T, ws=torch.empty(small, dtype=torch.uint8, device=DEV))
    assert saved.ws.numel() == small and torch.equal(ll, want[3])
    del kept
    torch.cuda.empty_cache()
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda d=None: (7 * full, 0))
    p = [t.clone().requires_grad_(True) for t in args[:3]]
    ll = api.HMMLogLik.apply(*p, *args[3:], api.HMM_FP32_LOG, max_T)
    assert ll.grad_fn.saved.ws.numel() == small
    ll.sum().backward()
    assert torch.equal(ll.detach(), want[3])
    for a, b in zip(p, want):
        assert torch.equal(a.grad, b)


def test_captured_with_a_workspace_that_asks_the_driver():
    args, max_T = _inputs(128, 8, 600, 800, 1200)
    m = api._model(*args[:3])
    assert _lib.load().hmm_adjoint_workspace_size(C.byref(m), 600, args[3].numel(), max_T) > api._ADJ_ANY
    want = [t.clone() for t in api.hmm_adjoint(*args, max_T=max_T)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = api.hmm_adjoint(*args, max_T=max_T)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
