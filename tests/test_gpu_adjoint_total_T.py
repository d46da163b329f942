"""The adjoint called with a total_T that its offsets go past: the workspace holds the rows of total_T steps, so
the sequences beyond them are skipped and reported, nothing is written past it, and the others' results stand."""
import ctypes as C

import pytest
import torch

from paper_2211_00621_gb300 import _lib, api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("K,fit", [(37, 0), (64, 1), (128, 9), (200, 25), (256, 29)])
def test_sequences_past_total_T_are_skipped_and_reported(K, fit):
    S, M = 30, 6
    p = synth.hmm_workload(K, K, M, S, "uniform", 20, 80)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    obs, off = (torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets"))
    max_T = int(p["lengths"].max())
    short = int(p["offsets"][fit]) + 7                       # the first `fit` sequences, and part of the next
    lib, m = _lib.load(), api._model(*args)
    need = lib.hmm_adjoint_workspace_size(C.byref(m), S, short, max_T)
    guard = torch.full((need + (1 << 20),), 77, dtype=torch.uint8, device=DEV)
    ll = torch.full((S,), float("nan"), dtype=torch.float64, device=DEV)
    g = [torch.empty(s, device=DEV) for s in ((K, K), (K, M), (K,))]
    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    api.set_device_status(word)
    try:
        _lib.check("hmm_adjoint", lib.hmm_adjoint(C.byref(m), api._ptr(obs), api._ptr(off), S, short, max_T, None,
                                                  api._ptr(ll), *(api._ptr(t) for t in g), api._ptr(guard), need,
                                                  api._stream()))
        with pytest.raises(_lib.AccelError) as e:
            api.sync_status(word)
        assert e.value.status == 2
    finally:
        api.set_device_status(None)
    assert bool((guard[need:] == 77).all())
    assert bool(ll[fit:].isnan().all())
    if fit:
        want = api.hmm_adjoint(*args, obs[: int(off[fit])].contiguous(), off[: fit + 1].contiguous(), max_T=max_T)
        assert torch.equal(ll[:fit], want[3])
        for a, b in zip(g, want[:3]):
            # the rows of the products are cut at other places
            assert torch.all((a - b).abs() <= 1e-5 * b.abs() + 1e-7 * b.abs().sum())
    else:
        assert all(not t.any() for t in g)
