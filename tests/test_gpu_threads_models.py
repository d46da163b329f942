"""Host threads that call at once with models of different sizes: kernels they share are launched with different
amounts of dynamic shared memory, and no call takes another's away."""
import ctypes as C
import threading

import pytest
import torch

from paper_2211_00621_gb300 import _lib, api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, seed):
    p = synth.hmm_workload(seed, K, M, 6, "uniform", 3, 20)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    return args + [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")], int(p["lengths"].max())


def _at_once(calls, reps):
    """calls[q]() on a thread of its own, reps times; the statuses that were not OK."""
    bad, start = [], threading.Barrier(len(calls))

    def work(q):
        try:
            start.wait()
            for _ in range(reps):
                st = calls[q]()
                if st != 0:
                    bad.append((q, st, _lib.load().accel_last_error()))
                    return
        except Exception as e:                      # surfaced by the caller
            bad.append((q, e))

    th = [threading.Thread(target=work, args=(q,)) for q in range(len(calls))]
    for x in th:
        x.start()
    for x in th:
        x.join()
    torch.cuda.synchronize()
    return bad


# two models that need more than the 48 KB every launch may have, two that need less
@pytest.mark.parametrize("precision,models", [(api.HMM_FP32_LOG, [(64, 600), (64, 3), (50, 300), (40, 5)]),
                                              (api.HMM_BF16_SCALED, [(128, 300), (128, 3), (128, 200), (128, 4)])])
def test_forward(precision, models):
    lib, calls, outs, refs, keep = _lib.load(), [], [], [], []
    for q, (K, M) in enumerate(models):
        args, _ = _inputs(K, M, q)
        refs.append(api.hmm_forward(*args, precision))
        m, S, n = api._model(*args[:3]), 6, args[3].numel()
        ws = api._ws(lib.hmm_forward_workspace_size(C.byref(m), S, n, precision), DEV)
        out = torch.empty(S, dtype=torch.float64, device=DEV)
        stream = torch.cuda.Stream()
        keep.append((args, m, ws, stream))
        outs.append(out)
        a = (C.byref(m), precision, args[3].data_ptr(), args[4].data_ptr(), S, n, out.data_ptr(), ws.data_ptr(), ws.numel(),
             stream.cuda_stream)
        calls.append(lambda a=a: lib.hmm_forward(*a))
    torch.cuda.synchronize()
    assert not _at_once(calls, 5000)
    assert all(torch.equal(a, b) for a, b in zip(outs, refs))


def test_adjoint():
    lib, calls, outs, refs, keep = _lib.load(), [], [], [], []
    for q, (K, M) in enumerate([(256, 64), (256, 3), (64, 5), (128, 200)]):
        args, max_T = _inputs(K, M, q)
        refs.append(api.hmm_adjoint(*args, max_T=max_T))
        m, S, n = api._model(*args[:3]), 6, args[3].numel()
        ws = api._ws(lib.hmm_adjoint_workspace_size(C.byref(m), S, n, max_T), DEV)
        out = [torch.empty_like(t) for t in refs[-1]]
        stream = torch.cuda.Stream()
        keep.append((args, m, ws, stream))
        outs.append(out)
        a = (C.byref(m), args[3].data_ptr(), args[4].data_ptr(), S, n, max_T, None, out[3].data_ptr(),
             *(t.data_ptr() for t in out[:3]), ws.data_ptr(), ws.numel(), stream.cuda_stream)
        calls.append(lambda a=a: lib.hmm_adjoint(*a))
    torch.cuda.synchronize()
    assert not _at_once(calls, 1500)
    for out, ref in zip(outs, refs):
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
