"""The hand-overs between the warps of the BF16 forward: thousands of steps in a row, with tiles whose maxima are
taken by warps of their own (16 and 32 sequences) and with tiles where the epilogue takes them (64)."""
import json

import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# 128 and fewer states: one issuing warp; more: two, of which one may be a step ahead of the max warps
@pytest.mark.parametrize("K", [64, 128, 192, 256])
@pytest.mark.parametrize("n", [16, 32, 64])
def test_many_steps_without_a_lost_phase(tmp_path, K, n):
    M, S, T = 8, 200, 4001
    p = synth.hmm_workload(K + n, K, M, S, "fixed", T, T)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")]
    split, rows = (4, 32) if n == 16 else (2, n)
    path = tmp_path / "tile.jsonl"
    path.write_text(json.dumps({"kernel": "hmm_forward_bf16", "device": torch.cuda.get_device_name(), "K": K, "M": M,
                                "S_log2": S.bit_length() - 1, "split": split, "rows": rows, "pair": 0, "units": 0,
                                "ms": 1.0}) + "\n")
    assert api.hmm_autotune(*args, cache_path=str(path))[0] == 0.0
    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    api.set_device_status(word)
    try:
        runs = [api.hmm_forward(*args, api.HMM_BF16_SCALED) for _ in range(20)]
        api.sync_status(word)                      # no wait gave up
    finally:
        api.set_device_status(None)
    for r in runs[1:]:
        assert torch.equal(r, runs[0])
    at = list(range(0, S, 41))
    ref = ohmm.loglik_batch(p, seqs=at, params=ohmm.params_from_f32_logs(logs))
    assert np.all(np.abs(runs[0].cpu().numpy()[at] - ref) <= 1e-3 * np.abs(ref))
