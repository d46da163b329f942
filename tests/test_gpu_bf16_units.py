"""Saved configurations of the BF16 forward whose units were clusters of two or four CTAs: they launch as many CTAs."""
import json

import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _time(tmp_path, args, pair, units):
    K, M, S = args[0].shape[0], args[1].shape[1], args[4].numel() - 1
    path = tmp_path / f"saved{pair}_{units}.jsonl"
    path.write_text(json.dumps({"kernel": "hmm_forward_bf16", "device": torch.cuda.get_device_name(), "K": K, "M": M,
                                "S_log2": S.bit_length() - 1, "split": 2, "rows": 32, "pair": pair, "units": units,
                                "ms": 1.0}) + "\n")
    assert api.hmm_autotune(*args, cache_path=str(path)) == (0.0, (2, 32, pair, units))
    ms = []
    for _ in range(5):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        ll = api.hmm_forward(*args, api.HMM_BF16_SCALED)
        e[1].record()
        torch.cuda.synchronize()
        ms.append(e[0].elapsed_time(e[1]))
    return sorted(ms)[2], ll


def test_units_of_clusters_are_as_many_ctas(tmp_path):
    # 16 tiles of 32 sequences of one length, one after the other on a CTA: the time is the number of rounds
    p = synth.hmm_workload(1, 256, 8, 512, "fixed", 300, 300)
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")]
    one, ref = _time(tmp_path, args, 0, 1)
    for pair, units, ctas in ((1, 1, 2), (2, 1, 4), (1, 3, 6), (0, 4, 4)):
        ms, ll = _time(tmp_path, args, pair, units)
        rounds = -(-16 // ctas)
        assert 0.7 * rounds / 16 <= ms / one <= 1.4 * rounds / 16, (pair, units, ms, one)
        assert torch.equal(ll, ref)
