"""The BF16 forward's tiles: every tile size, partly filled tiles, one- and two-step sequences,
columns that take a second sequence, and the two emission table types."""
import json

import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, lengths, seed):
    p = synth.hmm_params(seed, K, M)
    obs, off = synth.observations(seed + 1, np.asarray(lengths, np.int64), M)
    p.update(obs=obs, offsets=off, lengths=np.asarray(lengths, np.int64), K=K, M=M, S=len(lengths))
    logs = synth.hmm_log_inputs_f32(p)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(obs).to(DEV), torch.from_numpy(off).to(DEV)]
    return p, logs, args


def _tile(tmp_path, args, n, units):
    """Make tiles of n sequences on at most `units` CTAs the configuration of these sizes."""
    K, M, S = args[0].shape[0], args[1].shape[1], args[4].numel() - 1
    split, rows = (4, 32) if n == 16 else (2, n)
    path = tmp_path / f"tile{n}.jsonl"
    path.write_text(json.dumps({"kernel": "hmm_forward_bf16", "device": torch.cuda.get_device_name(), "K": K, "M": M,
                                "S_log2": S.bit_length() - 1, "split": split, "rows": rows, "pair": 0, "units": units,
                                "ms": 1.0}) + "\n")
    ms, cfg = api.hmm_autotune(*args, cache_path=str(path))
    assert ms == 0.0 and cfg == (split, rows, 0, units)


# rows of 1, 15, 17 and 129 sequences leave a tile partly filled; one CTA (units = 1) takes every
# tile's overflow from the queue; M = 1000 and 600 take the BF16 emission table
@pytest.mark.parametrize("K,M,S,units", [(64, 5, 1, 0), (64, 1000, 15, 0), (128, 600, 17, 0), (128, 9, 129, 1),
                                         (192, 30, 70, 2), (256, 64, 129, 1), (256, 3, 300, 0)])
def test_every_tile_size(tmp_path, K, M, S, units):
    lengths = synth.seq_lengths(K + S, S, "loguniform", 1, 90)
    lengths[: min(S, 4)] = [1, 2, 3, 90][: min(S, 4)]
    p, logs, args = _inputs(K, M, lengths, 100 + S)
    ref = ohmm.loglik_batch(p, params=ohmm.params_from_f32_logs(logs))
    got = []
    for n in (16, 32, 64, 128):
        _tile(tmp_path, args, n, units)
        got.append(api.hmm_forward(*args, api.HMM_BF16_SCALED).cpu().numpy())
        # BF16 vectors (2^-9 relative an entry, averaged over the states): the stated 1e-3
        assert np.all(np.abs(got[-1] - ref) <= 1e-3 * np.abs(ref)), n
    for g in got[1:]:
        # the same products in the same order; only the exact powers of two differ, so logL differs by
        # the rounding of ln2 E + ln s in float64
        assert np.all(np.abs(g - got[0]) <= 1e-13 * np.abs(ref))


# past tiles of 16 on every SM the tile is picked on the device: equal lengths favour the larger
# size, a few long sequences among short ones the smaller
@pytest.mark.parametrize("K,kind", [(64, "equal"), (64, "skewed"), (256, "equal")])
def test_tile_picked_from_the_lengths(K, kind):
    S = 17 * torch.cuda.get_device_properties(0).multi_processor_count
    lengths = np.full(S, 12, np.int64)
    if kind == "skewed":
        lengths[:: S // 8] = 300
    p, logs, args = _inputs(K, 11, lengths, 7)
    ll = api.hmm_forward(*args, api.HMM_BF16_SCALED).cpu().numpy()
    at = list(range(0, S, S // 16))
    ref = ohmm.loglik_batch(p, seqs=at, params=ohmm.params_from_f32_logs(logs))
    assert np.all(np.isfinite(ll)) and np.all(np.abs(ll[at] - ref) <= 1e-3 * np.abs(ref))


def test_rare_symbols_in_a_row():
    # two consecutive symbols of probability ~1e-19 in every state (a floored emission): the
    # exponents, which follow the vector two steps behind, keep it in range
    K, M, T = 128, 4, 40
    p, logs, args = _inputs(K, M, [T] * 20, 3)
    logs["log_B"][:, 3] = -44.0
    args[1] = torch.from_numpy(logs["log_B"]).to(DEV)
    obs = p["obs"].reshape(20, T)
    obs[obs == 3] = 0
    for s in range(20):
        obs[s, s:s + 2] = 3
    p["obs"] = obs.reshape(-1)
    args[3] = torch.from_numpy(p["obs"]).to(DEV)
    ll = api.hmm_forward(*args, api.HMM_BF16_SCALED).cpu().numpy()
    ref = ohmm.loglik_batch(p, params=ohmm.params_from_f32_logs(logs))
    assert np.all(np.abs(ll - ref) <= 1e-3 * np.abs(ref))
