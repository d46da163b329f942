"""The FP32 forward: padded state counts, uneven slots, impossible states and
halves, the shortest sequences, offsets that start inside the observations."""
import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _inputs(K, M, S, lo, hi, seed):
    p = synth.hmm_workload(seed, K, M, S, "uniform", lo, hi)
    logs = synth.hmm_log_inputs_f32(p)
    return p, logs


def _run(logs, p, off=None):
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p["obs"]).to(DEV), torch.from_numpy(p["offsets"]).to(DEV) if off is None else off]
    return api.hmm_forward(*args).cpu().numpy()


def _bound(K, lengths):
    # a step: sums of K terms (an ulp each at worst), exp and log to 2^-21, log B added at magnitude < 16
    return np.asarray(lengths) * ((K + 32) * 2.0 ** -24 + 4 * 2.0 ** -21)


# K on both sides of the padded sizes; more sequences than the 8 slots of every cluster (2500, 1300),
# fewer than one cluster's; one- and two-step sequences
@pytest.mark.parametrize("K,M,S,lo,hi", [(65, 3, 30, 1, 50), (100, 20, 1, 777, 777), (128, 150, 7, 1, 90),
                                         (129, 9, 6, 1, 60), (200, 40, 33, 1, 2), (255, 64, 9, 5, 70),
                                         (256, 120, 9, 1, 40), (96, 7, 2500, 1, 9), (256, 6, 1300, 1, 6)])
def test_matches_the_oracle(K, M, S, lo, hi):
    p, logs = _inputs(K, M, S, lo, hi, K + 3 * S)
    got = _run(logs, p)
    ref = ohmm.loglik_batch(p, params=ohmm.params_from_f32_logs(logs))
    assert np.all(np.abs(got - ref) <= _bound(K, p["lengths"]))
    assert np.array_equal(got, _run(logs, p))


# A warp per sequence: K around the lanes' columns, lengths around the chunks of 32 symbols, warps without
# a sequence
@pytest.mark.parametrize("K", [1, 2, 5, 31, 32, 33, 63, 64])
@pytest.mark.parametrize("M,S,lo,hi", [(3, 70, 1, 70), (130, 9, 28, 36), (7, 1, 97, 97)])
def test_up_to_64_states(K, M, S, lo, hi):
    p, logs = _inputs(K, M, S, lo, hi, K + 3 * S)
    got = _run(logs, p)
    ref = ohmm.loglik_batch(p, params=ohmm.params_from_f32_logs(logs))
    assert np.all(np.abs(got - ref) <= _bound(K, p["lengths"]))


# One half of the states (and so one CTA of a pair) impossible at every step, at every other step, or
# improbable beyond the range of FP32
@pytest.mark.parametrize("K", [40, 80, 256])
@pytest.mark.parametrize("low", [-np.inf, -300.0])
@pytest.mark.parametrize("side", [0, 1])
def test_impossible_and_improbable_halves(K, low, side):
    p, logs = _inputs(K, 6, 20, 1, 60, K)
    half = slice(0, K // 2) if side == 0 else slice(K // 2, K)
    logs["log_B"] = logs["log_B"].copy()
    logs["log_B"][half, ::2] = low
    logs["log_pi"] = logs["log_pi"].copy()
    logs["log_pi"][half] = low
    with np.errstate(divide="ignore"):
        ref = np.array([_log_forward(logs, p["obs"][a:b]) for a, b in zip(p["offsets"], p["offsets"][1:])])
    assert np.all(np.abs(_run(logs, p) - ref) <= _bound(K, p["lengths"]) + p["lengths"] * 300 * 2.0 ** -24)


def _log_forward(logs, obs):
    A = np.exp(logs["log_A"].astype(np.float64))
    lb = logs["log_B"].astype(np.float64)
    la = logs["log_pi"].astype(np.float64) + lb[:, obs[0]]
    for o in obs[1:]:
        m = la.max()
        la = m + np.log(np.exp(la - m) @ A) + lb[:, o]
    return la.max() + np.log(np.exp(la - la.max()).sum())


@pytest.mark.parametrize("K", [70, 256])
def test_offsets_that_start_inside_the_observations(K):
    p, logs = _inputs(K, 12, 20, 3, 80, K)
    off = torch.from_numpy(p["offsets"][5:16].copy()).to(DEV)
    assert np.array_equal(_run(logs, p, off), _run(logs, p)[5:15])


def test_emission_tables_beyond_the_limit_are_refused():
    p, logs = _inputs(256, 130, 9, 1, 40, 1)
    with pytest.raises(api.L.AccelError, match="M\\*K too large"):
        _run(logs, p)
