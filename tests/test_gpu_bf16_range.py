"""The BF16 forward on emissions above 1 (densities), steady and sudden, up to e^43: X's target leaves room for them."""
import numpy as np
import pytest
import torch

from oracle import hmm as ohmm
from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# every symbol as large; one that is, in runs; large and small ones in turn; and on both sides of where the
# target begins to fall (2^25 = e^17.3)
@pytest.mark.parametrize("K", [64, 256])
@pytest.mark.parametrize("logs_B", [[17.0] * 4, [17.6] * 4, [30.0] * 4, [43.0] * 4, [0.0, 0.0, 0.0, 30.0],
                                    [40.0, -2.0, 40.0, -30.0], [43.0, 43.0, 0.0, -20.0]])
def test_emissions_above_one(K, logs_B):
    S, T, M = 40, 60, 4
    p = synth.hmm_workload(K, K, M, S, "fixed", T, T)
    logs = synth.hmm_log_inputs_f32(p)
    logs["log_B"] = (logs["log_B"] * 0.1 + np.asarray(logs_B)).astype(np.float32)
    obs = p["obs"].reshape(S, T)
    obs[: S // 2, 10:20] = int(np.argmax(logs_B))           # a run of the largest
    p["obs"] = obs.reshape(-1)
    args = [torch.from_numpy(logs[k]).to(DEV) for k in ("log_A", "log_B", "log_pi")]
    args += [torch.from_numpy(p[k]).to(DEV) for k in ("obs", "offsets")]
    ll = api.hmm_forward(*args, api.HMM_BF16_SCALED).cpu().numpy()
    ref = ohmm.loglik_batch(p, params=ohmm.params_from_f32_logs(logs))
    # the stated 1e-3 of logL, of the sum of its terms' magnitudes where those cancel
    size = np.abs(np.asarray(logs_B))[obs].sum(1) + 10.0
    assert np.all(np.abs(ll - ref) <= 1e-3 * np.maximum(np.abs(ref), size))
