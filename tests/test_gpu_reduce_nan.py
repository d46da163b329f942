"""Minimum and maximum of float data with NaNs: they are left out on every path (one CTA, whole vectors, ragged
ends), wherever they stand, and hide no neighbour."""
import numpy as np
import pytest
import torch

from paper_2211_00621_gb300 import api, synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n", [5, 1000, 65536, 65537, 70_003, 1_000_003, 5_000_001])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("start", [0, 1, 3])
def test_nans_are_left_out(n, dtype, start):
    x = synth.rng(n).uniform(-1.0, 1.0, size=n + start)
    t = torch.from_numpy(x).to(DEV).to(dtype)
    for step in (16, 5, 4, 3, 2):                  # the extremes beside NaNs at every place of a vector
        for k in range(min(step, n)):
            v = t.clone()[start:]
            v[k::step] = float("nan")
            for at, big in ((k + 1, 7.0), (n - 1, 9.0)):
                if at < n and (at - k) % step:
                    v[at] = big
                    v[(at + 1 if (at + 1 - k) % step and at + 1 < n else at)] = big
            want = v[~v.isnan()]
            if want.numel() == 0:
                continue
            assert api.accel_reduce(api.RED_MAX, v).item() == want.max().item(), (step, k)
            assert api.accel_reduce(api.RED_MIN, -v).item() == -want.max().item(), (step, k)


def test_nothing_but_nans_is_the_neutral_element():
    for n in (3, 100_000):
        v = torch.full((n,), float("nan"), device=DEV)
        assert api.accel_reduce(api.RED_MAX, v).item() == -np.inf
        assert api.accel_reduce(api.RED_MIN, v).item() == np.inf
