"""Rounding of the closed-form update (GPU): z = log s - 1/2 log n is rounded to
FP32 once, from FP64.

In a market of like users (no biases, unit capacities) log s less the
logarithm of the sum's fraction is the same for all of them, so rounding it
first would shift all log v alike (by 1e-8 at 464 x 1,142, sigma = 1, and their
rms error against float64 to 2.9e-8). Rounded once, what is left are the FP32
logarithms of the sum's fraction and of log1p, each to half a unit of a number in
[0.5, 1): 2 ** -24 / sqrt(12) = 1.72e-8 rms, together 2.43e-8; the bound is 2.5e-8
over three markets (3,400 users: the rms is settled to 1 %).
"""

import numpy as np
import pytest

from synth import make_market

from _parity import oracle_sweeps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["fused", "dense"])
def test_like_users_are_not_shifted(gpu_lib, path):
    err = []
    for seed in (5, 6, 7):
        mk = make_market(464, 1142, 24, sigma=1.0, seed=seed, dtype="bf16" if path == "fused" else "fp32")
        m = gpu_lib.from_synth(mk, path=path)
        try:
            m.sweep(1)
            _, v = m.potentials64()
        finally:
            m.close()
        err.append(v - oracle_sweeps(mk, 1)[1])
    err = np.concatenate(err)
    assert np.sqrt(np.mean(err * err)) < 2.5e-8, (np.sqrt(np.mean(err * err)), err.mean())
