"""Accuracy of half-sweeps of e4m3 rows of two 128-byte blocks with one scale per
side (GPU), whose g is folded into the MMA as g / c: the rounding of 1 / c does
not show in the potentials.

1 / c is rounded once, so without a correction every g is off by the same
fraction, and by its luck for a sigma the error is larger or smaller than with
g added in FP32 (d = 100, sigma = 0.35: rms of log u 7.9e-8 against 6.7e-8).
Corrected, what is left are the accumulator's and the FP32 logarithms' roundings,
which the sums average: below one unit of FP32 at 1, 2^-24 = 6.0e-8.
"""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _held(a, b):
    """[a | b] as e4m3 with one power-of-two scale, in float64."""
    x = torch.cat([a, b], 1)
    k = math.ceil(math.log2(float(x.abs().max()) / 448))
    return (x.double() / 2.0**k).float().to(torch.float8_e4m3fn).double() * 2.0**k


@pytest.mark.parametrize("sigma", [0.35, 0.5, 0.7, 1.0])
@pytest.mark.parametrize("d", [72, 100, 128])
def test_error_against_float64(gpu_lib, d, sigma):
    tu = gpu_lib
    N, M = 3001, 5003
    g = torch.Generator(device="cuda").manual_seed(d)
    F, K, G, L = (torch.randn(r, d, generator=g, device="cuda") / math.sqrt(d) for r in (N, N, M, M))
    lv = (torch.randn(M, generator=g, device="cuda", dtype=torch.float64) - 0.5 * math.log(N)).cpu().numpy()
    mkt = tu.Market(F, K, G, L, np.full(N, 2.0), np.ones(M), sigma, fp8="side")
    try:
        mkt.set_translation(False)
        tu.tu_set_potentials_f64(mkt.handle, np.zeros(N), lv)
        mkt.sweep(1)
        u, _ = mkt.potentials64()
    finally:
        mkt.close()
    t = _held(F, K) @ _held(G, L).T * (0.5 / sigma) + torch.from_numpy(lv).cuda()
    s = 0.5 * torch.exp(torch.logsumexp(t, 1)).cpu().numpy()
    e = u - (0.5 * math.log(2.0) - np.arcsinh(s / math.sqrt(2.0)))
    assert np.sqrt(np.mean(e * e)) < 2.0**-24
