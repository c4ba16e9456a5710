"""Exponents of wide half-sweeps (GPU): c * phi + g enters the sum with one
rounding, whatever the sizes of c * phi and g.

The market is built so that every exponent is known exactly: c = 75, integer
inner products P up to 13 (exact in BF16 and in the accumulator), and partner
potentials with g = q - 75 P for small q that FP32 holds exactly. c * phi and
g then reach 975 and cancel to q, and a row's sum is sum 2^q. A fused multiply-add
gives q itself; any rounding of g / c or of phi + g / c would show at the size
of the terms (975 * 2^-24 * 0.69 = 4e-5 on the log potential). Tolerance: 2^-22
for ex2.approx, four FP32 roundings for sums and logarithms: 5e-7, with a margin
of four 2e-6.
"""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

C = 75.0


@pytest.mark.parametrize("fp8", [False, "side", "rows"], ids=lambda v: f"fp8={v}")
@pytest.mark.parametrize("N,M,d", [(300, 1000, 24), (1100, 700, 24), (300, 1000, 50), (1100, 700, 50), (2100, 3300, 100)])
def test_exponents_that_cancel(gpu_lib, N, M, d, fp8):
    tu = gpu_lib
    sigma = math.log2(math.e) / (2 * C)
    rng = np.random.default_rng(N + d)
    P = rng.integers(0, 14, M)
    q = -rng.integers(0, 64, M) / 8.0
    P[0], q[0] = 0, 0.0  # the largest g is 0
    F, K, G, L = (np.zeros((r, d), np.float32) for r in (N, N, M, M))
    F[:, 0] = 8.0
    G[:, 0] = P / 8.0  # (e4m3: P / 8 is exact under a power-of-two scale)
    n, m = np.full(N, 2.0), np.ones(M)
    ell = (q - C * P) * math.log(2.0)
    t = [torch.from_numpy(x).cuda() for x in (F, K, G, L)]
    mkt = tu.Market(*(t if fp8 else [x.to(torch.bfloat16) for x in t]), n, m, sigma, path="fused", fp8=fp8)
    try:
        mkt.set_translation(False)
        tu.tu_set_potentials_f64(mkt.handle, np.zeros(N), ell)
        mkt.sweep(1)
        u, _ = mkt.potentials64()
    finally:
        mkt.close()
    s = 0.5 * np.exp2(q).sum()
    want = math.log(math.sqrt(2.0 + s * s) - s)
    np.testing.assert_allclose(u, want, rtol=0, atol=2e-6)
