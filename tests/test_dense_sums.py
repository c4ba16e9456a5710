"""Rounding of the dense path's one-pass sweep (GPU): the sums over a row of
A-hat keep what each addition rounds off, as the row pass does.

A-hat is 1 everywhere (no factors), and the partner weights are 1 for one
column and just under half a unit in the last place for the columns that the
same thread adds after it (columns 640 apart); the rest is negligible. Added
plainly every small term would be lost, 2^-24 of the sum each (15 of 10,240
columns: 8.8e-7 on the log potential; the shortest row here: 4.1e-7).
Compensated, what is left is one rounding of the sum (2^-24), the FP32
logarithm's (2^-24 of 0.69, one unit) and log1p's (2^-24): 1.6e-7, taken as
2.5e-7.
"""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [5120, 10_240, 20_480, 81_920])
def test_terms_below_half_a_unit_add_up(gpu_lib, M):
    tu = gpu_lib
    N, d = 600, 4
    width = min(M, 10_240)
    w = np.full(M, 1e-30)
    w[0] = 1.0
    w[640:width:640] = 0.98 * 2.0**-24
    z = [torch.zeros(r, d, device="cuda") for r in (N, N, M, M)]
    mkt = tu.Market(*z, np.ones(N), np.ones(M), 0.5, path="dense")
    try:
        mkt.set_translation(False)
        tu.tu_set_potentials_f64(mkt.handle, np.zeros(N), 5.0 + np.log(w))
        mkt.sweep(1)
        u, _ = mkt.potentials64()
    finally:
        mkt.close()
    s = 0.5 * math.exp(5.0) * math.fsum(w)
    np.testing.assert_allclose(u, -math.asinh(s), rtol=0, atol=2.5e-7)
