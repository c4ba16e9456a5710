"""Weights of the dense path's one-pass sweep (GPU): the column sums take every
row with the weight of its stored potential, rounded once.

128 groups of columns see one row each (inner products of 30 inside a group and
0 outside, every other row's weight negligible), so log v of a group holds the
rounding of one weight. Against float64 from the stored log u, with what all
groups share (the entries' and log1p's rounding) taken out, two independent
errors are left: the weight's, uniform to half a unit of FP32 (rms 2^-24
sqrt(0.541 / 3) = 2.5e-8 over the fractions of a binade), and the FP32
logarithm's of the column sum (0.7 of a unit at 2^-24: 2.4e-8). Together 3.5e-8;
512 samples settle the rms to 3 %, and the bound is a quarter above: 4.4e-8.
An FP32 exponent and exp2f give 5.1e-8.
"""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _errors(tu, M, sigma, seed):
    N, groups = 1024, 128
    d = groups // 2
    X, Y = np.zeros((N, groups), np.float32), np.zeros((M, groups), np.float32)
    s = np.float32(math.sqrt(30 * 2 * sigma))
    X[np.arange(groups), np.arange(groups)] = s
    Y[np.arange(M), np.arange(M) % groups] = s
    rng = np.random.default_rng(seed)
    n, bias = np.ones(N), np.full(N, -60 * 2 * sigma, np.float32)
    n[:groups] = rng.uniform(1, 8, groups)
    bias[:groups] = rng.uniform(0, 3, groups)
    parts = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (X[:, :d], X[:, d:], Y[:, :d], Y[:, d:])]
    mkt = tu.Market(*parts, n, np.ones(M), sigma, bias_x=torch.from_numpy(bias).cuda(), path="dense")
    try:
        mkt.set_translation(False)
        tu.tu_set_potentials_f64(mkt.handle, np.zeros(N), -40.0 + 0.5 * rng.normal(size=M))
        mkt.sweep(1)
        u, v = mkt.potentials64()
    finally:
        mkt.close()
    w = np.exp(u + bias.astype(np.float64) * (0.5 / sigma))
    own = math.exp(float(s) * float(s) * 0.5 / sigma) - 1.0
    e = v[:groups] + np.arcsinh(0.5 * (w.sum() + own * w[:groups]))
    return e - np.median(e)


def test_weights_are_the_stored_potentials(gpu_lib):
    e = np.concatenate([_errors(gpu_lib, M, sigma, seed) for seed, (M, sigma) in
                        enumerate([(2048, 0.5), (10_240, 0.5), (20_480, 0.5), (2048, 1.0)])])
    assert np.sqrt(np.mean(e * e)) < 4.4e-8
