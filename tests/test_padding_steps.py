"""Half-sweeps multiply only the 32-byte steps of a packed row that hold
factors: iterates against the oracle around the steps' edges, and batches whose
members end in different steps."""

import numpy as np
import pytest
import torch

from synth import fp8_quantized, make_market

from _parity import oracle_sweeps

pytestmark = pytest.mark.gpu

# 2d values: exactly whole steps (16 BF16, 32 e4m3 values each), one more and one less, whole rows
SHAPES = [(d, 0.5, False) for d in (1, 8, 9, 24, 25, 33, 40, 41, 63, 65, 72, 73, 96, 97, 127)]
SHAPES += [(d, 0.5, "side") for d in (16, 17, 65, 81, 129, 145)] + [(d, 0.5, "rows") for d in (16, 33, 81, 161)]


@pytest.mark.parametrize("d,sigma,fp8", SHAPES, ids=lambda v: str(v))
def test_iterates_at_step_edges(gpu_lib, d, sigma, fp8):
    mk = make_market(700, 530, d, sigma=sigma, seed=d, bias_x=True, bias_y=True, dtype="fp32" if fp8 else "bf16")
    m = gpu_lib.from_synth(mk, path="fused", fp8=fp8)
    try:
        m.sweep(2)
        u, v = m.potentials64()
    finally:
        m.close()
    if fp8:
        mk, _ = fp8_quantized(mk, "side" if fp8 == "side" else "row")
    ou, ov = oracle_sweeps(mk, 2)
    np.testing.assert_allclose(u, ou, rtol=0, atol=2e-5)
    np.testing.assert_allclose(v, ov, rtol=0, atol=2e-5)


def test_batch_members_of_different_steps(gpu_lib):
    ms = [make_market(n, k, d, sigma=0.5, seed=d, dtype="bf16") for n, k, d in ((300, 900, 3), (500, 200, 32), (70, 600, 17))]
    solo, batched = [], [gpu_lib.from_synth(mk, path="fused") for mk in ms]
    for mk in ms:
        m = gpu_lib.from_synth(mk, path="fused")
        m.sweep(3)
        solo.append(m.potentials64())
        m.close()
    b = gpu_lib.Batch(batched)
    try:
        b.sweep(3)
        torch.cuda.synchronize()
        for m, want in zip(batched, solo):
            for a, w in zip(m.potentials64(), want):
                np.testing.assert_array_equal(a, w)
    finally:
        b.close()
        for m in batched:
            m.close()
