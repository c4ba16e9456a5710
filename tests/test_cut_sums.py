"""Cut half-sweeps and pairs of CTAs (GPU): a market's row sums are formed in
ranges that belong to its shape, so every launch shape gives the same bits.

Sizes: fewer own tiles than SMs with spans that end inside and at the end of a
tile, one tile more than a wave (38,912 rows on 152 SMs), and both sides cut;
packed rows of one (d = 24), two and four 128-byte blocks, the latter on pairs
of CTAs (512-row tiles, an odd number of 256-row halves among them).
Against the oracle the fused path's 2e-5 per sweep holds (test_parity_fused.py
derives it).
"""

import numpy as np
import pytest

from synth import make_market

from _parity import oracle_sweeps

pytestmark = pytest.mark.gpu

SHAPES = [(1500, 3000, 24, 0.5, False), (4097, 2049, 24, 0.5, False), (39_000, 1100, 24, 0.5, False),
          (39_000, 1100, 24, 0.5, "rows"), (2100, 3300, 24, 0.5, "side"), (3000, 4100, 24, 0.01, False),
          (39_100, 1300, 24, 0.01, "rows"),
          (513, 700, 64, 0.5, False), (4097, 2049, 50, 0.5, False), (39_000, 1100, 64, 0.5, False),
          (3000, 4100, 64, 0.01, False), (2300, 3333, 100, 0.5, False), (39_000, 1100, 128, 0.01, False),
          (2300, 3333, 100, 0.5, "rows"), (2300, 3333, 200, 0.5, "side")]


def _run(tu, mk, fp8, mode):
    m = tu.from_synth(mk, path="fused", fp8=fp8)
    try:
        if mode is not None:
            tu.tu_market_set_small_tiles(m.handle, mode)
        m.sweep(3)
        return m.potentials64()
    finally:
        m.close()


@pytest.mark.parametrize("N,M,d,sigma,fp8", SHAPES, ids=lambda v: str(v))
def test_same_bits_in_every_launch_shape(gpu_lib, N, M, d, sigma, fp8):
    mk = make_market(N, M, d, sigma=sigma, seed=N + M, bias_x=True, bias_y=True, m_kind="uniform1to3",
                     dtype="fp32" if fp8 else "bf16")
    want = _run(gpu_lib, mk, fp8, 0)  # a row's ranges in turn
    for mode in (None, 2):            # a CTA per span; 128-row tiles
        for a, b in zip(want, _run(gpu_lib, mk, fp8, mode)):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("N,M,d", [(1500, 3000, 24), (4097, 2049, 24), (1500, 3000, 64), (2300, 1777, 100)])
def test_cut_sweeps_match_oracle(gpu_lib, N, M, d):
    mk = make_market(N, M, d, sigma=0.5, seed=N, bias_x=True, bias_y=True, dtype="bf16")
    u, v = _run(gpu_lib, mk, False, None)
    ou, ov = oracle_sweeps(mk, 3)
    np.testing.assert_allclose(u, ou, rtol=0, atol=2e-5)
    np.testing.assert_allclose(v, ov, rtol=0, atol=2e-5)
