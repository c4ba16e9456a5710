"""Half-sweeps of which whole waves of own tiles run as they are and the rest is
cut (GPU): the same bits in every launch shape.

Own sides of one wave of tiles (152 SMs: 38,912 rows) and a little more, against
enough partners that the rest is cut; the test computes the market's plan and
asserts both. Rows of one 128-byte block on single CTAs (BF16, e4m3 with one
scale per side and per row), of two and four blocks on pairs, the last of which
has one 256-row tile; narrow and wide.
"""

import numpy as np
import pytest
import torch

from synth import make_market

pytestmark = pytest.mark.gpu

SHAPES = [(39_000, 1700, 24, 0.5, False), (39_000, 1700, 24, 0.5, "side"), (39_000, 1700, 24, 0.5, "rows"),
          (39_000, 1700, 24, 0.01, False), (39_100, 1700, 64, 0.5, False), (39_100, 1700, 64, 0.01, False),
          (39_300, 1600, 100, 0.5, False), (39_100, 1600, 100, 0.01, False), (39_100, 1600, 128, 0.5, "rows"),
          (39_100, 1600, 128, 0.01, "rows"), (39_100, 1600, 128, 0.01, "side"), (39_100, 1600, 200, 0.5, "side")]


def _cut_plan(own, partner, blocks, sms):
    """(t0, span): whole tiles, and partner tiles per span of the rest (0: not cut)."""
    pair = blocks > 1 and sms % 2 == 0 and own > 512
    sms, tile = (sms // 2, 512) if pair else (sms, 256)
    T, P = -(-own // tile), -(-partner // 128)
    w, rest = divmod(T, sms)
    span = max(-(-rest * P // sms), 4)
    if rest == 0 or P <= 4 or w * (P + 4) + span + 8 > 0.92 * (w + 1) * (P + 4):
        return T, 0
    return w * sms, span


@pytest.mark.parametrize("N,M,d,sigma,fp8", SHAPES, ids=lambda v: str(v))
def test_same_bits_with_whole_waves(gpu_lib, N, M, d, sigma, fp8):
    tu = gpu_lib
    row = 2 * d * (1 if fp8 else 2)  # bytes that hold factors
    blocks = 1 if row <= 128 else (2 if row <= 256 else 4)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    t0, span = _cut_plan(N, M, blocks, sms)
    assert t0 > 0 and span > 0
    mk = make_market(N, M, d, sigma=sigma, seed=N + d, bias_x=True, bias_y=True, m_kind="uniform1to3",
                     dtype="fp32" if fp8 else "bf16")
    got = []
    for mode in (0, 1, 2):  # a row's ranges in turn; a CTA (or pair) per span; 128-row tiles
        m = tu.from_synth(mk, path="fused", fp8=fp8)
        try:
            tu.tu_market_set_small_tiles(m.handle, mode)
            m.sweep(2)
            got.append(m.potentials64())
        finally:
            m.close()
    for g in got[1:]:
        for a, b in zip(got[0], g):
            np.testing.assert_array_equal(a, b)
