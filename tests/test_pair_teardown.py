"""Pairs of CTAs launched back to back (GPU): the second CTA of a pair stays
until the last arrivals on its own barriers have landed, so none reaches the
shared memory of the kernel that takes the SM over.

Many launches of a few microseconds each, with list kernels (single CTAs, other
barriers at the same shared addresses) between them; the potentials have the
bits of the same sweeps on single CTAs. Sizes: one pair with a single 256-row
tile in its second CTA's place or beyond the end, several pairs, rows of two and
of four 128-byte blocks, folded and unfolded g.
"""

import numpy as np
import pytest

from synth import make_market

pytestmark = pytest.mark.gpu

SHAPES = [(513, 300, 64, 0.5, False), (700, 530, 50, 0.01, False), (1300, 1025, 100, 0.5, False),
          (1300, 1025, 128, 0.5, "rows"), (1300, 1025, 128, 0.5, "side")]


@pytest.mark.parametrize("N,M,d,sigma,fp8", SHAPES, ids=lambda v: str(v))
def test_short_pair_launches_back_to_back(gpu_lib, N, M, d, sigma, fp8):
    tu = gpu_lib
    mk = make_market(N, M, d, sigma=sigma, seed=N, bias_x=True, bias_y=True, m_kind="uniform1to3",
                     dtype="fp32" if fp8 else "bf16")
    got = []
    for mode in (1, 0):  # pairs; a CTA per tile
        m = tu.from_synth(mk, path="fused", fp8=fp8)
        try:
            tu.tu_market_set_small_tiles(m.handle, mode)
            lists = []
            for _ in range(20):
                m.sweep(10)
                lists.append(m.topk(1, 5))
            got.append((*m.potentials64(), *[t.cpu().numpy() for pair in lists for t in pair]))
        finally:
            m.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
