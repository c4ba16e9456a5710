"""Ranked lists of every length against the longest one.

Lists of up to 14 entries, of 15 to 32 and longer ones are kept in different
places and run on own tiles of different heights; entry i of a row's list does
not depend on the list's length, so a list of k entries is the first k of the
list of 64 bit for bit.
"""

import pytest
import torch

from synth import make_market

pytestmark = pytest.mark.gpu

SHAPES = [
    # N, M, d, fp8: rows around the tiles' edges, ragged partner tiles, one and two k blocks, lists that reach the end
    (1, 64, 8, False),
    (127, 65, 16, False),
    (129, 1333, 32, False),
    (257, 700, 64, False),
    (20001, 300, 16, False),
    (513, 641, 40, "side"),
    (300, 2049, 50, "rows"),
    (1025, 900, 200, "rows"),
]


@pytest.mark.parametrize("N,M,d,fp8", SHAPES, ids=lambda v: str(v))
def test_shorter_list_is_a_prefix(gpu_lib, N, M, d, fp8):
    mk = make_market(N, M, d, sigma=1.0, seed=5 + N, bias_x=True, bias_y=True, dtype="fp32" if fp8 else "bf16")
    if M > 600:  # ties inside a column half and across halves
        mk.G[300:600] = mk.G[:300]
        mk.L[300:600] = mk.L[:300]
    m = gpu_lib.from_synth(mk, path="fused", fp8=fp8)
    try:
        m.sweep(2)
        idx, score = m.topk(0, 64)
        for k in (1, 14, 15, 16, 20, 31, 32, 33):
            i, s = m.topk(0, k)
            assert torch.equal(i, idx[:, :k]), k
            assert torch.equal(s, score[:, :k]), k
    finally:
        m.close()
