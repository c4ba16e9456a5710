"""Batches of thousands of small markets (GPU): the kernels over a market's
users have as many blocks per market as the batch's size leaves, so a large
member among thousands shares few, and one block per market goes without the
count of finished blocks.

Every member's sweeps have the bits of its own; match counts differ only by the
order of an FP64 sum (relative 1e-12: fewer than 1e4 terms of like size at 1e-16).
"""

import numpy as np
import pytest
import torch

from synth import make_market

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("copies,large", [(330, (9000, 4100)), (1100, (5000, 300)), (1100, None)])
def test_members_as_alone(gpu_lib, copies, large):
    tu = gpu_lib
    shapes = [(100, 90), (1, 300), (257, 33), (513, 128), (80, 81), (130, 700), (300, 1), (256, 256), (90, 100)]
    mks = [make_market(N, M, 16, sigma=0.5, seed=50 + i, bias_x=True, bias_y=True, n_kind="uniform_real",
                       m_kind="uniform_real", dtype="bf16") for i, (N, M) in enumerate(shapes)]
    kinds = list(range(len(mks))) * (copies * 9 // len(shapes))
    if large is not None:
        mks.append(make_market(*large, 16, sigma=0.5, seed=77, bias_x=True, bias_y=True, dtype="bf16"))
        kinds.insert(len(kinds) // 2, len(mks) - 1)
    alone = [tu.from_synth(mk) for mk in mks]
    members = [tu.from_synth(mks[i]) for i in kinds]
    batch = tu.Batch(members)
    try:
        batch.sweep(2)
        torch.cuda.synchronize()
        for m in alone:
            m.sweep(2)
        for at in list(range(9)) + [len(kinds) // 2, len(kinds) - 1]:
            for a, b in zip(alone[kinds[at]].potentials64(), members[at].potentials64()):
                np.testing.assert_array_equal(a, b)
        _, infos = batch.solve(1e-6, 500)
        for at in list(range(9)) + [len(kinds) // 2, len(kinds) - 1]:
            want = alone[kinds[at]].solve(1e-6, 500)
            assert infos[at]["status"] == want["status"] and infos[at]["residual_inf"] <= 1e-6
            if infos[at]["sweeps"] == want["sweeps"]:
                assert infos[at]["match_count"] == pytest.approx(want["match_count"], rel=1e-12)
    finally:
        batch.close()
        for m in alone + members:
            m.close()
