"""A batch on another stream than its members', used as soon as they are made
(GPU): creation leaves work on the member's stream, which the batch waits for."""

import numpy as np
import pytest
import torch

from synth import make_market

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp8,d", [(False, 32), (False, 64), ("rows", 64)])
def test_batch_follows_creation_on_another_stream(gpu_lib, fp8, d):
    tu = gpu_lib
    mks = [make_market(N, M, d, sigma=0.5, seed=N, bias_x=True, bias_y=True, m_kind="uniform1to3",
                       dtype="fp32" if fp8 else "bf16") for N, M in ((30_000, 20_000), (700, 900), (5000, 1))]
    want = []
    for mk in mks:
        with tu.from_synth(mk, fp8=fp8) as m:
            m.sweep(2)
            want.append(m.potentials64())
    theirs, ours = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    members = [tu.from_synth(mk, fp8=fp8, stream=theirs) for mk in mks]
    batch = tu.Batch(members, stream=ours)
    try:
        batch.sweep(2)
        ours.synchronize()
        for w, m in zip(want, members):
            for a, b in zip(w, m.potentials64()):
                np.testing.assert_array_equal(a, b)
    finally:
        batch.close()
        for m in members:
            m.close()
