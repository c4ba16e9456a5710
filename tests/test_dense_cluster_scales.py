"""The column sums' scale in clusters (GPU): row potentials that span e^{+-60}
make the sums change their scale along a cluster's rows (rising) or keep the
first (falling). The factor travels to every CTA of the cluster with the row's
weight.

Clusters of two (five slots in the ring: one row at a time), of two and of four
with narrow slices (seven slots and more: two rows at a time, an odd number of
rows among them) and of eight; a few more than twenty rows for each cluster.
Tolerance as for the dense path: 1e-5 on the log potentials per sweep.
"""

import dataclasses

import numpy as np
import pytest

from synth import make_market

from _parity import oracle_sweeps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["rising", "falling"])
@pytest.mark.parametrize("N,M", [(1601, 20_003), (1599, 10_241), (801, 30_001), (451, 41_001)])
def test_cluster_scales(gpu_lib, N, M, order):
    mk = make_market(N, M, 8, sigma=0.5, seed=N, bias_x=True, bias_y=True, dtype="fp32")
    b = np.linspace(-60.0, 60.0, N).astype(np.float32)
    mk = dataclasses.replace(mk, bias_x=b if order == "rising" else b[::-1].copy())
    mkt = gpu_lib.from_synth(mk, path="dense")
    try:
        mkt.set_translation(False)
        mkt.sweep(1)
        lu, lv = mkt.potentials64()
    finally:
        mkt.close()
    ou, ov = oracle_sweeps(mk, 1, translate=False)
    np.testing.assert_allclose(lu, ou, rtol=0, atol=1e-5)
    np.testing.assert_allclose(lv, ov, rtol=0, atol=1e-5)
