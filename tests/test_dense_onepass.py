"""GPU parity of the dense path's one-pass sweep against the FP64 oracle.

Shapes at the edges of its layout: units of eight, four, two and one rows of
A-hat, the longest row of a single CTA (10,240 columns), the shortest of a
cluster, clusters of two, four and eight with ragged last slices, and fewer
rows than clusters. Tolerance as for the two-pass dense path (FP32 kernel
entries, compensated FP32 sums): 1e-5 on the log potentials per sweep.
"""

import dataclasses

import numpy as np
import pytest

import oracle
from synth import make_market

from _parity import oracle_sweeps

pytestmark = pytest.mark.gpu

ATOL_LOG = 1e-5

SHAPES = [(1999, 512), (1203, 1281), (517, 2561), (3001, 5119), (769, 10_240), (1031, 10_241), (600, 25_003),
          (513, 41_001)]


def _check(tu, mk, translate=True, omega=1.0, targets=(1, 3)):
    mkt = tu.from_synth(mk, path="dense")
    try:
        mkt.set_translation(translate)
        if omega != 1.0:
            mkt.set_relaxation(omega)
        done = 0
        for target in targets:
            mkt.sweep(target - done)
            done = target
            lu, lv = (t.double().cpu().numpy() for t in mkt.potentials())
            if omega == 1.0:
                ou, ov = oracle_sweeps(mk, target, translate=translate)
            else:
                f = mk.f64()
                Phi = oracle.phi_dense(f["F"], f["K"], f["G"], f["L"], f["bias_x"], f["bias_y"])
                r = oracle.ipfp_batch(Phi, f["n"], f["m"], f["sigma"], max_sweeps=target, tol=0.0, omega=omega,
                                      translate=translate)
                ou, ov = r["log_u"], r["log_v"]
            np.testing.assert_allclose(lu, ou, rtol=0, atol=ATOL_LOG, err_msg=f"log u after {target} sweeps")
            np.testing.assert_allclose(lv, ov, rtol=0, atol=ATOL_LOG, err_msg=f"log v after {target} sweeps")
    finally:
        mkt.close()


@pytest.mark.parametrize("N,M", SHAPES, ids=lambda v: str(v))
def test_sweeps_match_oracle(gpu_lib, N, M):
    mk = make_market(N, M, 8, sigma=0.5, seed=N + 3 * M, bias_y=True, m_kind="uniform1to5", dtype="fp32")
    _check(gpu_lib, mk)


@pytest.mark.parametrize("order", ["rising", "falling"])
def test_weights_beyond_one_scale(gpu_lib, order):
    """Row potentials that span e^{+-60}: the column sums change their scale
    along the rows (rising) or keep the first (falling)."""
    mk = make_market(1500, 700, 8, sigma=0.5, seed=11, bias_x=True, bias_y=True, dtype="fp32")
    b = np.linspace(-60.0, 60.0, mk.N).astype(np.float32)
    mk = dataclasses.replace(mk, bias_x=b if order == "rising" else b[::-1].copy())
    _check(gpu_lib, mk, translate=False, targets=(1, 2))


def test_relaxed_sweeps(gpu_lib):
    mk = make_market(900, 1100, 8, sigma=0.5, seed=12, bias_y=True, dtype="fp32")
    _check(gpu_lib, mk, omega=1.3)
