"""The FP32 CUDA-core transforms (k_gemm_f32) through the bond probe and one step of
the plain path, against the oracle: lengths that are and are not multiples of four
(float4 and scalar loads) and of the 16-wide K chunks, and row counts at the edges of
both tile sizes (the larger tiles from 152 blocks on).

Tolerance: a dot product of M terms in FP32 is within M 2^-24 of the sum of its terms'
magnitudes; the bond vectors are sums of M terms below chi R, so M 2^-24 times the
largest row sum of |chi| |R| bounds the error (with the rounding of R and chi to FP32,
M + 2)."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C", [(3, 1), (17, 5), (20, 11), (33, 7), (64, 43), (100, 21), (100, 1621), (101, 1700),
                                 (255, 5), (260, 650)])
def test_fp32_transforms_match_the_oracle(M, C):
    m = O.Model(M, dtau=1.0)
    R0 = np.stack([m.equilibrium_start(3, c % 7) for c in range(C)])
    with sfp.Batch([{"n_beads": M, "dtau": 1.0, "job_id": c} for c in range(C)], seed=3,
                   precision=sfp.SFP_FP32_SIMT) as b:
        b.set_modes(R0)
        b.step(1)
        u, out = b.probe(sfp.SFP_PROBE_BONDS), b.modes()
    chi = np.zeros((M, M))
    t = m.tables()
    phi = t["phi"]
    chi[1:, 1:] = phi[1:, 1:] - phi[:-1, 1:]
    ref = R0 @ chi.T
    bound = (M + 2) * 2.0 ** -24 * (np.abs(R0) @ np.abs(chi).T).max()
    assert np.abs(u - ref).max() < bound
    sub = list(range(min(C, 7))) + [C - 1]
    step = m.run_modes(R0[sub], 3, np.array(sub), 0, 1)
    err = np.linalg.norm((out[sub] - step)[:, :, 1:], axis=(1, 2)) / np.linalg.norm(step[:, :, 1:], axis=(1, 2))
    assert err.max() < 1e-5
