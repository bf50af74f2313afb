"""FP32 normals (polynomial Box-Muller) against the oracle's FP64 ones for the same
Philox words, through the noise probe of the plain path: lengths whose last Philox
call is full and partly used, and enough draws to reach both tails.

Tolerance: a normal is r cos(theta) with r = sqrt(-2 ln u) below 5.8.  The radius is
one approximate square root (2^-22 relative by its specification) of a logarithm with
polynomial and rounding errors below 2^-22, the sine or cosine is within 2^-23
absolute, so |error| < r (2^-22 / 2 + 2^-22 + 2^-23) < r 2^-21."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C,step", [(3, 5, 0), (64, 300, 2 ** 33 + 5), (101, 50, 1), (256, 400, 12345), (511, 40, 7)])
def test_fp32_normals_match_the_oracle(M, C, step):
    with sfp.Batch([{"n_beads": M, "dtau": 1.0}] * C, seed=9, precision=sfp.SFP_FP32_SIMT) as b:
        b.set_path(sfp.SFP_PATH_STAGED)
        b.set_step(step)
        b.step(1)
        z = b.probe(sfp.SFP_PROBE_NOISE)
    ref = np.stack([O.bead_normals(9, c, step, 0, M) for c in range(C)])
    assert z.shape == ref.shape
    assert np.abs(z - ref).max() < 5.8 * 2.0 ** -21
    assert abs(z.mean()) < 6 / np.sqrt(z.size)
