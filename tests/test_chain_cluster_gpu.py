"""The FP64 kernels of a cluster of CTAs per chain (16 for up to 9 chains, 8 for up to 19;
tables in shared memory up to 352 and 256 beads, from L2 beyond) against the kernel of a
CTA per chain that the same chains take in a batch of 20: lengths at both edges of each
form and shorter than the cluster, both noise keyings, sheared and unsheared chains, calls
of one and of several steps.

Tolerance: 9 steps of three sums of M terms in FP64, each term rounded twice:
9 * 3 * 2 M * 2^-53 of the largest mode."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


def run(M, C, keying):
    chains = [{"n_beads": M, "dtau": 10.0, "shear_rate_per_s": 5e7 if c % 2 else 0.0} for c in range(C)]
    with sfp.Batch(chains, seed=8, precision=sfp.SFP_FP64) as b:
        b.set_noise(keying)
        b.init_equilibrium()
        for n in (1, 5, 3):
            b.step(n)
        return b.modes(), b.observe(sfp.SFP_OBS_COM), b.observe(sfp.SFP_OBS_STEP)


@pytest.mark.parametrize("keying", [sfp.SFP_NOISE_BEADS, sfp.SFP_NOISE_MODES], ids=["beads", "modes"])
@pytest.mark.parametrize("C", [1, 9, 10, 19])
@pytest.mark.parametrize("M", [3, 7, 17, 64, 129, 256, 257, 352, 353])
def test_cluster_matches_one_cta_per_chain(M, C, keying):
    S, scom, steps = run(M, C, keying)
    R, com, _ = run(M, 20, keying)
    tol = 9 * 3 * 2 * M * 2.0 ** -53
    assert np.abs(R[:C] - S).max() < tol * np.abs(R).max()
    assert np.abs(com[:C] - scom).max() < tol * np.abs(com).max()
    assert (steps == 9).all()
