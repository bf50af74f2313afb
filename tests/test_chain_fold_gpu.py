"""The FP64 kernel of a CTA per chain, whose sums run in halves for an even number of
beads, against the cluster kernel (whole sums) that the same chains take in a batch of
few: even and odd lengths, thread counts below, at and above the chain's, both noise
keyings, sheared and unsheared chains.

Tolerance: 7 steps of three sums of M terms in FP64, each term rounded twice:
7 * 3 * 2 M * 2^-53 of the largest mode."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


def run(M, C, keying):
    chains = [{"n_beads": M, "dtau": 10.0, "shear_rate_per_s": 5e7 if c % 2 else 0.0} for c in range(C)]
    with sfp.Batch(chains, seed=3, precision=sfp.SFP_FP64) as b:
        b.set_noise(keying)
        b.init_equilibrium()
        b.step(7)
        return b.modes(), b.observe(sfp.SFP_OBS_COM)


@pytest.mark.parametrize("keying", [sfp.SFP_NOISE_BEADS, sfp.SFP_NOISE_MODES], ids=["beads", "modes"])
@pytest.mark.parametrize("M", [4, 6, 20, 64, 100, 101, 128, 300, 514])
def test_halved_sums_match_whole_sums(M, keying):
    R, com = run(M, 20, keying)
    S, scom = run(M, 4, keying)
    tol = 7 * 3 * 2 * M * 2.0 ** -53
    assert np.abs(R[:4] - S).max() < tol * np.abs(S).max()
    assert np.abs(com[:4] - scom).max() < tol * np.abs(scom).max()
