"""The FP64 cluster step over many steps in one call, at lengths that leave some CTAs of the
cluster, or some of their warps, without a bond or mode of their own, against the kernel of
a CTA per chain that the same chains take in a batch of 20.

Tolerance: n steps of three sums of M terms in FP64, each term rounded twice: n * 3 * 2 M
* 2^-53 of the largest mode."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


def run(M, C, n):
    chains = [{"n_beads": M, "dtau": 10.0, "shear_rate_per_s": 5e7 if c % 2 else 0.0} for c in range(C)]
    with sfp.Batch(chains, seed=12, precision=sfp.SFP_FP64) as b:
        b.init_equilibrium()
        b.step(n)
        return b.modes(), b.observe(sfp.SFP_OBS_COM), b.observe(sfp.SFP_OBS_STEP)


@pytest.mark.parametrize("C", [1, 9, 19])
@pytest.mark.parametrize("M", [3, 7, 17, 20, 31, 100])
def test_cluster_with_idle_ctas_and_warps(M, C, n=1500):
    S, scom, steps = run(M, C, n)
    R, com, _ = run(M, 20, n)
    tol = n * 3 * 2 * M * 2.0 ** -53
    assert np.abs(R[:C] - S).max() < tol * np.abs(R).max()
    assert np.abs(com[:C] - scom).max() < tol * np.abs(com).max()
    assert (steps == n).all()
