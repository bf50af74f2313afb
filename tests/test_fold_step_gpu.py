"""The FP32 fused step at 128 and 256 beads in the halves of the mirror symmetry
against the FP64 path of the same library from the same starts and noise keys: chain
counts at the edges of its tiles and of the noise warps' chunks (eight chains), bead-
and mode-keyed noise, with and without shear.

Tolerance: 1e-5 of a chain's mode norm, the bound of the fused steps elsewhere; the
centre of mass is a sum of noise projections in TF32 hi/lo parts (21 bits and the sum's
rounding), so 2^-18 of its largest value."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu

DTAU = {128: 50.0, 256: 100.0}


def run(M, C, n, shear, noise, precision):
    chains = [{"n_beads": M, "dtau": DTAU[M], "job_id": 3 + c,
               "shear_rate_per_s": shear if c % 2 == 0 else 0.0} for c in range(C)]
    with sfp.Batch(chains, seed=6, precision=precision) as b:
        b.init_equilibrium()
        b.set_noise(noise)
        b.step(n)
        return b.modes(), b.observe(sfp.SFP_OBS_COM), b.observe(sfp.SFP_OBS_STEP)


@pytest.mark.parametrize("noise", [sfp.SFP_NOISE_BEADS, sfp.SFP_NOISE_MODES])
@pytest.mark.parametrize("M", [128, 256])
@pytest.mark.parametrize("C,n,shear", [(1, 1, 0.0), (4, 2, 1e8), (7, 3, 0.0), (8, 40, 1e8), (9, 5, 0.0), (609, 3, 1e8),
                                       (1825, 4, 0.0), (4097, 3, 0.0), (6081, 2, 1e8)])
def test_folded_step_matches_fp64(M, C, n, shear, noise):
    got, com, steps = run(M, C, n, shear, noise, sfp.SFP_FP32)
    ref, rcom, _ = run(M, C, n, shear, noise, sfp.SFP_FP64)
    err = np.linalg.norm((got - ref)[:, :, 1:], axis=(1, 2)) / np.linalg.norm(ref[:, :, 1:], axis=(1, 2))
    assert err.max() < 1e-5, (err.max(), err.argmax())
    assert np.abs(com - rcom).max() < 2.0 ** -18 * np.abs(rcom).max()
    assert (steps == n).all()
