"""The lane step (bonds and modes on the TMEM lanes; BF16 hi/lo transforms at 64,
128, 256 and 512 beads) against the FP64 path of the same library from the same
equilibrium starts and noise keys: chain counts at the edges of its tiles and of
the groups that share a tile's chains, one and several steps per launch, with and
without shear.

Tolerance: 1e-5 of a chain's mode norm, the bound of the fused BF16 step after
1000 steps (a BF16 hi/lo product carries about 17 bits); the centre of mass is
the sum of n noise projections with the same 17 bits, so 2^-16 of its largest
value."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu

DTAU = {64: 10.0, 128: 50.0, 256: 100.0, 512: 100.0}


def run(M, C, n, shear, precision):
    chains = [{"n_beads": M, "dtau": DTAU[M], "job_id": 7 + c,
               "shear_rate_per_s": shear if c % 2 == 0 else 0.0} for c in range(C)]
    with sfp.Batch(chains, seed=5, precision=precision) as b:
        b.init_equilibrium()
        b.step(n)
        return b.modes(), b.observe(sfp.SFP_OBS_COM), b.observe(sfp.SFP_OBS_STEP)


@pytest.mark.parametrize("M", [64, 128, 256])
@pytest.mark.parametrize("C,n,shear", [(1, 1, 0.0), (2, 5, 1e8), (3, 2, 0.0), (4, 3, 0.0), (5, 40, 1e8), (31, 3, 0.0),
                                       (607, 4, 0.0), (609, 4, 1e8), (2500, 3, 0.0), (4865, 2, 1e8)])
def test_lane_step_matches_fp64(M, C, n, shear):
    got, com, steps = run(M, C, n, shear, sfp.SFP_MIXED_BF16)
    ref, rcom, _ = run(M, C, n, shear, sfp.SFP_FP64)
    err = np.linalg.norm((got - ref)[:, :, 1:], axis=(1, 2)) / np.linalg.norm(ref[:, :, 1:], axis=(1, 2))
    assert err.max() < 1e-5, (err.max(), err.argmax())
    assert np.abs(com - rcom).max() < 2.0 ** -16 * np.abs(rcom).max()
    assert (steps == n).all()


@pytest.mark.parametrize("C,n,shear", [(1, 1, 0.0), (2, 3, 1e8), (23, 4, 0.0), (24, 5, 1e8), (25, 40, 1e8), (77, 2, 0.0),
                                       (1824, 3, 0.0), (1825, 2, 1e8)])
def test_lane_step_of_512_beads_on_two_ctas_matches_fp64(C, n, shear):
    """A tile of up to 24 chains on a cluster of two CTAs, one parity of the modes
    each: bonds are sums over both, normals and forces are shared by both."""
    test_lane_step_matches_fp64(512, C, n, shear)


@pytest.mark.parametrize("C", [33, 4865, 6080])
def test_noise_keyings_by_turns(C):
    """Bead-, mode- and bead-keyed steps of one batch: each keying's kernel takes tiles of
    its own size, and the plan comes back to the lane step's."""
    def steps(precision):
        with sfp.Batch([{"n_beads": 64, "dtau": DTAU[64], "job_id": c} for c in range(C)], seed=5, precision=precision) as b:
            b.init_equilibrium()
            for keying in (sfp.SFP_NOISE_BEADS, sfp.SFP_NOISE_MODES, sfp.SFP_NOISE_BEADS):
                b.set_noise(keying)
                b.step(2)
            return b.modes()
    got, ref = steps(sfp.SFP_MIXED_BF16), steps(sfp.SFP_FP64)
    err = np.linalg.norm((got - ref)[:, :, 1:], axis=(1, 2)) / np.linalg.norm(ref[:, :, 1:], axis=(1, 2))
    assert err.max() < 1e-5, (err.max(), err.argmax())
