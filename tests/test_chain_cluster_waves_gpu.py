"""Small FP64 batches whose clusters the GPU can, and can no longer, hold all at once with the
tables in shared memory: one chain more must not make all of them take turns (twice the
time), and gives the same trajectories as the kernel of a CTA per chain (20 chains).

The time of one chain more is bounded by 1.8 times (1.1 to 1.6 measured; 2.0 in turns); the
trajectories by n steps of three sums of M terms in FP64, each term rounded twice."""
import time

import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


def batch(M, C):
    return sfp.Batch([{"n_beads": M, "dtau": 10.0}] * C, seed=3, precision=sfp.SFP_FP64)


def seconds(M, C, n=200):
    with batch(M, C) as b:
        best = 1e9
        for _ in range(6):
            t = time.perf_counter()
            b.step(n)
            b.observe(sfp.SFP_OBS_STEP)
            best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("M,C", [(256, 7), (250, 7), (256, 15), (184, 15)])
def test_one_chain_more_does_not_double_the_time(M, C):
    assert seconds(M, C + 1) < 1.8 * seconds(M, C)


@pytest.mark.parametrize("M,C", [(256, 7), (256, 8), (184, 15), (184, 16), (320, 9), (321, 9), (104, 16), (105, 16), (121, 15), (121, 16)])
def test_each_form_matches_one_cta_per_chain(M, C, n=9):
    def run(C):
        with batch(M, C) as b:
            b.init_equilibrium()
            b.step(n)
            return b.modes()
    S, R = run(C), run(20)
    assert np.abs(R[:C] - S).max() < n * 3 * 2 * M * 2.0 ** -53 * np.abs(R).max()
