"""Equilibrium starts and the FP64 transforms between beads and modes: shortest and
longest chains, odd and even numbers of beads (whole and halved transforms), one chain
and chain counts at the edges of the sampler's blocks, against the oracle.

Tolerance: a conformation is a chain of M rotations and sums in FP64, each with a few
roundings of the positions' scale (the contour length, at most 5 M in scaled units);
the transforms add M terms of that scale: 64 M roundings bound both."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from oracle import oracle as O

pytestmark = pytest.mark.gpu
D_NM = 0.33 * (1.0 - 2.0 * 0.35)


@pytest.mark.parametrize("M,C", [(3, 1), (4, 2), (5, 33), (20, 153), (63, 305), (64, 4900), (101, 3), (512, 16), (1025, 2),
                                 (4096, 1)])
def test_start_matches_the_oracle(M, C):
    m = O.Model(M, dtau=1.0)
    sub = sorted({0, C // 2, C - 1})
    with sfp.Batch([{"n_beads": M, "dtau": 1.0, "job_id": 5 + c} for c in range(C)], seed=4, precision=sfp.SFP_FP64) as b:
        b.init_equilibrium()
        R, pos = b.modes(), b.positions_nm()
        b.set_positions(pos)
        back = b.modes()
    tol = 64 * M * 2.0 ** -53 * 5 * M
    for c in sub:
        ref = m.equilibrium_start(4, 5 + c)
        assert np.abs(R[c] - ref).max() < tol
        assert np.abs(pos[c] / D_NM - m.modes_to_beads(ref)).max() < tol
    assert np.abs(back - R).max() < tol
