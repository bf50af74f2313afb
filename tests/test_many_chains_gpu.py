"""The FP32 CUDA-core step of more chains than one grid dimension of row tiles would take
(65535 tiles of 64 rows, three rows a chain): the last chains against the same chains in a
batch of their own.  Every output is the same sum in the same order, so the bits agree."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [8, 9])
def test_step_of_1_4_million_chains(M, C=64 * 65535 // 3 + 70, last=130):
    def run(ids):
        with sfp.Batch([{"n_beads": M, "dtau": 1.0, "job_id": i} for i in ids], seed=2, precision=sfp.SFP_FP32_SIMT) as b:
            b.step(2)
            return b.observe(sfp.SFP_OBS_MODES_F32)[-last:].copy()
    assert np.array_equal(run(range(C)), run(range(C - last, C)))
