"""Switching to mode-keyed noise within a batch's memory budget: where the tables and buffers
of all lengths together do not fit, the call is refused before anything is allocated and the
batch steps on with bead-keyed noise; where they fit, it switches and stays within."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from paper_1411_3487_gb300 import _lib

pytestmark = pytest.mark.gpu

DTAU = {64: 10.0, 128: 50.0, 256: 100.0}


def batch(lengths, precision, budget=0):
    return sfp.Batch([{"n_beads": M, "dtau": DTAU[M], "job_id": c} for c, M in enumerate(lengths)], seed=9,
                     precision=precision, hbm_budget_bytes=budget)


@pytest.mark.parametrize("precision", [sfp.SFP_MIXED_BF16, sfp.SFP_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("lengths", [[256] * 40, [64, 256, 128, 64, 256] * 9], ids=["one", "mixed"])
def test_mode_noise_is_held_to_the_budget(lengths, precision):
    def run(b, *keyings):
        b.init_equilibrium()
        for k in keyings:
            b.set_noise(k)
            b.step(3)
        return np.concatenate([np.ravel(x) for x in b.modes()])

    with batch(lengths, precision) as b:
        held = b.info()["device_bytes"]
        beads = run(b, sfp.SFP_NOISE_BEADS, sfp.SFP_NOISE_BEADS)
        both = run(b, sfp.SFP_NOISE_MODES, sfp.SFP_NOISE_BEADS)
        full = b.info()["device_bytes"]
    assert full > held
    for budget in (held, full - 1):
        with batch(lengths, precision, budget) as b:
            b.init_equilibrium()
            b.step(3)
            with pytest.raises(sfp.SfpError) as e:
                b.set_noise(sfp.SFP_NOISE_MODES)
            assert e.value.code == _lib.SFP_ENOMEM and b.info()["device_bytes"] == held
            b.step(3)
            assert np.array_equal(np.concatenate([np.ravel(x) for x in b.modes()]), beads)
    with batch(lengths, precision, full) as b:
        assert np.array_equal(run(b, sfp.SFP_NOISE_MODES, sfp.SFP_NOISE_BEADS), both)
        assert b.info()["device_bytes"] == full
