"""A stalled launch of the lane step over several steps (SFP_TEST_STALL=1: its MMA warps wait for
something that never comes): every role gives up without an arrival too many, the call reports
SFP_ETIMEDOUT, state and step counters are those before it, also of the chains whose modes lie
in global memory (256 beads, more than 20 chains a tile), and the next batch runs."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from paper_1411_3487_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C", [(64, 9), (128, 9), (256, 4096), (512, 100)])
def test_stalled_steps_leave_the_chains_as_they_were(monkeypatch, M, C, n=5):
    def read(b, what, out):
        return _lib.load().sfp_observe(b._h, what, out.ctypes.data, out.nbytes), out

    def batch():
        b = sfp.Batch([{"n_beads": M, "dtau": 10.0}] * C, seed=6, precision=sfp.SFP_MIXED_BF16)
        b.init_equilibrium()
        b.step(2)
        return b

    with batch() as b:
        ref = b.observe(sfp.SFP_OBS_MODES_F32)
        monkeypatch.setenv("SFP_TEST_STALL", "1")
        b.step(n)
        monkeypatch.delenv("SFP_TEST_STALL")
        rc, modes = read(b, sfp.SFP_OBS_MODES_F32, np.zeros_like(ref))
        assert rc == _lib.SFP_ETIMEDOUT and np.array_equal(modes, ref)
        rc, steps = read(b, sfp.SFP_OBS_STEP, np.zeros(C, dtype=np.int64))
        assert rc == _lib.SFP_ETIMEDOUT and (steps == 2).all()
    with batch() as b:
        b.step(n)
        assert (b.observe(sfp.SFP_OBS_STEP) == n + 2).all()
