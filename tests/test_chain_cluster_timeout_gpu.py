"""A wait of the FP64 cluster step that runs out (SFP_TEST_STALL=1: one CTA of each cluster
waits for something that nobody sends, and the others then wait in vain for its forces): the
call reports SFP_ETIMEDOUT, state, centre of mass and step counter are those before it, and
the context stays usable."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp
from paper_1411_3487_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,C", [(64, 2), (20, 10), (256, 1)])
def test_timeout_leaves_the_chain_as_it_was(monkeypatch, M, C):
    def batch():
        b = sfp.Batch([{"n_beads": M, "dtau": 10.0}] * C, seed=6, precision=sfp.SFP_FP64)
        b.init_equilibrium()
        b.step(3)
        return b

    def read(b, what, out):
        rc = _lib.load().sfp_observe(b._h, what, out.ctypes.data, out.nbytes)
        return rc, out

    with batch() as b:
        ref, com = b.modes(), b.observe(sfp.SFP_OBS_COM)
        monkeypatch.setenv("SFP_TEST_STALL", "1")
        b.step(5)
        monkeypatch.delenv("SFP_TEST_STALL")
        rc, modes = read(b, sfp.SFP_OBS_MODES, np.zeros((C, 3, M)))
        assert rc == _lib.SFP_ETIMEDOUT
        rc, steps = read(b, sfp.SFP_OBS_STEP, np.zeros(C, dtype=np.int64))
        assert rc == _lib.SFP_ETIMEDOUT
        rc, after = read(b, sfp.SFP_OBS_COM, np.zeros_like(com))
        assert rc == _lib.SFP_ETIMEDOUT
        assert (steps == 3).all() and np.array_equal(modes, ref) and np.array_equal(after, com)
    with batch() as b:
        b.step(5)
        assert (b.observe(sfp.SFP_OBS_STEP) == 8).all() and np.isfinite(b.modes()).all()
