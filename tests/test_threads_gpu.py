"""Batches of different sizes driven by host threads of their own at the same time: a kernel's
attributes belong to the process, so what one call sets must suit every other call.  Starts
(k_equilibrium: from 0.6 to 200 KB of shared memory a block) and FP64 steps of single chains
(k_chain_cluster: 80 to 220 KB), each against the same calls made one after another."""
import threading

import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu

CASES = {"start": (sfp.SFP_FP32, [(256, 3000), (20, 1), (512, 200)], lambda b: b.init_equilibrium()),
         "cluster": (sfp.SFP_FP64, [(256, 1), (150, 1), (200, 1)], lambda b: b.step(2))}


@pytest.mark.parametrize("kind", list(CASES))
def test_threads_do_not_disturb_each_other(kind, rounds=400):
    precision, shapes, call = CASES[kind]
    errors, out = [], {}

    def work(i, M, C, gate=None):
        try:
            with sfp.Batch([{"n_beads": M, "dtau": 10.0}] * C, seed=4, precision=precision) as b:
                if gate:
                    gate.wait(60)
                for _ in range(rounds):
                    call(b)
                out[i] = b.modes()
        except Exception as e:
            errors.append(e)

    for i, s in enumerate(shapes):
        work(i, *s)
    alone, gate = dict(out), threading.Barrier(len(shapes))
    threads = [threading.Thread(target=work, args=(i, *s, gate)) for i, s in enumerate(shapes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    for i in range(len(shapes)):
        assert np.array_equal(out[i], alone[i])
