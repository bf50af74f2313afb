"""Modes of a batch of several lengths are packed on the device: equal, value for
value, to what the batches of each length alone hand back, FP64 and FP32, after
set_modes of arbitrary values (no arithmetic lies between but the centre of mass'
sqrt(M) and 1 / sqrt(M)) and after steps."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[3, 4], [64, 7, 64, 512, 3, 7], [100, 64, 333, 64, 128, 3, 257] * 9])
@pytest.mark.parametrize("precision", [sfp.SFP_FP64, sfp.SFP_FP32])
def test_packed_modes_equal_those_of_single_length_batches(lengths, precision):
    chains = [{"n_beads": m, "dtau": 5.0, "job_id": i} for i, m in enumerate(lengths)]
    rng = np.random.default_rng(4)
    start = [rng.standard_normal((3, m)).astype(np.float32).astype(np.float64) + 5.0 for m in lengths]
    with sfp.Batch(chains, seed=9, precision=precision) as b:
        b.set_modes(start)
        steps = [0, 3]
        got = []
        for n in steps:
            b.step(n) if n else None
            got.append((b.observe(sfp.SFP_OBS_MODES), b.observe(sfp.SFP_OBS_MODES_F32)))
        pos = b.positions_nm()
    for m in set(lengths):
        idx = [i for i, x in enumerate(lengths) if x == m]
        with sfp.Batch([chains[i] for i in idx], seed=9, precision=precision) as s:
            s.set_modes(np.stack([start[i] for i in idx]))
            for n, (f64, f32) in zip(steps, got):
                s.step(n) if n else None
                a, c = s.observe(sfp.SFP_OBS_MODES), s.observe(sfp.SFP_OBS_MODES_F32)
                for k, i in enumerate(idx):
                    assert np.array_equal(f64[i], a[k]) and f64[i].shape == (3, m)
                    assert np.array_equal(f32[i], c[k]) and f32[i].dtype == np.float32
            p = s.positions_nm()
            for k, i in enumerate(idx):
                assert np.array_equal(pos[i], p[k])
