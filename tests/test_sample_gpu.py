"""One kernel samples every observable of a chain per warp: the accumulated shape, mode
power and window sums against the same sums formed here from the modes of every sample,
for lengths below, at and beyond a warp's lanes, one to eight lags (some beyond the run).

Tolerance: sums of M FP64 products, squared and summed over the samples: 8 M 2^-53 of the
sum of the terms' absolute values, which (sum_p |c_p| |R_p|)^2 bounds per sample and
axis."""
import numpy as np
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lags", [[1], [1, 2, 3, 5], [1, 2, 3, 4, 5, 6, 7, 100]])
@pytest.mark.parametrize("M", [3, 31, 32, 33, 64, 100])
def test_sampled_sums(M, lags):
    C, samples = 5, 7
    with sfp.Batch([{"n_beads": M, "dtau": 5.0, "job_id": c} for c in range(C)], seed=2, precision=sfp.SFP_FP64) as b:
        b.init_equilibrium()
        b.set_msd_lags(lags)
        b.set_sampling(2)
        R, com = [b.modes()], [b.observe(sfp.SFP_OBS_COM)]
        for _ in range(samples - 1):
            b.step(2)
            R.append(b.modes())
            com.append(b.observe(sfp.SFP_OBS_COM))
        acc, power = b.observe(sfp.SFP_OBS_ACCUM), b.observe(sfp.SFP_OBS_MODE_POWER)
        got = [b.observe(w) for w in (sfp.SFP_OBS_COM_MSD, sfp.SFP_OBS_E2E_MSD, sfp.SFP_OBS_BOND_MSD)]
    d = sfp.derive()["d_nm"]
    n, p = np.arange(M)[:, None], np.arange(M)[None]
    phi = np.sqrt(2.0 / M) * np.cos(np.pi * p * (n + 0.5) / M)
    phi[:, 0] = 1.0 / np.sqrt(M)
    R = np.array(R)
    com = np.array(com)
    beads = np.einsum("scap,np->scan", R, phi) * d
    L = beads[..., -1] - beads[..., 0]
    size = ((np.abs(R[..., 1:]).sum(-1) * d) ** 2).max()
    tol = samples * 8 * M * 2.0 ** -53 * max(size, (com ** 2).max())
    assert np.abs(acc[:, 0] - (L ** 2).sum(-1).sum(0)).max() < tol
    assert (acc[:, 3] == samples).all()
    assert np.allclose(power, (R ** 2).sum(0), rtol=samples * 2.0 ** -50, atol=0.0)

    def windows(x):
        out = np.zeros((C, len(lags), 2))
        for i, lag in enumerate(lags):
            edges = x[::lag]
            out[:, i, 0] = ((edges[1:] - edges[:-1]) ** 2).sum(-1).sum(0)
            out[:, i, 1] = len(edges) - 1
        return out

    bonds = [beads[..., m] - beads[..., m - 1] for m in range(1, M)]
    refs = [[windows(com)], [windows(L)], [windows(u) for u in bonds]]
    for g, ref in zip(got, refs):
        assert any((np.abs(g[..., 0] - r[..., 0]) < 4 * tol).all() for r in ref)
        assert (g[..., 1] == ref[0][..., 1]).all()
