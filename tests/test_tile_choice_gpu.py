"""Chains per tile of batches of mixed lengths, and the autotuner's candidates: neither counts
on tiles larger than a group's step takes (40 chains; three-pass BF16 32, 24 at 512 beads)."""
import pytest

import paper_1411_3487_gb300 as sfp

pytestmark = pytest.mark.gpu

LENGTHS = (64, 128, 256, 512)


def tiles(b):
    """The tiles in use (the autotuner of a staged batch reports them and tries none)."""
    b.set_path(sfp.SFP_PATH_STAGED)
    out = b.autotune(1)
    b.set_path(sfp.SFP_PATH_FUSED)
    return out


@pytest.mark.parametrize("precision", [sfp.SFP_MIXED_BF16, sfp.SFP_FP32], ids=["bf16", "fp32"])
@pytest.mark.parametrize("C", [12, 200, 600, 790, 830, 850, 900])
def test_mixed_lengths_take_one_wave_where_one_is_enough(C, precision):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def ctas(t):
        return sum((C + c - 1) // c * (2 if M == 512 else 1) for M, c in zip(LENGTHS, t))

    most = [32, 32, 32, 24] if precision == sfp.SFP_MIXED_BF16 else [40] * 4
    with sfp.Batch([{"n_beads": M, "dtau": 10.0} for M in LENGTHS] * C, seed=1, precision=precision) as b:
        got = tiles(b)
    if ctas(most) > sms:
        assert got == most
    else:
        assert ctas(got) <= sms
        smaller = [min(c, max(got) - 4) for c in most]
        assert max(got) == 4 or ctas(smaller) > sms


def test_the_autotuner_times_a_tile_once(steps=2):
    """5472 chains of 64 beads: every candidate is above the largest tile, so there is one
    (two launches), then the choice is run as a whole (two more)."""
    with sfp.Batch([{"n_beads": 64, "dtau": 10.0}] * 5472, seed=1, precision=sfp.SFP_MIXED_BF16) as b:
        before = b.info()["launches"]
        assert b.autotune(steps) == [32]
        assert b.info()["launches"] - before == 4
