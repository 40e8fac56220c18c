"""The rule that picks how a CTA takes two tiles of a causal run at d_head = 128 (csrc/plans.h), against measured times of both
forms: 32 / 8 heads, between one and two rounds of tiles, behind prefixes from none to eight times the run."""
import pytest

from tests import plans

# new tokens, prefix, us with a long and a short tile in turn, us with two neighbours together
MEASURED = [
    (608, 0, 27.28, 29.48), (608, 152, 33.96, 35.33), (608, 304, 40.27, 39.94), (608, 608, 52.22, 49.79), (608, 1216, 77.25, 69.07),
    (608, 2432, 126.77, 108.72), (608, 4864, 226.99, 187.90),
    (800, 0, 32.09, 36.01), (800, 200, 41.42, 43.85), (800, 400, 49.63, 50.16), (800, 800, 64.85, 62.63), (800, 1600, 98.13, 87.90),
    (800, 3200, 164.02, 140.12), (800, 6400, 296.36, 244.49),
    (1024, 0, 36.13, 43.52), (1024, 256, 46.76, 52.05), (1024, 512, 57.17, 60.25), (1024, 1024, 78.50, 76.97), (1024, 2048, 120.66, 109.91),
    (1024, 4096, 205.37, 176.43), (1024, 8192, 376.32, 310.02),
    # 37 tiles: a round and four CTAs
    (1184, 0, 45.31, 51.46), (1184, 296, 57.60, 61.70), (1184, 592, 68.50, 71.91), (1184, 1184, 92.38, 106.62), (1184, 2368, 141.57, 179.71),
    (1184, 4736, 237.91, 331.86), (1184, 9472, 432.38, 635.86),
]


@pytest.mark.parametrize("T, prefix, turn, together", MEASURED)
def test_the_form_taken_is_the_faster_one(T, prefix, turn, together):
    form = plans.prefill(prefix, T, 32, 8)
    assert (form.tiles_per_cta, form.splits) == (2, 1)
    assert (together if form.pair else turn) <= 1.02 * min(turn, together)


def test_forms_outside_that_range():
    assert plans.prefill(4096, 576, 32, 8).tiles_per_cta == 1          # 144 tiles: a CTA each
    for prefix in (0, 4096):                                            # 304 tiles: together whatever the prefix
        form = plans.prefill(prefix, 1200, 32, 8)
        assert form.tiles_per_cta == 2 and form.pair
    form = plans.prefill(8192, 1024, 32, 8, 64)                         # d_head = 64 has no form for two tiles together
    assert form.tiles_per_cta == 2 and not form.pair
    assert plans.prefill(0, 1200, 32, 8, 64).tiles_per_cta == 1


@pytest.mark.parametrize("T, prefix, Hq, Hkv, splits", [(32, 4000, 60, 15, 8), (32, 4000, 64, 16, 4), (64, 4000, 32, 8, 4), (32, 1200, 128, 32, 4)])
def test_clusters_of_eight_run_at_the_same_time_at_d_head_64(T, prefix, Hq, Hkv, splits):
    """Up to 15 of them: a second round costs more than the split gives."""
    assert plans.prefill(prefix, T, Hq, Hkv, 64).splits == splits
