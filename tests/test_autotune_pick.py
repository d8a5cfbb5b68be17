"""Which launch options the autotuner picks for given candidate times (no GPU): ties are not left to noise."""
import random

import pytest

from paper_2509_15117_gb300 import binding as Bd

CANDS = [(128, 1, 1), (128, 1, 4), (128, 1, 16), (64, 1, 1), (64, 1, 4), (256, 1, 1), (256, 1, 4), (128, 3, 1), (128, 3, 4)]


def pick(**faster):
    """Times of 280 ms for one register budget and 380 for the other, but for those given as percent faster."""
    ms = [(280.0 if m == 1 else 380.0) * (1.0 - faster.get(f"b{b}_{m}_{r}", 0.0) / 100.0) for b, m, r in CANDS]
    return Bd.ia_test_autotune_pick(ms)


def test_equal_blocks_do_not_fall_to_the_smallest():
    rng = random.Random(1)
    for _ in range(200):
        ms = [(280.0 if m == 1 else 380.0) * (1.0 - rng.uniform(0.0, 0.0099)) for b, m, r in CANDS]
        b, m, r = Bd.ia_test_autotune_pick(ms)
        assert b in (128, 256) and (m, r) == (1, 1)
        assert ms[CANDS.index((b, m, r))] == min(ms[0], ms[5])  # the faster of the two


@pytest.mark.parametrize("faster,want", [
    ({"b64_1_1": 0.9}, (128, 1, 1)), ({"b64_1_1": 2.0}, (64, 1, 1)), ({"b64_1_4": 2.0}, (64, 1, 4)),
    ({"b256_1_1": 0.5}, (256, 1, 1)), ({"b256_1_4": 0.9}, (128, 1, 1)), ({"b256_1_4": 3.0}, (256, 1, 4)),
    ({"b128_3_1": 50.0}, (128, 3, 1)), ({"b64_1_1": 5.0, "b256_1_1": 4.5}, (256, 1, 1))])
def test_rule(faster, want):
    assert pick(**faster) == want


def test_refuses_another_number_of_times():
    with pytest.raises(Bd.IaError):
        Bd.ia_test_autotune_pick([1.0] * 8)
