"""The chain kernel's barrier protocol (the model of test_protocol_model.py) with the six ring stages
and one O accumulator of the decode at D = 64: units of 1 to 32 items, also with the producer or
one softmax warpgroup slowed to one step in fifty."""
import random

import pytest

from test_protocol_model import Model

CASES = [(1, 1), (5, 1), (4, 2), (3, 5), (3, 8), (2, 32)]


@pytest.mark.parametrize("slow", [None, "producer", "softmax0", "softmax3"])
@pytest.mark.parametrize("n_units,n_items", CASES)
def test_decode_protocol_six_stages(n_units, n_items, slow):
    for seed in range(8):
        Model(rng=random.Random(seed), slow=slow, units=[4] * n_units, n_items=[n_items] * n_units,
              stages=6, abufs=2, obufs=1).run()
