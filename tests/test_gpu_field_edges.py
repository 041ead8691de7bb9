"""Carries of the field multiplication and squaring: operands whose words are
0, 1, 2^31, 2^32 - 1 or random in every mix, so that each carry chain of the
product and of the reduction runs both empty and full (exact, against Python
integers)."""
import random

import pytest

from paper_2504_14497_gb300 import pcmm
from tests.gpu_common import P, device, ints_to_planar_fe, planar_fe_to_ints

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


def _operands(seed, count):
    rng = random.Random(seed)
    words = (0, 0, 1, 1 << 31, (1 << 32) - 1, (1 << 32) - 1, None)
    out = []
    for _ in range(count):
        v = 0
        for i in range(8):
            w = rng.choice(words)
            v |= (rng.getrandbits(32) if w is None else w) << (32 * i)
        out.append(v)
    return out


@pytest.mark.parametrize("op", [2, 3])
@pytest.mark.parametrize("seed", [1, 2])
def test_products_of_full_and_empty_words(op, seed):
    dev = device()
    a, b = _operands(seed, 4096), _operands(seed + 100, 4096)
    out = pcmm.test_field(op, pcmm.to_device_words(ints_to_planar_fe(a), dev),
                          pcmm.to_device_words(ints_to_planar_fe(b), dev))
    got = planar_fe_to_ints(pcmm.to_host_words(out), len(a))
    for x, y, g in zip(a, b, got):
        assert g == x * (y if op == 2 else x) % P, (hex(x), hex(y))
