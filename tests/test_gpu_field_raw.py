"""The field operations that only kernels call, on words as they are: the
inversion that a warp shares, the subtraction of a canonical value, the fused
a b - c d with its rare second correction, and the square reduced twice (exact,
against Python integers)."""
import random

import pytest

from paper_2504_14497_gb300 import pcmm
from tests.gpu_common import P, device, ints_to_planar_fe, planar_fe_to_ints

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

R = 1 << 256
ONE = R % P
EDGES = ([0, 1, 2, P - 2, P - 1, P, P + 1, R - 1, R - 2, ONE, P - ONE, P + ONE - 1, (P + 1) // 2, R * R % P]
         + [1 << i for i in range(256)] + [R - (1 << i) for i in range(256)] + [(1 << i) - 1 for i in range(30, 256, 30)])


def _run(op, a, b=None):
    dev = device()
    words = [pcmm.to_device_words(ints_to_planar_fe(v), dev) for v in (a, b) if v is not None]
    return planar_fe_to_ints(pcmm.to_host_words(pcmm.test_field(op, *words)), len(a))


@pytest.mark.parametrize("count", [1, 31, 33, 0])
def test_shared_inversion(count):
    rng = random.Random(count)
    a = [rng.randrange(R) for _ in range(count)] or EDGES + [rng.randrange(R) for _ in range(3000)]
    for x, g in zip(a, _run(6, a)):
        assert g == (R * R * pow(x, -1, P) % P if x % P else 0), hex(x)


def _pairs(seed):
    rng = random.Random(seed)
    a = EDGES + [rng.randrange(R) for _ in range(2000)]
    b = a[::-1]
    b[:len(EDGES)] = rng.sample(EDGES, len(EDGES))
    return a, b


def test_subtraction_of_a_canonical_value():
    a, b = _pairs(1)
    b = [y if y <= P else y % P for y in b]
    for x, y, g in zip(a, b, _run(7, a, b)):
        assert g == (x - y) % P, (hex(x), hex(y))


def test_fused_difference_of_products():
    a, b = _pairs(2)
    small = [0, 1, 2, (1 << 31) + 5, 1 << 200]          # a' b' - a b > p R: corrected twice
    a, b = a + small, b + small[::-1]
    assert sum((R - 1 - x) * (R - 1 - y) - x * y > P * R for x, y in zip(a, b)) >= 5
    ri = pow(R, -1, P)
    for x, y, g in zip(a, b, _run(8, a, b)):
        assert g == (x * y - (R - 1 - x) * (R - 1 - y)) * ri % P, (hex(x), hex(y))


def test_square_reduced_twice():
    a, _ = _pairs(3)
    ri = pow(R * R, -1, P)
    for x, g in zip(a, _run(9, a)):
        assert g == x * x * ri % P, hex(x)


def test_shared_inversion_of_one_is_free():
    # Products of factors that are all 1 (affine points) need no division steps.
    import torch

    dev = device()
    count = 152 * 4 * 128
    times = []
    for v in (ONE, 3 * ONE % P):
        a = pcmm.to_device_words(ints_to_planar_fe([v]), dev).view(2, 1, 4).expand(2, count, 4).reshape(-1).contiguous()
        pcmm.test_field(6, a)
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        pcmm.test_field(6, a)
        end.record()
        end.synchronize()
        times.append(start.elapsed_time(end))
    assert times[0] < 0.5 * times[1], times
