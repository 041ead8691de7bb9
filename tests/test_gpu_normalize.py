"""Output normalisation on both of its paths (blocks whose Z's are all 0 or 1
only copy) at the edges of a block, and products whose sums have zero, one
and two table entries (exact, against the oracle)."""
import random

import numpy as np
import pytest

from oracle import oracle
from paper_2504_14497_gb300 import pcmm
from tests.gpu_common import P, Q, ct_from_aos, device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EDGE_Z = [1, 2, 3, P - 1, P - 2, (P + 1) // 2, 2**255 % P, 2**96, 2**32 - 1, 2**224 - 1]


def _points(count, seed):
    rng = random.Random(seed)
    s = [rng.randrange(1, Q) for _ in range(min(count, 64))]
    pts = oracle.base_mul(np.stack([oracle.int_to_words(v) for v in s]))
    return np.ascontiguousarray(np.resize(pts, (count, 16)))


def _scaled(pt, z):
    """Jacobian words of an affine point with Z = z (z = 0: infinity)."""
    x, y = oracle.point_to_ints(pt)
    z2 = z * z % P
    return np.concatenate([oracle.int_to_words(x * z2 % P if z else 1), oracle.int_to_words(y * z2 * z % P if z else 1),
                           oracle.int_to_words(z)])


@pytest.mark.parametrize("kind", ["plain", "edge", "mixed"])
@pytest.mark.parametrize("count", [1, 5, 127, 128, 129, 700])
def test_normalize(kind, count):
    dev = device()
    rng = random.Random(count)
    aff = _points(2 * count, count).reshape(count, 2, 16)
    jac = np.zeros((count, 2, 24), dtype=np.uint32)
    want = aff.copy()
    for i in range(count):
        for c in range(2):
            z = {"plain": [0, 1, 1], "edge": EDGE_Z, "mixed": [0, 1] + EDGE_Z + [rng.randrange(1, P)]}[kind]
            z = rng.choice(z)
            jac[i, c] = _scaled(aff[i, c], z)
            if z == 0:
                want[i, c] = 0
    got = pcmm.normalize(pcmm.to_device_words(pcmm.ct_to_planar(jac), dev), count)
    assert np.array_equal(pcmm.planar_to_ct(pcmm.to_host_words(got), count), want)


@pytest.mark.parametrize("l", [1, 33])
@pytest.mark.parametrize("n", [1, 2, 3, 40])
def test_sums_of_few_entries(n, l):
    # Row i has i mod 4 non-zero entries (0 .. 3); column 1 of Enc(B) holds infinity.
    dev = device()
    m, w = 9, 4
    A = np.zeros((m, n), dtype=np.uint8)
    for i in range(m):
        for t in range(min(i % 4, n)):
            A[i, (i + t) % n] = 1 + (i + 3 * t) % 15
    ct = _points(2 * n * l, 7 + n).reshape(n, l, 2, 16)
    if n > 1:
        ct[1] = 0
    got = pcmm.normalize(pcmm.cussen(torch.from_numpy(A).to(dev), ct_from_aos(dev, ct), l, w, k=1), m * l)
    got = pcmm.planar_to_ct(pcmm.to_host_words(got), m * l).reshape(m, l, 2, 16)
    for i in range(m):
        for j in (0, l - 1):
            for c in range(2):
                want = np.zeros(16, dtype=np.uint32)
                for k in range(n):
                    if A[i, k]:
                        want = oracle.point_add(want, oracle.scalar_mul(int(A[i, k]), ct[k, j, c]))
                assert np.array_equal(got[i, j, c], want), (i, j, c)
