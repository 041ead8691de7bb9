"""Strip tables built by digits, through whole products against the schoolbook
path (exact): every split of a code into digits and halves, ragged last
strips and column blocks, and pairs of points that the affine addition cannot
take (equal and opposite columns, columns at infinity)."""
import numpy as np
import pytest

from oracle import oracle
from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import P, ct_from_aos, device, encrypt_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _device_plain(A, w, dev):
    return pcmm.plaintext16(A, dev) if w > 8 else torch.from_numpy(A).to(dev)


def _same(A, ctB, m, l, w, k):
    want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
    ws = pcmm.workspace(m, A.shape[1], l, w, k, device=A.device)
    got = pcmm.normalize(pcmm.cussen(A, ctB, l, w, k=k, ws=ws), m * l)
    assert pcmm.workspace_status(ws) == 0
    assert torch.equal(got, want)


@pytest.mark.parametrize("w,k,m,n,l", [
    (1, 2, 40, 5, 33), (1, 6, 300, 13, 32), (1, 16, 300, 17, 3), (2, 3, 70, 7, 65), (2, 4, 300, 9, 32),
    (3, 2, 70, 5, 40), (3, 5, 600, 6, 32), (4, 2, 300, 3, 96), (4, 4, 700, 5, 32), (5, 1, 40, 3, 33),
    (5, 3, 700, 4, 32), (6, 2, 400, 3, 32), (7, 1, 140, 3, 64), (8, 1, 16, 3, 1), (8, 1, 300, 2, 130),
    (8, 2, 900, 3, 32), (9, 1, 100, 3, 33), (12, 1, 200, 2, 32), (13, 1, 300, 2, 64), (16, 1, 300, 3, 32),
])
def test_products(w, k, m, n, l):
    dev = device()
    pr = inputs.pcmm_problem(9000 + 100 * w + k, m, n, l, w)
    _same(_device_plain(pr["A"], w, dev), encrypt_gpu(dev, pr), m, l, w, k)


@pytest.mark.parametrize("w,k,m", [(1, 6, 64), (2, 3, 128), (4, 2, 300), (4, 4, 500), (8, 2, 700), (8, 1, 300)])
def test_related_columns(w, k, m):
    # Within every strip: a column, the same column, its negative, infinity.
    dev = device()
    n, l = 2 * k + 1, 34
    pr = inputs.pcmm_problem(9900 + 10 * w + k, m, n, l, w)
    ct = oracle.encrypt(oracle.keygen(pr["sk"]), pr["B"], pr["r"]).copy()     # [n, l, 2, 16]
    for s in range(0, n, k):
        for t in range(1, min(k, n - s)):
            for j in range(l):
                kind = (t + j) % 4
                if kind == 0:
                    ct[s + t, j] = 0
                elif kind < 3:
                    ct[s + t, j] = ct[s, j]
                    for c in range(2):
                        if kind == 2 and ct[s, j, c].any():
                            y = oracle.words_to_int(ct[s, j, c, 8:])
                            ct[s + t, j, c, 8:] = oracle.int_to_words((P - y) % P)
    _same(_device_plain(pr["A"], w, dev), ct_from_aos(dev, ct), m, l, w, k)
    # The same without infinity: no strip leaves the digit build.
    for s in range(0, n, k):
        for t in range(1, min(k, n - s)):
            for j in range(l):
                if (t + j) % 4 == 0:
                    ct[s + t, j] = ct[s, j]
    _same(_device_plain(pr["A"], w, dev), ct_from_aos(dev, ct), m, l, w, k)


@pytest.mark.parametrize("w,k,m,n,l", [
    (6, 1, 40, 3, 33), (6, 1, 300, 2, 1), (6, 2, 900, 3, 40), (7, 1, 20, 2, 32), (7, 2, 400, 3, 33), (8, 1, 17, 3, 33),
    (8, 1, 120, 2, 64), (8, 1, 1500, 2, 32), (8, 2, 600, 5, 20), (10, 1, 300, 2, 33), (11, 1, 300, 3, 32),
    (12, 1, 400, 2, 40), (14, 1, 300, 2, 32), (15, 1, 400, 2, 3), (16, 1, 900, 2, 40),
])
def test_signed_pairs(w, k, m, n, l):
    # Values around the multiples of 16, where an entry is the sum or the
    # difference of a pair, besides random ones.
    dev = device()
    pr = inputs.pcmm_problem(9300 + 100 * w + k, m, n, l, w)
    A = pr["A"].copy()
    near = (np.arange(m * n).reshape(m, n) * 16 + np.resize([0, 1, 7, 8, 9, 15], (m, n))) % (1 << w)
    A[::2] = near[::2]
    _same(_device_plain(A, w, dev), encrypt_gpu(dev, pr), m, l, w, k)


@pytest.mark.parametrize("w,k,m", [(8, 1, 20), (8, 1, 400), (4, 2, 40), (4, 1, 20), (2, 3, 70), (12, 1, 16), (16, 1, 300)])
def test_many_blocks(w, k, m):
    # More than two blocks per SM: the kernels with the smaller register share.
    dev = device()
    n, l = 125 * k, 160
    pr = inputs.pcmm_problem(9500 + 10 * w + k, m, n, l, w)
    _same(_device_plain(pr["A"], w, dev), encrypt_gpu(dev, pr), m, l, w, k)


def _small_order():
    """Points of orders 2, 3 and 4, each on the curve y^2 = x^3 - 3 x + b' of
    its own b', on which the same formulas add."""
    root = lambda a: pow(a, (P + 1) // 4, P)
    square = lambda a: a and pow(a, (P - 1) // 2, P) == 1
    pts = [(5, 0)]
    x = 2
    while True:          # 3 x^4 - 18 x^2 + 12 b x - 9 = 0: order 3
        b = (9 - 3 * x**4 + 18 * x * x) * pow(12 * x, -1, P) % P
        y2 = (x**3 - 3 * x + b) % P
        if square(y2):
            pts.append((x, root(y2)))
            break
        x += 1
    x2 = 2
    while True:          # twice the point is (x2, 0): (x - x2)^2 = 3 x2^2 - 3
        b = (3 * x2 - x2**3) % P
        if square((3 * x2 * x2 - 3) % P):
            x = (x2 + root((3 * x2 * x2 - 3) % P)) % P
            y2 = (x**3 - 3 * x + b) % P
            if square(y2):
                pts.append((x, root(y2)))
                break
        x2 += 1
    return pts


@pytest.mark.parametrize("w", [4, 6, 8, 12, 16])
def test_points_of_small_order_keep_to_their_lane(w):
    # Such a column is no ciphertext; its neighbours in the shared inversion are.
    dev = device()
    m, l = 300, 34
    pr = inputs.pcmm_problem(9700 + w, m, 1, l, w)
    ct = oracle.encrypt(oracle.keygen(pr["sk"]), pr["B"], pr["r"]).copy()
    for i, (x, y) in enumerate(_small_order()):
        for j in (i, 20 + i):
            ct[0, j, j % 2, :8] = oracle.int_to_words(x)
            ct[0, j, j % 2, 8:] = oracle.int_to_words(y)
    _same(_device_plain(pr["A"], w, dev), ct_from_aos(dev, ct), m, l, w, 1)


def _add(p, q):
    if p is None or q is None:
        return p or q
    if p[0] == q[0]:
        if (p[1] + q[1]) % P == 0:
            return None
        s = (3 * p[0] * p[0] - 3) * pow(2 * p[1], -1, P) % P
    else:
        s = (q[1] - p[1]) * pow(q[0] - p[0], -1, P) % P
    x = (s * s - p[0] - q[0]) % P
    return x, (s * (p[0] - x) - p[1]) % P


def _times(k, p):
    if k < 0:
        p, k = (p[0], (P - p[1]) % P), -k
    r = None
    while k:
        if k & 1:
            r = _add(r, p)
        p, k = _add(p, p), k >> 1
    return r


@pytest.mark.parametrize("k,m,n,l", [(2, 300, 5, 33), (2, 20, 2, 70), (3, 600, 4, 34), (3, 900, 5, 20), (4, 700, 9, 33),
                                     (4, 600, 6, 34)])
def test_signed_pairs_of_two_columns(k, m, n, l):
    # Beside random lanes, upper columns that are 0, 8, -8, -4, -2, -1, 1, 2 or 16
    # times the lower one (8 P0 + v P1 doubles or cancels), and lower columns, and
    # both, at infinity.
    dev = device()
    pr = inputs.pcmm_problem(9400 + 10 * k + m, m, n, l, 4)
    ct = oracle.encrypt(oracle.keygen(pr["sk"]), pr["B"], pr["r"]).copy()
    scale = [0, 8, -8, -4, -2, -1, 1, 2, 16]
    for col in range(1, n):
        for j in range(l):
            kind = (3 * col + j) % 15
            for c in range(2):
                if kind < len(scale):
                    base = ct[col - 1, j, c]
                    q = None
                    if base.any():
                        q = _times(scale[kind], (oracle.words_to_int(base[:8]), oracle.words_to_int(base[8:])))
                    ct[col, j, c, :8] = oracle.int_to_words(q[0]) if q else 0
                    ct[col, j, c, 8:] = oracle.int_to_words(q[1]) if q else 0
                if kind in (0, 10):
                    ct[col - 1, j, c] = 0
    _same(_device_plain(pr["A"], 4, dev), ct_from_aos(dev, ct), m, l, 4, k)
    _same(_device_plain(pr["A"], 4, dev), encrypt_gpu(dev, pr), m, l, 4, k)
