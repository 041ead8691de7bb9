"""Products on the paths for small and narrow shapes, against the schoolbook
path (exact): sums split into parts that a tree of lanes adds (part counts
that are and are not powers of two, on several passes), the copy of a
one-strip product, tables of a single digit, and inputs at infinity on every
table path."""
import pytest

from oracle import oracle
from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import ct_from_aos, device, encrypt_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(pr, m, n, l, w, k, ws=None):
    dev = device()
    A = torch.from_numpy(pr["A"]).to(dev)
    ctB = encrypt_gpu(dev, pr)
    want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
    ws = pcmm.workspace(m, n, l, w, k, device=dev) if ws is None else torch.empty(ws, dtype=torch.uint8, device=dev)
    got = pcmm.normalize(pcmm.cussen(A, ctB, l, w, k=k, ws=ws), m * l)
    assert pcmm.workspace_status(ws) == 0
    assert torch.equal(got, want)


@pytest.mark.parametrize("m,n,l", [(1, 8, 1), (1, 9, 1), (10, 12, 1), (3, 44, 2), (10, 128, 1), (2, 131, 33), (7, 60, 32)])
@pytest.mark.parametrize("w", [1, 4])
def test_parts(m, n, l, w):
    _check(inputs.pcmm_problem(7000 + m + n + l, m, n, l, w), m, n, l, w, 1)


@pytest.mark.parametrize("strips", [1, 5, 37])
def test_parts_over_several_passes(strips):
    m, n, l, w, k = 4, 75, 3, 3, 2
    _check(inputs.pcmm_problem(7100, m, n, l, w), m, n, l, w, k,
           ws=pcmm.cussen_workspace_bytes_for(m, n, l, w, k, strips))


@pytest.mark.parametrize("m,l,w,k,n", [(1, 1, 4, 1, 1), (33, 40, 4, 1, 1), (300, 64, 8, 1, 1), (70, 31, 2, 3, 3),
                                        (5, 129, 1, 1, 1)])
def test_one_strip(m, l, w, k, n):
    pr = inputs.pcmm_problem(7200 + m, m, n, l, w)
    pr["A"][m // 2] = 0          # a row that selects nothing
    _check(pr, m, n, l, w, k)


@pytest.mark.parametrize("w,m", [(2, 2), (3, 4), (4, 8), (4, 9), (4, 100)])
def test_one_digit(w, m):
    _check(inputs.pcmm_problem(7300 + w + m, m, 6, 34, w), m, 6, 34, w, 1)


@pytest.mark.parametrize("w,k,m", [
    (3, 1, 12), (4, 2, 40), (8, 1, 300), (8, 2, 700), (12, 1, 300), (16, 1, 400), (1, 6, 70), (1, 16, 300),   # digits
    (8, 1, 12), (12, 1, 40), (16, 1, 30), (5, 2, 20), (2, 7, 40), (7, 2, 50),                                 # chains
])
@pytest.mark.parametrize("l", [34, 65, 3])
def test_infinity_beside_points(w, k, m, l):
    # Every third ciphertext component is at infinity, the lanes beside it are
    # not: one product and the same product in a batch.
    dev = device()
    n = 2 * k + 1
    pr = inputs.pcmm_problem(7400 + 10 * w + k, m, n, l, w)
    ct = oracle.encrypt(oracle.keygen(pr["sk"]), pr["B"], pr["r"]).copy()
    for i in range(n):
        for j in range(l):
            for c in range(2):
                if (i + j + c) % 3 == 0:
                    ct[i, j, c] = 0
    A = pcmm.plaintext16(pr["A"], dev) if w > 8 else torch.from_numpy(pr["A"]).to(dev)
    ctB = ct_from_aos(dev, ct)
    want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
    assert torch.equal(pcmm.normalize(pcmm.cussen(A, ctB, l, w, k=k), m * l), want)
    if w <= 8:
        for out in pcmm.cussen_batched([(A, ctB, l, w, k)] * 3):
            assert torch.equal(pcmm.normalize(out, m * l), want)


@pytest.mark.parametrize("l", [1, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64, 65, 97])
@pytest.mark.parametrize("m,n,w,k", [(60, 1, 4, 1), (9, 40, 4, 1), (300, 5, 8, 1), (40, 4, 12, 1), (300, 5, 4, 2),
                                     (300, 9, 2, 4)])
def test_columns_that_fill_no_block(m, n, w, k, l):
    # Both components' chains in blocks of 32, packed where that saves one:
    # copies, parts, tables by digits and by chains, several passes, batched.
    pr = inputs.pcmm_problem(7600 + 100 * l + n, m, n, l, w)
    if w > 8:
        dev = device()
        A = pcmm.plaintext16(pr["A"], dev)
        ctB = encrypt_gpu(dev, pr)
        want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
        assert torch.equal(pcmm.normalize(pcmm.cussen(A, ctB, l, w, k=k), m * l), want)
        return
    _check(pr, m, n, l, w, k)
    _check(pr, m, n, l, w, k, ws=pcmm.cussen_workspace_bytes_for(m, n, l, w, k, 2))
    dev = device()
    A = torch.from_numpy(pr["A"]).to(dev)
    ctB = encrypt_gpu(dev, pr)
    want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
    for out in pcmm.cussen_batched([(A, ctB, l, w, k)] * 2):
        assert torch.equal(pcmm.normalize(out, m * l), want)


@pytest.mark.parametrize("m,n,l", [(60, 600, 30), (33, 700, 70), (300, 80, 130), (150, 300, 128)])
def test_lanes_that_add_several_parts(m, n, l):
    # Fewer lanes a point than parts (8, 8, 1 and 1), in one pass and in several.
    pr = inputs.pcmm_problem(7700 + m, m, n, l, 2)
    _check(pr, m, n, l, 2, 1)
    _check(pr, m, n, l, 2, 1, ws=pcmm.cussen_workspace_bytes_for(m, n, l, 2, 1, n // 2 + 1))
