"""Strips of few distinct codes beside dense ones, in one pass and in passes of
which some are built by chains of prefix sums and some by digits (exact, against
the schoolbook path); tables of few codes cost what they hold."""
import numpy as np
import pytest

from oracle import oracle
from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import ct_from_aos, device, encrypt_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _matrix(m, n, w, seed):
    """Runs of dense, empty, one-valued, two-valued and sparse columns."""
    rng = np.random.default_rng(seed)
    top = (1 << w) - 1
    A = rng.integers(0, top + 1, (m, n))
    for j in range(n):
        kind = (j // 3) % 5
        if kind == 1:
            A[:, j] = 0
        elif kind == 2:
            A[:, j] = top
        elif kind == 3:
            A[:, j] = np.where(rng.random(m) < 0.5, top, 1)
        elif kind == 4:
            A[:, j] *= rng.random(m) < 0.03
    return A.astype(np.uint8 if w <= 8 else np.uint16)


def _device_matrix(A, w, dev):
    return torch.from_numpy(A).to(dev) if w <= 8 else pcmm.plaintext16(A, dev)


@pytest.mark.parametrize("w,k,m", [(8, 1, 300), (12, 1, 300), (16, 1, 400), (5, 1, 40), (4, 2, 90), (5, 2, 200), (2, 3, 70),
                                   (1, 6, 70)])
@pytest.mark.parametrize("l", [5, 40, 97, 130])
def test_few_beside_dense(w, k, m, l):
    dev = device()
    n = 15 * k + 1
    A = _device_matrix(_matrix(m, n, w, 10 * w + k), w, dev)
    pr = inputs.pcmm_problem(8300 + w, m, n, l, 1)
    ct = oracle.encrypt(oracle.keygen(pr["sk"]), pr["B"], pr["r"]).reshape(-1, 2, 16)
    ct[::3, 0] = 0                                   # infinity in every third C1
    ctB = ct_from_aos(dev, ct)
    want = pcmm.normalize((pcmm.schoolbook if w <= 8 else pcmm.schoolbook16)(A, ctB, l, w), m * l)
    for strips in (n, 4):
        ws = torch.empty(pcmm.cussen_workspace_bytes_for(m, n, l, w, k, strips), dtype=torch.uint8, device=dev)
        got = pcmm.normalize(pcmm.cussen(A, ctB, l, w, k=k, ws=ws), m * l)
        assert pcmm.workspace_status(ws) == 0
        assert torch.equal(got, want)


@pytest.mark.parametrize("w,m", [(8, 300), (4, 90), (5, 40), (1, 70)])
def test_few_beside_dense_in_a_batch(w, m):
    # Blocks choose one by one, some of them with strips of both kinds.
    dev = device()
    items, want = [], []
    for l, k in ((5, 1), (40, 2), (97, 1), (130, 1)):
        n = 15 * k + 1
        A = _device_matrix(_matrix(m, n, w, 20 * w + l), w, dev)
        ctB = encrypt_gpu(dev, inputs.pcmm_problem(8350 + l, 1, n, l, 1))
        items.append((A, ctB, l, w, k))
        want.append(pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l))
    for max_strips in (0, 4):
        batch = pcmm.Batch(items, max_strips=max_strips)
        outs = batch.run()
        for out, (A, _, l, _, _), ref in zip(outs, items, want):
            assert torch.equal(pcmm.normalize(out, m * l), ref)
        assert pcmm.workspace_status(batch.ws) == 0


def test_batched_tables_of_few_codes_cost_what_they_hold():
    # Half a percent of the entries not zero against dense (about a tenth; tables that
    # make every digit's multiples take a quarter).
    dev = device()
    m, n, l, w = 128, 256, 256, 8
    ctB = encrypt_gpu(dev, inputs.pcmm_problem(8450, 1, n, l, 1))
    rng = np.random.default_rng(2)
    dense = rng.integers(1, 1 << w, (m, n))
    times = []
    for A in (dense * (rng.random((m, n)) < 0.005), dense):
        batch = pcmm.Batch([(_device_matrix(A.astype(np.uint8), w, dev), ctB, l, w, 1)])
        batch.run()
        pcmm.profile_enable(64)
        batch.run()
        times.append(pcmm.profile_read()["batched"][0])
        pcmm.profile_enable(0)
    assert times[0] < 0.17 * times[1], times


@pytest.mark.parametrize("w", [12, 16])
def test_tables_of_few_codes_cost_what_they_hold(w):
    # 256 columns of one value against dense ones (about an eleventh and a fifteenth).
    dev = device()
    m, n, l = 512, 256, 256
    ctB = encrypt_gpu(dev, inputs.pcmm_problem(8400, 1, n, l, 1))
    ws = pcmm.workspace(m, n, l, w, 1, device=dev)
    times = []
    for A in (np.full((m, n), (1 << w) - 1), np.random.default_rng(1).integers(0, 1 << w, (m, n))):
        A = _device_matrix(A.astype(np.uint16), w, dev)
        pcmm.cussen(A, ctB, l, w, k=1, ws=ws)
        pcmm.profile_enable(64)
        pcmm.cussen(A, ctB, l, w, k=1, ws=ws)
        times.append(pcmm.profile_read()["table"][0])
        pcmm.profile_enable(0)
    assert times[0] < 0.2 * times[1], times
