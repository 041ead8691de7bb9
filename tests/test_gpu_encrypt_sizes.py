"""Encryption at the counts where the split of a ciphertext's additions over
threads changes, and nonces with empty windows."""
import numpy as np
import pytest

from oracle import oracle
from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _encrypt(dev, H, msg, r):
    return pcmm.encrypt(H, torch.from_numpy(msg).to(dev), pcmm.to_device_words(pcmm.scalars_to_planar(r), dev))


def _rows(ct, count):
    return pcmm.planar_to_ct(pcmm.to_host_words(ct), count)


def test_counts_agree():
    dev = device()
    rng = np.random.default_rng(77)
    n = 9731
    r = rng.integers(0, 2**32, size=(n, 8), dtype=np.uint64).astype(np.uint32)
    r[:, 7] >>= 1
    msg = rng.integers(0, 256, size=n, dtype=np.uint8)
    _, H = _key()
    want = _rows(_encrypt(dev, H, msg, r), n)
    for count in (1, 2, 127, 129, 1216, 1217, 9728, 9729):
        got = _rows(_encrypt(dev, H, msg[:count], r[:count]), count)
        assert (got == want[:count]).all()


def _key():
    sk = inputs.uniform_scalars(inputs.streams(5)["sk"], (1,))[0]
    return sk, pcmm.public_key(sk)


@pytest.mark.parametrize("pad", [0, 1300, 9800])
def test_empty_windows(pad):
    dev = device()
    sk, H = _key()
    special = [0, 1, 255, 256, 1 << 248, (1 << 248) + 1, 0xFF << 120, (1 << 64) - 1, 0x01010101 << 32, 7 << 200]
    r = np.zeros((len(special) + pad, 8), dtype=np.uint32)
    for i, x in enumerate(special):
        r[i] = oracle.int_to_words(x)
    r[len(special):, 2] = 9
    msg = np.resize(np.array([0, 255, 1], dtype=np.uint8), len(r))
    got = _rows(_encrypt(dev, H, msg, r), len(r))
    k = len(special)
    assert not got[0].any()          # nonce 0, message 0 (the oracle refuses this nonce): infinity twice
    want = oracle.encrypt(oracle.keygen(sk), msg[1:k].reshape(1, k - 1), r[1:k].reshape(1, k - 1, 8))
    assert (got[1:k] == want.reshape(k - 1, 2, 16)).all()


@pytest.mark.parametrize("count", [58368, 58369])
def test_decryption_where_its_kernel_changes(count):
    dev = device()
    rng = np.random.default_rng(count)
    r = rng.integers(0, 2**32, size=(count, 8), dtype=np.uint64).astype(np.uint32)
    r[:, 7] >>= 1
    msg = rng.integers(0, 256, size=count, dtype=np.uint8)
    sk, H = _key()
    steps = pcmm.BabySteps.for_range(255, device=dev)
    out = pcmm.decrypt(sk, _encrypt(dev, H, msg, r), count, 255, steps)
    assert (out.cpu().numpy() == msg.astype(np.int64)).all()
