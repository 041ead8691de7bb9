"""Nonces that lie inside the output of the encryption: both components read
them before they are overwritten."""
import pytest

from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("quad", [0, 2, 3, 4, 6])
@pytest.mark.parametrize("count", [5, 3000, 250000])
def test_nonces_inside_the_output(count, quad):
    # The nonces' two quads are two of the eight that the ciphertexts of the same
    # index are written to.
    dev = device()
    g = torch.Generator(device="cuda")
    g.manual_seed(count)
    r = torch.randint(-(1 << 31), 1 << 31, (8 * count,), dtype=torch.int64, device=dev, generator=g).to(torch.int32)
    msg = torch.randint(0, 256, (count,), dtype=torch.uint8, device=dev, generator=g)
    H = pcmm.public_key(inputs.uniform_scalars(inputs.streams(5)["sk"], (1,))[0], device=dev)
    table = pcmm.keytable(H, device=dev)
    want = pcmm.encrypt_table(table, msg, r)
    out = torch.empty(pcmm.PCMM_AFF_WORDS * count, dtype=torch.int32, device=dev)
    inside = out[4 * quad * count:4 * (quad + 2) * count]
    inside.copy_(r)
    pcmm.encrypt_table(table, msg, inside, out=out)
    assert torch.equal(out, want)
