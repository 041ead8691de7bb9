"""Workspaces that hold every strip's tables and no partial sums: the room of
the sums may not turn one pass over the strips into several."""
import pytest

from paper_2504_14497_gb300 import inputs, pcmm
from tests.gpu_common import device, encrypt_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n,l,w,k", [(73, 41, 63, 1, 3), (170, 28, 30, 2, 2), (27, 8, 350, 4, 1), (251, 8, 31, 5, 1)])
@pytest.mark.parametrize("extra", [0, 1, 1 << 16, 1 << 23])
def test_all_strips_in_one_pass(m, n, l, w, k, extra):
    dev = device()
    pr = inputs.pcmm_problem(8100 + m, m, n, l, w)
    A = torch.from_numpy(pr["A"]).to(dev)
    ctB = encrypt_gpu(dev, pr)
    want = pcmm.normalize(pcmm.schoolbook(A, ctB, l, w), m * l)
    per_strip = pcmm.cussen_workspace_bytes_for(m, n, l, w, k, 2) - pcmm.cussen_workspace_bytes_for(m, n, l, w, k, 1)
    plan = pcmm.lib().pcmm_cussen_plan_bytes(m, n, w, k)
    ws = torch.empty(plan + -(-n // k) * per_strip + extra, dtype=torch.uint8, device=dev)
    pcmm.profile_enable(64)
    jac = pcmm.cussen(A, ctB, l, w, k=k, ws=ws)
    gathers = pcmm.profile_read()["gather"][1]
    pcmm.profile_enable(0)
    assert pcmm.workspace_status(ws) == 0
    assert torch.equal(pcmm.normalize(jac, m * l), want)
    assert gathers == 1


@pytest.mark.parametrize("count", [1, 8, 39])
def test_batched_workspace_holds_184_bytes_an_instance(count):
    # Workspaces of sizes that callers keep are still large enough.
    dev = device()
    A = torch.ones((4, 4), dtype=torch.uint8, device=dev)
    ctB = torch.zeros(32 * 4 * 2, dtype=torch.int32, device=dev)
    info = pcmm.Batch([(A, ctB, 2, 1, 1)] * count).info
    assert info.off_segs - info.off_insts <= (184 * count + 255) // 256 * 256
