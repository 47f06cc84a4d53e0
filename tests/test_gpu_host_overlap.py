"""The host call writes C over memory that held B: every element of B is read
before, as when the call ran in one piece."""
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# C starting at B's first column, and at a column of the last of five panels
@pytest.mark.parametrize("shift", [0, 7168])
def test_result_over_b(libbpx, shift):
    bpx = libbpx
    code, M, K, N = bpx.Code.systematic(8, 3, 8), 2050, 2048, 8192
    h = -(-M // code.num_sources)
    g = torch.Generator()
    g.manual_seed(shift)
    hA, B = torch.randn((M, K), generator=g).pin_memory(), torch.randn((K, N), generator=g)
    room = torch.zeros(shift + M * N).pin_memory()
    hB, hC = room[:K * N].view(K, N), room[shift:shift + M * N].view(M, N)
    hB.copy_(B)
    m = torch.from_numpy(W.erasure_mask(code.n, code.e, 3)).pin_memory()
    dev = [torch.empty(t.shape, dtype=t.dtype, device="cuda") for t in (hA, hB, m)]
    ws = bpx.Workspace(code, M, N, K, h, bpx.BF16X3)
    rc, _info = bpx.coded_matmul_host(code, hA, hB, h, bpx.BF16X3, m, hC, *dev, bpx.alloc_C(code, h, N), ws)
    assert rc == bpx.OK
    C, _info = bpx.coded_matmul(code, hA.cuda(), B.cuda(), h, bpx.BF16X3, m.cuda(), ws)
    assert torch.equal(hC, C[:M].cpu())
