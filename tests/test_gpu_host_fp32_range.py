"""The host call in panels with FP32 operands that the tensor-core parts cannot
hold or sum, in any panel: the bits of the device call."""
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

M, K, N = 2050, 2048, 4096  # two panels of 2048 columns


def _host(bpx, code, h, hA, hB, ws):
    m = torch.from_numpy(W.erasure_mask(code.n, code.e, 3)).pin_memory()
    hC = torch.full((M, N), 7.0).pin_memory()
    dev = [torch.empty(t.shape, dtype=t.dtype, device="cuda") for t in (hA, hB, m)]
    rc, info = bpx.coded_matmul_host(code, hA.pin_memory(), hB.pin_memory(), h, bpx.FP32, m, hC, *dev,
                                     bpx.alloc_C(code, h, N), ws)
    assert rc == bpx.OK and info[bpx.INFO_RECOVERED] == code.num_sources
    return hC


def _device(bpx, code, h, hA, hB):
    m = torch.from_numpy(W.erasure_mask(code.n, code.e, 3)).cuda()
    return bpx.coded_matmul(code, hA.cuda(), hB.cuda(), h, bpx.FP32, m,
                            bpx.Workspace(code, M, N, K, h, bpx.FP32))[0][:M].cpu()


@pytest.mark.parametrize("column", [0, 2047, 2048, 4095])
@pytest.mark.parametrize("value", [float("inf"), 2.0 ** -110, 1e30])
def test_one_element(libbpx, column, value):
    bpx = libbpx
    code = bpx.Code.systematic(8, 3, 8)
    h = -(-M // code.num_sources)
    g = torch.Generator()
    g.manual_seed(column)
    hA, hB = torch.randn((M, K), generator=g), torch.randn((K, N), generator=g)
    good = hB.clone()
    hB[7, column] = value
    if value == 1e30:
        hA[3, 7] = 1e20
    ws = bpx.Workspace(code, M, N, K, h, bpx.FP32)
    assert torch.equal(_host(bpx, code, h, hA, hB, ws).view(torch.int32),
                       _device(bpx, code, h, hA, hB).view(torch.int32))
    # and a good call after it
    if value != 1e30:
        assert torch.equal(_host(bpx, code, h, hA, good, ws), _device(bpx, code, h, hA, good))
