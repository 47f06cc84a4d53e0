"""The host call in panels of B's columns gives the bits of the device call,
leaves A, B and C on the device as the call in one piece does, and takes column
and cell masks, undecodable masks and page-locked or pageable memory."""
import numpy as np
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# widths: several whole panels, a ragged last one, one panel too narrow to cut
@pytest.mark.parametrize("args,M,K,N", [(("systematic", 8, 3, 8), 2050, 2048, 4096), (("table3",), 1500, 1200, 4100),
                                        (("mojette_a", 8, 6, 200), 1199, 1032, 5000),
                                        (("table1",), 700, 4200, 1000)])
@pytest.mark.parametrize("prec", ["fp32", "bf16", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("pinned", [True, False])
def test_panels_equal_device_call(libbpx, args, M, K, N, prec, pinned):
    bpx = libbpx
    code, P = getattr(bpx.Code, args[0])(*args[1:]), bpx.PRECISIONS[prec]
    h = -(-M // code.num_sources)
    g = torch.Generator()
    g.manual_seed(M)
    hA, hB = torch.randn((M, K), generator=g), torch.randn((K, N), generator=g)
    cells = prec == "bf16x3"
    m = W.erasure_mask(code.n, code.e, 3)
    m = torch.from_numpy(m[code.col_of_cell] if cells else m)
    hC = torch.full((M, N), 7.0)
    if pinned:
        hA, hB, hC, m = (t.pin_memory() for t in (hA, hB, hC, m))
    opts = bpx.default_opts(mask_cells=int(cells), direct_write=int(prec != "fp16x3"))
    dev = [torch.empty(t.shape, dtype=t.dtype, device="cuda") for t in (hA, hB, m)]
    dC = bpx.alloc_C(code, h, N)
    rc, info = bpx.coded_matmul_host(code, hA, hB, h, P, m, hC, dev[0], dev[1], dev[2], dC,
                                     bpx.Workspace(code, M, N, K, h, P), opts=opts)
    assert rc == bpx.OK and info[bpx.INFO_RECOVERED] == code.num_sources
    A, B = hA.cuda(), hB.cuda()
    assert torch.equal(dev[0], A) and torch.equal(dev[1], B) and torch.equal(dev[2].cpu(), m)
    C, dinfo = bpx.coded_matmul(code, A, B, h, P, m.cuda(), bpx.Workspace(code, M, N, K, h, P), opts=opts)
    assert np.array_equal(info, dinfo.cpu().numpy())
    assert torch.equal(dC, C) and torch.equal(hC, C[:M].cpu())


def test_undecodable_and_refused(libbpx):
    bpx = libbpx
    code, M, K, N = bpx.Code.table3(), 900, 2048, 4096
    h = M // code.num_sources
    hA, hB, hC = torch.randn((M, K)), torch.randn((K, N)), torch.zeros((M, N))
    m = torch.tensor([1, 1, 1, 0, 0], dtype=torch.uint8)
    dev = [t.cuda() for t in (hA, hB, m)]
    dC, ws = bpx.alloc_C(code, h, N), bpx.Workspace(code, M, N, K, h, bpx.BF16X3)
    rc, info = bpx.coded_matmul_host(code, hA, hB, h, bpx.BF16X3, m, hC, *dev, dC, ws)
    assert rc == bpx.ERR_UNDECODABLE and info[bpx.INFO_RECOVERED] < code.num_sources
    with pytest.raises(bpx.BpxError) as err:
        bpx.coded_matmul_host(code, hA, hB, h, bpx.BF16X3, m, hC, *dev, dC, ws, opts=bpx.default_opts(gemm_config=8083))
    assert err.value.code == bpx.ERR_INVAL
    small = bpx.Workspace(code, M, N // 2, K, h, bpx.BF16X3)
    with pytest.raises(bpx.BpxError) as err:
        bpx.coded_matmul_host(code, hA, hB, h, bpx.BF16X3, m, hC, *dev, dC, small)
    assert err.value.code == bpx.ERR_NOMEM
