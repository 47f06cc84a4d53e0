"""Column maxima of B, which scale split-fp16 and exact-slice products: eight
CTAs share a column's rows, 128 at a time, and meet in the first one's shared
memory.  Integer products are exact, so a maximum that misses one CTA's rows
(the scale then overflows fp16 or cuts digits) shows in whole numbers."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# K: one CTA with rows and seven without, two, all eight, a second run of the
# first; N: short of a cluster's 32 columns, several clusters
@pytest.mark.parametrize("K", [8, 128, 136, 1024, 1032])
@pytest.mark.parametrize("N", [4, 36, 516])
@pytest.mark.parametrize("prec", ["fp16x3", "exact"])
def test_column_maxima(libbpx, K, N, prec):
    bpx = libbpx
    code, P = bpx.Code.table1(), bpx.PRECISIONS[prec]
    M = 96
    h = M // code.num_sources
    g = torch.Generator()
    g.manual_seed(K + N)
    A = torch.randint(-4, 5, (M, K), generator=g).float().cuda()
    B = torch.randint(-3, 4, (K, N), generator=g).float()
    # one element of 2^12 a column, its row walking over every CTA's run of rows
    B[(torch.arange(N) * 61) % K, torch.arange(N)] = 4096.0
    B = B.cuda()
    R = (A.double() @ B.double()).float()  # below 2^24: exact
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[1, 3]] = 1
    ws = bpx.Workspace(code, M, N, K, h, P)
    for _ in range(3):
        C, info = bpx.coded_matmul(code, A, B, h, P, mask, ws)
        assert int(info[bpx.INFO_STATUS]) == bpx.OK
        assert torch.equal(C[:M], R)
