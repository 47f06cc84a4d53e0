"""FP32 products against FP64, element by element: on the tensor cores (three
bf16 parts per operand) at tile and K edges, with operands that the parts
cannot hold, and on the CUDA cores at the edges of each tile size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _direct(bpx, A, B):
    """C from the data columns alone (no erasure: every block is a product)."""
    code = bpx.Code.systematic(8, 3, 8)
    (M, K), N = A.shape, B.shape[1]
    h = -(-M // code.num_sources)
    ws = bpx.Workspace(code, M, N, K, h, bpx.FP32)
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    C, info = bpx.coded_matmul(code, A, B, h, bpx.FP32, mask, ws)
    assert int(info[bpx.INFO_STATUS]) == bpx.OK
    return C[:M]


# 128 x 128 and 256 x 256 tiles, ragged rows, columns and K; K just past the
# smallest the form takes, a multiple of 64, one 8-element chunk more
@pytest.mark.parametrize("M,K,N", [(2050, 136, 1540), (1000, 520, 1100), (640, 2056, 516), (4096, 1024, 2048),
                                   (4100, 1032, 2052), (8200, 128, 516)])
@pytest.mark.parametrize("spread", [0.0, 20.0])
def test_tile_edges(libbpx, M, K, N, spread):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K)
    A, B = (torch.randn(s, generator=g, device="cuda") *
            torch.exp(spread * (torch.rand(s, generator=g, device="cuda") - 0.5)) for s in ((M, K), (K, N)))
    C = _direct(libbpx, A, B).double()
    A, B = A.double(), B.double()
    # per element, relative to sum |a||b|: three dropped products (2^-25 each),
    # a 64-wide segment's truncating adds (24, the full-magnitude ones at
    # 2^-23), one rounded add per segment (2^-24)
    gamma = (-(-K // 64) + 2 * 24 + 2) * 2.0 ** -24
    assert ((C - A @ B).abs() <= gamma * (A.abs() @ B.abs())).all()


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.4e38, 1e-40, 2.0 ** -103])
@pytest.mark.parametrize("where", ["A", "B"])
def test_elements_the_parts_cannot_hold(libbpx, value, where):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    A = torch.randn((1000, 520), generator=g, device="cuda")
    B = torch.randn((520, 1100), generator=g, device="cuda")
    A[5, 17], B[17, 3] = 1.0, 0.5
    (A if where == "A" else B)[5 if where == "A" else 17, 17 if where == "A" else 3] = value
    if abs(value) < 1e-30:  # a row / column of such magnitudes: the products stay normal numbers
        if where == "A":
            A[5] *= 2.0 ** -103
            A[5, 17] = value
        else:
            B[:, 3] *= 2.0 ** -103
            B[17, 3] = value
    C = _direct(libbpx, A, B).double()
    R = A.double() @ B.double()
    big = R.abs() > 3.4028234e38  # past FP32's largest
    R = torch.where(big, torch.sign(R) * float("inf"), R)
    assert torch.equal(torch.isnan(C), torch.isnan(R))
    fin = torch.isfinite(R)
    assert torch.equal(C[~fin & ~torch.isnan(R)], R[~fin & ~torch.isnan(R)])
    S = A.double().abs() @ B.double().abs()
    # an FFMA chain of K terms: K roundings of 2^-24, plus the last bit of a subnormal sum
    assert ((C - R).abs()[fin] <= (520 * 2.0 ** -24 * S + 520 * 2.0 ** -149)[fin]).all()


# 32 x 32, 32 x 64, 64 x 64 and 128 x 256 tiles: ragged rows, columns and K
@pytest.mark.parametrize("M,K,N", [(512, 256, 128), (200, 264, 132), (65, 8, 4), (130, 40, 68), (520, 776, 516),
                                   (1000, 1000, 200), (8200, 264, 244), (2050, 72, 2052)])
def test_cuda_core_tile_edges(libbpx, M, K, N):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K)
    A = torch.randn((M, K), generator=g, device="cuda")
    B = torch.randn((K, N), generator=g, device="cuda")
    C = _direct(libbpx, A, B).double()
    A, B = A.double(), B.double()
    # one FMA chain of K terms
    assert ((C - A @ B).abs() <= K * 2.0 ** -24 * (A.abs() @ B.abs())).all()


# the tile that a default call takes (256 x 256 of a CTA pair, 128 x 128,
# 128 x 64) does not change a bit: against the pair tile asked for by name
@pytest.mark.parametrize("M,K,N", [(512, 256, 128), (1000, 1416, 1100), (4096, 4096, 512), (130, 72, 36)])
@pytest.mark.parametrize("prec,pair", [("bf16", 8080), ("bf16x3", 8080), ("fp16x3", 8020)])
def test_default_tile_same_bits(libbpx, M, K, N, prec, pair):
    bpx = libbpx
    code = bpx.Code.systematic(8, 3, 8)
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K)
    A = torch.randn((M, K), generator=g, device="cuda")
    B = torch.randn((K, N), generator=g, device="cuda")
    h = -(-M // code.num_sources)
    ws = bpx.Workspace(code, M, N, K, h, bpx.PRECISIONS[prec])
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[0, 9]] = 1
    C = [bpx.coded_matmul(code, A, B, h, bpx.PRECISIONS[prec], mask, ws, opts=bpx.default_opts(gemm_config=c))[0]
         for c in (0, pair)]
    assert torch.equal(C[0], C[1])


# two pairs a cluster (an even number of 256-wide tiles, the default of larger
# products) against single pairs, rows short of a tile and one wave or several
@pytest.mark.parametrize("M,K,N", [(4000, 200, 4096), (8190, 136, 1536), (2050, 72, 2300)])
@pytest.mark.parametrize("prec,pair", [("bf16", 8080), ("bf16x3", 8080), ("fp16x3", 8020)])
def test_pairs_sharing_rows_same_bits(libbpx, M, K, N, prec, pair):
    test_default_tile_same_bits(libbpx, M, K, N, prec, pair)


@pytest.mark.parametrize("M,K,w", [(2048, 200, 512), (1000, 72, 1000), (4096, 136, 256)])
@pytest.mark.parametrize("prec", ["bf16", "bf16x3"])
def test_two_dimensional_default_same_bits(libbpx, M, K, w, prec):
    bpx = libbpx
    code = bpx.Code.systematic(4, 2, 5)
    g = torch.Generator(device="cuda")
    g.manual_seed(M + K)
    N, h, P = code.k * w, -(-M // code.b), bpx.PRECISIONS[prec]
    A = torch.randn((M, K), generator=g, device="cuda")
    B = torch.randn((K, N), generator=g, device="cuda")
    ws = bpx.Workspace2D(code, M, N, K, h, P)
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[1, 4]] = 1
    C = [bpx.coded_matmul_2d(code, A, B, h, P, mask, ws, opts=bpx.default_opts(gemm_config=c))[0] for c in (0, 8080)]
    assert torch.equal(C[0], C[1])
