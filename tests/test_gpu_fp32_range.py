"""FP32 products whose sums leave FP32's range, or come near it: the infinities
and values of one rounded product after the other, and what stays on the
tensor cores."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

M, K, N = 1000, 520, 1100


def _call(bpx, A, B, erased=()):
    code = bpx.Code.systematic(8, 3, 8)
    h = -(-M // code.num_sources)
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[list(erased)] = 1
    C, info = bpx.coded_matmul(code, A, B, h, bpx.FP32, mask, bpx.Workspace(code, M, N, K, h, bpx.FP32))
    assert int(info[bpx.INFO_STATUS]) == bpx.OK
    return C[:M]


def _operands():
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    return torch.randn((M, K), generator=g, device="cuda"), torch.randn((K, N), generator=g, device="cuda"), g


def _chain(A, B):
    """A B as FMA chains over ascending k (the products exact in FP64)."""
    acc = torch.zeros((M, N), device="cuda")
    for k in range(K):
        acc = (acc.double() + A[:, k:k + 1].double() * B[k].double()).float()
    return acc


# one row and one column of magnitudes whose products all have one sign:
# beyond the range, and just inside it in one term and in 40
@pytest.mark.parametrize("a,b", [(1e30, 1e30), (-1e30, 1e30), (1e25, 1e25), (1e38, 1e4), (1e4, -1e38),
                                 (1.998 * 2.0 ** 63, 1.998 * 2.0 ** 63), (2.0 ** 61, 1.9 * 2.0 ** 61), (1e20, 1e17)])
@pytest.mark.parametrize("terms", [1, 40])
def test_large_products(libbpx, a, b, terms):
    A, B, g = _operands()
    A[5], B[:, 3] = 0, 0
    A[5, 100:100 + terms] = a * (0.75 + 0.25 * torch.rand(terms, generator=g, device="cuda"))
    B[100:100 + terms, 3] = b * (0.75 + 0.25 * torch.rand(terms, generator=g, device="cuda"))
    C, R = _call(libbpx, A, B).double(), _chain(A, B).double()
    # (a sum that leaves the range stays infinite, whatever the terms after it)
    assert torch.equal(torch.isinf(C), torch.isinf(R)) and torch.equal(C[torch.isinf(R)], R[torch.isinf(R)])
    S = A.double().abs() @ B.double().abs()
    rest = torch.isfinite(R)
    assert ((C - R).abs()[rest] <= (2 * (K + 1) * 2.0 ** -24 * S + K * 2.0 ** -149)[rest]).all()


# the line itself: K max|A| max|B| below 2^126 runs on the tensor cores, whose
# sums are not those of an FFMA chain; from it on the sums are the chain's own
def test_both_sides_of_the_line(libbpx):
    A, B, _ = _operands()
    A, B = A.clamp(-4, 4), B.clamp(-4, 4)
    A[0, 0] = B[0, 0] = 4.0
    plain = _call(libbpx, A, B, (1, 9))
    scaled = {e: _call(libbpx, A * 2.0 ** e, B * 2.0 ** 50, (1, 9)) * 2.0 ** -50 * 2.0 ** -e for e in (0, 40, 60, 66)}
    R = A.double() @ B.double()
    S = A.double().abs() @ B.double().abs()
    for e, C in scaled.items():
        # max|coded A| lies between 4 and 8 x 4 (eight sources at most): 520 (32) 4 2^(e + 50)
        # is below 2^126 up to e = 59, and 520 (4) 4 2^(e + 50) is not from e = 63 on
        same = torch.equal(C, plain)
        assert same or e > 59
        assert not same or e < 63
        assert ((C.double() - R).abs() <= 64 * (-(-K // 64) + 50) * 2.0 ** -24 * S).all()


# whole operands on both sides of 2^32, from where a warp notes its maximum
@pytest.mark.parametrize("scale", [2.0 ** 17, 2.0 ** 40])
def test_large_operands(libbpx, scale):
    A, B, _ = _operands()
    assert torch.equal(_call(libbpx, A * scale, B, (0, 4)) / scale, _call(libbpx, A, B, (0, 4)))
    assert torch.equal(_call(libbpx, A, B * scale, (0, 4)) / scale, _call(libbpx, A, B, (0, 4)))
