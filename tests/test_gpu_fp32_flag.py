"""FP32 operands that the tensor-core parts cannot hold decide about their own
call only: the calls after it, on the same plan or chained, give the bits that
they give alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

M, K, N = 1000, 520, 1100


def _operands():
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    return torch.randn((M, K), generator=g, device="cuda"), torch.randn((K, N), generator=g, device="cuda")


def _bad(X, value):
    X = X.clone()
    X[7, 11] = value
    return X


@pytest.mark.parametrize("value", [float("inf"), 2.0 ** -110])
@pytest.mark.parametrize("where", ["A", "B"])
def test_products_on_one_plan(libbpx, value, where):
    bpx = libbpx
    code = bpx.Code.systematic(8, 3, 8)
    h = -(-M // code.num_sources)
    A, B = _operands()
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[2, 9]] = 1

    def products(calls):
        ws = bpx.Workspace(code, M, N, K, h, bpx.FP32)
        bpx.schedule(code, mask, ws)
        for a, b in calls:
            P = bpx.coded_products(code, a, b, h, bpx.FP32, ws)
        return P

    bad = (_bad(A, value), B) if where == "A" else (A, _bad(B, value))
    assert torch.equal(products([bad, (A, B)]), products([(A, B)]))
    once, twice = products([bad]), products([(A, B), bad, bad])
    assert torch.equal(once.view(torch.int32), twice.view(torch.int32))


@pytest.mark.parametrize("captured", [False, True])
def test_whole_calls_back_to_back(libbpx, captured):
    bpx = libbpx
    code = bpx.Code.systematic(8, 3, 8)
    h = -(-M // code.num_sources)
    A, B = _operands()
    bad = _bad(B, float("inf"))
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[2, 9]] = 1
    ws = bpx.Workspace(code, M, N, K, h, bpx.FP32)
    alone = [bpx.coded_matmul(code, A, b, h, bpx.FP32, mask, bpx.Workspace(code, M, N, K, h, bpx.FP32))[0]
             for b in (B, bad)]
    out = [bpx.alloc_C(code, h, N) for _ in range(4)]
    info = torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda")

    def calls():
        for C, b in zip(out, (B, bad, B, bad)):
            bpx.coded_matmul(code, A, b, h, bpx.FP32, mask, ws, C=C, info=info)

    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            calls()
        graph.replay()
        graph.replay()
    else:
        calls()
    torch.cuda.synchronize()
    for i, C in enumerate(out):
        assert torch.equal(C.view(torch.int32), alone[i % 2].view(torch.int32))
