"""Chained launches: calls back to back on one workspace with new inputs
written right before each, from several threads on their own streams and in a
captured graph, give the bits of calls that run alone."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CASES = [(512, 256, 128, "fp32"), (900, 1000, 1300, "fp32"), (300, 200, 300, "bf16"), (700, 520, 900, "bf16x3"),
         (1000, 1416, 1100, "fp16x3"), (300, 384, 260, "mxfp8"), (640, 256, 640, "exact")]


def _inputs(M, K, N, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn((M, K), generator=g, device="cuda"), torch.randn((K, N), generator=g, device="cuda"))


@pytest.mark.parametrize("M,K,N,prec", CASES)
def test_back_to_back_equals_alone(libbpx, M, K, N, prec):
    bpx = libbpx
    code, P, h = bpx.Code.systematic(8, 3, 8), bpx.PRECISIONS[prec], -(-M // 64)
    masks = torch.zeros((2, code.n), dtype=torch.uint8, device="cuda")
    masks[0, [0, 4]] = 1
    masks[1, [2, 9, 10]] = 1
    inputs = [_inputs(M, K, N, s) for s in range(3)]
    alone = []
    for i in range(6):
        A, B = inputs[i % 3]
        torch.cuda.synchronize()
        C, _info = bpx.coded_matmul(code, A, B, h, P, masks[i % 2], bpx.Workspace(code, M, N, K, h, P))
        torch.cuda.synchronize()
        alone.append(C)
    wrong = []

    def work():
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            ws, C = bpx.Workspace(code, M, N, K, h, P), bpx.alloc_C(code, h, N)
            A, B = torch.empty_like(inputs[0][0]), torch.empty_like(inputs[0][1])
            mask, outs = torch.empty_like(masks[0]), []
            for i in range(24):
                A.copy_(inputs[i % 3][0])
                B.copy_(inputs[i % 3][1])
                mask.copy_(masks[i % 2])
                bpx.coded_matmul(code, A, B, h, P, mask, ws, C=C)
                outs.append(C.clone())
            st.synchronize()
            wrong.extend(i for i, C in enumerate(outs) if not torch.equal(C, alone[i % 6]))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_captured(libbpx):
    bpx = libbpx
    M, K, N, P = 700, 520, 900, bpx.BF16X3
    code, h = bpx.Code.systematic(8, 3, 8), 11
    A, B = _inputs(M, K, N, 0)
    mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
    mask[[0, 4]] = 1
    ws, C = bpx.Workspace(code, M, N, K, h, P), bpx.alloc_C(code, h, N)
    info = torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        bpx.coded_matmul(code, A, B, h, P, mask, ws, C=C, info=info)
        st.synchronize()
        alone = C.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            bpx.coded_matmul(code, A, B, h, P, mask, ws, C=C, info=info)
        C.zero_()
        graph.replay()
        st.synchronize()
    assert torch.equal(C, alone)
