"""Exact slices with B's digits in pairs (codes of more than 16 sources a
cell) and the narrow exact peel: bit for bit against the oracle, at the
accumulation bound, across segments, ragged sizes and both peel forms, and the
same decode from the separate diagonal planes."""
import numpy as np
import pytest

from oracle import bpx_oracle as o
from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _decode(bpx, code, A, B, h, m, split=False):
    (M, K), N = A.shape, B.shape[1]
    ws = bpx.Workspace(code, M, N, K, h, bpx.EXACT)
    A, B, m = (torch.from_numpy(x).cuda() for x in (A, B, m))
    if split:
        bpx.schedule(code, m, ws)
        C = bpx.peel_decode_exact(code, bpx.exact_products(code, A, B, h, ws), N, h, bpx.alloc_C(code, h, N), ws)
    else:
        C, info = bpx.coded_matmul(code, A, B, h, bpx.EXACT, m, ws)
        assert int(info[bpx.INFO_STATUS]) == bpx.OK
    return C[:M].cpu().numpy()


def _same(C, R, M):
    assert np.array_equal(C.view(np.uint32), R[:M].view(np.uint32))


# sigma 18 and 24 (4-bit digits, S = 6) and 36 (3-bit, S = 8); K below, at and
# past a segment and with a padded tail; N narrow, ragged, and wide enough for
# the peel's other form
@pytest.mark.parametrize("args,e", [((24, 18, 40), 6), ((32, 24, 26), 8), ((44, 36, 37), 8)])
@pytest.mark.parametrize("K,N", [(64, 4), (320, 68), (712, 36), (72, 5000)])
def test_pairs_bit_exact(libbpx, args, e, K, N):
    code, ref = libbpx.Code.mojette_a(*args), o.construction_a(*args)
    h = 1
    M = ref.num_sources - 3
    A, B = W.inputs(M, K, N, "normal", 7)
    m = W.erasure_mask(ref.n, e, 9)
    R, _Q, sch = o.exact_slice_coded_matmul(ref, A, B, h, list(np.nonzero(m)[0]))
    assert sch.ok
    C = _decode(libbpx, code, A, B, h, m)
    _same(C, R, M)
    _same(_decode(libbpx, code, A, B, h, m, split=True), R, M)


# Every entry's digits at their largest, (7, -8, -8, ...) or (3, -4, -4, ...):
# pairs of -136 or -36, and a cell of sigma sources sums to -8 sigma or -4
# sigma a digit
@pytest.mark.parametrize("args,w,S", [((32, 24, 26), 4, 6), ((44, 36, 37), 3, 8)])
def test_pairs_at_the_accumulation_bound(libbpx, args, w, S):
    code, ref = libbpx.Code.mojette_a(*args), o.construction_a(*args)
    p = libbpx.exact_params(code, 1024)
    assert (p["w"], p["S"], p["bits"]) == (w, S, 23)
    half = 2 ** (w - 1)
    xint = (half - 1) * 2 ** (w * (S - 1)) - half * sum(2 ** (w * i) for i in range(S - 1))
    x = np.float32(xint * 2.0 ** -23)
    A = np.full((ref.num_sources, 1024), x, dtype=np.float32)
    B = np.full((1024, 8), x, dtype=np.float32)
    m = W.erasure_mask(ref.n, 4, 3)
    for sign in (False, True):
        if sign:
            A[:, 1::7] = -x
        R, _Q, sch = o.exact_slice_coded_matmul(ref, A, B, 1, list(np.nonzero(m)[0]))
        assert sch.ok
        _same(_decode(libbpx, code, A, B, 1, m), R, len(A))
