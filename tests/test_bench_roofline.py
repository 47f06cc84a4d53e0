"""bench.py's account of what a coded GEMM runs on, and of the kernels of a
call, for FP32 products on either side of the line (no GPU needed)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

PEAKS = {"bf16_tflops": 1870.0, "sm_max_mhz": 2070.0}


@pytest.mark.parametrize("args,M,K,N,mult,bound,launches", [
    (("table1",), 512, 256, 128, 1, "alu", 4), (("systematic", 8, 3, 8), 8192, 8192, 8192, 6, "tensor", 7),
    (("mojette_a", 12, 9, 128), 1152, 64, 1024, 1, "alu", 5), (("mojette_a", 32, 24, 200), 4800, 512, 512, 6, "tensor", 9)])
def test_fp32(libbpx, args, M, K, N, mult, bound, launches):
    bpx = libbpx
    code = getattr(bpx.Code, args[0])(*args[1:])
    h = -(-M // code.num_sources)
    got, peak, _src, on, _kernel = bench._gemm_unit(bpx, code, "fp32", N, K, h, PEAKS, 152)
    assert (got, on) == (mult, bound)
    assert peak == pytest.approx(152 * 128 * 2 * 2070e6 / 1e12 if bound == "alu" else 1870.0)
    assert bench._launches(bpx, code, "fp32", N, K, h) == launches


# counted on the device: one call of each
@pytest.mark.parametrize("prec,launches", [("bf16x3", 5), ("bf16", 5), ("mxfp8", 5), ("exact", 7), ("fp16x3", 6),
                                           ("bf16x3-fused", 4)])
def test_launches(libbpx, prec, launches):
    code = libbpx.Code.systematic(8, 3, 8)
    assert bench._launches(libbpx, code, prec, 2048, 2048, 32) == launches
    tall = libbpx.Code.mojette_a(32, 24, 200)
    extra = {"fp16x3": 4, "exact": 3}.get(prec, 2)
    assert bench._launches(libbpx, tall, prec, 512, 512, 1) == launches + extra
