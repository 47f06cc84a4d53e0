"""The autotuners' built-in lists hold the defaults: tuning never ends slower
than not tuning."""
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# 128 x 64 tiles, which only the default takes, need two thirds of the time of
# the fastest named ones here (10.2 us against 14.8)
def test_small_product_keeps_the_default(libbpx):
    bpx = libbpx
    code, M, K, N, P = bpx.Code.systematic(8, 3, 8), 1024, 256, 128, bpx.BF16X3
    h = M // code.num_sources
    assert bpx.default_tile(code, P, N, K, h) == 64
    A, B = torch.randn((M, K), device="cuda"), torch.randn((K, N), device="cuda")
    mask = torch.from_numpy(W.erasure_mask(code.n, code.e, 1)).cuda()
    ws = bpx.Workspace(code, M, N, K, h, P)
    tuned = min(bpx.autotune(code, A, B, h, P, mask, ws)[1] for _ in range(5))
    default = min(bpx.autotune(code, A, B, h, P, mask, ws, configs=[0])[1] for _ in range(5))
    assert tuned <= 1.2 * default


def test_group_peel_list_holds_the_default_plan(libbpx):
    bpx = libbpx
    batch = []
    for i in range(3):
        code = bpx.Code.systematic(8, 3, 8)
        batch.append(dict(code=code, h=8, A=torch.randn((512, 128), device="cuda"), B=torch.randn((128, 256), device="cuda"),
                          C=bpx.alloc_C(code, 8, 256), mask=torch.from_numpy(W.erasure_mask(code.n, code.e, i)).cuda(),
                          info=torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda")))
    G = bpx.Group(batch, bpx.BF16X3)
    G.run()
    torch.cuda.synchronize()
    ref = [j["C"].clone() for j in batch]
    best, ms = G.autotune_peel()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert best in (0, sms // 8, sms // 4, sms // 2, sms, 2 * sms, 4 * sms, 8 * sms) and ms > 0
    G.run()
    torch.cuda.synchronize()
    assert all(torch.equal(j["C"], r) for j, r in zip(batch, ref))
    with pytest.raises(bpx.BpxError) as err:
        G.autotune_peel([0])
    assert err.value.code == bpx.ERR_INVAL
