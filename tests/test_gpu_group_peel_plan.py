"""The default plan of a small batch's peel against the same peel with the
plan of one CTA an SM and job (the same kernels and jobs): wide chunks, right
for many jobs, made four jobs' chains twice as long."""
import ctypes as ct

import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _peel_ms(bpx, G):
    """Best of five runs, by the events around the stage."""
    best = float("inf")
    for _ in range(7):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * bpx.NUM_STAGES)]
        for e in ev:
            e.record()
        opts = bpx.default_opts()
        arr = (ct.c_void_p * len(ev))(*[e.cuda_event for e in ev])
        opts.stage_events = ct.cast(arr, ct.POINTER(ct.c_void_p))
        G.run(opts)
        torch.cuda.synchronize()
        best = min(best, ev[2 * bpx.STAGE_PEEL].elapsed_time(ev[2 * bpx.STAGE_PEEL + 1]))
    return best


@pytest.mark.parametrize("jobs,hi", [(4, 1024), (4, 2048), (8, 2048)])
def test_small_batches(libbpx, jobs, hi):
    bpx = libbpx
    batch = []
    for i, sp in enumerate(W.batch_specs(jobs, 6, 256, hi)):
        kind, *a = sp["code"]
        if kind == "mojette_a":
            a[2] = min(a[2], 16)
        code = getattr(bpx.Code, kind)(*a)
        h = -(-sp["M"] // code.num_sources)
        batch.append(dict(code=code, A=torch.randn((sp["M"], sp["K"]), device="cuda"),
                          B=torch.randn((sp["K"], sp["N"]), device="cuda"), C=bpx.alloc_C(code, h, sp["N"]), h=h,
                          mask=torch.from_numpy(W.erasure_mask(code.n, sp["e"], sp["mask_seed"] + 1)).cuda(),
                          info=torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda")))
    G = bpx.Group(batch, bpx.BF16X3)
    default = _peel_ms(bpx, G)
    G.autotune_peel([152])
    tuned = _peel_ms(bpx, G)
    assert default <= 1.4 * tuned, (default, tuned)
