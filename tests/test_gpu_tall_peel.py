"""Pipelined peel of tall codes against the wave-by-wave forms, which a peel
over few CTAs takes: each result is the same chain of subtractions, so the bits
agree.  Widths at the edges: one float4, a last slice shorter than the others,
slices that do not divide the CTA's threads, the widest slices, and supports at
most of which a round holds eight positions."""
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CODES = {
    "supports of 9": (("mojette_a", 12, 9, 120), 3),
    "supports of 24": (("mojette_a", 32, 24, 60), 8),
    "supports of 32, the most": (("mojette_a", 40, 32, 34), 8),
    "systematic": (("systematic", 8, 3, 130), 3),
    "nothing erased": (("mojette_a", 12, 9, 120), 0),
    "not recovered": (("mojette_a", 12, 9, 120), 4),
}


@pytest.mark.parametrize("comp", [-1, 3])
@pytest.mark.parametrize("N,h", [(4, 1), (36, 1), (1000, 1), (4096, 2), (8192, 2), (4100, 4)])
@pytest.mark.parametrize("name", CODES)
def test_same_bits_as_by_waves(libbpx, name, N, h, comp):
    bpx = libbpx
    args, e = CODES[name]
    code = getattr(bpx.Code, args[0])(*args[1:])
    g = torch.Generator(device="cuda")
    g.manual_seed(N + h)
    wide = max(N, 1024)  # few CTAs take the other forms from 33 float4s a CTA on
    P = torch.randn((code.num_cells * h, wide), generator=g, device="cuda")
    m = torch.from_numpy(W.erasure_mask(code.n, e, 7)).cuda()
    out = []
    for n, ctas in ((N, 0), (wide, 1)):
        C = torch.zeros((code.num_sources * h, n), device="cuda")
        ws = bpx.Workspace(code, 0, n, 8, h, bpx.PRECISIONS["fp32"])
        bpx.peel_decode(code, P[:, :n].contiguous(), n, h, C, ws, mask=m,
                        opts=bpx.default_opts(peel_ctas=ctas, compensate_depth=comp))
        out.append(C[:, :N])
    assert torch.equal(out[0].contiguous().view(torch.int32), out[1].contiguous().view(torch.int32))
