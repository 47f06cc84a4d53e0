"""Grouped runs at the edges of their launch plans, job by job against single
calls (the same bits): tiles past the surviving rows, a CTA's rows over several
cells and jobs, one job and more jobs than the live-tile table holds, and peel
chunks of every size."""
import pytest

from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _check(bpx, specs, prec, config=0):
    jobs = []
    for i, (args, M, K, N, e) in enumerate(specs):
        code = getattr(bpx.Code, args[0])(*args[1:])
        g = torch.Generator(device="cuda")
        g.manual_seed(i)
        h = -(-M // code.num_sources)
        jobs.append(dict(code=code, h=h, A=torch.randn((M, K), generator=g, device="cuda"),
                         B=torch.randn((K, N), generator=g, device="cuda"), C=bpx.alloc_C(code, h, N),
                         mask=torch.from_numpy(W.erasure_mask(code.n, e, i)).cuda(),
                         info=torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda")))
    G = bpx.Group(jobs, prec)
    if config:
        G.set_config(config)
    for _ in range(2):
        G.run()
    torch.cuda.synchronize()
    for j in jobs:
        (M, K), N = j["A"].shape, j["B"].shape[1]
        C, info = bpx.coded_matmul(j["code"], j["A"], j["B"], j["h"], prec, j["mask"],
                                   bpx.Workspace(j["code"], M, N, K, j["h"], prec))
        assert torch.equal(j["info"][:5], info[:5])
        assert torch.equal(j["C"], C)


MIXED = [(("table1",), 130, 8, 4, 3), (("table3",), 700, 264, 260, 2), (("systematic", 8, 3, 8), 1000, 72, 516, 3),
         (("systematic", 20, 2, 60), 1250, 520, 132, 2), (("mojette_a", 12, 9, 16), 300, 1032, 36, 3),
         (("mojette_a", 16, 12, 100), 1200, 200, 1030 * 4, 4)]


@pytest.mark.parametrize("prec", ["bf16x3", "bf16"])
@pytest.mark.parametrize("config", [0, 8082, 8086])  # 256 x 256, 128 x 128 and 32-wide slices
def test_mixed(libbpx, prec, config):
    _check(libbpx, MIXED, libbpx.PRECISIONS[prec], config)


def test_one_job(libbpx):
    _check(libbpx, MIXED[3:4], libbpx.BF16X3)


@pytest.mark.parametrize("n", [65, 1030])  # past the live-tile tables of 32- and 64-wide slices
def test_many_jobs(libbpx, n):
    _check(libbpx, [(("table1",), 40 + i % 7, 64, 4 * (1 + i % 5), 1 + i % 3) for i in range(n)], libbpx.BF16X3,
           8086 if n < 1000 else 0)
