"""Performance cases: the coded multiplications a user of this library runs,
through its public entry points (``paper_1904_11563_gb300.bpx``).

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes what a caller holds before the call (device inputs, the code
handle, a bound workspace, output buffers), ``run`` is one pass, ``work`` what
the pass cannot do without, ``exact`` the result in 64 bits without this
library's code.
"""
import random

import numpy as np
import torch

from paper_1904_11563_gb300 import bpx, straggler
from paper_1904_11563_gb300 import workloads as W

F64 = torch.float64


def listed():
    return [
        # The smallest calls: the tiny plain-FP32 workload (Table I code) and
        # the tiny cancellation-stressing split-BF16 one (Table III code).
        # A few microseconds of work each: launches and latency count.
        dict(name="tiny_fp32", path="matmul", code="table1", M=512, K=256, N=128, precision="fp32",
             dist="uniform", e=2, stragglers=False),
        dict(name="tiny_logu_bf16x3", path="matmul", code="table3", M=576, K=256, N=128, precision="bf16x3",
             dist="loguniform", e=2, stragglers=False),
        # Ordinary calls of ragged size: the accurate tensor-core mode decoding
        # from the first decodable set of arrived processors, and plain FP32.
        dict(name="ragged_straggler_fp16x3", path="matmul", code="systematic 6 2 6", M=1000, K=1416, N=1100,
             precision="fp16x3", dist="normal", e=0, stragglers=True),
        dict(name="ragged_fp32", path="matmul", code="systematic 8 3 8", M=2000, K=1992, N=2044, precision="fp32",
             dist="normal", e=3, stragglers=False),
        # The benchmark workload (n = 11 columns, 3 erased, 8192 cubed) in its
        # headline precision and in plain FP32.
        dict(name="bench_bf16x3", path="matmul", code="systematic 8 3 8", M=8192, K=8192, N=8192,
             precision="bf16x3", dist="normal", e=3, stragglers=False),
        dict(name="bench_fp32", path="matmul", code="systematic 8 3 8", M=8192, K=8192, N=8192, precision="fp32",
             dist="normal", e=3, stragglers=False),
        # The large projection-code workload (Construction A, n = 32, 16392
        # one-row sources, 8 erased), stage by stage: schedule and FP8 coded
        # products, then the sink's decode of arrived products.  (The decode
        # of FP8 products of so deep a code is ill-conditioned; its stages are
        # what a caller can check.)
        dict(name="tall_products_mxfp8", path="products", code="mojette_a 32 24 683", M=16384, K=16384, N=8192,
             precision="mxfp8", dist="uniform", e=8, stragglers=False),
        dict(name="tall_peel", path="peel", code="mojette_a 32 24 683", M=16392, K=0, N=8192, precision="fp32",
             dist="int", e=8, stragglers=False),
        # Exact slices on a deep projection code (the b = 64 point of the
        # grid-height sweep): what a caller takes when the peel is deep.
        dict(name="deep_exact", path="matmul", code="mojette_a 32 24 64", M=1536, K=4096, N=1024, precision="exact",
             dist="uniform", e=8, stragglers=False),
        # Many independent multiplications of uneven shapes and codes in one
        # grouped run.
        dict(name="batch48_bf16x3", path="batch", jobs=48, lo=256, hi=4096, precision="bf16x3", dist="normal",
             spec_seed=5),
        # The two-dimensional scheme in plain BF16, 8 x 8 output blocks.
        dict(name="twod_bf16", path="twod", code="systematic 8 3 8", M=4096, K=4096, N=4096, precision="bf16",
             dist="normal", e=3, stragglers=False),
        # End to end from page-locked host memory, one call at a time.
        dict(name="host_bf16x3", path="host", code="systematic 8 3 8", M=4096, K=4096, N=4096, precision="bf16x3",
             dist="normal", e=3, stragglers=False),
    ]


def _log(rng, lo, hi, mult):
    """A multiple of mult, log-uniform on [lo, hi]."""
    return max(mult, int(round(np.exp(rng.uniform(np.log(lo), np.log(hi))) / mult)) * mult)


def draw(rng: random.Random):
    path = rng.choice(["matmul"] * 5 + ["products", "peel", "exact", "batch", "twod", "host"])
    dist = rng.choice(["normal", "uniform"])
    if path == "batch":
        return dict(path="batch", jobs=rng.randint(4, 48), lo=256, hi=rng.choice([1024, 2048, 4096]),
                    precision=rng.choice(["bf16x3", "bf16"]), dist=dist, spec_seed=rng.randint(6, 10 ** 6))
    if path == "peel" or path == "products":
        n = rng.choice([8, 12, 16, 32])
        k, b = n - n // 4, _log(rng, 48, 683, 1)
        rows = k * b
        if path == "peel":
            return dict(path="peel", code=f"mojette_a {n} {k} {b}", M=rows, K=0, N=_log(rng, 256, 8192, 4),
                        precision="fp32", dist="int", e=n // 4, stragglers=False)
        p = rng.choice(["mxfp8", "bf16x3", "fp16x3"])
        return dict(path="products", code=f"mojette_a {n} {k} {b}", M=rows - rng.randint(0, 7),
                    K=_log(rng, 512, 8192, 128 if p == "mxfp8" else 8), N=_log(rng, 256, 8192, 4), precision=p,
                    dist="uniform", e=n // 4, stragglers=False)
    if path == "exact":
        n = rng.choice([12, 16, 32])
        k, b = n - n // 4, _log(rng, 8, 128, 1)
        return dict(path="matmul", code=f"mojette_a {n} {k} {b}", M=k * b, K=_log(rng, 256, 4096, 8),
                    N=_log(rng, 128, 2048, 4), precision="exact", dist="uniform", e=n // 4, stragglers=False)
    if path == "twod":
        k, e, b = rng.choice([(8, 3, 8), (6, 2, 6), (4, 2, 5)])
        return dict(path="twod", code=f"systematic {k} {e} {b}", M=_log(rng, 512, 6144, 1), K=_log(rng, 512, 6144, 8),
                    N=k * _log(rng, 64, 768, 4), precision=rng.choice(["bf16", "bf16x3"]), dist=dist, e=e,
                    stragglers=False)
    code, e = rng.choice([("systematic 8 3 8", 3), ("systematic 6 2 6", 2), ("systematic 10 2 4", 2), ("xcode 7", 2),
                          ("table1", 2), ("table3", 2)])
    if path == "host":
        return dict(path="host", code=code, M=_log(rng, 512, 6144, 1), K=_log(rng, 512, 6144, 8),
                    N=_log(rng, 512, 6144, 4), precision=rng.choice(["bf16x3", "fp16x3", "fp32"]), dist=dist, e=e,
                    stragglers=False)
    p = rng.choice(["fp32", "fp32", "bf16x3", "bf16x3", "fp16x3", "bf16", "mxfp8", "exact"])
    stragglers = rng.random() < 0.25
    return dict(path="matmul", code=code, M=_log(rng, 128, 6144, 1), K=_log(rng, 128, 6144, 128 if p == "mxfp8" else 8),
                N=_log(rng, 64, 6144, 4), precision=p, dist=dist, e=0 if stragglers else e, stragglers=stragglers)


def _code(text):
    kind, *args = text.split()
    return getattr(bpx.Code, kind)(*(int(a) for a in args))


def _matrix(shape, dist, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if dist == "normal":
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    if dist == "uniform":
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32).mul_(2).sub_(1)
    if dist == "int":
        return torch.randint(-8, 9, shape, generator=g, device="cuda").to(torch.float32)
    # magnitudes log-uniform on [1e-3, 1e3], random signs
    mag = torch.rand(shape, generator=g, device="cuda").mul_(2 * np.log(1e3)).sub_(np.log(1e3)).exp_()
    return mag * torch.where(torch.rand(shape, generator=g, device="cuda") < 0.5, -1.0, 1.0)


def _inputs(case, seed):
    return (_matrix((case["M"], case["K"]), case["dist"], 2 * seed + 1),
            _matrix((case["K"], case["N"]), case["dist"], 2 * seed + 2))


def _columns(n, e, seed):
    m = np.zeros(n, dtype=np.uint8)
    m[np.random.default_rng(seed).choice(n, size=e, replace=False)] = 1
    return m


def _mask(case, code, seed):
    """One byte per column (e columns straggled), or per cell (all but the
    first decodable set of arrivals)."""
    if not case["stragglers"]:
        return _columns(code.n, case["e"], seed)
    order, first, _t, _r = straggler.arrivals(
        code, straggler.task_times(code, W.exponential_draws(code.num_cells, 1.0, seed)))
    m = np.ones(code.num_cells, dtype=np.uint8)
    m[order[:first]] = 0
    return m


def _projections(n, k, b):
    """The cells of Construction A (the sources on each discrete line of slope
    -floor((n-1)/2) .. ceil((n-1)/2) of the b x k grid) and their columns."""
    z, l = np.divmod(np.arange(b * k), k)
    cells, cols = [], []
    for j in range(n):
        line = -z - l * (j - (n - 1) // 2)
        order = np.argsort(line, kind="stable")
        cuts = np.nonzero(np.diff(line[order]))[0] + 1
        cells += np.split(order, cuts)
        cols += [j] * (len(cuts) + 1)
    return cells, np.array(cols)


def _coded(cells, X):
    """Per cell, the sum of its sources' rows of X (one row a source)."""
    ptr = torch.from_numpy(np.cumsum([0] + [len(c) for c in cells])).cuda()
    src = torch.from_numpy(np.concatenate(cells)).cuda()
    G = torch.sparse_csr_tensor(ptr, src, torch.ones(len(src), dtype=X.dtype, device="cuda"), (len(cells), X.shape[0]))
    return G @ X


def _batch_specs(case):
    """The batch workload's shapes and codes; projection codes with a grid of
    at most 16 rows, whose peel floating point can carry."""
    out = []
    for sp in W.batch_specs(case["jobs"], case["spec_seed"], case["lo"], case["hi"]):
        if sp["code"][0] == "mojette_a":
            _, n, k, b = sp["code"]
            b = min(b, 16)
            sp = dict(sp, code=("mojette_a", n, k, b), h=-(-sp["M"] // (k * b)))
        out.append(sp)
    return out


def prepare(case, seed):
    prec = bpx.PRECISIONS[case["precision"]]
    if case["path"] == "batch":
        jobs, specs = [], _batch_specs(case)
        infos = torch.zeros((len(specs), bpx.INFO_LEN), dtype=torch.int32, device="cuda")
        for i, sp in enumerate(specs):
            code = _code(" ".join(str(x) for x in sp["code"]))
            A = _matrix((sp["M"], sp["K"]), case["dist"], 1000003 * seed + 2 * i)
            B = _matrix((sp["K"], sp["N"]), case["dist"], 1000003 * seed + 2 * i + 1)
            m = torch.from_numpy(W.erasure_mask(code.n, sp["e"], sp["mask_seed"] + seed)).cuda()
            jobs.append(dict(code=code, A=A, B=B, C=bpx.alloc_C(code, sp["h"], sp["N"]), mask=m,
                             info=infos[i], h=sp["h"]))
        return dict(path="batch", jobs=jobs, infos=infos, group=bpx.Group(jobs, prec))
    code = _code(case["code"])
    M, K, N = case["M"], case["K"], case["N"]
    h = -(-M // (code.b if case["path"] == "twod" else code.num_sources))
    hmask = _mask(case, code, seed)
    st = dict(path=case["path"], code=code, h=h, prec=prec, mask=torch.from_numpy(hmask).cuda(),
              opts=bpx.default_opts(mask_cells=1) if case["stragglers"] else None,
              info=torch.zeros(bpx.INFO_LEN, dtype=torch.int32, device="cuda"))
    if case["path"] == "peel":
        blocks = _matrix((code.num_sources, N), case["dist"], seed)  # h = 1
        cells, _ = _projections(code.n, code.k, code.b)
        st.update(N=N, ws=bpx.Workspace(code, 0, N, 8, h, prec), C=bpx.alloc_C(code, h, N),
                  products=_coded(cells, blocks))
        return st
    A, B = _inputs(case, seed)
    if case["path"] == "twod":
        st.update(A=A, B=B, ws=bpx.Workspace2D(code, M, N, K, h, prec),
                  C=torch.zeros((code.b * h, N), dtype=torch.float32, device="cuda"))
        return st
    st.update(ws=bpx.Workspace(code, M, N, K, h, prec), C=bpx.alloc_C(code, h, N))
    if case["path"] == "host":
        st.update(hA=A.cpu().pin_memory(), hB=B.cpu().pin_memory(), hmask=torch.from_numpy(hmask).pin_memory(),
                  hC=torch.zeros((M, N), dtype=torch.float32).pin_memory(), A=torch.empty_like(A),
                  B=torch.empty_like(B))
        return st
    st.update(A=A, B=B)
    if case["path"] == "products":
        st["products"] = torch.zeros((code.num_cells * h, N), dtype=torch.float32, device="cuda")
    return st


def run(s):
    if s["path"] == "batch":
        s["group"].run()
        return [j["C"] for j in s["jobs"]], s["infos"]
    code, h, prec, ws, opts = s["code"], s["h"], s["prec"], s["ws"], s["opts"]
    if s["path"] == "matmul":
        return bpx.coded_matmul(code, s["A"], s["B"], h, prec, s["mask"], ws, C=s["C"], opts=opts, info=s["info"])
    if s["path"] == "twod":
        return bpx.coded_matmul_2d(code, s["A"], s["B"], h, prec, s["mask"], ws, C=s["C"], opts=opts, info=s["info"])
    if s["path"] == "products":
        order, rec, info = bpx.schedule(code, s["mask"], ws)
        return order, rec, info, bpx.coded_products(code, s["A"], s["B"], h, prec, ws, products=s["products"],
                                                    C=s["C"], opts=opts), s["C"]
    if s["path"] == "peel":
        return bpx.peel_decode(code, s["products"], s["N"], h, s["C"], ws, opts=opts, mask=s["mask"],
                               info=s["info"]), s["info"]
    status, info = bpx.coded_matmul_host(code, s["hA"], s["hB"], h, prec, s["hmask"], s["hC"], s["A"], s["B"],
                                         s["mask"], s["C"], ws, opts=opts)
    return s["hC"], info, status


def _arrived(case, code):
    """Cells whose products are computed, on average over the masks."""
    if case["stragglers"]:  # the first decodable set: a little more than the sources
        return min(code.num_cells, 1.25 * code.num_sources)
    return code.num_cells * (code.n - case["e"]) / code.n


def work(case):
    if case["path"] == "batch":
        by = fl = 0
        for sp in _batch_specs(case):
            code = _code(" ".join(str(x) for x in sp["code"]))
            by += 4 * (sp["M"] * sp["K"] + sp["K"] * sp["N"] + sp["M"] * sp["N"])
            fl += 2 * sp["h"] * sp["N"] * sp["K"] * code.num_cells * (code.n - sp["e"]) / code.n
        return dict(bytes=by, flops=fl)
    code = _code(case["code"])
    M, K, N = case["M"], case["K"], case["N"]
    cells = _arrived(case, code)
    if case["path"] == "twod":
        h, w = -(-M // code.b), N // code.k
        per, _ = bpx.terms_2d(code)
        return dict(bytes=4 * (M * K + K * N + M * N),
                    flops=2.0 * h * w * K * float(per.sum()) * (code.n - case["e"]) / code.n)
    h = -(-M // code.num_sources)
    if case["path"] == "peel":  # every source: its resolver's product in, the block out; one add an edge
        deg = code.num_edges / code.num_cells
        return dict(bytes=8 * code.num_sources * h * N, flops=code.num_sources * h * N * max(0.0, deg - 1))
    out = cells * h * N if case["path"] == "products" else M * N
    return dict(bytes=4 * (M * K + K * N + out), flops=2.0 * cells * h * N * K)


def _padded(A, B, rows):
    C = torch.zeros((rows, B.shape[1]), dtype=F64, device="cuda")
    torch.matmul(A.to(F64), B.to(F64), out=C[:A.shape[0]])
    return C


def exact(case, seed):
    if case["path"] == "batch":
        out = []
        for i, sp in enumerate(_batch_specs(case)):
            kind, *a = sp["code"]
            S = {"table1": 4, "table3": 9}.get(kind) or (a[0] * a[2] if kind == "systematic" else a[1] * a[2])
            A = _matrix((sp["M"], sp["K"]), case["dist"], 1000003 * seed + 2 * i)
            B = _matrix((sp["K"], sp["N"]), case["dist"], 1000003 * seed + 2 * i + 1)
            out.append(_padded(A, B, S * sp["h"]))
        return out, None
    kind, *args = case["code"].split()
    args = [int(x) for x in args]
    k, b = {"table1": (2, 2), "table3": (3, 3)}.get(kind) or (
        (args[0] - 2, args[0]) if kind == "xcode" else (args[0], args[2]) if kind == "systematic" else args[1:])
    if case["path"] == "peel":
        return _matrix((k * b, case["N"]), case["dist"], seed).to(F64), None
    A, B = _inputs(case, seed)
    if case["path"] == "host":
        return torch.matmul(A.to(F64), B.to(F64)), None, None
    blocks = b if case["path"] == "twod" else k * b
    if case["path"] in ("twod", "matmul"):
        return _padded(A, B, blocks * -(-case["M"] // blocks)), None
    # products (h = 1): every cell of an arrived column, but the lowest
    # degree-one cell of each source, whose product goes to that source's row of C
    cells, cols = _projections(args[0], k, b)
    gone = _columns(args[0], case["e"], seed)[cols] == 1
    direct = {}
    for c, src in enumerate(cells):
        if len(src) == 1 and not gone[c]:
            direct.setdefault(int(src[0]), c)
    X = torch.zeros((blocks, case["K"]), dtype=F64, device="cuda")
    X[:case["M"]] = A
    P = torch.matmul(_coded(cells, X), B.to(F64))
    C = torch.zeros((blocks, case["N"]), dtype=F64, device="cuda")
    C[list(direct)] = P[list(direct.values())]
    P[list(direct.values())] = 0
    P[torch.from_numpy(gone).cuda()] = 0
    return None, None, None, P, C
