"""The schedule's forms, bit for bit against the oracle: graphs computed from
the grid or read from tables, in shared or global memory, rounds wider than
one warp orders and than the ready ring, and the peel lists in each of their
ways (through a whole multiplication of small integers)."""
import numpy as np
import pytest

from oracle import bpx_oracle as o
from paper_1904_11563_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

CODES = {
    "grid in shared memory": (("systematic", 8, 3, 8), 3),
    "computed cells": (("mojette_a", 12, 9, 340), 3),       # 3060 sources, lists by the second launch
    "computed cells, in-kernel lists": (("mojette_a", 12, 9, 100), 3),  # supports of 9: a warp a position
    "more columns than the table": (("mojette_a", 70, 56, 40), 10),
    "cells from tables": (("mojette_b", 8, 6, 400, 1), 2),
    "wide rounds": (("systematic", 40, 3, 400), 3),           # first round wider than half the ring
    "wide rounds, small": (("systematic", 20, 2, 40), 2),     # 256 < first round, everything on chip
    "one row": (("mojette_a", 5, 4, 1), 1),
}


def _pair(bpx, spec):
    kind, *a = spec
    ref = {"systematic": o.systematic_mojette, "mojette_a": o.construction_a, "mojette_b": o.construction_b}[kind]
    return getattr(bpx.Code, kind)(*a), ref(*a)


@pytest.mark.parametrize("name", CODES)
@pytest.mark.parametrize("cells", [False, True])
def test_plan_bit_exact(libbpx, name, cells):
    bpx = libbpx
    spec, e = CODES[name]
    code, ref = _pair(bpx, spec)
    m = W.erasure_mask(code.n, e, 7)
    mask = m[code.col_of_cell] if cells else m
    if cells:  # and every 50th cell of the columns that arrived
        mask = mask.copy()
        mask[::50] = 1
    ws = bpx.Workspace(code, 0, 0, 0, 1, bpx.FP32)
    order, rec, info = bpx.schedule(code, torch.from_numpy(mask).cuda(), ws, cells=cells)
    alive = [c for c in range(code.num_cells) if not (mask[c] if cells else m[code.col_of_cell[c]])]
    sch = o.wave_schedule(ref, alive)
    exp = np.full((code.num_sources, 3), -1, dtype=np.int32)
    exp[:len(sch.order)] = np.array(sch.order, dtype=np.int32).reshape(-1, 3)
    assert np.array_equal(order.cpu().numpy(), exp)
    assert list(rec.cpu().numpy()) == sch.recovered
    inf = info.cpu().numpy()
    assert inf[bpx.INFO_WAVES] == sch.num_waves and inf[bpx.INFO_SURVIVING] == len(alive)
    assert inf[bpx.INFO_DIRECT] == sum(1 for _s, _r, d in sch.order if d == 1)


@pytest.mark.parametrize("name", [n for n in CODES if n != "one row"])
def test_whole_path_integers(libbpx, name):
    bpx = libbpx
    spec, e = CODES[name]
    code, ref = _pair(bpx, spec)
    M, K, N = code.num_sources - 1, 64, 36
    A, B = W.matrix((M, K), "int", 5), W.matrix((K, N), "int", 6)
    m = W.erasure_mask(code.n, e, 7)
    ws = bpx.Workspace(code, M, N, K, 1, bpx.BF16X3)
    C, info = bpx.coded_matmul(code, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), 1, bpx.BF16X3,
                               torch.from_numpy(m).cuda(), ws)
    sch = o.wave_schedule(ref, o.surviving_cells(ref, list(np.nonzero(m)[0])))
    rec = np.array(sch.recovered[:M], dtype=bool)
    assert int(info[bpx.INFO_RECOVERED]) == sum(sch.recovered)
    assert np.array_equal(C[:M].cpu().numpy()[rec], o.reference_product(A, B)[rec])
