"""Rounds of every width that the schedule orders in a way of its own, against
the oracle, and a middling round's time against a larger one's."""
import numpy as np
import pytest

from oracle import bpx_oracle as o

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


# one round of 2 b sources: a lane each, up to four a lane, by depth
@pytest.mark.parametrize("b", [1, 15, 16, 17, 32, 33, 48, 49, 63, 64, 65, 129, 300])
def test_one_round(libbpx, b):
    bpx = libbpx
    code, ref = bpx.Code.systematic(2, 1, b), o.systematic_mojette(2, 1, b)
    mask = np.zeros(code.n, dtype=np.uint8)
    mask[2] = 1  # the parity column: both data columns hold their sources
    order, rec, info = bpx.schedule(code, torch.from_numpy(mask).cuda(), bpx.Workspace(code, 0, 0, 0, 1, bpx.FP32))
    sch = o.wave_schedule(ref, o.surviving_cells(ref, [2]))
    assert np.array_equal(order.cpu().numpy(), np.array(sch.order, dtype=np.int32).reshape(-1, 3))
    assert int(info[bpx.INFO_WAVES]) == sch.num_waves and int(info[bpx.INFO_RECOVERED]) == 2 * b


def test_a_middling_round_costs_no_more_than_a_wide_one(libbpx):
    bpx = libbpx

    def us(*args):
        code = bpx.Code.mojette_a(*args)
        ws = bpx.Workspace(code, 0, 0, 0, 1, bpx.FP32)
        mask = torch.zeros(code.n, dtype=torch.uint8, device="cuda")
        mask[:code.n // 4] = 1
        best = float("inf")
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                bpx.schedule(code, mask, ws)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20 * 1e3)
        return best

    # one round of 252 sources in 3924 cells against one of 288 in 5904
    assert us(27, 21, 12) <= 1.4 * us(32, 24, 12)
