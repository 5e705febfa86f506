"""Row-unit decode at every way four consecutive stored rows can fall: one width
(2, 4, 6 or 8 bits), a change of width after one, two or three of them, FP16 pivot rows
among them. The oracle steps the same pages; tolerances are the parity tests'."""
import numpy as np
import pytest

import oracle as O
from paper_2609_38169_gb300 import api as A, workloads as W

from gpu_helpers import Tally, compare_pools, compare_y, plans, to_dev

pytestmark = pytest.mark.gpu

CASES = [(4, (2, 4, 6, 8), 26), (6, (4, 6, 8), 102), (4, (2, 4, 6, 8), 0), (8, (4, 6, 8), 0)]


def _cfg(bits, cands, pivots):
    return W.WORKLOADS["channel"].replace(nominal_bits=bits, candidates=cands, n_pivots=pivots, pool_slots=4)


@pytest.mark.parametrize("bits,cands,pivots", CASES)
def test_row_width_mixes(bits, cands, pivots):
    wl = _cfg(bits, cands, pivots)
    cfg, plan, oplan, _ = plans(wl)
    mp = W.model_params(wl)
    slots = np.array([2, 0], np.int32)
    pool_o = np.zeros(wl.pool_slots * oplan.slot_stride, np.uint8)
    O.pool_encode(oplan, pool_o, 0, slots, O.warmup_states(wl, 0, 2))
    (slots_d,) = to_dev(slots)
    pool_d = A.alloc_pool(plan, wl.pool_slots)
    t = Tally()
    for step in range(2):
        inp = W.step_inputs(wl, mp, W.STREAM_DECODE, step, 0, batch=2)
        pool_d.copy_(pool_d.new_tensor(pool_o))
        q, k, v, beta, gate = to_dev(inp.q, inp.k, inp.v, inp.beta, inp.gate)
        y = v.new_empty((2, wl.hv, 128))
        y2, delta = y.clone(), y.clone()
        A.stepq_decode_readout(plan, 0, pool_d, slots_d, q, k, v, beta, gate, y2, delta)
        halves = pool_d.clone()
        A.stepq_decode_writeback(plan, 0, halves, slots_d, k, beta, gate, delta)
        A.stepq_decode_step(plan, 0, pool_d, slots_d, q, k, v, beta, gate, y)
        assert np.array_equal(halves.cpu().numpy(), pool_d.cpu().numpy())
        assert np.array_equal(y2.cpu().numpy(), y.cpu().numpy())
        y_o = O.pool_step(oplan, pool_o, 0, slots, inp)
        compare_y(t, y.cpu().numpy(), y_o)
        compare_pools(t, pool_d.cpu().numpy(), pool_o, oplan, 0, slots)
    t.check()
    assert A.stepq_device_error() == 0


def test_row_widths_cover_the_mixes():
    kinds = set()
    for case in CASES:
        _, plan, _, _ = plans(_cfg(*case))
        for h in plan.unit_bits.reshape(-1, 128):
            for s in np.sort(h)[::-1].reshape(-1, 4):
                kinds.add((int(s[0]), int((s == s[0]).sum())))
    assert {(b, 4) for b in (2, 4, 6, 8, 16)} <= kinds
    assert {(b, n) for b in (4, 6, 8, 16) for n in (1, 2, 3)} <= kinds
