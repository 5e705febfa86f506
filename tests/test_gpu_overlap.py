"""Launches that may start before the previous kernel has ended: a chain in which every
call reads what the one before wrote gives the same bytes with and without a device
synchronisation between the calls."""
import pytest

from paper_2609_38169_gb300 import api as A, workloads as W

from gpu_helpers import plans

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


@pytest.mark.parametrize("name,B", [("gqa", 1), ("gqa", 40), ("channel", 1), ("channel", 40)])
def test_dependent_chain(torch, name, B):
    wl = W.WORKLOADS[name].replace(batch=B, pool_slots=B)
    cfg, plan, _, _ = plans(wl)
    mp = W.model_params_torch(W.model_params(wl), "cuda")
    inp = [W.torch_step_inputs(wl, mp, t, 0, "cuda", batch=B) for t in range(6)]
    T = 33
    pre = [torch.stack([x[i] for x in inp] * 6, dim=1)[:, :T].contiguous() for i in range(5)]
    slots = torch.arange(B, dtype=torch.int32, device="cuda")

    def chain(between):
        S = torch.zeros((B, wl.hv, 128, 128), device="cuda")
        ys, yp = torch.zeros((B, wl.hv, 128), device="cuda"), torch.empty((B, T, wl.hv, 128), device="cuda")
        pool = A.alloc_pool(plan, B)
        pool8 = torch.zeros(B * A.stepq_intb_slot_bytes(cfg, 8), dtype=torch.uint8, device="cuda")
        dense = torch.empty((B, 1, wl.hv, 128, 128), device="cuda")
        torch.cuda.synchronize()
        A.stepq_prefill_fp32(cfg, S, *pre, yp); between()
        A.stepq_quantize_pool(plan, 0, S, slots, pool); between()
        for q, k, v, beta, gate in inp:
            # the step reads the y that the previous launch wrote as its v
            A.stepq_decode_step(plan, 0, pool, slots, q, k, ys, beta, gate, ys); between()
            A.stepq_decode_step(plan, 0, pool, slots, q, k, v, beta, gate, ys); between()
        A.stepq_dequantize_pool(plan, 0, pool, slots, dense); between()
        A.stepq_intb_quantize_pool(cfg, 8, 0, dense, slots, pool8); between()
        for q, k, v, beta, gate in inp:
            A.stepq_fp32_decode_step(cfg, 0, dense, slots, q, k, ys, beta, gate, ys); between()
            A.stepq_intb_decode_step(cfg, 8, 0, pool8, slots, q, k, ys, beta, gate, ys); between()
        torch.cuda.synchronize()
        assert A.stepq_device_error() == 0
        return S, yp, pool, pool8, dense, ys

    want = chain(torch.cuda.synchronize)
    for _ in range(3):
        for a, b in zip(chain(lambda: None), want):
            assert torch.equal(a, b)
