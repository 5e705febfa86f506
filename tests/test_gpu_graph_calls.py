"""Every call whose kernel may start under the previous kernel's end, captured into one
CUDA graph in which each reads what the one before wrote: the replays give the bytes of
the same calls made one by one with a device synchronisation in between."""
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
def test_captured_chain(torch, name, B):
    wl = W.WORKLOADS[name].replace(batch=B, pool_slots=B)
    cfg, plan, _, _ = plans(wl)
    mp = W.model_params_torch(W.model_params(wl), "cuda")
    inp = [W.torch_step_inputs(wl, mp, t, 0, "cuda", batch=B) for t in range(3)]
    T = 33
    pre = [torch.stack([x[i] for x in inp] * 11, dim=1).contiguous() for i in range(5)]
    slots = torch.arange(B, dtype=torch.int32, device="cuda")
    S, yp = torch.empty((B, wl.hv, 128, 128), device="cuda"), torch.empty((B, T, wl.hv, 128), device="cuda")
    ys, d = (torch.empty((B, wl.hv, 128), device="cuda") for _ in range(2))
    pool, dense = A.alloc_pool(plan, B), torch.empty((B, 1, wl.hv, 128, 128), device="cuda")
    pool8 = torch.zeros(B * A.stepq_intb_slot_bytes(cfg, 8), dtype=torch.uint8, device="cuda")
    bufs = S, yp, ys, d, pool, dense, pool8

    def chain(between):
        A.stepq_prefill_fp32(cfg, S, *pre, yp); between()
        A.stepq_quantize_pool(plan, 0, S, slots, pool); between()
        for q, k, v, beta, gate in inp:
            A.stepq_decode_readout(plan, 0, pool, slots, q, k, v, beta, gate, ys, d); between()
            A.stepq_decode_writeback(plan, 0, pool, slots, k, beta, gate, d); between()
            A.stepq_decode_step(plan, 0, pool, slots, q, k, ys, beta, gate, ys); between()
        A.stepq_dequantize_pool(plan, 0, pool, slots, dense); between()
        A.stepq_intb_quantize_pool(cfg, 8, 0, dense, slots, pool8); between()
        for q, k, v, beta, gate in inp:
            A.stepq_fp32_decode_step(cfg, 0, dense, slots, q, k, ys, beta, gate, ys); between()
            A.stepq_intb_decode_step(cfg, 8, 0, pool8, slots, q, k, ys, beta, gate, ys); between()

    def clear():
        for b in bufs:
            b.zero_()

    clear()
    chain(torch.cuda.synchronize)
    want = [b.clone() for b in bufs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        clear()
        chain(lambda: None)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert A.stepq_device_error() == 0
        for got, b in zip(bufs, want):
            assert torch.equal(got, b)
