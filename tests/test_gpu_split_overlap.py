"""The split decode step with its two halves on two streams: how they share the chip."""
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


@pytest.mark.parametrize("name", ["pool", "drift"])
def test_writebacks_run_beside_the_readouts(torch, name):
    """With a token's readouts queued on one stream and its writebacks on another, the
    writebacks are not held back until the last readout is done: each runs beside the two
    readouts after its own, so that all but the last three are complete by then."""
    layers, B = 12, 128
    wl = W.WORKLOADS[name].replace(layers=1, batch=B, pool_slots=B)
    _, plan, _, _ = plans(wl)
    mp = W.model_params_torch(W.model_params(wl), "cuda")
    q, k, v, beta, gate = W.torch_step_inputs(wl, mp, 0, 0, "cuda", batch=B)
    slots = torch.arange(B, dtype=torch.int32, device="cuda")
    pools = [A.alloc_pool(plan, B) for _ in range(layers)]        # a pool per layer, of one plan
    S = torch.randn((B, wl.hv, 128, 128), device="cuda")
    for pool in pools:
        A.stepq_quantize_pool(plan, 0, S, slots, pool)
    y, d = (torch.empty((layers, B, wl.hv, 128), device="cuda") for _ in range(2))
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    done = [torch.cuda.Event(enable_timing=True) for _ in range(layers)]
    last = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    with torch.cuda.stream(main):
        torch.cuda._sleep(20_000_000)                            # about 10 ms: all is queued before it runs
        for n, pool in enumerate(pools):
            A.stepq_decode_readout(plan, 0, pool, slots, q, k, v, beta, gate, y[n], d[n])
            ready = torch.cuda.Event()
            ready.record()
            side.wait_event(ready)
            A.stepq_decode_writeback(plan, 0, pool, slots, k, beta, gate, d[n], stream=side)
            done[n].record(side)
        last.record()
    torch.cuda.synchronize()
    assert A.stepq_device_error() == 0
    early = sum(e.elapsed_time(last) > 0 for e in done)
    assert early >= layers - 3, early
