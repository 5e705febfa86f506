"""Pack and unpack over many items per CTA: one call over every layer equals calls of
one slot and one layer each, byte for byte, with slot ids out of range in between."""
import numpy as np
import pytest

from paper_2609_38169_gb300 import api as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


def _plan(gate, layers, hv, cands, nominal, pivots, iters):
    cfg = A.Config(n_layers=layers, n_key_heads=hv, n_value_heads=hv, gate_kind=gate, nominal_bits=nominal,
                   candidates=cands, n_pivots=pivots, fit_iters=iters)
    g = np.random.default_rng(5)
    n = A.stepq_num_units(cfg)
    dist = g.lognormal(0, 2, n)[:, None] * np.array([4.0 ** -b for b in cands] + [4.0 ** -11])[None]
    return A.stepq_fit_scales(cfg, g.lognormal(size=(layers, hv, 128)).astype(np.float32),
                              np.log(g.uniform(0.8, 0.999, n)), dist)


@pytest.mark.parametrize("gate,layers,hv,B,cands,nominal,pivots,iters", [
    (A.GATE_SCALAR, 2, 37, 9, (2, 4, 6, 8), 4, 3, 1),      # 666 items, every width and FP16 heads
    (A.GATE_SCALAR, 3, 1, 2, (6,), 6, 0, 3),
    (A.GATE_CHANNEL, 2, 23, 15, (2, 4, 6, 8), 4, 200, 1),  # 690 items, FP16 rows
    (A.GATE_CHANNEL, 1, 1, 1, (8,), 8, 0, 2),
])
def test_all_layers_equal_single_items(torch, gate, layers, hv, B, cands, nominal, pivots, iters):
    plan = _plan(gate, layers, hv, cands, nominal, pivots, iters)
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    S = torch.randn((B, layers, hv, 128, 128), generator=g, device="cuda")
    S *= torch.exp(torch.randn((B, layers, hv, 128, 1), generator=g, device="cuda"))
    S[B // 2, 0, 0] = 0.0                                   # scales at their floor
    S[0, -1, -1] *= 1e9                                     # a capped column start: clamped codes
    if B > 3:
        S[1, 0, 0, 3, 5] = float("inf")
    slots = torch.randperm(B + 2, generator=g, device="cuda")[:B].to(torch.int32)
    bad = [1, B - 2] if B > 4 else []
    given = slots.clone()
    for i, b in enumerate(bad):
        given[b] = (-1, B + 2)[i]
    pool, one = A.alloc_pool(plan, B + 2), A.alloc_pool(plan, B + 2)
    A.stepq_quantize_pool(plan, -1, S, given, pool)
    good = [b for b in range(B) if b not in bad]
    for b in good:
        for layer in range(layers):
            A.stepq_quantize_pool(plan, layer, S[b:b + 1, layer].contiguous(), slots[b:b + 1], one)
    assert A.stepq_device_error() == (2 if bad else 0)      # STEPQ_ERR_SLOT_RANGE
    assert torch.equal(pool, one)
    out, ref = torch.zeros_like(S), torch.zeros_like(S)
    A.stepq_dequantize_pool(plan, -1, pool, given, out)
    for b in good:
        for layer in range(layers):
            part = torch.empty((1, hv, 128, 128), device="cuda")
            A.stepq_dequantize_pool(plan, layer, pool, slots[b:b + 1], part)
            ref[b, layer] = part[0]
    assert A.stepq_device_error() == (2 if bad else 0)
    assert torch.equal(out.view(torch.int32), ref.view(torch.int32))
    # within a quantization step of the state where the scales are in range
    quiet = [b for b in good if b not in (0, 1, B // 2)]
    if quiet:
        err = torch.linalg.vector_norm(out[quiet] - S[quiet]) / torch.linalg.vector_norm(S[quiet])
        assert err < 0.5
