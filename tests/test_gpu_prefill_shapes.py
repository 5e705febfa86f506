"""Chunked prefill against the token recurrence in fp64 at the sizes where the chunk
pipeline can go wrong: one token, tails of one token short or long of a chunk, one chunk
an item, odd head groups, items fewer and more than CTAs, and strong gates."""
import pytest

from paper_2609_38169_gb300 import api as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


@pytest.mark.parametrize("channel", [False, True])
@pytest.mark.parametrize("B,hk,hv,T,lo", [(1, 1, 1, 1, 0.8), (2, 1, 3, 31, 0.8), (1, 2, 2, 33, 0.8), (3, 2, 6, 64, 0.15),
                                          (40, 4, 8, 97, 0.8), (1, 1, 2, 1030, 0.9), (160, 1, 1, 32, 0.8)])
def test_prefill_recurrence(torch, channel, B, hk, hv, T, lo):
    g = torch.Generator(device="cuda")
    g.manual_seed(17 * T + B)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    uni = lambda *s: torch.rand(s, generator=g, device="cuda")
    q, k, v = rnd(B, T, hk, 128), rnd(B, T, hk, 128), rnd(B, T, hv, 128)
    k /= torch.linalg.vector_norm(k, dim=-1, keepdim=True)
    beta = torch.sigmoid(rnd(B, T, hv))
    gate = lo + (0.999 - lo) * (uni(B, T, hv, 128) if channel else uni(B, T, hv))
    S = rnd(B, hv, 128, 128)
    Sd, y = S.double().reshape(B * hv, 128, 128), torch.empty((B, T, hv, 128), device="cuda")
    cfg = A.Config(1, hk, hv, A.GATE_CHANNEL if channel else A.GATE_SCALAR)
    A.stepq_prefill_fp32(cfg, S, q, k, v, beta, gate, y)
    want = torch.empty((B, T, hv, 128), dtype=torch.float64, device="cuda")
    per = lambda x, t: x[:, t].double().repeat_interleave(hv // hk, 1).reshape(B * hv, 128)
    for t in range(T):
        kt, qt = per(k, t), per(q, t)
        Sd = Sd * gate[:, t].double().reshape(B * hv, -1, 1)
        d = v[:, t].double().reshape(B * hv, 128) - torch.einsum("nij,ni->nj", Sd, kt)
        Sd = Sd + (beta[:, t].double().reshape(-1, 1) * kt)[:, :, None] * d[:, None, :]
        want[:, t] = torch.einsum("nij,ni->nj", Sd, qt).reshape(B, hv, 128)
    assert A.stepq_device_error() == 0
    # the bounds of the recurrence parity (1e-4) on each token's readout and the state
    rel = torch.linalg.vector_norm(y - want, dim=-1) / torch.linalg.vector_norm(want, dim=-1)
    assert rel.max() <= 1e-4, rel.max()
    Sd = Sd.reshape(B, hv, 128, 128)
    assert (S - Sd).abs().max() <= 1e-4 * Sd.abs().max()
