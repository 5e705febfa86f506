"""Failure detection in the prefill kernel without a fault: the test switch keeps the first
q and k of one item from being copied, so that the warps that wait for them, and those
that wait for these warps, give up one after the other. The launch returns and reports
STEPQ_ERR_TIMEOUT, and the next, normal call on the same context has the results of one
that came before."""
import pytest

from paper_2609_38169_gb300 import api as A

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


# one CTA an item, the CTA's only item or one of several; and a CTA's second item, with the
# tensor work of the first behind it
@pytest.mark.parametrize("channel", [False, True])
@pytest.mark.parametrize("B,hv,T,withhold", [(1, 2, 20, 0), (2, 4, 100, 5), (90, 4, 70, 3), (90, 4, 70, 157)])
def test_bounded_waits_run_out_and_recover(torch, B, hv, T, withhold, channel):
    g = torch.Generator(device="cuda")
    g.manual_seed(B + T)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    q, k, v, S0 = rnd(B, T, 1, 128), rnd(B, T, 1, 128), rnd(B, T, hv, 128), rnd(B, hv, 128, 128)
    k /= torch.linalg.vector_norm(k, dim=-1, keepdim=True)
    beta, gate = torch.sigmoid(rnd(B, T, hv)), 0.9 + 0.09 * torch.sigmoid(rnd(*([B, T, hv] + [128] * channel)))
    cfg = A.Config(1, 1, hv, A.GATE_CHANNEL if channel else A.GATE_SCALAR)

    def call():
        S, y = S0.clone(), torch.empty((B, T, hv, 128), device="cuda")
        A.stepq_prefill_fp32(cfg, S, q, k, v, beta, gate, y)
        return S, y, A.stepq_device_error()                                     # synchronises

    S, y, status = call()
    assert status == 0
    A.stepq_debug_stall(1_000_000, withhold)
    try:
        assert call()[2] == 8                                                   # STEPQ_ERR_TIMEOUT
    finally:
        A.stepq_debug_stall()
    S2, y2, status = call()
    assert status == 0 and torch.equal(S, S2) and torch.equal(y, y2)
