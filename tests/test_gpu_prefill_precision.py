"""Prefill's W = (I + A)^-1 R against fp64, read off one chunk: unit gates, a zero state, and
queries that are orthogonal to every other token's key, so that y_t is w_t. Keys, values and
beta lie on grids on which A and R are exact in fp32, so that the error is that of W alone."""
import numpy as np
import pytest

from paper_2609_38169_gb300 import api as A

pytestmark = pytest.mark.gpu
T = 32


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


def substitution(a, r):
    """Forward substitution, each fma rounded to fp32."""
    w = r.copy()
    for s in range(T - 1):
        w[s + 1:] = (w[s + 1:] - np.outer(a[s + 1:, s], w[s].astype(np.float64))).astype(np.float32)
    return w


@pytest.mark.parametrize("channel", [False, True])
@pytest.mark.parametrize("beta", [0.5, 1.0])
@pytest.mark.parametrize("corr", [0.0, 0.9, 0.99, 1.0])      # of the keys: random to all equal
def test_w(torch, corr, beta, channel):
    rng = np.random.default_rng([int(100 * corr), int(10 * beta)])
    B = 8
    k, q, v = (np.zeros((B, T, 1, 128), np.float32) for _ in range(3))
    want, plain = np.empty((B, T, 128)), np.empty((B, T, 128))
    for b in range(B):
        c = corr**0.5 * rng.standard_normal(96) + (1 - corr)**0.5 * rng.standard_normal((T, 96))
        c *= 0.96875 / np.linalg.norm(c, axis=1, keepdims=True)
        k[b, :, 0, :32], q[b, :, 0, :32] = 0.25 * np.eye(T), 4 * np.eye(T)
        k[b, :, 0, 32:] = np.round(256 * c) / 256
        v[b, :, 0] = np.round(256 * rng.standard_normal((T, 128))) / 256
        kd = k[b, :, 0].astype(np.float64)
        a, r = np.tril(beta * kd @ kd.T, -1), beta * v[b, :, 0]
        assert (a == a.astype(np.float32)).all()
        want[b], plain[b] = np.linalg.solve(np.eye(T) + a, r.astype(np.float64)), substitution(a, r)
    dev = lambda x: torch.from_numpy(x).cuda()
    S, y = torch.zeros((B, 1, 128, 128), device="cuda"), torch.empty((B, T, 1, 128), device="cuda")
    gate = torch.ones((B, T, 1, 128) if channel else (B, T, 1), device="cuda")
    A.stepq_prefill_fp32(A.Config(1, 1, 1, A.GATE_CHANNEL if channel else A.GATE_SCALAR), S, dev(q), dev(k), dev(v),
                         torch.full((B, T, 1), beta, device="cuda"), gate, y)
    assert A.stepq_device_error() == 0
    err = lambda x: np.linalg.norm(x - want) / np.linalg.norm(want)
    # No further off than the substitution; w_t reaches y_t as a head of 11 bits and a rest
    # rounded to 11, which is 2^-24 of it in the root mean square.
    assert err(y[:, :, 0].cpu().numpy()) <= np.hypot(err(plain), 2.0**-24)
