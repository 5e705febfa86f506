"""The one-launch passes of stepq_calibrate_from_trace against the same protocol
driven token by token through the single-step entry points (observe, FP32 decode,
distortion), over odd token counts, sampling intervals, head groups and fit passes."""
import numpy as np
import pytest

from paper_2609_38169_gb300 import api as A, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T
    if not T.cuda.is_available():
        pytest.skip("no CUDA device")
    return T


@pytest.mark.parametrize("name,layers,hk,hv,n,T,every,iters,pivots", [
    ("tiny", 1, 4, 4, 1, 1, 1, 1, 0),          # one token, one sample
    ("gqa", 2, 2, 6, 3, 37, 5, 2, 1),          # ragged tail, three value heads a key head
    ("channel", 2, 3, 3, 2, 21, 4, 1, 9),      # pivot rows: the second pass
    ("channel", 2, 3, 3, 2, 21, 4, 1, 2),      # pivot rows in some heads only
    ("channel", 1, 1, 2, 5, 64, 64, 2, 0),     # a single sample at the end
])
def test_calibration_equals_token_steps(torch, name, layers, hk, hv, n, T, every, iters, pivots):
    wl = W.WORKLOADS[name].replace(layers=layers, hk=hk, hv=hv, n_pivots=pivots, fit_iters=iters)
    cfg = A.Config.from_workload(wl)
    mp = W.model_params_torch(W.model_params(wl), "cuda")
    steps = [[W.torch_step_inputs(wl, mp, t, layer, "cuda", W.STREAM_CALIB, batch=n) for t in range(T)]
             for layer in range(layers)]
    trace = [torch.stack([torch.stack([s[i] for s in per]) for per in steps]).contiguous() for i in range(5)]
    got = A.stepq_calibrate_from_trace(cfg, *trace, every=every)

    f64 = dict(dtype=torch.float64, device="cuda")
    U, K1 = A.stepq_num_units(cfg), len(cfg.candidates) + 1
    om, lr = torch.zeros((layers, hv, 128), **f64), torch.zeros(U, **f64)
    for layer in range(layers):
        for t in range(T):
            q, k, v, beta, gate = [x[layer, t] for x in trace]
            A.stepq_calib_observe(cfg, layer, q, k, beta, gate, om, lr)
    omega = (om / (n * T)).float().cpu().numpy()
    # fp64 sums in another order: a few ulps of fp64, one of the rounding to fp32
    np.testing.assert_allclose(got.omega, omega, rtol=2e-7)
    np.testing.assert_allclose(got.mean_log_ret, lr.cpu().numpy() / (n * T), rtol=1e-12)

    w = torch.from_numpy(A.stepq_row_weights(cfg, got.omega)).cuda()
    one = A.Config.from_workload(wl.replace(layers=1))
    slots = torch.arange(n, dtype=torch.int32, device="cuda")
    y = torch.empty((n, hv, 128), device="cuda")

    def distortion(pivot_rows):
        acc = torch.zeros((U, K1), **f64)
        for layer in range(layers):
            S = torch.zeros((n, 1, hv, 128, 128), device="cuda")
            for t in range(T):
                A.stepq_fp32_decode_step(one, 0, S, slots, *[x[layer, t] for x in trace], y)
                if (t + 1) % every == 0:
                    A.stepq_calib_distortion(cfg, layer, w, pivot_rows, S[:, 0].contiguous(), acc)
        return acc.cpu().numpy() / (T // every * n)

    # the states are the same bit for bit; only the order of the fp64 sums differs
    np.testing.assert_allclose(got.dist_stage1, distortion(None), rtol=1e-12)
    np.testing.assert_array_equal(got.pivot, A.stepq_select_pivots(cfg, got.mean_log_ret, got.dist_stage1))
    rows = cfg.unit_rows and pivots > 0
    want = distortion(torch.from_numpy(got.pivot).cuda()) if rows else got.dist_stage1
    np.testing.assert_allclose(got.dist, want, rtol=1e-12)
    assert got.n_samples == T // every * n and got.n_tokens == n * T
