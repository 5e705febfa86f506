// The calibration protocol of App. A.3 behind one C entry point: it drives the
// observe kernel and the replay kernel (FP32 recurrence with its candidate
// distortions) over a recorded trace, forms the means, chooses the FP16 pivots and,
// for row units, repeats the replay with the pivot rows held out of the column fit
// (App. C.2).
//
// Each pass is one launch over all layers, sequences and heads. One launch per token
// and layer, as before, left the chip idle between and inside them (observe 26 us on
// 32 CTAs, replay 11 us on the state's way through memory): the four-layer channel-gate
// model with 8 sequences of 256 tokens took 147 ms, 9.3 ms now.
#include <algorithm>
#include <cstring>
#include <vector>

#include "internal.h"

using namespace stepq;

namespace {

size_t up256(size_t n) { return (n + 255) / 256 * 256; }

// Regions of the caller's workspace, each 256-byte aligned.
struct Workspace {
    double *omega_sum, *logret_sum, *acc, *scratch;
    float *w;
    uint8_t *pivot;
    int chunks;             // token chunks of the observe pass that scratch has room for
    size_t bytes;

    Workspace(const stepq_config *cfg, int n, uint8_t *base) {
        const size_t heads = (size_t)cfg->n_layers * cfg->n_value_heads;
        const size_t U = stepq_num_units(cfg), K1 = (size_t)cfg->n_candidates + 1;
        size_t o = 0;
        const auto take = [&](size_t nb) {
            uint8_t *p = base ? base + o : nullptr;
            o += up256(nb);
            return p;
        };
        omega_sum = (double *)take(heads * kD * sizeof(double));
        logret_sum = (double *)take(U * sizeof(double));
        acc = (double *)take(U * K1 * sizeof(double));
        w = (float *)take(heads * kD * sizeof(float));
        pivot = take(U);
        // About 16 observe CTAs per SM, within the size of n dense states of a layer.
        // (The bytes asked for do not depend on the device.)
        const size_t most = std::max<size_t>(1, 32 * (size_t)n / cfg->n_layers);
        chunks = base ? (int)std::min(most, (16 * (size_t)sm_count() + heads - 1) / heads) : 1;
        scratch = chunks > 1 ? (double *)(base + o) : nullptr;
        // The size is part of the interface, in what is asked for and in what is refused:
        // n slot ids, n dense states and n readouts of a layer, as when the replay went
        // through memory.
        take((size_t)n * sizeof(int32_t));
        take((size_t)n * cfg->n_value_heads * kN * sizeof(float));
        take((size_t)n * cfg->n_value_heads * kD * sizeof(float));
        bytes = o;
    }
};

stepq_status cuda_ok(cudaError_t e) { return e == cudaSuccess ? STEPQ_OK : STEPQ_ERR_CUDA; }

}  // namespace

extern "C" size_t stepq_calib_workspace_bytes(const stepq_config *cfg, int n) {
    if (validate_config(cfg, true) != STEPQ_OK || n <= 0) return 0;
    return Workspace(cfg, n, nullptr).bytes;
}

extern "C" stepq_status stepq_calibrate_from_trace(const stepq_config *cfg, int n, int T, int every,
                                                   const float *q, const float *k, const float *v,
                                                   const float *beta, const float *gate,
                                                   void *workspace, size_t workspace_bytes,
                                                   stepq_calib_result *out, stepq_stream_t stream) {
    stepq_status st = validate_config(cfg, true);
    if (st != STEPQ_OK) return st;
    if (n <= 0 || T <= 0 || every <= 0 || !q || !k || !v || !beta || !gate || !workspace || !out ||
        !out->omega || !out->mean_log_ret || !out->distortion || !out->pivot_mask)
        return STEPQ_ERR_ARG;
    if (((uintptr_t)workspace & 255) || ((uintptr_t)q & 15) || ((uintptr_t)k & 15) ||
        ((uintptr_t)v & 15) || ((uintptr_t)beta & 3) || ((uintptr_t)gate & 15))
        return STEPQ_ERR_ALIGN;
    Workspace ws(cfg, n, (uint8_t *)workspace);
    if (workspace_bytes < ws.bytes) return STEPQ_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int L = cfg->n_layers, Hv = cfg->n_value_heads;
    const bool rows = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    const size_t heads = (size_t)L * Hv, U = stepq_num_units(cfg), K1 = (size_t)cfg->n_candidates + 1;

    // Pass A: sums of g_{t,i}^2 (Sec. 4.1) and of log retention (Eq. calibration_lifetime).
    if ((st = cuda_ok(cudaMemsetAsync(ws.omega_sum, 0, heads * kD * sizeof(double), s))) != STEPQ_OK ||
        (st = cuda_ok(cudaMemsetAsync(ws.logret_sum, 0, U * sizeof(double), s))) != STEPQ_OK ||
        (st = launch_calib_observe(cfg, L, q, k, beta, gate, n * T, ws.omega_sum, ws.logret_sum, ws.scratch,
                                   ws.chunks, s)) != STEPQ_OK)
        return st;
    std::vector<double> osum(heads * kD), lsum(U);
    if ((st = cuda_ok(cudaMemcpyAsync(osum.data(), ws.omega_sum, osum.size() * sizeof(double),
                                      cudaMemcpyDeviceToHost, s))) != STEPQ_OK ||
        (st = cuda_ok(cudaMemcpyAsync(lsum.data(), ws.logret_sum, lsum.size() * sizeof(double),
                                      cudaMemcpyDeviceToHost, s))) != STEPQ_OK ||
        (st = cuda_ok(cudaStreamSynchronize(s))) != STEPQ_OK)
        return st;
    const double n_tok = (double)n * T;
    for (size_t e = 0; e < osum.size(); e++) out->omega[e] = (float)(osum[e] / n_tok);
    for (size_t u = 0; u < U; u++) out->mean_log_ret[u] = lsum[u] / n_tok;
    out->n_tokens = n * T;

    // Row-impact factors of the fit weights (footnote of Sec. 4.3).
    std::vector<float> w(heads * kD);
    if ((st = stepq_row_weights(cfg, out->omega, w.data())) != STEPQ_OK) return st;
    if ((st = cuda_ok(cudaMemcpyAsync(ws.w, w.data(), w.size() * sizeof(float), cudaMemcpyHostToDevice, s))) !=
        STEPQ_OK)
        return st;

    // Pass B: replay the FP32-state recurrence from zero in every layer and fit every
    // `every`-th state at each candidate width (Eqs. qwen_calibration_distortion,
    // kda_calibration_distortion); each sequence is one sample. The host forms the
    // lifetimes, which only need pass A, while the first replay runs.
    std::vector<double> life;
    const auto distortion_pass = [&](const uint8_t *pivot_rows, const int32_t *list, size_t count,
                                     double *dist) -> stepq_status {
        stepq_status e;
        if ((e = cuda_ok(cudaMemsetAsync(ws.acc, 0, U * K1 * sizeof(double), s))) != STEPQ_OK) return e;
        if ((e = launch_calib_replay(cfg, n, T, every, k, v, beta, gate, ws.w, pivot_rows, ws.acc, list, (int)count,
                                     s)) != STEPQ_OK)
            return e;
        if (life.empty()) life = lifetime_weights(cfg, out->mean_log_ret);
        const int n_samp = T / every * n;
        std::vector<double> acc(U * K1);
        if ((e = cuda_ok(cudaMemcpyAsync(acc.data(), ws.acc, acc.size() * sizeof(double),
                                         cudaMemcpyDeviceToHost, s))) != STEPQ_OK ||
            (e = cuda_ok(cudaStreamSynchronize(s))) != STEPQ_OK)
            return e;
        const double ns = n_samp > 0 ? n_samp : 1;
        for (size_t x = 0; x < acc.size(); x++) dist[x] = acc[x] / ns;
        out->n_samples = n_samp;
        return STEPQ_OK;
    };
    std::vector<double> d1(U * K1);
    if ((st = distortion_pass(nullptr, nullptr, heads, d1.data())) != STEPQ_OK) return st;
    if (out->distortion_stage1) std::memcpy(out->distortion_stage1, d1.data(), d1.size() * sizeof(double));
    if ((st = select_pivots(cfg, life, d1.data(), out->pivot_mask)) != STEPQ_OK) return st;
    // Row units: measure again with the chosen pivot rows kept in FP16. Only the heads that
    // have such rows fit differently; the others' figures stand. (102 pivots fall into 64 of
    // 128 heads: the second replay takes 2.4 ms, 4.2 ms over all heads.)
    std::vector<int32_t> list;
    for (size_t lh = 0; rows && lh < heads; lh++)
        if (std::memchr(out->pivot_mask + lh * kD, 1, kD)) list.push_back((int32_t)lh);
    if (list.empty()) {
        std::memcpy(out->distortion, d1.data(), d1.size() * sizeof(double));
        return STEPQ_OK;
    }
    int32_t *list_d = (int32_t *)ws.omega_sum;               // pass A's sums are on the host
    if ((st = cuda_ok(cudaMemcpyAsync(ws.pivot, out->pivot_mask, U, cudaMemcpyHostToDevice, s))) != STEPQ_OK ||
        (st = cuda_ok(cudaMemcpyAsync(list_d, list.data(), list.size() * sizeof(int32_t),
                                      cudaMemcpyHostToDevice, s))) != STEPQ_OK ||
        (st = distortion_pass(ws.pivot, list_d, list.size(), out->distortion)) != STEPQ_OK)
        return st;
    size_t at = 0;
    for (size_t lh = 0; lh < heads; lh++) {
        if (at < list.size() && (size_t)list[at] == lh) {
            at++;
            continue;
        }
        std::memcpy(out->distortion + lh * kD * K1, d1.data() + lh * kD * K1, kD * K1 * sizeof(double));
    }
    return STEPQ_OK;
}
