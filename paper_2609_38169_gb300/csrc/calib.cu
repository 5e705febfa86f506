// Calibration statistics on the device (App. A.3): row-impact scores
// omega_i = E[g_{t,i}^2] with g_t = A_t^T q_t = D_t (q_t - beta_t k_t (k_t^T q_t))
// (Sec. 4.1, Eq. kda_sensitivity) and the mean log retention ell_u
// (Eq. calibration_lifetime). Sums are kept in fp64; the caller divides.
//
// Bound by the fp64 pipe (two lanes a clock and SM): per entry a dot product term,
// g and g^2. The logarithms are taken of the product of four tokens' retentions, so
// that they cost a quarter of a log each.
#include "device.cuh"
#include "internal.h"

namespace stepq {

struct ObsArgs {
    const float *q, *k, *beta, *gate;      // [layers][n][..]
    int n, Hk, Hv, gate_per_row, chunk;
    double *omega, *logret;                // sums: [layers][Hv][128], [layers][Hv] or [layers][Hv][128]
    double *part;                          // chunk partials [chunks][layers][Hv][256], or null
};

// Adds log r of a run of retentions: the running product of up to four, then its
// log. Negative retentions (outside the gates' range) stay NaN.
struct LogSum {
    double sum = 0.0, prod = 1.0;
    int count = 0;
    __device__ __forceinline__ void add(float r) {
        prod *= r < 0.f ? nan("") : (double)r;
        if (++count == 4) flush();
    }
    __device__ __forceinline__ void flush() {
        if (count) sum += log(prod);
        prod = 1.0;
        count = 0;
    }
};

// One 128-thread CTA per (layer, value head, token chunk). Warp w takes tokens
// w, w + 4, ... of its chunk, lane l channels 4l..4l+3; the warps' sums meet in
// shared memory in warp order.
__global__ void __launch_bounds__(128) observe_kernel(ObsArgs a) {
    __shared__ double om_s[4][128], lr_s[4][128];
    const int lh = blockIdx.x, layer = lh / a.Hv, h = lh - layer * a.Hv;
    const int hk = h / (a.Hv / a.Hk), w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int t0 = blockIdx.y * a.chunk, t1 = min(a.n, t0 + a.chunk);
    double om[4] = {0, 0, 0, 0};
    LogSum lr[4];
    for (int t = t0 + w; t < t1; t += 4) {
        const size_t tok = (size_t)layer * a.n + t;
        const float4 q = ((const float4 *)&a.q[(tok * a.Hk + hk) * 128])[l];
        const float4 k = ((const float4 *)&a.k[(tok * a.Hk + hk) * 128])[l];
        const double beta = a.beta[tok * a.Hv + h];
        float4 d;
        if (a.gate_per_row) {
            d = ((const float4 *)&a.gate[(tok * a.Hv + h) * 128])[l];
        } else {
            d.x = d.y = d.z = d.w = a.gate[tok * a.Hv + h];
        }
        const double qd[4] = {q.x, q.y, q.z, q.w}, kd[4] = {k.x, k.y, k.z, k.w};
        const float df[4] = {d.x, d.y, d.z, d.w};
        double p = (qd[0] * kd[0] + qd[1] * kd[1]) + (qd[2] * kd[2] + qd[3] * kd[3]);
        for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
        const double bkq = beta * p;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const double g = (double)df[e] * (qd[e] - bkq * kd[e]);
            om[e] += g * g;
            if (a.gate_per_row || (l == 0 && e == 0)) lr[e].add(df[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {
        lr[e].flush();
        om_s[w][4 * l + e] = om[e];
        lr_s[w][4 * l + e] = lr[e].sum;
    }
    __syncthreads();
    const int i = threadIdx.x;
    const double o = ((om_s[0][i] + om_s[1][i]) + om_s[2][i]) + om_s[3][i];
    const double r = ((lr_s[0][i] + lr_s[1][i]) + lr_s[2][i]) + lr_s[3][i];
    if (a.part) {
        double *dst = a.part + ((size_t)blockIdx.y * gridDim.x + lh) * 256;
        dst[i] = o;
        dst[128 + i] = r;
        return;
    }
    a.omega[(size_t)lh * 128 + i] += o;
    if (a.gate_per_row) a.logret[(size_t)lh * 128 + i] += r;
    else if (i == 0) a.logret[lh] += r;
}

// The chunks' partials added in chunk order: one 128-thread CTA per (layer, head).
__global__ void __launch_bounds__(128) observe_sum_kernel(ObsArgs a, int chunks) {
    const size_t lh = blockIdx.x;
    const int i = threadIdx.x;
    double o = 0.0, r = 0.0;
    for (int c = 0; c < chunks; c++) {
        const double *p = a.part + ((size_t)c * gridDim.x + lh) * 256;
        o += p[i];
        r += p[128 + i];
    }
    a.omega[lh * 128 + i] += o;
    if (a.gate_per_row) a.logret[lh * 128 + i] += r;
    else if (i == 0) a.logret[lh] += r;
}

// Sums over the n tokens of `layers` layers, whose inputs, omega and logret slices
// follow each other. scratch (or null): room for `chunks` chunks of partials; a
// layer's tokens are split over that many CTAs so that few heads still fill the chip.
stepq_status launch_calib_observe(const stepq_config *cfg, int layers, const float *q, const float *k,
                                  const float *beta, const float *gate, int n, double *omega_sum,
                                  double *logret_sum, double *scratch, int chunks, cudaStream_t s) {
    ObsArgs a{};
    a.q = q; a.k = k; a.beta = beta; a.gate = gate;
    a.n = n;
    a.Hk = cfg->n_key_heads;
    a.Hv = cfg->n_value_heads;
    a.gate_per_row = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    a.omega = omega_sum;
    a.logret = logret_sum;
    if (!scratch || chunks > n) chunks = scratch ? n : 1;
    a.chunk = (n + chunks - 1) / chunks;
    chunks = (n + a.chunk - 1) / a.chunk;
    a.part = chunks > 1 ? scratch : nullptr;
    const unsigned heads = (unsigned)((size_t)layers * cfg->n_value_heads);
    observe_kernel<<<dim3(heads, (unsigned)chunks), 128, 0, s>>>(a);
    if (chunks > 1) observe_sum_kernel<<<heads, 128, 0, s>>>(a, chunks);
    return cudaGetLastError() == cudaSuccess ? STEPQ_OK : STEPQ_ERR_CUDA;
}

}  // namespace stepq
