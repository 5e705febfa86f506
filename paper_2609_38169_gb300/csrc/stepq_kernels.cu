// Row-unit (KDA) pool pack/unpack and the calibration distortion kernel
// (sm_103a), and the dispatch of the decode step: head units (GDN) run the
// pipelined kernel of heads.cu, row units the one of rows.cu.
//
// A 256-thread CTA holds one (slot, value head) tile in registers, fits the
// dual-axis scales and writes the packed segment (App. C.3 steps 4-6).
//
// Numerical contract (shared with the CPU oracle, which restates it in fp64):
// the tile X is fp32; r_i = fp16(clamp(sqrt(m_i) * w_i^(-1/2), 2^-14, 65504));
// rho_i = fp32(1/(r_i zs_i)); every code decision is the nearest integer (ties to
// even) to the exact product fp32(X rho_i) gamma_j with gamma_j = fp32(1/c_j), one
// fused multiply-add with 1.5 * 2^23;
// c is fitted from the clip-free start
// max_i fp32(fp32(|X_ij| rho_i) / qmax_i) by `fit_iters` fixed-code
// least-squares updates.
#include "async.cuh"
#include "device.cuh"
#include "internal.h"
#include "tile.cuh"

namespace stepq {

// ---------------------------------------------------------------- smem layout
// Scratch of the fit. Per-column values and the cross-warp partials are kept in
// 16-byte groups whose low two index bits are swizzled by the lane's column
// group (cpos), so that the 8 lanes of a quarter warp, which address columns 16
// apart, hit 8 different bank groups instead of 2.
constexpr int kFitRed = 0;                                   // float [2][8][128]
constexpr int kFitCol = kFitRed + 2 * 8 * 128 * 4;           // float [2][128]: c_j, 1 / c_j
constexpr int kFitRow = kFitCol + 2 * 128 * 4;               // float [5][128]: w^2, w^-1/2, rho, r, 1 / r
constexpr int kFitBits = kFitRow + 5 * 128 * 4;              // int [128] widths
constexpr int kFitWarp = kFitBits + 128 * 4;                 // float [8]
constexpr int kFitBytes = kFitWarp + 64;

struct FitSmem {
    float *red, *colC, *colG, *w2, *wis, *rho, *rr, *rho1, *warp;
    int *rbits;
    __device__ __forceinline__ explicit FitSmem(uint8_t *s) {
        red = (float *)(s + kFitRed);
        colC = (float *)(s + kFitCol);
        colG = colC + 128;
        w2 = (float *)(s + kFitRow);
        wis = w2 + 128;
        rho = w2 + 256;
        rr = w2 + 384;
        rho1 = w2 + 512;
        rbits = (int *)(s + kFitBits);
        warp = (float *)(s + kFitWarp);
    }
};

// 16-byte group e (0..3) of the 16 columns of group cg, and the position of column c.
__device__ __forceinline__ int cgroup(int cg, int e) { return 4 * cg + (e ^ (cg >> 1)); }
__device__ __forceinline__ int cpos(int c) { return 4 * cgroup(c >> 4, (c >> 2) & 3) + (c & 3); }

__device__ __forceinline__ int qmax_of(int b) { return (1 << (b - 1)) - 1; }

// Pairs (2e, 2e+1) of the lane's 16 values of a per-column vector, two at a time.
__device__ __forceinline__ void col_pairs(const float *v, const Lane &L, int e, uint64_t &lo, uint64_t &hi) {
    const uint4 q = *(const uint4 *)&v[4 * cgroup(L.cg, e)];
    lo = u2pair(q.x, q.y);
    hi = u2pair(q.z, q.w);
}

// Reduce-scatter of 16 per-column partials over the 4 lanes of a column group
// into the warp's row of `red` (the 8 warps' rows are summed by the column's owner).
template <bool MAX>
__device__ __forceinline__ void columns_to_red(const Lane &L, const float (&acc)[16], float *red) {
    const auto join = [](float x, float y) { return MAX ? fmaxf(x, y) : x + y; };
    float h8[8], h4[4];
    const bool hi16 = (L.rs & 2) != 0, hi8 = (L.rs & 1) != 0;
#pragma unroll
    for (int t = 0; t < 8; t++)
        h8[t] = join(hi16 ? acc[8 + t] : acc[t],
                     __shfl_xor_sync(0xffffffffu, hi16 ? acc[t] : acc[8 + t], 16));
#pragma unroll
    for (int t = 0; t < 4; t++)
        h4[t] = join(hi8 ? h8[4 + t] : h8[t], __shfl_xor_sync(0xffffffffu, hi8 ? h8[t] : h8[4 + t], 8));
    *(float4 *)&red[L.warp * 128 + 4 * cgroup(L.cg, L.rs)] = make_float4(h4[0], h4[1], h4[2], h4[3]);
}

// One fixed-code pass (App. C.1): the thread's sums of w_i^2 v_ij X_ij and
// w_i^2 v_ij^2 over its 4 rows, v_ij = r_i zs_i rne(X_ij rho_i gamma_j), per column
// pair. CLIP clamps the codes to +-qmax and leaves pivot rows out by a select;
// without it no code can exceed qmax, all values are finite and a pivot row adds
// exact zeros (rho = r = 0).
template <bool CLIP>
__device__ __forceinline__ void ls_partials(const Lane &L, const FitSmem &S, const uint64_t (&x)[4][8],
                                            int unit_rows, uint64_t (&n)[8], uint64_t (&d)[8]) {
    const uint64_t M2 = f2s(kMagic), nM2 = f2s(-kMagic);
#pragma unroll
    for (int e = 0; e < 8; e++) n[e] = d[e] = 0;
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int i = L.row(t), bits = S.rbits[i];
        const bool pivot = bits == kPivot;
        const float zs = unit_rows && !pivot ? (float)(1 << (8 - bits)) : 1.0f;
        const float lim = pivot ? 0.f : (float)qmax_of(bits);
        const uint64_t rho = f2s(S.rho[i]), rz = f2s(S.rr[i] * zs), w2 = f2s(S.w2[i]);
#pragma unroll
        for (int e4 = 0; e4 < 4; e4++) {
            uint64_t g[2];
            col_pairs(S.colG, L, e4, g[0], g[1]);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int e = 2 * e4 + h;
                uint64_t q = fadd2(ffma2(fmul2(x[t][e], rho), g[h], M2), nM2);   // rne of the product
                if (CLIP) q = clamp2(q, lim);
                const uint64_t v = fmul2(rz, q);                                 // v_ij = r_i z_ij
                const uint64_t nn = ffma2(w2, fmul2(v, x[t][e]), n[e]);
                const uint64_t dd = ffma2(w2, fmul2(v, v), d[e]);
                n[e] = CLIP && pivot ? n[e] : nn;
                d[e] = CLIP && pivot ? d[e] : dd;
            }
        }
    }
}

// Key-Row-Aware Dual-axis Fitting of the register tile x (Sec. 4.3, App. C.1), in two
// parts: the row factors with the columns' maxima, and the column factors.
// x[t][e] holds columns 16cg + 2e, 2e + 1 of row 16w + 4t + rs. msum[t]: sum_j
// |X_ij| of the thread's rows; row widths come from S.rbits.
//
// Bound by instruction issue (about 60% of it fp32 arithmetic), so the passes run
// on f32x2 column pairs, and the clamps, two min/max per code, only when the clip-free
// start was capped, the state holds a non-finite value or (last pass and final
// codes) some max_i |X'_ij| mu_i / c_j reaches 1 + 1/(2 qmax).

// Row factors r_i = m_i^(1/2) w_i^(-1/2) into S.rr (and the page, or null, which must no
// longer be read), rho_i = 1 / (r_i zs_i) into S.rho (0 for pivot rows). Thread tid < 128
// returns column tid's clip-free start c0_j = max_i fp32(fp32(|X_ij| rho_i) mu_i),
// mu_i = 1 / qmax_i; ANY leaves out the widths (mu_i = zs_i = 1, rho_i into S.rho1): a head
// of one width has that maximum and those rho_i times a power of two, and the start is
// rounded once more by mu (rounding keeps the order). `wild`: a non-finite row sum.
template <bool ANY>
__device__ __forceinline__ float fit_rows(const Lane &L, const FitSmem &S, const uint64_t (&x)[4][8],
                                          const float (&msum)[4], int unit_rows, uint8_t *page, bool &wild) {
    wild = false;
    float acc[16];
#pragma unroll
    for (int j = 0; j < 16; j++) acc[j] = 0.f;
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int i = L.row(t), bits = S.rbits[i];
        float rf = 0.f, rho = 0.f, zs = 1.f, mu = 0.f;
        if (bits != kPivot) {
            const float m = msum[t] * (1.0f / 128.0f);
            rf = __half2float(__float2half_rn(
                fminf(fmaxf(__fmul_rn(sqrtf(m), S.wis[i]), kF16Min), kF16Max)));
            if (!ANY) {
                zs = unit_rows ? (float)(1 << (8 - bits)) : 1.0f;
                mu = __frcp_rn((float)qmax_of(bits));
            }
            rho = __frcp_rn(rf * zs);
        }
        wild = wild || !(msum[t] <= 3.4028235e38f);
        if (L.cg == 0) {
            S.rr[i] = rf;
            (ANY ? S.rho1 : S.rho)[i] = rho;
            if (page) ((uint16_t *)page)[i] = f16_bits(rf);
        }
        const uint64_t rho2 = f2s(rho), mu2 = f2s(mu);
#pragma unroll
        for (int e = 0; e < 8; e++) {
            uint64_t z = fmul2(x[t][e], rho2);
            if (!ANY) z = fmul2(z, mu2);
            acc[2 * e] = fmaxf(acc[2 * e], fabsf(f2lo(z)));
            acc[2 * e + 1] = fmaxf(acc[2 * e + 1], fabsf(f2hi(z)));
        }
    }
    columns_to_red<true>(L, acc, S.red);
    __syncthreads();
    const int cp = cpos(L.tid & 127);
    float cm = 0.f;
    if (L.tid < 128) {
        cm = S.red[cp];
#pragma unroll
        for (int wv = 1; wv < 8; wv++) cm = fmaxf(cm, S.red[wv * 128 + cp]);
    }
    return cm;
}

// Column factors from the starts cm (thread tid < 128: column tid): S.colC the stored
// (FP16-rounded) ones, S.colG their reciprocals, the page (or null) the FP16 c. Returns
// whether a code may exceed qmax with these scales (uniform over the CTA).
__device__ __forceinline__ bool fit_columns(const Lane &L, const FitSmem &S, const uint64_t (&x)[4][8], float cm,
                                            bool wild, int unit_rows, uint8_t *page, int fit_iters) {
    const int cp = cpos(L.tid & 127);
    float acc[16], cc = 0.f;
    if (L.tid < 128) {
        wild = wild || cm > kF16Max;                         // start capped: codes may clip
        cc = fminf(fmaxf(cm, kF16Min), kF16Max);
        S.colG[cp] = __frcp_rn(cc);
    }
    wild = __syncthreads_or(wild);
    // Fixed-code least-squares updates over the non-pivot rows.
    bool clip = wild;
    for (int it = 0; it < fit_iters; it++) {
        {
            uint64_t n[8], d[8];
            if (it > 0 || wild) ls_partials<true>(L, S, x, unit_rows, n, d);
            else ls_partials<false>(L, S, x, unit_rows, n, d);
#pragma unroll
            for (int e = 0; e < 8; e++) {
                acc[2 * e] = f2lo(n[e]);
                acc[2 * e + 1] = f2hi(n[e]);
            }
            columns_to_red<false>(L, acc, S.red);
#pragma unroll
            for (int e = 0; e < 8; e++) {
                acc[2 * e] = f2lo(d[e]);
                acc[2 * e + 1] = f2hi(d[e]);
            }
            columns_to_red<false>(L, acc, S.red + 8 * 128);
        }
        __syncthreads();
        if (L.tid < 128) {
            float num = S.red[cp], den = S.red[8 * 128 + cp];
#pragma unroll
            for (int wv = 1; wv < 8; wv++) {
                num += S.red[wv * 128 + cp];
                den += S.red[(8 + wv) * 128 + cp];
            }
            if (den > 0.f) cc = fminf(fmaxf(__fdiv_rn(num, den), kF16Min), kF16Max);
            if (it + 1 < fit_iters) {
                S.colG[cp] = __frcp_rn(cc);
            } else {                                          // storage precision of c
                const float cf = __half2float(__float2half_rn(cc)), g = __frcp_rn(cf);
                S.colC[cp] = cf;
                S.colG[cp] = g;
                if (page) ((uint16_t *)(page + 256))[L.tid] = f16_bits(cf);
                clip = clip || __fmul_rn(cm, g) >= (1.0f + 0.5f / 127.0f) * 0.999999f;
            }
        }
        clip = __syncthreads_or(clip);
    }
    return clip;
}

// Final codes rne(X_ij rho_i gamma_j) of the thread's 16 columns of a row, as the
// float bit patterns 0x4B400000 | (q + 2^(b-1)); with `clip` clamped to +-qmax.
__device__ __forceinline__ void row_codes(const Lane &L, const FitSmem &S, const uint64_t (&x)[8], float rho,
                                          int bits, bool clip, uint32_t (&f)[16]) {
    const float mb = kMagic + (float)(1 << (bits - 1)), lim = (float)qmax_of(bits);
    const uint64_t rho2 = f2s(rho), mb2 = f2s(mb), lo = f2s(mb - lim), hi = f2s(mb + lim);
#pragma unroll
    for (int e4 = 0; e4 < 4; e4++) {
        uint64_t g[2];
        col_pairs(S.colG, L, e4, g[0], g[1]);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            uint64_t u = ffma2(fmul2(x[2 * e4 + h], rho2), g[h], mb2);
            if (clip) u = clamp2r(u, lo, hi);
            f[4 * e4 + 2 * h] = (uint32_t)u;
            f[4 * e4 + 2 * h + 1] = (uint32_t)(u >> 32);
        }
    }
}

// Sixteen biased codes of width B packed LSB-first: the plain sum of the shifted bit
// patterns minus the shifted constants (mod 2^32), one shift-add per code.
template <int B>
__device__ __forceinline__ void pack_biased(const uint32_t (&f)[16], uint32_t (&wd)[B / 2]) {
    if (B == 8) {
#pragma unroll
        for (int t = 0; t < 4; t++)
            wd[t] = __byte_perm(__byte_perm(f[4 * t], f[4 * t + 1], 0x0040),
                                __byte_perm(f[4 * t + 2], f[4 * t + 3], 0x0040), 0x5410);
        return;
    }
#pragma unroll
    for (int k = 0; k < B / 2; k++) wd[k] = 0u - pack_bias(B, k);
#pragma unroll
    for (int r = 0; r < 16; r++) {
        const int p = r * B, k = p >> 5, s = p & 31;
        wd[k] += f[r] << s;
        if (s + B > 32) wd[k + 1] += f[r] >> (32 - s);
    }
}

// Packs the tile with the stored scales into the staged page (App. C.3 step 6);
// roff: payload offset of each row.
__device__ __forceinline__ void pack_page(const Lane &L, const FitSmem &S, uint8_t *page, const int *roff,
                                          const uint64_t (&x)[4][8], bool clip) {
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const int i = L.row(t), bits = S.rbits[i];
        uint8_t *row = page + roff[i];
        if (bits == kPivot) {
            uint32_t wd[8];
#pragma unroll
            for (int e = 0; e < 8; e++)
                wd[e] = (uint32_t)f16_bits(f16_round_sat(f2lo(x[t][e]))) |
                        ((uint32_t)f16_bits(f16_round_sat(f2hi(x[t][e]))) << 16);
            uint4 *p = (uint4 *)(row + 32 * L.cg);
            p[0] = make_uint4(wd[0], wd[1], wd[2], wd[3]);
            p[1] = make_uint4(wd[4], wd[5], wd[6], wd[7]);
            continue;
        }
        uint32_t f[16];
        row_codes(L, S, x[t], S.rho[i], bits, clip, f);
        switch (bits) {
        case 2: {
            uint32_t wd[1];
            pack_biased<2>(f, wd);
            *(uint32_t *)(row + 4 * L.cg) = wd[0];
        } break;
        case 4: {
            uint32_t wd[2];
            pack_biased<4>(f, wd);
            *(uint2 *)(row + 8 * L.cg) = make_uint2(wd[0], wd[1]);
        } break;
        case 6: {
            uint32_t wd[3];
            pack_biased<6>(f, wd);
            uint32_t *p = (uint32_t *)(row + 12 * L.cg);
            p[0] = wd[0];
            p[1] = wd[1];
            p[2] = wd[2];
        } break;
        default: {
            uint32_t wd[4];
            pack_biased<8>(f, wd);
            *(uint4 *)(row + 16 * L.cg) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
        } break;
        }
    }
}

// The thread's part of a dense state (row stride 128) and its rows' sums of |X_ij|.
__device__ __forceinline__ void load_dense(const Lane &L, const float *X, uint64_t (&x)[4][8], float (&msum)[4]) {
#pragma unroll
    for (int t = 0; t < 4; t++) {
        const float4 *src = (const float4 *)(X + L.row(t) * 128 + L.col0());
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const float4 f = src[e];
            x[t][2 * e] = f2(f.x, f.y);
            x[t][2 * e + 1] = f2(f.z, f.w);
            s += fabsf(f.x) + fabsf(f.y) + fabsf(f.z) + fabsf(f.w);
        }
        msum[t] = row_allreduce(s);
    }
}

// ---------------------------------------------------------- quantize / dequantize
struct PoolArgs {
    uint8_t *pool;
    uint64_t stride;
    int pool_slots;
    const int32_t *slots;
    LayerTables tab;
    int heads, items;         // heads per batch entry (one layer's or all layers'); item = entry * heads + head
    int fit_iters;
    float *states;            // [B][..][heads][128][128]
    size_t state_stride_b;    // floats between consecutive batch entries
    unsigned int *err;
};

// Pack of dense states, persistent, two CTAs per SM. A state is 64 KB and its fit is
// bound by instruction issue (about 8,000 warp instructions an item), so the loads
// have to run under it: once an item's tile is in registers its shared-memory copy is
// refilled with the next item's state (16-byte cp.async, swizzled as cgroup), and the
// page leaves by a bulk store. One CTA per item with plain loads exposed their
// latency (stalled on it 18% of the time at 24% occupancy): 4096 heads at 6 bits
// took 143 us, 109 us now (47 us at the copy rate of HBM).
constexpr int kQTile = 0;                                    // float [128][128], 16-byte groups swizzled
constexpr int kQPage = kN * 4;
constexpr int kQFit = kQPage + (int)kMaxHeadBytes;
constexpr int kQRoff = kQFit + kFitBytes;                    // int [128]
constexpr int kQSmem = kQRoff + 128 * 4;

__global__ void __launch_bounds__(kThreads, 2) quantize_kernel(PoolArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const Lane L;
    float *tile = (float *)(smem + kQTile);
    uint8_t *page = smem + kQPage;
    const FitSmem S(smem + kQFit);
    int *roff = (int *)(smem + kQRoff);
    const int tid = L.tid;
    griddep_wait();
    griddep_launch();
    const auto slot_of = [&](int item) { return item < a.items ? a.slots[item / a.heads] : -1; };
    const auto ok = [&](int slot) { return slot >= 0 && slot < a.pool_slots; };
    const auto start = [&](int item) {
        const int b = item / a.heads, h = item - b * a.heads;
        const float4 *X = (const float4 *)(a.states + (size_t)b * a.state_stride_b + (size_t)h * kN);
#pragma unroll
        for (int j = 0; j < 16; j++) {
            const int e = tid + j * kThreads, row = e >> 5, f = e & 31;
            cp_async16(&tile[row * 128 + 4 * cgroup(f >> 2, f & 3)], X + e);
        }
    };
    // Row tables of an item's head: one row per thread of the first half.
    int fbits = 0, froff = 0;
    float fw2 = 0.f, fwis = 0.f;
    const auto fetch = [&](int item) {
        if (tid < 128) {
            const int h = item % a.heads;
            fbits = a.tab.row_bits[h * 128 + tid];
            froff = (int)a.tab.row_off[h * 128 + tid];
            fw2 = a.tab.w2[h * 128 + tid];
            fwis = a.tab.wis[h * 128 + tid];
        }
    };
    int slot = slot_of(blockIdx.x);
    if (ok(slot)) {
        start(blockIdx.x);
        fetch(blockIdx.x);
    }
    for (int item = blockIdx.x; item < a.items; item += gridDim.x) {
        const int next = item + gridDim.x, nslot = slot_of(next);
        if (!ok(slot)) {                                      // uniform over the CTA
            if (tid == 0) raise_error(a.err, STEPQ_ERR_SLOT_RANGE);
            if (ok(nslot)) {
                start(next);
                fetch(next);
            }
            slot = nslot;
            continue;
        }
        if (tid < 128) {
            S.rbits[tid] = fbits;
            roff[tid] = froff;
            S.w2[tid] = fw2;
            S.wis[tid] = fwis;
        }
        cp_async_wait_all();
        __syncthreads();
        uint64_t x[4][8];
        float msum[4];
#pragma unroll
        for (int t = 0; t < 4; t++) {
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const float4 f = *(const float4 *)&tile[L.row(t) * 128 + 4 * cgroup(L.cg, e)];
                x[t][2 * e] = f2(f.x, f.y);
                x[t][2 * e + 1] = f2(f.z, f.w);
                s += fabsf(f.x) + fabsf(f.y) + fabsf(f.z) + fabsf(f.w);
            }
            msum[t] = row_allreduce(s);
        }
        if (tid == 0) bulk_wait_read_all();                   // the previous page has left
        __syncthreads();
        if (ok(nslot)) {
            start(next);
            fetch(next);
        }
        bool wild;
        const float cm = fit_rows<false>(L, S, x, msum, 1, page, wild);
        const bool clip = fit_columns(L, S, x, cm, wild, 1, page, a.fit_iters);
        pack_page(L, S, page, roff, x, clip);
        fence_async_smem();
        __syncthreads();
        if (tid == 0) {
            const int h = item % a.heads;
            bulk_store(a.pool + (uint64_t)slot * a.stride + a.tab.head_off[h], page, a.tab.head_bytes[h]);
            bulk_commit();
        }
        slot = nslot;
    }
    if (tid == 0) bulk_wait_all();
}

// Unpack, one CTA per (slot, head) and bound by the 64 KB it writes. Warp w takes rows
// 16w..16w+15 and lane l columns 4l..4l+3, so that a row's width is uniform over the
// warp, its codes are read straight from the page and its 512 bytes leave as one
// store instruction. (Staging the page in shared memory with 16 columns of a row per
// thread wrote in 16-byte pieces 64 bytes apart and waited for the staging: 88 us for
// 4096 heads at 6 bits, 51 us now; 47 us at the copy rate of HBM.)
__global__ void __launch_bounds__(kThreads, 4) dequantize_kernel(PoolArgs a) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int b = blockIdx.x / a.heads, h = blockIdx.x - b * a.heads;
    griddep_wait();
    griddep_launch();
    const int slot = a.slots[b];
    if (slot < 0 || slot >= a.pool_slots) {
        if (threadIdx.x == 0) raise_error(a.err, STEPQ_ERR_SLOT_RANGE);
        return;
    }
    const uint8_t *page = a.pool + (uint64_t)slot * a.stride + a.tab.head_off[h];
    float *out = a.states + (size_t)b * a.state_stride_b + (size_t)h * kN;
    // Lanes 0..15: width, payload offset and r_i zs_i (exact) of the warp's rows.
    int tbits = 0, toff = 0;
    float trz = 0.f;
    if (l < 16) {
        const int i = 16 * w + l;
        tbits = a.tab.row_bits[h * 128 + i];
        toff = (int)a.tab.row_off[h * 128 + i];
        const float r = f16_val(((const uint16_t *)page)[i]);
        if (tbits != kPivot) trz = r * (float)(1 << (8 - tbits));
    }
    const uint2 c4 = ((const uint2 *)(page + 256))[l];
    const uint64_t c01 = f2(f16_val((uint16_t)(c4.x & 0xFFFFu)), f16_val((uint16_t)(c4.x >> 16)));
    const uint64_t c23 = f2(f16_val((uint16_t)(c4.y & 0xFFFFu)), f16_val((uint16_t)(c4.y >> 16)));
#pragma unroll
    for (int r0 = 0; r0 < 16; r0 += 8) {
        // The words that hold the lane's 4b bits of eight rows (its first byte is
        // l b / 2; an FP16 row has two whole words). The second word is read only
        // where the lane's bits reach it, so no read passes the row.
        uint32_t w0[8], w1[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int bits = __shfl_sync(0xffffffffu, tbits, r0 + u), off = __shfl_sync(0xffffffffu, toff, r0 + u);
            const int at = (l * bits) >> 1;
            const uint32_t *p = (const uint32_t *)(page + off + (at & ~3));
            w0[u] = p[0];
            w1[u] = 8 * (at & 3) + 4 * bits > 32 ? p[1] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int bits = __shfl_sync(0xffffffffu, tbits, r0 + u);
            const float rz = __shfl_sync(0xffffffffu, trz, r0 + u);
            float4 v;
            if (bits == kPivot) {
                v = make_float4(f16_val((uint16_t)(w0[u] & 0xFFFFu)), f16_val((uint16_t)(w0[u] >> 16)),
                                f16_val((uint16_t)(w1[u] & 0xFFFFu)), f16_val((uint16_t)(w1[u] >> 16)));
            } else {
                const uint32_t s = __funnelshift_r(w0[u], w1[u], 8 * (((l * bits) >> 1) & 3)), m = (1u << bits) - 1u;
                const uint64_t off = f2s(-(kMagic + (float)(1 << (bits - 1)))), rz2 = f2s(rz);
                // q is exact, r c zs is exact (22 bits), their product rounds once
                const uint64_t q01 = fadd2(u2pair(and_or(s, m, kMagicBits), and_or(s >> bits, m, kMagicBits)), off);
                const uint64_t q23 =
                    fadd2(u2pair(and_or(s >> (2 * bits), m, kMagicBits), and_or(s >> (3 * bits), m, kMagicBits)), off);
                const uint64_t v01 = fmul2(fmul2(rz2, c01), q01), v23 = fmul2(fmul2(rz2, c23), q23);
                v = make_float4(f2lo(v01), f2hi(v01), f2lo(v23), f2hi(v23));
            }
            *(float4 *)(out + (16 * w + r0 + u) * 128 + 4 * l) = v;
        }
    }
}

// ------------------------------------------------------ calibration distortion
// A reference state head fitted at every candidate width with the codec above
// (uniform over the head; pivot rows kept in FP16 and out of the column fit), and
// its reconstruction errors (Eqs. qwen_calibration_distortion,
// kda_calibration_distortion). add(k, i, e): row units, the mean error of key row i
// at candidate k; add(k, 0, e): head units, the weighted mean over the head (by one
// thread). S.w2 and S.wis hold the head's weights; `piv` its pivot rows or null.
struct FitCands {
    int unit_rows, n_cand, fit_iters;
    int cands[4];
};

template <class Add>
__device__ __forceinline__ void distortion_of(const Lane &L, const FitSmem &S, const uint64_t (&x)[4][8],
                                              const float (&msum)[4], const uint8_t *piv, const FitCands &a,
                                              const Add &add) {
    const int K1 = a.n_cand + 1;
    // The row factors and the columns' maxima serve every candidate (formed anew for each
    // of three, the four-layer model's calibration took 12.0 ms; 11.0 ms now).
    if (L.tid < 128) S.rbits[L.tid] = piv && piv[L.tid] ? kPivot : a.cands[0];
    __syncthreads();
    bool wild;
    const float top = fit_rows<true>(L, S, x, msum, a.unit_rows, nullptr, wild);
    for (int k = 0; k < K1; k++) {
        const bool fp16_col = (k == a.n_cand);
        const int b = fp16_col ? kPivot : a.cands[k];
        const float step = fp16_col || !a.unit_rows ? 1.f : 1.0f / (float)(1 << (8 - b));
        if (L.tid < 128) {
            S.rbits[L.tid] = piv && piv[L.tid] ? kPivot : b;
            S.rho[L.tid] = S.rho1[L.tid] * step;              // 0 stays 0 for a pivot row
        }
        __syncthreads();
        bool clip = false;
        if (!fp16_col) {
            const float cm = __fmul_rn(top * step, __frcp_rn((float)qmax_of(b)));
            clip = fit_columns(L, S, x, cm, wild, a.unit_rows, nullptr, a.fit_iters);
        }
        float head_err = 0.f;
#pragma unroll
        for (int t = 0; t < 4; t++) {
            const int i = L.row(t);
            const int bits = S.rbits[i];
            float e = 0.f;
            if (bits == kPivot) {
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const float x0 = f2lo(x[t][j]), x1 = f2hi(x[t][j]);
                    const float d0 = f16_round_sat(x0) - x0, d1 = f16_round_sat(x1) - x1;
                    e = fmaf(d0, d0, e);
                    e = fmaf(d1, d1, e);
                }
            } else {
                const float lim = (float)qmax_of(bits);
                const uint64_t zs = f2s(a.unit_rows ? (float)(1 << (8 - bits)) : 1.0f);
                const uint64_t rho = f2s(S.rho[i]), rr = f2s(S.rr[i]);
                const uint64_t M2 = f2s(kMagic), nM2 = f2s(-kMagic), m1 = f2s(-1.0f);
#pragma unroll
                for (int e4 = 0; e4 < 4; e4++) {
                    uint64_t g[2], c[2];
                    col_pairs(S.colG, L, e4, g[0], g[1]);
                    col_pairs(S.colC, L, e4, c[0], c[1]);
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        const uint64_t xv = x[t][2 * e4 + h];
                        uint64_t q = fadd2(ffma2(fmul2(xv, rho), g[h], M2), nM2);
                        if (clip) q = clamp2(q, lim);
                        const uint64_t rec = fmul2(fmul2(rr, c[h]), fmul2(zs, q));
                        const uint64_t d = ffma2(xv, m1, rec);                  // rec - x
                        e = fmaf(f2lo(d), f2lo(d), e);
                        e = fmaf(f2hi(d), f2hi(d), e);
                    }
                }
            }
            e = row_allreduce(e);
            if (a.unit_rows) {
                if (L.cg == 0) add(k, i, (double)e / 128.0);
            } else {
                head_err += S.w2[i] * e;
            }
        }
        if (!a.unit_rows) {
            // rows of one lane group share head_err; take it once per group
            float v = (L.cg == 0) ? head_err : 0.f;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (L.lane == 0) S.warp[L.warp] = v;
            __syncthreads();
            if (L.tid == 0) {
                double sum = 0.0;
                for (int wv = 0; wv < 8; wv++) sum += S.warp[wv];
                add(k, 0, sum / (double)kN);
            }
        }
        __syncthreads();
    }
}

// One CTA per (sample, head).
struct DistArgs {
    const float *states;          // [n][Hv][128][128]
    const float *w;               // [Hv][128] of the layer
    const uint8_t *pivot_rows;    // [Hv][128] of the layer, or null
    double *acc;                  // head: [Hv][K+1]; row: [Hv*128][K+1] (layer slice)
    int Hv;
    FitCands fit;
};

__device__ __forceinline__ void load_weights(const Lane &L, const FitSmem &S, const float *w) {
    if (L.tid < 128) {
        const float wv = w[L.tid];
        S.w2[L.tid] = __fmul_rn(wv, wv);
        S.wis[L.tid] = __frsqrt_rn(wv);
    }
}

__global__ void __launch_bounds__(kThreads, 2) distortion_kernel(DistArgs a) {
    __shared__ __align__(16) uint8_t smem[kFitBytes];
    const Lane L;
    const FitSmem S(smem);
    const int s = blockIdx.x / a.Hv, h = blockIdx.x - s * a.Hv;
    const int K1 = a.fit.n_cand + 1;
    load_weights(L, S, a.w + h * 128);
    uint64_t x[4][8];
    float msum[4];
    load_dense(L, a.states + ((size_t)s * a.Hv + h) * kN, x, msum);
    const size_t rows = a.fit.unit_rows ? 128 : 1;
    distortion_of(L, S, x, msum, a.pivot_rows ? a.pivot_rows + h * 128 : nullptr, a.fit,
                  [&](int k, int i, double e) { atomicAdd(&a.acc[(h * rows + i) * K1 + k], e); });
}

// ------------------------------------------------- calibration replay (App. A.3)
// The FP32 recurrence of one (layer, sequence, value head) from a zero state over T
// tokens, with every `every`-th state fitted in place at each candidate width: one
// CTA carries the state in registers for all tokens, so a token costs one CTA
// barrier and about 200 instructions a thread instead of a launch and two passes of
// the state over memory, and the layers run side by side. The arithmetic and its
// order are the FP32 decode kernel's (fp32.cu): warp w owns key rows 16w..16w+15,
// lane l columns 4l..4l+3; the eight warps' retrieval partials are summed in warp
// order, by every warp for itself. A sampled state goes through shared memory into
// the fit's tile mapping (the replay's registers are reloaded from there).
// Bound by the fits (three candidate widths plus FP16: about nine tenths of the
// instructions at one sample in 8 tokens). 4 layers x 8 sequences x 32 heads, 256
// tokens, 32 samples: 4.2 ms a pass over all heads, against about 28 ms of per-token launches.
struct ReplayArgs {
    const float *k, *v, *beta, *gate;   // trace [L][T][n][..]
    const float *w;                     // [L][Hv][128]
    const uint8_t *pivot_rows;          // [L][Hv][128] or null
    double *acc;                        // [L][Hv or Hv*128][K+1]
    const int32_t *heads;               // the heads to replay, layer * Hv + head, or null: all
    int n_heads, n, T, Hk, Hv, every, gate_per_row;
    FitCands fit;
};

constexpr int kRpTile = 0;                                   // float [128][128] (16-byte groups swizzled)
constexpr int kRpRed = kRpTile + kN * 4;                     // float [2][8][128]
constexpr int kRpRowA = kRpRed + 2 * 8 * 128 * 4;            // float4 [3][128]: d d k k
constexpr int kRpRowB = kRpRowA + 3 * 128 * 16;              // float2 [3][128]: beta k, twice
constexpr int kRpV = kRpRowB + 3 * 128 * 8;                  // float [3][128]
constexpr int kRpFit = kRpV + 3 * 128 * 4;
constexpr int kRpAcc = (kRpFit + kFitBytes + 15) / 16 * 16;  // double [128][5]
constexpr int kRpSmem = kRpAcc + 128 * 5 * 8;

__global__ void __launch_bounds__(kThreads, 2) replay_kernel(ReplayArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const Lane L;
    const FitSmem S(smem + kRpFit);
    float *tile = (float *)(smem + kRpTile), *red = (float *)(smem + kRpRed), *vs = (float *)(smem + kRpV);
    float4 *rowA = (float4 *)(smem + kRpRowA);
    float2 *rowB = (float2 *)(smem + kRpRowB);
    double *acc = (double *)(smem + kRpAcc);
    const int tid = L.tid, w = L.warp, l = L.lane;
    const int at = blockIdx.x % a.n_heads, b = blockIdx.x / a.n_heads;
    const size_t lh = a.heads ? a.heads[at] : at;
    const int layer = (int)(lh / a.Hv), h = (int)(lh % a.Hv);
    const int hk = h / (a.Hv / a.Hk), K1 = a.fit.n_cand + 1;
    load_weights(L, S, a.w + lh * 128);
    for (int e = tid; e < 128 * K1; e += kThreads) acc[e] = 0.0;
    // A token's vectors: loaded two tokens ahead by threads 0..127 (one channel
    // each), in shared memory one token ahead, three buffers.
    float fk = 0.f, fv = 0.f, fd = 0.f, fb = 0.f;
    const auto fetch = [&](int t) {
        if (tid < 128 && t < a.T) {
            const size_t tok = ((size_t)layer * a.T + t) * a.n + b;
            fk = a.k[(tok * a.Hk + hk) * 128 + tid];
            fv = a.v[(tok * a.Hv + h) * 128 + tid];
            fd = a.gate_per_row ? a.gate[(tok * a.Hv + h) * 128 + tid] : a.gate[tok * a.Hv + h];
            fb = a.beta[tok * a.Hv + h];
        }
    };
    const auto put = [&](int buf) {
        if (tid < 128) {
            rowA[buf * 128 + tid] = make_float4(fd, fd, fk, fk);
            const float bk = fb * fk;
            rowB[buf * 128 + tid] = make_float2(bk, bk);
            vs[buf * 128 + tid] = fv;
        }
    };
    fetch(0);
    put(0);
    fetch(1);
    __syncthreads();
    uint64_t x2[16][2];
#pragma unroll
    for (int r = 0; r < 16; r++) x2[r][0] = x2[r][1] = 0;
    const uint8_t *piv = a.pivot_rows ? a.pivot_rows + lh * 128 : nullptr;
    int left = a.every;
    for (int t = 0, cur = 0; t < a.T; t++) {
        const int nxt = cur == 2 ? 0 : cur + 1;
        float *rd = red + (t & 1) * 8 * 128;
        // P = D S and the retrieval u_j = sum_i k_i P_ij.
        uint64_t ua[2] = {0, 0}, ub[2] = {0, 0};
#pragma unroll
        for (int r = 0; r < 16; r++) {
            const uint4 q = *(const uint4 *)&rowA[cur * 128 + 16 * w + r];
            const uint64_t dd = u2pair(q.x, q.y), kk = u2pair(q.z, q.w);
            x2[r][0] = fmul2(x2[r][0], dd);
            x2[r][1] = fmul2(x2[r][1], dd);
            uint64_t(&ac)[2] = (r & 1) ? ub : ua;
            ac[0] = ffma2(kk, x2[r][0], ac[0]);
            ac[1] = ffma2(kk, x2[r][1], ac[1]);
        }
        {
            const uint64_t s0 = fadd2(ua[0], ub[0]), s1 = fadd2(ua[1], ub[1]);
            *(float4 *)&rd[w * 128 + 4 * l] = make_float4(f2lo(s0), f2hi(s0), f2lo(s1), f2hi(s1));
        }
        // The next token's buffer was last read two tokens ago, behind the previous
        // token's barrier; this one's barrier publishes it.
        put(nxt);
        fetch(t + 2);
        __syncthreads();
        // delta_j = v_j - u_j; S = P + beta k_i delta_j.
        uint64_t s0 = 0, s1 = 0;
#pragma unroll
        for (int wv = 0; wv < 8; wv++) {
            const uint4 p = *(const uint4 *)&rd[wv * 128 + 4 * l];
            s0 = fadd2(s0, u2pair(p.x, p.y));
            s1 = fadd2(s1, u2pair(p.z, p.w));
        }
        const float4 v4 = *(const float4 *)&vs[cur * 128 + 4 * l];
        const uint64_t d0 = f2(v4.x - f2lo(s0), v4.y - f2hi(s0)), d1 = f2(v4.z - f2lo(s1), v4.w - f2hi(s1));
#pragma unroll
        for (int r = 0; r < 16; r++) {
            const uint64_t bk = *(const uint64_t *)&rowB[cur * 128 + 16 * w + r];
            x2[r][0] = ffma2(bk, d0, x2[r][0]);
            x2[r][1] = ffma2(bk, d1, x2[r][1]);
        }
        if (--left == 0) {
            left = a.every;
#pragma unroll
            for (int r = 0; r < 16; r++)
                *(uint4 *)&tile[(16 * w + r) * 128 + 4 * cgroup(l >> 2, l & 3)] =
                    make_uint4((uint32_t)x2[r][0], (uint32_t)(x2[r][0] >> 32), (uint32_t)x2[r][1],
                               (uint32_t)(x2[r][1] >> 32));
            __syncwarp();                                     // both mappings give warp w rows 16w..16w+15
            {
                uint64_t x[4][8];
                float msum[4];
#pragma unroll
                for (int t4 = 0; t4 < 4; t4++) {
                    float s = 0.f;
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float4 f = *(const float4 *)&tile[L.row(t4) * 128 + 4 * cgroup(L.cg, e)];
                        x[t4][2 * e] = f2(f.x, f.y);
                        x[t4][2 * e + 1] = f2(f.z, f.w);
                        s += fabsf(f.x) + fabsf(f.y) + fabsf(f.z) + fabsf(f.w);
                    }
                    msum[t4] = row_allreduce(s);
                }
                // one adder per entry and a fixed order within the CTA
                distortion_of(L, S, x, msum, piv, a.fit, [&](int k, int i, double e) { acc[i * K1 + k] += e; });
            }
#pragma unroll
            for (int r = 0; r < 16; r++) {
                const uint4 p = *(const uint4 *)&tile[(16 * w + r) * 128 + 4 * cgroup(l >> 2, l & 3)];
                x2[r][0] = u2pair(p.x, p.y);
                x2[r][1] = u2pair(p.z, p.w);
            }
        }
        cur = nxt;
    }
    __syncthreads();
    const int entries = (a.fit.unit_rows ? 128 : 1) * K1;
    for (int e = tid; e < entries; e += kThreads) atomicAdd(&a.acc[lh * entries + e], acc[e]);
}

// ------------------------------------------------------------------ launchers
static stepq_status launched() {
    return cudaGetLastError() == cudaSuccess ? STEPQ_OK : STEPQ_ERR_CUDA;
}

stepq_status launch_decode(const stepq_plan *p, int layer, uint8_t *pool, int pool_slots,
                           const int32_t *slots, int B, const float *q, const float *k,
                           const float *v, const float *beta, const float *gate, float *y,
                           cudaStream_t s) {
    if (p->cfg.gate_kind == STEPQ_GATE_SCALAR)
        return launch_decode_heads(p, layer, pool, pool_slots, slots, B, q, k, v, beta, gate, y, s);
    return launch_decode_rows(p, layer, pool, pool_slots, slots, B, q, k, v, beta, gate, y, s);
}

// layer >= 0: one layer's heads; layer = -1: all layers' in one launch (their tables,
// and their states in a batch entry, follow each other).
static PoolArgs pool_args(const stepq_plan *p, int layer, const float *states, const int32_t *slots, int B,
                          uint8_t *pool, int pool_slots) {
    const int heads = p->cfg.n_value_heads * (layer < 0 ? p->cfg.n_layers : 1);
    return {pool, p->slot_stride, pool_slots, slots, p->layer(layer < 0 ? 0 : layer), heads, B * heads,
            p->cfg.fit_iters, (float *)states, (size_t)heads * kN, device_error_word()};
}

stepq_status launch_quantize(const stepq_plan *p, int layer, const float *states, const int32_t *slots, int B,
                             uint8_t *pool, int pool_slots, cudaStream_t s) {
    if (p->cfg.gate_kind == STEPQ_GATE_SCALAR)
        return launch_quantize_heads(p, layer, states, slots, B, pool, pool_slots, s);
    static SmemOptIn opt;
    const stepq_status st = opt((const void *)quantize_kernel, kQSmem);
    if (st != STEPQ_OK) return st;
    const PoolArgs a = pool_args(p, layer, states, slots, B, pool, pool_slots);
    const int grid = 2 * sm_count();
    return launch_overlapped(quantize_kernel, grid < a.items ? grid : a.items, kThreads, kQSmem, s, a);
}

stepq_status launch_dequantize(const stepq_plan *p, int layer, const uint8_t *pool, int pool_slots,
                               const int32_t *slots, int B, float *states, cudaStream_t s) {
    if (p->cfg.gate_kind == STEPQ_GATE_SCALAR)
        return launch_dequantize_heads(p, layer, pool, pool_slots, slots, B, states, s);
    const PoolArgs a = pool_args(p, layer, states, slots, B, (uint8_t *)pool, pool_slots);
    return launch_overlapped(dequantize_kernel, a.items, kThreads, 0, s, a);
}

static FitCands fit_cands(const stepq_config *cfg) {
    FitCands f{};
    f.unit_rows = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    f.n_cand = cfg->n_candidates;
    f.fit_iters = cfg->fit_iters;
    for (int k = 0; k < cfg->n_candidates; k++) f.cands[k] = cfg->candidates[k];
    return f;
}

stepq_status launch_calib_distortion(const stepq_config *cfg, int layer, const float *w,
                                     const uint8_t *pivot_rows, const float *states, int n,
                                     double *acc, cudaStream_t s) {
    const size_t Hv = (size_t)cfg->n_value_heads;
    const bool rows = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    const size_t K1 = (size_t)cfg->n_candidates + 1;
    DistArgs a{};
    a.states = states;
    a.w = w + (size_t)layer * Hv * kD;
    a.pivot_rows = (rows && pivot_rows) ? pivot_rows + (size_t)layer * Hv * kD : nullptr;
    a.acc = acc + (size_t)layer * Hv * (rows ? kD : 1) * K1;
    a.Hv = (int)Hv;
    a.fit = fit_cands(cfg);
    distortion_kernel<<<(unsigned)(n * Hv), kThreads, 0, s>>>(a);
    return launched();
}

stepq_status launch_calib_replay(const stepq_config *cfg, int n, int T, int every, const float *k,
                                 const float *v, const float *beta, const float *gate, const float *w,
                                 const uint8_t *pivot_rows, double *acc, const int32_t *heads, int n_heads,
                                 cudaStream_t s) {
    static SmemOptIn opt;
    const stepq_status st = opt((const void *)replay_kernel, kRpSmem);
    if (st != STEPQ_OK) return st;
    const bool rows = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    ReplayArgs a{k, v, beta, gate, w, rows ? pivot_rows : nullptr, acc, heads, n_heads, n, T,
                 cfg->n_key_heads, cfg->n_value_heads, every, rows, fit_cands(cfg)};
    const size_t ctas = (size_t)n * n_heads;
    if (ctas > 0x7fffffffu) return STEPQ_ERR_UNSUPPORTED;
    replay_kernel<<<(unsigned)ctas, kThreads, kRpSmem, s>>>(a);
    return launched();
}

}  // namespace stepq
