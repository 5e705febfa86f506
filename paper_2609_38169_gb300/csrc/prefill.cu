// Chunked FP32-state prefill: the gated Delta rule (Eq. delta_update) over T
// tokens, 32 tokens at a time, producing the boundary state that
// stepq_quantize_pool packs (the prefill side of App. C.3 / App. F.1: the
// native chunk computation runs on an uncompressed state, and the state is
// packed once at the boundary).
//
// Within a chunk with cumulative gates g_t = d_1 ... d_t (per key channel; a
// scalar gate is the same value in every channel) and S_0 the state before it:
//   S_t = G_t S_0 + sum_{s<=t} G_t G_s^-1 k_s w_s^T,
//   w_t = beta_t (v_t - S_0^T g_t k_t - sum_{s<t} (k_s/g_s . g_t k_t) w_s),
// i.e. (I + A) W = diag(beta) (V - K~ S_0) with K~ = G K, K^ = G^-1 K and
// A_ts = beta_t (K~_t . K^_s) for s < t; the outputs are
//   Y = Q~ S_0 + Bm W,  Bm = tril(Q~ K^T) (Q~ = G Q, lower triangle with the diagonal),
// and the state after the chunk is S_C = G_C S_0 + K_bar^T W, K_bar = K g_C / g.
//
// Every product runs on the tensor cores (tcgen05, kind::tf32) in split
// precision: an fp32 operand is its TF32 head, which is all the tensor core reads of
// it, plus a remainder, and a product is head*head + head*rest + rest*head (P0 and PW
// also take rest*rest), which keeps fp32 accuracy. The state stays in tensor memory as
// S^T (lane j = value column, column i = key row):
//   P0  [Q~ ; K~] K^T        -> Bm, A      M = 128, N = 64, K = 128, A, B in smem
//   P1  S_0^T [Q~ ; K~]^T    -> [Q~ S_0 ; K~ S_0]^T    M = 128, N = 128 / 64, K = 128, A in tmem
//   PW  W^T - R^T = R^T (T - I)^T, T = (I + A)^-1, R = diag(beta) (V - K~ S_0)   M = 128, N = 64, K = 32
//   P2  S^T += W^T K_bar and Y^T = (Q~ S_0)^T + W^T Bm^T   M = 128, N = 160, K = 32, A in tmem
// An MMA with M = 128 takes N / 2 cycles, but not less than the 35 to 45 that its issue
// takes, so operands are stacked until N is 128 where they can be: P0's A rows and P1's B
// rows are [Q~ ; K~] (64) over its rests (64), P0's B rows K^ (32) over its rests (32),
// PW's T (32) over its rests (32), P2's K_bar^T (128) over Bm (32). The partial products
// of stacked rests land in columns (or, P0, lanes) of their own and are added when they
// are read. Shared-memory operands are K-major core matrices (8 rows x 16 bytes). The
// FMA pipe keeps the element-wise work, the inverse T and the scaling of S by g_C.
//
// Precision of W: the identity's part of T R is R itself, added in fp32, so that only
// (T - I) R goes through split operands; the rests of R and W are rounded, not truncated,
// to what the tensor core keeps of them; and the lower blocks of T are formed as
// T22 (N21 T11), the order whose rounding T11 does not amplify. W then is as near to fp64 as
// by a forward substitution in fp32 or nearer (0.7 to 0.96 of its error with keys from
// random to equal and beta up to 1; W = T R from truncated rests: 1.2 to 1.5). Whole outputs,
// 512 tokens, random keys, scalar gates 0.85 to 0.999: y 1.08e-6 and the final state 4.4e-7
// off, at 1.76 ms as below; with W = T R 1.30e-6 and 6.7e-7 at 1.75 ms; with the substitution,
// P0 without rest*rest, 1.88e-6 and 5.8e-7. (The state's rest rounded too gives 1.05e-6 and
// 4.4e-7, but lies on the chain: 1.82 ms.)
//
// One persistent CTA of 20 warps per SM; it owns all 512 tensor-memory columns:
//   [0, 128) S^T | [128, 160) Y^T | [160, 192) (K~ S_0)^T, then R^T | [192, 256) the rests'
//   part of both | [256, 384) S^T rest | [384, 448) P0 result | [448, 480) W^T |
//   [480, 512) W^T rest
// The chunks of a head are a serial chain P1 -> R -> PW -> P2 -> P1, so the time of a
// chunk is that chain's latency, and the rest runs beside it:
//   warps 0-7   the chain: S's rest (under P1's first half), A and Bm from P0 (under P1),
//               R, W, the scaling of S (under PW); a chunk's y leaves under the next one
//   warps 8-15  the next chunk's operands: cumulative gates, products and rests, written
//               as soon as the products of this chunk have read theirs
//   warp 16     issues the MMAs, P0 of the next chunk right after P2
//   warp 17     T from A
//   warp 18     q and k of the next chunk by bulk copies
// With 8 warps doing all of it in turn a chunk took 17,700 cycles: 6,700 the operands,
// 5,500 waiting on P0 and P1 (96 MMAs then, 48 now), 2,200 a triangular solve for W, 1,500
// the outputs. It takes 7,800 now, of which 2,200 are T and 1,250 A and Bm (both wait on
// P0, 900, which follows P2, 1,100) and 900 R, PW and W.
// 128 slots x 32 heads x 512 tokens: 4.05 ms then, 1.76 ms now.
//
// Hand-over, all by mbarriers, one phase a chunk, every wait bounded: `full1` (warps
// 8-15: Q~, K~, K^, V, beta, g_C) starts P0, which completes `p0`; `ready` (warps 0-7: S,
// Y read) and `rest` start P1's halves, which complete `p1`; `a` (warps 0-7: A) starts
// warp 17, which completes `t`; `rready` (warps 0-7: R) and `t` start PW, which completes
// `pw`; `wready` (warps 0-7: W, Bm, scaled S) and `full2` (warps 8-15: K_bar) start P2,
// which completes `p2`. Warps 8-15 refill K^ after p0, Q~ and K~ after p1 and K_bar after
// p2; q and k are refilled after full1 and complete `in`; V, beta and g_C have two buffers.
#include "async.cuh"
#include "device.cuh"
#include "internal.h"
#include "tcgen05.cuh"

namespace stepq {
namespace pf {

constexpr int C = 32;                                  // tokens per chunk
constexpr int kGroup = 256;                            // threads of warps 0-7 and of warps 8-15
constexpr int kBlock = 2 * kGroup + 128;
// Registers a thread: 96 at launch (20 warps), then the shares of the three groups.
constexpr int kRegs = 96, kRegsChain = 112, kRegsProduce = 88, kRegsIssue = 80;
static_assert(kGroup * (kRegsChain + kRegsProduce) + 128 * kRegsIssue <= kBlock * kRegs, "register shares");
constexpr uint32_t kColS = 0, kColY = 128, kColX = 160, kColYl = 192, kColXl = 224, kColSl = 256, kColP0 = 384,
                   kColW = 448, kColWl = 480;
constexpr uint32_t kCols = 512;
constexpr uint32_t kIdescP0 = tc::idesc_tf32(128, 64);
constexpr uint32_t kIdescP1 = tc::idesc_tf32(128, 128), kIdescP1l = tc::idesc_tf32(128, 64);
constexpr uint32_t kIdescPw = tc::idesc_tf32(128, 64);
constexpr uint32_t kIdescP2 = tc::idesc_tf32(128, 160);

// Shared-memory operands: K-major core matrices of 8 rows x 4 fp32 (128 B). Strides are
// chosen for the stores alone (the tensor core's time does not depend on them): with
// K = 128 the matrices are back to back and a quarter warp stores 8 tokens of one; with
// K = 32 they are 144 B apart along K and 1184 B between row groups, so that a warp's
// scalar stores (8 tokens x 4 channels) hit 32 banks.
constexpr int kLbo128 = 128, kSbo128 = 32 * kLbo128;
constexpr int kLbo32 = 144, kSbo32 = 8 * kLbo32 + 32;
constexpr int kQRow = 132;                             // padded row of q and k
constexpr int kOffB1 = 0;                              // [Q~ ; K~] 64 rows x K 128, then its rests
constexpr int kOffB1l = kOffB1 + 8 * kSbo128;
constexpr int kOffB3 = kOffB1l + 8 * kSbo128;          // K^ 32 rows (s) x K 128, then its rests
constexpr int kOffB3l = kOffB3 + 4 * kSbo128;
constexpr int kOffB2 = kOffB3l + 4 * kSbo128;          // K_bar^T 128 rows (i) x K 32 (t), then Bm 32 rows (t) x K 32 (s)
constexpr int kOffB4 = kOffB2 + 16 * kSbo32;
constexpr int kOffB2l = kOffB4 + 4 * kSbo32;           // the rests of both
constexpr int kOffB4l = kOffB2l + 16 * kSbo32;
constexpr int kOffV = kOffB4l + 4 * kSbo32;            // float [2][C][128] V (16-byte group f of token t at f ^ (t & 7))
constexpr int kOffGc = kOffV + 2 * C * 128 * 4;        // float [2][128] g_C
constexpr int kOffBeta = kOffGc + 2 * 128 * 4;         // float [2][C]
constexpr int kMRow = C + 4;                           // padded row of A, T and F
constexpr int kOffA = kOffBeta + 2 * C * 4;            // float [C][kMRow] -A (zero from the diagonal on)
constexpr int kOffTm = kOffA + C * kMRow * 4;          // float [C][kMRow] T as it forms
constexpr int kOffF = kOffTm + C * kMRow * 4;          // float [64][kMRow] P0 partials of the rest rows
constexpr int kOffT = kOffF;                           // T 32 rows (t) x K 32 (s), then its rests; after F is read
constexpr int kOffTl = kOffT + 4 * kSbo32;
constexpr int kOffQK = kOffT + 8 * kSbo32;             // float [2 C][kQRow] the next chunk's q, then k
constexpr int kOffBar = kOffQK + 2 * C * kQRow * 4;        // uint64 [14] mbarriers
constexpr int kOffTmem = kOffBar + 112;                 // u32 tensor-memory base
constexpr int kSmem = kOffTmem + 16;
static_assert(kSmem <= kSmemMax, "one CTA's shared memory");
static_assert(64 * kMRow * 4 <= 8 * kSbo32 && kOffF % 16 == 0, "T in the place of F");
enum { kIn, kReady, kRest, kFull1, kP0, kA, kT, kP1, kRready, kPw, kWready, kFull2, kP2, kDrain };

// Byte offset of element (row r, k) of a K-major operand.
__device__ __forceinline__ int off128(int r, int k) { return (r >> 3) * kSbo128 + (k >> 2) * kLbo128 + (r & 7) * 16; }
__device__ __forceinline__ int off32(int r, int k) {
    return (r >> 3) * kSbo32 + (k >> 2) * kLbo32 + (r & 7) * 16 + (k & 3) * 4;
}

// Four consecutive K elements of one row (off 16-byte aligned) and their rests.
__device__ __forceinline__ void put4(uint8_t *base, uint8_t *rest, int off, float4 x) {
    *(float4 *)(base + off) = x;
    *(float4 *)(rest + off) =
        make_float4(tc::tf32_rest(x.x), tc::tf32_rest(x.y), tc::tf32_rest(x.z), tc::tf32_rest(x.w));
}
__device__ __forceinline__ float4 mul4(float4 a, float4 b) {
    return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}
__device__ __forceinline__ float rcp(float x) {          // within 1 ulp
    float d;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(d) : "f"(x));
    return d;
}
// Barrier over the 256 threads of warps 0-7; returns the OR of their predicates.
__device__ __forceinline__ bool group_any(bool p) {
    uint32_t r;
    asm volatile(
        "{ .reg .pred p, q; setp.ne.u32 p, %1, 0; barrier.cta.red.or.pred q, 1, 256, p; selp.u32 %0, 1, 0, q; }"
        : "=r"(r)
        : "r"((uint32_t)p)
        : "memory");
    return r != 0;
}

struct Args {
    const float *q, *k, *v, *beta, *gate;
    float *states, *y;
    int T, Hk, Hv, gate_per_row, items;      // item = batch entry * Hv + head
    unsigned int *err;
    StallKnob stall;
};

// Cumulative gates of a chunk: this thread's float4 of four channels at tokens 8 m + tl
// (m = 0..3, tl = lane & 7), multiplied up over the tokens by a scan over the 8 lanes
// of a token block and the blocks before it; kept above 1e-30 so that K / g stays
// finite. Returns g_C.
__device__ __forceinline__ float4 scan_channels(float4 (&g)[4], int tl) {
    const auto up = [&](float x, int o) {
        const float y = __shfl_up_sync(0xffffffffu, x, o, 8);
        return tl >= o ? x * y : x;
    };
    const auto floor4 = [](float4 a, float4 b) {
        return make_float4(fmaxf(a.x * b.x, 1e-30f), fmaxf(a.y * b.y, 1e-30f), fmaxf(a.z * b.z, 1e-30f),
                           fmaxf(a.w * b.w, 1e-30f));
    };
    float4 run = make_float4(1.f, 1.f, 1.f, 1.f);
#pragma unroll
    for (int m = 0; m < 4; m++) {
#pragma unroll
        for (int o = 1; o < 8; o *= 2) g[m] = make_float4(up(g[m].x, o), up(g[m].y, o), up(g[m].z, o), up(g[m].w, o));
        const float4 all = make_float4(__shfl_sync(0xffffffffu, g[m].x, 7, 8), __shfl_sync(0xffffffffu, g[m].y, 7, 8),
                                       __shfl_sync(0xffffffffu, g[m].z, 7, 8), __shfl_sync(0xffffffffu, g[m].w, 7, 8));
        g[m] = floor4(run, g[m]);
        run = floor4(run, all);
    }
    return run;
}

// Warps 8-15: the operands of this CTA's chunks, in order. Warp pw holds channels
// 16 pw .. +15; lane l holds channels 16 pw + 4 (l >> 3) .. +3 at tokens 8 m + (l & 7),
// so that a load covers 64-byte pieces of 8 tokens, a quarter warp's operand store one
// core matrix, and the gates' product over the tokens stays inside the warp. No input is
// loaded through registers but the gates (64 more registers spilled as they arrived and
// held the warps for their latency): warp 18 brings q and k, cp.async V to where the
// solve reads it. Missing tokens of a ragged tail are the identity step (gate 1, beta 0,
// zero k, q, v).
__device__ __forceinline__ bool produce(const Args &a, uint8_t *smem, uint64_t *bars) {
    uint8_t *B1 = smem + kOffB1, *B1l = smem + kOffB1l, *B2 = smem + kOffB2, *B2l = smem + kOffB2l;
    uint8_t *B3 = smem + kOffB3, *B3l = smem + kOffB3l;
    const int l = threadIdx.x & 31, tl = l & 7, pw = (threadIdx.x - kGroup) >> 5, c4 = 16 * pw + 4 * (l >> 3);
    const float *Q = (const float *)(smem + kOffQK) + c4, *K = Q + C * kQRow;
    float4 g[4];
    float ds = 1.f, bt = 0.f;
    int fn = 0;
    // gates and beta of a chunk; its V (buffer vb) once that buffer is free
    const auto fetch = [&](int item, int c0) {
        const int b = item / a.Hv, h = item - b * a.Hv;
        fn = min(C, a.T - c0);
        const size_t tok0 = (size_t)b * a.T + c0, tok = tok0 + min(l, fn - 1);
        if (a.gate_per_row) {
#pragma unroll
            for (int m = 0; m < 4; m++)
                g[m] = *(const float4 *)&a.gate[((tok0 + min(8 * m + tl, fn - 1)) * a.Hv + h) * 128 + c4];
        } else {
            ds = a.gate[tok * a.Hv + h];
        }
        if (pw == 0) bt = a.beta[tok * a.Hv + h];
    };
    const auto fetch_v = [&](int item, int c0, uint32_t vb) {
        const int b = item / a.Hv, h = item - b * a.Hv, n = min(C, a.T - c0);
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const int t = 8 * m + tl;
            const size_t tok = (size_t)b * a.T + c0 + (t < n ? t : 0);
            cp_async16_or_zero(smem + kOffV + ((vb * C + t) * 128 + (c4 ^ 4 * tl)) * 4, &a.v[(tok * a.Hv + h) * 128 + c4], t < n);
        }
    };
    const auto token = [&](const float *p, int t) {
        return t < fn ? *(const float4 *)(p + t * kQRow) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    const auto wait = [&](int bar, uint32_t ph) {
        return (bool)__all_sync(0xffffffffu, mbar_wait(&bars[bar], ph, a.stall.wait_cycles));
    };
    int item = blockIdx.x, c0 = 0;
    if (item < a.items) {
        fetch(item, 0);
        fetch_v(item, 0, 0);
    }
    for (uint32_t n = 0; item < a.items; n++) {
        const uint32_t buf = n & 1u, prev = buf ^ 1u;      // prev: parity of chunk n - 1's phases
        float4 gC;
        if (a.gate_per_row) {
#pragma unroll
            for (int m = 0; m < 4; m++)
                if (8 * m + tl >= fn) g[m] = make_float4(1.f, 1.f, 1.f, 1.f);
            gC = scan_channels(g, tl);
        } else {                                           // lane l: token l
            float d = l < fn ? ds : 1.f;
#pragma unroll
            for (int o = 1; o < 32; o *= 2) {
                const float y = __shfl_up_sync(0xffffffffu, d, o);
                d = l >= o ? d * y : d;
            }
            d = fmaxf(d, 1e-30f);
            const float dC = __shfl_sync(0xffffffffu, d, 31);
            gC = make_float4(dC, dC, dC, dC);
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const float x = __shfl_sync(0xffffffffu, d, 8 * m + tl);
                g[m] = make_float4(x, x, x, x);
            }
        }
        cp_async_wait_all();                               // V
        if (!wait(kIn, buf)) return false;                 // q and k
        // P0 of the chunk before has read K^, its P1 Q~ and K~; beta and g_C of two
        // chunks ago are used up (S's rest was formed before that P1 started).
        if (n > 0 && !wait(kP0, prev)) return false;
        float4 kb[4];                                      // K_bar at the thread's tokens
#pragma unroll
        for (int m = 0; m < 4; m++) {
            float4 kr = make_float4(rcp(g[m].x), 0.f, 0.f, 0.f);
            kr.y = a.gate_per_row ? rcp(g[m].y) : kr.x;
            kr.z = a.gate_per_row ? rcp(g[m].z) : kr.x;
            kr.w = a.gate_per_row ? rcp(g[m].w) : kr.x;
            kr = mul4(token(K, 8 * m + tl), kr);
            put4(B3, B3l, off128(8 * m + tl, c4), kr);                              // K^
            kb[m] = mul4(kr, gC);
        }
        if (n > 0 && !wait(kP1, prev)) return false;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const int t = 8 * m + tl;
            put4(B1, B1l, off128(t, c4), mul4(g[m], token(Q, t)));                  // Q~
            put4(B1, B1l, off128(C + t, c4), mul4(g[m], token(K, t)));              // K~
        }
        if (tl == 0) *(float4 *)(smem + kOffGc + (buf * 128 + c4) * 4) = gC;
        if (pw == 0) ((float *)(smem + kOffBeta))[buf * C + l] = l < fn ? bt : 0.f;
        fence_async_smem();
        mbar_arrive(&bars[kFull1]);
        c0 += C;
        if (c0 >= a.T) {
            item += gridDim.x;
            c0 = 0;
        }
        if (item < a.items) fetch(item, c0);
        // P2 of the chunk before has read K_bar.
        if (n > 0 && !wait(kP2, prev)) return false;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const float e4[4] = {kb[m].x, kb[m].y, kb[m].z, kb[m].w};
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int o = off32(c4 + e, 8 * m + tl);
                *(float *)(B2 + o) = e4[e];
                *(float *)(B2l + o) = tc::tf32_rest(e4[e]);
            }
        }
        fence_async_smem();
        mbar_arrive(&bars[kFull2]);
        if (item < a.items) fetch_v(item, c0, prev);       // V of the chunk before is used up
    }
    return true;
}

// Warp 18: q and k of every chunk, one bulk copy of 512 bytes a token and vector, once
// the operands of the chunk before are written. (The phases of full1 and `in` cannot
// run ahead of this warp: each needs the copies it starts in between.)
__device__ __forceinline__ bool load_qk(const Args &a, uint8_t *smem, uint64_t *bars) {
    const int l = threadIdx.x & 31, grp = a.Hv / a.Hk;
    uint8_t *dst = smem + kOffQK + l * kQRow * 4;
    uint32_t n = 0;
    bool ok = true;
    for (int item = blockIdx.x; ok && item < a.items; item += gridDim.x) {
        const int b = item / a.Hv, hk = (item - b * a.Hv) / grp;
        for (int c0 = 0; c0 < a.T; c0 += C, n++) {
            ok = n == 0 || __all_sync(0xffffffffu, mbar_wait(&bars[kFull1], (n - 1) & 1u, a.stall.wait_cycles));
            if (!ok) break;
            if (item == a.stall.withhold_item && c0 == 0) continue;   // test switch: these copies never start
            const int tokens = min(C, a.T - c0);
            if (l == 0) mbar_arrive_tx(&bars[kIn], (uint32_t)tokens * 1024u);
            __syncwarp();
            if (l < tokens) {
                const size_t e = (((size_t)b * a.T + c0 + l) * a.Hk + hk) * 128;
                bulk_load(dst, a.q + e, 512, &bars[kIn]);
                bulk_load(dst + C * kQRow * 4, a.k + e, 512, &bars[kIn]);
            }
        }
    }
    // no copy is in flight when the CTA ends, whatever stalled
    return (n == 0 || mbar_wait(&bars[kIn], (n - 1) & 1u, a.stall.wait_cycles)) && ok;
}

// Warp 16: the MMAs of this CTA's chunks, issued by one elected lane; the whole warp runs
// the loop, converged, so that descriptors stay in uniform registers.
__device__ __forceinline__ bool issue_mma(const Args &a, uint8_t *smem, uint64_t *bars, uint32_t tm) {
    // Descriptors of each operand's first K step; a step of 8 adds 2 core matrices.
    const uint64_t d1 = tc::sdesc(smem + kOffB1, kLbo128, kSbo128), d3 = tc::sdesc(smem + kOffB3, kLbo128, kSbo128);
    const uint64_t d2 = tc::sdesc(smem + kOffB2, kLbo32, kSbo32), d2l = tc::sdesc(smem + kOffB2l, kLbo32, kSbo32);
    const uint64_t dT = tc::sdesc(smem + kOffT, kLbo32, kSbo32);
    constexpr uint64_t k128 = 2 * kLbo128 / 16, k32 = 2 * kLbo32 / 16;
    const int per = (a.T + C - 1) / C, mine = (a.items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const long long chunks = (long long)per * mine;
    const uint32_t lead = tc::elect();
    const auto wait = [&](int bar, uint32_t ph) {
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&bars[bar], ph, a.stall.wait_cycles));
        tc::fence_after();
        return ok;
    };
    const auto p0 = [&]() {
#pragma unroll
        for (int s = 0; s < 16; s++)
            tc::mma_tf32_ss(lead, tm + kColP0, d1 + s * k128, d3 + s * k128, kIdescP0, s > 0 ? 1u : 0u);
        tc::commit(lead, &bars[kP0]);
    };
    bool ok = wait(kFull1, 0);
    if (ok) p0();
    for (long long n = 0; ok && n < chunks; n++) {
        const uint32_t ph = (uint32_t)n & 1u;
        if (!(ok = wait(kReady, ph))) break;
        // the heads' part of P1 needs the state alone; its rest is formed under it
#pragma unroll
        for (int s = 0; s < 16; s++)
            tc::mma_tf32_ts(lead, tm + kColY, tm + kColS + 8 * s, d1 + s * k128, kIdescP1, s > 0 ? 1u : 0u);
        if (!(ok = wait(kRest, ph))) break;
#pragma unroll
        for (int s = 0; s < 16; s++)
            tc::mma_tf32_ts(lead, tm + kColY, tm + kColSl + 8 * s, d1 + s * k128, kIdescP1l, 1u);
        tc::commit(lead, &bars[kP1]);
        if (!(ok = wait(kT, ph) && wait(kRready, ph))) break;
#pragma unroll
        for (int s = 0; s < 4; s++) {
            tc::mma_tf32_ts(lead, tm + kColW, tm + kColX + 8 * s, dT + s * k32, kIdescPw, s > 0 ? 1u : 0u);
            tc::mma_tf32_ts(lead, tm + kColW, tm + kColXl + 8 * s, dT + s * k32, kIdescPw, 1u);
        }
        tc::commit(lead, &bars[kPw]);
        if (!(ok = wait(kFull2, ph) && wait(kWready, ph))) break;
#pragma unroll
        for (int s = 0; s < 4; s++) {
            tc::mma_tf32_ts(lead, tm + kColS, tm + kColW + 8 * s, d2 + s * k32, kIdescP2, 1u);
            tc::mma_tf32_ts(lead, tm + kColS, tm + kColW + 8 * s, d2l + s * k32, kIdescP2, 1u);
            tc::mma_tf32_ts(lead, tm + kColS, tm + kColWl + 8 * s, d2 + s * k32, kIdescP2, 1u);
        }
        tc::commit(lead, &bars[kP2]);
        if (n + 1 < chunks && (ok = wait(kFull1, ph ^ 1u))) p0();
    }
    // every MMA has ended before the tensor memory is given back
    tc::commit(lead, &bars[kDrain]);
    return wait(kDrain, 0) && ok;
}

// Warp 17: T = (I + A)^-1 of every chunk from N = -A, by blocks: the 8 x 8 diagonal
// blocks by substitution (a row per lane), then the lower parts of the 16 x 16 and the
// 32 x 32 blocks as T22 (N21 T11), two dense products each. One substitution over 32 rows
// is a chain of 31 dependent steps (2,400 cycles or more; this takes 2,200 beside the
// other warps' shared-memory traffic). A lane holds a row of the
// left factor and reads the right one's rows, 16 bytes at a time, eight loads in flight.
__device__ __forceinline__ bool invert(const Args &a, uint8_t *smem, uint64_t *bars) {
    const float *N = (const float *)(smem + kOffA);
    float *T = (float *)(smem + kOffTm);
    const int l = threadIdx.x & 31;
    const int per = (a.T + C - 1) / C, mine = (a.items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    const long long chunks = (long long)per * mine;
    const auto quad4 = [](const float *p) { return *(const uint4 *)p; };
    const auto put = [](float *p, uint64_t lo, uint64_t hi) {
        *(uint4 *)p = make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
    };
    const auto acc4 = [](const uint4 &m, uint32_t u, uint64_t &lo, uint64_t &hi) {
        const uint64_t uu = u2pair(u, u);
        lo = ffma2(u2pair(m.x, m.y), uu, lo);
        hi = ffma2(u2pair(m.z, m.w), uu, hi);
    };
    // (lo, hi) = x[0..8) m, x a row of eight, m eight rows kMRow apart (four columns of each)
    const auto row8 = [&](const float *x, const float *m, uint64_t &lo, uint64_t &hi) {
        const uint4 x0 = quad4(x), x1 = quad4(x + 4);
        uint4 r[8];
#pragma unroll
        for (int s = 0; s < 8; s++) r[s] = quad4(m + s * kMRow);
        const uint32_t xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
        for (int s = 0; s < 8; s++) acc4(r[s], xv[s], lo, hi);
    };
    for (long long n = 0; n < chunks; n++) {
        const uint32_t ph = (uint32_t)n & 1u;
        if (!__all_sync(0xffffffffu, mbar_wait(&bars[kA], ph, a.stall.wait_cycles))) return false;
        {   // 8 x 8 blocks: lane 8 b + r holds row r of block b
            const int o = l & 24, r = l & 7;
            const float *m = N + o * kMRow + o;
            uint4 lo[8], hi[8];
#pragma unroll
            for (int q = 1; q < 8; q++) {
                lo[q] = quad4(m + q * kMRow);
                if (q > 4) hi[q] = quad4(m + q * kMRow + 4);
            }
            uint64_t x[4];
#pragma unroll
            for (int p = 0; p < 4; p++) x[p] = f2(2 * p == r ? 1.f : 0.f, 2 * p + 1 == r ? 1.f : 0.f);
#pragma unroll
            for (int q = 7; q > 0; q--) {                             // row q of N is zero from column q on
                const uint32_t xq = (uint32_t)(q & 1 ? x[q >> 1] >> 32 : x[q >> 1]);
                acc4(lo[q], xq, x[0], x[1]);
                if (q > 4) acc4(hi[q], xq, x[2], x[3]);
            }
            float *t = T + (o + r) * kMRow + o;
            put(t, x[0], x[1]);
            put(t + 4, x[2], x[3]);
            if (!(o & 8)) {                                           // read as part of the 16 x 16 block
                put(t + 8, 0, 0);
                put(t + 12, 0, 0);
            }
        }
        __syncwarp();
        {   // 16 x 16: lane holds columns c .. c + 3 of row r of the pair of blocks at o
            const int o = l & 16, r = l & 7, c = 4 * ((l >> 3) & 1);
            float *v = T + ((o >> 1) + r) * kMRow + 16;               // in T's zero part
            uint64_t lo = 0, hi = 0;
            row8(N + (o + 8 + r) * kMRow + o, T + o * kMRow + o + c, lo, hi);
            put(v + c, lo, hi);
            __syncwarp();
            lo = hi = 0;
            row8(T + (o + 8 + r) * kMRow + o + 8, v - r * kMRow + c, lo, hi);
            put(T + (o + 8 + r) * kMRow + o + c, lo, hi);
        }
        __syncwarp();
        {   // 32 x 32: lane holds columns c .. c + 7 of row r
            const int r = l & 15, c = 8 * (l >> 4);
            float *v = T + r * kMRow + 16;
            uint64_t y[4] = {0, 0, 0, 0};
#pragma unroll
            for (int s = 0; s < 16; s += 8) {
                row8(N + (16 + r) * kMRow + s, T + s * kMRow + c, y[0], y[1]);
                row8(N + (16 + r) * kMRow + s, T + s * kMRow + c + 4, y[2], y[3]);
            }
            put(v + c, y[0], y[1]);
            put(v + c + 4, y[2], y[3]);
            __syncwarp();
            y[0] = y[1] = y[2] = y[3] = 0;
#pragma unroll
            for (int s = 0; s < 16; s += 8) {
                row8(T + (16 + r) * kMRow + 16 + s, T + s * kMRow + 16 + c, y[0], y[1]);
                row8(T + (16 + r) * kMRow + 16 + s, T + s * kMRow + 16 + c + 4, y[2], y[3]);
            }
            put(T + (16 + r) * kMRow + c, y[0], y[1]);
            put(T + (16 + r) * kMRow + c + 4, y[2], y[3]);
        }
        __syncwarp();
        // The operand T - I: row t = lane, zero from the diagonal on.
#pragma unroll
        for (int s = 0; s < C; s += 4) {
            const float4 x = *(const float4 *)(T + l * kMRow + s);
            put4(smem + kOffT, smem + kOffTl, off32(l, s),
                 make_float4(s < l ? x.x : 0.f, s + 1 < l ? x.y : 0.f, s + 2 < l ? x.z : 0.f, s + 3 < l ? x.w : 0.f));
        }
        fence_async_smem();
        mbar_arrive(&bars[kT]);
    }
    return true;
}

// Warps 0-7: the chain of this CTA's chunks. Warps w and w + 4 share tensor-memory
// lanes 32 (w % 4) ..; lane j = value column (and row of P0's result).
__device__ __forceinline__ bool chain(const Args &a, uint8_t *smem, uint64_t *bars, uint32_t tm) {
    uint8_t *B4 = smem + kOffB4, *B4l = smem + kOffB4l;
    float *A = (float *)(smem + kOffA), *F = (float *)(smem + kOffF);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, quad = w & 3, half = w >> 2;
    const int j = 32 * quad + l;
    const uint32_t tl = tm + ((uint32_t)(32 * quad) << 16);   // this warp's lanes
    uint32_t ph = 0;
    bool ok = true;
    float yv[16], *yp = nullptr;                          // the previous chunk's outputs
    int yn = 0;
    const auto store_y = [&]() {
#pragma unroll
        for (int e = 0; e < 16; e++)
            if (e < yn) yp[(size_t)e * a.Hv * 128] = yv[e];
    };
    for (int item = blockIdx.x; item < a.items; item += gridDim.x) {
        const int b = item / a.Hv, h = item - b * a.Hv;
        float *Sg = a.states + (size_t)item * kN;
        // S^T into tensor memory: this thread's lane j, the 64 key rows of its half.
        {
            float sv[64];
#pragma unroll
            for (int e = 0; e < 64; e++) sv[e] = Sg[(size_t)(64 * half + e) * 128 + j];
            tc::st64(tl + kColS + 64 * half, sv);
#pragma unroll
            for (int e = 0; e < 64; e++) sv[e] = tc::tf32_rest(sv[e]);
            tc::st64(tl + kColSl + 64 * half, sv);
        }
        for (int t0 = 0; t0 < a.T; t0 += C, ph ^= 1u) {
            const int n = min(C, a.T - t0);               // tokens in this chunk (ragged tail)
            const bool last = t0 + C >= a.T;
            const float *V = (const float *)(smem + kOffV) + ph * C * 128;
            const float *gC = (const float *)(smem + kOffGc) + ph * 128;
            const float *bet = (const float *)(smem + kOffBeta) + ph * C;
            // full1 first: its next phase then cannot end before this thread has seen this one
            ok = mbar_wait(&bars[kFull1], ph, a.stall.wait_cycles) && ok;
            if (t0 == 0) tc::wait_st();
            tc::fence_before();
            mbar_arrive(&bars[kReady]);
            if (t0 > 0) {                                 // the state's rest, under P1's first half
                float sv[64];
                tc::ld64(tl + kColS + 64 * half, sv);
#pragma unroll
                for (int e = 0; e < 64; e++) sv[e] = tc::tf32_rest(sv[e]);
                tc::st64(tl + kColSl + 64 * half, sv);
                tc::wait_st();
                tc::fence_before();
            }
            mbar_arrive(&bars[kRest]);
            // P0's result, row r = lane: [Q~ ; K~] in lanes 0-63, its rests in 64-127;
            // columns s over K^, 32 + s over its rests. This half takes columns
            // 16 half .. +15.
            ok = mbar_wait(&bars[kP0], ph, a.stall.wait_cycles) && ok;
            tc::fence_after();
            float d[16];
            {
                float e[16];
                tc::ld16(tl + kColP0 + 16 * half, d);
                tc::ld16(tl + kColP0 + 32 + 16 * half, e);
#pragma unroll
                for (int s = 0; s < 16; s++) d[s] += e[s];
            }
            if (quad >= 2) {
#pragma unroll
                for (int s = 0; s < 16; s += 4)
                    *(float4 *)&F[(j - 64) * kMRow + 16 * half + s] = make_float4(d[s], d[s + 1], d[s + 2], d[s + 3]);
            }
            tc::fence_before();
            if (group_any(!ok)) return false;
            // Bm = lower (with diagonal) of Q~ K^T (row t = lane t), an operand, and
            // A = strict lower of diag(beta) K~ K^T (row t = lane 32 + t), kept negated.
            if (quad < 2) {
#pragma unroll
                for (int s = 0; s < 16; s += 4) {
                    const float4 f = *(const float4 *)&F[j * kMRow + 16 * half + s];
                    d[s] += f.x;
                    d[s + 1] += f.y;
                    d[s + 2] += f.z;
                    d[s + 3] += f.w;
                }
                if (quad == 1) {
                    const float nb = -bet[l];
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        const int s = 16 * half + e;
                        *(float4 *)&A[l * kMRow + s] =
                            make_float4(s < l ? nb * d[e] : 0.f, s + 1 < l ? nb * d[e + 1] : 0.f,
                                        s + 2 < l ? nb * d[e + 2] : 0.f, s + 3 < l ? nb * d[e + 3] : 0.f);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        const int s = 16 * half + e;
                        put4(B4, B4l, off32(l, s),
                             make_float4(s <= l ? d[e] : 0.f, s + 1 <= l ? d[e + 1] : 0.f,
                                         s + 2 <= l ? d[e + 2] : 0.f, s + 3 <= l ? d[e + 3] : 0.f));
                    }
                    fence_async_smem();
                }
            }
            mbar_arrive(&bars[kA]);
            store_y();
            // R = diag(beta) (V - K~ S_0), tokens 16 half .. +15 of column j, and its rest,
            // in the place of K~ S_0 and its rest.
            ok = mbar_wait(&bars[kP1], ph, a.stall.wait_cycles);
            tc::fence_after();
            float r[16];                                  // W = R + (T - I) R takes R again
            {
                float xl[16];
                tc::ld16(tl + kColX + 16 * half, r);
                tc::ld16(tl + kColXl + 16 * half, xl);
#pragma unroll
                for (int e = 0; e < 16; e++) {
                    const int t = 16 * half + e;
                    r[e] = bet[t] * (V[t * 128 + (j ^ 4 * (t & 7))] - (r[e] + xl[e]));
                    xl[e] = tc::tf32_rest_rn(r[e]);
                }
                tc::st16(tl + kColX + 16 * half, r);
                tc::st16(tl + kColXl + 16 * half, xl);
            }
            tc::wait_st();
            tc::fence_before();
            mbar_arrive(&bars[kRready]);
            // While W = T R forms: S^T <- S^T diag(g_C), key row i scaled by its cumulative gate.
            {
                float sv[64];
                tc::ld64(tl + kColS + 64 * half, sv);
#pragma unroll
                for (int e = 0; e < 64; e += 4) {
                    const float4 g = *(const float4 *)&gC[64 * half + e];
                    sv[e] *= g.x;
                    sv[e + 1] *= g.y;
                    sv[e + 2] *= g.z;
                    sv[e + 3] *= g.w;
                }
                tc::st64(tl + kColS + 64 * half, sv);
            }
            ok = mbar_wait(&bars[kPw], ph, a.stall.wait_cycles) && ok;
            tc::fence_after();
            {
                float x[16], xl[16];
                tc::ld16(tl + kColW + 16 * half, x);
                tc::ld16(tl + kColWl + 16 * half, xl);
#pragma unroll
                for (int e = 0; e < 16; e++) {
                    x[e] = r[e] + (x[e] + xl[e]);
                    xl[e] = tc::tf32_rest_rn(x[e]);
                }
                tc::st16(tl + kColW + 16 * half, x);
                tc::st16(tl + kColWl + 16 * half, xl);
            }
            tc::wait_st();
            tc::fence_before();
            mbar_arrive(&bars[kWready]);
            ok = mbar_wait(&bars[kP2], ph, a.stall.wait_cycles) && ok;
            tc::fence_after();
            // Outputs: tokens 16 half .. 16 half + 15 of column j, stored once the next
            // chunk can start.
            tc::ld16(tl + kColY + 16 * half, yv);
            {
                float yl[16];
                tc::ld16(tl + kColYl + 16 * half, yl);
#pragma unroll
                for (int e = 0; e < 16; e++) yv[e] += yl[e];
            }
            if (last) {                                   // the boundary state back to global memory
                float sv[64];
                tc::ld64(tl + kColS + 64 * half, sv);
#pragma unroll
                for (int e = 0; e < 64; e++) Sg[(size_t)(64 * half + e) * 128 + j] = sv[e];
            }
            yp = a.y + (((size_t)b * a.T + t0 + 16 * half) * a.Hv + h) * 128 + j;
            yn = n - 16 * half;
        }
    }
    store_y();
    return ok;
}

__global__ void __launch_bounds__(kBlock, 1) prefill_kernel(Args a) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = (uint64_t *)(smem + kOffBar);
    uint32_t *tbase = (uint32_t *)(smem + kOffTmem);
    const int tid = threadIdx.x, w = __shfl_sync(0xffffffffu, tid >> 5, 0);   // uniform
    if (w == 0) {
        tc::tmem_alloc(tbase, kCols);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&bars[kReady], kGroup);
        mbar_init(&bars[kFull1], kGroup);
        mbar_init(&bars[kP0], 1);
        mbar_init(&bars[kP1], 1);
        mbar_init(&bars[kWready], kGroup);
        mbar_init(&bars[kFull2], kGroup);
        mbar_init(&bars[kP2], 1);
        mbar_init(&bars[kRest], kGroup);
        mbar_init(&bars[kRready], kGroup);
        mbar_init(&bars[kA], kGroup);
        mbar_init(&bars[kIn], 1);
        mbar_init(&bars[kT], 32);
        mbar_init(&bars[kPw], 1);
        mbar_init(&bars[kDrain], 1);
        mbar_init_fence();
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    griddep_wait();
    griddep_launch();
    const uint32_t tm = *tbase;                            // lane 0, first column
    bool ok = true;
    if (w < 8) {
        tc::regs_inc<kRegsChain>();
        ok = chain(a, smem, bars, tm);
    } else if (w < 16) {
        tc::regs_dec<kRegsProduce>();
        ok = produce(a, smem, bars);
    } else {
        tc::regs_dec<kRegsIssue>();
        if (w == 16) ok = issue_mma(a, smem, bars, tm);
        else if (w == 17) ok = invert(a, smem, bars);
        else if (w == 18) ok = load_qk(a, smem, bars);
    }
    if (!ok) raise_error(a.err, STEPQ_ERR_TIMEOUT);
    __syncwarp();
    tc::fence_before();
    __syncthreads();
    if (w == 0) {
        tc::fence_after();
        tc::tmem_dealloc(tm, kCols);
    }
}

}  // namespace pf

stepq_status launch_prefill(const stepq_config *cfg, const float *q, const float *k, const float *v,
                            const float *beta, const float *gate, int B, int T, float *states, float *y,
                            cudaStream_t s) {
    pf::Args a{};
    a.q = q; a.k = k; a.v = v; a.beta = beta; a.gate = gate;
    a.states = states; a.y = y;
    a.T = T;
    a.Hk = cfg->n_key_heads;
    a.Hv = cfg->n_value_heads;
    a.gate_per_row = cfg->gate_kind == STEPQ_GATE_CHANNEL;
    a.items = B * a.Hv;
    a.err = device_error_word();
    a.stall = stall_knob();
    static SmemOptIn opt;
    const stepq_status st = opt((const void *)pf::prefill_kernel, pf::kSmem);
    if (st != STEPQ_OK) return st;
    // the register shares are taken from what the kernel is launched with
    static std::atomic<int> regs{0};                       // kept once known
    if (regs.load(std::memory_order_relaxed) == 0) {
        cudaFuncAttributes f{};
        const stepq_status e = cuda_status(cudaFuncGetAttributes(&f, (const void *)pf::prefill_kernel));
        if (e != STEPQ_OK) return e;
        regs.store(f.numRegs, std::memory_order_relaxed);
    }
    if (regs.load(std::memory_order_relaxed) < pf::kRegs) return STEPQ_ERR_CUDA;
    int grid = sm_count();
    if (grid > a.items) grid = a.items;
    return launch_overlapped(pf::prefill_kernel, grid, pf::kBlock, pf::kSmem, s, a);
}

}  // namespace stepq
