// ra_attn_tile.cuh -- one tile of cache rows against a head's query rows on mma.sync, shared by the
// attention kernels of ra_attn.cu and ra_attn_cluster.cu.
#pragma once

#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "ra_internal.h"
#include "ra_ptx.cuh"

namespace ra {
namespace {

constexpr float kTau = 8.0f;                       // lazy-rescale threshold (log2 units)
constexpr uint64_t kWaitLimitNs = 2000000000ull;   // bounded mbarrier waits: 2 s
constexpr int kHalfCh = 64;                        // channels per swizzled TMA box (128 bytes)

// Byte offset of (row j, 16-byte chunk c of 16) inside a swizzled K or V tile: two boxes of 64
// channels, HALF bytes each; within a box the chunk index is xored with j mod 8.
template <int HALF>
__device__ __forceinline__ uint32_t swz_tile(int j, int c)
{
    return (uint32_t)((c >> 3) * HALF + j * 128 + (((c & 7) ^ (j & 7)) << 4));
}

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// C[16x8] += A[16x16] B[16x8], bf16 inputs, fp32 accumulators (register-only: not volatile, so the
// compiler may interleave independent products).
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Transpose of an 8x8 bf16 matrix held in fragment layout (lane l: row l / 4, columns 2 (l % 4) + {0, 1}).
__device__ __forceinline__ uint32_t movtrans(uint32_t x)
{
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

// What the rounding of two weights to bf16 (w) left out.
__device__ __forceinline__ uint32_t residual_bf16x2(float lo, float hi, uint32_t w)
{
    return pack_bf16x2(lo - bf16lo(w), hi - bf16hi(w));
}
// A sum of products with the residuals, onto that with the rounded weights (an infinite one stays: V's infinities
// times a residual of zero are NaN).
__device__ __forceinline__ float add_residual(float o, float res) { return isinf(o) ? o : o + res; }

// Residuals of the weights.  Weights rounded to bf16 relative to a running maximum are exact where they are the
// maximum, so a head in short pieces loses less than one in long pieces: 64 layers of one sequence, launched one by one
// (a tile per piece), were 2.11e-3 from 64 bits, in one launch 2.33e-3, of which the output's own rounding is
// 1.65e-3.  Launches over several layers therefore multiply V with the residuals too (1.66e-3): in the columns that
// at most four query heads leave free, whose lanes hold the same logits once more (kResCols), else as products of
// their own (kResAcc).  Launches that stream from memory take the same time (36 layers of 16 sequences 902 us, 16 layers
// of the Qwen3-32B shape 2729 and 2731 us); of small stacks, whose time is the chain of a few tiles, those of more than
// four query heads per KV head take 3 to 5% longer (40 layers of 8 heads of 600 rows, G = 8: 24.0 and 25.2 us; G = 4:
// 21.4 and 21.6).
constexpr int kResNone = 0, kResCols = 1, kResAcc = 2;

// The transposed products' running state of a head piece, per lane: O^T (m-tile mt = channels 16 mt..:
// {ch 16 mt + gq: heads hA, hB; ch 16 mt + gq + 8: hA, hB}, gq = lane / 4, hA = 2 (lane % 4), hB = hA + 1), the
// running max and the (lane-partial) sum of the two heads.  kResCols: columns 4 .. 7 are the residuals' of heads 0 .. 3;
// kResAcc: R holds the residuals'.
template <int RES>
struct PieceT {
    float O[8][4];
    float R[RES == kResAcc ? 8 : 1][4];
    float mA, mB, lA, lB;
    __device__ __forceinline__ void clear()
    {
        mA = mB = -INFINITY;
        lA = lB = 0.f;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                O[mt][e] = 0.f;
                if (RES == kResAcc) R[mt][e] = 0.f;
            }
    }
    // The piece's end: the residuals' products into O (kResCols: of the lanes that hold heads 0 .. 3).
    __device__ __forceinline__ void add_residuals()
    {
        if constexpr (RES != kResNone) {
#pragma unroll
            for (int mt = 0; mt < 8; ++mt)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    O[mt][e] = add_residual(O[mt][e], RES == kResAcc ? R[mt][e] : __shfl_xor_sync(0xffffffffu, O[mt][e], 2));
        }
    }
    __device__ __forceinline__ void sum_lanes(float& la, float& lb) const  // over the 8 lanes of a head pair
    {
        la = lA;
        lb = lB;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            la += __shfl_xor_sync(0xffffffffu, la, o);
            lb += __shfl_xor_sync(0xffffffffu, lb, o);
        }
    }
    // O, m and l to a record: heads `stride` floats apart, then m [G], l [G].
    template <int G>
    __device__ __forceinline__ void store(float* rec, int stride, float la, float lb, int lane) const
    {
        const int gq = lane >> 2, hA = 2 * (lane & 3), hB = hA + 1;
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            const int ch = 16 * mt + gq;
            if (hA < G) {
                rec[hA * stride + ch] = O[mt][0];
                rec[hA * stride + ch + 8] = O[mt][2];
            }
            if (hB < G) {
                rec[hB * stride + ch] = O[mt][1];
                rec[hB * stride + ch + 8] = O[mt][3];
            }
        }
        if (gq == 0) {
            if (hA < G) {
                rec[G * stride + hA] = mA;
                rec[G * stride + G + hA] = la;
            }
            if (hB < G) {
                rec[G * stride + hB] = mB;
                rec[G * stride + G + hB] = lb;
            }
        }
    }
};

// S^T = K Q^T of 16 rows from bs on (two accumulator chains), scaled; this lane: rows bs + gq and bs + 8 + gq
// (gq = lane / 4) for heads hA, hB.  Rows from n on, and with MASK those whose bit of ev_hi:ev_lo is set, are
// -infinity.
template <int HALF, bool MASK>
__device__ __forceinline__ void tile_logits(float (&sv)[4], uint32_t ks, int bs, int n, const uint32_t (&qa)[8][2], float sl,
                                            uint32_t ev_lo, uint32_t ev_hi, int lane)
{
    const int gq = lane >> 2, mi = lane >> 3, ri = lane & 7;  // ldmatrix: matrix and row this lane addresses
    float x[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kk = 0; kk < 8; kk += 2) {
        uint32_t a0[4], a1[4];
        ldsm_x4(a0, ks + swz_tile<HALF>(bs + (mi & 1) * 8 + ri, 2 * kk + (mi >> 1)));
        ldsm_x4(a1, ks + swz_tile<HALF>(bs + (mi & 1) * 8 + ri, 2 * kk + 2 + (mi >> 1)));
        mma16816(x, a0, qa[kk][0], qa[kk][1]);
        mma16816(y, a1, qa[kk + 1][0], qa[kk + 1][1]);
    }
    const int r0 = bs + gq, r1 = r0 + 8;
    bool v0 = r0 < n, v1 = r1 < n;
    if (MASK) {
        v0 = v0 && !(((r0 < 32 ? ev_lo >> r0 : ev_hi >> (r0 - 32)) & 1u));
        v1 = v1 && !(((r1 < 32 ? ev_lo >> r1 : ev_hi >> (r1 - 32)) & 1u));
    }
    sv[0] = v0 ? (x[0] + y[0]) * sl : -INFINITY;
    sv[1] = v0 ? (x[1] + y[1]) * sl : -INFINITY;
    sv[2] = v1 ? (x[2] + y[2]) * sl : -INFINITY;
    sv[3] = v1 ? (x[3] + y[3]) * sl : -INFINITY;
}

// The running max of both heads raised where xA, xB (this lane's largest logits) exceed it by more than 2^8.
template <int RES>
__device__ __forceinline__ void raise_max(PieceT<RES>& s, float xA, float xB)
{
    if (!__any_sync(0xffffffffu, xA > s.mA + kTau || xB > s.mB + kTau)) return;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {  // over the 8 lanes that share a head pair
        xA = fmaxf(xA, __shfl_xor_sync(0xffffffffu, xA, o));
        xB = fmaxf(xB, __shfl_xor_sync(0xffffffffu, xB, o));
    }
    const float nA = xA > s.mA + kTau ? xA : s.mA, nB = xB > s.mB + kTau ? xB : s.mB;
    const float aA = (nA == s.mA) ? 1.f : exp2f(s.mA - nA), aB = (nB == s.mB) ? 1.f : exp2f(s.mB - nB);
    s.mA = nA;
    s.mB = nB;
    s.lA *= aA;
    s.lB *= aB;
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
        s.O[mt][0] *= aA;
        s.O[mt][2] *= aA;
        s.O[mt][1] *= aB;
        s.O[mt][3] *= aB;
        if (RES == kResAcc) {
            s.R[mt][0] *= aA;
            s.R[mt][2] *= aA;
            s.R[mt][1] *= aB;
            s.R[mt][3] *= aB;
        }
    }
}

// The weights of 16 rows, added to the sums; P^T as B fragments in b, with kResAcc their residuals' in c.
template <bool MASK, int RES>
__device__ __forceinline__ void tile_weights(PieceT<RES>& s, const float (&sv)[4], uint32_t (&b)[2], uint32_t (&c)[2], int lane)
{
    float pr[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float m = (e & 1) ? s.mB : s.mA;
        pr[e] = (MASK && sv[e] == -INFINITY) ? 0.f : exp2f(sv[e] - m);
    }
    s.lA += pr[0] + pr[2];
    s.lB += pr[1] + pr[3];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t w = pack_bf16x2(pr[2 * i], pr[2 * i + 1]);
        const uint32_t left = RES == kResNone ? 0u : residual_bf16x2(pr[2 * i], pr[2 * i + 1], w);
        b[i] = movtrans(RES == kResCols && (lane & 2) ? left : w);
        if (RES == kResAcc) c[i] = movtrans(left);
    }
}

// O^T += V^T P^T of one m-tile (v: V transposed), and the residuals'.
template <int RES>
__device__ __forceinline__ void add_product(PieceT<RES>& s, int mt, const uint32_t (&v)[4], const uint32_t (&b)[2],
                                            const uint32_t (&c)[2])
{
    mma16816(s.O[mt], v, b[0], b[1]);
    if (RES == kResAcc) mma16816(s.R[mt], v, c[0], c[1]);
}

// n rows of a tile (K at shared address ks, V at vs): S^T = K Q^T, online softmax, O^T += V^T P^T.  qa: the
// head's query rows as B fragments of the 8 k-steps (kResCols: twice, as columns 0 .. 3 and 4 .. 7).  32 rows at a time, so that two batches' products and
// exponentials run beside each other (36 layers of 16 sequences 1167 us, 16 rows at a time; 1152 us this way),
// then 16 for what is left.
template <int HALF, bool MASK, int RES>
__device__ __forceinline__ void attend_tile(PieceT<RES>& s, uint32_t ks, uint32_t vs, int n, const uint32_t (&qa)[8][2], float sl,
                                            uint32_t ev_lo, uint32_t ev_hi, int lane)
{
    const int mi = lane >> 3, ri = lane & 7;
    int bs = 0;
    for (; bs + 16 < n; bs += 32) {
        float s0[4], s1[4];
        tile_logits<HALF, MASK>(s0, ks, bs, n, qa, sl, ev_lo, ev_hi, lane);
        tile_logits<HALF, MASK>(s1, ks, bs + 16, n, qa, sl, ev_lo, ev_hi, lane);
        raise_max(s, fmaxf(fmaxf(s0[0], s0[2]), fmaxf(s1[0], s1[2])), fmaxf(fmaxf(s0[1], s0[3]), fmaxf(s1[1], s1[3])));
        uint32_t b0[2], b1[2], c0[2], c1[2];
        tile_weights<MASK>(s, s0, b0, c0, lane);
        tile_weights<MASK>(s, s1, b1, c1, lane);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            uint32_t v4[4], w4[4];
            ldsm_x4_t(v4, vs + swz_tile<HALF>(bs + (mi >> 1) * 8 + ri, 2 * mt + (mi & 1)));
            ldsm_x4_t(w4, vs + swz_tile<HALF>(bs + 16 + (mi >> 1) * 8 + ri, 2 * mt + (mi & 1)));
            add_product(s, mt, v4, b0, c0);
            add_product(s, mt, w4, b1, c1);
        }
    }
    if (bs < n) {
        float s0[4];
        tile_logits<HALF, MASK>(s0, ks, bs, n, qa, sl, ev_lo, ev_hi, lane);
        raise_max(s, fmaxf(s0[0], s0[2]), fmaxf(s0[1], s0[3]));
        uint32_t b0[2], c0[2];
        tile_weights<MASK>(s, s0, b0, c0, lane);
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            uint32_t v4[4];
            ldsm_x4_t(v4, vs + swz_tile<HALF>(bs + (mi >> 1) * 8 + ri, 2 * mt + (mi & 1)));
            add_product(s, mt, v4, b0, c0);
        }
    }
}

}  // namespace
}  // namespace ra
