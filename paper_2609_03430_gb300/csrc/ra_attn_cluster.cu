// ra_attn_cluster.cu -- decode attention of a layer of few heads: a thread-block cluster per head (sm_103a).
//
// The same computation as ra_attn.cu (one layer, no compaction inside).  A layer of one sequence has 8
// heads of a few thousand rows: 11 MB, under 2 us of memory time.  What it costs is the chain from one
// layer's end to the next one's: launch, first rows, products, merge.  Splitting such a head over CTAs of
// different SMs through global memory makes that chain long (records, a fence, an atomic, and the last
// CTA reading every record back).  Here the head's CTAs are one cluster: each merges its warps' pieces in
// shared memory and sends every channel slice to the CTA that owns it through distributed shared memory;
// one cluster barrier later each CTA merges its slice and writes the output.  A stage per warp (98 KB
// a CTA, two CTAs per SM) leaves room for the next layer's CTAs beside this layer's, so that their first
// tiles are on the way (p.early) before this layer ends.
// 36 layers of one sequence (8 heads of 2.7K rows) take 203 us instead of 300, a layer of 8 heads of 450 rows
// called on its own 4.0 us instead of 7.9 (device time).  What is left is the chain itself, about 4 us.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "ra_attn_tile.cuh"
#include "ra_internal.h"
#include "ra_ptx.cuh"

namespace ra {
namespace {

constexpr int kTile = 32;                  // the narrow shape's tiles (and tensor maps)
constexpr int kHalf = kTile * 128;         // one 64-channel half of K or V
constexpr int kKv = 2 * kHalf;             // a K (or V) tile
constexpr int kStage = 2 * kKv;
constexpr int kWarps = kClusterWarps;
constexpr int kThreads = kWarps * 32;
constexpr int kMaxCl = 16;
constexpr int kDepRow = kHeadDim + 4;      // a deposit's heads: no bank conflicts
constexpr int kVec = kHeadDim / 4;         // float4 columns of a query head
static_assert(kPromptPage % kTile == 0, "a prompt tile lies inside one page");

template <int G>
struct ClCfg {
    // what a CTA receives: for each column of its slice and each CTA of the cluster, four channels, m and l
    static constexpr int LAND = G * kVec + kMaxCl;  // columns of a slice times CTAs, at most
    static constexpr int LAND_OFF = kWarps * kStage;
    static constexpr int ML_OFF = LAND_OFF + LAND * 16;
    static constexpr int BAR_OFF = ML_OFF + LAND * 8;
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + kWarps * 8;
    static_assert((G * kDepRow + 2 * G) * 4 <= kStage, "a deposit fits the warp's stage");
    static_assert(SMEM <= 113 * 1024, "two CTAs per SM");
};

__device__ __forceinline__ uint32_t cluster_nctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void st_dsmem_f4(uint32_t addr, const float4& v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_dsmem_f2(uint32_t addr, float x, float y)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x), "f"(y) : "memory");
}

using Params = AttnParamsN<kSmallBatch>;

template <int G>
__global__ void __launch_bounds__(kThreads, 2)
    attn_cluster_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap tk,
                        const __grid_constant__ CUtensorMap tv)
{
    using C = ClCfg<G>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const DevLayout& L = p.lay;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint8_t* st = smem + (size_t)warp * kStage;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF) + warp;
    const int CL = (int)cluster_nctarank(), rank = (int)cluster_ctarank();

    if (lane == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        prefetch_tensormap(&tk);
        prefetch_tensormap(&tv);
    }
    __syncwarp();
    cluster_arrive();  // (waited for before the first store into another CTA: they have started by then)

    // the cluster's head: KV head h of the (index / KVH)-th sequence that holds rows
    const int index = (int)blockIdx.x / CL, h = index % L.KVH;
    int b = 0;
    for (int left = index / L.KVH; b < L.B - 1; ++b)
        if (p.seq_base[b + 1] > p.seq_base[b] && left-- == 0) break;
    const int hid = b * L.KVH + h;
    const int nt = (p.seq_base[b + 1] - p.seq_base[b]) / L.KVH;
    const int lp = p.seq_lp[b], gen = p.seq_gen[b], tp = (lp + kTile - 1) / kTile;
    const int W = (nt + CL * kWarps - 1) / (CL * kWarps);  // tiles per warp, in the head's order
    const int t0 = min(nt, (rank * kWarps + warp) * W), t1 = min(nt, t0 + W);
    const long long grow = L.gen_row0 + (long long)(p.seq_region[b] * L.KVH + h) * L.Cmax;
    const bool pending = p.k_new && ((p.pending[b >> 5] >> (b & 31)) & 1u);
    // p.early: no tile, every tile, or (the previous kernel wrote each head's newest cached row) every
    // tile but those that hold that row or lie past it may be requested before the wait
    const int newest = gen - (pending ? 2 : 1);
    auto late = [&](int k) { return p.early == kEarlyNone || (p.early == kEarlyButNewest && k >= tp && (k - tp + 1) * kTile > newest); };
    auto rows = [&](int k) { return k < tp ? min(kTile, lp - k * kTile) : min(kTile, gen - (k - tp) * kTile); };
    auto first_row = [&](int k) -> int {
        if (k >= tp) return (int)(grow + (long long)(k - tp) * kTile);
        const int p0 = k * kTile, pi = p0 / kPromptPage;
        const int page = p.seq_page0[b] >= 0 ? p.seq_page0[b] + pi : __ldg(L.pages + (size_t)b * L.max_pages + pi);
        return (int)(prompt_row(L, p.layer, page, h, p0));
    };
    auto issue = [&](int k) {  // tile k into the warp's stage
        const int row = first_row(k);
        if (lane == 0) {
            mbar_arrive_expect_tx(bar, (uint32_t)kStage);
            tma_load_2d(st, &tk, 0, row, bar);
            tma_load_2d(st + kHalf, &tk, kHalfCh, row, bar);
            tma_load_2d(st + kKv, &tv, 0, row, bar);
            tma_load_2d(st + kKv + kHalf, &tv, kHalfCh, row, bar);
        }
    };
    const bool first_late = t0 < t1 && late(t0);
    if (t0 < t1 && !first_late) issue(t0);
    pdl_wait();
    pdl_launch_dependents();  // only now: the successor may assume our predecessor has completed
    if (first_late) issue(t0);

    const int gq = lane >> 2, tq = lane & 3;
    PieceT<kResNone> acc;
    acc.clear();
    if (t0 < t1) {
        uint32_t qa[8][2];  // the query rows as B fragments of the 8 k-steps
        const uint32_t* Q = reinterpret_cast<const uint32_t*>(p.q + (size_t)hid * G * kHeadDim) + gq * (kHeadDim / 2) + tq;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            qa[kk][0] = gq < G ? Q[8 * kk] : 0u;
            qa[kk][1] = gq < G ? Q[8 * kk + 4] : 0u;
        }
        uint4 fresh = make_uint4(0u, 0u, 0u, 0u);  // the new token's row: lanes 0-15 K, 16-31 V
        if (pending && t1 == nt)
            fresh = reinterpret_cast<const uint4*>((lane < 16 ? p.k_new : p.v_new) + (size_t)hid * kHeadDim)[lane & 15];
        if (t0 == 0 && p.qring) {  // the scored policy's window: this step's query rows of the head
            int slot = (p.seq_g[b] + p.ring_off) % L.r;
            if (slot < 0) slot += L.r;
            const uint4* from = reinterpret_cast<const uint4*>(p.q + (size_t)hid * G * kHeadDim);
            uint4* to = reinterpret_cast<uint4*>(
                p.qring + (((size_t)p.layer * L.B * L.KVH + hid) * L.r + slot) * (size_t)(G * kHeadDim));
            for (int i = lane; i < G * 16; i += 32) to[i] = from[i];
        }
        const uint32_t ks = smem_u32(st), vs = ks + kKv;
        for (int k = t0; k < t1; ++k) {
            if (!mbar_wait_bounded(bar, (uint32_t)((k - t0) & 1), kWaitLimitNs)) {
                if (lane == 0) atomicExch(L.err, kDeviceErrTimeout);
                break;  // (to the barriers that the other warps and CTAs wait at)
            }
            const int n = rows(k);
            if (pending && k == nt - 1) {  // fused append: the tile's last row, and the cache's
                const int c = lane & 15;
                *reinterpret_cast<uint4*>((lane < 16 ? st : st + kKv) + swz_tile<kHalf>(n - 1, c)) = fresh;
                const long long row = grow + gen - 1;
                reinterpret_cast<uint4*>((lane < 16 ? L.kpool : L.vpool) + row * kHeadDim)[c] = fresh;
                if (lane == 0) L.pos[row - L.gen_row0] = lp + p.seq_g[b];
                __syncwarp();
            }
            if (n < kTile) {  // rows past the valid ones hold stale data: zero V there so 0 * V stays 0
                const int nb = (n + 15) & ~15;
                for (int i = lane; i < (nb - n) * 16; i += 32)
                    *reinterpret_cast<uint4*>(st + kKv + swz_tile<kHalf>(n + (i >> 4), i & 15)) = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
            }
            attend_tile<kHalf, false>(acc, ks, vs, n, qa, p.qk_scale_log2, 0u, 0u, lane);
            __syncwarp();
            if (k + 1 < t1) {
                if (lane == 0) fence_proxy_async_smem();
                issue(k + 1);
            }
        }
        // the piece, in the warp's stage (its tiles are consumed)
        float la, lb;
        acc.sum_lanes(la, lb);
        acc.store<G>(reinterpret_cast<float*>(st), kDepRow, la, lb, lane);
    }
    __syncthreads();
    cluster_wait();  // every CTA of the cluster has started

    // the CTA's pieces merged per column (four channels of a query head), each to the CTA that owns the column
    const int per = (G * kVec + CL - 1) / CL;  // columns of a slice
    const int nw = min(kWarps, (max(0, nt - rank * kWarps * W) + W - 1) / W);  // warps that hold a piece
    float4* land = reinterpret_cast<float4*>(smem + C::LAND_OFF);
    float2* land_ml = reinterpret_cast<float2*>(smem + C::ML_OFF);
    if (nw > 0)
        for (int col = tid; col < G * kVec; col += kThreads) {
            const int g = col / kVec, c4 = col % kVec;
            float m[kWarps], M = -INFINITY, l = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                m[w] = w < nw ? reinterpret_cast<const float*>(smem + w * kStage)[G * kDepRow + g] : -INFINITY;
                M = fmaxf(M, m[w]);
            }
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < kWarps; ++w)
                if (w < nw) {
                    const float* rec = reinterpret_cast<const float*>(smem + w * kStage);
                    const float e = exp2f(m[w] - M);
                    l = fmaf(e, rec[G * kDepRow + G + g], l);
                    const float4 v = reinterpret_cast<const float4*>(rec + g * kDepRow)[c4];
                    o.x = fmaf(e, v.x, o.x);
                    o.y = fmaf(e, v.y, o.y);
                    o.z = fmaf(e, v.z, o.z);
                    o.w = fmaf(e, v.w, o.w);
                }
            const int owner = col / per, at = rank * per + (col - owner * per);
            st_dsmem_f4(dsmem_addr(land + at, (uint32_t)owner), o);
            st_dsmem_f2(dsmem_addr(land_ml + at, (uint32_t)owner), M, l);
        }
    __syncwarp();
    cluster_sync();  // every slice is complete; no CTA touches another's memory after it
    const int nr = (nt + W * kWarps - 1) / (W * kWarps);  // CTAs that hold a piece
    // a group of `span` lanes per column, a lane per CTA that sent it (one thread over all of them takes a chain
    // of shared-memory reads, half a microsecond for 14)
    int span = 1;
    while (span < nr) span <<= 1;
    for (int i0 = 0; i0 < per; i0 += kThreads / span) {
        const int i = i0 + tid / span, k = tid & (span - 1), col = rank * per + i;
        const bool mine = i < per && col < G * kVec;
        float m = -INFINITY, l = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (mine && k < nr) {
            const float2 ml = land_ml[k * per + i];
            m = ml.x;
            l = ml.y;
            o = land[k * per + i];
        }
        float M = m;
        for (int d = 1; d < span; d <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, d));
        const float e = m == -INFINITY ? 0.f : exp2f(m - M);
        l *= e;
        o.x *= e;
        o.y *= e;
        o.z *= e;
        o.w *= e;
        for (int d = 1; d < span; d <<= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, d);
            o.x += __shfl_xor_sync(0xffffffffu, o.x, d);
            o.y += __shfl_xor_sync(0xffffffffu, o.y, d);
            o.z += __shfl_xor_sync(0xffffffffu, o.z, d);
            o.w += __shfl_xor_sync(0xffffffffu, o.w, d);
        }
        if (!mine || k > 0) continue;
        const int g = col / kVec, c4 = col % kVec;
        if (p.qring && c4 == 0) {  // the window query's softmax normaliser
            int slot = (p.seq_g[b] + p.ring_off) % L.r;
            if (slot < 0) slot += L.r;
            L.qstats[(((size_t)p.layer * L.B * L.KVH + hid) * L.r + slot) * G + g] = make_float2(p.qk_scale_log2, M + log2f(l));
        }
        const float inv = 1.f / l;
        *reinterpret_cast<uint2*>(p.out + ((size_t)hid * G + g) * kHeadDim + 4 * c4) =
            make_uint2(pack_bf16x2(o.x * inv, o.y * inv), pack_bf16x2(o.z * inv, o.w * inv));
    }
}

cudaLaunchConfig_t cluster_config(int ctas, int cl, size_t smem, cudaStream_t s, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

template <int G>
cudaError_t launch_g(const Params& p, const CUtensorMap* tk, const CUtensorMap* tv, int heads, int cl, cudaStream_t s)
{
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(heads * cl, cl, ClCfg<G>::SMEM, s, attr);
    return cudaLaunchKernelEx(&cfg, attn_cluster_kernel<G>, p, *tk, *tv);
}

template <int G>
cudaError_t prepare_g(int* active)
{
    auto kernel = attn_cluster_kernel<G>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ClCfg<G>::SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    active[0] = 0;
    for (int cl = 1; cl <= kMaxCl; ++cl) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config(cl, cl, ClCfg<G>::SMEM, 0, attr);
        cfg.numAttrs = 1;  // the cluster shape only
        active[cl] = 0;
        if (cudaOccupancyMaxActiveClusters(&active[cl], kernel, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            active[cl] = 0;
        }
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t attn_cluster_prepare(int G, int* active)
{
    switch (G) {
        case 1: return prepare_g<1>(active);
        case 2: return prepare_g<2>(active);
        case 3: return prepare_g<3>(active);
        case 4: return prepare_g<4>(active);
        case 5: return prepare_g<5>(active);
        case 6: return prepare_g<6>(active);
        case 7: return prepare_g<7>(active);
        case 8: return prepare_g<8>(active);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_attn_cluster(const AttnParamsN<kSmallBatch>& p, const CUtensorMap* tk, const CUtensorMap* tv, int heads,
                                int cl, cudaStream_t s)
{
    if (cl < 1 || cl > kMaxCl || heads < 1) return cudaErrorInvalidValue;
    switch (p.lay.G) {
        case 1: return launch_g<1>(p, tk, tv, heads, cl, s);
        case 2: return launch_g<2>(p, tk, tv, heads, cl, s);
        case 3: return launch_g<3>(p, tk, tv, heads, cl, s);
        case 4: return launch_g<4>(p, tk, tv, heads, cl, s);
        case 5: return launch_g<5>(p, tk, tv, heads, cl, s);
        case 6: return launch_g<6>(p, tk, tv, heads, cl, s);
        case 7: return launch_g<7>(p, tk, tv, heads, cl, s);
        case 8: return launch_g<8>(p, tk, tv, heads, cl, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace ra
