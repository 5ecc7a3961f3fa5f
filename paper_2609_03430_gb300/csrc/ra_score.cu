// ra_score.cu -- window attention of the scored comparator on sm_103a.
//
// The comparator ranks a head's eviction candidates by the SnapKV score of
// section 2 ("Baselines as choices of s"): the attention that the window of
// the last r decode queries gives each candidate, summed over the window and
// over the G query heads of the KV group (max-pooling and top-K happen in the
// select kernel).  A window query attends, as at its own decode step, to the
// keys at positions up to its own: the prompt, every candidate, and the first
// u buffer rows, u = its rank in the window.
//
// Between two eviction rounds the cache only grows, so each window query saw
// at its own step exactly the keys it sees now, and the decode attention
// kernel records its softmax normaliser beside it.  The eviction therefore
// needs one pass over the candidate rows only:
//   summation pass (score_sum_tc_kernel<ROWS>)  per triggered (sequence, KV
//       head), the logits of the M = r * G window rows against the candidate
//       tiles, normalised by the recorded normalisers and summed over all M
//       rows: one fp32 score per candidate.  Each CTA holds all M rows, so
//       every candidate's sum is complete inside it -- no atomics, and the
//       result does not depend on the launch shape.  It runs on tcgen05 with
//       the accumulators in tensor memory (see the kernel).
//   restore pass (score_stats_tc_kernel<MQ> + score_merge_kernel)  only when a
//       window is loaded from outside (ra_restore_queries): the normalisers,
//       recomputed over the prompt and the cached rows each query sees (by
//       position), split over chunks of key tiles and merged.
// The contraction of the window rows with the key rows is a dense GEMM
// (M x keys x 128), so both passes run on tcgen05 with the accumulators in
// tensor memory: the summation pass with the keys on the M side (a thread
// holds a key and sums over the window), the restore pass with the window on
// the M side (a thread holds a window row and sums over the keys), so that
// neither needs a reduction across threads.  Rows arrive by 2-D TMA (64-row x
// 64-channel boxes, 128-byte swizzle).  Logits are in base 2 with the scale
// folded in.
#include <cuda.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "ra_internal.h"
#include "ra_ptx.cuh"

namespace ra {
static_assert(kPromptPage % kScoreTile == 0, "a scoring tile of the prompt lies inside one page");
namespace {

constexpr int kHalfBytes = kScoreTile * 128;      // one 64-channel box of a key tile
constexpr uint64_t kWaitLimitNs = 2000000000ull;  // bounded mbarrier waits: 2 s
static_assert(kHalfBytes % 1024 == 0, "128-byte-swizzled TMA boxes start 1024-byte aligned");

// Tiles of one head in the restore pass: its prompt rows, then its c cached generated rows.
__device__ __forceinline__ int head_tiles(int lp, int n_gen, int* tp)
{
    *tp = (lp + kScoreTile - 1) / kScoreTile;
    return *tp + (n_gen + kScoreTile - 1) / kScoreTile;
}

// Restore pass: the decode step whose query sits in window slot `slot` when g tokens have been
// generated (the r latest steps fill the r slots), and how many of the head's c cached generated
// rows (positions pos[0..c), increasing) that query sees: those at positions up to its own.
__device__ __forceinline__ int visible_rows(const int32_t* pos, int c, int lp, int g, int r, int slot)
{
    const int d = ((g - 1 - slot) % r + r) % r;
    const int step = g - d;
    if (step < 1) return 0;  // no such step yet: the slot is never read before a real query fills it
    const int qpos = lp + step - 1;
    // nothing is evicted between two rounds, so the tokens after the query are the newest d cached
    // ones: two reads confirm it (the search's chain of dependent reads takes several microseconds)
    const int guess = max(c - d, 0);
    const int below = guess > 0 ? __ldcg(pos + guess - 1) : INT_MIN, after = guess < c ? __ldcg(pos + guess) : INT_MAX;
    if (below <= qpos && after > qpos) return guess;
    int lo = 0, hi = c;      // first ordinal whose position is after qpos
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldcg(pos + mid) <= qpos) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------------
// Both passes on the 5th-generation tensor cores (tcgen05, accumulators in tensor memory).
//
// Operands are K-major in shared memory with the 128-byte swizzle the TMA copies already produce (rows
// of 128 bytes, 8-row groups 1024 bytes apart, the two 64-channel halves one after the other); a K-step
// of 16 channels advances the descriptors' start address by 32 bytes.  One warp of its own loads key
// tiles and issues products, the others read accumulators: stages and accumulator buffers go round by
// mbarriers, so that neither side waits for the other (issue_tiles).  A CTA's start -- tables, tensor
// memory, 64 KB of window rows -- takes as long as several tiles, so windows of at most 256 rows run
// two CTAs per SM (one key stage and 256 accumulator columns each): one CTA's start, loads and products
// run beside the other's exponentials.
//
// Summation pass.  The product is taken transposed, D = K Q^T: the 128 candidate key rows of a tile are
// the M side of the MMA and the window rows are the N side (up to 256 per instruction), so that TMEM
// lane j holds every window row's logit against key j.  The thread that reads lane j then sums its own
// key's weights exp2(logit * scale_R - lse_R) over its warpgroup's part of the window rows, with no
// reduction across lanes.  Six layers of 10 heads with 4160 candidates and 256 window rows: 42 us with
// one CTA of two warpgroups per SM, 31 us this way.

constexpr int kTcRows = 128;                        // key rows per tile: the MMA's M
constexpr int kTcHalf = kTcRows * 128;              // one 64-channel half of a key tile
constexpr int kTcStage = 2 * kTcHalf;               // a key tile: 128 rows x 256 bytes

template <int ROWS>  // window rows held: r * G padded to a multiple of 128, at most 512
struct TcCfg {
    static constexpr bool TWO = ROWS <= 256;                   // two CTAs per SM
    static constexpr int WGS = TWO ? 2 : 4;                    // warpgroups that sum, each a part of the window rows
    static constexpr int THREADS = (WGS * 4 + 1) * 32;         // and the issuing warp
    static constexpr int NCH = ROWS > 256 ? 2 : 1;             // MMAs per K-step (N <= 256 each)
    static constexpr int NC = ROWS / NCH;                      // N of each MMA
    static constexpr int NST = TWO ? 1 : 2;                    // key tiles on the way
    static constexpr int NBUF = 2 * ROWS <= 256 ? 2 : 1;      // accumulator buffers in TMEM
    static constexpr uint32_t COLS = TWO ? 256u : 512u;        // columns allocated (a power of 2)
    static constexpr int Q_OFF = NST * kTcStage;               // after the key stages
    static constexpr int Q_HALF = ROWS * 128;
    static constexpr int STAT_OFF = Q_OFF + ROWS * kRowBytes;
    static constexpr int RED_OFF = STAT_OFF + 2 * ROWS * 4;    // two tiles' parts, taken in turn
    static constexpr int BAR_OFF = RED_OFF + 2 * WGS * kTcRows * 4;  // full, free (stages), done, read (buffers), TMEM base
    static constexpr int NBAR = 2 * NST + 2 * NBUF;
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + NBAR * 8 + 16;
    static_assert(ROWS % 128 == 0 && ROWS <= 512, "window rows");
    static_assert(NC % 16 == 0 && NC <= 256, "UMMA N for M = 128");
    static_assert(ROWS / WGS % 32 == 0 && NBUF * ROWS <= (int)COLS, "whole reads of the accumulators");
    static_assert(SMEM <= (TWO ? 113 * 1024 : 232448), "one or two CTAs per SM");
};

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // bits 0-13: start address >> 4
    d |= (uint64_t)1 << 16;                            // bits 16-29: leading byte offset (unused here)
    d |= (uint64_t)(1024 >> 4) << 32;                  // bits 32-45: stride byte offset >> 4
    d |= (uint64_t)1 << 46;                            // bits 46-48: fixed 0b001
    d |= (uint64_t)2 << 61;                            // bits 61-63: 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: fp32 accumulate, bf16 A and B, both K-major, M x N.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4)                        // D: f32
           | (1u << 7) | (1u << 10)         // A, B: bf16
           | ((uint32_t)(N >> 3) << 17)     // N / 8
           | ((uint32_t)(M >> 4) << 24);    // M / 16
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int accum)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive fp32 columns of this warp's 32 TMEM lanes (one lane per thread).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// The issuing thread of a scoring CTA: tile i goes through stage i % NST and accumulator buffer i % NBUF.
// load(i) issues the copies of tile i (completing on full[i % NST]), product(i) its MMAs.  A stage is loaded
// again when the products that read it have completed, a buffer written again when its readers have
// arrived on read[].  Every wait is bounded; false after one ran out, with everything issued waited for.
template <int NST, int NBUF, class Load, class Product>
__device__ bool issue_tiles(int ntile, uint64_t* full, uint64_t* sfree, uint64_t* done, uint64_t* read, Load load,
                            Product product)
{
    int loaded = 0, issued = 0;  // tiles whose copies, whose products are issued
    while (loaded < min(NST, ntile)) load(loaded++);
    bool ok = true;
    while (ok && issued < ntile) {
        const int i = issued;
        ok = mbar_wait_bounded(&full[i % NST], (uint32_t)((i / NST) & 1), kWaitLimitNs) &&
             (i < NBUF || mbar_wait_bounded(&read[i % NBUF], (uint32_t)((i / NBUF - 1) & 1), kWaitLimitNs));
        if (!ok) break;
        tmem_fence_after();
        product(i);
        umma_commit(&done[i % NBUF]);
        umma_commit(&sfree[i % NST]);
        ++issued;
        const int old = loaded - NST;  // the tile whose stage the next one takes
        if (loaded < ntile && old <= i - (NST > 1 ? 1 : 0)) {
            ok = mbar_wait_bounded(&sfree[old % NST], (uint32_t)((old / NST) & 1), kWaitLimitNs);
            if (ok) load(loaded++);
        }
    }
    if (!ok) {
        for (int i = max(0, issued - NST); i < issued; ++i)
            (void)mbar_wait_bounded(&sfree[i % NST], (uint32_t)((i / NST) & 1), kWaitLimitNs);
        for (int i = issued; i < loaded; ++i)
            (void)mbar_wait_bounded(&full[i % NST], (uint32_t)((i / NST) & 1), kWaitLimitNs);
    }
    return ok;
}

// A scoring CTA's set-up, by all threads: the accumulators' tensor memory (held until tc_leave) and the barriers.
template <int NST, int NBUF>
__device__ __forceinline__ uint32_t tc_enter(uint64_t* full, uint64_t* sfree, uint64_t* done, uint64_t* read, uint32_t* slot,
                                             uint32_t cols, int readers)
{
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&sfree[i], 1);
        }
        for (int i = 0; i < NBUF; ++i) {
            mbar_init(&done[i], 1);
            mbar_init(&read[i], readers);
        }
        fence_mbar_init();
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    return *slot;
}

__device__ __forceinline__ void tc_leave(uint32_t tmem, uint32_t cols)
{
    __syncwarp();
    tmem_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
    }
}

template <int ROWS>
__global__ void __launch_bounds__(TcCfg<ROWS>::THREADS, TcCfg<ROWS>::TWO ? 2 : 1)
    score_sum_tc_kernel(const __grid_constant__ EvictParams p, const __grid_constant__ CUtensorMap tk,
                        const __grid_constant__ CUtensorMap tw)
{
    using C = TcCfg<ROWS>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);  // stage: key tile (and the window) landed
    uint64_t* sfree = full + C::NST;                                    // stage: the products that read it completed
    uint64_t* mdone = sfree + C::NST;                                   // buffer: a tile's products completed
    uint64_t* bread = mdone + C::NBUF;                                  // buffer: its warps have read it
    float2* s_st = reinterpret_cast<float2*>(smem + C::STAT_OFF);  // (scale, -lse) of each window row
    float* red = reinterpret_cast<float*>(smem + C::RED_OFF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // With p.early everything read here was written by kernels that completed before the predecessor
    // started, and the scores are read only by the successor.
    if (!p.early) {
        pdl_wait();
        pdl_launch_dependents();
    }
    const DevLayout& L = p.lay;
    const int t = blockIdx.y / L.KVH, h = blockIdx.y - t * L.KVH;
    const int b = p.trig[t];
    const int N = p.trig_n[t], M = L.r * L.G;
    const int r_lo = blockIdx.x * p.ch2 * kScoreTile;  // this CTA's candidate rows [r_lo, r_hi)
    if (r_lo >= N) {
        if (p.early) {
            pdl_wait();
            pdl_launch_dependents();
        }
        return;
    }
    const int r_hi = min(N, r_lo + p.ch2 * kScoreTile);
    const int ntile = (r_hi - r_lo + kTcRows - 1) / kTcRows;
    const size_t lbh = ((size_t)(p.layer + blockIdx.z) * L.B + b) * L.KVH + h;
    {  // the normaliser each window query had at its decode step
        const float2* qst = L.qstats + lbh * (size_t)M;
        for (int R = tid; R < ROWS; R += C::THREADS) {
            const float2 f = R < M ? __ldcg(qst + R) : make_float2(0.f, INFINITY);  // padding rows weigh 0
            s_st[R] = make_float2(f.x, -f.y);
        }
    }
    const uint32_t tmem = tc_enter<C::NST, C::NBUF>(full, sfree, mdone, bread, reinterpret_cast<uint32_t*>(bread + C::NBUF),
                                                    C::COLS, C::WGS * 4);
    if (warp == C::WGS * 4) {
        if (lane == 0) {
            prefetch_tensormap(&tk);
            prefetch_tensormap(&tw);
            const long long grow = L.gen_row0 + (long long)L.region[lbh] * L.Cmax;
            const uint32_t idesc = umma_idesc_bf16(kTcRows, C::NC), sbase = smem_u32(smem);
            auto load = [&](int i) {
                uint8_t* st = smem + (size_t)(i % C::NST) * kTcStage;
                uint64_t* bar = &full[i % C::NST];
                const int row = (int)(grow + r_lo + (long long)i * kTcRows);
                // The window rows (row R = slot * G + g) complete with the first key tile; rows past M are
                // another head's (or read as zero): finite, and given no weight.
                mbar_arrive_expect_tx(bar, (uint32_t)kTcStage + (i == 0 ? (uint32_t)(ROWS * kRowBytes) : 0u));
                for (int q = 0; q < kTcRows; q += kScoreTile) {
                    tma_load_2d(st + q * 128, &tk, 0, row + q, bar);
                    tma_load_2d(st + kTcHalf + q * 128, &tk, 64, row + q, bar);
                }
                if (i > 0) return;
                const int row0 = (int)(lbh * (size_t)M);
                for (int rb = 0; rb < ROWS; rb += kScoreTile) {
                    tma_load_2d(smem + C::Q_OFF + rb * 128, &tw, 0, row0 + rb, bar);
                    tma_load_2d(smem + C::Q_OFF + C::Q_HALF + rb * 128, &tw, 64, row0 + rb, bar);
                }
            };
            auto product = [&](int i) {
                const uint32_t d0 = tmem + (uint32_t)((i % C::NBUF) * ROWS);
                const uint32_t a0 = sbase + (uint32_t)((i % C::NST) * kTcStage);
#pragma unroll
                for (int kh = 0; kh < 2; ++kh)        // 64-channel half
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)    // 16-channel K-step inside the half
#pragma unroll
                        for (int c = 0; c < C::NCH; ++c)
                            umma_bf16(d0 + c * C::NC, umma_desc_sw128(a0 + kh * kTcHalf + kk * 32),
                                      umma_desc_sw128(sbase + C::Q_OFF + kh * C::Q_HALF + c * C::NC * 128 + kk * 32), idesc,
                                      (kh | kk) != 0);
            };
            if (!issue_tiles<C::NST, C::NBUF>(ntile, full, sfree, mdone, bread, load, product))
                atomicExch(L.err, kDeviceErrTimeout);
        }
    } else {
        // this thread: key row wq * 32 + lane of a tile, window rows [wg, wg + 1) * ROWS / WGS
        const int wg = warp >> 2, wq = warp & 3;
        float* scores = L.scores + lbh * L.Cmax;
        bool ok = true;
        for (int i = 0; i < ntile; ++i) {
            // (after a wait that ran out the warp only keeps the others' barrier going)
            if (ok && !mbar_wait_bounded(&mdone[i % C::NBUF], (uint32_t)((i / C::NBUF) & 1), kWaitLimitNs)) {
                if (lane == 0) atomicExch(L.err, kDeviceErrTimeout);
                ok = false;
            }
            ok = __all_sync(0xffffffffu, ok);
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
            if (ok) {
                tmem_fence_after();
                const uint32_t tl = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)((i % C::NBUF) * ROWS);
#pragma unroll 1
                for (int c0 = wg * (ROWS / C::WGS); c0 < (wg + 1) * (ROWS / C::WGS); c0 += 32) {
                    uint32_t v[32];
                    tmem_ld32(tl + c0, v);
#pragma unroll
                    for (int j = 0; j < 32; j += 2) {
                        const float4 f = *reinterpret_cast<const float4*>(s_st + c0 + j);  // two rows' (one address: a broadcast)
                        sum[j & 2] += exp2f(fmaf(__uint_as_float(v[j]), f.x, f.y));
                        sum[(j & 2) + 1] += exp2f(fmaf(__uint_as_float(v[j + 1]), f.z, f.w));
                    }
                }
                tmem_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bread[i % C::NBUF]);
            }
            float* part = red + (i & 1) * (C::WGS * kTcRows);
            part[wg * kTcRows + wq * 32 + lane] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            asm volatile("bar.sync 1, %0;" ::"n"(C::WGS * 128) : "memory");  // every part of the tile is summed
            const int row = r_lo + i * kTcRows + tid;
            if (ok && tid < kTcRows && row < r_hi) {
                float all = 0.f;
#pragma unroll
                for (int k = 0; k < C::WGS; ++k) all += part[k * kTcRows + tid];
                scores[row] = all;
            }
        }
    }
    tc_leave(tmem, C::COLS);
    if (p.early) {
        pdl_wait();
        pdl_launch_dependents();
    }
}

// ---------------------------------------------------------------------------------------------
// Restore pass on tcgen05: per window row, (max, sum of exp2) over one chunk of the keys it sees.
//
// D = Q K^T: the window rows are the M side (MQ tiles of 128), the 128 keys of a tile the N side, so
// that a TMEM lane holds one window row's logits and the thread that reads it keeps that row's
// running maximum and sum in registers.  The warpgroups take the M tiles, or parts of the keys of one
// (merged at the end).  A tile is two runs of kScoreTile cache rows (a prompt page holds three).  Bound by
// exp2 (one per logit) and the few instructions around it.  160 heads of 3.3K keys and 256 window rows:
// 167 us with mma.sync and two shuffles per 16 keys of a row; here 85 us with one CTA per SM of two
// warpgroups and a barrier of all threads per tile, 63 us with four warpgroups and the issuing warp,
// 55 us with two such CTAs of two warpgroups.
template <int MQ>
struct StCfg {
    static constexpr bool TWO = MQ <= 2;                       // two CTAs per SM
    static constexpr int WGS = TWO ? 2 : 4;                    // warpgroups that keep statistics
    static constexpr int THREADS = (WGS * 4 + 1) * 32;         // and the issuing warp
    static constexpr int ROWS = 128 * MQ;
    static constexpr int NST = TWO ? 1 : MQ == 3 ? 3 : 2;      // key tiles on the way
    static constexpr int BUF_COLS = kTcRows * MQ;              // columns of one buffer: 128 keys per M tile
    static constexpr int NBUF = MQ == 1 ? 2 : 1;               // accumulator buffers in TMEM
    static constexpr uint32_t COLS = TWO ? 256u : 512u;        // columns allocated (a power of 2)
    static constexpr int PARTS = WGS > MQ ? WGS / MQ : 1;      // warpgroups that share an M tile's keys
    static constexpr int PCOLS = kTcRows / PARTS;
    static constexpr int Q_OFF = NST * kTcStage;               // after the key stages
    static constexpr int Q_HALF = ROWS * 128;
    static constexpr int RED_OFF = Q_OFF + ROWS * kRowBytes;   // statistics of the parts but the first
    static constexpr int BAR_OFF = RED_OFF + MQ * (PARTS - 1) * 128 * 8;  // full, free (stages), done, read (buffers), TMEM base
    static constexpr int NBAR = 2 * NST + 2 * NBUF;
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + NBAR * 8 + 16;
    static_assert(NBUF * BUF_COLS <= (int)COLS && PCOLS % 32 == 0, "tensor memory");
    static_assert(SMEM <= (TWO ? 113 * 1024 : 232448), "one or two CTAs per SM");
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Running (max, sum of exp2) of one row over 32 more logits, of which the first `valid` count.  The maximum
// is raised only past 2^8 (the result is the same up to rounding).
template <bool MASK>
__device__ __forceinline__ void add_stats(const uint32_t (&v)[32], int valid, float sl, float& m, float& l)
{
    float x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = !MASK || j < valid ? __uint_as_float(v[j]) : -INFINITY;
    float c[4] = {x[0], x[1], x[2], x[3]};
#pragma unroll
    for (int j = 4; j < 32; ++j) c[j & 3] = fmaxf(c[j & 3], x[j]);
    const float top = fmaxf(fmaxf(c[0], c[1]), fmaxf(c[2], c[3])) * sl;
    if (top == -INFINITY) return;  // nothing visible
    if (top > m + 8.f) {
        l *= m == -INFINITY ? 0.f : ex2(m - top);
        m = top;
    }
    float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 32; ++j) a[j & 3] += ex2(fmaf(x[j], sl, -m));
    l += (a[0] + a[1]) + (a[2] + a[3]);
}

template <int MQ>
__global__ void __launch_bounds__(StCfg<MQ>::THREADS, StCfg<MQ>::TWO ? 2 : 1)
    score_stats_tc_kernel(const __grid_constant__ EvictParams p, const __grid_constant__ CUtensorMap tk,
                          const __grid_constant__ CUtensorMap tw)
{
    using C = StCfg<MQ>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);  // stage: key tile (and the window) landed
    uint64_t* sfree = full + C::NST;                                    // stage: the products that read it completed
    uint64_t* mdone = sfree + C::NST;                                   // buffer: a tile's products completed
    uint64_t* bread = mdone + C::NBUF;                                  // buffer: its warps have read it
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    pdl_wait();  // the window, the cache and the tables come from earlier kernels
    pdl_launch_dependents();

    const DevLayout& L = p.lay;
    const int t = blockIdx.y / L.KVH, h = blockIdx.y - t * L.KVH;
    const int b = p.trig[t];
    const int N = p.trig_n[t], r = L.r, G = L.G, M = r * G;
    const int lp = L.seq_lp[b];
    int tp;
    const int nt_head = head_tiles(lp, N, &tp);
    const int t0 = blockIdx.x * p.ch1;           // this CTA's runs [t0, t1) of kScoreTile rows
    if (t0 >= nt_head) return;  // (exiting counts as letting the successor start)
    const int t1 = min(t0 + p.ch1, nt_head), ntile = (t1 - t0 + 1) / 2;
    const size_t lbh = ((size_t)p.layer * L.B + b) * L.KVH + h;
    const int reg = L.region[lbh];

    const uint32_t tmem = tc_enter<C::NST, C::NBUF>(full, sfree, mdone, bread, reinterpret_cast<uint32_t*>(bread + C::NBUF),
                                                    C::COLS, MQ * C::PARTS * 4);

    // this thread's window row: lane wq * 32 + lane of M tile q, the keys of part `part`
    const int wg = warp >> 2, wq = warp & 3, q = wg / C::PARTS, part = wg % C::PARTS;
    const int R = q * 128 + wq * 32 + lane;
    float mrow = -INFINITY, lrow = 0.f;
    if (warp == C::WGS * 4) {
        if (lane == 0) {
            const long long pbase = prompt_row(L, p.layer, 0, h, 0);
            const int32_t* ptab = L.pages + (size_t)b * L.max_pages;
            const long long grow = L.gen_row0 + (long long)reg * L.Cmax;
            auto run_row = [&](int k) -> int {  // first cache row of the head's run k
                // (a run of the prompt lies inside one page: kPromptPage is a multiple of kScoreTile)
                return (int)(k < tp ? pbase + (long long)__ldg(ptab + k * kScoreTile / kPromptPage) * L.KVH * kPromptPage +
                                          (k * kScoreTile) % kPromptPage
                                    : grow + (long long)(k - tp) * kScoreTile);
            };
            // Tile i: runs t0 + 2 i and the next, if this CTA has it (else its rows are old ones, whose logits
            // count nothing).  The window rows (row R = slot * G + g) complete with the first tile; rows past M
            // are another head's (or read as zero) and belong to no thread's statistics.
            prefetch_tensormap(&tk);
            prefetch_tensormap(&tw);
            const uint32_t idesc = umma_idesc_bf16(128, kTcRows), sbase = smem_u32(smem);
            auto load = [&](int i) {
                const int k = t0 + 2 * i, n = min(2, t1 - k);
                uint8_t* st = smem + (size_t)(i % C::NST) * kTcStage;
                uint64_t* bar = &full[i % C::NST];
                mbar_arrive_expect_tx(bar, (uint32_t)(n * kScoreTile * kRowBytes) + (i == 0 ? (uint32_t)(C::ROWS * kRowBytes) : 0u));
                for (int u = 0; u < n; ++u) {
                    const int row = run_row(k + u);
                    tma_load_2d(st + u * kHalfBytes, &tk, 0, row, bar);
                    tma_load_2d(st + kTcHalf + u * kHalfBytes, &tk, 64, row, bar);
                }
                if (i > 0) return;
                const int row0 = (int)(lbh * (size_t)M);
                for (int rb = 0; rb < C::ROWS; rb += kScoreTile) {
                    tma_load_2d(smem + C::Q_OFF + rb * 128, &tw, 0, row0 + rb, bar);
                    tma_load_2d(smem + C::Q_OFF + C::Q_HALF + rb * 128, &tw, 64, row0 + rb, bar);
                }
            };
            auto product = [&](int i) {
                const uint32_t d0 = tmem + (uint32_t)((i % C::NBUF) * C::BUF_COLS);
                const uint32_t b0 = sbase + (uint32_t)((i % C::NST) * kTcStage);
#pragma unroll
                for (int m = 0; m < MQ; ++m)
#pragma unroll
                    for (int kh = 0; kh < 2; ++kh)        // 64-channel half
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)    // 16-channel K-step inside the half
                            umma_bf16(d0 + m * kTcRows,
                                      umma_desc_sw128(sbase + C::Q_OFF + kh * C::Q_HALF + m * 128 * 128 + kk * 32),
                                      umma_desc_sw128(b0 + kh * kTcHalf + kk * 32), idesc, (kh | kk) != 0);
            };
            if (!issue_tiles<C::NST, C::NBUF>(ntile, full, sfree, mdone, bread, load, product))
                atomicExch(L.err, kDeviceErrTimeout);
        }
    } else if (q < MQ) {
        // generated rows the row sees
        const int lim = R < M ? visible_rows(L.pos + (size_t)reg * L.Cmax, N, lp, p.trig_g[t], r, R / G) : 0;
        const float sl = p.qk_scale_log2;  // the scale the restored queries are taken at
        for (int i = 0; i < ntile; ++i) {
            if (!mbar_wait_bounded(&mdone[i % C::NBUF], (uint32_t)((i / C::NBUF) & 1), kWaitLimitNs)) {
                if (lane == 0) atomicExch(L.err, kDeviceErrTimeout);
                break;
            }
            tmem_fence_after();
            const uint32_t tl = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)((i % C::NBUF) * C::BUF_COLS + q * kTcRows);
#pragma unroll 1
            for (int c0 = part * C::PCOLS; c0 < (part + 1) * C::PCOLS; c0 += 32) {
                const int k = t0 + 2 * i + (c0 >> 6);  // the run these columns belong to
                if (k >= t1) break;
                const int valid = (k < tp ? lp - k * kScoreTile : lim - (k - tp) * kScoreTile) - (c0 & 63);
                uint32_t v[32];
                __syncwarp();
                tmem_ld32(tl + c0, v);
                if (__all_sync(0xffffffffu, valid >= 32)) add_stats<false>(v, valid, sl, mrow, lrow);
                else add_stats<true>(v, valid, sl, mrow, lrow);
            }
            tmem_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bread[i % C::NBUF]);
        }
        if (part > 0)
            reinterpret_cast<float2*>(smem + C::RED_OFF)[(q * (C::PARTS - 1) + part - 1) * 128 + wq * 32 + lane] =
                make_float2(mrow, lrow);
    }
    tc_leave(tmem, C::COLS);
    if (warp >= C::WGS * 4 || q >= MQ || part > 0) return;
#pragma unroll
    for (int k = 0; k < C::PARTS - 1; ++k) {
        const float2 o = reinterpret_cast<const float2*>(smem + C::RED_OFF)[(q * (C::PARTS - 1) + k) * 128 + wq * 32 + lane];
        const float mx = fmaxf(mrow, o.x);
        if (mx != -INFINITY)
            lrow = (mrow == -INFINITY ? 0.f : lrow * ex2(mrow - mx)) + (o.x == -INFINITY ? 0.f : o.y * ex2(o.x - mx));
        mrow = mx;
    }
    // this chunk's statistics of every real row
    if (R < M)
        reinterpret_cast<float2*>(L.stats)[((size_t)(b * L.KVH + h) * L.stats_chunks + blockIdx.x) * M + R] = make_float2(mrow, lrow);
}

// Restore pass, last step: merge each window row's chunk statistics into its normaliser.
__global__ void __launch_bounds__(256) score_merge_kernel(const __grid_constant__ EvictParams p)
{
    pdl_wait();
    pdl_launch_dependents();
    const DevLayout& L = p.lay;
    const int t = blockIdx.x / L.KVH, h = blockIdx.x - t * L.KVH;
    const int b = p.trig[t];
    const int M = L.r * L.G;
    int tp;
    const int nch = (head_tiles(L.seq_lp[b], p.trig_n[t], &tp) + p.ch1 - 1) / p.ch1;
    const float* st = L.stats + (size_t)(b * L.KVH + h) * L.stats_chunks * M * 2;
    float2* qst = L.qstats + (((size_t)p.layer * L.B + b) * L.KVH + h) * (size_t)M;
    for (int R = threadIdx.x; R < M; R += blockDim.x) {
        float mx = -INFINITY;
        for (int k = 0; k < nch; ++k) mx = fmaxf(mx, st[((size_t)k * M + R) * 2]);
        float sum = 0.f;
        if (mx != -INFINITY)
            for (int k = 0; k < nch; ++k) {
                const float mk = st[((size_t)k * M + R) * 2];
                if (mk != -INFINITY) sum += st[((size_t)k * M + R) * 2 + 1] * exp2f(mk - mx);
            }
        qst[R] = make_float2(p.qk_scale_log2, mx + log2f(sum));
    }
}

template <int MT>
cudaError_t launch_stats(const EvictParams& p, const CUtensorMap* tk, const CUtensorMap* tq, cudaStream_t s)
{
    const dim3 grid(p.nch1, p.n_trig * p.lay.KVH);
    return launch_pdl(score_stats_tc_kernel<MT>, grid, dim3(StCfg<MT>::THREADS), StCfg<MT>::SMEM, s, p, *tk, *tq);
}

template <int MT>
cudaError_t prepare_mt()
{
    cudaError_t e = cudaFuncSetAttribute(score_stats_tc_kernel<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)StCfg<MT>::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(score_sum_tc_kernel<128 * MT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)TcCfg<128 * MT>::SMEM);
}

template <int MT>
cudaError_t launch_sum_tc(const EvictParams& p, const CUtensorMap* tk, const CUtensorMap* tq, cudaStream_t s)
{
    const dim3 grid(p.nch2, p.n_trig * p.lay.KVH, p.layers);
    return launch_pdl(score_sum_tc_kernel<128 * MT>, grid, dim3(TcCfg<128 * MT>::THREADS), TcCfg<128 * MT>::SMEM, s, p, *tk, *tq);
}

}  // namespace

int score_window_tiles(int M) { return (M + 127) / 128; }

cudaError_t score_prepare()
{
    cudaError_t e;
    if ((e = prepare_mt<1>()) != cudaSuccess) return e;
    if ((e = prepare_mt<2>()) != cudaSuccess) return e;
    if ((e = prepare_mt<3>()) != cudaSuccess) return e;
    return prepare_mt<4>();
}

cudaError_t launch_score_merge(const EvictParams& p, cudaStream_t s)
{
    return launch_pdl(score_merge_kernel, dim3(p.n_trig * p.lay.KVH), dim3(256), 0, s, p);
}

cudaError_t launch_score(const EvictParams& p, int pass, const CUtensorMap* tk, const CUtensorMap* tq, cudaStream_t s)
{
    const int MT = score_window_tiles(p.lay.r * p.lay.G);
    if (pass == 1) {
        switch (MT) {
            case 1: return launch_stats<1>(p, tk, tq, s);
            case 2: return launch_stats<2>(p, tk, tq, s);
            case 3: return launch_stats<3>(p, tk, tq, s);
            case 4: return launch_stats<4>(p, tk, tq, s);
        }
    } else {
        switch (MT) {
            case 1: return launch_sum_tc<1>(p, tk, tq, s);
            case 2: return launch_sum_tc<2>(p, tk, tq, s);
            case 3: return launch_sum_tc<3>(p, tk, tq, s);
            case 4: return launch_sum_tc<4>(p, tk, tq, s);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace ra
