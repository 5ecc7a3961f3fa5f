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

constexpr int kThreads = 512;  // summation pass: four warpgroups
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
// Summation pass on the 5th-generation tensor cores (tcgen05, accumulators in tensor memory).
//
// The product is taken transposed, D = K Q^T: the 128 candidate key rows of a tile are the M
// side of the MMA and the window rows are the N side (up to 256 per instruction), so that TMEM
// lane j holds every window row's logit against key j.  The thread that reads lane j then sums
// its own key's weights exp2(logit * scale_R - lse_R) over the window rows R, with no
// cross-thread reduction; the four warpgroups take a quarter of the window rows each.  Both operands
// are K-major in shared memory with the 128-byte swizzle the TMA copies already produce (rows of
// 128 bytes, 8-row groups 1024 bytes apart, the two 64-channel halves one after the other); a
// K-step of 16 channels advances the descriptors' start address by 32 bytes.  One thread issues
// the MMAs and commits them to an mbarrier.  With a window of at most 256 rows the accumulator
// is double-buffered in TMEM, so the MMAs of tile i + 1 run while tile i's weights are summed.

constexpr int kTcRows = 128;                        // key rows per tile: the MMA's M
constexpr int kTcHalf = kTcRows * 128;              // one 64-channel half of a key tile
constexpr int kTcStage = 2 * kTcHalf;               // a key tile: 128 rows x 256 bytes

template <int ROWS>  // window rows held: r * G padded to a multiple of 128, at most 512
struct TcCfg {
    static constexpr int NCH = ROWS > 256 ? 2 : 1;             // MMAs per K-step (N <= 256 each)
    static constexpr int NC = ROWS / NCH;                      // N of each MMA
    static constexpr int NBUF = 2 * ROWS <= 512 ? 2 : 1;      // accumulator buffers in TMEM (512 columns)
    static constexpr uint32_t COLS = NBUF * ROWS <= 256 ? 256u : 512u;  // columns allocated (a power of 2)
    static constexpr int Q_OFF = 2 * kTcStage;                 // after the two key stages
    static constexpr int Q_HALF = ROWS * 128;
    static constexpr int STAT_OFF = Q_OFF + ROWS * kRowBytes;
    static constexpr int RED_OFF = STAT_OFF + 2 * ROWS * 4;
    static constexpr int BAR_OFF = RED_OFF + kThreads / 128 * kTcRows * 4;  // full[2], mma_done[2], TMEM base
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + 4 * 8 + 16;
    static_assert(ROWS % 128 == 0 && ROWS <= 512, "window rows");
    static_assert(NC % 16 == 0 && NC <= 256, "UMMA N for M = 128");
    static_assert(SMEM <= 232448, "fits the 227 KB opt-in shared memory");
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

template <int ROWS>
__global__ void __launch_bounds__(kThreads, 1) score_sum_tc_kernel(const __grid_constant__ EvictParams p,
                                                                  const __grid_constant__ CUtensorMap tk,
                                                                  const __grid_constant__ CUtensorMap tw)
{
    using C = TcCfg<ROWS>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);  // key tile (and the window) landed
    uint64_t* mdone = full + 2;                                          // the tile's MMAs completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(full + 4);
    float2* s_st = reinterpret_cast<float2*>(smem + C::STAT_OFF);  // (scale, -lse) of each window row
    float* red = reinterpret_cast<float*>(smem + C::RED_OFF);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // As the mma.sync pass: with p.early everything read here was written by kernels that
    // completed before the predecessor started, and the scores are read only by the successor.
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
    const long long grow = L.gen_row0 + (long long)L.region[lbh] * L.Cmax;

    auto issue_tile = [&](int i, uint32_t extra) {  // thread 0: key tile i into stage i % 2
        const int s = i % 2;
        uint8_t* st = smem + (size_t)s * kTcStage;
        const int row = (int)(grow + r_lo + (long long)i * kTcRows);
        mbar_arrive_expect_tx(&full[s], (uint32_t)kTcStage + extra);
        for (int q = 0; q < kTcRows; q += kScoreTile) {
            tma_load_2d(st + q * 128, &tk, 0, row + q, &full[s]);
            tma_load_2d(st + kTcHalf + q * 128, &tk, 64, row + q, &full[s]);
        }
    };
    if (warp == 0) {  // the accumulators' tensor memory (held until the end)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(C::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&mdone[s], 1);
        }
        fence_mbar_init();
        prefetch_tensormap(&tk);
        prefetch_tensormap(&tw);
        // The window rows (row R = slot * G + g) complete on full[0] with the first key tile;
        // rows past M are another head's (or read as zero): finite, and given no weight below.
        issue_tile(0, (uint32_t)(ROWS * kRowBytes));
        const int row0 = (int)(lbh * (size_t)M);
        for (int rb = 0; rb < ROWS; rb += kScoreTile) {
            tma_load_2d(smem + C::Q_OFF + rb * 128, &tw, 0, row0 + rb, &full[0]);
            tma_load_2d(smem + C::Q_OFF + C::Q_HALF + rb * 128, &tw, 64, row0 + rb, &full[0]);
        }
        if (ntile > 1) issue_tile(1, 0u);
    }
    // thread 0's counts of tiles: copies issued, MMAs issued, MMAs waited for
    int n_loaded = min(ntile, 2), n_mma = 0, done = 0;
    {  // the normaliser each window query had at its decode step
        const float2* qst = L.qstats + lbh * (size_t)M;
        for (int R = tid; R < ROWS; R += kThreads) {
            const float2 f = R < M ? __ldcg(qst + R) : make_float2(0.f, INFINITY);  // padding rows weigh 0
            s_st[R] = make_float2(f.x, -f.y);
        }
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t idesc = umma_idesc_bf16(kTcRows, C::NC);
    const uint32_t sbase = smem_u32(smem);

    // Thread 0: the MMAs of tile i into accumulator buffer i % NBUF, committed to mdone[i % 2].
    auto issue_mma = [&](int i) -> bool {
        if (!mbar_wait_bounded(&full[i % 2], (uint32_t)((i / 2) & 1), kWaitLimitNs)) return false;
        tmem_fence_after();
        const uint32_t d0 = tmem + (uint32_t)((i % C::NBUF) * ROWS);
        const uint32_t a0 = sbase + (uint32_t)((i % 2) * kTcStage);
#pragma unroll
        for (int kh = 0; kh < 2; ++kh)        // 64-channel half
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {  // 16-channel K-step inside the half
                const uint64_t ad = umma_desc_sw128(a0 + kh * kTcHalf + kk * 32);
#pragma unroll
                for (int c = 0; c < C::NCH; ++c) {
                    const uint64_t bd = umma_desc_sw128(sbase + C::Q_OFF + kh * C::Q_HALF + c * C::NC * 128 + kk * 32);
                    umma_bf16(d0 + c * C::NC, ad, bd, idesc, (kh | kk) != 0);
                }
            }
        umma_commit(&mdone[i % 2]);
        n_mma = i + 1;
        return true;
    };

    float* scores = L.scores + lbh * L.Cmax;
    constexpr int kWgs = kThreads / 128;
    const int wg = warp >> 2, wq = warp & 3;  // warpgroup (its part of the window rows), TMEM lane quarter
    bool ok = true;
    if (tid == 0) ok = issue_mma(0);
    for (int i = 0; i < ntile; ++i) {
        if (C::NBUF == 2 && tid == 0 && ok && i + 1 < ntile) ok = issue_mma(i + 1);
        const bool got = mbar_wait_bounded(&mdone[i % 2], (uint32_t)((i / 2) & 1), kWaitLimitNs);
        if (!__syncthreads_and(got && ok)) {  // give up together
            if (tid == 0) atomicExch(L.err, kDeviceErrTimeout);
            break;
        }
        done = i + 1;
        tmem_fence_after();
        if (tid == 0 && i + 2 < ntile) {  // the tile's MMAs have read stage i % 2: refill it
            fence_proxy_async_smem();
            issue_tile(i + 2, 0u);
            n_loaded = i + 3;
        }
        // this thread: key row wq * 32 + lane of the tile, window rows [wg, wg + 1) * ROWS / kWgs
        const uint32_t tl = tmem + ((uint32_t)(wq * 32) << 16) + (uint32_t)((i % C::NBUF) * ROWS);
        float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int c0 = wg * (ROWS / kWgs); c0 < (wg + 1) * (ROWS / kWgs); c0 += 32) {
            uint32_t v[32];
            tmem_ld32(tl + c0, v);
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                const float4 f = *reinterpret_cast<const float4*>(s_st + c0 + j);  // two rows' (one address: a broadcast)
                sum[j & 2] += exp2f(fmaf(__uint_as_float(v[j]), f.x, f.y));
                sum[(j & 2) + 1] += exp2f(fmaf(__uint_as_float(v[j + 1]), f.z, f.w));
            }
        }
        red[wg * kTcRows + wq * 32 + lane] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
        tmem_fence_before();
        __syncthreads();  // every part summed; the accumulator buffer is free again
        if (tid < kTcRows) {
            const int row = r_lo + i * kTcRows + tid;
            float all = 0.f;
#pragma unroll
            for (int k = 0; k < kWgs; ++k) all += red[k * kTcRows + tid];
            if (row < r_hi) scores[row] = all;
        }
        if (C::NBUF == 1 && tid == 0 && ok && i + 1 < ntile) {
            tmem_fence_after();
            ok = issue_mma(i + 1);
        }
        __syncthreads();  // red is rewritten by the next tile
    }
    // Leave only with nothing in flight: after a timeout, the MMAs issued but not waited for and
    // the copies issued but not consumed are waited for once more, bounded.
    if (tid == 0) {
        for (int i = done; i < n_mma; ++i) (void)mbar_wait_bounded(&mdone[i % 2], (uint32_t)((i / 2) & 1), kWaitLimitNs);
        for (int i = n_mma; i < n_loaded; ++i) (void)mbar_wait_bounded(&full[i % 2], (uint32_t)((i / 2) & 1), kWaitLimitNs);
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::COLS) : "memory");
    }
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
// running maximum and sum in registers.  Four warpgroups take the M tiles, or parts of the keys of
// one (merged at the end), and a warp of its own loads tiles and issues products, so that neither
// waits for the other: a tile's accumulator is handed back by an mbarrier.  A tile is two runs of
// kScoreTile cache rows (a prompt page holds three); with at most 256 window rows the accumulator is
// double-buffered, and the products of tile i + 1 run while tile i is summed.  Bound by exp2 (one per
// logit) and the few instructions around it, with four warps per scheduler to hide their latency, and
// by a CTA's start (64 KB of window rows).  160 heads of 3.3K keys and 256 window rows: 167 us with
// mma.sync and two shuffles per 16 keys of a row, 85 us with two warpgroups and a barrier of all
// threads per tile, 63 us this way.
constexpr int kStWgs = 4, kStThreads = (kStWgs * 4 + 1) * 32;  // four warpgroups and the issuing warp

template <int MQ>
struct StCfg {
    static constexpr int ROWS = 128 * MQ;
    static constexpr int NST = MQ <= 3 ? 3 : 2;                // key tiles on the way
    static constexpr int NBUF = MQ <= 2 ? 2 : 1;               // accumulator buffers in TMEM
    static constexpr int BUF_COLS = kTcRows * MQ;              // columns of one buffer: 128 keys per M tile
    static constexpr uint32_t COLS = MQ == 1 ? 256u : 512u;    // columns allocated (a power of 2)
    static constexpr int PARTS = MQ <= 2 ? kStWgs / MQ : 1;    // warpgroups that share an M tile's keys
    static constexpr int PCOLS = kTcRows / PARTS;
    static constexpr int Q_OFF = NST * kTcStage;               // after the key stages
    static constexpr int Q_HALF = ROWS * 128;
    static constexpr int RED_OFF = Q_OFF + ROWS * kRowBytes;   // statistics of the parts but the first
    static constexpr int BAR_OFF = RED_OFF + MQ * (PARTS - 1) * 128 * 8;  // full, free (stages), done, read (buffers), TMEM base
    static constexpr int NBAR = 2 * NST + 2 * NBUF;
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + NBAR * 8 + 16;
    static_assert(NBUF * BUF_COLS <= (int)COLS && SMEM <= 232448 && PCOLS % 32 == 0, "tensor and shared memory");
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
__global__ void __launch_bounds__(kStThreads, 1) score_stats_tc_kernel(const __grid_constant__ EvictParams p,
                                                                      const __grid_constant__ CUtensorMap tk,
                                                                      const __grid_constant__ CUtensorMap tw)
{
    using C = StCfg<MQ>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);  // stage: key tile (and the window) landed
    uint64_t* sfree = full + C::NST;                                    // stage: the products that read it completed
    uint64_t* mdone = sfree + C::NST;                                   // buffer: a tile's products completed
    uint64_t* bread = mdone + C::NBUF;                                  // buffer: its warps have read it
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bread + C::NBUF);
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

    if (warp == 0) {  // the accumulators' tensor memory (held until the end)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(C::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < C::NST; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&sfree[i], 1);
        }
        for (int i = 0; i < C::NBUF; ++i) {
            mbar_init(&mdone[i], 1);
            mbar_init(&bread[i], MQ * C::PARTS * 4);
        }
        fence_mbar_init();
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = *tmem_slot;

    // this thread's window row: lane wq * 32 + lane of M tile q, the keys of part `part`
    const int wg = warp >> 2, wq = warp & 3, q = wg / C::PARTS, part = wg % C::PARTS;
    const int R = q * 128 + wq * 32 + lane;
    float mrow = -INFINITY, lrow = 0.f;
    if (warp == kStWgs * 4) {
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
            // Tile i (runs t0 + 2 i and the next, if this CTA has it) into stage i % NST; `extra` bytes of other
            // copies complete on the same barrier.  A missing second run leaves old rows, whose logits count
            // nothing.
            auto issue_tile = [&](int i, uint32_t extra) {
                const int k = t0 + 2 * i, n = min(2, t1 - k);
                uint8_t* st = smem + (size_t)(i % C::NST) * kTcStage;
                uint64_t* bar = &full[i % C::NST];
                mbar_arrive_expect_tx(bar, (uint32_t)(n * kScoreTile * kRowBytes) + extra);
                for (int u = 0; u < n; ++u) {
                    const int row = run_row(k + u);
                    tma_load_2d(st + u * kHalfBytes, &tk, 0, row, bar);
                    tma_load_2d(st + kTcHalf + u * kHalfBytes, &tk, 64, row, bar);
                }
            };
            prefetch_tensormap(&tk);
            prefetch_tensormap(&tw);
            // The window rows (row R = slot * G + g) complete on full[0] with the first key tile; rows past M
            // are another head's (or read as zero) and belong to no thread's statistics.
            issue_tile(0, (uint32_t)(C::ROWS * kRowBytes));
            const int row0 = (int)(lbh * (size_t)M);
            for (int rb = 0; rb < C::ROWS; rb += kScoreTile) {
                tma_load_2d(smem + C::Q_OFF + rb * 128, &tw, 0, row0 + rb, &full[0]);
                tma_load_2d(smem + C::Q_OFF + C::Q_HALF + rb * 128, &tw, 64, row0 + rb, &full[0]);
            }
            int loaded = 1, issued = 0;  // tiles whose copies, whose products are issued
            for (; loaded < min(C::NST, ntile); ++loaded) issue_tile(loaded, 0u);
            const uint32_t idesc = umma_idesc_bf16(128, kTcRows), sbase = smem_u32(smem);
            bool ok = true;
            while (ok && issued < ntile) {
                const int i = issued;
                ok = mbar_wait_bounded(&full[i % C::NST], (uint32_t)((i / C::NST) & 1), kWaitLimitNs) &&
                     (i < C::NBUF || mbar_wait_bounded(&bread[i % C::NBUF], (uint32_t)((i / C::NBUF - 1) & 1), kWaitLimitNs));
                if (!ok) break;
                tmem_fence_after();
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
                umma_commit(&mdone[i % C::NBUF]);
                umma_commit(&sfree[i % C::NST]);
                ++issued;
                if (i >= 1 && loaded < ntile) {  // tile i - 1 + NST into tile i - 1's stage
                    ok = mbar_wait_bounded(&sfree[(i - 1) % C::NST], (uint32_t)(((i - 1) / C::NST) & 1), kWaitLimitNs);
                    if (ok) issue_tile(loaded++, 0u);
                }
            }
            if (!ok) {  // leave only with nothing in flight: everything issued is waited for once more, bounded
                atomicExch(L.err, kDeviceErrTimeout);
                for (int i = max(0, issued - C::NST); i < issued; ++i)
                    (void)mbar_wait_bounded(&sfree[i % C::NST], (uint32_t)((i / C::NST) & 1), kWaitLimitNs);
                for (int i = issued; i < loaded; ++i)
                    (void)mbar_wait_bounded(&full[i % C::NST], (uint32_t)((i / C::NST) & 1), kWaitLimitNs);
            }
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
    __syncwarp();
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
        tmem_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::COLS) : "memory");
    }
    if (warp >= kStWgs * 4 || q >= MQ || part > 0) return;
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
    return launch_pdl(score_stats_tc_kernel<MT>, grid, dim3(kStThreads), StCfg<MT>::SMEM, s, p, *tk, *tq);
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
    return launch_pdl(score_sum_tc_kernel<128 * MT>, grid, dim3(kThreads), TcCfg<128 * MT>::SMEM, s, p, *tk, *tq);
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
