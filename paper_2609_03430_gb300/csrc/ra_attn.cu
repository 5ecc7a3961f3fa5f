// ra_attn.cu -- GQA split-K flash-decode attention over the per-head caches (sm_103a).
//
// Computes, for every active sequence b and query head qh (KV head h = qh / G),
//     o = sum_i softmax_i(scale * q . k_i) v_i
// over the prompt rows and the cached generated rows of (b, h) -- section 2
// ("Notation"), with the grouped-query sharing of Appendix F.  In the fused
// form the step's new token (Appendix F: appended post-RoPE every step) is the
// last generated row: it is read from the caller's k_new/v_new rows, placed in
// its head's last tile, attended, and written into the cache by the warp that
// consumes that tile.
//
// Work split: every head is cut into tiles of TILE rows (its prompt rows, then
// its generated rows); the tiles of all heads of the launch are laid end to end
// (layer-major, then sequence, then KV head) and cut into equal chunks of W
// tiles, one per warp, so every warp makes the same number of pipeline trips.
// A launch takes one layer, or every layer of a stacked step: its ramp and its
// tail (about 10 us together, during which the memory idles) then come once a
// step instead of once a layer.  36 layers of 174 MB, one launch each: 1340 us
// a step, in one launch 921 us; 64 layers of 8.7 MB: 1747 and 95 us.  A
// warp runs its own pipeline: lane 0 streams the tiles of K and V -- each as
// two 64-channel boxes stored with the 128-byte swizzle -- plus, at the first
// tile of each head piece, the G query rows, into a ring of SPW shared-memory
// stages with 2-D TMA loads completing on per-stage mbarriers; all 32 lanes
// consume.  A head that fits in one chunk is finished in registers.  Otherwise
// each (head, chunk) piece writes an fp32 partial (unnormalised o, running max
// m, sum l) to one of its chunk's two records -- record 1 for the head that
// starts in the chunk and goes on in the next, record 0 for the head that
// began before it -- and the last warp to finish a piece of that head (an
// arrival counter per chunk, that of the head's first) merges all of them.
//
// The narrow build merges inside the CTA first.  Small layers have more warps
// than heads: one sequence's 8 heads of 2.7K rows were 85 one-tile pieces each,
// 177 KB of partials that one warp merged, 20.6 us a layer.  A CTA's warps hold
// consecutive chunks, so their pieces of a head are deposited in shared memory
// and merged there by the last of them; at most two records per CTA (the head it
// shares with the CTA before and the one it shares with the next) go to global
// memory, announced at the CTA's end, and the last CTA merges a head with all
// its threads.  8.5 us a layer of one sequence, 33.1 instead of 36.6 us one of 16.
//
// Equal chunks end unequally: in a stacked launch of 2.6 ms the CTAs of some SMs
// (always the same ones) end 2.7% after the median.  A long stacked launch of the
// wide shape therefore cuts its last 3% of tiles into chunks of 1.5% of a warp's
// share, at least 8 tiles, which warps claim as they finish.  Smaller or more of
// them cut heads into more pieces, whose merges cost what the balance gives.  16
// layers of the Qwen3-32B shape 2817 -> 2767 us (2778 with 1% chunks, 2771 with
// 5% in 2.5% chunks, 2778 with 8% in 2%), 64 layers 10.81 -> 10.54 ms, 36 layers of
// 16 Qwen3-4B-shape sequences 932 -> 915 us.
//
// With the scored comparator's buffers bound, the warp that consumes a head's
// first tile also copies the head's G query rows into the query window, and
// whoever finishes a head records each query's softmax normaliser beside it:
// until the next eviction, the window score needs exactly these normalisers.
//
// Per-warp compute: the contraction of the G query rows with a tile of cache
// rows runs on the tensor cores (mma.sync m16n8k16, bf16 in, fp32 accumulate):
// S = Q K^T takes the query heads as the 16 M rows (G <= 8 used, the rest
// zero) and 8 cache rows per N tile; O += P V reuses the S accumulator
// fragments as the A operand (P rounded to bf16; launches over several layers
// take what the rounding left out as the A rows 8..15, which are otherwise
// zero, into accumulators of their own: see ra_attn_tile.cuh).  Q fragments stay in
// registers for a whole head piece; K and V are read with ldmatrix from TMA
// tiles stored with the 128-byte swizzle, so the reads are bank-conflict free.
// Each lane owns one query head (lane / 4): the softmax statistics need only
// two shuffles per 16 rows, and O needs no cross-lane reduction.  The softmax
// is online in base 2 with the scale folded into one multiply; the running max
// is only raised when a batch exceeds it by more than 2^8 (the result is
// unchanged up to rounding, as softmax is shift invariant), so rescaling the
// accumulators is rare.
//
// The narrow build (RA_ATTN_TRANSPOSED) takes the products transposed, so
// that the 16-row M side holds cache rows and the 8-wide N side the query
// heads: S^T = K Q^T (A = 16 cache rows x 16 channels of K; B = the same Q
// fragments), then O^T += V^T P^T (A = V read transposed; B = P^T, the S^T
// accumulators rounded to bf16 and transposed in registers with movmatrix).
// That is half the products per row.  A lane then holds rows lane / 4 and
// lane / 4 + 8 of a batch for query heads 2 (lane % 4) and 2 (lane % 4) + 1,
// and a raised max needs a reduction over the 8 lanes of a head pair.  On
// small layers, where warps share sub-partitions, it measured 1.5% faster;
// the wide build keeps the other layout, which measured 2-4% faster there.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "ra_attn_tile.cuh"
#include "ra_internal.h"
#include "ra_ptx.cuh"

namespace ra {
namespace {

#if RA_ATTN_CTA_MERGE
constexpr int kSmemBudget = 232448 - 1024 - 256;  // all an SM gives, but the alignment and the statics
#else
constexpr int kSmemBudget = 220 * 1024;
#endif

// Kernel shape: rows per stage (a multiple of 16), stages per warp, warps per CTA
// (one CTA per SM; the warp count is capped by what fits in shared memory).  The library
// builds this file twice, into the namespaces attn_wide (48-row tiles, 4 warps: large
// layers) and attn_narrow (32-row tiles, 6 warps: small layers, finer work split).
#ifndef RA_ATTN_NS
#define RA_ATTN_NS attn_wide
#endif
#ifndef RA_ATTN_TILE
#define RA_ATTN_TILE 48
#endif
#ifndef RA_ATTN_SPW
#define RA_ATTN_SPW 2
#endif
#ifndef RA_ATTN_WARPS
#define RA_ATTN_WARPS 4
#endif
// Contraction layout: 0 = the query heads are the MMA's M rows (the wide shape); 1 = the cache rows
// are, transposed (the narrow shape).  See the comment at the top of the file.
#ifndef RA_ATTN_TRANSPOSED
#define RA_ATTN_TRANSPOSED 0
#endif
// 1: a CTA merges its warps' pieces of a head in shared memory before anything goes to global memory
// (the narrow shape; see the comment at the top of the file).
#define RA_ATTN_CTA_MERGE RA_ATTN_TRANSPOSED

template <int G>
struct Cfg {
    static constexpr int TILE = RA_ATTN_TILE;                                // rows per stage
    static constexpr int HALF_BYTES = TILE * 128;                            // one 64-channel half of K or V
    static constexpr int KV_BYTES = 2 * HALF_BYTES;                          // a K (or V) tile
    static constexpr int STAGE_BYTES = 2 * KV_BYTES;
    static constexpr int SPW = RA_ATTN_SPW;
    // Beside the stages, per warp: the query rows of a piece and the fused new token's K and V rows
    // (unswizzled).  A slot per stage, or with RA_ATTN_CTA_MERGE one per warp (a second piece start or
    // new token among the tiles on the way is then read straight from global memory), which leaves
    // room for the deposits: O (rows DEP_ROW floats apart: no bank conflicts), m and l of a piece.
    static constexpr bool CTA_MERGE = RA_ATTN_CTA_MERGE;
    static constexpr int SLOTS = CTA_MERGE ? 1 : SPW;
    static constexpr int Q_BYTES = G * kRowBytes;
    static constexpr int SLOT_BYTES = Q_BYTES + 2 * kRowBytes;
    static constexpr int DEP_ROW = kHeadDim + 4;
    static constexpr int DEP_FLOATS = G * DEP_ROW + (2 * G + 3) / 4 * 4;
    static constexpr int DEP_BYTES = CTA_MERGE ? DEP_FLOATS * 4 : 0;
    static constexpr int WARP_BYTES = SPW * (STAGE_BYTES + 16 + 8) + SLOTS * SLOT_BYTES + DEP_BYTES;
    static constexpr int WARPS_FIT = kSmemBudget / WARP_BYTES;
    static constexpr int WARPS = WARPS_FIT < RA_ATTN_WARPS ? WARPS_FIT : RA_ATTN_WARPS;
    static constexpr int NSTAGE = WARPS * SPW;
    // [stages][slots][deposits][tile headers][mbarriers]
    static constexpr int SLOT_OFF = NSTAGE * STAGE_BYTES;
    static constexpr int DEP_OFF = SLOT_OFF + WARPS * SLOTS * SLOT_BYTES;
    static constexpr int HDR_OFF = DEP_OFF + WARPS * DEP_BYTES;
    static constexpr int BAR_OFF = HDR_OFF + NSTAGE * 16;
    static constexpr size_t SMEM = 1024 + (size_t)BAR_OFF + NSTAGE * 8;
    static_assert(DEP_BYTES <= STAGE_BYTES && DEP_BYTES % 16 == 0, "a deposit fits a stage");
    // merge layout: LG lanes per query head, MCH channels per lane
    static constexpr int GP = G <= 1 ? 1 : (G <= 2 ? 2 : (G <= 4 ? 4 : 8));
    static constexpr int LG = 32 / GP;
    static constexpr int MCH = kHeadDim / LG;
    static_assert(G >= 1 && G <= 8, "the 16-row MMA holds up to 8 query heads");
    static_assert(TILE % 16 == 0 && TILE <= 256, "whole 16-row MMA batches; TMA box rows <= 256");
    static_assert(kPromptPage % TILE == 0, "a prompt tile lies inside one page");
    static_assert(HALF_BYTES % 1024 == 0, "128-byte-swizzled TMA boxes start 1024-byte aligned");
    static_assert(WARPS >= 2, "shared-memory budget too small");
    static_assert(SMEM + (CTA_MERGE ? 256 : 0) <= 232448, "fits the 227 KB opt-in shared memory of sm_100+");
};

// What a launch does: one layer; one layer with the compaction of the heads in p.compacting; several
// layers.  Instantiations of their own, so that plain launches run code free of the others' branches
// and registers (with the layer walk in it, a layer of one sequence took 6% longer).
constexpr int kModePlain = 0, kModeCompact = 1, kModeStack = 2;

// Tile header flags; the chunk index sits above them (<< kFlagBits).
// kNewest: the tile holds the newest cached row or rows past it.  kQDirect, kNtDirect: the query rows, the new token's rows are read straight from global memory.
constexpr int kFirst = 1, kLast = 2, kNewTok = 4, kHead0 = 8, kCompact = 16, kQDirect = 32, kNtDirect = 64,
              kNewest = 128, kFlagBits = 8;

// Producer-side walk over the warp's chunks (chunks and cursors count tiles).
struct TileIter {
    int chunk;                       // this warp's chunk (-1: not started)
    int f, end;                      // flattened tile cursor and end of the current chunk
    int l, b, h, k;                  // current layer (of the launch), sequence, KV head, tile within the head
    int nt, tp;                      // tiles in the head, prompt tiles among them
    int lp, gen;                     // prompt rows, generated rows (incl. a fused new token)
    bool comp;                       // the head compacts in this launch: its generated rows are the old region's
    long long pbase, grow;           // the head's prompt rows: pbase + page * KVH * kPromptPage + offset; first generated row
    const int32_t* ptab;             // the sequence's page table (null: its pages are page0, page0 + 1, ...)
    int page0;
    int pg_i, pg_cur, pg_next;       // page-table entry i of the current prompt tile, and entry i + 1 (read ahead)
    int reg_hid, reg_next;           // several layers: the head whose region was read ahead, and that region
    bool piece_start;
};

struct TileDesc {
    long long row;  // first cache row of the tile
    int n, hid, flags, chunk;
};

// The sequence of head `hid` of the launch, (layer * B + sequence) * KVH + KV head.
template <int MODE, class PT>
__device__ __forceinline__ int hid_seq(const PT& p, int hid)
{
    const int lb = hid / p.lay.KVH;
    return MODE == kModeStack ? lb % p.lay.B : lb;
}

template <class PT>
__device__ __forceinline__ int seq_head_tiles(const PT& p, int b)
{
    return (p.seq_base[b + 1] - p.seq_base[b]) / p.lay.KVH;
}

// First tile of head `hid` in the launch's tile order, and the head's tiles.
template <int MODE, class PT>
__device__ __forceinline__ long long head_tile0(const PT& p, int hid, int* nth)
{
    const int lb = hid / p.lay.KVH, h = hid - lb * p.lay.KVH;
    const int l = MODE == kModeStack ? lb / p.lay.B : 0, b = lb - l * p.lay.B;
    *nth = seq_head_tiles(p, b);
    return (long long)l * p.layer_tiles + p.seq_base[b] + (long long)h * *nth;
}

template <int MODE, class PT>
__device__ __forceinline__ void enter_head(TileIter& it, const PT& p)
{
    const DevLayout& L = p.lay;
    it.lp = p.seq_lp[it.b];
    it.gen = p.seq_gen[it.b];
    it.tp = (it.lp + p.tile - 1) / p.tile;
    it.pbase = prompt_row(L, p.layer + (MODE == kModeStack ? it.l : 0), 0, it.h, 0);
    it.page0 = p.seq_page0[it.b];
    it.ptab = it.page0 >= 0 ? nullptr : L.pages + (size_t)it.b * L.max_pages;
    it.pg_i = 0;
    if (it.lp > 0) {
        it.pg_cur = it.ptab ? __ldg(it.ptab) : it.page0;
        it.pg_next = it.lp > kPromptPage ? (it.ptab ? __ldg(it.ptab + 1) : it.page0 + 1) : 0;
    }
    it.comp = MODE == kModeCompact && ((p.compacting[it.b >> 5] >> (it.b & 31)) & 1u);
    int reg;
    if (MODE == kModeStack) {  // the next head's region is read one head ahead
        const int hid = (it.l * L.B + it.b) * L.KVH + it.h, last = p.layers * L.B * L.KVH - 1;
        const int32_t* tab = L.region + (size_t)p.layer * L.B * L.KVH;
        reg = it.reg_hid == hid ? it.reg_next : __ldcg(tab + hid);
        it.reg_hid = hid + 1;
        it.reg_next = hid < last ? __ldcg(tab + hid + 1) : 0;
    } else {
        reg = it.comp ? L.plan[(size_t)(it.b * L.KVH + it.h) * (kPlanHeader + L.r)]  // the old region
                      : p.seq_region[it.b] * L.KVH + it.h;
    }
    it.grow = L.gen_row0 + (long long)reg * L.Cmax;
    it.piece_start = true;
}

template <int MODE, class PT>
__device__ void iter_init(TileIter& it, const PT& p, int R0, int R1)
{
    it.f = R0;
    it.end = R1;
    it.reg_hid = -1;
    it.l = MODE == kModeStack ? R0 / p.layer_tiles : 0;
    const int F = R0 - it.l * p.layer_tiles;
    int lo = 0, hi = p.lay.B - 1;  // largest b with seq_base[b] <= F (empty sequences skipped below)
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.seq_base[mid] <= F) lo = mid; else hi = mid - 1;
    }
    int b = lo;
    while (b < p.lay.B && p.seq_base[b + 1] <= F) ++b;
    it.b = b;
    it.nt = seq_head_tiles(p, b);
    const int off = F - p.seq_base[b];
    it.h = off / it.nt;
    it.k = off - it.h * it.nt;
    enter_head<MODE>(it, p);
}

// The chunk that tile `f` of the launch lies in.
template <int MODE, class PT>
__device__ __forceinline__ int chunk_of(const PT& p, long long f)
{
    if (MODE == kModeStack && p.nstatic > 0 && f >= p.tail_tile) return p.nstatic + (int)(f - p.tail_tile) / p.tail_size;
    return (int)(f / p.W);
}

// The warp's next chunk: false once there is none.  One chunk per warp; in a long stacked launch, then
// chunks claimed one by one.
template <int MODE, class PT>
__device__ bool iter_next_chunk(TileIter& it, const PT& p, int warp_id)
{
    if (MODE == kModeStack && p.nstatic > 0 && it.chunk >= 0) {
        int c = 0;
        if ((threadIdx.x & 31) == 0) {
            c = p.nstatic + atomicAdd(p.ticket, 1);
            // every warp (nstatic of them) claims until a claim fails: the last failing one is the launch's last
            if (c == p.nchunks + p.nstatic - 1) *p.ticket = 0;
        }
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= p.nchunks) return false;
        const int R0 = p.tail_tile + (c - p.nstatic) * p.tail_size;
        it.chunk = c;
        iter_init<MODE>(it, p, R0, min(p.total, R0 + p.tail_size));
        return true;
    }
    if (it.chunk >= 0 || warp_id >= p.nchunks) return false;
    it.chunk = warp_id;
    const int R0 = warp_id * p.W;
    iter_init<MODE>(it, p, R0, min(p.total, R0 + p.W));
    return true;
}

template <int MODE, class PT>
__device__ bool iter_next(TileIter& it, const PT& p, TileDesc& d, int warp_id)
{
    if (it.f >= it.end && !iter_next_chunk<MODE>(it, p, warp_id)) return false;
    const int T = p.tile;
    d.flags = (it.piece_start ? kFirst : 0) | (it.k == 0 ? kHead0 : 0);
    if (it.k < it.tp) {  // a prompt tile lies inside one page (kPromptPage is a multiple of T)
        const int p0 = it.k * T, pi = p0 / kPromptPage;
        if (pi != it.pg_i) {  // another page: the next one's entry was read ahead (a chunk may start mid-prompt)
            it.pg_cur = pi == it.pg_i + 1 ? it.pg_next : (it.ptab ? __ldg(it.ptab + pi) : it.page0 + pi);
            it.pg_i = pi;
            it.pg_next = (pi + 1) * kPromptPage < it.lp ? (it.ptab ? __ldg(it.ptab + pi + 1) : it.page0 + pi + 1) : 0;
        }
        d.row = it.pbase + (long long)it.pg_cur * p.lay.KVH * kPromptPage + p0 % kPromptPage;
        d.n = min(T, it.lp - p0);
    } else {
        const int kg = it.k - it.tp;
        d.row = it.grow + (long long)kg * T;
        d.n = min(T, it.gen - kg * T);
        const bool pending = p.k_new && ((p.pending[it.b >> 5] >> (it.b & 31)) & 1u);
        if (pending && kg * T + d.n == it.gen) d.flags |= kNewTok;  // its last row is the step's new token
        if (kg * T + d.n > it.gen - (pending ? 2 : 1)) d.flags |= kNewest;
        if (MODE == kModeCompact && it.comp) d.flags |= kCompact;
    }
    if (it.k + 1 == it.nt || it.f + 1 == it.end) d.flags |= kLast;
    d.hid = ((MODE == kModeStack ? it.l * p.lay.B : 0) + it.b) * p.lay.KVH + it.h;
    d.chunk = it.chunk;
    it.piece_start = false;
    ++it.k;
    ++it.f;
    if (it.k == it.nt && it.f < it.end) {  // next head (skipping finished sequences)
        if (++it.h == p.lay.KVH) {
            it.h = 0;
            do {
                ++it.b;
                if (MODE == kModeStack && it.b == p.lay.B) {  // (only with layers left: it.f < it.end)
                    it.b = 0;
                    ++it.l;
                }
            } while (seq_head_tiles(p, it.b) == 0);
            it.nt = seq_head_tiles(p, it.b);
        }
        it.k = 0;
        enter_head<MODE>(it, p);
    }
    return true;
}

template <int G>
__device__ __forceinline__ uint32_t swz(int j, int c)
{
    return swz_tile<Cfg<G>::HALF_BYTES>(j, c);
}

#if !RA_ATTN_TRANSPOSED
#pragma nv_diag_suppress 550  // d2, d3: the product's padding rows, discarded
// D[16x8] += A[16x16] B[16x8], bf16 inputs, fp32 accumulators.  Only rows 0..7 of A
// (the query heads) are nonzero, so only c0/c1 of the accumulator are kept.
__device__ __forceinline__ void mma_rows8(float& c0, float& c1, uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1)
{
    float d2, d3;
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %11, %12, %13};"
        : "=f"(c0), "=f"(c1), "=f"(d2), "=f"(d3)
        : "r"(a0), "r"(0u), "r"(a2), "r"(0u), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(0.f), "f"(0.f));
    (void)d2;  // rows 8..15 of the product: padding
    (void)d3;
}
#pragma nv_diag_default 550

// The same with all 16 rows: the weights in rows 0..7 (a0, a2), their residuals in rows 8..15 (a1, a3).
__device__ __forceinline__ void mma_rows16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                           uint32_t b1)
{
    const uint32_t a[4] = {a0, a1, a2, a3};
    mma16816(c, a, b0, b1);
}
#endif

// The scored policy's window: the softmax normaliser of query head g of head `hid` at this
// step, as (scale * log2 e, log2 sum_i exp2(scale * log2 e * q.k_i)), beside its query rows.
template <int G, int MODE, class PT>
__device__ __forceinline__ void record_stats(const PT& p, int hid, int g, float lse2)
{
    const int r = p.lay.r;
    int slot = (p.seq_g[hid_seq<MODE>(p, hid)] + p.ring_off) % r;
    if (slot < 0) slot += r;
    p.lay.qstats[(((size_t)p.layer * p.lay.B * p.lay.KVH + hid) * r + slot) * G + g] =
        make_float2(p.qk_scale_log2, lse2);
}

#if !RA_ATTN_CTA_MERGE
// Merge every piece of head `hid` (P chunks from w0 on: record 1 of chunk w0, record 0 of the
// others) into the bf16 output rows of its G query heads.  One warp, two rounds of L2 reads: first every lane
// reads the statistics of its pieces (lane q: piece q, q + 32, ...) and the warp reduces them
// to each query head's max M and normaliser L; then lanes split as (query head g, channel
// group), and for every piece load its max (one address per head: a broadcast) and their
// channels together, so the loads of all pieces are independent.  Partials come from other
// SMs: read through L2.
template <int G, int MODE, class PT>
__device__ void merge_head(const PT& p, int hid, int w0, int P, int lane)
{
    using C = Cfg<G>;
    constexpr int rs = partial_stride(G);
    const float* base = p.partial + (size_t)w0 * 2 * rs;
    auto piece = [&](int q) { return base + (size_t)(q == 0 ? rs : 2 * q * rs); };
    float M[G], Lh[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        M[g] = -INFINITY;
        Lh[g] = 0.f;
    }
    for (int q = lane; q < P; q += 32)
#pragma unroll
        for (int g = 0; g < G; ++g) M[g] = fmaxf(M[g], __ldcg(piece(q) + G * kHeadDim + g));
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) M[g] = fmaxf(M[g], __shfl_xor_sync(0xffffffffu, M[g], o));
    for (int q = lane; q < P; q += 32)
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float* st = piece(q) + G * kHeadDim;
            Lh[g] = fmaf(exp2f(__ldcg(st + g) - M[g]), __ldcg(st + G + g), Lh[g]);
        }
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) Lh[g] += __shfl_xor_sync(0xffffffffu, Lh[g], o);

    const int g = lane / C::LG, sub = lane % C::LG;
    const int gg = g < G ? g : 0;  // lanes of padding heads shadow head 0 (results unused)
    float Mg = M[0], Lg = Lh[0];
#pragma unroll
    for (int k = 1; k < G; ++k)
        if (gg == k) {
            Mg = M[k];
            Lg = Lh[k];
        }
    const int ch0 = sub * C::MCH;
    float4 acc[C::MCH / 4];
#pragma unroll
    for (int j = 0; j < C::MCH / 4; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int q = 0; q < P; ++q) {
        const float* rec = piece(q);
        const float a = exp2f(__ldcg(rec + G * kHeadDim + gg) - Mg);
        const float4* o = reinterpret_cast<const float4*>(rec + gg * kHeadDim + ch0);
#pragma unroll
        for (int k = 0; k < C::MCH / 4; ++k) {
            const float4 v = __ldcg(o + k);
            acc[k].x = fmaf(a, v.x, acc[k].x);
            acc[k].y = fmaf(a, v.y, acc[k].y);
            acc[k].z = fmaf(a, v.z, acc[k].z);
            acc[k].w = fmaf(a, v.w, acc[k].w);
        }
    }
    if (g >= G) return;
    const float inv = 1.f / Lg;
    if (p.qring && sub == 0) record_stats<G, MODE>(p, hid, g, Mg + log2f(Lg));
    uint16_t* out = p.out + ((size_t)hid * G + g) * kHeadDim + ch0;
#pragma unroll
    for (int k = 0; k < C::MCH / 4; ++k) {
        const uint2 w = make_uint2(pack_bf16x2(acc[k].x * inv, acc[k].y * inv), pack_bf16x2(acc[k].z * inv, acc[k].w * inv));
        *reinterpret_cast<uint2*>(out + 4 * k) = w;
    }
}
#else
// The CTA's own merge.  A warp that ends its piece of a head which other warps of the CTA hold too
// deposits it in shared memory; the last of them to do so merges the deposits, into the output or,
// where the head goes on in another CTA, into one of the CTA's two global records (0: the head began
// in an earlier CTA, 1: it starts here).
struct CtaMerge {
    int arrived[8];            // deposits made, by the first warp that holds a piece of the head (one head each)
    int stage[8];              // the stage a warp's last piece ended in
    struct Part {
        int hid, c0, P;        // the record's head, the first CTA that holds a piece, how many do (0: no record)
    } part[2];
    int last[2];
};

// Where a warp deposits: its last piece goes to its stage other than `s` (nothing is on the way there any
// more), a piece that ends before its chunk does to the warp's deposit slot.
template <int G>
__device__ __forceinline__ uint8_t* deposit(uint8_t* smem, int warp, bool last_piece, int s)
{
    using C = Cfg<G>;
    static_assert(C::SPW == 2 || !C::CTA_MERGE, "the other stage");
    return last_piece ? smem + (size_t)(warp * C::SPW + (s ^ 1)) * C::STAGE_BYTES : smem + C::DEP_OFF + (size_t)warp * C::DEP_BYTES;
}

// Warps a .. z of the CTA have deposited head `hid`, whose chunks are w0 .. w1.  One warp: lanes split
// as (query head g, channel group).
template <int G, int MODE, class PT>
__device__ void merge_deposits(const PT& p, CtaMerge& cm, uint8_t* smem, int hid, int w0, int w1, int a, int z, int lane)
{
    using C = Cfg<G>;
    const int cta0 = (int)blockIdx.x * C::WARPS;
    const int g = lane / C::LG, sub = lane % C::LG, ch0 = sub * C::MCH;
    if (g < G) {
        auto piece = [&](int w) { return reinterpret_cast<const float*>(deposit<G>(smem, w, cta0 + w < w1, cm.stage[w])); };
        float M = -INFINITY, l = 0.f;
        for (int w = a; w <= z; ++w) M = fmaxf(M, piece(w)[G * C::DEP_ROW + g]);
        float4 acc[C::MCH / 4];
#pragma unroll
        for (int j = 0; j < C::MCH / 4; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int w = a; w <= z; ++w) {
            const float* rec = piece(w);
            const float m = rec[G * C::DEP_ROW + g];
            const float e = m == -INFINITY ? 0.f : exp2f(m - M);  // (a piece whose rows are all evicted weighs nothing)
            l = fmaf(e, rec[G * C::DEP_ROW + G + g], l);
            const float4* o = reinterpret_cast<const float4*>(rec + g * C::DEP_ROW + ch0);
#pragma unroll
            for (int k = 0; k < C::MCH / 4; ++k) {
                const float4 v = o[k];
                acc[k].x = fmaf(e, v.x, acc[k].x);
                acc[k].y = fmaf(e, v.y, acc[k].y);
                acc[k].z = fmaf(e, v.z, acc[k].z);
                acc[k].w = fmaf(e, v.w, acc[k].w);
            }
        }
        if (w0 >= cta0 && w1 < cta0 + C::WARPS) {  // the whole head is here
            if (p.qring && sub == 0) record_stats<G, MODE>(p, hid, g, M + log2f(l));
            const float inv = 1.f / l;
            uint16_t* out = p.out + ((size_t)hid * G + g) * kHeadDim + ch0;
#pragma unroll
            for (int k = 0; k < C::MCH / 4; ++k)
                *reinterpret_cast<uint2*>(out + 4 * k) = make_uint2(pack_bf16x2(acc[k].x * inv, acc[k].y * inv),
                                                                    pack_bf16x2(acc[k].z * inv, acc[k].w * inv));
        } else {
            float* rec = p.partial + (size_t)(2 * blockIdx.x + (w0 >= cta0 ? 1 : 0)) * partial_stride(G);
#pragma unroll
            for (int k = 0; k < C::MCH / 4; ++k) *reinterpret_cast<float4*>(rec + g * kHeadDim + ch0 + 4 * k) = acc[k];
            if (sub == 0) {
                rec[G * kHeadDim + g] = M;
                rec[G * kHeadDim + G + g] = l;
            }
        }
    }
    if (lane == 0 && (w0 < cta0 || w1 >= cta0 + C::WARPS))
        cm.part[w0 >= cta0 ? 1 : 0] = {hid, w0 / C::WARPS, w1 / C::WARPS - w0 / C::WARPS + 1};
}

// The CTA's end: its records are announced, and where this CTA is the last to hold a piece of a head,
// all its threads merge the head's records, four channels of a query head each, up to eight records
// on the way per thread.  Partials come from other SMs: read through L2.
template <int G, int MODE, class PT>
__device__ void finish_cta(const PT& p, CtaMerge& cm)
{
    using C = Cfg<G>;
    constexpr int rs = partial_stride(G), kBatch = 8;
    __syncthreads();  // the records are written
    if (threadIdx.x < 2) {
        const CtaMerge::Part q = cm.part[threadIdx.x];
        int last = 0;
        if (q.P > 0) {
            __threadfence();
            last = atomicAdd(p.arrive + q.c0, 1) == q.P - 1;
            if (last) {
                p.arrive[q.c0] = 0;  // ready for the next launch
                __threadfence();
            }
        }
        cm.last[threadIdx.x] = last;
    }
    __syncthreads();
#pragma unroll 1
    for (int slot = 0; slot < 2; ++slot) {
        if (!cm.last[slot]) continue;
        const CtaMerge::Part q = cm.part[slot];
        const float* base = p.partial + (size_t)q.c0 * 2 * rs;
        for (int col = threadIdx.x; col < G * (kHeadDim / 4); col += C::WARPS * 32) {
            const int g = col / (kHeadDim / 4), c4 = col % (kHeadDim / 4);
            float M = -INFINITY, l = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int q0 = 0; q0 < q.P; q0 += kBatch) {
                float m[kBatch], s[kBatch], nM = M;
                float4 o[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    m[j] = -INFINITY;
                    s[j] = 0.f;
                    o[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (q0 + j < q.P) {
                        const float* rec = base + (size_t)(q0 + j == 0 ? 1 : 2 * (q0 + j)) * rs;
                        m[j] = __ldcg(rec + G * kHeadDim + g);
                        s[j] = __ldcg(rec + G * kHeadDim + G + g);
                        o[j] = __ldcg(reinterpret_cast<const float4*>(rec + g * kHeadDim) + c4);
                    }
                }
#pragma unroll
                for (int j = 0; j < kBatch; ++j) nM = fmaxf(nM, m[j]);
                if (nM == -INFINITY) {  // no logit in these pieces: all rows evicted, which sum to 0, or NaN, which stays
#pragma unroll
                    for (int j = 0; j < kBatch; ++j) l += s[j];
                    continue;
                }
                const float sc = exp2f(M - nM);
                M = nM;
                l *= sc;
                acc.x *= sc;
                acc.y *= sc;
                acc.z *= sc;
                acc.w *= sc;
#pragma unroll
                for (int j = 0; j < kBatch; ++j) {
                    const float e = exp2f(m[j] - M);
                    l = fmaf(e, s[j], l);
                    acc.x = fmaf(e, o[j].x, acc.x);
                    acc.y = fmaf(e, o[j].y, acc.y);
                    acc.z = fmaf(e, o[j].z, acc.z);
                    acc.w = fmaf(e, o[j].w, acc.w);
                }
            }
            if (p.qring && c4 == 0) record_stats<G, MODE>(p, q.hid, g, M + log2f(l));
            const float inv = 1.f / l;
            *reinterpret_cast<uint2*>(p.out + ((size_t)q.hid * G + g) * kHeadDim + 4 * c4) =
                make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
        }
    }
}
#endif

template <int G, int MODE, int NB>
__global__ void __launch_bounds__(Cfg<G>::WARPS * 32, 1)
    attn_kernel(const __grid_constant__ AttnParamsN<NB> p, const __grid_constant__ CUtensorMap tk,
                const __grid_constant__ CUtensorMap tv)
{
    using C = Cfg<G>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t* wstage = smem + (size_t)warp * C::SPW * C::STAGE_BYTES;
    uint8_t* wslot = smem + C::SLOT_OFF + (size_t)warp * C::SLOTS * C::SLOT_BYTES;
    int4* hdrs = reinterpret_cast<int4*>(smem + C::HDR_OFF) + warp * C::SPW;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF) + warp * C::SPW;

    const int gw = blockIdx.x * C::WARPS + warp;
#if RA_ATTN_CTA_MERGE
    __shared__ CtaMerge cm;
    if (threadIdx.x < 8) cm.arrived[threadIdx.x] = 0;
    if (threadIdx.x < 2) cm.part[threadIdx.x].P = 0;
    __syncthreads();
#else
    if (gw >= p.nchunks) {  // no chunk for this warp
        pdl_wait();
        pdl_launch_dependents();
        return;
    }
#endif

    if (lane == 0) {
        for (int s = 0; s < C::SPW; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
        prefetch_tensormap(&tk);
        prefetch_tensormap(&tv);
    }
    __syncwarp();
    // The cache, the region table and the inputs may come from the previous kernel.  With
    // p.early (the host has checked that the previous kernel writes none of this layer's
    // cache or tables, or only each head's newest cached row) the first tiles' K and V are requested
    // before waiting; the query rows and the new token's row, which the caller may have just
    // produced, come after.
    bool waited = p.early == kEarlyNone;
    if (waited) pdl_wait();

    TileIter it;
    it.chunk = -1;
    it.f = it.end = 0;
    int issued = 0;
    bool q_busy = false, nt_busy = false;  // the warp's only slot holds rows not consumed yet (SLOTS == 1)
    // The caller's rows of a stage: the query rows (first tile of a piece), the new token's row.
    auto issue_inputs = [&](int s) {
        const int4 hd = hdrs[s];
        uint8_t* sl = wslot + (size_t)(s % C::SLOTS) * C::SLOT_BYTES;
        if ((hd.y & (kNewTok | kNtDirect)) == kNewTok) {
            const size_t src = (size_t)hd.z * kHeadDim;
            bulk_load(sl + C::Q_BYTES, p.k_new + src, (uint32_t)kRowBytes, &bars[s]);
            bulk_load(sl + C::Q_BYTES + kRowBytes, p.v_new + src, (uint32_t)kRowBytes, &bars[s]);
        }
        if ((hd.y & (kFirst | kQDirect)) == kFirst)
            bulk_load(sl, p.q + (size_t)hd.z * G * kHeadDim,
                      (uint32_t)C::Q_BYTES, &bars[s]);
    };
    auto issue = [&](int t) -> bool {
        TileDesc d;
        if (!iter_next<MODE>(it, p, d, gw)) return false;
        const int s = t % C::SPW;
        if (!waited && p.early == kEarlyButNewest && (d.flags & kNewest)) {
            waited = true;
            pdl_wait();
            if (lane == 0)
                for (int u = 0; u < t; ++u) issue_inputs(u);
        }
        if (C::SLOTS == 1) {
            if (d.flags & kFirst) {
                if (q_busy) d.flags |= kQDirect;
                q_busy = true;
            }
            if (d.flags & kNewTok) {
                if (nt_busy) d.flags |= kNtDirect;
                nt_busy = true;
            }
        }
        if (lane == 0) {
            uint8_t* st = wstage + (size_t)s * C::STAGE_BYTES;
            hdrs[s] = make_int4(d.n, d.flags | (d.chunk << kFlagBits), d.hid, (int)d.row);
            const bool first = (d.flags & (kFirst | kQDirect)) == kFirst;
            const bool newtok = (d.flags & (kNewTok | kNtDirect)) == kNewTok;
            mbar_arrive_expect_tx(&bars[s], 2u * C::KV_BYTES + (first ? (uint32_t)C::Q_BYTES : 0u) +
                                                (newtok ? 2u * kRowBytes : 0u));
            tma_load_2d(st, &tk, 0, (int)d.row, &bars[s]);
            tma_load_2d(st + C::HALF_BYTES, &tk, kHalfCh, (int)d.row, &bars[s]);
            tma_load_2d(st + C::KV_BYTES, &tv, 0, (int)d.row, &bars[s]);
            tma_load_2d(st + C::KV_BYTES + C::HALF_BYTES, &tv, kHalfCh, (int)d.row, &bars[s]);
            if (waited) issue_inputs(s);
        }
        return true;
    };
    bool more = true;
    for (int t = 0; t < C::SPW && more; ++t) {
        more = issue(t);
        if (more) ++issued;
    }
    if (!waited) {
        waited = true;
        pdl_wait();
        if (lane == 0)
            for (int t = 0; t < issued; ++t) issue_inputs(t);
    }
    pdl_launch_dependents();  // only now: the successor may assume our predecessor has completed

    const int gq = lane >> 2;  // this lane's query head (rows >= G are padding)
    const int tq = lane & 3;
    uint32_t qa[8][2];  // fragments of Q (rows 0..7) for the 8 k-steps of 16 channels (A, or B of Q^T)
#if RA_ATTN_TRANSPOSED
    const int hA = 2 * tq, hB = 2 * tq + 1;  // the query heads of this lane's accumulator columns
    constexpr int RES = MODE != kModeStack ? kResNone : (G <= 4 ? kResCols : kResAcc);
    const int qh = RES == kResCols ? gq & 3 : gq;  // the head whose query rows this lane's fragments hold
    PieceT<RES> acc;
    acc.clear();
#else
    const int mi = lane >> 3, ri = lane & 7;  // ldmatrix: matrix and row this lane addresses
    constexpr bool RES = MODE == kModeStack;  // the weights' residuals count too
    const int qh = gq;
    float O[16][RES ? 4 : 2];  // O[head gq][n-tile * 8 + 2 tq + {0, 1}]; then the residuals'
    float m_run = -INFINITY, l_run = 0.f;
    auto clear = [&] {
        m_run = -INFINITY;
        l_run = 0.f;
#pragma unroll
        for (int nt = 0; nt < 16; ++nt)
#pragma unroll
            for (int e = 0; e < (RES ? 4 : 2); ++e) O[nt][e] = 0.f;
    };
    clear();
#endif

    for (int t = 0; t < issued; ++t) {
        const int s = t % C::SPW;
        if (!mbar_wait_bounded(&bars[s], (uint32_t)((t / C::SPW) & 1), kWaitLimitNs)) {
            // Give up: flag it, let the copies already issued land (bounded), leave.
            if (lane == 0) atomicExch(p.lay.err, kDeviceErrTimeout);
            for (int u = t + 1; u < issued; ++u)
                (void)mbar_wait_bounded(&bars[u % C::SPW], (uint32_t)((u / C::SPW) & 1), kWaitLimitNs);
#if RA_ATTN_CTA_MERGE
            break;  // (to the CTA's last barrier)
#else
            return;
#endif
        }
        const int4 hd = hdrs[s];
        const int n = hd.x;
        uint8_t* Ks = wstage + (size_t)s * C::STAGE_BYTES;
        uint8_t* Vs = Ks + C::KV_BYTES;
        const uint32_t ks = smem_u32(Ks), vs = smem_u32(Vs);
        uint8_t* slot = wslot + (size_t)(s % C::SLOTS) * C::SLOT_BYTES;
        if (hd.y & kFirst) {  // first tile of a head piece: fresh query fragments
            const uint8_t* Qs = slot;
            if (C::SLOTS == 1) {
                if (hd.y & kQDirect) Qs = reinterpret_cast<const uint8_t*>(p.q + (size_t)hd.z * G * kHeadDim);
                else q_busy = false;
            }
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                qa[kk][0] = qh < G ? *reinterpret_cast<const uint32_t*>(Qs + qh * kRowBytes + (16 * kk + 2 * tq) * 2) : 0u;
                qa[kk][1] = qh < G ? *reinterpret_cast<const uint32_t*>(Qs + qh * kRowBytes + (16 * kk + 8 + 2 * tq) * 2) : 0u;
            }
            if ((hd.y & kHead0) && p.qring) {  // the scored policy's window: this step's query rows of the head
                const int r = p.lay.r;
                int slot = (p.seq_g[hid_seq<MODE>(p, hd.z)] + p.ring_off) % r;
                if (slot < 0) slot += r;
                uint4* dst = reinterpret_cast<uint4*>(
                    p.qring + (((size_t)p.layer * p.lay.B * p.lay.KVH + hd.z) * r + slot) * (size_t)(G * kHeadDim));
                for (int i = lane; i < G * 16; i += 32) dst[i] = lds128(Qs + i * 16);
            }
        }
        // A tile of a head that compacts in this launch: which of its rows were evicted (a 64-bit
        // mask, from the ascending list of at most 64 evicted ordinals) and how many before it.
        uint32_t ev_lo = 0u, ev_hi = 0u;
        int ev_before = 0, j0 = 0;
        if (MODE == kModeCompact && (hd.y & kCompact)) {
            const int32_t* plan = p.lay.plan + (size_t)hd.z * (kPlanHeader + p.lay.r);
            const int m = plan[3];
            j0 = (int)((long long)hd.w - p.lay.gen_row0 - (long long)plan[0] * p.lay.Cmax);
            const int e0 = lane < m ? plan[kPlanHeader + lane] - j0 : INT_MAX;
            const int e1 = lane + 32 < m ? plan[kPlanHeader + 32 + lane] - j0 : INT_MAX;
            ev_before = __popc(__ballot_sync(0xffffffffu, e0 < 0)) + __popc(__ballot_sync(0xffffffffu, e1 < 0));
            const uint32_t lo = ((e0 >= 0 && e0 < 32) ? 1u << e0 : 0u) | ((e1 >= 0 && e1 < 32) ? 1u << e1 : 0u);
            const uint32_t hi = ((e0 >= 32 && e0 < 64) ? 1u << (e0 - 32) : 0u) | ((e1 >= 32 && e1 < 64) ? 1u << (e1 - 32) : 0u);
            ev_lo = __reduce_or_sync(0xffffffffu, lo);
            ev_hi = __reduce_or_sync(0xffffffffu, hi);
        }
        if (hd.y & kNewTok) {  // fused append: put the new token in row n-1 of the tile and into the cache
            const int b = hid_seq<MODE>(p, hd.z);
            const int c = lane & 15;
            uint4 v;
            if (C::SLOTS == 1 && (hd.y & kNtDirect)) {
                v = reinterpret_cast<const uint4*>((lane < 16 ? p.k_new : p.v_new) + (size_t)hd.z * kHeadDim)[c];
            } else {
                v = lds128(slot + C::Q_BYTES + (lane >> 4) * kRowBytes + c * 16);
                nt_busy = false;
            }
            *reinterpret_cast<uint4*>((lane < 16 ? Ks : Vs) + swz<G>(n - 1, c)) = v;
            if (!(MODE == kModeCompact && (hd.y & kCompact))) {  // (a compacting head writes it with its survivors)
                const long long row = (long long)hd.w + n - 1;
                reinterpret_cast<uint4*>((lane < 16 ? p.lay.kpool : p.lay.vpool) + row * kHeadDim)[c] = v;
                if (lane == 0) p.lay.pos[row - p.lay.gen_row0] = p.seq_lp[b] + p.seq_g[b];
            }
            __syncwarp();
        }
        if (n < C::TILE) {  // rows past the valid ones hold stale data: zero V there so 0 * V stays 0
            const int nb = (n + 15) & ~15;  // only rows inside the last used 16-row batch matter
            for (int idx = lane; idx < (nb - n) * 16; idx += 32) {
                const int j = n + (idx >> 4), c = idx & 15;
                *reinterpret_cast<uint4*>(Vs + swz<G>(j, c)) = make_uint4(0u, 0u, 0u, 0u);
            }
            __syncwarp();
        }

#if RA_ATTN_TRANSPOSED
        attend_tile<C::HALF_BYTES, MODE == kModeCompact>(acc, ks, vs, n, qa, p.qk_scale_log2, ev_lo, ev_hi, lane);

        if (hd.y & kLast) {  // last tile of the piece
            float la, lb;
            acc.add_residuals();
            acc.sum_lanes(la, lb);
            const int hid = hd.z;
            int nth;
            const long long A = head_tile0<MODE>(p, hid, &nth);
            const int w0 = (int)(A / p.W), w1 = (int)((A + nth - 1) / p.W);
            if (w0 == w1) {  // the whole head was this warp's: normalise and write the output
                if (p.qring && gq == 0) {
                    if (hA < G) record_stats<G, MODE>(p, hid, hA, acc.mA + log2f(la));
                    if (hB < G) record_stats<G, MODE>(p, hid, hB, acc.mB + log2f(lb));
                }
                const float iA = 1.f / la, iB = 1.f / lb;
                __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(p.out + (size_t)hid * G * kHeadDim);
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) {
                    const int ch = 16 * mt + gq;
                    if (hA < G) {
                        ob[hA * kHeadDim + ch] = __float2bfloat16_rn(acc.O[mt][0] * iA);
                        ob[hA * kHeadDim + ch + 8] = __float2bfloat16_rn(acc.O[mt][2] * iA);
                    }
                    if (hB < G) {
                        ob[hB * kHeadDim + ch] = __float2bfloat16_rn(acc.O[mt][1] * iB);
                        ob[hB * kHeadDim + ch + 8] = __float2bfloat16_rn(acc.O[mt][3] * iB);
                    }
                }
            } else {
                // a piece: the CTA's chunks of this head are a .. z
                const int chunk = hd.y >> kFlagBits, cta0 = (int)blockIdx.x * C::WARPS;
                const int a = max(w0, cta0), z = min(w1, cta0 + C::WARPS - 1);
                float* rec;
                int rs;
                if (a == z) {  // the only one of this CTA: to global memory
                    rec = p.partial + (size_t)(2 * blockIdx.x + (a == w0 ? 1 : 0)) * partial_stride(G);
                    rs = kHeadDim;
                } else {  // deposited for the CTA's merge
                    rec = reinterpret_cast<float*>(deposit<G>(smem, warp, chunk < w1, s));
                    rs = C::DEP_ROW;
                }
                acc.template store<G>(rec, rs, la, lb, lane);
                if (a == z) {
                    if (lane == 0) cm.part[a == w0 ? 1 : 0] = {hid, w0 / C::WARPS, w1 / C::WARPS - w0 / C::WARPS + 1};
                } else {
                    if (lane == 0 && chunk < w1) cm.stage[warp] = s;
                    __threadfence_block();
                    __syncwarp();
                    int old = 0;
                    if (lane == 0) old = atomicAdd(&cm.arrived[a - cta0], 1);
                    old = __shfl_sync(0xffffffffu, old, 0);
                    if (old == z - a) {  // every other piece of the head in this CTA is deposited
                        __threadfence_block();
                        merge_deposits<G, MODE>(p, cm, smem, hid, w0, w1, a - cta0, z - cta0, lane);
                    }
                }
            }
            acc.clear();
        }
#else
        for (int bs = 0; bs < n; bs += 16) {
            // S = Q K^T for rows bs..bs+15: n-tile 0 = rows bs..bs+7, n-tile 1 = rows bs+8..bs+15
            float s0a = 0.f, s0b = 0.f, s1a = 0.f, s1b = 0.f;
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                uint32_t b[4];
                ldsm_x4(b, ks + swz<G>(bs + (mi >> 1) * 8 + ri, 2 * kk + (mi & 1)));
                mma_rows8(s0a, s0b, qa[kk][0], qa[kk][1], b[0], b[1]);
                mma_rows8(s1a, s1b, qa[kk][0], qa[kk][1], b[2], b[3]);
            }
            // this lane: head gq, rows bs + 2tq + {0,1} and bs + 8 + 2tq + {0,1}
            const int r0 = bs + 2 * tq;
            const float sl = p.qk_scale_log2;
            float sc[4] = {r0 < n ? s0a * sl : -INFINITY, r0 + 1 < n ? s0b * sl : -INFINITY,
                           r0 + 8 < n ? s1a * sl : -INFINITY, r0 + 9 < n ? s1b * sl : -INFINITY};
            if (MODE == kModeCompact && (hd.y & kCompact)) {  // evicted rows get no weight
                const int rr[4] = {r0, r0 + 1, r0 + 8, r0 + 9};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (((rr[e] < 32 ? ev_lo >> rr[e] : ev_hi >> (rr[e] - 32)) & 1u)) sc[e] = -INFINITY;
            }
            float bm = fmaxf(fmaxf(sc[0], sc[1]), fmaxf(sc[2], sc[3]));
            bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 1));
            bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 2));
            const bool need = bm > m_run + kTau;
            if (__any_sync(0xffffffffu, need)) {
                const float m_new = need ? bm : m_run;
                const float a = (m_new == m_run) ? 1.f : exp2f(m_run - m_new);
                l_run *= a;
                m_run = m_new;
#pragma unroll
                for (int nt = 0; nt < 16; ++nt)
#pragma unroll
                    for (int e = 0; e < (RES ? 4 : 2); ++e) O[nt][e] *= a;
            }
            float pr[4];
#pragma unroll
            // masked rows: exp2(-inf) = 0; a compacting head can have a whole batch evicted, with
            // m_run still -inf (the difference would be NaN), so there a masked row weighs 0 outright
            for (int e = 0; e < 4; ++e) pr[e] = (MODE == kModeCompact && sc[e] == -INFINITY) ? 0.f : exp2f(sc[e] - m_run);
            l_run += (pr[0] + pr[1]) + (pr[2] + pr[3]);
            const uint32_t pa0 = pack_bf16x2(pr[0], pr[1]), pa2 = pack_bf16x2(pr[2], pr[3]);
            const uint32_t pa1 = residual_bf16x2(pr[0], pr[1], pa0), pa3 = residual_bf16x2(pr[2], pr[3], pa2);
            // O += P V: 16 n-tiles of 8 channels, k = the 16 rows
#pragma unroll
            for (int np = 0; np < 8; ++np) {
                uint32_t b[4];
                ldsm_x4_t(b, vs + swz<G>(bs + (mi & 1) * 8 + ri, 2 * np + (mi >> 1)));
                if constexpr (RES) {
                    mma_rows16(O[2 * np], pa0, pa1, pa2, pa3, b[0], b[1]);
                    mma_rows16(O[2 * np + 1], pa0, pa1, pa2, pa3, b[2], b[3]);
                } else {
                    mma_rows8(O[2 * np][0], O[2 * np][1], pa0, pa2, b[0], b[1]);
                    mma_rows8(O[2 * np + 1][0], O[2 * np + 1][1], pa0, pa2, b[2], b[3]);
                }
            }
        }

        if (hd.y & kLast) {  // last tile of the piece
            if constexpr (RES) {
#pragma unroll
                for (int nt = 0; nt < 16; ++nt) {
                    O[nt][0] = add_residual(O[nt][0], O[nt][2]);
                    O[nt][1] = add_residual(O[nt][1], O[nt][3]);
                }
            }
            float l = l_run;
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            const int hid = hd.z;
            int nth;
            const long long A = head_tile0<MODE>(p, hid, &nth);
            const int w0 = chunk_of<MODE>(p, A), w1 = chunk_of<MODE>(p, A + nth - 1);
            if (w0 == w1) {  // the whole head was this warp's: normalise and write the output
                if (gq < G) {
                    if (p.qring && tq == 0) record_stats<G, MODE>(p, hid, gq, m_run + log2f(l));
                    const float inv = 1.f / l;
                    uint32_t* out = reinterpret_cast<uint32_t*>(p.out + ((size_t)hid * G + gq) * kHeadDim);
#pragma unroll
                    for (int nt = 0; nt < 16; ++nt) out[nt * 4 + tq] = pack_bf16x2(O[nt][0] * inv, O[nt][1] * inv);
                }
            } else {
                const int chunk = hd.y >> kFlagBits;
                float* rec = p.partial + (size_t)(2 * chunk + (chunk == w0 ? 1 : 0)) * partial_stride(G);
                if (gq < G) {
#pragma unroll
                    for (int nt = 0; nt < 16; ++nt)
                        *reinterpret_cast<float2*>(rec + gq * kHeadDim + nt * 8 + 2 * tq) = make_float2(O[nt][0], O[nt][1]);
                    if (tq == 0) {
                        rec[G * kHeadDim + gq] = m_run;
                        rec[G * kHeadDim + G + gq] = l;
                    }
                }
                __threadfence();
                __syncwarp();
                int old = 0;
                if (lane == 0) old = atomicAdd(p.arrive + w0, 1);
                old = __shfl_sync(0xffffffffu, old, 0);
                if (old == w1 - w0) {  // every other piece of this head is already written
                    __threadfence();
                    merge_head<G, MODE>(p, hid, w0, w1 - w0 + 1, lane);
                    if (lane == 0) p.arrive[w0] = 0;  // ready for the next launch
                }
            }
            clear();
        }
#endif

        if (MODE == kModeCompact && (hd.y & kCompact)) {
            // Compaction fused into the pass: every surviving row of the tile (the new token
            // included) goes from the staged tile to its slot in the new region, ordinal
            // j - (evicted before j); positions follow.  One row per step, 16-byte lanes
            // (0-15: K, 16-31: V).
            const int32_t* plan = p.lay.plan + (size_t)hd.z * (kPlanHeader + p.lay.r);
            const long long drow0 = p.lay.gen_row0 + (long long)plan[1] * p.lay.Cmax;
            const int32_t* spos = p.lay.pos + (size_t)plan[0] * p.lay.Cmax;
            int32_t* dpos = p.lay.pos + (size_t)plan[1] * p.lay.Cmax;
            const int c = lane & 15;
            uint16_t* pool = lane < 16 ? p.lay.kpool : p.lay.vpool;
            const uint8_t* tile = lane < 16 ? Ks : Vs;
            auto evicted = [&](int jj) { return ((jj < 32 ? ev_lo >> jj : ev_hi >> (jj - 32)) & 1u) != 0u; };
            auto dest = [&](int jj) {
                const int below = jj < 32 ? __popc(ev_lo & ((1u << jj) - 1u))
                                          : __popc(ev_lo) + __popc(ev_hi & ((1u << (jj - 32)) - 1u));
                return j0 + jj - ev_before - below;
            };
            for (int jj = 0; jj < n; ++jj) {
                if (evicted(jj)) continue;
                reinterpret_cast<uint4*>(pool + (drow0 + dest(jj)) * kHeadDim)[c] = lds128(tile + swz<G>(jj, c));
            }
            for (int jj = lane; jj < n; jj += 32) {
                if (evicted(jj)) continue;
                const int b = hid_seq<MODE>(p, hd.z);
                const bool newtok = (hd.y & kNewTok) && jj == n - 1;
                dpos[dest(jj)] = newtok ? p.seq_lp[b] + p.seq_g[b] : __ldg(spos + j0 + jj);
            }
        }

        __syncwarp();
        if (more) {
            if (lane == 0) fence_proxy_async_smem();
            more = issue(t + C::SPW);
            if (more) ++issued;
        }
    }
#if RA_ATTN_CTA_MERGE
    finish_cta<G, MODE>(p, cm);
#endif
}

// Active sequences whose heads hold no slot at all (empty prompt, nothing generated)
// attend over nothing: their output rows are zero.
__global__ void __launch_bounds__(256) zero_empty_kernel(const __grid_constant__ AttnParams p)
{
    pdl_wait();
    pdl_launch_dependents();
    const int b = blockIdx.x;
    if (!((p.active[b >> 5] >> (b & 31)) & 1u) || p.seq_base[b + 1] != p.seq_base[b]) return;
    uint16_t* out = p.out + (size_t)b * p.lay.H * kHeadDim;
    for (int i = threadIdx.x; i < p.lay.H * kHeadDim / 8; i += blockDim.x)
        reinterpret_cast<uint4*>(out)[i] = make_uint4(0u, 0u, 0u, 0u);
}

template <int G>
cudaError_t launch_attn_g(const AttnParams& p, const CUtensorMap* tk, const CUtensorMap* tv, int ctas, cudaStream_t s)
{
    using C = Cfg<G>;
    bool compact = false;
    for (int i = 0; i < RA_MAX_BATCH / 32; ++i) compact |= p.compacting[i] != 0u;
    const dim3 grid(ctas), block(C::WARPS * 32);
    if (p.layers == 1 && !compact && p.lay.B <= kSmallBatch) {  // (p.cluster implies it)
        AttnParamsN<kSmallBatch> sp;
        static_cast<AttnScalars&>(sp) = p;
        auto take = [&](auto& to, const auto& from, int n) { std::copy(from, from + n, to); };
        const int B = p.lay.B, words = (B + 31) / 32;
        take(sp.active, p.active, words);
        take(sp.pending, p.pending, words);
        take(sp.seq_base, p.seq_base, B + 1);
        take(sp.seq_gen, p.seq_gen, B);
        take(sp.seq_g, p.seq_g, B);
        take(sp.seq_lp, p.seq_lp, B);
        take(sp.seq_page0, p.seq_page0, B);
        take(sp.seq_region, p.seq_region, B);
        if (p.cluster > 0) return launch_attn_cluster(sp, tk, tv, p.cluster_heads, p.cluster, s);
        return launch_pdl(attn_kernel<G, kModePlain, kSmallBatch>, grid, block, C::SMEM, s, sp, *tk, *tv);
    }
    auto kernel = p.layers > 1 ? attn_kernel<G, kModeStack, RA_MAX_BATCH>
                  : compact    ? attn_kernel<G, kModeCompact, RA_MAX_BATCH>
                               : attn_kernel<G, kModePlain, RA_MAX_BATCH>;
    return launch_pdl(kernel, grid, block, C::SMEM, s, p, *tk, *tv);
}

template <int G>
cudaError_t prepare_g()
{
    auto set = [](auto* kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<G>::SMEM);
    };
    cudaError_t e = set(attn_kernel<G, kModePlain, kSmallBatch>);
    if (e == cudaSuccess) e = set(attn_kernel<G, kModePlain, RA_MAX_BATCH>);
    if (e == cudaSuccess) e = set(attn_kernel<G, kModeCompact, RA_MAX_BATCH>);
    if (e == cudaSuccess) e = set(attn_kernel<G, kModeStack, RA_MAX_BATCH>);
    return e;
}

}  // namespace

namespace RA_ATTN_NS {

int attn_warps_per_cta(int G)
{
    switch (G) {
        case 1: return Cfg<1>::WARPS;
        case 2: return Cfg<2>::WARPS;
        case 3: return Cfg<3>::WARPS;
        case 4: return Cfg<4>::WARPS;
        case 5: return Cfg<5>::WARPS;
        case 6: return Cfg<6>::WARPS;
        case 7: return Cfg<7>::WARPS;
        case 8: return Cfg<8>::WARPS;
    }
    return 0;
}

int attn_tile_rows(int G)
{
    switch (G) {
        case 1: return Cfg<1>::TILE;
        case 2: return Cfg<2>::TILE;
        case 3: return Cfg<3>::TILE;
        case 4: return Cfg<4>::TILE;
        case 5: return Cfg<5>::TILE;
        case 6: return Cfg<6>::TILE;
        case 7: return Cfg<7>::TILE;
        case 8: return Cfg<8>::TILE;
    }
    return 0;
}

cudaError_t attn_prepare(int G)
{
    switch (G) {
        case 1: return prepare_g<1>();
        case 2: return prepare_g<2>();
        case 3: return prepare_g<3>();
        case 4: return prepare_g<4>();
        case 5: return prepare_g<5>();
        case 6: return prepare_g<6>();
        case 7: return prepare_g<7>();
        case 8: return prepare_g<8>();
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_attention(const AttnParams& p, const CUtensorMap* tk, const CUtensorMap* tv, int ctas,
                             cudaStream_t s)
{
    bool any_empty = false;
    for (int b = 0; b < p.lay.B; ++b)
        if (((p.active[b >> 5] >> (b & 31)) & 1u) && p.seq_base[b + 1] == p.seq_base[b]) any_empty = true;
    if (any_empty) {
        cudaError_t e = launch_pdl(zero_empty_kernel, dim3(p.lay.B), dim3(256), 0, s, p);
        if (e != cudaSuccess) return e;
    }
    if (p.total == 0) return cudaSuccess;
    switch (p.lay.G) {
        case 1: return launch_attn_g<1>(p, tk, tv, ctas, s);
        case 2: return launch_attn_g<2>(p, tk, tv, ctas, s);
        case 3: return launch_attn_g<3>(p, tk, tv, ctas, s);
        case 4: return launch_attn_g<4>(p, tk, tv, ctas, s);
        case 5: return launch_attn_g<5>(p, tk, tv, ctas, s);
        case 6: return launch_attn_g<6>(p, tk, tv, ctas, s);
        case 7: return launch_attn_g<7>(p, tk, tv, ctas, s);
        case 8: return launch_attn_g<8>(p, tk, tv, ctas, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace RA_ATTN_NS
}  // namespace ra
