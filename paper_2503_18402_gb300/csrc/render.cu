// render.cu -- Eq. 1 compositing per tile (forward) and its adjoint (backward).
//
// Persistent launches over all views: one CTA per resident slot, each taking
// work items from an atomic counter until none are left, so items of very
// different cost balance across the SMs and all views of a batch share one
// launch.  Each warp owns an 8-pixel-wide block of 4*PPT rows of a B x B
// tile, each lane PPT vertically adjacent pixels of one column.  A work item's
// list entries are streamed through shared memory in batches of B*B/PPT
// records (one coalesced 48-byte gather per thread per batch); every staged
// record is then evaluated for the thread's PPT pixels.
//
// Work items.  Without splitting, an item is a whole tile.  A tile's list is
// walked in order, so a tile with a long list is a serial chain that no other
// SM can help with; at low resolution (few tiles, thousands of entries each)
// those chains set the time of the launch.  With splitting, a tile whose list
// is longer than L entries becomes ceil(n/L) chunks of L entries, each its own
// work item.  Eq. 1 composes over chunks: the transmittance in front of
// chunk c is the product of the (1 - alpha) factors of chunks 0..c-1, and the
// colour is the sum of the chunks' contributions.  Three passes keep the
// result that of the sequential rule, early stop included:
//   1. product pass: each chunk but the last computes, per pixel, the product
//      of its (1 - alpha) factors starting from 1, stopping as soon as the
//      product drops below the stop threshold (from then on the pixel has
//      stopped whatever the transmittance in front of the chunk);
//   2. compositing pass: each chunk starts from T_in = product of the earlier
//      chunks' products and applies Eq. 1 with the stop rule exactly; a pixel
//      whose T_in is already below the threshold stopped in an earlier chunk;
//   3. combine: per pixel, the colour sum over chunks, T_final from the chunk
//      where compositing stopped (else the last chunk), last = the largest
//      last of any chunk; and, for the backward, the colour behind each chunk.
// The backward takes the same items: a chunk starts from its own end
// transmittance and the colour behind it instead of T_final and T_final * bg.
// By default lists are split only when the batch has fewer than two tiles per
// resident CTA, with L = max(64, M / resident CTAs); L is raised where needed
// to keep the chunk count within the workspace.
//
//   Forward: front to back; an item stops once every pixel has terminated
//   (__syncthreads_count).
//   Backward: back to front from each pixel's last contributor; the
//   transmittance in front of entry j is recovered as T_j = T_{j+1} / (1 - a_j).
//   A thread first sums its PPT pixels' partial gradients, the warp then sums
//   the nine values by recursive halving (12 shuffles) and nine lanes add the
//   totals with one atomic instruction; warps with no contributing pixel skip
//   the reduction.
// Tile-level skip: while a batch is staged, each entry is tested once against
// the whole tile: the minimum of its quadratic form over the rectangle of the
// tile's pixel centres (closed form on the four edges when the mean lies
// outside).  If even that maximum alpha is below 1/255 (with a margin that
// absorbs float32 rounding of the per-pixel evaluation), every pixel would
// skip the entry, so it is dropped from the batch (stable compaction; the
// original list position is kept for `last`).  Results are unchanged.
#include <climits>
#include <stdlib.h>
#include <string.h>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "scan.cuh"

namespace dg {


// Pixel layout of a work item: warp w owns an 8-pixel-wide block of 4*PPT
// rows (blocks tile the B x B tile row-major); lane l owns column l % 8 and the
// PPT adjacent rows (l / 8) * PPT + k.
template <int B, int PPT>
__device__ inline void pix_of(int tid, int* lx, int* ly0)
{
    constexpr int NBX = B / 8;
    const int w = tid >> 5, l = tid & 31;
    *lx = (w % NBX) * 8 + (l & 7);
    *ly0 = (w / NBX) * (4 * PPT) + (l >> 3) * PPT;
}

// 2^x on the MUFU unit (ex2.approx, flush-to-zero).
__device__ inline float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Forward: list entries evaluated per loop iteration (a launch-shape constant;
// the result does not depend on it).
#ifndef DG_FWD_UNROLL
#define DG_FWD_UNROLL 2
#endif
constexpr int kFwdUnroll = DG_FWD_UNROLL;
// Backward: list entries whose quadratic forms are formed per loop iteration.
#ifndef DG_BWD_UNROLL
#define DG_BWD_UNROLL 1
#endif
constexpr int kBwdUnroll = DG_BWD_UNROLL;

constexpr float kLog2e = 1.4426950408889634f;
// log2(1/255): the alpha >= 1/255 test is taken in the log2 domain, before the
// exponential, identically in the forward and the backward
constexpr float kLog2AlphaMin = -7.994353436858858f;

// Backward: a warp whose contributing lanes number at most this many adds their
// partial gradients with per-lane vector atomics instead of reducing first
// (0: always reduce; 16 measured fastest on the 2M-Gaussian full-resolution
// step).  A launch-shape constant: results differ only in the
// order of the float additions.
#ifndef DG_BWD_DIRECT_LANES
#define DG_BWD_DIRECT_LANES 16
#endif
constexpr int kBwdDirectLanes = DG_BWD_DIRECT_LANES;

// Stable block-wide compaction index of `keep`; *total = number kept.  Ends with a barrier.
template <int NT>
__device__ inline int compact_index(bool keep, int* s_w, int* total)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_w[w] = __popc(bal);
    __syncthreads();
    int pre = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const int c = s_w[i];
        pre += i < w ? c : 0;
        tot += c;
    }
    *total = tot;
    __syncthreads();
    return pre + __popc(bal & ((1u << lane) - 1u));
}

// One projected record as (u, v, A, B), (C, o, r, g), b.  REC 0: the FP32
// record of dg_project (three float4).  REC 1: the mixed-precision record of
// dg_pack_records (24 bytes: u, v float32 | A, B float16 | C, o float16 |
// r, g bfloat16 | b bfloat16, pad), widened to float32 here; all arithmetic
// after the load is float32.
template <int REC>
__device__ inline void load_record(const void* __restrict__ feat, uint32_t g, float4& a, float4& b, float& c)
{
    if (REC == 0) {
        const float4* f = (const float4*)feat + 3 * (size_t)g;
        a = f[0];
        b = f[1];
        c = f[2].x;
    } else {
        const uint2* f = (const uint2*)feat + 3 * (size_t)g;
        const uint2 w0 = f[0], w1 = f[1], w2 = f[2];
        __half2 ab, co;
        __nv_bfloat162 rg;
        memcpy(&ab, &w1.x, 4);
        memcpy(&co, &w1.y, 4);
        memcpy(&rg, &w2.x, 4);
        const float2 fab = __half22float2(ab), fco = __half22float2(co), frg = __bfloat1622float2(rg);
        a = make_float4(__uint_as_float(w0.x), __uint_as_float(w0.y), fab.x, fab.y);
        b = make_float4(fco.x, fco.y, frg.x, frg.y);
        c = __uint_as_float(w2.y << 16);  // bfloat16 in the low half: its float32 is the bits shifted up
    }
}

// Views of one launch: image sizes, tile grids and where each view's tiles and
// pixels start in the global tile range table and the concatenated images.
struct RViews {
    int n;
    int total;                      // tiles of all views
    int W[DG_MAX_VIEWS], H[DG_MAX_VIEWS], TX[DG_MAX_VIEWS];
    int toff[DG_MAX_VIEWS + 1];
    long long poff[DG_MAX_VIEWS];   // first pixel of each view
    float bg0, bg1, bg2;
};

// Head of the render workspace.  The forward writes the split plan here and
// in the arrays after it; the backward of the same batch reads it.
struct RHdr {
    int cnt_prod, cnt_fwd, cnt_bwd;           // work counters of the three persistent launches
    int colours;                              // set by k_render_fwd_w: 1 it ran, 2 it met a colour that is not finite
    int planned;                              // 1: items/sitems hold a split plan
    int L;                                    // chunk length of that plan
    int n_items, n_slots;                     // items (all chunks), chunks of split tiles
    long long M;                              // entries in the range table
    long long totals;                         // scan total: items (low 32 bits), split chunks (high 32)
};
static_assert(sizeof(RHdr) <= 256, "render header");

// Per-pixel state of split chunks: planes [cap][B*B], chunk slot s = slot0 + c.
struct Slots {
    float* prod;   // product of the chunk's (1 - alpha), pass 1
    float* tout;   // transmittance at the chunk's end (or where compositing stopped)
    float* c0;     // colour added by the chunk; after the combine, the colour behind it
    float* c1;
    float* c2;
    int* last;     // 1-based list position of the chunk's last blend | kStopFlag if it stopped there
    int* nbl;      // entries blended in the chunk
    int* stop;     // list position where compositing stopped (-1 if not in this chunk)
};
constexpr int kStopFlag = 1 << 30;

struct SplitCfg {
    int Lreq;  // > 0: requested chunk length; 0: automatic
    int R;     // resident CTAs of the compositing launch
    int cap;   // chunk slots in the workspace
};

// Shortest automatic chunk (entries): shorter chunks fill more CTAs but give
// the combine pass more chunks to walk per pixel.
#ifndef DG_SPLIT_MIN_LEN
#define DG_SPLIT_MIN_LEN 64
#endif

// Chunk length for M entries: requested or max(DG_SPLIT_MIN_LEN, M/R), raised
// to 2M/cap so that the chunks of split tiles (each tile has n > L, so
// ceil(n/L) < 2n/L) never exceed the slots.
__host__ __device__ inline int split_len(long long M, SplitCfg s)
{
    long long L = s.Lreq > 0 ? s.Lreq : (M + s.R - 1) / s.R;
    if (s.Lreq <= 0 && L < DG_SPLIT_MIN_LEN) L = DG_SPLIT_MIN_LEN;
    const long long Lcap = (2 * M + s.cap - 1) / s.cap;
    if (L < Lcap) L = Lcap;
    if (L < 1) L = 1;
    if (L > (INT_MAX >> 2)) L = INT_MAX >> 2;
    return (int)L;
}

struct LoadLen {
    const uint2* ranges;
    __device__ uint64_t operator()(long long t) const { const uint2 r = ranges[t]; return (uint64_t)(r.y - r.x); }
};
// Items (low 32 bits) and split chunks (high 32 bits) of tile t.
struct LoadChunks {
    const uint2* ranges;
    const RHdr* hdr;
    SplitCfg cfg;
    __device__ uint64_t operator()(long long t) const
    {
        const long long L = split_len(hdr->M, cfg);
        const uint2 r = ranges[t];
        const long long n = (long long)(r.y - r.x);
        if (n <= L) return 1;
        const uint64_t k = (uint64_t)((n + L - 1) / L);
        return (k << 32) | k;
    }
};

__global__ void k_plan_items(const uint2* __restrict__ ranges, int n_tiles, RHdr* hdr, SplitCfg cfg,
                             const uint64_t* __restrict__ toff, int4* __restrict__ items, int4* __restrict__ sitems)
{
    const long long M = hdr->M;
    const int L = split_len(M, cfg);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned long long tot = (unsigned long long)hdr->totals;
        hdr->L = L;
        hdr->n_items = (int)(tot & 0xffffffffull);
        hdr->n_slots = (int)(tot >> 32);
        hdr->planned = 1;
    }
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_tiles; t += gridDim.x * blockDim.x) {
        const uint2 r = ranges[t];
        const long long n = (long long)(r.y - r.x);  // as counted by LoadChunks
        const uint64_t off = toff[t];
        const int io = (int)(off & 0xffffffffull), so = (int)(off >> 32);
        if (n <= L) {
            items[io] = make_int4(t, 0, 1, -1);
            continue;
        }
        const int k = (int)((n + L - 1) / L);
        for (int c = 0; c < k; ++c) {
            const int4 w = make_int4(t, c, k, so);
            items[io + c] = w;
            sitems[so + c] = w;
        }
    }
}

// The whole plan in one block, for up to PLAN_TILES tiles: every automatic split
// of 8x8 tiles (it happens below two tiles per resident CTA, 4864 here) and of
// 16x16 tiles of common images.  A plan of a few tiles is launch-bound: the scans'
// six launches take 30 us in a row.  Every item finds its tile by a search over the
// tiles' first items, so all threads write items: written tile by tile by the warp
// that holds the tile (consecutive tiles, so few warps worked), they took 21 us on 120
// tiles and 37 on 351: the forward of 5 views of 85x62, 440 tiles, 80 -> 50 us.  Above
// PLAN_TILES the scan's blocks read the ranges in parallel.
constexpr int PLAN_THREADS = 1024;
constexpr int PLAN_TILES = PLAN_THREADS * 8;
__global__ void __launch_bounds__(PLAN_THREADS)
k_plan_small(const uint2* __restrict__ ranges, int n_tiles, RHdr* hdr, SplitCfg cfg, int4* __restrict__ items,
             int4* __restrict__ sitems)
{
    __shared__ uint64_t sm[33];
    __shared__ uint32_t s_off[PLAN_TILES];    // list length, then first item of each tile
    __shared__ uint32_t s_slot[PLAN_THREADS]; // first chunk slot of each thread's tiles
    const int tid = threadIdx.x;
    uint64_t acc = 0, tot;
    for (int t = tid; t < n_tiles; t += PLAN_THREADS) {
        const uint2 r = ranges[t];
        s_off[t] = r.y - r.x;
        acc += r.y - r.x;
    }
    block_excl_scan<uint64_t>(acc, sm, &tot);
    const long long M = (long long)tot;
    const uint32_t L = (uint32_t)split_len(M, cfg);
    // a thread's tiles: 1 << sh consecutive ones
    const int sh = n_tiles <= PLAN_THREADS ? 0 : n_tiles <= 2 * PLAN_THREADS ? 1 : n_tiles <= 4 * PLAN_THREADS ? 2 : 3;
    const int t0 = tid << sh, t1 = min(n_tiles, t0 + (1 << sh));
    auto chunks = [&](uint32_t len) { return len <= L ? 1u : (uint32_t)(((uint64_t)len + L - 1) / L); };
    // items (low 32 bits) and split chunks (high 32 bits)
    uint64_t cnt = 0;
    for (int t = t0; t < t1; ++t) {
        const uint32_t k = chunks(s_off[t]);
        cnt += (uint64_t)k | (k > 1 ? (uint64_t)k << 32 : 0);
    }
    const uint64_t off = block_excl_scan<uint64_t>(cnt, sm, &tot);
    const uint32_t n_items = (uint32_t)tot;
    if (tid == 0) {
        hdr->M = M;
        hdr->totals = (long long)tot;
        hdr->L = (int)L;
        hdr->n_items = (int)n_items;
        hdr->n_slots = (int)(tot >> 32);
        hdr->planned = 1;
    }
    s_slot[tid] = (uint32_t)(off >> 32);
    uint32_t at = (uint32_t)off;
    for (int t = t0; t < t1; ++t) {
        const uint32_t k = chunks(s_off[t]);
        s_off[t] = at;
        at += k;
    }
    __syncthreads();
    auto first = [&](int t) { return t < n_tiles ? s_off[t] : n_items; };
    for (uint32_t i = tid; i < n_items; i += PLAN_THREADS) {
        int lo = 0, hi = n_tiles - 1;  // the last tile whose first item is not behind i
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_off[mid] <= i) lo = mid; else hi = mid - 1;
        }
        const uint32_t f = s_off[lo], k = first(lo + 1) - f;
        int4 w = make_int4(lo, (int)(i - f), (int)k, -1);
        if (k > 1) {
            uint32_t slot = s_slot[lo >> sh];
            for (int t = (lo >> sh) << sh; t < lo; ++t) {
                const uint32_t kt = first(t + 1) - s_off[t];
                slot += kt > 1 ? kt : 0u;
            }
            w.w = (int)slot;
            sitems[slot + (i - f)] = w;
        }
        items[i] = w;
    }
}

// A work item: tile (global over views), chunk c of nch, first chunk slot
// (-1: the tile is not split), and the tile's place in its view.
struct Item { int tile, c, nch, slot0, v, tx, ty, W, H; long long poff; };

// Next work item of this CTA from `list` (or tile `index` when list is null);
// item.tile < 0: none left.  Ends with a barrier.
__device__ inline Item next_item(int* counter, int count, const int4* list, const RViews& rv, int4* s_item)
{
    if (threadIdx.x == 0) {
        const int i = atomicAdd(counter, 1);
        int4 w = make_int4(-1, 0, 1, -1);
        if (i < count) w = list ? list[i] : make_int4(i, 0, 1, -1);
        *s_item = w;
    }
    __syncthreads();
    const int4 w = *s_item;
    __syncthreads();
    Item it;
    it.tile = w.x; it.c = w.y; it.nch = w.z; it.slot0 = w.w;
    if (it.tile < 0) return it;
    int v = 0;
    while (v + 1 < rv.n && it.tile >= rv.toff[v + 1]) ++v;
    const int t = it.tile - rv.toff[v];
    it.v = v;
    it.tx = t % rv.TX[v];
    it.ty = t / rv.TX[v];
    it.W = rv.W[v];
    it.H = rv.H[v];
    it.poff = rv.poff[v];
    return it;
}

// Per-pair blend flag written by the forward: 0 when no pixel of the item
// blended the entry; otherwise bit w set when a pixel of warp w's block did.
// With 8x8 tiles and one pixel per thread (two warps of 8x4 pixels, the
// layout of k_render_bwd_ep) bit 7 marks that the low bits are per-warp bits
// of that layout; other layouts set bit 0 only.
constexpr uint8_t kFlagWarpBits = 0x80;
template <int B, int PPT, int NW, int NS>
__device__ inline uint8_t blend_flag(const uint8_t (&s_bl)[NW][NS], int slot)
{
    uint8_t f = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) f |= s_bl[w][slot] ? 1 : 0;
    if (B == 8 && PPT == 1 && f) {
        f = kFlagWarpBits;
#pragma unroll
        for (int w = 0; w < NW; ++w) f |= s_bl[w][slot] ? (uint8_t)(1u << w) : 0;
    }
    return f;
}

// Compositing of one work item.  PROD: pass 1 of a split tile (product of
// the chunk's (1 - alpha) factors from 1, no colour).  Otherwise Eq. 1 over
// the item's entries from T_in, writing the final pixels (whole tile) or the
// chunk's slot (split tile).
template <int B, int PPT, bool PROD, int REC>
__global__ void __launch_bounds__(B * B / PPT)
k_render_fwd(const void* __restrict__ feat, const uint32_t* __restrict__ gid,
             const uint2* __restrict__ ranges, RViews rv, RHdr* hdr, const int4* __restrict__ items,
             const int4* __restrict__ sitems, Slots sl, uint8_t* __restrict__ flags, long long flags_cap,
             float* __restrict__ img, float* __restrict__ Tout, int* __restrict__ lastout,
             int* __restrict__ exout, int* __restrict__ blout)
{
    constexpr int NT = B * B / PPT;
    constexpr int NPIX = B * B;
    __shared__ float4 s_a[NT];    // u, v, a', b'  (prescaled conic, see below)
    __shared__ float2 s_q[NT];    // c', log2 o
    __shared__ float4 s_col[NT];  // r, g, b, list position (int bits)
    // staged entry blended by some pixel of warp w's block (one row per warp, no
    // two warps write the same byte)
    constexpr int NW = NT / 32;
    __shared__ uint8_t s_bl[NW][NT];
    __shared__ int s_w[NT / 32];
    __shared__ int4 s_item;
    const bool planned = hdr->planned != 0 && items != nullptr;
    const int L = planned ? hdr->L : INT_MAX;
    const int count = PROD ? hdr->n_slots : (planned ? hdr->n_items : rv.total);
    const int4* list = PROD ? sitems : (planned ? items : nullptr);
    int* counter = PROD ? &hdr->cnt_prod : &hdr->cnt_fwd;
    for (;;) {
    const Item it = next_item(counter, count, list, rv, &s_item);
    if (it.tile < 0) break;
    if (PROD && it.c == it.nch - 1) continue;  // the last chunk's product is never needed
    const int tile = it.tile, tx = it.tx, ty = it.ty, W = it.W, H = it.H;
    int lx, ly0;
    pix_of<B, PPT>(threadIdx.x, &lx, &ly0);
    const int x = tx * B + lx;
    const int y0 = ty * B + ly0;
    const float pxc = (float)x + 0.5f;
    const float tpx0 = (float)(tx * B) + 0.5f, tpx1 = tpx0 + (float)(B - 1);
    const float tpy0 = (float)(ty * B) + 0.5f, tpy1 = tpy0 + (float)(B - 1);
    const uint2 rg = ranges[tile];
    const int n = (int)(rg.y - rg.x);
    const bool split = it.slot0 >= 0;
    const int lo = split ? it.c * L : 0;
    const int hi = split ? (int)min((long long)n, (long long)lo + L) : n;
    float pyc[PPT], T[PPT], c0[PPT], c1[PPT], c2[PPT];
    int last[PPT], stop[PPT], nbl[PPT];
    bool done[PPT];
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int y = y0 + k;
        pyc[k] = (float)y + 0.5f;
        T[k] = 1.f; c0[k] = c1[k] = c2[k] = 0.f;
        last[k] = 0; stop[k] = -1; nbl[k] = 0;
        done[k] = !(x < W && y < H);
        if (!PROD && split && it.c > 0) {
            // transmittance in front of the chunk: product of the earlier chunks' products
            const int p = (ly0 + k) * B + lx;
            for (int c = 0; c < it.c; ++c) T[k] *= sl.prod[(size_t)(it.slot0 + c) * NPIX + p];
            if (T[k] < kTMin) done[k] = true;  // stopped in an earlier chunk
        }
    }
    bool alldone = true;
#pragma unroll
    for (int k = 0; k < PPT; ++k) alldone = alldone && done[k];
    // flag bytes of the previous batch, written once the next barrier has
    // passed (every lane's blends of that batch are then in s_bl, and the next
    // staging writes s_bl only after compact_index's barriers)
    int pj = -1, pslot = 0;
    bool pkeep = false;
    auto write_flags = [&]() {
        if (PROD || !flags || pj < 0) return;
        const long long gj = (long long)rg.x + pj;
        if (pj < hi && gj < flags_cap) flags[gj] = pkeep ? blend_flag<B, PPT>(s_bl, pslot) : 0;
    };
    for (int base = lo; base < hi; base += NT) {
        if (__syncthreads_count(alldone) == NT) break;
        write_flags();
        const int j = base + (int)threadIdx.x;
        bool keep = false;
        float4 ga, gb;
        float gc = 0.f;
        if (j < hi) {
            const uint32_t g = gid[rg.x + j];
            load_record<REC>(feat, g, ga, gb, gc);
            keep = !tile_skip(ga, gb, tpx0, tpx1, tpy0, tpy1);
        }
        int cnt;
        const int slot = compact_index<NT>(keep, s_w, &cnt);
        if (keep) {
            // prescaled: p = log2(e) * power = dx (a' dx + b' dy) + c' dy^2, alpha = 2^(p + log2 o)
            s_a[slot] = make_float4(ga.x, ga.y, -0.5f * kLog2e * ga.z, -kLog2e * ga.w);
            s_q[slot] = make_float2(-0.5f * kLog2e * gb.x, __log2f(gb.y));
            s_col[slot] = make_float4(gb.z, gb.w, gc, __int_as_float(j));
#pragma unroll
            for (int w = 0; w < NW; ++w) s_bl[w][slot] = 0;
        }
        __syncthreads();
        // Eq. 1 for entry kk at the thread's pixel k, given the entry's power p
        // (log2 scale) and e = p + log2 o
        auto blend = [&](int k, int kk, float p, float e) {
            if (done[k] || !(p <= 0.f && e >= kLog2AlphaMin)) return;
            const float alpha = fminf(kAlphaMax, ex2_approx(e));
            const float Tn = fmaf(-alpha, T[k], T[k]);
            const float4 col = s_col[kk];
            const int pos = __float_as_int(col.w);
            if (Tn < kTMin) {
                done[k] = true;
                stop[k] = pos;
                if (PROD) T[k] = Tn;  // below the threshold: every later chunk is stopped
            } else {
                if (!PROD) {
                    const float w = alpha * T[k];
                    c0[k] += w * col.x;
                    c1[k] += w * col.y;
                    c2[k] += w * col.z;
                    last[k] = pos + 1;
                    ++nbl[k];
                    s_bl[threadIdx.x >> 5][kk] = 1;
                }
                T[k] = Tn;
            }
        };
        // DG_FWD_UNROLL entries per iteration: their quadratic forms do not depend
        // on the transmittance chain, so all are evaluated before any is blended
        for (int kk = 0; kk < cnt && !alldone; kk += kFwdUnroll) {
            float pu[kFwdUnroll][PPT], eu[kFwdUnroll][PPT];
#pragma unroll
            for (int u = 0; u < kFwdUnroll; ++u) {
                const int ku = kk + u < cnt ? kk + u : cnt - 1;
                const float4 a = s_a[ku];
                const float2 q = s_q[ku];
                const float dx = a.x - pxc;
                const float adx = a.z * dx;
#pragma unroll
                for (int k = 0; k < PPT; ++k) {
                    const float dy = a.y - pyc[k];
                    pu[u][k] = fmaf(dx, fmaf(a.w, dy, adx), q.x * dy * dy);
                    eu[u][k] = pu[u][k] + q.y;
                }
            }
#pragma unroll
            for (int u = 0; u < kFwdUnroll; ++u) {
                if (kk + u < cnt) {
#pragma unroll
                    for (int k = 0; k < PPT; ++k) blend(k, kk + u, pu[u][k], eu[u][k]);
                }
            }
            alldone = true;
#pragma unroll
            for (int k = 0; k < PPT; ++k) alldone = alldone && done[k];
        }
        // per list entry: blended by some pixel of this item (the backward
        // stages only those); every entry of the batch gets its byte
        pj = j;
        pkeep = keep;
        pslot = slot;
    }
    if (!PROD && flags) {
        __syncthreads();
        write_flags();
    }
    if (split) {
        const size_t s0 = (size_t)(it.slot0 + it.c) * NPIX;
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            const size_t s = s0 + (size_t)((ly0 + k) * B + lx);
            if (PROD) {
                sl.prod[s] = T[k];
            } else {
                sl.tout[s] = T[k];
                sl.c0[s] = c0[k]; sl.c1[s] = c1[k]; sl.c2[s] = c2[k];
                sl.last[s] = last[k] | (stop[k] >= 0 ? kStopFlag : 0);
                sl.nbl[s] = nbl[k];
                sl.stop[s] = stop[k];
            }
        }
        continue;
    }
    const size_t HW = (size_t)W * H;
    float* im = img + 3 * it.poff;
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int y = y0 + k;
        if (x < W && y < H) {
            const size_t pix = (size_t)y * W + x;
            im[pix] = c0[k] + T[k] * rv.bg0;
            im[HW + pix] = c1[k] + T[k] * rv.bg1;
            im[2 * HW + pix] = c2[k] + T[k] * rv.bg2;
            Tout[it.poff + pix] = T[k];
            lastout[it.poff + pix] = last[k];
            // entries visited: up to and including the one that stopped compositing
            if (exout) exout[it.poff + pix] = stop[k] >= 0 ? stop[k] + 1 : n;
            if (blout) blout[it.poff + pix] = nbl[k];
        }
    }
    }  // work items
}

// Pass 3 of split tiles: one CTA per split tile, one thread per pixel.
template <int B>
__global__ void __launch_bounds__(B * B)
k_render_combine(const uint2* __restrict__ ranges, RViews rv, const RHdr* hdr, const int4* __restrict__ sitems,
                 Slots sl, float* __restrict__ img, float* __restrict__ Tout, int* __restrict__ lastout,
                 int* __restrict__ exout, int* __restrict__ blout)
{
    constexpr int NPIX = B * B;
    if (!hdr->planned) return;
    const int count = hdr->n_slots;
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int4 w = sitems[i];
        if (w.y != 0) continue;
        int v = 0;
        while (v + 1 < rv.n && w.x >= rv.toff[v + 1]) ++v;
        const int t = w.x - rv.toff[v];
        const int W = rv.W[v], H = rv.H[v];
        const int lx = (int)(threadIdx.x % B), ly = (int)(threadIdx.x / B);
        const int x = (t % rv.TX[v]) * B + lx, y = (t / rv.TX[v]) * B + ly;
        if (!(x < W && y < H)) continue;
        const uint2 rg = ranges[w.x];
        const int n = (int)(rg.y - rg.x);
        const int nch = w.z;
        const size_t p = (size_t)threadIdx.x;
        // A few tiles hold dozens of chunks each and only their blocks work, so
        // each walk loads CB chunks' fields before using any (chunk order, and
        // so every sum's rounding, unchanged).
        constexpr int CB = 8;
        float C0 = 0.f, C1 = 0.f, C2 = 0.f;
        int lastv = 0, nb = 0, cstop = -1;
        for (int cb = 0; cb < nch; cb += CB) {
            int lt[CB], nbv[CB];
            float a0[CB], a1[CB], a2[CB];
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                if (cb + j < nch) {
                    const size_t s = (size_t)(w.w + cb + j) * NPIX + p;
                    lt[j] = sl.last[s]; nbv[j] = sl.nbl[s];
                    a0[j] = sl.c0[s]; a1[j] = sl.c1[s]; a2[j] = sl.c2[s];
                }
            }
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                if (cb + j < nch) {
                    C0 += a0[j]; C1 += a1[j]; C2 += a2[j];
                    lastv = max(lastv, lt[j] & (kStopFlag - 1));
                    nb += nbv[j];
                    if ((lt[j] & kStopFlag) && cstop < 0) cstop = cb + j;
                }
            }
        }
        // T at the end: from the chunk where the pixel stopped, else the last chunk
        const size_t sf = (size_t)(w.w + (cstop >= 0 ? cstop : nch - 1)) * NPIX + p;
        const float Tf = sl.tout[sf];
        const int ex = cstop >= 0 ? sl.stop[sf] + 1 : n;
        // colour behind each chunk (the backward's starting S), back to front
        float S0 = Tf * rv.bg0, S1 = Tf * rv.bg1, S2 = Tf * rv.bg2;
        for (int cb = nch - 1; cb >= 0; cb -= CB) {
            float a0[CB], a1[CB], a2[CB];
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                if (cb - j >= 0) {
                    const size_t s = (size_t)(w.w + cb - j) * NPIX + p;
                    a0[j] = sl.c0[s]; a1[j] = sl.c1[s]; a2[j] = sl.c2[s];
                }
            }
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                if (cb - j >= 0) {
                    const size_t s = (size_t)(w.w + cb - j) * NPIX + p;
                    sl.c0[s] = S0; sl.c1[s] = S1; sl.c2[s] = S2;
                    S0 += a0[j]; S1 += a1[j]; S2 += a2[j];
                }
            }
        }
        const size_t HW = (size_t)W * H;
        const size_t pix = (size_t)y * W + x;
        float* im = img + 3 * rv.poff[v];
        im[pix] = C0 + Tf * rv.bg0;
        im[HW + pix] = C1 + Tf * rv.bg1;
        im[2 * HW + pix] = C2 + Tf * rv.bg2;
        Tout[rv.poff[v] + pix] = Tf;
        lastout[rv.poff[v] + pix] = lastv;
        if (exout) exout[rv.poff[v] + pix] = ex;
        if (blout) blout[rv.poff[v] + pix] = nb;
    }
}

// Sum of 9 per-lane values over the warp by recursive halving: at each step a
// lane keeps half of its values and receives its partner's partial sums of
// that half (12 shuffles instead of 45).  Returns the total of value `*idx`
// (0..8) on the lanes where *idx is valid (*idx = -1 elsewhere); both lanes of
// each final pair hold it, only the even one reports it.
__device__ inline float warp_sum9(const float v[9], int lane, int* idx)
{
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    float a1[6];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float lo = v[i], hi = i + 5 < 9 ? v[i + 5] : 0.f;
        const float keep = b4 ? hi : lo, send = b4 ? lo : hi;
        a1[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    a1[5] = 0.f;
    float a2[4];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float keep = b3 ? a1[i + 3] : a1[i], send = b3 ? a1[i] : a1[i + 3];
        a2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    a2[3] = 0.f;
    float a3[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float keep = b2 ? a2[i + 2] : a2[i], send = b2 ? a2[i] : a2[i + 2];
        a3[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    float a4;
    {
        const float keep = b1 ? a3[1] : a3[0], send = b1 ? a3[0] : a3[1];
        a4 = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    a4 += __shfl_xor_sync(0xffffffffu, a4, 1);
    const int i2 = (b2 ? 2 : 0) + (b1 ? 1 : 0);        // index into a2 (3 = padding)
    const int i1 = (b3 ? 3 : 0) + i2;                   // index into a1 (5 = padding)
    const int i0 = (b4 ? 5 : 0) + i1;                   // original index (9 = padding)
    *idx = ((lane & 1) == 0 && i2 < 3 && i1 < 5 && i0 < 9) ? i0 : -1;
    return a4;
}

template <int B, int PPT, int REC>
__global__ void __launch_bounds__(B * B / PPT)
k_render_bwd(const void* __restrict__ feat, const uint32_t* __restrict__ gid,
             const uint2* __restrict__ ranges, RViews rv, RHdr* hdr, const int4* __restrict__ items, Slots sl,
             const uint8_t* __restrict__ flags, long long flags_cap,
             const float* __restrict__ Tfin, const int* __restrict__ lastin,
             const float* __restrict__ dLdimg, float4* __restrict__ grad2d)
{
    constexpr int NT = B * B / PPT;
    constexpr int NPIX = B * B;
    __shared__ float4 s_a[NT];    // u, v, a', b'  (the forward's prescaled conic)
    __shared__ float2 s_q[NT];    // c', log2 o
    __shared__ float4 s_k[NT];    // A, B, C, 1/o
    __shared__ float4 s_col[NT];  // r, g, b, list position (int bits)
    __shared__ uint32_t s_g[NT];
    __shared__ int s_w[NT / 32];
    __shared__ int s_n;
    __shared__ int4 s_item;
    const float bg0 = rv.bg0, bg1 = rv.bg1, bg2 = rv.bg2;
    // (a whole-tile walk is exact whatever the forward did; items is null when
    // the workspace was laid out without splitting)
    const bool planned = hdr->planned != 0 && items != nullptr;
    const int L = planned ? hdr->L : INT_MAX;
    const int count = planned ? hdr->n_items : rv.total;
    for (;;) {
    const Item it = next_item(&hdr->cnt_bwd, count, planned ? items : nullptr, rv, &s_item);
    if (it.tile < 0) break;
    const int tile = it.tile, tx = it.tx, ty = it.ty, W = it.W, H = it.H;
    int lx, ly0;
    pix_of<B, PPT>(threadIdx.x, &lx, &ly0);
    const int x = tx * B + lx;
    const int y0 = ty * B + ly0;
    const float pxc = (float)x + 0.5f;
    const float tpx0 = (float)(tx * B) + 0.5f, tpx1 = tpx0 + (float)(B - 1);
    const float tpy0 = (float)(ty * B) + 0.5f, tpy1 = tpy0 + (float)(B - 1);
    const uint2 rg = ranges[tile];
    const int nlist = (int)(rg.y - rg.x);
    const bool split = it.slot0 >= 0;
    const int lo = split ? it.c * L : 0;
    const int hi = split ? (int)min((long long)nlist, (long long)lo + L) : nlist;
    const size_t HW = (size_t)W * H;
    // per pixel: transmittance, dL/dC, and gS = dL/dC . S where S is the
    // colour composited behind the current entry (the only way S enters the
    // gradient: dL/dalpha_j = T_j (g . c_j) - (g . S_j) / (1 - alpha_j))
    float pyc[PPT], T[PPT], g0[PPT], g1[PPT], g2[PPT], gS[PPT];
    int lastp[PPT];
    int mylast = 0;
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int y = y0 + k;
        pyc[k] = (float)y + 0.5f;
        T[k] = 1.f; g0[k] = g1[k] = g2[k] = 0.f; lastp[k] = 0;
        gS[k] = 0.f;
        if (x < W && y < H) {
            const size_t pix = (size_t)y * W + x;
            const float* dl = dLdimg + 3 * it.poff;
            lastp[k] = lastin[it.poff + pix];
            g0[k] = dl[pix];
            g1[k] = dl[HW + pix];
            g2[k] = dl[2 * HW + pix];
            if (split) {
                // the chunk's end transmittance and the colour behind the chunk
                const size_t s = (size_t)(it.slot0 + it.c) * NPIX + (size_t)((ly0 + k) * B + lx);
                T[k] = sl.tout[s];
                gS[k] = g0[k] * sl.c0[s] + g1[k] * sl.c1[s] + g2[k] * sl.c2[s];
            } else {
                T[k] = Tfin[it.poff + pix];
                gS[k] = T[k] * (g0[k] * bg0 + g1[k] * bg1 + g2[k] * bg2);  // behind the last entry: T bg
            }
        }
        mylast = max(mylast, lastp[k]);
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    if (mylast > 0) atomicMax(&s_n, mylast);
    __syncthreads();
    // never walk past the item's own entries, whatever `last` holds
    const int top = min(s_n, hi);
    const int lane = threadIdx.x & 31;
    // this lane's partial gradient of the current entry: du, dv, dA, dB, dC,
    // d opacity, d r, d g, d b.  With one pixel per thread each blending lane
    // assigns all nine (no per-entry zeroing; lanes that did not blend are
    // masked at the reduction); with several pixels they accumulate from zero.
    float vd[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) vd[i] = 0.f;
    for (int base = top > lo ? lo + ((top - lo - 1) / NT) * NT : lo - 1; base >= lo; base -= NT) {
        const int j = base + (int)threadIdx.x;
        bool keep = false;
        float4 ga, gb;
        float gc = 0.f;
        uint32_t g = 0;
        if (j < top) {
            const long long gj = (long long)rg.x + j;
            if (flags && gj < flags_cap) {
                // the forward's record of this entry: blended by some pixel of the
                // tile or not (an entry no pixel blended has no gradient)
                keep = flags[gj] != 0;
                if (keep) {
                    g = gid[gj];
                    load_record<REC>(feat, g, ga, gb, gc);
                }
            } else {
                g = gid[gj];
                load_record<REC>(feat, g, ga, gb, gc);
                keep = !tile_skip(ga, gb, tpx0, tpx1, tpy0, tpy1);
            }
        }
        int cnt;
        const int slot = compact_index<NT>(keep, s_w, &cnt);
        if (keep) {
            s_g[slot] = g;
            s_a[slot] = make_float4(ga.x, ga.y, -0.5f * kLog2e * ga.z, -kLog2e * ga.w);
            s_q[slot] = make_float2(-0.5f * kLog2e * gb.x, __log2f(gb.y));
            s_k[slot] = make_float4(ga.z, ga.w, gb.x, __frcp_rn(gb.y));
            s_col[slot] = make_float4(gb.z, gb.w, gc, __int_as_float(j));
        }
        __syncthreads();
        // one list entry, given its quadratic forms at this thread's pixels
        auto entry = [&](int kk, const float4& col, float dx, const float* dyv, const float* pv) {
            const int pos = __float_as_int(col.w);
            if (!__any_sync(0xffffffffu, pos < mylast)) return;
            const float cr = col.x, cg = col.y, cb = col.z;
            const float qy = s_q[kk].y;
            if (PPT > 1) {
#pragma unroll
                for (int i = 0; i < 9; ++i) vd[i] = 0.f;
            }
            bool any = false;
#pragma unroll
            for (int k = 0; k < PPT; ++k) {
                if (pos < lastp[k]) {
                    // the forward's blend test and alpha, bit for bit
                    const float dy = dyv[k];
                    const float p = pv[k];
                    const float e = p + qy;
                    if (p <= 0.f && e >= kLog2AlphaMin) {
                        const float raw = ex2_approx(e);
                        const float alpha = fminf(kAlphaMax, raw);
                        const float4 kc = s_k[kk];  // A, B, C, 1/o
                        any = true;
                        // hardware reciprocal (about 1 ulp; 1 - alpha is in [0.01, 1]): the
                        // exactly rounded one costs a measured 6% of the kernel
                        const float inv = __fdividef(1.f, 1.f - alpha);
                        T[k] *= inv;  // transmittance in front of this entry
                        const float wT = alpha * T[k];
                        const float gcol = fmaf(g0[k], cr, fmaf(g1[k], cg, g2[k] * cb));
                        const float dLda = fmaf(T[k], gcol, -gS[k] * inv);
                        gS[k] = fmaf(wT, gcol, gS[k]);
                        // below the clamp: d alpha / d o = exp(power), d alpha / d power = alpha
                        const float dp = raw <= kAlphaMax ? dLda * alpha : 0.f;
                        const float dopa = raw <= kAlphaMax ? dLda * raw * kc.w : 0.f;
                        const float qx = dp * dx, qdy = dp * dy;
                        const float v[9] = {-fmaf(kc.x, qx, kc.y * qdy), -fmaf(kc.y, qx, kc.z * qdy),
                                            -0.5f * qx * dx, -qx * dy, -0.5f * qdy * dy, dopa,
                                            wT * g0[k], wT * g1[k], wT * g2[k]};
#pragma unroll
                        for (int i = 0; i < 9; ++i) vd[i] = PPT == 1 ? v[i] : vd[i] + v[i];
                    }
                }
            }
            const unsigned anym = __ballot_sync(0xffffffffu, any);
            if (!anym) return;
            if (kBwdDirectLanes > 0 && __popc(anym) <= kBwdDirectLanes) {
                // few contributing lanes: each adds its own partial sums (three
                // vector atomics) instead of the 12-shuffle warp reduction
                if (any) {
                    float4* gp = grad2d + 3 * (size_t)s_g[kk];
                    atomicAdd(gp, make_float4(vd[0], vd[1], vd[2], vd[3]));
                    atomicAdd(gp + 1, make_float4(vd[4], vd[5], vd[6], vd[7]));
                    atomicAdd((float*)(gp + 2), vd[8]);
                }
                return;
            }
            float vals[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) vals[i] = any ? vd[i] : 0.f;
            int idx;
            const float tot = warp_sum9(vals, lane, &idx);
            if (idx >= 0) atomicAdd((float*)(grad2d + 3 * (size_t)s_g[kk]) + idx, tot);
        };
        // kBwdUnroll entries per iteration, back to front: their quadratic forms
        // are formed first (independent of the transmittance chain)
        for (int kk = cnt - 1; kk >= 0; kk -= kBwdUnroll) {
            float4 colu[kBwdUnroll];
            float dxu[kBwdUnroll], dyu[kBwdUnroll][PPT], pu[kBwdUnroll][PPT];
#pragma unroll
            for (int u = 0; u < kBwdUnroll; ++u) {
                const int ku = kk - u >= 0 ? kk - u : kk;
                colu[u] = s_col[ku];
                const float4 a = s_a[ku];
                const float2 q = s_q[ku];
                dxu[u] = a.x - pxc;
                const float adx = a.z * dxu[u];
#pragma unroll
                for (int k = 0; k < PPT; ++k) {
                    dyu[u][k] = a.y - pyc[k];
                    pu[u][k] = fmaf(dxu[u], fmaf(a.w, dyu[u][k], adx), q.x * dyu[u][k] * dyu[u][k]);
                }
            }
#pragma unroll
            for (int u = 0; u < kBwdUnroll; ++u)
                if (kk - u >= 0) entry(kk - u, colu[u], dxu[u], dyu[u], pu[u]);
        }
        __syncthreads();
    }
    }  // work items
}

constexpr int kEpG = 16;                      // entries per group
constexpr int kEpRing = 48;                   // staged entries: a group less one, and a batch of 32
constexpr int kEpPitch = 33;                  // float4 per entry pair of the (pair, pixel) matrix: 32 pixels + 1
constexpr int kPairW = 5;                     // float4 per staged entry pair

// Next work item of this warp: item index w covers tile (or chunk) w / 2 and
// the 8x4 pixel block w % 2 of it; *blk receives the block.  Warp-uniform.
__device__ inline Item next_item_warp(int* counter, int count, const int4* list, const RViews& rv, int* blk)
{
    int w = 0;
    if ((threadIdx.x & 31) == 0) w = atomicAdd(counter, 1);
    w = __shfl_sync(0xffffffffu, w, 0);
    Item it;
    it.tile = -1;
    if (w >= 2 * count) return it;
    const int i = w >> 1;
    *blk = w & 1;
    const int4 q = list ? list[i] : make_int4(i, 0, 1, -1);
    it.tile = q.x; it.c = q.y; it.nch = q.z; it.slot0 = q.w;
    int v = 0;
    while (v + 1 < rv.n && it.tile >= rv.toff[v + 1]) ++v;
    const int t = it.tile - rv.toff[v];
    it.v = v;
    it.tx = t % rv.TX[v];
    it.ty = t / rv.TX[v];
    it.W = rv.W[v];
    it.H = rv.H[v];
    it.poff = rv.poff[v];
    return it;
}

// True unless a colour channel is infinite or NaN.
__device__ __forceinline__ bool finite_colour(float r, float g, float b)
{
    return fmaf(b, 0.f, fmaf(g, 0.f, r * 0.f)) == 0.f;
}

// Reciprocal on the special-function unit (rcp.approx: about 1 ulp; exactly 1 for 1).
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Backward of 8x8 tiles with one pixel per thread, entry-parallel gradient
// sums, each warp on its own.  A work item is one 8x4 block of a tile (or of a
// chunk of a split tile), taken by the warp from the shared counter; no
// CTA-wide barrier, so the two blocks of a tile, whose lists and walks
// differ, do not wait for each other.  The warp walks back from the largest
// `last` of its own 32 pixels over batches of 32 candidates and stages, last
// entry first, only those that some pixel of its block blended (the forward's
// per-block bit, or every flagged entry when the forward ran at another launch
// shape; the block-rectangle alpha test when there are no flags).  The staged
// entries form a ring that carries over from batch to batch, so every group but
// the walk's last is full.  Per group of 16 entries:
//   A. pixel-parallel (lane = pixel): walks the group's entries exactly as
//      k_render_bwd (the forward's blend test bit for bit, T recovered through
//      1/(1 - alpha), dL/dalpha from the running g . S) and stores per (entry,
//      pixel) the two scalars the gradient needs, dp = dL/dpower and wT =
//      alpha T.  One straight line for the whole warp, two entries a step in
//      packed float32: where the pixel does not blend, alpha is 0, which leaves
//      T and g . S alone and gives dp = wT = 0;
//   B. entry-parallel (lane = entry pair of the group and one row of the block):
//      the sums over the pixels of dp dx, dp dy, dp dx^2, dp dx dy, dp dy^2 (dx,
//      dy: Gaussian centre minus pixel centre) follow from moments of dp about
//      the block's centre (per row sum dp, sum dp ox, sum dp ox^2 with ox in
//      -3.5 .. 3.5; expanding about the block's own centre keeps cancellation
//      small), packed over the two entries, plus the colour sums sum wT dL/dC with
//      the row's dL/dC in registers.  Two rounds of shuffles join the rows, the
//      first also leaving one entry per lane; then two lanes hold each entry's
//      sums and add their parts of its record.
// The opacity term uses d alpha / d o = alpha / o below the clamp: sum(dp) / o.
// Bound by issue and the shared-memory pipe together (77% of the issue slots,
// 85% of the pipe's wavefronts).  Measured on 16 views of 1237x822, 480k
// Gaussians, mixed records: 4.14 ms with groups cut at every batch (9.5 entries
// of 16 on average) and a scalar walk with branches -> 3.55 ms (on four of the
// views 1097M -> 740M warp instructions; then the shared-memory pipe was full)
// -> 3.25 ms with a pair and a row per lane instead of an entry and half the
// block -> 3.20 ms with the row's dL/dC in registers instead of read from shared
// memory per group (12 blocks of 64 threads per SM; 9, 10, 11 blocks 3.21, 3.23,
// 3.20 ms) -> 3.13 ms with the shared arrays as one struct and the body inlined once
// per form of k_render_bwd_ep.
struct EpShared {
    // staged entry pairs: (u, u', v, v'), (a, a', b, b') the forward's prescaled
    // conic, (c, c', log2 o, log2 o'), (r, r', g, g'), (b, b', list positions)
    float4 pair[2][kEpRing / 2 * kPairW];
    float4 k[2][kEpRing];                // A, B, C, 1/o
    uint32_t g[2][kEpRing];
    float4 m[2][kEpG / 2 * kEpPitch];    // [pair][pixel] (dp, dp', wT, wT')
    float4 px[2][32];                    // per pixel dL/dC
};

// APART: some staged colour may be infinite or NaN.
template <int REC, bool APART>
__device__ __forceinline__ void
render_bwd_ep(const void* __restrict__ feat, const uint32_t* __restrict__ gid,
              const uint2* __restrict__ ranges, RViews rv, RHdr* hdr, const int4* __restrict__ items, Slots sl,
              const uint8_t* __restrict__ flags, long long flags_cap,
              const float* __restrict__ Tfin, const int* __restrict__ lastin,
              const float* __restrict__ dLdimg, float4* __restrict__ grad2d, EpShared& sh)
{
    constexpr int B = 8, NPIX = 64;
    const float bg0 = rv.bg0, bg1 = rv.bg1, bg2 = rv.bg2;
    const bool planned = hdr->planned != 0 && items != nullptr;
    const int L = planned ? hdr->L : INT_MAX;
    const int count = planned ? hdr->n_items : rv.total;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    float4* const sp = sh.pair[wp];
    float4* const sm = sh.m[wp];
    float4* const wk = sh.k[wp];
    uint32_t* const wg = sh.g[wp];
    const uint32_t above = ~((2u << lane) - 1u);  // lanes behind this one in the list
    for (;;) {
    int blk = 0;
    const Item it = next_item_warp(&hdr->cnt_bwd, count, planned ? items : nullptr, rv, &blk);
    if (it.tile < 0) break;
    const int tile = it.tile, tx = it.tx, ty = it.ty, W = it.W, H = it.H;
    const int lx = lane & 7, ly0 = 4 * blk + (lane >> 3);
    const int x = tx * B + lx;
    const int y = ty * B + ly0;
    const float pxc = (float)x + 0.5f, pyc = (float)y + 0.5f;
    // this block's pixel centres: [bx0, bx1] x [by0, by1]
    const float bx0 = (float)(tx * B) + 0.5f, bx1 = bx0 + 7.f;
    const float by0 = (float)(ty * B + 4 * blk) + 0.5f, by1 = by0 + 3.f;
    const uint2 rg = ranges[tile];
    const int nlist = (int)(rg.y - rg.x);
    const bool split = it.slot0 >= 0;
    const int lo = split ? it.c * L : 0;
    const int hi = split ? (int)min((long long)nlist, (long long)lo + L) : nlist;
    const size_t HW = (size_t)W * H;
    float T = 1.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, gS = 0.f;
    int lastp = 0;
    if (x < W && y < H) {
        const size_t pix = (size_t)y * W + x;
        const float* dl = dLdimg + 3 * it.poff;
        lastp = lastin[it.poff + pix];
        g0 = dl[pix];
        g1 = dl[HW + pix];
        g2 = dl[2 * HW + pix];
        if (split) {
            const size_t sidx = (size_t)(it.slot0 + it.c) * NPIX + (size_t)(ly0 * B + lx);
            T = sl.tout[sidx];
            gS = g0 * sl.c0[sidx] + g1 * sl.c1[sidx] + g2 * sl.c2[sidx];
        } else {
            T = Tfin[it.poff + pix];
            gS = T * (g0 * bg0 + g1 * bg1 + g2 * bg2);
        }
    }
    __syncwarp();
    sh.px[wp][lane] = make_float4(g0, g1, g2, 0.f);
    __syncwarp();
    // phase B: dL/dC of the 8 pixels of this lane's row
    float gpr[8], gpg[8], gpb[8];
#pragma unroll
    for (int px = 0; px < 8; ++px) {
        const float4 c = sh.px[wp][8 * (lane >> 3) + px];
        gpr[px] = c.x; gpg[px] = c.y; gpb[px] = c.z;
    }
    const int top = min(__reduce_max_sync(0xffffffffu, lastp), hi);
    // phase B: this lane's entry pair of the group and row of the block; the
    // entry it is left with after the first exchange
    const int bp8 = lane & 7, br = lane >> 3, be = 2 * bp8 + (br & 1);
    const float bcx = bx0 + 3.5f, bcy = by0 + 1.5f;
    const float oyo = (float)br - 1.5f, oyp = (float)(br ^ 1) - 1.5f;  // this row's and the exchanged row's offsets
    const f32x2 npx = f2_pack(-pxc, -pxc), npy = f2_pack(-pyc, -pyc);
    const f32x2 gr = f2_pack(g0, g0), gg = f2_pack(g1, g1), gb2 = f2_pack(g2, g2);
    __syncwarp();
    // the flag byte and Gaussian index of a batch are loaded one batch ahead,
    // so a batch waits only for its records (kNoFlag: no flag for the entry)
    constexpr uint32_t kNoFlag = 0x100u;
    int base = top > lo ? lo + ((top - lo - 1) / 32) * 32 : lo - 1;
    uint32_t fn = kNoFlag, gn = 0;
    auto fetch = [&](int b) {
        const int jj = b + lane;
        fn = kNoFlag;
        gn = 0;
        if (b >= lo && jj < top) {
            const long long gj = (long long)rg.x + jj;
            if (flags && gj < flags_cap) fn = flags[gj];
            gn = gid[gj];
        }
    };
    fetch(base);
    int pend = 0, gslot = 0;  // staged entries, and the ring slot of the first
    for (;;) {
        while (pend < kEpG && base >= lo) {
            const int j = base + lane;
            const uint32_t fcur = fn, g = gn;
            base -= 32;
            fetch(base);
            bool keep = false;
            float4 ga, gb;
            float gc = 0.f, lo2 = 0.f;
            if (j < top) {
                if (fcur != kNoFlag) {
                    keep = (fcur & kFlagWarpBits) ? ((fcur >> blk) & 1u) != 0 : fcur != 0;
                    if (keep) {
                        load_record<REC>(feat, g, ga, gb, gc);
                        lo2 = __log2f(gb.y);
                    }
                } else {
                    load_record<REC>(feat, g, ga, gb, gc);
                    lo2 = __log2f(gb.y);
                    keep = !block_skip(ga, gb, lo2, bx0, bx1, by0, by1);
                }
            }
            const uint32_t km = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                int slot = gslot + pend + __popc(km & above);
                if (slot >= kEpRing) slot -= kEpRing;
                float4* q = sp + (slot >> 1) * kPairW;
                float* f = (float*)q + (slot & 1);
                f[0] = ga.x; f[2] = ga.y;
                f[4] = -0.5f * kLog2e * ga.z; f[6] = -kLog2e * ga.w;
                f[8] = -0.5f * kLog2e * gb.x; f[10] = lo2;
                f[12] = gb.z; f[14] = gb.w;
                f[16] = gc; f[18] = __int_as_float(j);
                wg[slot] = g;
                wk[slot] = make_float4(ga.z, ga.w, gb.x, __frcp_rn(gb.y));
            }
            pend += __popc(km);
        }
        if (pend == 0) break;
        const int n = min(pend, kEpG);
        if ((n & 1) && lane == 0) {  // (only the walk's last group) an entry no pixel blends
            float* f = (float*)(sp + ((gslot + n) >> 1) * kPairW) + 1;
#pragma unroll
            for (int i = 0; i < 18; i += 2) f[i] = 0.f;
            f[18] = __int_as_float(INT_MAX);
        }
        __syncwarp();
        // A: this lane's pixel over the group's entries, back to front, two at a time
        uint32_t mine = 0;
        {
            const float4* q = sp + (gslot >> 1) * kPairW;
            float4* out = sm + lane;
            uint32_t bit = 1u;
            for (int k = 0; k < n; k += 2, q += kPairW, out += kEpPitch, bit <<= 2) {
                const float4 uv = q[0], ab = q[1], cl = q[2], rgc = q[3], bp = q[4];
                const f32x2 dx = f2_add(f2_pack(uv.x, uv.y), npx), dy = f2_add(f2_pack(uv.z, uv.w), npy);
                const f32x2 pu = f2_fma(dx, f2_fma(f2_pack(ab.z, ab.w), dy, f2_mul(f2_pack(ab.x, ab.y), dx)),
                                        f2_mul(f2_mul(f2_pack(cl.x, cl.y), dy), dy));
                const f32x2 eu = f2_add(pu, f2_pack(cl.z, cl.w));
                const f32x2 gu = f2_fma(gr, f2_pack(rgc.x, rgc.y),
                                        f2_fma(gg, f2_pack(rgc.z, rgc.w), f2_mul(gb2, f2_pack(bp.x, bp.y))));
                float p0, p1, e0, e1, gc0, gc1;
                f2_unpack(pu, p0, p1);
                f2_unpack(eu, e0, e1);
                f2_unpack(gu, gc0, gc1);
                const bool b0 = __float_as_int(bp.z) < lastp && p0 <= 0.f && e0 >= kLog2AlphaMin;
                const bool b1 = __float_as_int(bp.w) < lastp && p1 <= 0.f && e1 >= kLog2AlphaMin;
                if (APART) {  // the colour of an entry that is not blended stays out of g . S
                    if (!b0) gc0 = 0.f;
                    if (!b1) gc1 = 0.f;
                }
                const float r0 = ex2_approx(e0), r1 = ex2_approx(e1);
                const float a0 = b0 ? fminf(kAlphaMax, r0) : 0.f, a1 = b1 ? fminf(kAlphaMax, r1) : 0.f;
                const float i0 = rcp_approx(1.f - a0), i1 = rcp_approx(1.f - a1);
                // transmittance in front of the entry, then dL/dalpha and the colour behind the next
                T *= i0;
                const float w0 = a0 * T;
                const float d0 = fmaf(T, gc0, -gS * i0);
                gS = fmaf(w0, gc0, gS);
                T *= i1;
                const float w1 = a1 * T;
                const float d1 = fmaf(T, gc1, -gS * i1);
                gS = fmaf(w1, gc1, gS);
                // below the clamp d alpha / d power = alpha
                const float dp0 = b0 && r0 <= kAlphaMax ? d0 * a0 : 0.f;
                const float dp1 = b1 && r1 <= kAlphaMax ? d1 * a1 : 0.f;
                if (b0) mine |= bit;
                if (b1) mine |= bit << 1;
                *out = make_float4(dp0, dp1, w0, w1);
            }
        }
        const uint32_t used = __reduce_or_sync(0xffffffffu, mine);
        __syncwarp();
        if (used) {
            // (slots of a partial group hold an earlier group's entries: their sums are not used)
            const float4* const row = sm + bp8 * kEpPitch + 8 * br;
            // (both entries at once) sum dp, sum dp ox, sum dp ox^2: ox = -3.5 .. 3.5, so
            // pixels px and 7 - px share their sum and difference
            f32x2 s0, sx, sxx;
            float c0[3], c1[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) c0[i] = c1[i] = 0.f;
#pragma unroll
            for (int px = 0; px < 4; ++px) {
                const float4 m = row[7 - px], n2 = row[px];
                const float k = 3.5f - (float)px;
                const f32x2 d = f2_pack(m.x, m.y), e = f2_pack(n2.x, n2.y);
                const f32x2 su = f2_add(d, e), di = f2_fma(e, f2_pack(-1.f, -1.f), d);
                s0 = px ? f2_add(s0, su) : su;
                sx = px ? f2_fma(di, f2_pack(k, k), sx) : f2_mul(di, f2_pack(k, k));
                sxx = px ? f2_fma(su, f2_pack(k * k, k * k), sxx) : f2_mul(su, f2_pack(k * k, k * k));
                c0[0] = fmaf(m.z, gpr[7 - px], fmaf(n2.z, gpr[px], c0[0]));
                c0[1] = fmaf(m.z, gpg[7 - px], fmaf(n2.z, gpg[px], c0[1]));
                c0[2] = fmaf(m.z, gpb[7 - px], fmaf(n2.z, gpb[px], c0[2]));
                c1[0] = fmaf(m.w, gpr[7 - px], fmaf(n2.w, gpr[px], c1[0]));
                c1[1] = fmaf(m.w, gpg[7 - px], fmaf(n2.w, gpg[px], c1[1]));
                c1[2] = fmaf(m.w, gpb[7 - px], fmaf(n2.w, gpb[px], c1[2]));
            }
            // even rows keep the pair's first entry, odd rows the second
            float va[6], vb[6];
            f2_unpack(s0, va[0], vb[0]); f2_unpack(sx, va[1], vb[1]); f2_unpack(sxx, va[2], vb[2]);
#pragma unroll
            for (int i = 0; i < 3; ++i) { va[3 + i] = c0[i]; vb[3 + i] = c1[i]; }
            const bool odd = (br & 1) != 0;
            float acc[9];  // S0, Sx, Sxx, red, green, blue, Sy, Sxy, Syy
            {
                float own[6], oth[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    own[i] = odd ? vb[i] : va[i];
                    oth[i] = __shfl_xor_sync(0xffffffffu, odd ? va[i] : vb[i], 8);
                    acc[i] = own[i] + oth[i];
                }
                const float yo = oyo * own[0], yp = oyp * oth[0];
                acc[6] = yo + yp;
                acc[7] = fmaf(oyo, own[1], oyp * oth[1]);
                acc[8] = fmaf(oyo, yo, oyp * yp);
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
            if ((used >> be) & 1u) {
                const int slot = gslot + be;
                const float4 kc = wk[slot];
                const float* f = (const float*)(sp + (slot >> 1) * kPairW) + (slot & 1);
                const float dx0 = f[0] - bcx, dy0 = f[2] - bcy;
                const float S0 = acc[0], Sx = acc[1], Sy = acc[6];
                float4* const gq = grad2d + 3 * (size_t)wg[slot];
                if (br < 2) {
                    const float qx = fmaf(dx0, S0, -Sx), qy = fmaf(dy0, S0, -Sy);
                    const float gA = fmaf(dx0, fmaf(dx0, S0, -2.f * Sx), acc[2]);
                    const float gB = fmaf(dx0, fmaf(dy0, S0, -Sy), fmaf(-dy0, Sx, acc[7]));
                    atomicAdd(gq, make_float4(-fmaf(kc.x, qx, kc.y * qy), -fmaf(kc.y, qx, kc.z * qy), -0.5f * gA, -gB));
                } else {
                    const float gC = fmaf(dy0, fmaf(dy0, S0, -2.f * Sy), acc[8]);
                    atomicAdd(gq + 1, make_float4(-0.5f * gC, S0 * kc.w, acc[3], acc[4]));
                    atomicAdd((float*)(gq + 2), acc[5]);
                }
            }
        }
        __syncwarp();
        pend -= n;
        gslot += kEpG;
        if (gslot == kEpRing) gslot = 0;
    }
    __syncwarp();
    }  // work items
}

// The walk for finite colours unless the forward met others, or was another pass
// (then nothing is known): a weight of 0 leaves g . S alone only where the colour is
// finite, and keeping the others out takes two more instructions per step.  On 16
// views of 1237x822, 480k Gaussians, mixed records: 3.12 ms without the test, 3.20
// with it in every step, 3.16 with two walks side by side in one body, 3.05 with a
// body for each form.
template <int REC>
__global__ void __launch_bounds__(64, 12)
k_render_bwd_ep(const void* __restrict__ feat, const uint32_t* __restrict__ gid,
                const uint2* __restrict__ ranges, RViews rv, RHdr* hdr, const int4* __restrict__ items, Slots sl,
                const uint8_t* __restrict__ flags, long long flags_cap,
                const float* __restrict__ Tfin, const int* __restrict__ lastin,
                const float* __restrict__ dLdimg, float4* __restrict__ grad2d)
{
    __shared__ EpShared sh;
    if (hdr->colours == 1) render_bwd_ep<REC, false>(feat, gid, ranges, rv, hdr, items, sl, flags, flags_cap, Tfin, lastin, dLdimg, grad2d, sh);
    else render_bwd_ep<REC, true>(feat, gid, ranges, rv, hdr, items, sl, flags, flags_cap, Tfin, lastin, dLdimg, grad2d, sh);
}

// Forward of 8x8 tiles with one pixel per thread, each warp on its own: a work
// item is one 8x4 block of a tile (or of a chunk of a split tile), taken per
// warp from the counter (the same compositing as k_render_fwd, pixel for
// pixel and bit for bit).  The warp stages its block's candidates in batches
// of 32 with the alpha test over the block's rectangle of pixel centres
// (tighter than the tile's), stops as soon as its own 32 pixels are done, and
// needs no CTA barrier.  Blend flags: the flag bytes are cleared before the
// launch, and each entry some pixel of the block blended gets bit 7 and the
// block's bit OR-ed into its byte (one 32-bit atomic OR per entry and block).
//
// Bound by instruction issue (87% of the slots busy), so the walk over the
// staged entries is one straight line for the whole warp, two entries a step:
// a pixel that an entry does not blend takes alpha 0, which changes neither T
// nor the colour; a pixel that has stopped (or lies outside the image) gets an
// alpha threshold no entry reaches; the stop rule is tested once per step, on
// the transmittance behind both entries (it never grows), and the rare step
// where some pixel stops is sorted out on the side; list positions and blend
// counts follow from the batch's blend mask.  Measured on 16 views of 1237x822,
// 480k Gaussians, mixed records: 2.82 ms with a walk that diverged per lane and
// a branch per entry -> 2.27 ms -> 2.09 ms with one address per staged pair and
// only the facing edges in the cull (on four of the views 781M -> 595M -> 543M
// warp instructions).
//
// An entry whose colour is not finite leaves no finite sum in any lane, whatever its
// weight; such a block's colours are formed again, entry by entry and only from those
// the pixel blends (a test of every batch's colours cost 0.6%, a second round of the
// walk's own loop 2.3%, this call 0.5% of the pass when all colours are finite).
template <int REC>
__device__ __noinline__ float3 blended_colour(const void* feat, const uint32_t* gid, int count, float pxc, float pyc,
                                              float T, bool on)
{
    float3 c = make_float3(0.f, 0.f, 0.f);
    for (int j = 0; j < count && __any_sync(0xffffffffu, on); ++j) {
        float4 ga, gb;
        float gc;
        load_record<REC>(feat, gid[j], ga, gb, gc);
        // (the roundings of the walk)
        const float dx = __fadd_rn(ga.x, -pxc), dy = __fadd_rn(ga.y, -pyc);
        const float p = fmaf(dx, fmaf(-kLog2e * ga.w, dy, __fmul_rn(-0.5f * kLog2e * ga.z, dx)),
                             __fmul_rn(__fmul_rn(-0.5f * kLog2e * gb.x, dy), dy));
        const float e = __fadd_rn(p, __log2f(gb.y));
        if (!on || !(gb.y >= kAlphaMin) || !(p <= 0.f && e >= kLog2AlphaMin)) continue;
        const float a = fminf(kAlphaMax, ex2_approx(e));
        const float Tn = fmaf(-a, T, T);
        if (Tn < kTMin) {
            on = false;
            continue;
        }
        const float w = __fmul_rn(a, T);
        c.x = fmaf(w, gb.z, c.x);
        c.y = fmaf(w, gb.w, c.y);
        c.z = fmaf(w, gc, c.z);
        T = Tn;
    }
    return c;
}

template <bool PROD, int REC>
// (16 blocks of 64 threads per SM, 64 registers: 0.366 -> 0.353 ms against the
// compiler's 56-register choice of 18 blocks)
__global__ void __launch_bounds__(64, 16)
k_render_fwd_w(const void* __restrict__ feat, const uint32_t* __restrict__ gid,
               const uint2* __restrict__ ranges, RViews rv, RHdr* hdr, const int4* __restrict__ items,
               const int4* __restrict__ sitems, Slots sl, uint8_t* __restrict__ flags, long long flags_cap,
               float* __restrict__ img, float* __restrict__ Tout, int* __restrict__ lastout,
               int* __restrict__ exout, int* __restrict__ blout)
{
    constexpr int B = 8, NPIX = 64;
    // staged entry pairs, five float4 each: (u, u', v, v'), (a, a', b, b')
    // prescaled conic, (c, c', log2 o, log2 o'), then r, g, b and the list
    // position (int bits) of either entry; one address per step
    __shared__ float4 s_pair[2][16 * kPairW];
    const bool planned = hdr->planned != 0 && items != nullptr;
    const int L = planned ? hdr->L : INT_MAX;
    const int count = PROD ? hdr->n_slots : (planned ? hdr->n_items : rv.total);
    const int4* list = PROD ? sitems : (planned ? items : nullptr);
    int* counter = PROD ? &hdr->cnt_prod : &hdr->cnt_fwd;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    float4* const sp = s_pair[wp];
    auto pos_of = [&](int slot) { return __float_as_int(sp[(slot >> 1) * kPairW + 3 + (slot & 1)].w); };
    const uint32_t lt = (1u << lane) - 1u;
    // threshold of a pixel that takes no entry: NaN, which no alpha reaches, not even an
    // infinite opacity's
    const float kNever = __int_as_float(0x7fc00000);
    auto never = [](float t) { return t != t; };
    if (!PROD && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&hdr->colours, 1);
    for (;;) {
    int blk = 0;
    const Item it = next_item_warp(counter, count, list, rv, &blk);
    if (it.tile < 0) break;
    if (PROD && it.c == it.nch - 1) continue;  // the last chunk's product is never needed
    const int tile = it.tile, tx = it.tx, ty = it.ty, W = it.W, H = it.H;
    const int lx = lane & 7, ly0 = 4 * blk + (lane >> 3);
    const int x = tx * B + lx;
    const int y = ty * B + ly0;
    const float pxc = (float)x + 0.5f, pyc = (float)y + 0.5f;
    const float bx0 = (float)(tx * B) + 0.5f, bx1 = bx0 + 7.f;
    const float by0 = (float)(ty * B + 4 * blk) + 0.5f, by1 = by0 + 3.f;
    const uint2 rg = ranges[tile];
    const int n = (int)(rg.y - rg.x);
    const bool split = it.slot0 >= 0;
    const int lo = split ? it.c * L : 0;
    const int hi = split ? (int)min((long long)n, (long long)lo + L) : n;
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    int last = 0, stop = -1, nbl = 0;
    // alpha threshold (log2): kNever once the pixel takes no further entry; Tend
    // is its transmittance when that differs from the one the walk keeps
    float thr = x < W && y < H ? kLog2AlphaMin : kNever;
    float Tend = -1.f;
    const int p = ly0 * B + lx;  // pixel within the tile
    if (!PROD && split && it.c > 0) {
        for (int c = 0; c < it.c; ++c) T *= sl.prod[(size_t)(it.slot0 + c) * NPIX + p];
        if (T < kTMin) {  // stopped in an earlier chunk
            thr = kNever;
            Tend = T;
            T = 1.f;
        }
    }
    bool alldone = __all_sync(0xffffffffu, never(thr));
    const f32x2 npx = f2_pack(-pxc, -pxc), npy = f2_pack(-pyc, -pyc);
    // the Gaussian indices of a batch are loaded one batch ahead, so a batch
    // waits only for its records
    uint32_t gn = lo + lane < hi ? gid[rg.x + lo + lane] : 0u;
    for (int base = lo; base < hi && !alldone; base += 32) {
        const int j = base + lane;
        const uint32_t g = gn;
        gn = j + 32 < hi ? gid[rg.x + j + 32] : 0u;
        bool keep = false;
        float4 ga, gb;
        float gc = 0.f, lo2 = 0.f;
        if (j < hi) {
            load_record<REC>(feat, g, ga, gb, gc);
            lo2 = __log2f(gb.y);
            keep = !block_skip(ga, gb, lo2, bx0, bx1, by0, by1);
        }
        const uint32_t km = __ballot_sync(0xffffffffu, keep);
        const int cnt = __popc(km);
        if (keep) {
            const int slot = __popc(km & lt);
            float4* q = sp + (slot >> 1) * kPairW;
            float* f = (float*)q + (slot & 1);
            f[0] = ga.x; f[2] = ga.y;
            f[4] = -0.5f * kLog2e * ga.z; f[6] = -kLog2e * ga.w;
            f[8] = -0.5f * kLog2e * gb.x; f[10] = lo2;
            q[3 + (slot & 1)] = make_float4(gb.z, gb.w, gc, __int_as_float(j));
        }
        if ((cnt & 1) && lane == 0) {  // the last pair's second half: an entry no pixel blends
            float4* q = sp + (cnt >> 1) * kPairW;
            float* f = (float*)q + 1;
            f[0] = 0.f; f[2] = 0.f; f[4] = 0.f; f[6] = 0.f; f[8] = 0.f; f[10] = __int_as_float(0xff800000);
            q[4] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncwarp();
        uint32_t mine = 0;  // staged entries this pixel blended
        // Offsets, quadratic forms and log2 alphas of the step's two entries run as
        // packed float32 pairs (the staging keeps an entry pair's fields side by
        // side): the same roundings as the scalar form, so the backward's test
        // agrees bit for bit.
        const float4* const qend = sp + ((cnt + 1) >> 1) * kPairW;
        uint32_t bit = 1u;
        for (const float4* q = sp; q < qend; q += kPairW, bit <<= 2) {
            const float4 uv = q[0], ab = q[1], cl = q[2];
            const f32x2 dx = f2_add(f2_pack(uv.x, uv.y), npx), dy = f2_add(f2_pack(uv.z, uv.w), npy);
            const f32x2 pu = f2_fma(dx, f2_fma(f2_pack(ab.z, ab.w), dy, f2_mul(f2_pack(ab.x, ab.y), dx)),
                                    f2_mul(f2_mul(f2_pack(cl.x, cl.y), dy), dy));
            const f32x2 eu = f2_add(pu, f2_pack(cl.z, cl.w));
            float p0, p1, e0, e1;
            f2_unpack(pu, p0, p1);
            f2_unpack(eu, e0, e1);
            const bool b0 = p0 <= 0.f && e0 >= thr, b1 = p1 <= 0.f && e1 >= thr;
            float a0 = b0 ? fminf(kAlphaMax, ex2_approx(e0)) : 0.f;
            float a1 = b1 ? fminf(kAlphaMax, ex2_approx(e1)) : 0.f;
            float T0 = fmaf(-a0, T, T);   // behind the first entry
            float T1 = fmaf(-a1, T0, T0);
            if (b0) mine |= bit;
            if (b1) mine |= bit << 1;
            bool leave = false;
            if (__any_sync(0xffffffffu, T1 < kTMin)) {
                if (T1 < kTMin) {  // this pixel stops, at the first entry that takes it below the threshold
                    const bool first = T0 < kTMin;
                    stop = __float_as_int(first ? q[3].w : q[4].w);
                    if (PROD) Tend = first ? T0 : T1;  // below the threshold: every later chunk is stopped
                    mine &= first ? bit - 1u : 2u * bit - 1u;
                    a1 = 0.f;
                    if (first) {
                        a0 = 0.f;
                        T0 = T;
                    }
                    T1 = T0;
                    thr = kNever;
                }
                leave = __all_sync(0xffffffffu, never(thr));
            }
            if (!PROD) {
                const float4 q0 = q[3], q1 = q[4];
                const float w0 = a0 * T, w1 = a1 * T0;
                c0 = fmaf(w1, q1.x, fmaf(w0, q0.x, c0));
                c1 = fmaf(w1, q1.y, fmaf(w0, q0.y, c1));
                c2 = fmaf(w1, q1.z, fmaf(w0, q0.z, c2));
            }
            T = T1;
            if (leave) break;
        }
        if (!PROD) {
            nbl += __popc(mine);
            if (mine) last = pos_of(31 - __clz((int)mine)) + 1;
            if (flags) {
                const uint32_t bm = __reduce_or_sync(0xffffffffu, mine);
                if (lane < cnt && ((bm >> lane) & 1u)) {
                    const long long gj = (long long)rg.x + pos_of(lane);
                    if ((gj | 3) < flags_cap)
                        atomicOr((unsigned int*)(flags + (gj & ~3ll)),
                                 (unsigned int)(kFlagWarpBits | (1u << blk)) << (8 * (int)(gj & 3)));
                }
            }
        }
        alldone = __all_sync(0xffffffffu, never(thr));
        __syncwarp();
    }
    if (Tend >= 0.f) T = Tend;
    if (!PROD && __any_sync(0xffffffffu, !finite_colour(c0, c1, c2))) {
        if (lane == 0) atomicOr(&hdr->colours, 2);
        float T0 = 1.f;
        for (int c = 0; split && c < it.c; ++c) T0 *= sl.prod[(size_t)(it.slot0 + c) * NPIX + p];
        const float3 c = blended_colour<REC>(feat, gid + rg.x + lo, hi - lo, pxc, pyc, T0,
                                             x < W && y < H && !(T0 < kTMin));
        c0 = c.x; c1 = c.y; c2 = c.z;
    }
    if (split) {
        const size_t s0 = (size_t)(it.slot0 + it.c) * NPIX + (size_t)p;
        if (PROD) {
            sl.prod[s0] = T;
        } else {
            sl.tout[s0] = T;
            sl.c0[s0] = c0; sl.c1[s0] = c1; sl.c2[s0] = c2;
            sl.last[s0] = last | (stop >= 0 ? kStopFlag : 0);
            sl.nbl[s0] = nbl;
            sl.stop[s0] = stop;
        }
        continue;
    }
    if (x < W && y < H) {
        const size_t HW = (size_t)W * H;
        float* im = img + 3 * it.poff;
        const size_t pix = (size_t)y * W + x;
        im[pix] = c0 + T * rv.bg0;
        im[HW + pix] = c1 + T * rv.bg1;
        im[2 * HW + pix] = c2 + T * rv.bg2;
        Tout[it.poff + pix] = T;
        lastout[it.poff + pix] = last;
        if (exout) exout[it.poff + pix] = stop >= 0 ? stop + 1 : n;
        if (blout) blout[it.poff + pix] = nbl;
    }
    }  // work items
}

}  // namespace dg

static dg::RViews make_rviews(const dg_camera* cams, int n, int B, const dg_raster_opts* o)
{
    dg::RViews rv;
    rv.n = n;
    int tiles = 0;
    long long pix = 0;
    for (int v = 0; v < n; ++v) {
        rv.W[v] = cams[v].width;
        rv.H[v] = cams[v].height;
        rv.TX[v] = (cams[v].width + B - 1) / B;
        rv.toff[v] = tiles;
        rv.poff[v] = pix;
        tiles += rv.TX[v] * ((cams[v].height + B - 1) / B);
        pix += (long long)cams[v].width * cams[v].height;
    }
    rv.toff[n] = tiles;
    rv.total = tiles;
    rv.bg0 = o->bg[0]; rv.bg1 = o->bg[1]; rv.bg2 = o->bg[2];
    return rv;
}

// Resident CTAs of a kernel on this device.
template <typename Kern>
static int resident_ctas(Kern kern, int threads)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0);
    const long long g = (long long)(sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
    return (int)(g < (1 << 20) ? g : (1 << 20));
}

// Layout of the render workspace for n_tiles tiles of edge B.
struct RenderWs {
    dg::RHdr* hdr;
    uint8_t* flags;       // per pair: blended by some pixel of its tile (written by the forward)
    long long flags_cap;  // pairs the flag array holds
    int4* items;
    int4* sitems;
    uint64_t* toff;
    uint64_t* bsum;
    dg::Slots sl;
    int cap;
    size_t bytes;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Chunk slots: 2^20 pixels' worth (32 MiB of per-pixel chunk state).
static int slot_cap(int B) { return (1 << 20) / (B * B); }

// Layout of the render workspace; the per-pair flag array takes whatever
// follows the fixed part (ws_bytes - fixed bytes).
static RenderWs render_ws_fixed(void* base, long long n_tiles, int B, bool split);
static RenderWs render_ws(void* base, long long n_tiles, int B, bool split, size_t ws_bytes = 0)
{
    RenderWs w = render_ws_fixed(base, n_tiles, B, split);
    w.flags = (uint8_t*)base + w.bytes;
    w.flags_cap = ws_bytes > w.bytes ? (long long)(ws_bytes - w.bytes) : 0;
    if (!base) w.flags = nullptr;
    return w;
}

static RenderWs render_ws_fixed(void* base, long long n_tiles, int B, bool split)
{
    RenderWs w{};
    char* p = (char*)base;
    size_t off = 256;
    w.hdr = (dg::RHdr*)p;
    if (!split) { w.bytes = off; return w; }
    const int cap = slot_cap(B);
    const long long nb = (n_tiles + dg::SCAN_TILE - 1) / dg::SCAN_TILE;
    const size_t npix = (size_t)cap * B * B;
    w.cap = cap;
    w.items = (int4*)(p + off);  off = align256(off + sizeof(int4) * (size_t)(n_tiles + cap));
    w.sitems = (int4*)(p + off); off = align256(off + sizeof(int4) * (size_t)cap);
    w.toff = (uint64_t*)(p + off); off = align256(off + sizeof(uint64_t) * (size_t)(n_tiles > 0 ? n_tiles : 1));
    w.bsum = (uint64_t*)(p + off); off = align256(off + sizeof(uint64_t) * (size_t)(nb > 0 ? nb : 1));
    float** fp[5] = {&w.sl.prod, &w.sl.tout, &w.sl.c0, &w.sl.c1, &w.sl.c2};
    for (int i = 0; i < 5; ++i) { *fp[i] = (float*)(p + off); off = align256(off + sizeof(float) * npix); }
    int** ip[3] = {&w.sl.last, &w.sl.nbl, &w.sl.stop};
    for (int i = 0; i < 3; ++i) { *ip[i] = (int*)(p + off); off = align256(off + sizeof(int) * npix); }
    w.bytes = off;
    return w;
}

// Split plan of n tiles: hdr and the item arrays.
static void plan_items(const uint2* rg, int n, const RenderWs& w, const dg::SplitCfg& cfg, cudaStream_t s)
{
    if (n <= dg::PLAN_TILES) {
        dg::k_plan_small<<<1, dg::PLAN_THREADS, 0, s>>>(rg, n, w.hdr, cfg, w.items, w.sitems);
        dg_note_launch();
        return;
    }
    const int nb = (int)(((long long)n + dg::SCAN_TILE - 1) / dg::SCAN_TILE);
    dg::k_scan_reduce<<<nb, dg::SCAN_THREADS, 0, s>>>(dg::LoadLen{rg}, n, w.bsum);
    dg::k_scan_top<<<1, 1024, 0, s>>>(w.bsum, nb, &w.hdr->M);
    dg_note_launch(2);
    dg::exclusive_scan(dg::LoadChunks{rg, w.hdr, cfg}, n, w.toff, w.bsum, &w.hdr->totals, s);
    const int pg = (n + 255) / 256;
    dg::k_plan_items<<<pg < 1024 ? pg : 1024, 256, 0, s>>>(rg, n, w.hdr, cfg, w.toff, w.items, w.sitems);
    dg_note_launch();
}

// Tile 8, one pixel per thread: the warp-per-block forward (k_render_fwd_w).
template <int REC>
static dg_status launch_fwd_w(const float* feat, const uint32_t* gid, const uint32_t* ranges, const dg::RViews& rv,
                              const RenderWs& w, int split_req, float* img, float* T, int* last, int* ex, int* bl,
                              cudaStream_t s)
{
    const uint2* rg = (const uint2*)ranges;
    auto kern = dg::k_render_fwd_w<false, REC>;
    const int R = resident_ctas(kern, 64);
    cudaMemsetAsync(w.hdr, 0, 256, s);
    if (w.flags && w.flags_cap > 0) cudaMemsetAsync(w.flags, 0, (size_t)w.flags_cap, s);
    const bool split = rv.total > 0 && (split_req > 0 || (split_req == 0 && rv.total < 2LL * R));
    if (split) {
        const dg::SplitCfg cfg{split_req, R, w.cap};
        plan_items(rg, rv.total, w, cfg, s);
        auto kprod = dg::k_render_fwd_w<true, REC>;
        kprod<<<resident_ctas(kprod, 64), 64, 0, s>>>((const void*)feat, gid, rg, rv, w.hdr, w.items, w.sitems, w.sl,
                                                      nullptr, 0, img, T, last, ex, bl);
        dg_note_launch();
    }
    const int grid = split ? R : (R < rv.total ? R : (rv.total > 0 ? rv.total : 1));
    kern<<<grid, 64, 0, s>>>((const void*)feat, gid, rg, rv, w.hdr, w.items, w.sitems, w.sl, w.flags, w.flags_cap,
                             img, T, last, ex, bl);
    dg_note_launch();
    if (split) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        dg::k_render_combine<8><<<4 * (sms > 0 ? sms : 1), 64, 0, s>>>(rg, rv, w.hdr, w.sitems, w.sl, img, T, last,
                                                                      ex, bl);
        dg_note_launch();
    }
    return DG_OK;
}

template <int B, int PPT, int REC>
static dg_status launch_fwd(const float* feat, const uint32_t* gid, const uint32_t* ranges, const dg::RViews& rv,
                            const RenderWs& w, int split_req, float* img, float* T, int* last, int* ex, int* bl,
                            cudaStream_t s)
{
    const uint2* rg = (const uint2*)ranges;
    if (B == 8 && PPT == 1) return launch_fwd_w<REC>(feat, gid, ranges, rv, w, split_req, img, T, last, ex, bl, s);
    auto kern = dg::k_render_fwd<B, PPT, false, REC>;
    const int R = resident_ctas(kern, B * B / PPT);
    cudaMemsetAsync(w.hdr, 0, 256, s);
    // automatic: split only when the tiles alone leave resident CTAs idle
    // (with at least two tiles per CTA the persistent launch balances itself,
    // and splitting costs the product pass)
    const bool split = rv.total > 0 && (split_req > 0 || (split_req == 0 && rv.total < 2LL * R));
    if (split) {
        const dg::SplitCfg cfg{split_req, R, w.cap};
        plan_items(rg, rv.total, w, cfg, s);
        auto kprod = dg::k_render_fwd<B, PPT, true, REC>;
        kprod<<<resident_ctas(kprod, B * B / PPT), B * B / PPT, 0, s>>>(
            (const void*)feat, gid, rg, rv, w.hdr, w.items, w.sitems, w.sl, nullptr, 0, img, T, last, ex, bl);
        dg_note_launch();
    }
    const int grid = split ? R : (R < rv.total ? R : (rv.total > 0 ? rv.total : 1));
    kern<<<grid, B * B / PPT, 0, s>>>((const void*)feat, gid, rg, rv, w.hdr, w.items, w.sitems, w.sl, w.flags,
                                      w.flags_cap, img, T, last, ex, bl);
    dg_note_launch();
    if (split) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        dg::k_render_combine<B><<<4 * (sms > 0 ? sms : 1), B * B, 0, s>>>(rg, rv, w.hdr, w.sitems, w.sl, img, T,
                                                                         last, ex, bl);
        dg_note_launch();
    }
    return DG_OK;
}

// Backward of 8x8 tiles, one pixel per thread: entry-parallel gradient sums
// (k_render_bwd_ep) unless DG_BWD_EP is defined to 0.
#ifndef DG_BWD_EP
#define DG_BWD_EP 1
#endif

template <int B, int PPT, int REC>
static void launch_bwd(const float* feat, const uint32_t* gid, const uint32_t* ranges, const dg::RViews& rv,
                       const RenderWs& w, const float* T, const int* last, const float* dL, float* g2, cudaStream_t s)
{
    if (DG_BWD_EP && B == 8 && PPT == 1) {
        auto kew = dg::k_render_bwd_ep<REC>;
        const int grid = resident_ctas(kew, 64);
        cudaMemsetAsync(&w.hdr->cnt_bwd, 0, sizeof(int), s);
        kew<<<grid, 64, 0, s>>>((const void*)feat, gid, (const uint2*)ranges, rv, w.hdr, w.items, w.sl, w.flags,
                                w.flags_cap, T, last, dL, (float4*)g2);
        dg_note_launch();
        return;
    }
    auto kern = dg::k_render_bwd<B, PPT, REC>;
    const int grid = resident_ctas(kern, B * B / PPT);
    cudaMemsetAsync(&w.hdr->cnt_bwd, 0, sizeof(int), s);
    kern<<<grid, B * B / PPT, 0, s>>>((const void*)feat, gid, (const uint2*)ranges, rv, w.hdr, w.items, w.sl,
                                      w.flags, w.flags_cap, T, last, dL, (float4*)g2);
    dg_note_launch();
}

template <int REC>
static void fwd_dispatch(int B, int ppt, const float* feat, const uint32_t* gid, const uint32_t* ranges,
                         const dg::RViews& rv, const RenderWs& w, int sp, float* img, float* T, int* last, int* ex,
                         int* bl, cudaStream_t s)
{
    if (B == 8 && ppt == 2) launch_fwd<8, 2, REC>(feat, gid, ranges, rv, w, sp, img, T, last, ex, bl, s);
    else if (B == 8) launch_fwd<8, 1, REC>(feat, gid, ranges, rv, w, sp, img, T, last, ex, bl, s);
    else if (ppt == 1) launch_fwd<16, 1, REC>(feat, gid, ranges, rv, w, sp, img, T, last, ex, bl, s);
    else if (ppt == 2) launch_fwd<16, 2, REC>(feat, gid, ranges, rv, w, sp, img, T, last, ex, bl, s);
    else launch_fwd<16, 4, REC>(feat, gid, ranges, rv, w, sp, img, T, last, ex, bl, s);
}

template <int REC>
static void bwd_dispatch(int B, int ppt, const float* feat, const uint32_t* gid, const uint32_t* ranges,
                         const dg::RViews& rv, const RenderWs& w, const float* T, const int* last, const float* dL,
                         float* g2, cudaStream_t s)
{
    if (B == 8 && ppt == 2) launch_bwd<8, 2, REC>(feat, gid, ranges, rv, w, T, last, dL, g2, s);
    else if (B == 8) launch_bwd<8, 1, REC>(feat, gid, ranges, rv, w, T, last, dL, g2, s);
    else if (ppt == 1) launch_bwd<16, 1, REC>(feat, gid, ranges, rv, w, T, last, dL, g2, s);
    else if (ppt == 2) launch_bwd<16, 2, REC>(feat, gid, ranges, rv, w, T, last, dL, g2, s);
    else launch_bwd<16, 4, REC>(feat, gid, ranges, rv, w, T, last, dL, g2, s);
}

// Pixels per thread used for (tile, request): tile 16 -> 1, 2 or 4 (0 selects
// the default of each pass), tile 8 -> 1 or 2 (default 1).
static int resolve_ppt(const dg_raster_opts* o, bool backward)
{
    const int req = o->pixels_per_thread;
    if (o->tile == 8) return req == 2 ? 2 : 1;
    if (req == 1 || req == 2 || req == 4) return req;
    return backward ? 4 : 2;
}

bool dg_check_cameras(const dg_camera* cams, int n_views);

static long long total_tiles(const dg_camera* cams, int n_views, int B)
{
    long long t = 0;
    for (int v = 0; v < n_views; ++v)
        t += (long long)((cams[v].width + B - 1) / B) * ((cams[v].height + B - 1) / B);
    return t;
}

static bool render_args(const dg_camera* cams, int n_views, const dg_raster_opts* opts, void* ws, size_t ws_bytes)
{
    if (!dg_check_cameras(cams, n_views)) return false;
    if (!opts) { dg_set_error("opts null"); return false; }
    if (opts->tile != 8 && opts->tile != 16) { dg_set_error("render supports tile 8 or 16, got %d", opts->tile); return false; }
    const int p = opts->pixels_per_thread;
    if (p != 0 && p != 1 && p != 2 && p != 4) { dg_set_error("pixels_per_thread must be 0, 1, 2 or 4, got %d", p); return false; }
    if (total_tiles(cams, n_views, opts->tile) >= (1LL << 30)) { dg_set_error("too many tiles"); return false; }
    if (opts->record != 0 && opts->record != 1) { dg_set_error("record must be 0 (float32) or 1 (mixed), got %d", opts->record); return false; }
    const size_t need = dg_render_workspace_size(cams, n_views, opts, 0);  // the fixed part; flags use the rest
    if (!ws || ws_bytes < need) { dg_set_error("render workspace missing or too small (%zu < %zu bytes)", ws_bytes, need); return false; }
    if (((uintptr_t)ws) & 255u) { dg_set_error("render workspace must be 256-byte aligned"); return false; }
    return true;
}

extern "C" size_t dg_render_workspace_size(const dg_camera* cams, int32_t n_views, const dg_raster_opts* opts,
                                           int64_t M_cap)
{
    if (!cams || !opts || n_views < 1 || n_views > DG_MAX_VIEWS || (opts->tile != 8 && opts->tile != 16)) return 0;
    if (M_cap < 0) return 0;
    for (int v = 0; v < n_views; ++v)
        if (cams[v].width <= 0 || cams[v].height <= 0) return 0;
    const size_t fixed = render_ws_fixed(nullptr, total_tiles(cams, n_views, opts->tile), opts->tile,
                                         opts->split_len >= 0).bytes;
    return fixed + (((size_t)M_cap + 255) & ~(size_t)255);
}

extern "C" dg_status dg_render_fwd(const float* feat, const uint32_t* gid, const uint32_t* ranges,
                                   const dg_camera* cams, int32_t n_views, const dg_raster_opts* opts, float* img,
                                   float* T_final, int32_t* last, int32_t* examined, int32_t* blended, void* ws,
                                   size_t ws_bytes, dg_stream stream)
{
    if (!render_args(cams, n_views, opts, ws, ws_bytes)) return DG_ERR_ARG;
    if (!ranges || !img || !T_final || !last) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    if (feat && (((uintptr_t)feat) & 15u)) { dg_set_error("feat must be 16-byte aligned"); return DG_ERR_ARG; }
    cudaStream_t s = (cudaStream_t)stream;
    const int B = opts->tile;
    const dg::RViews rv = make_rviews(cams, n_views, B, opts);
    const RenderWs w = render_ws(ws, rv.total, B, opts->split_len >= 0, ws_bytes);
    const int sp = opts->split_len;
    const int ppt = resolve_ppt(opts, false);
    if (opts->record == 1) fwd_dispatch<1>(B, ppt, feat, gid, ranges, rv, w, sp, img, T_final, last, examined, blended, s);
    else fwd_dispatch<0>(B, ppt, feat, gid, ranges, rv, w, sp, img, T_final, last, examined, blended, s);
    return dg_check_launch("render_fwd");
}

extern "C" dg_status dg_render_bwd(const float* feat, const uint32_t* gid, const uint32_t* ranges,
                                   const dg_camera* cams, int32_t n_views, const dg_raster_opts* opts,
                                   const float* T_final, const int32_t* last, const float* dL_dimg, int64_t n_records,
                                   float* grad2d, void* ws, size_t ws_bytes, dg_stream stream)
{
    if (!render_args(cams, n_views, opts, ws, ws_bytes)) return DG_ERR_ARG;
    if (n_records < 0) { dg_set_error("n_records < 0"); return DG_ERR_ARG; }
    if (!ranges || !T_final || !last || !dL_dimg || (n_records > 0 && !grad2d)) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    if (grad2d && (((uintptr_t)grad2d) & 15u)) { dg_set_error("grad2d must be 16-byte aligned"); return DG_ERR_ARG; }
    cudaStream_t s = (cudaStream_t)stream;
    if (n_records > 0) cudaMemsetAsync(grad2d, 0, sizeof(float) * DG_FEAT_FLOATS * (size_t)n_records, s);
    const int B = opts->tile;
    const dg::RViews rv = make_rviews(cams, n_views, B, opts);
    const RenderWs w = render_ws(ws, rv.total, B, opts->split_len >= 0, ws_bytes);
    const int ppt = resolve_ppt(opts, true);
    if (opts->record == 1) bwd_dispatch<1>(B, ppt, feat, gid, ranges, rv, w, T_final, last, dL_dimg, grad2d, s);
    else bwd_dispatch<0>(B, ppt, feat, gid, ranges, rv, w, T_final, last, dL_dimg, grad2d, s);
    return dg_check_launch("render_bwd");
}
