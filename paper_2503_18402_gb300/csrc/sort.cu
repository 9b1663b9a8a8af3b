// sort.cu -- tile binning: depth order, pair emission, stable tile sort, ranges.
//
// The per-tile lists must come out ordered by (tile, depth bits, Gaussian
// index).  Instead of one radix sort over 64-bit (tile | depth) keys of all
// M pairs (6 passes of 8 bits), the order is built in two cheaper stages:
//   1. a stable 32-bit LSD radix sort of the visible depths (ties keep the
//      index order);
//   2. pairs are emitted in depth order, then stably sorted by tile id alone
//      (ceil(log2(tiles)) bits: 2 passes at 1237x822 / 8^2 = 15965 tiles).
// Stability of stage 2 preserves the depth order inside each tile, so the
// result equals the lexicographic (tile, depth bits, index) order.
// Several views: records are r = v * P + i; each view's records and pairs are
// a segment sorted on its own (onesweep.cuh), with tile ids local to the view;
// view v's pairs follow view v - 1's, and its ranges start at its first tile
// of the global range table.  The pair payload is the record index r.
//
// Stage 1 (dg_bin_count): one kernel counts the digits of all four depth
// passes, the visible records and the pairs of each view; the first pass then
// drops the culled records, so the other three move only the visible ones.
// Stage 2 (dg_bin_sort): one kernel walks the records in depth order, forms
// each one's tile rect (16 bytes), scans their pair counts (look-back) and
// counts the lowest tile digit (each tile pass counts the next one); the first
// tile pass emits its pairs straight into its ranking, so unsorted pairs never
// reach memory; the last one extends the ranges of the tiles whose runs it
// stages, so sorted keys are never stored.
// Measured (2M Gaussians, one 1237x822 view, 5.9M pairs / 653k Gaussians, 16
// views of 1237x822 to 309x205, 33M pairs): 0.315 / 1.16 ms both stages, against
// 0.41 / 1.88 ms with all views sorted as one sequence, culled records carried
// along, the pairs emitted to memory and histogram, scan and scatter kernels per
// tile pass.
#include "onesweep.cuh"
#include "tilekey.cuh"

namespace dg {

// Zeroed at the start of each phase: phase 1's counters ...
struct BinCtl1 {
    uint32_t ctr[4];
    int32_t err;                                // DG_ERR_TIMEOUT once a wait gave up
    unsigned long long nvis[DG_MAX_VIEWS];      // visible records of each view
    unsigned long long npair[DG_MAX_VIEWS];     // pairs of each view
    uint32_t hist[DG_MAX_VIEWS][4][OS_BINS];    // depth digit counts
};
// ... and phase 2's.
struct BinCtl2 {
    uint32_t ctr[1 + BIN_MAXPASS];              // records, tile passes
    int32_t err;                                // DG_ERR_TIMEOUT or DG_ERR_CUDA
    int32_t bad;                                // the records' pairs are not usable: emit nothing
    uint32_t hist[DG_MAX_VIEWS][BIN_MAXPASS][OS_BINS];  // tile digit counts
};

// --------------------------------------------------------------- depth order
constexpr int DH_THREADS = 512;
constexpr int DH_IPT = 8;

// Digit counts of the four depth passes and the visible records and pairs of
// each view (blockIdx.y) in one read of depths and tile counts.
__global__ void __launch_bounds__(DH_THREADS)
k_depth_hist(const float* __restrict__ depth, const int* __restrict__ tiles, long long P, BinCtl1* ctl)
{
    __shared__ uint32_t h[4][OS_BINS];
    __shared__ unsigned long long s_pairs;
    for (int i = threadIdx.x; i < 4 * OS_BINS; i += DH_THREADS) (&h[0][0])[i] = 0;
    if (threadIdx.x == 0) s_pairs = 0;
    __syncthreads();
    const int v = blockIdx.y;
    const float* d = depth + (size_t)v * P;
    const int* tl = tiles + (size_t)v * P;
    unsigned long long pairs = 0;
    for (long long base = (long long)blockIdx.x * (DH_THREADS * DH_IPT); base < P;
         base += (long long)gridDim.x * (DH_THREADS * DH_IPT)) {
        int n[DH_IPT];
        uint32_t k[DH_IPT];
#pragma unroll
        for (int q = 0; q < DH_IPT; ++q) {
            const long long i = base + q * DH_THREADS + threadIdx.x;
            n[q] = i < P ? tl[i] : 0;
            k[q] = i < P ? __float_as_uint(d[i]) : 0u;
        }
#pragma unroll
        for (int q = 0; q < DH_IPT; ++q) {
            if (n[q] > 0) {
                pairs += (unsigned long long)n[q];
                atomicAdd(&h[0][k[q] & 255u], 1u);
                atomicAdd(&h[1][(k[q] >> 8) & 255u], 1u);
                atomicAdd(&h[2][(k[q] >> 16) & 255u], 1u);
                atomicAdd(&h[3][k[q] >> 24], 1u);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    if ((threadIdx.x & 31) == 0 && pairs) atomicAdd(&s_pairs, pairs);
    __syncthreads();
    uint32_t* g = &ctl->hist[v][0][0];
    uint32_t vis = 0;
    for (int i = threadIdx.x; i < 4 * OS_BINS; i += DH_THREADS) {
        const uint32_t c = (&h[0][0])[i];
        if (c) atomicAdd(&g[i], c);
        if (i < OS_BINS) vis += c;
    }
    vis = __reduce_add_sync(0xffffffffu, vis);
    if ((threadIdx.x & 31) == 0 && vis) atomicAdd(&ctl->nvis[v], (unsigned long long)vis);
    if (threadIdx.x == 0 && s_pairs) atomicAdd(&ctl->npair[v], s_pairs);
}

// First depth pass: the visible records of the view, key = depth bits.
struct SrcDepth {
    const float* depth;
    const int* tiles;
    template <int IPT>
    __device__ __forceinline__ uint32_t load(const SegTile& st, int nv, uint32_t*, uint32_t*, uint32_t (&key)[IPT],
                                             int warp, int lane) const
    {
        const int seg = warp * 32 * IPT + lane;
        const long long first = st.off + (long long)st.t * (OS_THREADS * IPT) + seg;
        const float* dp = depth + first;
        const int* tp = tiles + first;
        uint32_t ok = 0;
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const bool on = seg + 32 * i < nv;
            key[i] = on ? __float_as_uint(dp[32 * i]) : 0u;
            ok |= (on && tp[32 * i] > 0 ? 1u : 0u) << i;
        }
        return ok;
    }
    template <int IPT>
    __device__ __forceinline__ void values(const SegTile& st, int, const uint32_t*, uint32_t (&val)[IPT], int warp,
                                           int lane) const
    {
        const uint32_t first = (uint32_t)(st.off + (long long)st.t * (OS_THREADS * IPT)) + warp * 32 * IPT + lane;
#pragma unroll
        for (int i = 0; i < IPT; ++i) val[i] = first + 32 * i;
    }
};

// --------------------------------------------------------------- records in depth order
// Records per thread: four, or one while that many records fill at most two blocks
// per SM at four: a lone block's chain (gathers, counts, look-back) is most of the
// kernel then (5k records on 120 tiles, phase 2: 38 -> 30 us; 334k records 36 with one
// or four, 504k 46 with four and 54 with one).
constexpr long long REC_SMALL_MAX = 152LL * 2 * OS_THREADS * 4;
static int rec_ipt(long long n) { return n <= REC_SMALL_MAX ? 1 : 4; }

// A record in depth order: its tiles (RecTiles), and its index in the view in .w.

// One tile of a view's records in depth order: gathers each one's
// rect or tile mask, writes it and its first pair (relative to the view's
// pairs), the record holding each pair tile's first pair, and the counts of the
// lowest tile digit.  Also clears the range table.  Positions fit 32 bits: with
// more pairs than M_cap (< 2^32) nothing is written.  The prefix comes first and
// the digits are counted while the first warp looks back.
template <int REC_IPT>
__global__ void __launch_bounds__(OS_THREADS)
k_records(const float4* __restrict__ feat, const int* __restrict__ radius, const uint32_t* __restrict__ order,
          long long P, int B, TileGrid tg, TileKey tk, Segs sg, const unsigned long long* __restrict__ npair,
          long long M_cap, int pair_tile, const int* __restrict__ err1, BinCtl2* ctl, uint64_t* __restrict__ look,
          uint4* __restrict__ rec, uint32_t* __restrict__ poff, uint32_t* __restrict__ bstart,
          uint2* __restrict__ ranges)
{
    constexpr int REC_TILE = OS_THREADS * REC_IPT;
    __shared__ int diff[OS_BINS];
    __shared__ uint32_t direct[OS_BINS];
    __shared__ uint32_t s_cycles;
    __shared__ uint32_t ssum[OS_WARPS];
    __shared__ uint32_t s_ex;
    __shared__ long long s_tb;     // first pair tile of the view
    __shared__ SegTile s_st;
    __shared__ int s_dsum[OS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_tiles = tg.off[tg.n];
    for (long long i = (long long)blockIdx.x * OS_THREADS + threadIdx.x; i < n_tiles;
         i += (long long)gridDim.x * OS_THREADS)
        ranges[i] = make_uint2(0u, 0u);
    if (warp == 0) {
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(&ctl->ctr[0], 1u);
        b = __shfl_sync(0xffffffffu, b, 0);
        seg_tile(sg, b, REC_TILE, &s_st, lane);
        __syncwarp();
        const long long m = lane < sg.V ? (long long)npair[lane] : 0;
        const long long mt = warp_incl_scan<long long>((m + pair_tile - 1) / pair_tile, lane) -
                             (m + pair_tile - 1) / pair_tile;
        if (lane == s_st.v) s_tb = mt;
        const long long msum = __shfl_sync(0xffffffffu, warp_incl_scan<long long>(m, lane), 31);
        __syncwarp();
        if (lane == 0 && msum > M_cap) s_st.v = -1;  // too many pairs: nothing is emitted
        if (lane == 0 && *err1 != 0) {               // the order is not complete: nothing is read by it
            s_st.v = -1;
            ctl->bad = 1;
        }
    }
    diff[threadIdx.x] = 0;
    direct[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_cycles = 0;
    __syncthreads();
    const SegTile st = s_st;
    if (st.v < 0) return;
    const int TX = tg.TX[st.v], TY = tg.TY[st.v];
    const long long m_view = (long long)npair[st.v];
    const long long first = (long long)st.t * REC_TILE + warp * (32 * REC_IPT) + lane;  // position in the view
    const uint32_t* ord = order + st.off;
    uint32_t r[REC_IPT];
#pragma unroll
    for (int k = 0; k < REC_IPT; ++k) r[k] = first + 32 * k < st.n ? ord[first + 32 * k] : 0u;
    float2 uv[REC_IPT];
    float4 f2[REC_IPT];
    int rad[REC_IPT];
#pragma unroll
    for (int k = 0; k < REC_IPT; ++k) {
        const float4* f = feat + 3 * (size_t)r[k];
        uv[k] = *(const float2*)f;
        f2[k] = f[2];
        rad[k] = radius[r[k]];
    }
    uint32_t cnt[REC_IPT], ex[REC_IPT];
    uint4 out[REC_IPT];
    uint32_t run = 0;
#pragma unroll
    for (int k = 0; k < REC_IPT; ++k) {
        const Rect q = tile_rect(uv[k].x, uv[k].y, rad[k], B, TX, TY);
        const RecTiles t = pack_tiles((uint32_t)q.x0, (uint32_t)q.y0, (uint32_t)(q.x1 - q.x0), (uint32_t)(q.y1 - q.y0),
                                      __float_as_uint(f2[k].y), __float_as_uint(f2[k].z), TX);
        out[k] = make_uint4(t.corner, t.lo, t.hi, (uint32_t)(r[k] - (uint32_t)(st.v * P)));
        cnt[k] = first + 32 * k >= st.n ? 0u
               : t.lo ? (uint32_t)(__popc(t.lo) + __popc(t.hi)) : rect_width(t.hi, TX) * rect_height(t.hi, TX);
        const uint32_t inc = warp_incl_scan<uint32_t>(cnt[k], lane);
        ex[k] = run + inc - cnt[k];
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) ssum[warp] = run;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < OS_WARPS; ++w) {
        pre += w < warp ? ssum[w] : 0u;
        tot += ssum[w];
    }
    if (warp == 0) {
        uint64_t* lk = look + st.tbase + st.t;
        if (lane == 0) st_relaxed(lk, (st.t == 0 ? kLbInc : kLbAgg) | tot);
        uint64_t e = 0;
        if (st.t > 0) {
            if (!os_lookback_warp(lk - st.t, st.t, &e, lane)) {
                if (lane == 0) atomicExch(&ctl->err, DG_ERR_TIMEOUT);
                ctl->bad = 1;
            }
            if (lane == 0) st_relaxed(lk, kLbInc | ((e + tot) & kLbCount));
        }
        if (lane == 0) {
            s_ex = (uint32_t)e;
            // (cannot differ for the depths, tiles, records and radii of one projection)
            if ((long long)(st.t + 1) * REC_TILE >= st.n && (long long)(e + tot) != m_view) {
                atomicCAS(&ctl->err, 0, DG_ERR_CUDA);
                ctl->bad = 1;
            }
        }
    }
    // counts of the lowest digit (or of the whole key, when it is one digit)
    const uint32_t dm = (1u << tk.width[0]) - 1u;
#pragma unroll
    for (int k = 0; k < REC_IPT; ++k) {
        if (cnt[k] == 0) continue;
        const uint32_t x0 = out[k].x & 0xffffu, y0 = out[k].x >> 16;
        const bool masked = out[k].y != 0;
        const uint32_t rw = rect_width(out[k].z, TX), rh = rect_height(out[k].z, TX);
        if (tk.linear) {
            auto add = [&](uint32_t i, int n) { atomicAdd(&diff[i], n); };
            auto cyc = [&](uint32_t n) { atomicAdd(&s_cycles, n); };
            const uint32_t a = y0 * (uint32_t)TX + x0;
            if (masked) count_linear_mask(a, TX, out[k].y, out[k].z, tk.width[0], add, cyc);
            else count_linear_rect(a, TX, rw, rh, tk.width[0], add, cyc);
        } else if (masked) {
            // pairs of each of the mask's eight columns
            uint32_t any = out[k].y | out[k].z;
            any |= any >> 16;
            any = (any | (any >> 8)) & 255u;
#pragma unroll 1
            for (; any; any &= any - 1) {
                const int c = __ffs((int)any) - 1;
                const uint32_t col = 0x01010101u << c;
                atomicAdd(&direct[(x0 + c) & dm], (uint32_t)(__popc(out[k].y & col) + __popc(out[k].z & col)));
            }
        } else {
            // columns x0 .. x0 + w - 1, each h times: cyclic through the digit's values
            count_run(x0, rw, rh, tk.width[0], [&](uint32_t i, int n) { atomicAdd(&diff[i], n); },
                      [&](uint32_t n) { atomicAdd(&s_cycles, n); });
        }
    }
    __syncthreads();
    const int mine = diff[threadIdx.x];
    const int dinc = warp_incl_scan<int>(mine, lane);
    if (lane == 31) s_dsum[warp] = dinc;
    __syncthreads();
    uint32_t c0 = (uint32_t)dinc + s_cycles + direct[threadIdx.x];
#pragma unroll
    for (int w = 0; w < OS_WARPS; ++w) c0 += w < warp ? (uint32_t)s_dsum[w] : 0u;
    if (threadIdx.x <= dm && c0) atomicAdd(&ctl->hist[st.v][0][threadIdx.x], c0);
    pre += s_ex;
#pragma unroll
    for (int k = 0; k < REC_IPT; ++k) {
        const long long s = first + 32 * k;
        if (s >= st.n) continue;
        const uint32_t a = pre + ex[k];
        rec[st.off + s] = out[k];
        poff[st.off + s] = a;
        const long long e = (long long)a + cnt[k];
        for (long long b = ((long long)a + pair_tile - 1) / pair_tile; b * pair_tile < e && b * pair_tile < m_view; ++b)
            bstart[s_tb + b] = (uint32_t)s;
    }
}

// First tile pass: the pairs of its tile, formed from the records in depth
// order.  A thread takes a record and writes its pairs to their places in
// shared memory (tile mask: a walk over the set bits, at most 64); the rects
// larger than a mask are written by the whole warp, 32 pairs at a time (small
// whole rects too took the pass 280 instead of 40 us on 1.6M records of one or
// two tiles).  (One thread per 16 consecutive pairs, walking along the records, left
// 16-way bank conflicts and a chain of dependent record loads.  A warp-round
// of 32 records takes about 240 instructions; issue and the pass behind it bound
// the kernel: 96 us on 5.9M pairs.)
struct SrcEmit {
    const uint4* rec;
    const uint32_t* poff;
    const uint32_t* bstart;
    const unsigned long long* nvis;
    long long P;
    TileGrid tg;
    int linear, xbits;
    BinCtl2* ctl;
    template <int IPT>
    __device__ __forceinline__ uint32_t load(const SegTile& st, int nv, uint32_t* sk, uint32_t* sv,
                                             uint32_t (&key)[IPT], int warp, int lane) const
    {
        constexpr int TILE = OS_THREADS * IPT;
        const uint32_t base = st.t * (uint32_t)TILE;  // first pair (relative to the view's)
        const uint4* rv = rec + st.v * P;
        const uint32_t* pv = poff + st.v * P;
        const uint32_t s_lo = bstart[st.tbase + st.t];
        const uint32_t s_hi = (long long)base + TILE < st.n ? bstart[st.tbase + st.t + 1] : (uint32_t)nvis[st.v] - 1u;
        const int nr = (int)(s_hi - s_lo) + 1;
        const uint32_t row = key_row(linear, xbits, tg.TX[st.v]);
        const uint32_t n_keys = (uint32_t)tg.TY[st.v] * row;
        const uint32_t rbase = (uint32_t)(st.v * P);
        bool bad = false;
        // (whole warps step together: the last round's idle lanes hold an empty mask)
        for (int i0 = warp * 32; i0 < nr; i0 += OS_THREADS) {
            const bool on = i0 + lane < nr;
            const uint32_t s = s_lo + (uint32_t)(on ? i0 + lane : 0);
            const uint4 c = rv[s];
            const int p0 = (int)(pv[s] - base);  // of the record's first pair in this tile's array (may be negative)
            const bool whole = on && c.y == 0;
            const uint32_t g = rbase + c.w;
            const uint32_t k0 = (c.x >> 16) * row + (c.x & 0xffffu);
            // the mask's two words in turn (most masks have no bit above the fourth tile row)
            int p = p0;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t mk = on && !whole ? (half ? c.z : c.y) : 0u;
                const uint32_t kh = k0 + 4u * half * row;
#pragma unroll 1
                for (; mk; ++p, mk &= mk - 1) {
                    const uint32_t b = (uint32_t)__ffs((int)mk) - 1u;
                    const uint32_t kk = kh + (b >> 3) * row + (b & 7u);
                    if ((uint32_t)p < (uint32_t)nv) {
                        bad = bad || kk >= n_keys;
                        sk[p] = kk < n_keys ? kk : 0u;
                        sv[p] = g;
                    }
                }
            }
            uint32_t todo = __ballot_sync(0xffffffffu, whole);
            while (todo) {
                const int l = __ffs((int)todo) - 1;
                todo &= todo - 1;
                const int q0 = __shfl_sync(0xffffffffu, p0, l);
                const uint32_t size = __shfl_sync(0xffffffffu, c.z, l);
                const uint32_t w = rect_width(size, tg.TX[st.v]), h = rect_height(size, tg.TX[st.v]);
                const uint32_t kb = __shfl_sync(0xffffffffu, k0, l), gg = __shfl_sync(0xffffffffu, g, l);
                const int a = q0 < 0 ? 0 : q0;
                const long long end = (long long)q0 + (long long)w * h;
                const int e = end < nv ? (int)end : nv;
                for (int i = a + lane; i < e; i += 32) {
                    const uint32_t j = (uint32_t)(i - q0), y = j / w;
                    const uint32_t kk = kb + y * row + (j - y * w);
                    bad = bad || kk >= n_keys;
                    sk[i] = kk < n_keys ? kk : 0u;
                    sv[i] = gg;
                }
            }
        }
        // (cannot happen for consistent inputs; no key leaves the grid)
        if (bad) atomicCAS(&ctl->err, 0, DG_ERR_CUDA);
        __syncthreads();
        const int seg = warp * 32 * IPT + lane;
        uint32_t ok = 0;
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const bool in = seg + 32 * i < nv;
            key[i] = in ? sk[seg + 32 * i] : 0u;
            ok |= (in ? 1u : 0u) << i;
        }
        return ok;
    }
    template <int IPT>
    __device__ __forceinline__ void values(const SegTile&, int nv, const uint32_t* sv, uint32_t (&val)[IPT], int warp,
                                           int lane) const
    {
        const int seg = warp * 32 * IPT + lane;
#pragma unroll
        for (int i = 0; i < IPT; ++i) val[i] = seg + 32 * i < nv ? sv[seg + 32 * i] : 0u;
    }
};

// Ranges from their (complement of the start, end) form, and the call's status.  With
// any error every range is empty: gid may hold words of an earlier call then, and the
// passes that read the lists are launched before the host sees the status.
__global__ void k_ranges_final(uint2* __restrict__ ranges, int n_tiles, const long long* M, long long M_cap,
                               const int* err1, const BinCtl2* ctl, int* status)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int st = *M > M_cap ? DG_ERR_CAPACITY : (*err1 != 0 ? *err1 : ctl->err);
    if (i < n_tiles) {
        const uint2 r = ranges[i];
        if (st != 0) ranges[i] = make_uint2(0u, 0u);
        else if (r.y != 0u) ranges[i].x = ~r.x;
    }
    if (i == 0) *status = st;
}

// Workspace layout (offsets 256-byte aligned).  The pair count and the
// record-sized buffers come first so that their offsets do not depend on
// M_cap: phase 1 and phase 2 may be called with workspaces laid out for
// different capacities as long as the record part was carried over.
struct BinWs {
    long long* M;                       // total pair count
    BinCtl1* ctl1;                      // phase 1 control block, then its look-back words
    void* look1;                        // [4][tiles][256]
    size_t look1_pass;                  // bytes of one pass
    size_t zero1;                       // bytes phase 1 clears from ctl1 on
    uint32_t *dk0, *dv0, *dk1, *dv1;   // depth sort, N each
    uint4* rec;                         // records in depth order, N
    uint32_t* poff;                     // N first pairs
    BinCtl2* ctl2;                      // phase 2 control block, then its look-back words
    uint64_t* rlook;                    // records scan
    void* look2;                        // [BIN_MAXPASS][pair tiles][256], 2^width words of a tile used
    size_t zero2_fixed;                 // bytes phase 2 clears from ctl2 up to look2
    uint32_t *pk0, *pv0, *pk1, *pv1;   // pair sort, M_cap each
    uint32_t* bstart;                   // record holding each pair tile's first pair
    size_t bytes;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Items per thread of a pass over at most n items, and the look-back word size.
static int os_ipt(long long n, long long small_max) { return n <= small_max ? OS_IPT_SMALL : OS_IPT_BIG; }
static size_t os_word(long long n) { return n < (1ll << 30) ? 4 : 8; }
// Tiles of `views` segments holding n items together (each ends in a partial tile).
static long long os_tiles(long long n, int views, int tile) { return n / tile + views; }
// The largest number of such tiles for any count up to n, when counts up to small_max
// take tiles of small_tile items: the layout's sizes do not shrink as counts grow, so
// that a workspace laid out for more serves fewer.
static long long os_tiles_upto(long long n, int views, long long small_max, int small_tile, int big_tile)
{
    const long long s = os_tiles(n < small_max ? n : small_max, views, small_tile);
    const long long b = n > small_max ? os_tiles(n, views, big_tile) : 0;
    return s > b ? s : b;
}
static long long pass_tiles_upto(long long n, int views, long long small_max)
{
    return os_tiles_upto(n, views, small_max, OS_THREADS * OS_IPT_SMALL, OS_THREADS * OS_IPT_BIG);
}

static BinWs bin_layout(char* base, long long P, int n_views, long long M_cap)
{
    const long long N = P * n_views;
    BinWs w;
    size_t o = 0;
    auto take = [&](size_t bytes) { char* p = base + o; o += align256(bytes); return p; };
    w.M = (long long*)take(8);
    const size_t c1 = o;
    w.ctl1 = (BinCtl1*)take(sizeof(BinCtl1));
    w.look1_pass = align256(os_word(N) * OS_BINS * (size_t)os_tiles(N, n_views, OS_THREADS * os_ipt(N, OS_SMALL_DEPTH)));
    w.zero1 = o - c1 + 4 * w.look1_pass;
    w.look1 = take(4 * align256(os_word(N) * OS_BINS * (size_t)pass_tiles_upto(N, n_views, OS_SMALL_DEPTH)));
    w.dk0 = (uint32_t*)take(4 * N); w.dv0 = (uint32_t*)take(4 * N);
    w.dk1 = (uint32_t*)take(4 * N); w.dv1 = (uint32_t*)take(4 * N);
    w.rec = (uint4*)take(16 * N);
    w.poff = (uint32_t*)take(4 * N);
    const size_t c2 = o;
    w.ctl2 = (BinCtl2*)take(sizeof(BinCtl2));
    w.rlook = (uint64_t*)take(8 * os_tiles_upto(N, n_views, REC_SMALL_MAX, OS_THREADS, OS_THREADS * 4));
    w.zero2_fixed = o - c2;
    // (from here on the offsets depend on M_cap)
    const long long pt = pass_tiles_upto(M_cap, n_views, OS_SMALL_PAIRS);
    w.look2 = take(BIN_MAXPASS * align256(os_word(M_cap) * OS_BINS * pt));
    w.pk0 = (uint32_t*)take(4 * M_cap); w.pv0 = (uint32_t*)take(4 * M_cap);
    w.pk1 = (uint32_t*)take(4 * M_cap); w.pv1 = (uint32_t*)take(4 * M_cap);
    w.bstart = (uint32_t*)take(4 * (pt + 1));
    w.bytes = o;
    return w;
}

// One pass over at most n_max items; the kernel's form by the item count.
template <int NB, class Src>
static void os_pass(const Src& src, const Segs& sg, const OsPass& ps, long long n_max, int ipt, cudaStream_t s)
{
    const int grid = (int)os_tiles(n_max, sg.V, OS_THREADS * ipt);
    if (ipt == OS_IPT_SMALL) k_os_pass<OS_IPT_SMALL, uint32_t, NB><<<grid, OS_THREADS, 0, s>>>(src, sg, ps);
    else if (os_word(n_max) == 4) k_os_pass<OS_IPT_BIG, uint32_t, NB><<<grid, OS_THREADS, 0, s>>>(src, sg, ps);
    else k_os_pass<OS_IPT_BIG, uint64_t, NB><<<grid, OS_THREADS, 0, s>>>(src, sg, ps);
    dg_note_launch();
}

}  // namespace dg

extern "C" size_t dg_bin_workspace_size(int64_t P, int32_t n_views, int64_t M_cap)
{
    if (P < 0 || M_cap < 0 || n_views < 1 || n_views > DG_MAX_VIEWS) return 0;
    return dg::bin_layout(nullptr, P, n_views, M_cap).bytes;
}

extern "C" dg_status dg_bin_count(const float* depth, const int32_t* tiles, int64_t P, int32_t n_views, void* ws,
                                  size_t ws_bytes, int64_t M_cap, int64_t* M_out, dg_stream stream)
{
    if (P < 0 || n_views < 1 || n_views > DG_MAX_VIEWS || P * n_views > (int64_t)UINT32_MAX || M_cap < 0 ||
        M_cap > (int64_t)UINT32_MAX) {
        dg_set_error("bad sizes P=%lld n_views=%d M_cap=%lld", (long long)P, n_views, (long long)M_cap);
        return DG_ERR_ARG;
    }
    if (!ws || !M_out || (P > 0 && (!depth || !tiles))) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    const long long N = P * n_views;
    const dg::BinWs w = dg::bin_layout((char*)ws, P, n_views, M_cap);
    if (ws_bytes < w.bytes) { dg_set_error("workspace %zu < %zu bytes", ws_bytes, w.bytes); return DG_ERR_CAPACITY; }
    cudaStream_t s = (cudaStream_t)stream;
    cudaMemsetAsync(w.ctl1, 0, w.zero1, s);  // counters, error word, look-back words
    if (N == 0) {
        cudaMemsetAsync(w.M, 0, sizeof(long long), s);
        cudaMemsetAsync(M_out, 0, sizeof(long long), s);
        return dg_check_launch("bin_count");
    }
    using namespace dg;
    const long long per_block = DH_THREADS * DH_IPT;
    long long hb = (P + per_block - 1) / per_block;
    const long long hmax = (152 * 4 + n_views - 1) / n_views;
    if (hb > hmax) hb = hmax;
    k_depth_hist<<<dim3((unsigned)hb, (unsigned)n_views), DH_THREADS, 0, s>>>(depth, tiles, P, w.ctl1);
    dg_note_launch();
    // depth passes: (depth, record) -> 1 -> 0 -> 1 -> records only in dv0
    auto pass = [&](int p, uint32_t* ko, uint32_t* vo) {
        OsPass ps{};
        ps.look = (char*)w.look1 + p * w.look1_pass;
        ps.ctr = &w.ctl1->ctr[p];
        ps.hist = &w.ctl1->hist[0][p][0];
        ps.hist_stride = 4 * OS_BINS;
        ps.err = &w.ctl1->err;
        ps.shift = 8 * p;
        ps.mask = OS_BINS - 1;
        ps.kout = ko;
        ps.vout = vo;
        if (p == 0) {
            ps.m_views = w.ctl1->npair;
            ps.m_ws = w.M;
            ps.m_out = (long long*)M_out;
        }
        return ps;
    };
    const Segs all{n_views, nullptr, P, P, LLONG_MAX, nullptr};
    const Segs vis{n_views, w.ctl1->nvis, 0, P, LLONG_MAX, nullptr};
    const int ipt = os_ipt(N, OS_SMALL_DEPTH);
    os_pass<8>(SrcDepth{depth, tiles}, all, pass(0, w.dk1, w.dv1), N, ipt, s);
    os_pass<8>(SrcKV{w.dk1, w.dv1}, vis, pass(1, w.dk0, w.dv0), N, ipt, s);
    os_pass<8>(SrcKV{w.dk0, w.dv0}, vis, pass(2, w.dk1, w.dv1), N, ipt, s);
    // (the highest digit, sign and upper exponent bits, has few distinct values)
    os_pass<0>(SrcKV{w.dk1, w.dv1}, vis, pass(3, nullptr, w.dv0), N, ipt, s);
    return dg_check_launch("bin_count");
}

bool dg_check_cameras(const dg_camera* cams, int n_views);

extern "C" dg_status dg_bin_sort(const float* feat, const int32_t* radius, int64_t P, const dg_camera* cams,
                                 int32_t n_views, int32_t tile, void* ws, size_t ws_bytes, int64_t M_cap,
                                 uint32_t* gid, uint32_t* ranges, int32_t* status, dg_stream stream)
{
    if (!dg_check_cameras(cams, n_views)) return DG_ERR_ARG;
    if (tile < 1 || tile > 64) { dg_set_error("bad tile %d", tile); return DG_ERR_ARG; }
    if (P < 0 || P * n_views > (int64_t)UINT32_MAX || M_cap < 0 || M_cap > (int64_t)UINT32_MAX) {
        dg_set_error("bad sizes");
        return DG_ERR_ARG;
    }
    if (!ws || !ranges || !status || (P > 0 && (!feat || !radius)) || (M_cap > 0 && !gid)) {
        dg_set_error("null buffer");
        return DG_ERR_ARG;
    }
    using namespace dg;
    const long long N = P * n_views;
    const BinWs w = bin_layout((char*)ws, P, n_views, M_cap);
    if (ws_bytes < w.bytes) { dg_set_error("workspace %zu < %zu bytes", ws_bytes, w.bytes); return DG_ERR_CAPACITY; }
    TileGrid tg;
    tg.n = n_views;
    long long n_tiles = 0, most = 1;
    for (int v = 0; v < n_views; ++v) {
        tg.TX[v] = (cams[v].width + tile - 1) / tile;
        tg.TY[v] = (cams[v].height + tile - 1) / tile;
        tg.off[v] = (int)n_tiles;
        const long long nt = (long long)tg.TX[v] * tg.TY[v];
        n_tiles += nt;
        if (nt > most) most = nt;
    }
    tg.off[n_views] = (int)n_tiles;
    if (n_tiles > (1ll << 30)) { dg_set_error("too many tiles"); return DG_ERR_ARG; }
    cudaStream_t s = (cudaStream_t)stream;
    const TileKey tk = tile_key(tg);
    const int ipt = os_ipt(M_cap, OS_SMALL_PAIRS);
    const int pair_tile = OS_THREADS * ipt;
    size_t look_at[BIN_MAXPASS + 1] = {0};
    for (int p = 0; p < tk.npass; ++p)
        look_at[p + 1] = look_at[p] + align256((os_word(M_cap) << tk.width[p]) * (size_t)os_tiles(M_cap, n_views, pair_tile));
    if (N > 0 && M_cap > 0) {
        cudaMemsetAsync(w.ctl2, 0, w.zero2_fixed + look_at[tk.npass], s);
        const Segs vis{n_views, w.ctl1->nvis, 0, P, LLONG_MAX, nullptr};
        auto records = rec_ipt(N) == 1 ? k_records<1> : k_records<4>;
        records<<<(int)os_tiles(N, n_views, OS_THREADS * rec_ipt(N)), OS_THREADS, 0, s>>>(
            (const float4*)feat, radius, w.dv0, P, tile, tg, tk, vis, w.ctl1->npair, M_cap, pair_tile,
            &w.ctl1->err, w.ctl2, w.rlook, w.rec, w.poff, w.bstart, (uint2*)ranges);
        dg_note_launch();
        const Segs pairs{n_views, w.ctl1->npair, 0, -1, M_cap, &w.ctl2->bad};
        uint32_t *ki = nullptr, *vi = nullptr;
        for (int p = 0; p < tk.npass; ++p) {
            const bool last = p == tk.npass - 1;
            uint32_t* ko = last ? nullptr : (p & 1) ? w.pk1 : w.pk0;
            uint32_t* vo = last ? gid : (p & 1) ? w.pv1 : w.pv0;
            OsPass ps{};
            ps.look = (char*)w.look2 + look_at[p];
            ps.ctr = &w.ctl2->ctr[1 + p];
            ps.hist = &w.ctl2->hist[0][p][0];
            ps.hist_stride = BIN_MAXPASS * OS_BINS;
            ps.err = &w.ctl2->err;
            ps.shift = tk.shift[p];
            ps.mask = (1u << tk.width[p]) - 1u;
            ps.kout = ko;
            ps.vout = vo;
            ps.hist_next = last ? nullptr : &w.ctl2->hist[0][p + 1][0];
            ps.mask_next = last ? 0u : (1u << tk.width[p + 1]) - 1u;
            if (last) {
                ps.linear = tk.linear;
                ps.xbits = tk.xbits;
                for (int v = 0; v < n_views; ++v) ps.TX[v] = tg.TX[v];
                ps.ranges = (uint2*)ranges;
                for (int v = 0; v <= n_views; ++v) ps.toff[v] = tg.off[v];
            }
            if (p == 0) os_pass<8>(SrcEmit{w.rec, w.poff, w.bstart, w.ctl1->nvis, P, tg, tk.linear, tk.xbits, w.ctl2}, pairs, ps, M_cap, ipt, s);
            else os_pass<8>(SrcKV{ki, vi}, pairs, ps, M_cap, ipt, s);
            ki = ko;
            vi = vo;
        }
    } else {
        cudaMemsetAsync(w.ctl2, 0, sizeof(BinCtl2), s);
        cudaMemsetAsync(ranges, 0, sizeof(uint32_t) * 2 * n_tiles, s);
    }
    k_ranges_final<<<(int)((n_tiles + 255) / 256), 256, 0, s>>>((uint2*)ranges, (int)n_tiles, w.M, M_cap,
                                                              &w.ctl1->err, w.ctl2, status);
    dg_note_launch();
    return dg_check_launch("bin_sort");
}

// ------------------------------------------------------------ look-back probe
namespace dg {
// One warp: form 0 and 1 run in its first lane, form 2 in all of them.
__global__ void k_lookback_probe(const void* look, long long t, int stride, int d, int max_polls, int form,
                                 uint64_t* sum, int* err)
{
    const int lane = threadIdx.x;
    if (lane == 0) *err = 0;
    __threadfence();
    __syncwarp();
    if (form == 2) {
        uint64_t s = 0;
        const bool ok = os_lookback_warp((const uint64_t*)look, t, &s, lane, max_polls);
        if (lane == 0) {
            *sum = s;
            if (!ok) atomicExch(err, DG_ERR_TIMEOUT);
        }
    } else if (lane == 0) {
        *sum = form == 0 ? os_lookback((const uint64_t*)look, t, stride, d, err, max_polls)
                         : (uint64_t)os_lookback((const uint32_t*)look, t, stride, d, err, max_polls);
    }
}
}  // namespace dg

extern "C" dg_status dg_lookback_probe_form(const void* look, int64_t tile, int32_t stride, int32_t digit,
                                            int32_t max_polls, int32_t form, uint64_t* sum, int32_t* err,
                                            dg_stream stream)
{
    if (!sum || !err || (tile > 0 && !look)) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    if (form < 0 || form > 2) { dg_set_error("bad look-back form %d", form); return DG_ERR_ARG; }
    if (tile < 0 || stride < 1 || digit < 0 || digit >= stride || (form == 2 && stride != 1)) {
        dg_set_error("bad look-back probe: tile=%lld stride=%d digit=%d", (long long)tile, stride, digit);
        return DG_ERR_ARG;
    }
    if (max_polls < 0 || max_polls > dg::kLbPolls) {
        dg_set_error("max_polls %d outside 0..%d", max_polls, dg::kLbPolls);
        return DG_ERR_ARG;
    }
    dg::k_lookback_probe<<<1, 32, 0, (cudaStream_t)stream>>>(look, tile, stride, digit, max_polls, form, sum, err);
    dg_note_launch();
    return dg_check_launch("lookback_probe");
}

extern "C" dg_status dg_lookback_probe(const uint64_t* look, int64_t tile, int32_t stride, int32_t digit,
                                       int32_t max_polls, uint64_t* sum, int32_t* err, dg_stream stream)
{
    return dg_lookback_probe_form(look, tile, stride, digit, max_polls, 0, sum, err, stream);
}
