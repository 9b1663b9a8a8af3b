// onesweep.cuh -- stable single-kernel radix passes over the views of a batch,
// built on decoupled look-back (Merrill & Garland, "Single-pass Parallel
// Prefix Scan with Decoupled Look-back", 2016; the radix form follows
// Adinets & Merrill, "Onesweep: A Faster Least Significant Digit Radix Sort
// for GPUs", 2022).  Both stages of the binning use them: the depth order of
// the records and the tile order of the pairs.
//
// Segments.  Each view's items are a segment of their own: a block belongs to
// one view, counts and look-back stay within it, and the view index is never a
// sort digit.  (Sorting all views as one sequence took one more pass over the
// records and, at 16 views of 1237x822, three 6-bit passes over the pairs
// instead of two 7-bit ones.)
//
// A pass is one kernel.  Each CTA takes a tile number from a counter when it
// starts, ranks its THREADS x IPT items by digit within warp-owned segments
// (so the pass is stable), publishes its per-digit totals, and sums the totals
// of its view's earlier tiles by walking back over their published words until
// one holds an inclusive prefix.  A CTA only waits on tiles taken by CTAs that
// started before it and that never wait on a later tile, so every wait ends;
// each is bounded all the same, and a wait that gives up records
// DG_ERR_TIMEOUT and carries on with what it has.  The start of each digit
// comes from the digit counts of the whole view, counted before the first pass
// and scanned by every CTA together with its own totals.
//
// What bounds a pass: about 170 instructions per warp and 32 items at 40% of
// the issue slots, the rest waits (a lone tile's chain of ticket, loads, ranking,
// prefix, look-back and scatter takes 7-9 us), not its 16 B per item.  Measured
// on 1.7M (key, value) items with 8-bit digits: 32 us with 2048-item tiles,
// 64-bit words, a 16-word look-back window polled without pause and 64-bit
// match masks; 22 us with 4096-item tiles, a 4-word window and a pause between
// polls (more words in flight flood L2: a 32-word window took 55 us).  Four
// votes' worth of instructions per digit bit became four instructions, and a
// value is loaded only after its rank is known, so that four CTAs fit an SM (on
// 33M pairs 1.16 against 1.23 ms for the whole binning with three; tiles of
// 2048, 3072 or 5120 items 1.40, 1.23 and 1.37).  At 64 registers for that the
// 4096-item passes keep 72 to 104 bytes of a thread in local memory.  At 100k items a
// 1024-item tile takes 6 us against 9 for 4096: the small tile is used while the
// items fill at most two and a half of them per SM in the depth order (334k items,
// four passes and counts, 50 -> 45 us; 467k items 53 -> 58, 531k 54 -> 60) and five,
// the most that are resident, in the tile order, whose first pass also emits (330k
// to 690k pairs: 7 to 15 us less of 45 to 64; 840k to 1.1M pairs 52 to 71 us, up to 9
// more, with small tiles).
#pragma once

#include "scan.cuh"
#include "tilekey.cuh"

namespace dg {
namespace {

constexpr int OS_THREADS = 256;
constexpr int OS_WARPS = OS_THREADS / 32;
constexpr int OS_BINS = 256;              // 8-bit digits, one thread per digit
constexpr int OS_IPT_BIG = 16;
constexpr int OS_IPT_SMALL = 4;
constexpr long long OS_SMALL_DEPTH = 152LL * 5 / 2 * OS_THREADS * OS_IPT_SMALL;
constexpr long long OS_SMALL_PAIRS = 152LL * 5 * OS_THREADS * OS_IPT_SMALL;
constexpr uint64_t kLbAgg = 1ull << 62;   // 64-bit word holding the tile's own total
constexpr uint64_t kLbInc = 2ull << 62;   // 64-bit word holding the inclusive prefix
constexpr uint64_t kLbCount = (1ull << 62) - 1;
constexpr int kLbPolls = 1 << 20;         // polls of one word before giving up

// Look-back words: the top two bits hold the state (0 not published, 1 own
// total, 2 inclusive prefix), the rest the count.  32-bit words serve segments
// below 2^30 items, 64-bit ones the rest.
template <typename Word>
struct LbWord {
    static constexpr int kShift = 8 * (int)sizeof(Word) - 2;
    static constexpr Word kCount = ((Word)1 << kShift) - 1;
    static __device__ __forceinline__ Word agg(Word c) { return ((Word)1 << kShift) | c; }
    static __device__ __forceinline__ Word inc(Word c) { return ((Word)2 << kShift) | c; }
};

__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t* p)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(uint64_t* p, uint64_t v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Sum of the counts the tiles before tile t published in column d of a
// [tiles][stride] word array, up to and including the nearest inclusive word;
// OS_WINDOW predecessors are read at once.
constexpr int OS_WINDOW = 4;
template <typename Word>
__device__ inline Word os_lookback(const Word* look, long long t, int stride, int d, int* err,
                                   int max_polls = kLbPolls)
{
    Word sum = 0;
    long long j = t;  // the window covers tiles j - OS_WINDOW .. j - 1
    int polls = 0;
    while (j > 0) {
        Word w[OS_WINDOW];
#pragma unroll
        for (int q = 0; q < OS_WINDOW; ++q)
            w[q] = j - 1 - q >= 0 ? ld_relaxed(look + (j - 1 - q) * stride + d) : LbWord<Word>::inc(0);
        int used = OS_WINDOW;
#pragma unroll
        for (int q = 0; q < OS_WINDOW; ++q) {
            if (used < OS_WINDOW) break;
            const Word st = w[q] >> LbWord<Word>::kShift;
            if (st == 0) {
                used = q;  // tile j - 1 - q has not published yet: read again from there
            } else {
                sum += w[q] & LbWord<Word>::kCount;
                if (st == 2) return sum;
            }
        }
        j -= used;
        if (used < OS_WINDOW) {
            if (++polls > max_polls) {
                atomicExch(err, DG_ERR_TIMEOUT);
                return sum;
            }
            __nanosleep(40);
        }
    }
    return sum;
}

// The same sum for one column of 64-bit words, taken by a whole warp, 32
// predecessors a time; false when a wait gave up.
__device__ inline bool os_lookback_warp(const uint64_t* look, long long t, uint64_t* out, int lane,
                                        int max_polls = kLbPolls)
{
    uint64_t& sum = *out;
    sum = 0;
    long long j = t;
    int polls = 0;
    while (j > 0) {
        const uint64_t w = j - 1 - lane >= 0 ? ld_relaxed(look + (j - 1 - lane)) : kLbInc;
        const uint32_t none = __ballot_sync(0xffffffffu, (w >> 62) == 0);
        const uint32_t inc = __ballot_sync(0xffffffffu, (w >> 62) == 2);
        // lanes before the first unpublished word and up to the first inclusive one
        const int lim = none ? __ffs(none) - 1 : 32;
        const int first = inc ? __ffs(inc) - 1 : 32;
        const int use = first < lim ? first + 1 : lim;
        uint64_t x = lane < use ? w & kLbCount : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        sum += x;
        if (first < lim) return true;
        j -= use;
        if (use < 32) {
            if (++polls > max_polls) return false;
            __nanosleep(40);
        }
    }
    return true;
}

// The views' items: view v holds cnt[v] items (or `fixed` when cnt is null),
// starting at v * stride, or right behind view v - 1's when stride < 0.  When
// all views hold more than `cap` items together, or *bad is set, there is
// nothing to do.
struct Segs {
    int V;
    const unsigned long long* cnt;
    long long fixed, stride, cap;
    const int* bad;
};

// A block's tile: view (-1: none left), tile number in the view, the view's
// item count, first item and first tile (over all views).
struct SegTile {
    int v;
    uint32_t t;
    long long n, off, tbase;
};

// Tile b of the views in `tile`-item tiles; called by one whole warp.
__device__ inline void seg_tile(const Segs& sg, uint32_t b, int tile, SegTile* out, int lane)
{
    const long long n = lane < sg.V ? (sg.cnt ? (long long)sg.cnt[lane] : sg.fixed) : 0;
    const long long nt = (n + tile - 1) / tile;
    const long long nt_inc = warp_incl_scan<long long>(nt, lane);
    const long long n_inc = warp_incl_scan<long long>(n, lane);
    const long long total = __shfl_sync(0xffffffffu, n_inc, 31);
    const bool run = total <= sg.cap && !(sg.bad && *sg.bad != 0);
    const bool mine = run && lane < sg.V && (long long)b >= nt_inc - nt && (long long)b < nt_inc;
    if (lane == 0) out->v = -1;
    __syncwarp();
    if (mine) {
        out->v = lane;
        out->t = (uint32_t)((long long)b - (nt_inc - nt));
        out->n = n;
        out->off = sg.stride < 0 ? n_inc - n : lane * sg.stride;
        out->tbase = nt_inc - nt;
    }
}

struct OsPass {
    void* look;            // [tiles][mask + 1] look-back words of this pass, zero before the launch
    uint32_t* ctr;         // this pass's tile counter, zero before the launch
    const uint32_t* hist;  // view v's digit counts of this pass at hist + v * hist_stride
    int hist_stride;
    uint32_t* hist_next;   // nullable: counts of the next digit to add this tile's to
    uint32_t mask_next;
    int* err;
    int shift;
    uint32_t mask;
    uint32_t* kout;        // nullable: values only
    uint32_t* vout;
    uint2* ranges;         // nullable: the last tile pass's ranges (complement of the start, end), zero before the launch
    int linear, xbits;     // with ranges: the form of the keys (TileKey)
    int TX[DG_MAX_VIEWS], toff[DG_MAX_VIEWS + 1];  // with ranges: tiles per row and first tile of each view
    const unsigned long long* m_views;  // nullable: the views' pair counts, summed into *m_ws and *m_out
    long long* m_ws;
    long long* m_out;
};

// Key sources of a pass: load() fills the warp-striped keys (item k of lane l
// of warp w at position w * 32 IPT + 32 k + l of the tile) and returns the bit
// mask of those that exist; values() fills their values, after the ranks are
// known (held from the start they would not fit the registers of four CTAs per
// SM).  sk, sv: IPT * OS_THREADS words of scratch each; sv is left as load()
// wrote it until values() returns on every thread.
struct SrcKV {
    const uint32_t* k;
    const uint32_t* v;
    template <int IPT>
    __device__ __forceinline__ uint32_t load(const SegTile& st, int nv, uint32_t*, uint32_t*, uint32_t (&key)[IPT],
                                             int warp, int lane) const
    {
        const int seg = warp * 32 * IPT + lane;
        const uint32_t* kp = k + st.off + (long long)st.t * (OS_THREADS * IPT) + seg;
        if (nv == OS_THREADS * IPT) {
#pragma unroll
            for (int i = 0; i < IPT; ++i) key[i] = kp[32 * i];
            return (1u << IPT) - 1u;
        }
        uint32_t ok = 0;
#pragma unroll
        for (int i = 0; i < IPT; ++i) {
            const bool on = seg + 32 * i < nv;
            key[i] = on ? kp[32 * i] : 0u;
            ok |= (on ? 1u : 0u) << i;
        }
        return ok;
    }
    template <int IPT>
    __device__ __forceinline__ void values(const SegTile& st, int nv, const uint32_t*, uint32_t (&val)[IPT], int warp,
                                           int lane) const
    {
        const int seg = warp * 32 * IPT + lane;
        const uint32_t* vp = v + st.off + (long long)st.t * (OS_THREADS * IPT) + seg;
#pragma unroll
        for (int i = 0; i < IPT; ++i) val[i] = seg + 32 * i < nv ? vp[32 * i] : 0u;
    }
};

// Lanes of the warp with this lane's NB-bit digit, among those in `on` (which
// holds this lane): per digit bit one vote, and the vote or its complement kept
// by the lane's own bit.
template <int NB>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, uint32_t on)
{
    uint32_t m = on;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        asm("{\n\t.reg .pred p;\n\t.reg .b32 t, b;\n\t"
            "and.b32 t, %1, %2;\n\t"
            "setp.ne.u32 p, t, 0;\n\t"
            "vote.sync.ballot.b32 b, p, 0xffffffff;\n\t"
            "@p and.b32 %0, %0, b;\n\t"
            "@!p lop3.b32 %0, %0, b, 0, 0x30;\n\t}"
            : "+r"(m) : "r"(d), "r"(1u << q));
    }
    return m;
}

// Stable rank of a warp's items among its items of the same digit, in position
// order; wcnt: the warp's running count per digit (zero on entry, the totals on
// return).  FULL: every item exists.  NB: digit bits to vote on, 0 for
// __match_any_sync (fewer instructions when a warp holds few distinct digits).
template <int IPT, int NB, bool FULL>
__device__ __forceinline__ void os_rank(const uint32_t (&key)[IPT], uint32_t (&rank)[IPT], uint32_t ok,
                                        uint32_t shift, uint32_t mask, uint32_t* wcnt, int lane)
{
    const uint32_t lt = (1u << lane) - 1u;
    // all peer masks first, then the running counts (a chain through shared memory)
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const uint32_t d = (key[k] >> shift) & mask;
        const bool on = FULL || ((ok >> k) & 1u);
        if (NB == 0) rank[k] = __match_any_sync(0xffffffffu, on ? d : 0x10000u + (uint32_t)lane);
        else rank[k] = digit_peers<NB>(d, FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, on));
    }
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const uint32_t m = rank[k];
        uint32_t* c = wcnt + ((key[k] >> shift) & mask);
        const uint32_t before = *c, below = __popc(m & lt);
        __syncwarp();
        if (below == 0 && (FULL || ((ok >> k) & 1u))) *c = before + __popc(m);
        __syncwarp();
        rank[k] = before + below;
    }
}

// One stable pass on digit (key >> shift) & mask; NB as os_rank's (at least the
// digit's width, or 0).
template <int IPT, typename Word, int NB, class Src>
__global__ void __launch_bounds__(OS_THREADS, IPT == OS_IPT_BIG ? 4 : 5)
k_os_pass(Src src, Segs sg, OsPass ps)
{
    constexpr int TILE = OS_THREADS * IPT;
    __shared__ uint32_t cnt[OS_WARPS][OS_BINS];  // per warp: items of a digit so far, then the digit's place in the tile
    __shared__ uint32_t gstart[OS_BINS];
    __shared__ __align__(16) uint32_t sk[TILE];
    __shared__ __align__(16) uint32_t sv[TILE];
    __shared__ uint64_t ssum[OS_WARPS];
    __shared__ uint32_t hnext[OS_BINS];
    __shared__ SegTile s_st;
    __shared__ int s_bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    hnext[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_bad = 0;
    if (warp == 0) {
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(ps.ctr, 1u);
        b = __shfl_sync(0xffffffffu, b, 0);
        seg_tile(sg, b, TILE, &s_st, lane);
        if (ps.m_views && b == 0 && lane == 0) {
            unsigned long long m = 0;
            for (int v = 0; v < sg.V; ++v) m += ps.m_views[v];
            *ps.m_ws = (long long)m;
            *ps.m_out = (long long)m;
        }
    }
    const int nbins = (int)ps.mask + 1;
    const int d0 = threadIdx.x;
    uint32_t* wcnt = cnt[warp];
    for (int d = lane; d < nbins; d += 32) wcnt[d] = 0;
    __syncthreads();
    const SegTile& st = s_st;
    if (st.v < 0) return;
    const uint32_t hv = d0 < nbins ? ps.hist[(long long)st.v * ps.hist_stride + d0] : 0u;
    Word* look = (Word*)ps.look + (st.tbase + st.t) * nbins;  // this tile's words; earlier tiles' before them
    const long long rest = st.n - (long long)st.t * TILE;
    const int nv = rest < TILE ? (int)rest : TILE;
    const uint32_t shift = (uint32_t)ps.shift, mask = ps.mask;
    uint32_t key[IPT], rank[IPT];
    const uint32_t ok = src.template load<IPT>(st, nv, sk, sv, key, warp, lane);
    const bool full = __all_sync(0xffffffffu, ok == (1u << IPT) - 1u);
    if (full) os_rank<IPT, NB, true>(key, rank, ok, shift, mask, wcnt, lane);
    else os_rank<IPT, NB, false>(key, rank, ok, shift, mask, wcnt, lane);
    if (ps.hist_next) {
        const int sh = ps.shift + __popc(mask);
        const uint32_t mn = ps.mask_next;
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            if (full || ((ok >> k) & 1u)) atomicAdd(&hnext[(key[k] >> sh) & mn], 1u);
    }
    __syncthreads();
    // per digit the tile's total, published at once so that later tiles can pass it
    uint32_t total = 0;
    if (d0 < nbins) {
#pragma unroll
        for (int w = 0; w < OS_WARPS; ++w) total += cnt[w][d0];
        st_relaxed(look + d0, st.t == 0 ? LbWord<Word>::inc(total) : LbWord<Word>::agg(total));
    }
    // one scan for the tile's digit starts (low half) and the view's (high half)
    const uint64_t both = (uint64_t)total | ((uint64_t)hv << 32);
    const uint64_t inc = warp_incl_scan<uint64_t>(both, lane);
    if (lane == 31) ssum[warp] = inc;
    __syncthreads();
    uint64_t ex = inc - both;
    uint32_t have = 0;
#pragma unroll
    for (int w = 0; w < OS_WARPS; ++w) {
        const uint64_t x = ssum[w];
        ex += w < warp ? x : 0;
        have += (uint32_t)x;
    }
    if (d0 < nbins) {
        uint32_t run = (uint32_t)ex;
#pragma unroll
        for (int w = 0; w < OS_WARPS; ++w) {
            const uint32_t c = cnt[w][d0];
            cnt[w][d0] = run;
            run += c;
        }
    }
    if (ps.hist_next && threadIdx.x <= ps.mask_next && hnext[threadIdx.x])
        atomicAdd(&ps.hist_next[(long long)st.v * ps.hist_stride + threadIdx.x], hnext[threadIdx.x]);
    uint32_t val[IPT];
    src.template values<IPT>(st, nv, sv, val, warp, lane);
    __syncthreads();
    // stage the tile in digit order
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        if (full || ((ok >> k) & 1u)) {
            const uint32_t p = wcnt[(key[k] >> shift) & mask] + rank[k];
            sk[p] = key[k];
            sv[p] = val[k];
        }
    }
    // the digit's place among the view's items: its start, plus the counts of earlier tiles
    if (d0 < nbins) {
        uint32_t before = 0;
        if (st.t > 0) {
            before = (uint32_t)os_lookback(look - (long long)st.t * nbins, st.t, nbins, d0, ps.err);
            st_relaxed(look + d0, LbWord<Word>::inc((Word)before + (Word)total));
        }
        const uint32_t at = (uint32_t)(ex >> 32) + before;
        // (always inside the view's items, unless a wait gave up in this pass or before
        // or the digit counts are not those of the items; the tile is dropped then, so
        // what the pass leaves is not to be used)
        if ((unsigned long long)at + total > (unsigned long long)st.n) {
            s_bad = 1;
            atomicCAS(ps.err, 0, DG_ERR_CUDA);
        }
        gstart[d0] = (uint32_t)st.off + at - (uint32_t)ex;
    }
    __syncthreads();
    if (s_bad) return;
    uint32_t* const vout = ps.vout;
    uint32_t* const kout = ps.kout;
    if (kout) {
#pragma unroll
        for (int k = 0; k < IPT; ++k) {
            const uint32_t j = threadIdx.x + k * OS_THREADS;
            if (j >= have) break;
            const uint32_t kk = sk[j], pos = gstart[(kk >> shift) & mask] + j;
            kout[pos] = kk;
            vout[pos] = sv[j];
        }
    } else {
#pragma unroll
        for (int k = 0; k < IPT; ++k) {
            const uint32_t j = threadIdx.x + k * OS_THREADS;
            if (j >= have) break;
            vout[gstart[(sk[j] >> shift) & mask] + j] = sv[j];
        }
    }
    if (ps.ranges && total > 0) {
        // the staged tile is in full key order (earlier passes sorted the lower
        // bits), so each key is one run of it whose ends extend the key's range;
        // mostly the tile holds one value of the lower bits: one key per digit
        const uint32_t TX = (uint32_t)ps.TX[st.v], nt = (uint32_t)(ps.toff[st.v + 1] - ps.toff[st.v]);
        uint2* const rg = ps.ranges + ps.toff[st.v];
        const uint32_t g = gstart[d0], j1 = (uint32_t)ex + total;
        for (uint32_t j = (uint32_t)ex; j < j1;) {
            const uint32_t kk = sk[j];
            uint32_t e = j1;
            if (sk[j1 - 1] != kk)
                for (e = j + 1; sk[e] == kk; ++e) {}
            const uint32_t tile = key_tile(kk, ps.linear, ps.xbits, TX);
            if (tile < nt) {
                atomicMax(&rg[tile].x, ~(g + j));
                atomicMax(&rg[tile].y, g + e);
            }
            j = e;
        }
    }
}

}  // namespace
}  // namespace dg
