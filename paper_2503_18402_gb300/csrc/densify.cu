// densify.cu -- DashGaussian's scheduled densification (supplementary
// "Densification of DashGaussian"): prune first, then clone or split the
// top-(P_i - N'_GS) Gaussians by densification score among those meeting the
// backbone's condition (3DGS: mean view-space positional gradient >= thresh).
//
// Every decision that yields an integer (prune, candidate, split, selection)
// is taken on float32 values against float32 thresholds computed once on the
// host, so the result does not depend on transcendental rounding: opacity is
// tested as logit < logit(min_opacity), scales as max log-scale > log(t).
// Selection needs only the set of the best n, not their order: a radix select
// (three digit counts of 11, 11 and 10 bits, highest first, over the bit-inverted
// float score) gives the key of the last one taken, and candidates of just that
// key are taken in index order.  One look-back scan then places survivors, which
// keep their order, and appended Gaussians, which follow in index order of their
// source.  Measured on 480k Gaussians, 8% of them
// selected, both phases: 400 us in 39 launches with the candidates sorted by score
// (four radix passes of five launches) and a scan of three launches per sum ->
// 226 us in 9, of which the copies take 127 (5.6 TB/s).
#include <math.h>

#include "onesweep.cuh"

namespace dg {

enum : uint8_t { F_KEEP = 1, F_CAND = 2, F_SPLIT = 4, F_SEL = 8 };

struct HalfSizes {
    int n;
    float hw[DG_MAX_VIEWS], hh[DG_MAX_VIEWS];
};

__global__ void k_dstats(const float4* __restrict__ grad2d, const int* __restrict__ radius, int P, HalfSizes hs,
                         float* __restrict__ accum, float* __restrict__ denom, float* __restrict__ maxr)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    float acc = 0.f, den = 0.f, mr = maxr[i];
    for (int v = 0; v < hs.n; ++v) {
        const size_t r = (size_t)v * P + i;
        const int rad = radius[r];
        if (rad <= 0) continue;
        const float4 g = grad2d[3 * r];
        const float gx = g.x * hs.hw[v], gy = g.y * hs.hh[v];
        acc += sqrtf(gx * gx + gy * gy);
        den += 1.f;
        mr = fmaxf(mr, (float)rad);
    }
    if (den > 0.f) {
        accum[i] += acc;
        denom[i] += den;
        maxr[i] = mr;
    }
}

struct DThresh {
    float grad, logit_min_op, log_split, max_screen, log_max_world;
    int use_screen, use_world;
};

__global__ void k_dmark(const float* __restrict__ prm, long long stride, int P, const float* __restrict__ accum,
                        const float* __restrict__ denom, const float* __restrict__ maxr, DThresh t,
                        uint8_t* __restrict__ flags, float* __restrict__ score, long long* counts)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool keep = false, cand = false;
    if (i < P) {
        const float logit = prm[10 * stride + i];
        const float ls = fmaxf(prm[3 * stride + i], fmaxf(prm[4 * stride + i], prm[5 * stride + i]));
        bool prune = logit < t.logit_min_op;
        if (t.use_screen) prune = prune || (maxr[i] > t.max_screen);
        if (t.use_world) prune = prune || (ls > t.log_max_world);
        keep = !prune;
        const float den = denom[i];
        const float sc = den > 0.f ? accum[i] / den : 0.f;
        cand = keep && den > 0.f && sc >= t.grad;
        flags[i] = (uint8_t)((keep ? F_KEEP : 0) | (cand ? F_CAND : 0) | (ls > t.log_split ? F_SPLIT : 0));
        score[i] = sc;
    }
    // one addition per block and counter (per warp they queue on two addresses: 22 us
    // at 480k Gaussians)
    const int nk = __syncthreads_count(keep), nc = __syncthreads_count(cand);
    if (threadIdx.x == 0) {
        if (nk) atomicAdd((unsigned long long*)&counts[0], (unsigned long long)nk);
        if (nc) atomicAdd((unsigned long long*)&counts[1], (unsigned long long)nc);
    }
}

// --------------------------------------------------------------- selection
constexpr int SEL_BINS = 2048;
constexpr int SEL_THREADS = 256;

// Zeroed at the start of dg_densify_apply, with the look-back words behind it.
struct DensCtl {
    uint32_t hist[3][SEL_BINS];
    uint32_t ctr;
    int32_t err;
    long long n_keep, n_all;  // survivors; with the appended Gaussians
};

// Sort key of a score (>= 0): ascending key = descending score.
__device__ __forceinline__ uint32_t sel_key(float score) { return ~__float_as_uint(score); }
// Digit `level` of a key.
__device__ __forceinline__ uint32_t sel_digit(uint32_t key, int level)
{
    return level == 0 ? key >> 21 : level == 1 ? (key >> 10) & 2047u : key & 1023u;
}

// Whole block: the digit value in which the n-th smallest item (n >= 1) of the
// counts lies, and how many items lie below it.
__device__ inline void sel_bin(const uint32_t* __restrict__ hist, unsigned long long n, uint32_t* s_bin,
                               unsigned long long* s_below, uint32_t* s_sum)
{
    constexpr int PER = SEL_BINS / SEL_THREADS;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) {  // (stays so only when there are fewer than n items)
        *s_bin = 0;
        *s_below = 0;
    }
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        c[i] = hist[t * PER + i];
        sum += c[i];
    }
    const uint32_t inc = warp_incl_scan<uint32_t>(sum, lane);
    if (lane == 31) s_sum[warp] = inc;
    __syncthreads();
    unsigned long long below = inc - sum;
    for (int w = 0; w < warp; ++w) below += s_sum[w];
    if (below < n && n <= below + sum) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (below < n && n <= below + c[i]) {
                *s_bin = (uint32_t)(t * PER + i);
                *s_below = below;
            }
            below += c[i];
        }
    }
    __syncthreads();
}

// Whole block: the first `levels` digits of the key of the n-th best candidate
// (digits[l]) and how many candidates are better than those digits say.
__device__ inline unsigned long long sel_prefix(const DensCtl* ctl, int levels, unsigned long long n, uint32_t* digits,
                                                uint32_t* s_bin, unsigned long long* s_below, uint32_t* s_sum)
{
    unsigned long long better = 0;
    for (int l = 0; l < levels; ++l) {
        sel_bin(ctl->hist[l], n - better, s_bin, s_below, s_sum);
        digits[l] = *s_bin;
        better += *s_below;
        __syncthreads();
    }
    return better;
}

// Counts digit `level` of the candidates that share the higher digits of the n-th best.
__global__ void __launch_bounds__(SEL_THREADS)
k_sel_hist(const uint8_t* __restrict__ flags, const float* __restrict__ score, int P, unsigned long long n, int level,
           DensCtl* ctl)
{
    __shared__ uint32_t h[SEL_BINS];
    __shared__ uint32_t s_bin, s_sum[SEL_THREADS / 32];
    __shared__ unsigned long long s_below;
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS) h[i] = 0;
    uint32_t dg[2] = {0, 0};
    sel_prefix(ctl, level, n, dg, &s_bin, &s_below, s_sum);
    __syncthreads();
    for (int i = blockIdx.x * SEL_THREADS + threadIdx.x; i < P; i += gridDim.x * SEL_THREADS) {
        if (!(flags[i] & F_CAND)) continue;
        const uint32_t key = sel_key(score[i]);
        if ((level >= 1 && sel_digit(key, 0) != dg[0]) || (level >= 2 && sel_digit(key, 1) != dg[1])) continue;
        atomicAdd(&h[sel_digit(key, level)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SEL_BINS; i += SEL_THREADS)
        if (h[i]) atomicAdd(&ctl->hist[level][i], h[i]);
}

// Places: one tile of Gaussians per block, three prefix sums by look-back: the
// candidates tied with the last selected key (needed only to decide which of them
// are taken), survivors, and selected | selected splits.  mode 0: nothing is
// selected, 1: the best n_sel, 2: every candidate.
constexpr int PL_IPT = 8;
constexpr int PL_TILE = SEL_THREADS * PL_IPT;
__global__ void __launch_bounds__(SEL_THREADS)
k_places(uint8_t* __restrict__ flags, const float* __restrict__ score, int P, int mode, unsigned long long n_sel,
         DensCtl* ctl, uint64_t* __restrict__ look, int n_tiles, uint32_t* __restrict__ keep_pos,
         uint32_t* __restrict__ app_pos, uint32_t* __restrict__ sel_rank)
{
    __shared__ uint32_t s_bin, s_sum[SEL_THREADS / 32];
    __shared__ unsigned long long s_below;
    __shared__ uint32_t s_t;
    __shared__ uint32_t w_tie[SEL_THREADS / 32];
    __shared__ uint64_t w_cnt[SEL_THREADS / 32][2];
    __shared__ uint64_t s_ex[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_t = atomicAdd(&ctl->ctr, 1u);
    uint32_t dg[3] = {0, 0, 0};
    unsigned long long better = 0;
    if (mode == 1) better = sel_prefix(ctl, 3, n_sel, dg, &s_bin, &s_below, s_sum);
    __syncthreads();
    const uint32_t last = (dg[0] << 21) | (dg[1] << 10) | dg[2];
    const unsigned long long take = n_sel - better;  // of the tied ones, in index order
    const int t = (int)s_t;
    // warp-striped: item k of a lane at 32 k + lane of the warp's segment
    const uint32_t seg = (uint32_t)t * PL_TILE + warp * 32 * PL_IPT + lane, n = (uint32_t)P;
    uint8_t f[PL_IPT];
    uint32_t tied = 0, ties = 0, tie_at[PL_IPT];
#pragma unroll
    for (int k = 0; k < PL_IPT; ++k) {
        const uint32_t i = seg + 32 * k;
        f[k] = i < n ? (uint8_t)(flags[i] & ~F_SEL) : (uint8_t)0;
        if (mode != 0 && (f[k] & F_CAND)) {
            const uint32_t key = mode == 1 ? sel_key(score[i]) : 0u;
            if (mode == 2 || key < last) f[k] |= F_SEL;
            else if (key == last) tied |= 1u << k;
        }
        const uint32_t m = __ballot_sync(0xffffffffu, (tied >> k) & 1u);
        tie_at[k] = ties + __popc(m & ((1u << lane) - 1u));
        ties += __popc(m);
    }
    if (mode == 1) {  // rank of each tied candidate among all of them
        if (lane == 0) w_tie[warp] = ties;
        __syncthreads();
        uint32_t pre = 0, tot = 0;
        for (int w = 0; w < SEL_THREADS / 32; ++w) {
            pre += w < warp ? w_tie[w] : 0u;
            tot += w_tie[w];
        }
        if (warp == 0) {
            uint64_t e = 0;
            if (lane == 0) st_relaxed(look + t, (t == 0 ? kLbInc : kLbAgg) | tot);
            if (t > 0) {
                if (!os_lookback_warp(look, t, &e, lane) && lane == 0) atomicExch(&ctl->err, DG_ERR_TIMEOUT);
                if (lane == 0) st_relaxed(look + t, kLbInc | (e + tot));
            }
            if (lane == 0) s_ex[0] = e;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < PL_IPT; ++k)
            if (((tied >> k) & 1u) && s_ex[0] + pre + tie_at[k] < take) f[k] |= F_SEL;
    }
    // survivors, and selected (low 31 bits) | selected splits (high 31 bits)
    uint32_t kc[PL_IPT], keeps = 0, sels = 0, spl = 0, sc[PL_IPT], pc[PL_IPT];
#pragma unroll
    for (int k = 0; k < PL_IPT; ++k) {
        const bool sel = f[k] & F_SEL, split = sel && (f[k] & F_SPLIT), keep = (f[k] & F_KEEP) && !split;
        const uint32_t below = (1u << lane) - 1u;
        const uint32_t mk = __ballot_sync(0xffffffffu, keep), ms = __ballot_sync(0xffffffffu, sel),
                       mp = __ballot_sync(0xffffffffu, split);
        kc[k] = keeps + __popc(mk & below);
        sc[k] = sels + __popc(ms & below);
        pc[k] = spl + __popc(mp & below);
        keeps += __popc(mk);
        sels += __popc(ms);
        spl += __popc(mp);
    }
    if (lane == 0) {
        w_cnt[warp][0] = keeps;
        w_cnt[warp][1] = (uint64_t)sels | ((uint64_t)spl << 31);
    }
    __syncthreads();
    uint64_t pre[2] = {0, 0}, tot[2] = {0, 0};
    for (int w = 0; w < SEL_THREADS / 32; ++w)
        for (int q = 0; q < 2; ++q) {
            pre[q] += w < warp ? w_cnt[w][q] : 0;
            tot[q] += w_cnt[w][q];
        }
    if (warp < 2) {  // one warp per sum
        uint64_t* lk = look + (size_t)(1 + warp) * n_tiles;
        const uint64_t mine = warp ? tot[1] : tot[0];
        uint64_t e = 0;
        if (lane == 0) st_relaxed(lk + t, (t == 0 ? kLbInc : kLbAgg) | mine);
        if (t > 0) {
            if (!os_lookback_warp(lk, t, &e, lane) && lane == 0) atomicExch(&ctl->err, DG_ERR_TIMEOUT);
            if (lane == 0) st_relaxed(lk + t, kLbInc | (e + mine));
        }
        if (lane == 0) s_ex[1 + warp] = e;
    }
    __syncthreads();
    constexpr uint64_t k31 = (1ull << 31) - 1;
    const uint32_t k0 = (uint32_t)(s_ex[1] + pre[0]);
    const uint64_t sp = s_ex[2] + pre[1];
    const uint32_t s0 = (uint32_t)(sp & k31), p0 = (uint32_t)(sp >> 31);
#pragma unroll
    for (int k = 0; k < PL_IPT; ++k) {
        const uint32_t i = seg + 32 * k;
        if (i >= n) continue;
        keep_pos[i] = k0 + kc[k];
        if (f[k] & F_CAND) flags[i] = f[k];
        if (f[k] & F_SEL) {  // one place per selected Gaussian, one more per split
            sel_rank[i] = s0 + sc[k];
            app_pos[i] = s0 + sc[k] + p0 + pc[k];
        }
    }
    if (t == n_tiles - 1 && threadIdx.x == 0) {
        const uint64_t all = s_ex[2] + tot[1];
        const long long nk = (long long)(s_ex[1] + tot[0]);
        ctl->n_keep = nk;
        ctl->n_all = nk + (long long)(all & k31) + (long long)(all >> 31);
    }
}

__device__ inline void quat_rot(float q0, float q1, float q2, float q3, float R[9])
{
    const float inv = 1.f / sqrtf(q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3);
    const float w = q0 * inv, x = q1 * inv, y = q2 * inv, z = q3 * inv;
    R[0] = 1.f - 2.f * (y * y + z * z); R[1] = 2.f * (x * y - w * z);       R[2] = 2.f * (x * z + w * y);
    R[3] = 2.f * (x * y + w * z);       R[4] = 1.f - 2.f * (x * x + z * z); R[5] = 2.f * (y * z - w * x);
    R[6] = 2.f * (x * z - w * y);       R[7] = 2.f * (y * z + w * x);       R[8] = 1.f - 2.f * (x * x + y * y);
}

// Writes survivors and appended Gaussians with their moments, DW_ROWS parameter
// rows per block (blockIdx.y): a thread loads its Gaussian's rows of all three
// arrays before it stores any, so 24 loads are in flight (row after row, one
// thread per Gaussian, took 149 us at 480k Gaussians against 127).
constexpr int DW_ROWS = 8;
__global__ void __launch_bounds__(256)
k_densify_write(const float* __restrict__ prm, const float* __restrict__ m, const float* __restrict__ v,
                long long stride, int P, const uint8_t* __restrict__ flags, const uint32_t* __restrict__ keep_pos,
                const uint32_t* __restrict__ app_pos, const uint32_t* __restrict__ sel_rank, const DensCtl* ctl,
                const float* __restrict__ noise, float log_div, float* __restrict__ dp, float* __restrict__ dm,
                float* __restrict__ dv, long long dstride, long long* __restrict__ P_out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // (here, not in the kernel of the places: only behind it is its error word final)
    if (i == 0 && blockIdx.y == 0) *P_out = ctl->err != 0 ? (long long)ctl->err : ctl->n_all;
    if (i >= P || ctl->err != 0) return;  // (a wait gave up: the places are not known)
    const uint8_t f = flags[i];
    const bool sel = f & F_SEL, split = sel && (f & F_SPLIT), keep = (f & F_KEEP) && !split;
    if (!keep && !sel) return;
    const int r0 = blockIdx.y * DW_ROWS;
    float p[DW_ROWS], mm[DW_ROWS], vv[DW_ROWS];
#pragma unroll
    for (int k = 0; k < DW_ROWS; ++k) {
        const long long at = (long long)(r0 + k) * stride + i;
        const bool in = r0 + k < DG_NPARAM;
        p[k] = in ? prm[at] : 0.f;
        mm[k] = in && keep ? m[at] : 0.f;
        vv[k] = in && keep ? v[at] : 0.f;
    }
    auto put = [&](long long o, bool moments) {
#pragma unroll
        for (int k = 0; k < DW_ROWS; ++k) {
            if (r0 + k >= DG_NPARAM) break;
            const long long at = (long long)(r0 + k) * dstride + o;
            dp[at] = p[k];
            dm[at] = moments ? mm[k] : 0.f;
            dv[at] = moments ? vv[k] : 0.f;
        }
    };
    if (keep) put(keep_pos[i], true);
    if (!sel) return;
    const long long base = ctl->n_keep + app_pos[i];
    if (!split) {
        put(base, false);
        return;
    }
    if (r0 > 0) {
        put(base, false);
        put(base + 1, false);
        return;
    }
    // rows 0..7 of the two samples: means, log scales, two of the quaternion
    float R[9];
    quat_rot(prm[6 * stride + i], prm[7 * stride + i], prm[8 * stride + i], prm[9 * stride + i], R);
    float s[3], mu[3], ls[3];
    for (int c = 0; c < 3; ++c) {
        s[c] = expf(p[3 + c]);
        mu[c] = p[c];
        ls[c] = p[3 + c] - log_div;
    }
    const float* eps = noise + 6 * (size_t)sel_rank[i];
    for (int k = 0; k < 2; ++k) {
        const float e0 = s[0] * eps[3 * k], e1 = s[1] * eps[3 * k + 1], e2 = s[2] * eps[3 * k + 2];
        for (int c = 0; c < 3; ++c) {
            p[c] = mu[c] + R[3 * c] * e0 + R[3 * c + 1] * e1 + R[3 * c + 2] * e2;
            p[3 + c] = ls[c];
        }
        put(base + k, false);
    }
}
static_assert(DW_ROWS >= 6, "the first row group holds the rows a split changes");

struct DensWs {
    uint8_t* flags;
    float* score;
    uint32_t *keep_pos, *app_pos, *sel_rank;
    DensCtl* ctl;
    uint64_t* look;     // [3][tiles]
    size_t zero;        // bytes dg_densify_apply clears from ctl on
    size_t bytes;
};

static size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

static DensWs dens_layout(char* b, long long P)
{
    DensWs w;
    size_t o = 0;
    auto take = [&](size_t n) { char* p = b + o; o += al(n); return p; };
    w.flags = (uint8_t*)take(P);
    w.score = (float*)take(4 * P);
    w.keep_pos = (uint32_t*)take(4 * P);
    w.app_pos = (uint32_t*)take(4 * P);
    w.sel_rank = (uint32_t*)take(4 * P);
    const size_t c = o;
    w.ctl = (DensCtl*)take(sizeof(DensCtl));
    w.look = (uint64_t*)take(8 * 3 * ((P + PL_TILE - 1) / PL_TILE));
    w.zero = o - c;
    w.bytes = o;
    return w;
}

static bool thresholds(const dg_densify_opts* o, DThresh* t)
{
    if (!(o->grad_thresh >= 0.f) || !(o->min_opacity > 0.f && o->min_opacity < 1.f) ||
        !(o->percent_dense > 0.f) || !(o->extent > 0.f))
        return false;
    t->grad = o->grad_thresh;
    t->logit_min_op = (float)log((double)o->min_opacity / (1.0 - (double)o->min_opacity));
    t->log_split = (float)log((double)o->percent_dense * (double)o->extent);
    t->use_screen = o->max_screen_radius > 0.f;
    t->max_screen = o->max_screen_radius;
    t->use_world = o->max_world_scale > 0.f;
    t->log_max_world = t->use_world ? (float)log((double)o->max_world_scale) : 0.f;
    return true;
}

}  // namespace dg

bool dg_check_cameras(const dg_camera* cams, int n_views);

extern "C" dg_status dg_densify_stats(const float* grad2d, const int32_t* radius, int64_t P, const dg_camera* cams,
                                      int32_t n_views, float* grad_accum, float* denom, float* max_radius,
                                      dg_stream stream)
{
    if (!dg_check_cameras(cams, n_views)) return DG_ERR_ARG;
    if (P < 0 || P > INT32_MAX) { dg_set_error("bad sizes"); return DG_ERR_ARG; }
    if (P == 0) return DG_OK;
    if (!grad2d || !radius || !grad_accum || !denom || !max_radius) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    dg::HalfSizes hs;
    hs.n = n_views;
    for (int v = 0; v < n_views; ++v) {
        hs.hw[v] = 0.5f * cams[v].width;
        hs.hh[v] = 0.5f * cams[v].height;
    }
    dg::k_dstats<<<(int)((P + 255) / 256), 256, 0, (cudaStream_t)stream>>>(
        (const float4*)grad2d, radius, (int)P, hs, grad_accum, denom, max_radius);
    dg_note_launch();
    return dg_check_launch("densify_stats");
}

extern "C" size_t dg_densify_workspace_size(int64_t P)
{
    if (P < 0) return 0;
    return dg::dens_layout(nullptr, P).bytes;
}

extern "C" dg_status dg_densify_mark(const float* params, int64_t stride, int64_t P, const float* grad_accum,
                                     const float* denom, const float* max_radius, const dg_densify_opts* opts,
                                     void* ws, size_t ws_bytes, int64_t* counts, dg_stream stream)
{
    dg::DThresh t;
    if (!opts || !dg::thresholds(opts, &t)) { dg_set_error("bad densify options"); return DG_ERR_ARG; }
    if (P < 0 || P > INT32_MAX || stride < P) { dg_set_error("bad P/stride"); return DG_ERR_ARG; }
    if (!ws || !counts || (P > 0 && (!params || !grad_accum || !denom || !max_radius))) {
        dg_set_error("null buffer");
        return DG_ERR_ARG;
    }
    const dg::DensWs w = dg::dens_layout((char*)ws, P);
    if (ws_bytes < w.bytes) { dg_set_error("densify workspace too small"); return DG_ERR_CAPACITY; }
    cudaStream_t s = (cudaStream_t)stream;
    cudaMemsetAsync(counts, 0, 2 * sizeof(int64_t), s);
    if (P == 0) return dg_check_launch("densify_mark");
    dg::k_dmark<<<(int)((P + 255) / 256), 256, 0, s>>>(params, (long long)stride, (int)P, grad_accum, denom,
                                                       max_radius, t, w.flags, w.score, (long long*)counts);
    dg_note_launch();
    return dg_check_launch("densify_mark");
}

extern "C" dg_status dg_densify_apply(const float* params, const float* m, const float* v, int64_t stride, int64_t P,
                                      int64_t n_cand, int64_t budget, const float* noise, void* ws, size_t ws_bytes,
                                      float* dst_params, float* dst_m, float* dst_v, int64_t dst_stride,
                                      int64_t* P_out, dg_stream stream)
{
    if (P < 0 || P > INT32_MAX || stride < P || n_cand < 0 || n_cand > P || budget < 0) {
        dg_set_error("bad sizes");
        return DG_ERR_ARG;
    }
    const long long n_sel = n_cand < budget ? n_cand : budget;
    if (!ws || !P_out || !dst_params || !dst_m || !dst_v || (P > 0 && (!params || !m || !v)) || (n_sel > 0 && !noise)) {
        dg_set_error("null buffer");
        return DG_ERR_ARG;
    }
    const dg::DensWs w = dg::dens_layout((char*)ws, P);
    if (ws_bytes < w.bytes) { dg_set_error("densify workspace too small"); return DG_ERR_CAPACITY; }
    if (dst_stride < P + n_sel) {
        dg_set_error("dst_stride %lld below the largest possible count %lld", (long long)dst_stride, (long long)(P + n_sel));
        return DG_ERR_CAPACITY;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (P == 0) {
        cudaMemsetAsync(P_out, 0, sizeof(int64_t), s);
        return dg_check_launch("densify_apply");
    }
    cudaMemsetAsync(w.ctl, 0, w.zero, s);
    const int mode = n_sel == 0 ? 0 : n_cand > budget ? 1 : 2;
    if (mode == 1) {
        const long long per = dg::SEL_THREADS * 8;
        const int hb = (int)((P + per - 1) / per < 152 * 4 ? (P + per - 1) / per : 152 * 4);
        for (int level = 0; level < 3; ++level)
            dg::k_sel_hist<<<hb, dg::SEL_THREADS, 0, s>>>(w.flags, w.score, (int)P, (unsigned long long)n_sel, level,
                                                         w.ctl);
        dg_note_launch(3);
    }
    const int nt = (int)((P + dg::PL_TILE - 1) / dg::PL_TILE);
    dg::k_places<<<nt, dg::SEL_THREADS, 0, s>>>(w.flags, w.score, (int)P, mode, (unsigned long long)n_sel, w.ctl, w.look,
                                              nt, w.keep_pos, w.app_pos, w.sel_rank);
    const dim3 grid((unsigned)((P + 255) / 256), (DG_NPARAM + dg::DW_ROWS - 1) / dg::DW_ROWS);
    dg::k_densify_write<<<grid, 256, 0, s>>>(params, m, v, (long long)stride, (int)P, w.flags, w.keep_pos, w.app_pos,
                                             w.sel_rank, w.ctl, noise, (float)log(1.6), dst_params, dst_m, dst_v,
                                             (long long)dst_stride, (long long*)P_out);
    dg_note_launch(2);
    return dg_check_launch("densify_apply");
}
