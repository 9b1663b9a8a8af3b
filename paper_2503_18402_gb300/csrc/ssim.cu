// ssim.cu -- the backbone's photometric loss (1 - lambda) L1 + lambda (1 - SSIM)
// and its gradient, for one or several views per call.
//
// SSIM (Wang et al. 2004): per channel, window sums under an 11 x 11 Gaussian
// (sigma 1.5, normalised, zero padding outside the image) give mu_x, mu_y and
// a = E[x^2], b = E[y^2], c = E[xy]; per pixel
//   S = (2 mu_x mu_y + C1)(2 (c - mu_x mu_y) + C2)
//       / ((mu_x^2 + mu_y^2 + C1)((a - mu_x^2) + (b - mu_y^2) + C2)).
// Its gradient is the adjoint of the window sums applied to three per-pixel
// partial derivatives of S (with respect to mu_x, a and c):
//   dS/dx(q) = F[dS/dmu_x](q) + 2 x(q) F[dS/da](q) + y(q) F[dS/dc](q),
// F the same symmetric, zero-padded window.
//
// Two passes, over tiles (k_ssim_fwd_t, k_ssim_bwd_t) for small or narrow images, else
// (k_ssim_fwd, k_ssim_bwd) over strips of SS_W output columns and segments of rows,
// a thread per two adjacent columns.  Going down the rows,
// two at a time are staged in shared memory; a thread forms the horizontal window
// sums of its two columns from twelve staged inputs and feeds them to the vertical
// windows, which it keeps as ten partial sums per column in registers (a new row
// adds its eleven taps), so nothing but the inputs passes through shared memory
// and the only halo that is computed is the ten rows at a segment's start.  The
// statistics run as packed float32 pairs: (mu_x, mu_y) and (E[x^2] + E[y^2], E[xy])
// (S uses E[x^2] and E[y^2] only through their sum) in the forward, (dS/dmu_x,
// dS/da) and dS/dc alone in the backward; every sum's taps are added in ascending
// order, the horizontal window first.  The forward writes the three partial-
// derivative maps (in padded strips) and per-block sums of 1 - S and |x - y|; the
// backward filters the maps and writes dL/dx including the L1 term; its first
// block sums the forward's block sums per view in a fixed order (FP64).
// HBM per pixel and channel: forward reads x, y (8 B) and writes 3 maps (12 B);
// backward reads the maps and x, y (20 B) and writes dL/dx (4 B).  Bound by issue
// and the FP32 pipe (packed operations take it twice).  Measured on 16 views of
// 1237x822: 0.97 ms with 32x32 tiles (42x42 staged, both windows through shared
// memory, a third of the threads idle in the horizontal pass's second round) and
// a separate summing launch -> 0.615 ms, the gradient the same bits (six blocks per
// SM, 160 registers; five 0.644, seven 0.618, eight 0.655); 0.620 with
// compensated sums.  The vertical window first, four outputs per thread in the
// horizontal one, took 0.535 ms, but rounds the gradient differently (3e-6 relative,
// no nearer to the exact one).
#include <math.h>

#include "common.cuh"

namespace dg {
namespace {

constexpr int SS_R = 5;               // window radius
constexpr int SS_THREADS = 64;
constexpr int SS_W = 2 * SS_THREADS;  // output columns of a strip, and floats per map row of a strip
constexpr int SS_E = SS_W + 2 * SS_R; // staged columns (138)
constexpr int SS_ROWS = 2;            // rows staged together
constexpr int SS_LD = (SS_E + SS_THREADS - 1) / SS_THREADS;  // staged columns per thread (3, the last for few)
constexpr int SS_FWD_BLOCKS = 6, SS_BWD_BLOCKS = 6;  // blocks per SM
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

struct Win { float w[SS_R + 1]; };    // symmetric: tap k has weight w[min(k, 10 - k)]

struct SViews {
    int n;
    int rows;                      // rows of a segment (even)
    int W[DG_MAX_VIEWS], H[DG_MAX_VIEWS], TX[DG_MAX_VIEWS], TY[DG_MAX_VIEWS];
    int boff[DG_MAX_VIEWS + 1];    // first block of each view (3 channels x strips x segments)
    long long poff[DG_MAX_VIEWS];  // first pixel of each view
    long long moff[DG_MAX_VIEWS];  // first map value of each view (maps [3 channels][strip][H][SS_W])
};

struct Blk { int v, ch, tx, y0, W, H; long long plane, map; };

__device__ inline Blk decode(const SViews& sv, int i)
{
    Blk b;
    int v = 0;
    while (v + 1 < sv.n && i >= sv.boff[v + 1]) ++v;
    const int r = i - sv.boff[v];
    const int per = sv.TX[v] * sv.TY[v];
    b.v = v;
    b.ch = r / per;
    const int t = r % per;
    b.tx = t % sv.TX[v];
    b.y0 = (t / sv.TX[v]) * sv.rows;
    b.W = sv.W[v];
    b.H = sv.H[v];
    b.plane = 3 * sv.poff[v] + (long long)b.ch * b.W * b.H;  // first element of this channel plane
    b.map = sv.moff[v] + (long long)b.ch * sv.TX[v] * b.H * SS_W;  // first map value of this channel
    return b;
}

// Vertical window of one column, packed pairs: acc[i] holds the taps so far of
// the output that is complete i + 1 rows from now.  Feeding row value v
// returns the output completed by it; the shift of the partial sums is part of
// the multiply-adds.
struct Col2 {
    f32x2 acc[2 * SS_R];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < 2 * SS_R; ++i) acc[i] = f2_pack(0.f, 0.f);
    }
    __device__ __forceinline__ f32x2 feed(f32x2 v, const f32x2 (&w)[SS_R + 1])
    {
        const f32x2 out = f2_fma(w[0], v, acc[0]);
#pragma unroll
        for (int i = 0; i < 2 * SS_R - 1; ++i) {
            const int k = 2 * SS_R - 1 - i;  // tap of the output i + 1 rows ahead
            acc[i] = f2_fma(w[k <= SS_R ? k : 2 * SS_R - k], v, acc[i + 1]);
        }
        acc[2 * SS_R - 1] = f2_mul(w[0], v);
        return out;
    }
};
struct Col1 {
    float acc[2 * SS_R];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < 2 * SS_R; ++i) acc[i] = 0.f;
    }
    __device__ __forceinline__ float feed(float v, const float (&w)[SS_R + 1])
    {
        const float out = fmaf(w[0], v, acc[0]);
#pragma unroll
        for (int i = 0; i < 2 * SS_R - 1; ++i) {
            const int k = 2 * SS_R - 1 - i;
            acc[i] = fmaf(w[k <= SS_R ? k : 2 * SS_R - k], v, acc[i + 1]);
        }
        acc[2 * SS_R - 1] = w[0] * v;
        return out;
    }
};

// Two sums with a running compensation (Kahan), packed: a thread adds up to 128
// values, whose plain float32 sum carries their roundings one on another (1.9e-6 of a
// constant |x - y|, against at most 11 roundings here).  1 - S is summed, not S: close
// images lose nothing to sums near the pixel count (relative error of the loss at
// |x - y| about 1e-3: 7.4e-7 -> 5.5e-7).  615 -> 620 us on 16 views of 1237x822.
struct KSum2 {
    f32x2 s, c;  // c: what the sum lacks
    __device__ __forceinline__ void clear() { s = c = f2_pack(0.f, 0.f); }
    __device__ __forceinline__ void add(float v0, float v1)
    {
        const f32x2 y = f2_add(f2_pack(v0, v1), c), t = f2_add(s, y);
        c = f2_add(f2_fma(t, f2_pack(-1.f, -1.f), s), y);
        s = t;
    }
};

// Horizontal window of two adjacent outputs from their twelve inputs.
__device__ __forceinline__ void hsum2(const f32x2 (&v)[2 * SS_R + 2], const f32x2 (&w)[SS_R + 1], f32x2 (&out)[2])
{
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        f32x2 a = f2_mul(w[0], v[o]);
#pragma unroll
        for (int k = 1; k <= 2 * SS_R; ++k) a = f2_fma(w[k <= SS_R ? k : 2 * SS_R - k], v[o + k], a);
        out[o] = a;
    }
}
__device__ __forceinline__ void hsum1(const float (&v)[2 * SS_R + 2], const float (&w)[SS_R + 1], float (&out)[2])
{
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        float a = w[0] * v[o];
#pragma unroll
        for (int k = 1; k <= 2 * SS_R; ++k) a = fmaf(w[k <= SS_R ? k : 2 * SS_R - k], v[o + k], a);
        out[o] = a;
    }
}

__global__ void __launch_bounds__(SS_THREADS, SS_FWD_BLOCKS)
k_ssim_fwd(const float* __restrict__ img, const float* __restrict__ tgt, SViews sv, Win win,
           float* __restrict__ dm, float* __restrict__ da, float* __restrict__ dc, float2* __restrict__ part)
{
    __shared__ __align__(16) float2 s_in[2][SS_ROWS][SS_E + 2];  // (x, y)
    __shared__ float red[2][SS_THREADS / 32];
    const Blk b = decode(sv, blockIdx.x);
    const int tid = threadIdx.x;
    const int x0 = b.tx * SS_W;
    const int nrow = min(sv.rows, b.H - b.y0);       // output rows of this segment
    // staged columns of this thread (tid, tid + 64, ...); row offsets from the
    // segment's first row fit 32 bits
    const float* px = img + b.plane + (long long)b.y0 * b.W;
    const float* py = tgt + b.plane + (long long)b.y0 * b.W;
    int col[SS_LD];
    bool cin[SS_LD];
#pragma unroll
    for (int q = 0; q < SS_LD; ++q) {
        const int s = tid + q * SS_THREADS;
        col[q] = x0 - SS_R + s;
        cin[q] = s < SS_E && col[q] >= 0 && col[q] < b.W;
    }
    float nx[SS_ROWS][SS_LD], ny[SS_ROWS][SS_LD];
    auto fetch = [&](int r) {  // rows r, r + 1 of the segment (from -SS_R on)
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i) {
            const bool yin = (unsigned)(b.y0 + r + i) < (unsigned)b.H;
            const int at = (r + i) * b.W;
#pragma unroll
            for (int q = 0; q < SS_LD; ++q) {
                nx[i][q] = yin && cin[q] ? px[at + col[q]] : 0.f;
                ny[i][q] = yin && cin[q] ? py[at + col[q]] : 0.f;
            }
        }
    };
    f32x2 w[SS_R + 1];
#pragma unroll
    for (int k = 0; k <= SS_R; ++k) w[k] = f2_pack(win.w[k], win.w[k]);
    Col2 cm[2], cq[2];
#pragma unroll
    for (int o = 0; o < 2; ++o) { cm[o].clear(); cq[o].clear(); }
    KSum2 sum;                                        // |x - y| and 1 - S over the thread's outputs
    sum.clear();
    float l1r = 0.f, dr = 0.f;                        // theirs since the last addition to it
    const int xo = x0 + 2 * tid;                      // this thread's two output columns
    const bool in0 = xo < b.W, in1 = xo + 1 < b.W;
    const float nin = (in0 ? 1.f : 0.f) + (in1 ? 1.f : 0.f);
    const long long mcol = b.map + ((long long)b.tx * b.H + b.y0) * SS_W + 2 * tid;
    fetch(-SS_R);
    int buf = 0;
    for (int r = -SS_R; r < nrow + SS_R; r += SS_ROWS, buf ^= 1) {
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i)
#pragma unroll
            for (int q = 0; q < SS_LD; ++q)
                if (tid + q * SS_THREADS < SS_E) s_in[buf][i][tid + q * SS_THREADS] = make_float2(nx[i][q], ny[i][q]);
        if (r + SS_ROWS < nrow + SS_R) fetch(r + SS_ROWS);
        __syncthreads();  // (the buffer written next round is read by no one after this)
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i) {
            f32x2 v[2 * SS_R + 2], h[2], mu[2], qq[2];
            const float4* c = (const float4*)s_in[buf][i] + tid;
#pragma unroll
            for (int j = 0; j < SS_R + 1; ++j) {
                const float4 t = c[j];
                v[2 * j] = f2_pack(t.x, t.y);
                v[2 * j + 1] = f2_pack(t.z, t.w);
            }
            if ((unsigned)(r + i) < (unsigned)nrow) {
                float x, y;
                f2_unpack(v[SS_R], x, y);
                if (in0) l1r += fabsf(x - y);
                f2_unpack(v[SS_R + 1], x, y);
                if (in1) l1r += fabsf(x - y);
            }
            hsum2(v, w, h);
#pragma unroll
            for (int o = 0; o < 2; ++o) mu[o] = cm[o].feed(h[o], w);
#pragma unroll
            for (int j = 0; j < 2 * SS_R + 2; ++j) {
                float x, y;
                f2_unpack(v[j], x, y);
                v[j] = f2_pack(fmaf(x, x, y * y), x * y);
            }
            hsum2(v, w, h);
#pragma unroll
            for (int o = 0; o < 2; ++o) qq[o] = cq[o].feed(h[o], w);
            const int yo = r + i - SS_R;  // the output row this row completes
            if (yo < 0 || yo >= nrow) continue;
            float2 o0, o1, o2;
            float *p0 = &o0.x, *p1 = &o1.x, *p2 = &o2.x;
            dr += nin;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                float mx, my, ab, cc;
                f2_unpack(mu[o], mx, my);
                f2_unpack(qq[o], ab, cc);
                const float A1 = 2.f * mx * my + kC1;
                const float A2 = 2.f * (cc - mx * my) + kC2;
                const float B1 = mx * mx + my * my + kC1;
                const float B2 = (ab - mx * mx - my * my) + kC2;
                const float inv = 1.f / (B1 * B2);
                const float S = A1 * A2 * inv;
                p0[o] = 2.f * my * (A2 - A1) * inv - 2.f * mx * S * (B2 - B1) * inv;
                p1[o] = -S * B1 * inv;
                p2[o] = 2.f * A1 * inv;
                if (o ? in1 : in0) dr -= S;
            }
            const long long m = mcol + yo * SS_W;
            *(float2*)(dm + m) = o0;
            *(float2*)(da + m) = o1;
            *(float2*)(dc + m) = o2;
        }
        sum.add(l1r, dr);
        l1r = dr = 0.f;
    }
    float l1sum, ssum;
    f2_unpack(sum.s, l1sum, ssum);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
        l1sum += __shfl_xor_sync(0xffffffffu, l1sum, o);
    }
    if ((tid & 31) == 0) { red[0][tid >> 5] = ssum; red[1][tid >> 5] = l1sum; }
    __syncthreads();
    if (tid == 0) {
        float s = 0.f, l = 0.f;
        for (int k = 0; k < SS_THREADS / 32; ++k) { s += red[0][k]; l += red[1][k]; }
        part[blockIdx.x] = make_float2(s, l);
    }
}

// loss[v] = (1 - lam) l1_v + lam (1 - ssim_v); loss[n] = mean over views.  One
// block: NW warps shared evenly by the views, or, with more views than warps, each
// warp taking every NW-th view; a warp sums a fixed stride of its view's block sums in
// FP64, and the warps' and the views' sums are added in a fixed order, so the
// result does not depend on timing.  It is the backward's first block: as a launch
// of its own behind the backward it took 8 us for one view and 12 us for 16.
template <int NW>
__device__ void ssim_final(const float2* __restrict__ part, const SViews& sv, float lam, float* __restrict__ loss)
{
    __shared__ double sm[2][DG_MAX_VIEWS][NW];
    __shared__ double lv_s[DG_MAX_VIEWS];
    const int nv = sv.n;
    const int wpv = nv >= NW ? 1 : NW / nv;  // warps per view
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int v = w / wpv; v < nv; v += NW / wpv) {
        double s = 0.0, l = 0.0;
        // eight loads in flight per round, added in index order
        const int step = 32 * wpv, end = sv.boff[v + 1];
        for (int i0 = sv.boff[v] + 32 * (w % wpv) + lane; i0 < end; i0 += 8 * step) {
            float2 p[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) p[u] = i0 + u * step < end ? part[i0 + u * step] : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                s += (double)p[u].x;
                l += (double)p[u].y;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            l += __shfl_xor_sync(0xffffffffu, l, o);
        }
        if (lane == 0) { sm[0][v][w % wpv] = s; sm[1][v][w % wpv] = l; }
    }
    __syncthreads();
    if ((int)threadIdx.x < nv) {
        const int v = threadIdx.x;
        double S = 0.0, Lv = 0.0;  // of 1 - S and |x - y|
        for (int q = 0; q < wpv; ++q) { S += sm[0][v][q]; Lv += sm[1][v][q]; }
        const double n = 3.0 * (double)sv.W[v] * (double)sv.H[v];
        const double lv = (1.0 - (double)lam) * (Lv / n) + (double)lam * (S / n);
        loss[v] = (float)lv;
        lv_s[v] = lv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double mean = 0.0;
        for (int q = 0; q < nv; ++q) mean += lv_s[q];
        loss[nv] = (float)(mean / nv);
    }
}

__global__ void __launch_bounds__(SS_THREADS, SS_BWD_BLOCKS)
k_ssim_bwd(const float* __restrict__ img, const float* __restrict__ tgt, SViews sv, Win win,
           const float* __restrict__ dm, const float* __restrict__ da, const float* __restrict__ dc,
           float lam, float* __restrict__ grad, const float2* __restrict__ part, float* __restrict__ loss)
{
    __shared__ __align__(16) float2 s_in[2][SS_ROWS][SS_E + 2];  // (dS/dmu_x, dS/da)
    __shared__ __align__(16) float s_c[2][SS_ROWS][SS_E + 2];    // dS/dc
    if (blockIdx.x == 0) {  // the losses, from the forward's block sums
        ssim_final<SS_THREADS / 32>(part, sv, lam, loss);
        return;
    }
    const Blk b = decode(sv, blockIdx.x - 1);
    const int tid = threadIdx.x;
    const int x0 = b.tx * SS_W;
    const int nrow = min(sv.rows, b.H - b.y0);
    // map offsets of this thread's staged columns (each in the strip that owns it)
    long long mc[SS_LD];
    bool cin[SS_LD];
#pragma unroll
    for (int q = 0; q < SS_LD; ++q) {
        const int s = tid + q * SS_THREADS, x = x0 - SS_R + s;
        cin[q] = s < SS_E && x >= 0 && x < b.W;
        const int st = cin[q] ? x / SS_W : 0;
        mc[q] = b.map + ((long long)st * b.H + b.y0) * SS_W + (cin[q] ? x - st * SS_W : 0);
    }
    const int xo = x0 + 2 * tid;
    const bool in0 = xo < b.W, in1 = xo + 1 < b.W;
    const long long ocol = b.plane + (long long)b.y0 * b.W + xo;
    const float *px = img + ocol, *py = tgt + ocol;
    float* const pg = grad + ocol;
    float n0[SS_ROWS][SS_LD], n1[SS_ROWS][SS_LD], n2[SS_ROWS][SS_LD];
    auto fetch = [&](int r) {
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i) {
            const bool yin = (unsigned)(b.y0 + r + i) < (unsigned)b.H;
            const int at = (r + i) * SS_W;
#pragma unroll
            for (int q = 0; q < SS_LD; ++q) {
                const bool in = yin && cin[q];
                n0[i][q] = in ? dm[mc[q] + at] : 0.f;
                n1[i][q] = in ? da[mc[q] + at] : 0.f;
                n2[i][q] = in ? dc[mc[q] + at] : 0.f;
            }
        }
    };
    f32x2 w[SS_R + 1];
    float w1[SS_R + 1];
#pragma unroll
    for (int k = 0; k <= SS_R; ++k) {
        w1[k] = win.w[k];
        w[k] = f2_pack(win.w[k], win.w[k]);
    }
    Col2 cm[2];
    Col1 cc[2];
#pragma unroll
    for (int o = 0; o < 2; ++o) { cm[o].clear(); cc[o].clear(); }
    // d/dx of the mean over views of (1 - lam) mean|x - y| + lam (1 - mean S)
    const float scale = 1.f / ((float)sv.n * 3.f * (float)b.W * (float)b.H);
    fetch(-SS_R);
    int buf = 0;
    for (int r = -SS_R; r < nrow + SS_R; r += SS_ROWS, buf ^= 1) {
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i)
#pragma unroll
            for (int q = 0; q < SS_LD; ++q)
                if (tid + q * SS_THREADS < SS_E) {
                    s_in[buf][i][tid + q * SS_THREADS] = make_float2(n0[i][q], n1[i][q]);
                    s_c[buf][i][tid + q * SS_THREADS] = n2[i][q];
                }
        if (r + SS_ROWS < nrow + SS_R) fetch(r + SS_ROWS);
        // x and y at the outputs these rows complete
        float xv[SS_ROWS][2], yv[SS_ROWS][2];
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i) {
            const int yo = r + i - SS_R;
            const bool yin = yo >= 0 && yo < nrow;
            const int at = yo * b.W;
            xv[i][0] = yin && in0 ? px[at] : 0.f; xv[i][1] = yin && in1 ? px[at + 1] : 0.f;
            yv[i][0] = yin && in0 ? py[at] : 0.f; yv[i][1] = yin && in1 ? py[at + 1] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SS_ROWS; ++i) {
            f32x2 v[2 * SS_R + 2], h[2], fm[2];
            float u[2 * SS_R + 2], g[2], fc[2];
            const float4* c = (const float4*)s_in[buf][i] + tid;
            const float2* d = (const float2*)s_c[buf][i] + tid;
#pragma unroll
            for (int j = 0; j < SS_R + 1; ++j) {
                const float4 t = c[j];
                v[2 * j] = f2_pack(t.x, t.y);
                v[2 * j + 1] = f2_pack(t.z, t.w);
                const float2 e = d[j];
                u[2 * j] = e.x;
                u[2 * j + 1] = e.y;
            }
            hsum2(v, w, h);
            hsum1(u, w1, g);
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                fm[o] = cm[o].feed(h[o], w);
                fc[o] = cc[o].feed(g[o], w1);
            }
            const int yo = r + i - SS_R;
            if (yo < 0 || yo >= nrow) continue;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                float f0, f1;
                f2_unpack(fm[o], f0, f1);
                const float f2 = fc[o];
                const float x = xv[i][o], y = yv[i][o];
                const float dS = f0 + 2.f * x * f1 + y * f2;
                const float dd = x - y;
                const float sg = dd > 0.f ? 1.f : (dd < 0.f ? -1.f : 0.f);
                if (o ? in1 : in0) pg[yo * b.W + o] = scale * ((1.f - lam) * sg - lam * dS);
            }
        }
    }
}

// ------------------------------------------------------------ tiles
// The same pass pair over 32x32 tiles of 256 threads: a tile and its halo are staged,
// the horizontal and then the vertical window sums go through shared memory.  More
// work per pixel than the strips, but a block is done in a fraction of a segment's
// serial rounds and narrow images waste less of it (ssim_plan says which runs).  Maps in
// the image's own layout [3 channels][H][W]; the gradient has the strips' bits (every
// sum's taps in ascending order, the horizontal window first).
constexpr int ST_T = 32;               // output tile edge
constexpr int ST_E = ST_T + 2 * SS_R;  // staged edge (42)
constexpr int ST_THREADS = 256;        // 32 x 8

__device__ __forceinline__ float tap(const Win& win, int k) { return win.w[k <= SS_R ? k : 2 * SS_R - k]; }

// Stage plane[y0 - R .. y0 + T + R) x [x0 - R ..) into s (zero outside the image).
// Thread t < 252 keeps column t % 42 and takes the rows t / 42 + 6 k (k < 7),
// so its column test and offsets are formed once; all of its loads are issued
// before its first shared store.
constexpr int ST_SR = ST_THREADS / ST_E;  // staged rows per pass (6)
static_assert(ST_E % ST_SR == 0, "the staged rows split evenly into passes");
__device__ inline void stage(const float* __restrict__ plane, int W, int H, int x0, int y0, float (*s)[ST_E + 1])
{
    constexpr int NR = ST_E / ST_SR;
    const int t = threadIdx.x;
    if (t >= ST_SR * ST_E) return;
    const int c = t % ST_E, r0 = t / ST_E;
    const int x = x0 - SS_R + c;
    const bool xok = x >= 0 && x < W;
    const int ys = y0 - SS_R + r0;
    float v[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int y = ys + ST_SR * k;
        v[k] = (xok && y >= 0 && y < H) ? plane[(size_t)y * W + x] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) s[r0 + ST_SR * k][c] = v[k];
}

// Work split of the two window passes: the horizontal pass gives each thread
// ST_SL adjacent outputs of one staged row (one load per input, reused by the
// ST_SL sums), the vertical pass ST_SL adjacent output rows of one column.
constexpr int ST_SL = 4;
static_assert((ST_THREADS / 32) * ST_SL == ST_T && ST_T / ST_SL == 8, "vertical: one warp per ST_SL rows; horizontal: 8 groups per row");

__global__ void __launch_bounds__(ST_THREADS)
k_ssim_fwd_t(const float* __restrict__ img, const float* __restrict__ tgt, SViews sv, Win win,
           float* __restrict__ dm, float* __restrict__ da, float* __restrict__ dc, float2* __restrict__ part)
{
    __shared__ float sx[ST_E][ST_E + 1];
    __shared__ float sy[ST_E][ST_E + 1];
    // horizontal sums: mu_x, mu_y, a + b, c (S needs E[x^2] and E[y^2] only
    // through their sum, so one window sum serves both)
    __shared__ float hs[4][ST_E][ST_T];
    __shared__ float red[2][ST_THREADS / 32];
    const Blk b = decode(sv, blockIdx.x);
    const int x0 = b.tx * ST_T, y0 = b.y0;
    stage(img + b.plane, b.W, b.H, x0, y0, sx);
    stage(tgt + b.plane, b.W, b.H, x0, y0, sy);
    __syncthreads();
    // (lanes: 8 groups of ST_SL columns x 4 rows per warp; banks all distinct)
    for (int it = threadIdx.x; it < ST_E * (ST_T / ST_SL); it += ST_THREADS) {
        const int r = it / (ST_T / ST_SL), c0 = (it % (ST_T / ST_SL)) * ST_SL;
        float xv[ST_SL + 2 * SS_R], yv[ST_SL + 2 * SS_R];
#pragma unroll
        for (int q = 0; q < ST_SL + 2 * SS_R; ++q) { xv[q] = sx[r][c0 + q]; yv[q] = sy[r][c0 + q]; }
#pragma unroll
        for (int o = 0; o < ST_SL; ++o) {
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * SS_R; ++k) {
                const float x = xv[o + k], y = yv[o + k], w = tap(win, k);
                s0 = fmaf(w, x, s0);
                s1 = fmaf(w, y, s1);
                s2 = fmaf(w, fmaf(x, x, y * y), s2);
                s3 = fmaf(w, x * y, s3);
            }
            hs[0][r][c0 + o] = s0; hs[1][r][c0 + o] = s1; hs[2][r][c0 + o] = s2;
            hs[3][r][c0 + o] = s3;
        }
    }
    __syncthreads();
    // vertical pass: lane = column, warp w = output rows ST_SL w .. ST_SL w + ST_SL - 1
    const int c = threadIdx.x & 31, rb = (threadIdx.x >> 5) * ST_SL;
    float st[4][ST_SL];  // window sums of the four statistics at this thread's outputs
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        float col[ST_SL + 2 * SS_R];
#pragma unroll
        for (int q = 0; q < ST_SL + 2 * SS_R; ++q) col[q] = hs[t][rb + q][c];
#pragma unroll
        for (int j = 0; j < ST_SL; ++j) {
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * SS_R; ++k) acc = fmaf(tap(win, k), col[j + k], acc);
            st[t][j] = acc;
        }
    }
    float ssum = 0.f, l1sum = 0.f;  // of 1 - S and |x - y|
#pragma unroll
    for (int j = 0; j < ST_SL; ++j) {
        const int r = rb + j;
        const int x = x0 + c, y = y0 + r;
        if (x >= b.W || y >= b.H) continue;
        const float mx = st[0][j], my = st[1][j], ab = st[2][j], cc = st[3][j];
        const float A1 = 2.f * mx * my + kC1;
        const float A2 = 2.f * (cc - mx * my) + kC2;
        const float B1 = mx * mx + my * my + kC1;
        const float B2 = (ab - mx * mx - my * my) + kC2;
        const float inv = 1.f / (B1 * B2);
        const float S = A1 * A2 * inv;
        const size_t o = (size_t)b.plane + (size_t)y * b.W + x;
        dm[o] = 2.f * my * (A2 - A1) * inv - 2.f * mx * S * (B2 - B1) * inv;
        da[o] = -S * B1 * inv;
        dc[o] = 2.f * A1 * inv;
        ssum += 1.f - S;
        l1sum += fabsf(sx[r + SS_R][c + SS_R] - sy[r + SS_R][c + SS_R]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ssum += __shfl_xor_sync(0xffffffffu, ssum, o);
        l1sum += __shfl_xor_sync(0xffffffffu, l1sum, o);
    }
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = ssum; red[1][threadIdx.x >> 5] = l1sum; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f, l = 0.f;
        for (int w = 0; w < ST_THREADS / 32; ++w) { s += red[0][w]; l += red[1][w]; }
        part[blockIdx.x] = make_float2(s, l);
    }
}

__global__ void __launch_bounds__(ST_THREADS, 4)
k_ssim_bwd_t(const float* __restrict__ img, const float* __restrict__ tgt, SViews sv, Win win,
           const float* __restrict__ dm, const float* __restrict__ da, const float* __restrict__ dc,
           float lam, float* __restrict__ grad, const float2* __restrict__ part, float* __restrict__ loss)
{
    __shared__ float s0[ST_E][ST_E + 1];
    __shared__ float s1[ST_E][ST_E + 1];
    __shared__ float s2[ST_E][ST_E + 1];
    __shared__ float hs[3][ST_E][ST_T];
    if (blockIdx.x == 0) {  // the losses, from the forward's block sums
        ssim_final<ST_THREADS / 32>(part, sv, lam, loss);
        return;
    }
    const Blk b = decode(sv, blockIdx.x - 1);
    const int x0 = b.tx * ST_T, y0 = b.y0;
    // this thread's outputs (column c, rows rb ..): their x and y are loaded
    // first, so the loads' latency passes during the window sums
    const int c = threadIdx.x & 31, rb = (threadIdx.x >> 5) * ST_SL;
    float xo[ST_SL], yo[ST_SL];
#pragma unroll
    for (int j = 0; j < ST_SL; ++j) {
        const int x = x0 + c, y = y0 + rb + j;
        const bool in = x < b.W && y < b.H;
        const size_t o = (size_t)b.plane + (size_t)(in ? y : 0) * b.W + (in ? x : 0);
        xo[j] = in ? img[o] : 0.f;
        yo[j] = in ? tgt[o] : 0.f;
    }
    stage(dm + b.plane, b.W, b.H, x0, y0, s0);
    stage(da + b.plane, b.W, b.H, x0, y0, s1);
    stage(dc + b.plane, b.W, b.H, x0, y0, s2);
    __syncthreads();
    for (int it = threadIdx.x; it < ST_E * (ST_T / ST_SL); it += ST_THREADS) {
        const int r = it / (ST_T / ST_SL), c0 = (it % (ST_T / ST_SL)) * ST_SL;
        float v0[ST_SL + 2 * SS_R], v1[ST_SL + 2 * SS_R], v2[ST_SL + 2 * SS_R];
#pragma unroll
        for (int q = 0; q < ST_SL + 2 * SS_R; ++q) { v0[q] = s0[r][c0 + q]; v1[q] = s1[r][c0 + q]; v2[q] = s2[r][c0 + q]; }
#pragma unroll
        for (int o = 0; o < ST_SL; ++o) {
            float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * SS_R; ++k) {
                const float w = tap(win, k);
                a0 = fmaf(w, v0[o + k], a0);
                a1 = fmaf(w, v1[o + k], a1);
                a2 = fmaf(w, v2[o + k], a2);
            }
            hs[0][r][c0 + o] = a0; hs[1][r][c0 + o] = a1; hs[2][r][c0 + o] = a2;
        }
    }
    __syncthreads();
    // d/dx of the mean over views of (1 - lam) mean|x - y| + lam (1 - mean S)
    const float scale = 1.f / ((float)sv.n * 3.f * (float)b.W * (float)b.H);
    float fs[3][ST_SL];  // filtered partial-derivative maps at this thread's outputs
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        float col[ST_SL + 2 * SS_R];
#pragma unroll
        for (int q = 0; q < ST_SL + 2 * SS_R; ++q) col[q] = hs[t][rb + q][c];
#pragma unroll
        for (int j = 0; j < ST_SL; ++j) {
            float acc = 0.f;
#pragma unroll
            for (int k = 0; k <= 2 * SS_R; ++k) acc = fmaf(tap(win, k), col[j + k], acc);
            fs[t][j] = acc;
        }
    }
#pragma unroll
    for (int j = 0; j < ST_SL; ++j) {
        const int r = rb + j;
        const int x = x0 + c, y = y0 + r;
        if (x >= b.W || y >= b.H) continue;
        const float f0 = fs[0][j], f1 = fs[1][j], f2 = fs[2][j];
        const size_t o = (size_t)b.plane + (size_t)y * b.W + x;
        const float xv = xo[j], yv = yo[j];
        const float dS = f0 + 2.f * xv * f1 + yv * f2;
        const float d = xv - yv;
        const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        grad[o] = scale * ((1.f - lam) * sg - lam * dS);
    }
}

}  // namespace
}  // namespace dg

// Strips of SS_W columns or tiles (see k_ssim_fwd_t), and the blocks of the call.
struct SsimPlan {
    dg::SViews sv;
    bool tiles;
    long long nmap;    // values of one map
    size_t map_bytes;  // of the three maps, as the workspace holds them
    size_t ws_bytes;
};

// Views cut into blocks of cols x rows pixels; maps in strips of map_cols columns (0: as
// the image).
static void ssim_blocks(const int32_t* wh, int n, int cols, int rows, int map_cols, SsimPlan* p)
{
    dg::SViews& sv = p->sv;
    long long blocks = 0, pix = 0, map = 0;
    sv.n = n;
    sv.rows = rows;
    for (int v = 0; v < n; ++v) {
        const int W = wh[2 * v], H = wh[2 * v + 1];
        sv.W[v] = W; sv.H[v] = H;
        sv.TX[v] = (W + cols - 1) / cols;
        sv.TY[v] = (H + rows - 1) / rows;
        sv.boff[v] = (int)blocks;
        sv.poff[v] = pix;
        sv.moff[v] = map;
        blocks += 3LL * sv.TX[v] * sv.TY[v];  // (at most 65536 x 65536 in each of 16 views)
        pix += (long long)W * H;
        map += 3LL * H * (map_cols ? sv.TX[v] * map_cols : W);
    }
    sv.boff[n] = (int)blocks;
    p->nmap = map;
}

static bool ssim_plan(const int32_t* wh, int n_views, SsimPlan* p)
{
    if (!wh) { dg_set_error("wh is null"); return false; }
    if (n_views < 1 || n_views > DG_MAX_VIEWS) { dg_set_error("n_views %d outside 1..%d", n_views, DG_MAX_VIEWS); return false; }
    long long plain = 0, padded = 0, tile_blocks = 0;
    for (int v = 0; v < n_views; ++v) {
        const int W = wh[2 * v], H = wh[2 * v + 1];
        if (W <= 0 || H <= 0 || W > (1 << 16) || H > (1 << 16)) { dg_set_error("view %d: image size %dx%d", v, W, H); return false; }
        const long long strips = (W + dg::SS_W - 1) / dg::SS_W;
        plain += (long long)W * H;
        padded += strips * dg::SS_W * H;
        tile_blocks += 3LL * ((W + dg::ST_T - 1) / dg::ST_T) * ((H + dg::ST_T - 1) / dg::ST_T);
    }
    // rows of a segment: 64 when that gives at least five blocks per SM, else 32: a
    // segment repeats the window sums of ten rows.  (16 views of 1237x822: 64 rows
    // 0.615 ms, 128 0.635; one view, in a training step: 32 rows 8 us less than 16.)
    ssim_blocks(wh, n_views, dg::SS_W, 64, dg::SS_W, p);
    if (p->sv.boff[n_views] < 5 * 152) ssim_blocks(wh, n_views, dg::SS_W, 32, dg::SS_W, p);
    // Tiles while they are few (a strip's rounds are one chain: up to 2432 tiles, 16 per
    // SM, 0.66 to 0.95 of the strips' time), and where the strips' padding or repeated
    // rows cost more than the tiles' windows: a tile takes as long as about 11.5 rows of
    // a strip (19 ns against 1.4 to 1.9).  One view of 1237x822: tiles 60 us, strips 52;
    // 16 of 309x205 67 and 75, of 129x1000 146 and 172, of 16x3000 86 and 228, of 385x500
    // 189 and 177.  (padded <= 1.5 plain holds the workspace's maps to that, too.)
    long long strip_rows = 0;
    for (int v = 0; v < n_views; ++v)
        strip_rows += 3LL * p->sv.TX[v] * (p->sv.H[v] + 2 * dg::SS_R * p->sv.TY[v]);
    p->tiles = padded * 2 > plain * 3 || tile_blocks <= 16 * 152 || 23 * tile_blocks < 2 * strip_rows;
    if (p->tiles) ssim_blocks(wh, n_views, dg::ST_T, dg::ST_T, 0, p);
    // the workspace: maps, then the block sums (of the tiles: never fewer than the strips'
    // segments), so that it grows with every size and serves smaller images too; 16 bytes
    // for the maps' alignment
    const long long maps = padded * 2 <= plain * 3 ? padded : plain + (plain + 1) / 2;
    p->map_bytes = ((size_t)3 * 3 * maps * sizeof(float) + 255) & ~(size_t)255;
    p->ws_bytes = 16 + p->map_bytes + sizeof(float2) * (size_t)tile_blocks;
    return true;
}

extern "C" size_t dg_ssim_workspace_size(const int32_t* wh, int32_t n_views)
{
    SsimPlan p;
    return ssim_plan(wh, n_views, &p) ? p.ws_bytes : 0;
}

extern "C" dg_status dg_loss_l1_dssim(const float* img, const float* target, const int32_t* wh, int32_t n_views,
                                      float lambda, float* dL_dimg, float* loss, void* ws, size_t ws_bytes,
                                      dg_stream stream)
{
    SsimPlan p;
    if (!ssim_plan(wh, n_views, &p)) return DG_ERR_ARG;
    if (!img || !target || !dL_dimg || !loss) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    if (!(lambda >= 0.f && lambda <= 1.f)) { dg_set_error("lambda must be in [0, 1]"); return DG_ERR_ARG; }
    if (!ws || ws_bytes < p.ws_bytes) { dg_set_error("ssim workspace missing or too small (%zu < %zu bytes)", ws_bytes, p.ws_bytes); return DG_ERR_ARG; }
    dg::Win win;
    double sum = 0.0, w[2 * dg::SS_R + 1];
    for (int k = 0; k <= 2 * dg::SS_R; ++k) {
        const double x = (double)(k - dg::SS_R);
        w[k] = exp(-x * x / (2.0 * 1.5 * 1.5));
        sum += w[k];
    }
    for (int k = 0; k <= dg::SS_R; ++k) win.w[k] = (float)(w[k] / sum);
    float* dm = (float*)(((uintptr_t)ws + 15) & ~(uintptr_t)15);
    float* da = dm + p.nmap;
    float* dc = da + p.nmap;
    float2* part = (float2*)((char*)dm + p.map_bytes);
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = p.sv.boff[p.sv.n];
    if (p.tiles) {
        dg::k_ssim_fwd_t<<<nb, dg::ST_THREADS, 0, s>>>(img, target, p.sv, win, dm, da, dc, part);
        dg::k_ssim_bwd_t<<<nb + 1, dg::ST_THREADS, 0, s>>>(img, target, p.sv, win, dm, da, dc, lambda, dL_dimg, part, loss);
    } else {
        dg::k_ssim_fwd<<<nb, dg::SS_THREADS, 0, s>>>(img, target, p.sv, win, dm, da, dc, part);
        dg::k_ssim_bwd<<<nb + 1, dg::SS_THREADS, 0, s>>>(img, target, p.sv, win, dm, da, dc, lambda, dL_dimg, part, loss);
    }
    dg_note_launch(2);
    return dg_check_launch("loss_l1_dssim");
}
