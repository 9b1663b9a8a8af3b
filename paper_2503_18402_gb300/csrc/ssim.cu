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
// Two passes (k_ssim_fwd, k_ssim_bwd), each over strips of SS_W output columns
// and segments of rows, a thread per two adjacent columns.  Going down the rows,
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
// SM, 160 registers; five 0.644, seven 0.618, eight 0.655).  The vertical window
// first, four outputs per thread in the horizontal one, took 0.535 ms, but rounds
// the gradient differently (3e-6 relative, no nearer to the exact one).
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
// |x - y| about 1e-3: 7.4e-7 -> 5.5e-7).  630 -> 636 us on 16 views of 1237x822.
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
// block: with one or two views four or two warps share a view, else each warp
// takes every fourth one; a warp sums a fixed stride of its view's block sums in
// FP64, and the warps' and the views' sums are added in a fixed order, so the
// result does not depend on timing.  It is the backward's first block: as a launch
// of its own behind the backward it took 8 us for one view and 12 us for 16.
__device__ void ssim_final(const float2* __restrict__ part, const SViews& sv, float lam, float* __restrict__ loss)
{
    constexpr int NW = SS_THREADS / 32;
    __shared__ double sm[2][DG_MAX_VIEWS][NW];
    __shared__ double lv_s[DG_MAX_VIEWS];
    const int nv = sv.n;
    const int wpv = nv == 1 ? NW : nv == 2 ? NW / 2 : 1;  // warps per view
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
        ssim_final(part, sv, lam, loss);
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

}  // namespace
}  // namespace dg

// Rows of a segment: the longest of 64, 32, 16 that gives at least five blocks
// per SM, else 8: a segment repeats the window sums of ten rows.  (16 views of
// 1237x822: 64 rows 0.615 ms, 128 0.635; one view, in a training step: 32 rows 8 us
// less than 16.)
static bool ssim_views(const int32_t* wh, int n_views, dg::SViews* sv, long long* nmap)
{
    if (!wh) { dg_set_error("wh is null"); return false; }
    if (n_views < 1 || n_views > DG_MAX_VIEWS) { dg_set_error("n_views %d outside 1..%d", n_views, DG_MAX_VIEWS); return false; }
    sv->n = n_views;
    for (int v = 0; v < n_views; ++v) {
        const int W = wh[2 * v], H = wh[2 * v + 1];
        if (W <= 0 || H <= 0 || W > (1 << 16) || H > (1 << 16)) { dg_set_error("view %d: image size %dx%d", v, W, H); return false; }
    }
    for (int rows = 64;; rows /= 2) {
        long long blocks = 0, pix = 0, map = 0;
        sv->rows = rows;
        for (int v = 0; v < n_views; ++v) {
            const int W = wh[2 * v], H = wh[2 * v + 1];
            sv->W[v] = W; sv->H[v] = H;
            sv->TX[v] = (W + dg::SS_W - 1) / dg::SS_W;
            sv->TY[v] = (H + rows - 1) / rows;
            sv->boff[v] = (int)blocks;
            sv->poff[v] = pix;
            sv->moff[v] = map;
            blocks += 3LL * sv->TX[v] * sv->TY[v];
            pix += (long long)W * H;
            map += 3LL * sv->TX[v] * H * dg::SS_W;
            if (blocks >= (1LL << 31) - 1) { dg_set_error("images too large"); return false; }
        }
        sv->boff[n_views] = (int)blocks;
        *nmap = map;
        if (blocks >= 5 * 152 || rows == 8) return true;
    }
}

// Maps, then the block sums, with room for the shortest segments (so that a
// workspace serves smaller images too) and for the maps' 16-byte alignment.
static size_t ssim_map_bytes(long long nmap) { return ((size_t)3 * nmap * sizeof(float) + 255) & ~(size_t)255; }
static size_t ssim_ws_bytes(const dg::SViews& sv, long long nmap)
{
    size_t blocks = 0;
    for (int v = 0; v < sv.n; ++v) blocks += (size_t)3 * sv.TX[v] * ((sv.H[v] + 7) / 8);
    return 16 + ssim_map_bytes(nmap) + sizeof(float2) * blocks;
}

extern "C" size_t dg_ssim_workspace_size(const int32_t* wh, int32_t n_views)
{
    dg::SViews sv;
    long long nmap = 0;
    if (!ssim_views(wh, n_views, &sv, &nmap)) return 0;
    return ssim_ws_bytes(sv, nmap);
}

extern "C" dg_status dg_loss_l1_dssim(const float* img, const float* target, const int32_t* wh, int32_t n_views,
                                      float lambda, float* dL_dimg, float* loss, void* ws, size_t ws_bytes,
                                      dg_stream stream)
{
    dg::SViews sv;
    long long nmap = 0;
    if (!ssim_views(wh, n_views, &sv, &nmap)) return DG_ERR_ARG;
    if (!img || !target || !dL_dimg || !loss) { dg_set_error("null buffer"); return DG_ERR_ARG; }
    if (!(lambda >= 0.f && lambda <= 1.f)) { dg_set_error("lambda must be in [0, 1]"); return DG_ERR_ARG; }
    const size_t need = ssim_ws_bytes(sv, nmap);
    if (!ws || ws_bytes < need) { dg_set_error("ssim workspace missing or too small (%zu < %zu bytes)", ws_bytes, need); return DG_ERR_ARG; }
    dg::Win win;
    double sum = 0.0, w[2 * dg::SS_R + 1];
    for (int k = 0; k <= 2 * dg::SS_R; ++k) {
        const double x = (double)(k - dg::SS_R);
        w[k] = exp(-x * x / (2.0 * 1.5 * 1.5));
        sum += w[k];
    }
    for (int k = 0; k <= dg::SS_R; ++k) win.w[k] = (float)(w[k] / sum);
    float* dm = (float*)(((uintptr_t)ws + 15) & ~(uintptr_t)15);
    float* da = dm + nmap;
    float* dc = da + nmap;
    float2* part = (float2*)((char*)dm + ssim_map_bytes(nmap));
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = sv.boff[sv.n];
    dg::k_ssim_fwd<<<nb, dg::SS_THREADS, 0, s>>>(img, target, sv, win, dm, da, dc, part);
    dg::k_ssim_bwd<<<nb + 1, dg::SS_THREADS, 0, s>>>(img, target, sv, win, dm, da, dc, lambda, dL_dimg, part, loss);
    dg_note_launch(2);
    return dg_check_launch("loss_l1_dssim");
}
