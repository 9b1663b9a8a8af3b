// scan.cuh -- warp and block prefix sums (binning, densification) and the
// device-wide exclusive scan of the render split plan.  Kernels live in an
// anonymous namespace: each including translation unit gets its own copy.
#pragma once

#include "common.cuh"

namespace dg {
namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_IPT = 16;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_IPT;

template <typename T>
__device__ inline T warp_incl_scan(T x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Block-wide exclusive scan of one value per thread; *total receives the sum.
// smem: at least 33 elements.  Ends with a barrier so smem can be reused.
template <typename T>
__device__ inline T block_excl_scan(T v, T* smem, T* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const T inc = warp_incl_scan(v, lane);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? smem[lane] : T(0);
        w = warp_incl_scan(w, lane);
        smem[lane] = w;
    }
    __syncthreads();
    const T pre = warp > 0 ? smem[warp - 1] : T(0);
    *total = smem[nw - 1];
    __syncthreads();
    return pre + inc - v;
}

// --------------------------------------------------------------- scan
template <typename Load>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(Load ld, long long n, uint64_t* bsum)
{
    __shared__ uint64_t sm[33];
    const long long base = (long long)blockIdx.x * SCAN_TILE;
    uint64_t acc = 0;
#pragma unroll
    for (int k = 0; k < SCAN_IPT; ++k) {
        const long long i = base + (long long)k * SCAN_THREADS + threadIdx.x;
        if (i < n) acc += ld(i);
    }
    uint64_t tot;
    block_excl_scan<uint64_t>(acc, sm, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_top(uint64_t* bsum, int nb, long long* total_out)
{
    __shared__ uint64_t sm[33];
    uint64_t carry = 0;
    for (int base = 0; base < nb; base += 1024) {
        const int i = base + threadIdx.x;
        const uint64_t v = i < nb ? bsum[i] : 0;
        uint64_t tot;
        const uint64_t ex = block_excl_scan<uint64_t>(v, sm, &tot);
        if (i < nb) bsum[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0 && total_out) *total_out = (long long)carry;
}

template <typename Load, typename TOut>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(Load ld, long long n, const uint64_t* bsum, TOut* out)
{
    __shared__ uint64_t sm[33];
    const long long base = (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_IPT;
    uint64_t v[SCAN_IPT];
    uint64_t acc = 0;
#pragma unroll
    for (int k = 0; k < SCAN_IPT; ++k) {
        const long long i = base + k;
        v[k] = i < n ? ld(i) : 0;
        acc += v[k];
    }
    uint64_t tot;
    uint64_t run = block_excl_scan<uint64_t>(acc, sm, &tot) + bsum[blockIdx.x];
#pragma unroll
    for (int k = 0; k < SCAN_IPT; ++k) {
        const long long i = base + k;
        if (i < n) out[i] = (TOut)run;
        run += v[k];
    }
}

template <typename Load, typename TOut>
static void exclusive_scan(Load ld, long long n, TOut* out, uint64_t* bsum, long long* total, cudaStream_t s)
{
    const int nb = (int)((n + SCAN_TILE - 1) / SCAN_TILE);
    if (nb == 0) {
        if (total) cudaMemsetAsync(total, 0, sizeof(long long), s);
        return;
    }
    k_scan_reduce<<<nb, SCAN_THREADS, 0, s>>>(ld, n, bsum);
    dg_note_launch();
    k_scan_top<<<1, 1024, 0, s>>>(bsum, nb, total);
    dg_note_launch();
    k_scan_down<<<nb, SCAN_THREADS, 0, s>>>(ld, n, bsum, out);
    dg_note_launch();
}

}  // namespace
}  // namespace dg
