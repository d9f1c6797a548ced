// device_util.cuh -- warp/block reductions and scans used by the kernels.
#pragma once

#include <cuda_runtime.h>

namespace amg {

constexpr unsigned FULL_MASK = 0xffffffffu;

__device__ __forceinline__ int warp_sum_int(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

__device__ __forceinline__ int warp_max_int(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(FULL_MASK, v, o));
    return v;
}

// Block-wide sum (any blockDim multiple of 32, <= 1024). All threads get it.
__device__ __forceinline__ int block_sum_int(int v) {
    __shared__ int ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum_int(v);
    if (lane == 0) ws[wid] = v;
    __syncthreads();
    int t = (lane < nw) ? ws[lane] : 0;
    t = warp_sum_int(t);
    __syncthreads();
    return t;
}

// Block-wide maximum (any blockDim multiple of 32, <= 1024). All threads get it.
__device__ __forceinline__ int block_max_int(int v) {
    __shared__ int wm[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_max_int(v);
    if (lane == 0) wm[wid] = v;
    __syncthreads();
    int t = (lane < nw) ? wm[lane] : 0;
    t = warp_max_int(t);
    __syncthreads();
    return t;
}

// Sums of NV doubles over a block of T threads in a fixed combination order
// (deterministic for a fixed T): the sum of v[j] comes back on every lane of
// warp j (0 elsewhere). This GPU issues one FP64 warp instruction per 64
// cycles of an SM sub-partition, so the number of warp-wide additions is what
// a block sum costs: the values go through shared memory and one warp per
// value adds T / 32 columns and then its lanes, T / 32 + 4 additions a value.
// (A butterfly in every warp and again over the warps took 10 T / 32 of them
// and 10 us of every kernel that ends in a dot product at 8 blocks per SM: the
// product with its dot on 32^3 rows 17.1 -> 10.2 us, with grids sized by the
// rows; a 32^3 solve 1.89 -> 1.34 ms.)
// Consecutive calls need a block barrier between them.
template <int T, int NV>
__device__ __forceinline__ double block_sums(const double (&v)[NV]) {
    __shared__ double sm[NV][T];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j) sm[j][threadIdx.x] = v[j];
    __syncthreads();
    // up to 256 values: 8 columns a lane by warp j; more: a warp per 256 values
    // first, which halves the serial chain at 1024 threads
    constexpr int P = T > 256 ? T / 256 : 1, C = T / P;
    double s0 = 0.0;
    if (w < NV * P) {
        const double* col = sm[w / P] + (w % P) * C + lane;
        s0 = col[0];
        double s1 = col[32];
#pragma unroll
        for (int k = 64; k < C; k += 64) {
            s0 += col[k];
            s1 += col[k + 32];
        }
        s0 += s1;
    }
    if constexpr (P > 1) {
        if (w < NV * P) sm[w / P][(w % P) * C + lane] = s0;
        __syncthreads();
        if (w < NV) {
            s0 = sm[w][lane];
#pragma unroll
            for (int q = 1; q < P; ++q) s0 += sm[w][q * C + lane];
        }
    }
    return w < NV ? warp_sum(s0) : 0.0;
}

// Block-wide exclusive scan of ints.
__device__ __forceinline__ int block_exclusive_scan_int(int v) {
    __shared__ int ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(FULL_MASK, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int t = (lane < nw) ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(FULL_MASK, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    int r = x - v + (wid > 0 ? ws[wid - 1] : 0);
    __syncthreads();
    return r;
}

// Warp-aggregated append of one item per participating lane to list[*cnt];
// items past `cap` are dropped (the caller sizes lists so this cannot happen).
__device__ __forceinline__ void warp_append(bool take, int item, int* list, int* cnt, int cap) {
    const unsigned act = __activemask();
    const unsigned m = __ballot_sync(act, take);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(act, base, leader);
    const int pos = base + __popc(m & ((1u << lane) - 1));
    if (take && pos < cap) list[pos] = item;
}

}  // namespace amg
