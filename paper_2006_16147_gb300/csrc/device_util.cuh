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
// warp j (0 elsewhere). This GPU issues one FP64 warp instruction per 76
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

// Programmatic dependent launch: a kernel started with launch_dep
// (amg_internal.cuh) may begin while the kernel before it on the stream still
// runs. It does what needs only the hierarchy's arrays, then dep_wait() returns
// when that kernel is done and its writes are visible; and only then may the
// next one begin, so at most two kernels overlap. Vectors that an earlier kernel
// wrote are read after the wait and with ldv: an ordinary load, never ld.nc,
// which the compiler picks for const __restrict__ pointers and which the wait
// does not order.
__device__ __forceinline__ void dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename T>
__device__ __forceinline__ T ldv(const T* p) { return __ldca(p); }

// ----------------------------------------- FP64 beside a slow FP64 pipe ----
// An FP64 instruction takes 76 cycles of a sub-partition's pipe per warp here
// (measured with independent FMAs, adds and multiplies: 0.53 T lanes/s at 2070
// MHz), a conversion from or to float twice that, also where a predicate turns it off;
// FP32 and integer instructions take one or two. f2d is the same value moved
// field by field without a branch.
__device__ __forceinline__ double f2d(float f) {
    const unsigned a0 = __float_as_uint(f) & 0x7fffffffu;
    const bool small = a0 < 0x00800000u;                          // zero or subnormal: scaled to a normal first
    const unsigned u = __float_as_uint(small ? f * 0x1p64f : f), a = u & 0x7fffffffu;
    unsigned off = small ? 0x38000000u - (64u << 20) : 0x38000000u;
    off = a0 >= 0x7f800000u ? 0x70000000u : off;                  // infinity, NaN
    return __hiloint2double((int)((a ? (a >> 3) + off : 0u) | (u & 0x80000000u)), (int)(u << 29));
}

// The nearest float, for results that are normal; else by the conversion, in a
// call so that it is not predicated.
static __device__ __noinline__ float d2f_rare(double d) { return (float)d; }
__device__ __forceinline__ float d2f(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e - 897u >= 253u && ((hi << 1) | lo)) return d2f_rare(d);   // else the result is in 2^-126 .. 2^127, or zero
    unsigned t = (__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7fffffffu;
    const unsigned rest = lo << 3;                                // the 29 bits below the result's last
    t += rest > 0x80000000u || (rest == 0x80000000u && (t & 1u));
    return __uint_as_float((e ? t : 0u) | (hi & 0x80000000u));
}

__device__ __forceinline__ float rcp_approx(float y) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

// Correctly rounded quotient of doubles without the FP64 pipe (a division
// holds it for some ten instructions of 76 cycles a warp). Mantissas n, d: the
// integer Q = floor(n 2^53 / d), by a 24-bit reciprocal, one Newton step in
// 64-bit integers and an exact remainder that corrects the last bits; the
// quotient of two doubles is never half-way between two, so Q's last bit alone
// decides the rounding. Zero, subnormal, infinite or NaN operands and quotients
// near the ends of the range take the division instruction sequence.
__device__ __forceinline__ double div_rn(double a, double b) {
    const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
    const unsigned long long ub = (unsigned long long)__double_as_longlong(b);
    const int ea = (int)(ua >> 52) & 0x7ff, eb = (int)(ub >> 52) & 0x7ff;
    int e = ea - eb + 1023;
    if ((unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || (unsigned)(e - 2) >= 2044u) return __ddiv_rn(a, b);
    const unsigned long long one = 1ull << 52;
    unsigned long long n = (ua & (one - 1)) | one;
    const unsigned long long d = (ub & (one - 1)) | one;
    if (n < d) {                                          // quotient in [1, 2)
        n <<= 1;
        --e;
    }
    // x 2^-23 ~ 2^53 / d, in (1, 2]: from d's top 24 bits as a float in [1, 2)
    const float y = __uint_as_float(0x3f800000u | (unsigned)((d >> 29) & 0x7fffffu));
    const unsigned x = (unsigned)(rcp_approx(y) * 0x1p24f);
    const long long r0 = -(long long)(d * x);             // 2^76 - x d, below 2^55
    const unsigned long long x1 = ((unsigned long long)x << 36) + (unsigned long long)(((r0 >> 20) * (long long)x) >> 20);
    // x1 2^-59 ~ 2^53 / d; Q ~ n x1 2^-59
    unsigned long long q = __umul64hi(n << 10, x1) >> 5;
    long long r = (long long)((n << 53) - q * d);         // exact: below 2^63
    const long long dq = ((r >> 30) * (long long)x) >> 46;
    q += (unsigned long long)dq;
    r -= dq * (long long)d;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        if (r < 0) { r += (long long)d; --q; }
        else if (r >= (long long)d) { r -= (long long)d; ++q; }
    }
    q = (q + 1) >> 1;                                     // at most 2^53: then the exponent below carries
    return __longlong_as_double((long long)(((ua ^ ub) & (1ull << 63)) | (((unsigned long long)(e - 1) << 52) + q)));
}

// A double of magnitude 2^-104 .. 2^103 times 2^SPLIT_UP as three floats,
// exactly: 24, 23 and 6 bits of its mantissa. Anything else but zero gives NaN.
constexpr unsigned SPLIT_UP = 24;
struct Split3 {
    float h, m, l;
    bool one;         // the double is a float: m = l = 0
};
__device__ __forceinline__ Split3 split3(double a) {
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
    const unsigned sgn = hi & 0x80000000u, t = (__funnelshift_l(lo, hi, 3) - ((896u - SPLIT_UP) << 23)) & 0x7fffffffu;
    const unsigned rest = lo & 0x1fffffffu;
    Split3 s{__uint_as_float(t | sgn), 0.0f, 0.0f, rest == 0u};
    if (rest) {
        const unsigned e = (t & 0x7f800000u) | sgn, em = e - (23u << 23), el = e - (46u << 23);
        s.m = __uint_as_float(em | (rest >> 6)) - __uint_as_float(em);
        s.l = __uint_as_float(el | ((rest & 63u) << 17)) - __uint_as_float(el);
    }
    if (((hi >> 20) & 0x7ffu) - (943u - SPLIT_UP) > 207u) s.h = ((hi << 1) | lo) ? __uint_as_float(0x7fc00000u) : 0.0f;
    return s;
}

// Sum of products a z of doubles a (split) and floats z without the FP64 pipe:
// the products' high parts summed exactly into s1 + s2 (an error-free product
// by fma, Knuth's two-sum), what those leave, 2^-46 of the largest product and
// below, into s3. value() rounds twice in FP64, so the sum is nearer than a
// chain of FP64 FMAs, as long as ok(): the largest product lies in
// 2^-84 .. 2^96 and nothing was infinite or NaN. The pieces stand 2^SPLIT_UP
// higher, which puts that window in the middle of a float's exponents. Where the
// largest product lies in 2^-112 .. 2^103, ok_far(), the pieces hold the sum too,
// but for parts below a float's last bit, 2^-56 of that product and 2^-60 more
// per entry; value_far() takes some ten instructions more to move them into a
// double, which every row would pay for in value() (a solve of 112^3 rows x 64
// columns 140 ms, 144 ms with them). Beyond, the caller takes the FP64 chain after
// the pieces: with right-hand sides scaled by 2^-70 that solve took 209 ms while
// the window ended at 2^-60, 143 ms now.
struct SplitSum {
    float s1 = 0.0f, s2 = 0.0f, s3 = 0.0f, big = 0.0f;
    static __device__ __forceinline__ float two_sum(float& s, float x) {
        const float t = __fadd_rn(s, x), b = __fadd_rn(t, -s);
        const float e = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -b)), __fadd_rn(x, -b));
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(const Split3& a, float z) {
        const float h = __fmul_rn(a.h, z), e = __fmaf_rn(a.h, z, -h);
        big = fmaxf(big, fabsf(h));
        const float t = two_sum(s1, h);
        s3 = __fadd_rn(s3, two_sum(s2, t));
        s3 = __fadd_rn(s3, two_sum(s2, e));
        if (!a.one) {
            const float g = __fmul_rn(a.m, z);
            s3 = __fadd_rn(s3, two_sum(s2, g));
            s3 = __fadd_rn(s3, __fmaf_rn(a.m, z, -g));
            s3 = __fmaf_rn(a.l, z, s3);
        }
    }
    __device__ __forceinline__ bool ok() const {
        return big >= 0x1p-60f && big <= 0x1p120f && fabsf(s1) <= 0x1p126f;   // false for NaN
    }
    // f 2^-SPLIT_UP field by field as in f2d, from f 2^UP, whose magnitudes below 2^-126 are taken as zero
    template <unsigned UP>
    static __device__ __forceinline__ double wide(float f) {
        const unsigned u = __float_as_uint(UP ? f * (float)(1u << UP) : f), a = u & 0x7fffffffu;
        constexpr unsigned off = 0x38000000u - ((UP + SPLIT_UP) << 20);
        return a < 0x00800000u ? 0.0 : __hiloint2double((int)((a >> 3) + off | (u & 0x80000000u)), (int)(u << 29));
    }
    __device__ __forceinline__ double value() const { return wide<0>(s1) + (wide<0>(s2) + wide<0>(s3)); }
    // s2 and s3 keep below infinity when scaled up; a sum that overflowed on the way stays infinite or NaN in s1
    __device__ __forceinline__ bool ok_far() const {
        return big >= 0x1p-88f && fabsf(s1) <= 0x1.fffffep127f && fabsf(s2) + fabsf(s3) <= 0x1p107f;
    }
    __device__ __forceinline__ double value_far() const {
        return (fabsf(s1) < 0x1p-100f ? wide<20>(s1) : wide<0>(s1)) + (wide<20>(s2) + wide<20>(s3));
    }
};

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
