// block.cu -- several right-hand sides at once (multi-RHS block solve).
//
// Every column runs its own preconditioned CG (its own alpha, beta, rho and
// convergence), while each sparse product and the V-cycle (Eq. 2) serve all k
// columns in one pass over the matrices: the matrix is read once per k
// columns. Vectors are row-major n x k. A group of G lanes handles one row;
// lane gl owns the CPL consecutive columns gl * CPL .. gl * CPL + CPL - 1, so
// the group reads each matrix entry once (broadcast) and a gathered row of X
// as one coalesced segment, each lane's part as one vector load (float4,
// float2 or double2) when the row stride is a multiple of CPL.
//
// Columns carry a state (ColMode): START columns enter at the V-cycle half of
// a step (r given, z = B r, p = z), ACTIVE columns take a full CG step, a
// column whose recursive residual meets rtol goes to CHECK, where the true
// residual decides DONE or a restart. Columns in other states are carried
// along but never updated, so columns can join and leave between steps.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <memory>
#include <type_traits>

#include "amg_internal.cuh"
#include "device_util.cuh"

namespace amg {

BlockWork::~BlockWork() {
    for (auto& g : gstep)
        if (g) cudaGraphExecDestroy(g);
    if (mode_host) cudaFreeHost(mode_host);
    if (iters_host) cudaFreeHost(iters_host);
    if (rr_host) cudaFreeHost(rr_host);
    if (bb_host) cudaFreeHost(bb_host);
}

namespace {

constexpr int TPB = 256;
constexpr int WARPS = TPB / 32;
constexpr int MAXK = 256;
constexpr int CC_TPB = 512;   // threads of the iterative coarsest solve's blocks, one block per SM

struct SellV {
    int n, nslices;
    const int* __restrict__ sptr;
    const int* __restrict__ col;
    const int* __restrict__ perm;
};

__device__ __forceinline__ int rowid(const SellV& S, int ip) { return S.perm ? __ldg(S.perm + ip) : ip; }

struct Grp {
    int G, gl, gw, ngroups;
};

__device__ __forceinline__ Grp make_grp(int G) {
    Grp g;
    g.G = G;
    const int lane = threadIdx.x & 31;
    g.gl = lane & (G - 1);
    const int gpw = 32 / G;
    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    g.gw = warp * gpw + lane / G;
    g.ngroups = (int)((gridDim.x * blockDim.x) >> 5) * gpw;
    return g;
}

// The CPL consecutive values at p (a lane's columns of one row; lim of them
// are live columns). With VEC the row stride is a multiple of CPL, so the
// address is aligned to CPL values and all CPL lie inside the row: the loads
// are vectors. Without VEC only the live columns are read. Never ld.nc (see
// dep_wait).
template <bool VEC, int CPL, typename T>
__device__ __forceinline__ void ld_cols(const T* p, T (&v)[CPL], int lim) {
    if constexpr (VEC && std::is_same<T, float>::value && CPL >= 4) {
#pragma unroll
        for (int q = 0; q < CPL / 4; ++q) {
            const float4 f = __ldca(reinterpret_cast<const float4*>(p) + q);
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    } else if constexpr (VEC && std::is_same<T, float>::value && CPL == 2) {
        const float2 f = __ldca(reinterpret_cast<const float2*>(p));
        v[0] = f.x; v[1] = f.y;
    } else if constexpr (VEC && std::is_same<T, double>::value && CPL >= 2) {
#pragma unroll
        for (int q = 0; q < CPL / 2; ++q) {
            const double2 f = __ldca(reinterpret_cast<const double2*>(p) + q);
            v[2 * q] = f.x; v[2 * q + 1] = f.y;
        }
    } else {
#pragma unroll
        for (int m = 0; m < CPL; ++m) v[m] = m < lim ? __ldca(p + m) : T(0);
    }
}

// Plain loads of a lane's columns of a row that this kernel also writes.
template <bool VEC, int CPL, typename T>
__device__ __forceinline__ void ld_own(const T* p, T (&v)[CPL], int lim) {
    if constexpr (VEC && std::is_same<T, float>::value && CPL >= 4) {
#pragma unroll
        for (int q = 0; q < CPL / 4; ++q) {
            const float4 f = reinterpret_cast<const float4*>(p)[q];
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    } else if constexpr (VEC && std::is_same<T, float>::value && CPL == 2) {
        const float2 f = *reinterpret_cast<const float2*>(p);
        v[0] = f.x; v[1] = f.y;
    } else if constexpr (VEC && std::is_same<T, double>::value && CPL >= 2) {
#pragma unroll
        for (int q = 0; q < CPL / 2; ++q) {
            const double2 f = reinterpret_cast<const double2*>(p)[q];
            v[2 * q] = f.x; v[2 * q + 1] = f.y;
        }
    } else {
#pragma unroll
        for (int m = 0; m < CPL; ++m) v[m] = m < lim ? p[m] : T(0);
    }
}

// Stores a lane's columns of a row: one vector store when VEC and all of them
// are live columns (c0 + CPL <= k), else one store per live column.
template <bool VEC, int CPL, typename T>
__device__ __forceinline__ void st_cols(T* p, const T (&v)[CPL], int c0, int k) {
    if constexpr (VEC && std::is_same<T, float>::value && CPL >= 4) {
        if (c0 + CPL <= k) {
#pragma unroll
            for (int q = 0; q < CPL / 4; ++q)
                reinterpret_cast<float4*>(p)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            return;
        }
    } else if constexpr (VEC && std::is_same<T, float>::value && CPL == 2) {
        if (c0 + CPL <= k) {
            *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
            return;
        }
    } else if constexpr (VEC && std::is_same<T, double>::value && CPL >= 2) {
        if (c0 + CPL <= k) {
#pragma unroll
            for (int q = 0; q < CPL / 2; ++q) reinterpret_cast<double2*>(p)[q] = make_double2(v[2 * q], v[2 * q + 1]);
            return;
        }
    }
#pragma unroll
    for (int m = 0; m < CPL; ++m)
        if (c0 + m < k) p[m] = v[m];
}

// acc[m] += sum_e val_e * X[col_e * ld + c0 + m] for the row at SELL position
// ip, in entry order (a lane's columns c0 .. c0 + CPL - 1; a lane without a
// live column returns at once). Four entries at a time (the last group
// predicated): their indices and values are loaded first and the four
// gathered rows of X are in flight together, so a row costs about two memory
// latencies per four entries instead of two per entry.
template <bool VEC, int CPL, typename T>
__device__ __forceinline__ void sell_row_k(const SellV& S, const T* __restrict__ val, int ip, int c0, int k,
                                           const T* X, int ld, T (&acc)[CPL]) {
    if (c0 >= k) return;
    const int s = ip >> 5, r = ip & 31;
    const int s0 = __ldg(S.sptr + s);
    const int w = __ldg(S.sptr + s + 1) - s0;
    long long base = (long long)s0 * 32 + r;
    int e = 0;
    for (; e + 4 <= w; e += 4, base += 128) {
        int j[4];
        T a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            j[u] = __ldg(S.col + base + 32 * u);
            a[u] = __ldg(val + base + 32 * u);
        }
        T xs[4][CPL];
#pragma unroll
        for (int u = 0; u < 4; ++u) ld_cols<VEC, CPL>(X + (size_t)j[u] * ld + c0, xs[u], k - c0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int m = 0; m < CPL; ++m) acc[m] = fma(a[u], xs[u][m], acc[m]);
    }
    if (e < w) {                      // the last 1-3 entries as one predicated group of four
        int j[4];
        T a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool ok = e + u < w;
            j[u] = ok ? __ldg(S.col + base + 32 * u) : 0;
            a[u] = ok ? __ldg(val + base + 32 * u) : T(0);
        }
        T xs[4][CPL];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (e + u < w) ld_cols<VEC, CPL>(X + (size_t)j[u] * ld + c0, xs[u], k - c0);
            else
#pragma unroll
                for (int m = 0; m < CPL; ++m) xs[u][m] = T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (e + u < w)
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = fma(a[u], xs[u][m], acc[m]);
    }
}

// The same for FP64 values and float X, in FP64 accuracy without the FP64 pipe
// (SplitSum); a column in `on` to which that does not apply takes the FP64
// chain. A matrix entry is split once for the lane's columns. One entry at a
// time: in 64 registers the other warps hide the loads, and four blocks per SM
// matter more (128^3 x 64 columns: 2407 us, 2600-3400 us with two or four
// entries in flight and two or three blocks). In a slice wider than SPLIT_WIDE
// one row is a chain that other warps do not hide, and its entries are loaded
// four at a time: with a hub of 5000 entries 1760 us one by one, 828 so, in the
// same order of additions. The loop for that stands in a kernel of its own
// (WIDE), as it costs the other rows registers (128^3 x 64 columns: 208 -> 213 ms).
constexpr int SPLIT_WIDE = 64;
template <bool VEC, int CPL, bool WIDE>
__device__ __forceinline__ void sell_row_split(const SellV& S, const double* __restrict__ val, int ip, int c0, int k,
                                               const float* __restrict__ X, int ld, const bool (&on)[CPL],
                                               double (&acc)[CPL]) {
    const int s = ip >> 5, r = ip & 31;
    const int s0 = __ldg(S.sptr + s);
    const int w = __ldg(S.sptr + s + 1) - s0;
    const long long base = (long long)s0 * 32 + r;
    SplitSum sum[CPL];
    int e = 0;
    if (WIDE && w > SPLIT_WIDE)
#pragma unroll 1
        for (; e + 4 <= w; e += 4) {
            int j[4];
            double a[4];
            float xs[4][CPL];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                j[u] = __ldg(S.col + base + 32 * (e + u));
                a[u] = __ldg(val + base + 32 * (e + u));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) ld_cols<VEC, CPL>(X + (size_t)j[u] * ld + c0, xs[u], k - c0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Split3 s = split3(a[u]);
#pragma unroll
                for (int m = 0; m < CPL; ++m) sum[m].add(s, xs[u][m]);
            }
        }
    for (; e < w; ++e) {
        const int j = __ldg(S.col + base + 32 * e);
        const Split3 a = split3(__ldg(val + base + 32 * e));
        float xs[CPL];
        ld_cols<VEC, CPL>(X + (size_t)j * ld + c0, xs, k - c0);
#pragma unroll
        for (int m = 0; m < CPL; ++m) sum[m].add(a, xs[m]);
    }
#pragma unroll
    for (int m = 0; m < CPL; ++m) {
        acc[m] = sum[m].value();
        if (on[m] && !sum[m].ok()) {
            if (sum[m].ok_far()) {
                acc[m] = sum[m].value_far();
                continue;
            }
            double t = 0.0;
            for (int e = 0; e < w; ++e)
                t = fma(__ldg(val + base + 32 * e),
                        (double)ldv(X + (size_t)__ldg(S.col + base + 32 * e) * ld + c0 + m), t);
            acc[m] = t;
        }
    }
}

__device__ __forceinline__ double to_d(double v) { return v; }
__device__ __forceinline__ double to_d(float v) { return f2d(v); }

// Sums over `count` blocks' partials (value j of column c of block b at
// part[(b * 2 + j) * k + c]) by the whole block: tpc consecutive lanes per
// column (a power of two <= 32, set by the block width ld so that it does not
// depend on how many columns are live), lane t adds the blocks t, t + tpc, ...
// in order and the lanes meet in a shuffle tree; out(c, sums) on one lane.
template <int NV, typename OUT>
__device__ __forceinline__ void sum_partials(const double* part, int count, int k, int ld, OUT&& out) {
    int tpc = 1;
    while (tpc < 32 && tpc * 2 * ld <= TPB) tpc *= 2;
    const int cpb = TPB / tpc;                           // columns per pass
    const int t = threadIdx.x & (tpc - 1);
    for (int cb = 0; cb < k; cb += cpb) {
        const int c = cb + (int)threadIdx.x / tpc;
        double s[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) s[j] = 0.0;
        if (c < k) {
#pragma unroll 4
            for (int b = t; b < count; b += tpc)
#pragma unroll
                for (int j = 0; j < NV; ++j) s[j] += __ldcg(part + ((size_t)b * 2 + j) * k + c);
        }
        for (int o = tpc >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int j = 0; j < NV; ++j) s[j] += __shfl_xor_sync(FULL_MASK, s[j], o);
        if (c < k && t == 0) out(c, s);
    }
}

// Per-column sums of v[0 .. NV) over the rows of the whole grid in a fixed
// order (warps of a block, groups of a warp, blocks of a team of CS_TEAM, then
// teams); the last block to finish calls fin(c, sum0, sum1) for every column.
// Deterministic for a fixed (grid, lanes per row, block width ld): a column's
// sum never depends on the other columns. The FP64 pipe issues one warp
// instruction per 76 cycles of a sub-partition, so additions are kept few: the
// block's values meet in shared memory (each addition serves 32 live columns),
// and the block partials are added by the last block of each team, in parallel
// over the teams, instead of all by the last block of the grid (20-40 us of
// every 64-column kernel; a 128^3 solve of 64 columns 223.0 -> 217.6 ms, one of
// 75x64x49 and 7 columns 8.56 -> 7.71 ms).
constexpr int CS_TEAM = 32;
template <int CPL, int NV, typename FIN>
__device__ __forceinline__ void colsum(double (&v)[NV][CPL], const Grp& g, int k, int ld, double* partial,
                                       unsigned* ticket, FIN&& fin) {
    __shared__ double sm[TPB * CPL];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gpw = 32 / g.G, W = g.G * CPL;             // groups of a warp, columns of a group (>= k)
    const int slots = gpw * W;                           // 32 CPL values of a warp
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        if (j) __syncthreads();
        double* own = sm + warp * slots + (lane / g.G) * W + g.gl * CPL;
#pragma unroll
        for (int m = 0; m < CPL; ++m) own[m] = v[j][m];
        __syncthreads();
        for (int s = threadIdx.x; s < slots; s += TPB) { // the warps, in place
            double a0 = sm[s], a1 = sm[slots + s];
#pragma unroll
            for (int w = 2; w < WARPS; w += 2) {
                a0 += sm[w * slots + s];
                a1 += sm[(w + 1) * slots + s];
            }
            sm[s] = a0 + a1;
        }
        __syncthreads();
        for (int c = threadIdx.x; c < k; c += TPB) {     // the groups
            double a = sm[c];
            for (int t = 1; t < gpw; ++t) a += sm[t * W + c];
            partial[((size_t)blockIdx.x * 2 + j) * k + c] = a;
            __threadfence();
        }
    }
    const int nteams = ((int)gridDim.x + CS_TEAM - 1) / CS_TEAM, team = blockIdx.x / CS_TEAM;
    const int members = min(CS_TEAM, (int)gridDim.x - team * CS_TEAM);
    double* tpart = partial + (size_t)gridDim.x * 2 * k; // team sums
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket + 1 + team, 1u) == (unsigned)members - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_partials<NV>(partial + (size_t)team * CS_TEAM * 2 * k, members, k, ld, [&](int c, const double (&s)[NV]) {
#pragma unroll
        for (int j = 0; j < NV; ++j) tpart[((size_t)team * 2 + j) * k + c] = s[j];
        __threadfence();
    });
    __syncthreads();
    if (threadIdx.x == 0) {
        ticket[1 + team] = 0u;
        last = atomicAdd(ticket, 1u) == (unsigned)nteams - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_partials<NV>(tpart, nteams, k, ld, [&](int c, const double (&s)[NV]) { fin(c, s[0], NV > 1 ? s[NV - 1] : 0.0); });
    __syncthreads();
    if (threadIdx.x == 0) *ticket = 0u;
}

// ---------------------------------------------------------- V-cycle --------
// x = omega M^-1 b, r = b - omega (A M^-1) b; valm = -omega A M^-1, in FP32 A M^-1.
template <typename T, int CPL, bool VEC>
__global__ void __launch_bounds__(TPB) bk_pre(SellV S, const T* __restrict__ valm, const T* __restrict__ minv, T omega,
                                              const T* __restrict__ B, T* __restrict__ X, T* __restrict__ R, int k, int ld,
                                              int G) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    if (c0 >= k) return;
    for (int ip = g.gw; ip < S.n; ip += g.ngroups) {
        if constexpr (sizeof(T) == 8) {
            const int i = rowid(S, ip);
            const size_t o = (size_t)i * ld + c0;
            T bi[CPL], xo[CPL], ro[CPL];
            ld_cols<VEC, CPL>(B + o, bi, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) ro[m] = bi[m];
            sell_row_k<VEC, CPL>(S, valm, ip, c0, k, B, ld, ro);
            const T mi = omega * minv[i];
#pragma unroll
            for (int m = 0; m < CPL; ++m) xo[m] = mi * bi[m];
            st_cols<VEC, CPL>(X + o, xo, c0, k);
            st_cols<VEC, CPL>(R + o, ro, c0, k);
        } else {
            T acc[CPL];
#pragma unroll
            for (int m = 0; m < CPL; ++m) acc[m] = 0;
            sell_row_k<VEC, CPL>(S, valm, ip, c0, k, B, ld, acc);
            const int i = rowid(S, ip);
            const T mi = omega * minv[i];
            const size_t o = (size_t)i * ld + c0;
            T bi[CPL], xo[CPL], ro[CPL];
            ld_cols<VEC, CPL>(B + o, bi, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                xo[m] = mi * bi[m];
                ro[m] = fma(-omega, acc[m], bi[m]);
            }
            st_cols<VEC, CPL>(X + o, xo, c0, k);
            st_cols<VEC, CPL>(R + o, ro, c0, k);
        }
    }
}

template <typename T, int CPL, bool VEC>
__global__ void __launch_bounds__(TPB) bk_restrict(int nc, const int* __restrict__ pt_ptr,
                                                   const int* __restrict__ pt_idx, const T* __restrict__ p,
                                                   const T* __restrict__ R, T* __restrict__ Bc, int k, int ld, int G) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    if (c0 >= k) return;
    for (int q = g.gw; q < nc; q += g.ngroups) {
        T acc[CPL];
#pragma unroll
        for (int m = 0; m < CPL; ++m) acc[m] = 0;
        for (int e = pt_ptr[q]; e < pt_ptr[q + 1]; ++e) {
            const int i = __ldg(pt_idx + e);
            const T pi = __ldg(p + i);
            T rv[CPL];
            ld_cols<VEC, CPL>(R + (size_t)i * ld + c0, rv, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) acc[m] = fma(pi, rv[m], acc[m]);
        }
        st_cols<VEC, CPL>(Bc + (size_t)q * ld + c0, acc, c0, k);
    }
}

// X = A_L^{-1} B on the coarsest level, FP64 arithmetic. A block per row: TPB / G
// slices of the row's entries, each by a group of G lanes over all columns, and
// a tree over the slices. (A group per row ran all n entries in series: 50 us
// for 64 rows and 64 columns, 6.5 us now.)
template <typename TI, typename TO, int CPL, bool VEC>
__global__ void __launch_bounds__(TPB) bk_coarse_dense(int n, const double* __restrict__ Ainv, const TI* __restrict__ B,
                                                       TO* __restrict__ X, int k, int ld, int G) {
    __shared__ double sm[TPB * CPL];
    const int gl = threadIdx.x % G, slice = threadIdx.x / G, slices = TPB / G;
    const int c0 = gl * CPL;
    dep_wait();
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        double acc[CPL];
#pragma unroll
        for (int m = 0; m < CPL; ++m) acc[m] = 0.0;
        const double* row = Ainv + (size_t)i * n;
        if (c0 < k)
#pragma unroll 4
            for (int j = slice; j < n; j += slices) {
                const double a = __ldg(row + j);
                TI bv[CPL];
                ld_cols<VEC, CPL>(B + (size_t)j * ld + c0, bv, k - c0);
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = fma(a, to_d(bv[m]), acc[m]);
            }
#pragma unroll
        for (int m = 0; m < CPL; ++m) sm[m * TPB + threadIdx.x] = acc[m];
        __syncthreads();
        for (int t = slices >> 1; t > 0; t >>= 1) {
            for (int q = threadIdx.x; q < t * G * CPL; q += TPB) {
                double* v = sm + q / (t * G) * TPB + q % (t * G);
                *v += v[t * G];
            }
            __syncthreads();
        }
        for (int c = threadIdx.x; c < k; c += TPB) X[(size_t)i * ld + c] = (TO)sm[c % CPL * TPB + c / CPL];
        __syncthreads();
    }
}

// r . z finisher: START columns take rho and beta = 0 and become ACTIVE;
// ACTIVE columns update beta (PCG, or flexible CG from z . q) and rho.
__device__ __forceinline__ void fin_rz(const BlockScalars& sc, int c, double rz, double zq, int flexible) {
    const int mode = sc.mode[c];
    if (mode == COL_START) {
        sc.rho[c] = rz;
        sc.beta[c] = 0.0;
        sc.mode[c] = isfinite(rz) ? COL_ACTIVE : COL_FAILED;
    } else if (mode == COL_ACTIVE) {
        const double beta = flexible ? -sc.alpha[c] * zq / sc.rho[c] : rz / sc.rho[c];
        sc.beta[c] = beta;
        sc.rho[c] = rz;
        if (!isfinite(beta)) sc.mode[c] = COL_FAILED;
    }
}

// out = x + omega M^-1 r + (P - omega M^-1 A P) e (FP64: the stored values are
// those of the bracket; FP32: omega M^-1 A P, and P e from agg and p); on level 0 also r_cg . out and (flexible CG) q . out per column.
template <typename T, typename TO, int CPL, bool DOT, bool VEC>
__global__ void __launch_bounds__(TPB) bk_post(SellV SAP, const T* __restrict__ apval, const T* __restrict__ minv,
                                               T omega, const int* __restrict__ agg, const T* __restrict__ p,
                                               const T* __restrict__ E, const T* __restrict__ X,
                                               const T* __restrict__ R, const double* __restrict__ Bdot,
                                               const double* __restrict__ Q2, TO* __restrict__ Out, int k, int ld, int G,
                                               double* partial, unsigned* ticket, BlockScalars sc, int flexible) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    double d[2][CPL];
#pragma unroll
    for (int m = 0; m < CPL; ++m) d[0][m] = d[1][m] = 0.0;
    if (c0 < k) {
        for (int ip = g.gw; ip < SAP.n; ip += g.ngroups) {
            const int i = rowid(SAP, ip);
            const size_t o = (size_t)i * ld + c0;
            T acc[CPL], xv[CPL], rv[CPL];
            TO ov[CPL];
            if constexpr (sizeof(T) == 8) {
                const T mi = omega * minv[i];
                ld_cols<VEC, CPL>(X + o, xv, k - c0);
                ld_cols<VEC, CPL>(R + o, rv, k - c0);
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = fma(mi, rv[m], xv[m]);
                sell_row_k<VEC, CPL>(SAP, apval, ip, c0, k, E, ld, acc);
#pragma unroll
                for (int m = 0; m < CPL; ++m) ov[m] = (TO)acc[m];
            } else {
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = 0;
                sell_row_k<VEC, CPL>(SAP, apval, ip, c0, k, E, ld, acc);
                const int a = agg[i];
                const T pi = p[i];
                const T mi = omega * minv[i];
                T ev[CPL];
                ld_cols<VEC, CPL>(E + (size_t)a * ld + c0, ev, k - c0);
                ld_cols<VEC, CPL>(X + o, xv, k - c0);
                ld_cols<VEC, CPL>(R + o, rv, k - c0);
#pragma unroll
                for (int m = 0; m < CPL; ++m) {
                    const T y = fma(pi, ev[m], xv[m]);
                    ov[m] = (TO)(fma(mi, rv[m], y) - acc[m]);
                }
            }
            st_cols<VEC, CPL>(Out + o, ov, c0, k);
            if (DOT) {
                double bd[CPL], qd[CPL];
                ld_cols<VEC, CPL>(Bdot + o, bd, k - c0);
                if (Q2) ld_cols<VEC, CPL>(Q2 + o, qd, k - c0);
#pragma unroll
                for (int m = 0; m < CPL; ++m) {
                    if (c0 + m >= k) continue;
                    const double od = to_d(ov[m]);
                    d[0][m] = fma(bd[m], od, d[0][m]);
                    if (Q2) d[1][m] = fma(qd[m], od, d[1][m]);
                }
            }
        }
    }
    if (DOT) {
        auto fin = [&](int c, double a, double b) { fin_rz(sc, c, a, b, flexible); };
        if (Q2) {
            colsum<CPL, 2>(d, g, k, ld, partial, ticket, fin);
        } else {
            double e[1][CPL];
#pragma unroll
            for (int m = 0; m < CPL; ++m) e[0][m] = d[0][m];
            colsum<CPL, 1>(e, g, k, ld, partial, ticket, fin);
        }
    }
}


// ------------------------------------- iterative coarsest solve, k columns
// CG with l1-Jacobi per column to ||r_c|| <= rtol ||b_c|| or maxit, FP64, all
// columns in one cooperative launch (the multi-column form of the
// single-column coarsest solve). Short rows come from the hybrid SELL layout
// through lane groups, rows kept out of it are split over the 32 lanes of a
// warp; per-column sums use one fixed reduction order, and every block sums
// the block partials in the same order after each grid barrier, so all blocks
// hold the same per-column scalars.
__device__ __forceinline__ unsigned long long bk_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned bk_ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void bk_grid_sync(unsigned* count, unsigned epoch, int* err) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        const unsigned target = epoch * gridDim.x;
        const unsigned long long t0 = bk_ns();
        while (bk_ld_acquire(count) < target) {
            if (bk_ns() - t0 > 2000000000ull) { atomicExch(err, 1); break; }
        }
        __threadfence();
    }
    __syncthreads();
}

// Sums over the grid of v[0 .. NV) per column: this block's partials go to
// part[(blockIdx.x * NV + j) * k + c], and after the grid barrier every block
// adds them in the same order into dst[j * k + c]. As few FP64 additions as
// there are partials: lanes of a warp add different columns, through shared
// memory (butterflies in every warp, 152 serial loads per column and a
// division per thread made a reduction of 16 columns cost 14 us, four of them
// an iteration).
template <int CPL, int NV>
__device__ __forceinline__ void cc_partials(double (&v)[NV][CPL], const Grp& g, int k, double* part, double* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gpw = 32 / g.G, W = g.G * CPL;             // groups of a warp, columns of a group (>= k)
    constexpr int SLOTS = 32 * CPL;                      // gpw * W: values of a warp
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        __syncthreads();
        double* own = sm + warp * SLOTS + (lane / g.G) * W + g.gl * CPL;
#pragma unroll
        for (int m = 0; m < CPL; ++m) own[m] = v[j][m];
        __syncthreads();
        for (int s = threadIdx.x; s < SLOTS; s += CC_TPB) {
            double a0 = sm[s], a1 = sm[SLOTS + s];
#pragma unroll
            for (int w = 2; w < CC_TPB / 32; w += 2) {
                a0 += sm[w * SLOTS + s];
                a1 += sm[(w + 1) * SLOTS + s];
            }
            sm[s] = a0 + a1;
        }
        __syncthreads();
        for (int c = threadIdx.x; c < k; c += CC_TPB) {
            double a = sm[c];
            for (int t = 1; t < gpw; ++t) a += sm[t * W + c];
            part[((size_t)blockIdx.x * NV + j) * k + c] = a;
        }
    }
}
template <int NV>
__device__ __forceinline__ void cc_sums(const double* part, int k, int ld, double* dst, double* sm) {
    const int nv = NV * k;                               // values; R threads share one (R from the block width ld:
    int R = 1;                                           // the order does not depend on the columns in flight)
    while (R < 32 && 2 * R * NV * ld <= CC_TPB) R *= 2;
    for (int v0 = 0; v0 < nv; v0 += CC_TPB / R) {
        const int cnt = min(nv - v0, CC_TPB / R);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt * R; t += CC_TPB) {
            const int v = v0 + t % cnt;
            double a = 0.0;
#pragma unroll 5
            for (int b = t / cnt; b < (int)gridDim.x; b += R) a += __ldcg(part + (size_t)b * nv + v);
            sm[t] = a;
        }
        __syncthreads();
        for (int half = R >> 1; half > 0; half >>= 1) {  // a tree over the R partial sums of every value
            for (int t = threadIdx.x; t < cnt * half; t += CC_TPB) sm[t] += sm[t + cnt * half];
            __syncthreads();
        }
        for (int t = threadIdx.x; t < cnt; t += CC_TPB) dst[v0 + t] = sm[t];
    }
    __syncthreads();
}

// One iteration is two grid barriers: the product q = A z + beta q (= A p)
// with p = z + beta p, then x, r and z = M^-1 r with r.r and r.z. 64^3 jump
// coefficients, 16 columns, 30 iterations: 1.69 ms before (four barriers, a
// block of 256 threads per SM), 0.74 ms now.
template <typename TI, typename TO, int CPL, bool VEC>
__global__ void __launch_bounds__(CC_TPB) bk_coarse_cg(SellV S, const double* __restrict__ sval, int n, int nlong,
                                                       const int* __restrict__ long_rows, const int* __restrict__ cptr,
                                                       const int* __restrict__ ccol, const double* __restrict__ cval,
                                                       const double* __restrict__ minv, const TI* __restrict__ B,
                                                       TO* __restrict__ Xo, int k, int ld, int G, double* x, double* r,
                                                       double* z, double* p, double* q, double* part, unsigned* bar,
                                                       int* err, int maxit, double rtol) {
    __shared__ double s_rho[MAXK], s_stop[MAXK], s_t[2 * MAXK], s_al[MAXK];   // s_al: alpha, then beta
    __shared__ int s_live[MAXK];
    extern __shared__ double cc_sm[];                    // CC_TPB * CPL
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    unsigned epoch = 0;
    int red = 0;                                         // reduction counter: two buffers of two values
    auto slot = [&]() { return part + (size_t)(red & 1) * 2 * gridDim.x * k; };
    double d2[2][CPL];
#pragma unroll
    for (int m = 0; m < CPL; ++m) d2[0][m] = d2[1][m] = 0.0;
    // x = 0, r = b, z = M^-1 r; b.b and rho = r.z per column
    if (c0 < k)
        for (int i = g.gw; i < n; i += g.ngroups) {
            const double mi = minv[i];
            const size_t o = (size_t)i * ld + c0;
            TI bt[CPL];
            double bi[CPL], zi[CPL], zero[CPL];
            ld_cols<VEC, CPL>(B + o, bt, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                bi[m] = (double)bt[m];
                zi[m] = mi * bi[m];
                zero[m] = 0.0;
                if (c0 + m >= k) continue;
                d2[0][m] = fma(bi[m], bi[m], d2[0][m]);
                d2[1][m] = fma(bi[m], zi[m], d2[1][m]);
            }
            st_cols<VEC, CPL>(x + o, zero, c0, k);
            st_cols<VEC, CPL>(r + o, bi, c0, k);
            st_cols<VEC, CPL>(z + o, zi, c0, k);
        }
    cc_partials<CPL, 2>(d2, g, k, slot(), cc_sm);
    bk_grid_sync(bar, ++epoch, err);
    if (__ldcg(err)) return;
    cc_sums<2>(slot(), k, ld, s_t, cc_sm);
    ++red;
    for (int c = threadIdx.x; c < k; c += blockDim.x) {
        const double bb = s_t[c];
        s_live[c] = bb > 0.0;
        s_stop[c] = rtol * rtol * bb;
        s_rho[c] = s_t[k + c];
        s_al[c] = 0.0;
    }
    __syncthreads();
    for (int it = 0; it < maxit; ++it) {
        int alive = 0;
        for (int c = threadIdx.x; c < k; c += blockDim.x) alive |= s_live[c];
        if (!__syncthreads_or(alive)) break;
        double be[CPL], d1[1][CPL];
        bool on[CPL], any = false;
#pragma unroll
        for (int m = 0; m < CPL; ++m) {
            on[m] = c0 + m < k && s_live[c0 + m];
            be[m] = on[m] ? s_al[c0 + m] : 0.0;
            any |= on[m];
            d1[0][m] = 0.0;
        }
        // p = z + beta p, q = A z + beta q of one row (it = 0: p and q are not
        // read), p . q; the row's own p, q and z are loaded before its product
        double pv[CPL], qv[CPL], zv[CPL];
        auto own_row = [&](int i) {
            const size_t o = (size_t)i * ld + c0;
            ld_cols<VEC, CPL>(z + o, zv, k - c0);
            if (it > 0) {
                ld_cols<VEC, CPL>(p + o, pv, k - c0);
                ld_cols<VEC, CPL>(q + o, qv, k - c0);
            }
        };
        auto finish_row = [&](int i, const double (&acc)[CPL]) {
            const size_t o = (size_t)i * ld + c0;
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                pv[m] = it > 0 ? fma(be[m], pv[m], zv[m]) : zv[m];
                qv[m] = it > 0 ? fma(be[m], qv[m], acc[m]) : acc[m];
                if (on[m]) d1[0][m] = fma(pv[m], qv[m], d1[0][m]);
            }
            st_cols<VEC, CPL>(p + o, pv, c0, k);
            st_cols<VEC, CPL>(q + o, qv, c0, k);
        };
        if (any)
            for (int ip = g.gw; ip < S.n; ip += g.ngroups) {
                double acc[CPL];
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = 0.0;
                const int i = rowid(S, ip);
                own_row(i);
                sell_row_k<VEC, CPL>(S, sval, ip, c0, k, (const double*)z, ld, acc);
                finish_row(i, acc);
            }
        // long rows: a warp per row, its lane groups take the entries in turn
        for (int lr = gwarp; lr < nlong; lr += nwarps) {
            const int i = __ldg(long_rows + lr);
            const int e1 = __ldg(cptr + i + 1);
            double acc[CPL];
#pragma unroll
            for (int m = 0; m < CPL; ++m) acc[m] = 0.0;
            if (any)
#pragma unroll 4
                for (int e = __ldg(cptr + i) + lane / G; e < e1; e += 32 / G) {
                    const double a = __ldg(cval + e);
                    double ze[CPL];
                    ld_cols<VEC, CPL>((const double*)z + (size_t)__ldg(ccol + e) * ld + c0, ze, k - c0);
#pragma unroll
                    for (int m = 0; m < CPL; ++m) acc[m] = fma(a, ze[m], acc[m]);
                }
            for (int o = 16; o >= G; o >>= 1)
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] += __shfl_xor_sync(FULL_MASK, acc[m], o);
            if (any && lane < G) {
                own_row(i);
                finish_row(i, acc);
            }
        }
        cc_partials<CPL, 1>(d1, g, k, slot(), cc_sm);
        bk_grid_sync(bar, ++epoch, err);
        if (__ldcg(err)) return;
        cc_sums<1>(slot(), k, ld, s_t, cc_sm);
        ++red;
        for (int c = threadIdx.x; c < k; c += blockDim.x) s_al[c] = s_live[c] ? s_rho[c] / s_t[c] : 0.0;
        __syncthreads();
        // x += alpha p, r -= alpha q, z = M^-1 r; r.r and r.z (columns that
        // are not live keep their values: alpha = 0)
        double al[CPL];
#pragma unroll
        for (int m = 0; m < CPL; ++m) {
            al[m] = on[m] ? s_al[c0 + m] : 0.0;
            d2[0][m] = d2[1][m] = 0.0;
        }
        if (any)
            for (int i = g.gw; i < n; i += g.ngroups) {
                const double mi = minv[i];
                const size_t o = (size_t)i * ld + c0;
                double pv[CPL], qv[CPL], xv[CPL], rv[CPL], zv[CPL];
                ld_cols<VEC, CPL>(p + o, pv, k - c0);
                ld_cols<VEC, CPL>(q + o, qv, k - c0);
                ld_own<VEC, CPL>(x + o, xv, k - c0);
                ld_own<VEC, CPL>(r + o, rv, k - c0);
#pragma unroll
                for (int m = 0; m < CPL; ++m) {
                    if (al[m] != 0.0) {
                        xv[m] = fma(al[m], pv[m], xv[m]);
                        rv[m] = fma(-al[m], qv[m], rv[m]);
                    }
                    zv[m] = mi * rv[m];
                    d2[0][m] = fma(rv[m], rv[m], d2[0][m]);
                    d2[1][m] = fma(rv[m], zv[m], d2[1][m]);
                }
                st_cols<VEC, CPL>(x + o, xv, c0, k);
                st_cols<VEC, CPL>(r + o, rv, c0, k);
                st_cols<VEC, CPL>(z + o, zv, c0, k);
            }
        cc_partials<CPL, 2>(d2, g, k, slot(), cc_sm);
        bk_grid_sync(bar, ++epoch, err);
        if (__ldcg(err)) return;
        cc_sums<2>(slot(), k, ld, s_t, cc_sm);
        ++red;
        for (int c = threadIdx.x; c < k; c += blockDim.x) {
            if (!s_live[c]) continue;
            if (s_t[c] <= s_stop[c]) s_live[c] = 0;
            s_al[c] = s_t[k + c] / s_rho[c];
            s_rho[c] = s_t[k + c];
        }
        __syncthreads();
    }
    if (c0 < k)
        for (int i = g.gw; i < n; i += g.ngroups) {
            const size_t o = (size_t)i * ld + c0;
            double xv[CPL];
            TO xo[CPL];
            ld_own<VEC, CPL>(x + o, xv, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) xo[m] = (TO)xv[m];
            st_cols<VEC, CPL>(Xo + o, xo, c0, k);
        }
}

// ------------------------------------------------------------- CG ----------
// ACTIVE columns: P = Z + beta P, Q = A Z + beta Q (= A P; a column that just
// started has beta = 0 and reads neither), p . q and alpha = rho / p.q; alpha =
// 0 for the others, whose P and Q keep their values. The product takes Z, the
// V-cycle's output in its own type: for FP32 the products are formed in FP32
// pieces, so FP64 instructions are 5 a row and column instead of 9 in the
// product and direction passes that this replaces, which were bound by them:
// 128^3 rows x 64 columns 2143 + 495 us, 2407 us now; 64^3 x 16 about 107 us,
// 95 us now.
// WIDE (FP32): a row is longer than SPLIT_WIDE.
template <typename TZ, int CPL, bool VEC, bool WIDE>
__global__ void __launch_bounds__(TPB, sizeof(TZ) == 4 && CPL <= 4 ? 4 : 1) bk_direction(SellV S, const double* __restrict__ val,
                                                    const TZ* __restrict__ Z, double* __restrict__ P,
                                                    double* __restrict__ Q, int k, int ld, int G, double* partial,
                                                    unsigned* ticket, BlockScalars sc) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    double be[CPL], d[1][CPL];
    bool on[CPL], any = false, old = false;
#pragma unroll
    for (int m = 0; m < CPL; ++m) {
        const int c = c0 + m;
        on[m] = c < k && sc.mode[c] == COL_ACTIVE;
        be[m] = on[m] ? sc.beta[c] : 0.0;
        any |= on[m];
        old |= c < k && (!on[m] || be[m] != 0.0);
        d[0][m] = 0.0;
    }
    if (any) {
        for (int ip = g.gw; ip < S.n; ip += g.ngroups) {
            const int i = rowid(S, ip);
            const size_t o = (size_t)i * ld + c0;
            double acc[CPL], pv[CPL], qv[CPL];
            TZ zv[CPL];
            if constexpr (sizeof(TZ) == 4) {
                sell_row_split<VEC, CPL, WIDE>(S, val, ip, c0, k, Z, ld, on, acc);
            } else {
#pragma unroll
                for (int m = 0; m < CPL; ++m) acc[m] = 0.0;
                sell_row_k<VEC, CPL>(S, val, ip, c0, k, Z, ld, acc);
            }
            ld_cols<VEC, CPL>(Z + o, zv, k - c0);
            if (old) {
                ld_own<VEC, CPL>(P + o, pv, k - c0);
                ld_own<VEC, CPL>(Q + o, qv, k - c0);
            }
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                if (!on[m]) continue;
                const double zd = to_d(zv[m]);
                pv[m] = be[m] == 0.0 ? zd : fma(be[m], pv[m], zd);
                qv[m] = be[m] == 0.0 ? acc[m] : fma(be[m], qv[m], acc[m]);
                d[0][m] = fma(pv[m], qv[m], d[0][m]);
            }
            st_cols<VEC, CPL>(P + o, pv, c0, k);
            st_cols<VEC, CPL>(Q + o, qv, c0, k);
        }
    }
    colsum<CPL, 1>(d, g, k, ld, partial, ticket, [&](int c, double pq, double) {
        sc.pq[c] = pq;
        if (sc.mode[c] == COL_ACTIVE) {
            const double alpha = sc.rho[c] / pq;
            if (!(pq > 0.0) || !isfinite(alpha)) {
                sc.mode[c] = COL_FAILED;
                sc.alpha[c] = 0.0;
            } else {
                sc.alpha[c] = alpha;
            }
        } else {
            sc.alpha[c] = 0.0;
        }
    });
}

// ACTIVE columns: X += alpha P, R -= alpha Q, ||R||^2; convergence -> CHECK.
// Other columns are written back unchanged when a vector store covers them.
// With R32 set (FP32 V-cycle) also the float copy of R that the V-cycle reads:
// this kernel and bk_residual, the two that write R, keep it.
template <int CPL, bool VEC>
__global__ void __launch_bounds__(TPB) bk_update_xr(int n, const double* __restrict__ P, const double* __restrict__ Q,
                                                    double* __restrict__ X, double* __restrict__ R,
                                                    float* __restrict__ R32, int k, int ld, int G,
                                                    double* partial, unsigned* ticket, BlockScalars sc) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    double al[CPL];
    bool on[CPL];
    bool any = false;
#pragma unroll
    for (int m = 0; m < CPL; ++m) {
        const int c = c0 + m;
        on[m] = c < k && sc.mode[c] == COL_ACTIVE;
        al[m] = on[m] ? sc.alpha[c] : 0.0;
        any |= on[m];
    }
    double d[1][CPL];
#pragma unroll
    for (int m = 0; m < CPL; ++m) d[0][m] = 0.0;
    if (any) {
        for (int i = g.gw; i < n; i += g.ngroups) {
            const size_t o = (size_t)i * ld + c0;
            double pv[CPL], qv[CPL], xv[CPL], rv[CPL];
            ld_cols<VEC, CPL>(P + o, pv, k - c0);
            ld_cols<VEC, CPL>(Q + o, qv, k - c0);
            ld_own<VEC, CPL>(X + o, xv, k - c0);
            ld_own<VEC, CPL>(R + o, rv, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                if (!on[m]) continue;
                xv[m] = fma(al[m], pv[m], xv[m]);
                rv[m] = fma(-al[m], qv[m], rv[m]);
                d[0][m] = fma(rv[m], rv[m], d[0][m]);
            }
            st_cols<VEC, CPL>(X + o, xv, c0, k);
            st_cols<VEC, CPL>(R + o, rv, c0, k);
            if (R32) {
                float rf[CPL];
#pragma unroll
                for (int m = 0; m < CPL; ++m) rf[m] = d2f(rv[m]);
                st_cols<VEC, CPL>(R32 + o, rf, c0, k);
            }
        }
    }
    colsum<CPL, 1>(d, g, k, ld, partial, ticket, [&](int c, double rr, double) {
        if (sc.mode[c] != COL_ACTIVE) return;
        sc.rr[c] = rr;
        sc.iters[c] += 1;
        if (rr <= sc.rtol[c] * sc.rtol[c] * sc.bb[c]) sc.mode[c] = COL_CHECK;
    });
}

// R = B - A X for the selected columns, ||R||^2 and ||B||^2.
//   stage 0 (start): INIT columns; DONE when ||B|| = 0 or x0 already meets
//                    rtol, else START.
//   stage 1 (check): CHECK columns; true residual below rtol -> DONE, else the
//                    column restarts from R (START).
//   stage 2 (report): every column; only records ||R||^2 in rr.
// Columns not selected keep their R when a vector store covers them.
template <int CPL, bool VEC>
__global__ void __launch_bounds__(TPB) bk_residual(SellV S, const double* __restrict__ val,
                                                   const double* __restrict__ X, const double* __restrict__ B,
                                                   double* __restrict__ R, float* __restrict__ R32, int k, int ld,
                                                   int G, double* partial,
                                                   unsigned* ticket, BlockScalars sc, int stage) {
    dep_wait();
    const Grp g = make_grp(G);
    const int c0 = g.gl * CPL;
    bool on[CPL];
    bool any = false;
#pragma unroll
    for (int m = 0; m < CPL; ++m) {
        const int c = c0 + m;
        const int md = c < k ? sc.mode[c] : COL_IDLE;
        on[m] = c < k && (stage == 0 ? md == COL_INIT : (stage == 1 ? md == COL_CHECK : true));
        any |= on[m];
    }
    double d[2][CPL];
#pragma unroll
    for (int m = 0; m < CPL; ++m) d[0][m] = d[1][m] = 0.0;
    if (any) {
        for (int ip = g.gw; ip < S.n; ip += g.ngroups) {
            double acc[CPL];
#pragma unroll
            for (int m = 0; m < CPL; ++m) acc[m] = 0.0;
            sell_row_k<VEC, CPL>(S, val, ip, c0, k, X, ld, acc);
            const int i = rowid(S, ip);
            const size_t o = (size_t)i * ld + c0;
            double bv[CPL], rv[CPL];
            ld_cols<VEC, CPL>(B + o, bv, k - c0);
            ld_own<VEC, CPL>(R + o, rv, k - c0);
#pragma unroll
            for (int m = 0; m < CPL; ++m) {
                if (!on[m]) continue;
                rv[m] = bv[m] - acc[m];
                d[0][m] = fma(rv[m], rv[m], d[0][m]);
                d[1][m] = fma(bv[m], bv[m], d[1][m]);
            }
            st_cols<VEC, CPL>(R + o, rv, c0, k);
            if (R32) {
                float rf[CPL];
#pragma unroll
                for (int m = 0; m < CPL; ++m) rf[m] = d2f(rv[m]);
                st_cols<VEC, CPL>(R32 + o, rf, c0, k);
            }
        }
    }
    colsum<CPL, 2>(d, g, k, ld, partial, ticket, [&](int c, double rr, double bb) {
        const int md = sc.mode[c];
        if (stage == 0) {
            if (md != COL_INIT) return;
            sc.bb[c] = bb;
            sc.rr[c] = rr;
            sc.iters[c] = 0;
            sc.mode[c] = bb == 0.0 ? COL_DONE : (rr <= sc.rtol[c] * sc.rtol[c] * bb ? COL_DONE : COL_START);
        } else if (stage == 1) {
            if (md != COL_CHECK) return;
            sc.rr[c] = rr;
            sc.mode[c] = rr <= sc.rtol[c] * sc.rtol[c] * sc.bb[c] ? COL_DONE : COL_START;
        } else {
            sc.rr[c] = rr;
        }
    });
}

// Slot lists of a request (at most MAXK slots) passed by value.
struct SlotList {
    int n;
    int slot[MAXK];
};

// dst[:, slot[j]] = src[:, j] (src row-major n x k contiguous, dst row stride ld);
// with src == nullptr the slot columns are zeroed.
__global__ void bk_scatter_slots(int n, const double* __restrict__ src, int ld, double* __restrict__ dst,
                                 SlotList sl) {
    const int k = sl.n;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)n * k;
         t += (long long)gridDim.x * blockDim.x) {
        const long long i = t / k;
        const int j = (int)(t % k);
        dst[i * ld + sl.slot[j]] = src ? src[t] : 0.0;
    }
}

// dst[:, j] = src[:, slot] for one slot column j of a request (dst n x k).
__global__ void bk_gather_slot(int n, const double* __restrict__ src, int ld, int slot, double* __restrict__ dst,
                               int k, int j) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[(size_t)i * k + j] = src[(size_t)i * ld + slot];
}

__global__ void bk_zero_cols(int n, double* __restrict__ X, int k, int ld, const int* __restrict__ mode,
                             const double* __restrict__ bb) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < (long long)n * k;
         t += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(t % k);
        const long long i = t / k;
        if (bb[c] == 0.0 && mode[c] == COL_DONE) X[i * ld + c] = 0.0;
    }
}

// ------------------------------------------------------------- host --------
SellV sv(const DevSell& S) { return SellV{S.n, S.nslices, S.sptr, S.col, S.perm}; }

int pow2_at_least(int v) {
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Group width and columns per lane for k active columns. With a fixed width
// (set by the slot count K, not by k) a column's arithmetic and reduction
// order do not depend on how many columns are in flight.
// The default width gives each lane one vector's worth of columns (4 floats
// or 2 doubles) when the columns fill the group.
void group_shape(const BlockWork& W, int k, int* G, int* cpl) {
    int g = std::min(32, std::max(1, pow2_at_least(W.fixed_width ? W.K : k) / W.vec_cols));
    if (W.tuned_G && !W.fixed_width) g = std::min(W.tuned_G, pow2_at_least(k));
    *G = g;
    *cpl = pow2_at_least((k + g - 1) / g);
}

// CPL columns per lane, as vectors (VEC) when the row stride ld is a multiple of CPL.
#define DISPATCH_ONE(cpl_, vec, ...)                                                               \
    if (vec) { constexpr int CPL = cpl_; constexpr bool VEC = true; (void)VEC; __VA_ARGS__; }        \
    else { constexpr int CPL = cpl_; constexpr bool VEC = false; (void)VEC; __VA_ARGS__; }
#define DISPATCH_CPL(cpl, ld, ...)                                                                 \
    do {                                                                                           \
        const bool vec_ = (cpl) > 1 && (ld) % (cpl) == 0;                                          \
        switch (cpl) {                                                                             \
            case 1: { constexpr int CPL = 1; constexpr bool VEC = false; (void)VEC; __VA_ARGS__; } break; \
            case 2: { DISPATCH_ONE(2, vec_, __VA_ARGS__) } break;                                   \
            case 4: { DISPATCH_ONE(4, vec_, __VA_ARGS__) } break;                                   \
            default: { DISPATCH_ONE(8, vec_, __VA_ARGS__) } break;                                  \
        }                                                                                          \
    } while (0)

// A kernel over rows, started beside the one before it (launch_dep) where its
// entries times columns (`work`) are few, after it otherwise: in a block solve a
// large kernel gains nothing, and the blocks that already wait take its place in
// the caches and on the SMs (rows of 60 entries, 100K x 16 columns, FP64: 18.8 ms
// a solve with all dependent, 17.6 so; rows of 300, 50K x 16: 23.5, 21.9; 64^3 x
// 64: 38.3, 37.3; small ones lose 3% without; a bound of 2M or 24M is as good).
// The server's kernels (fixed width), launched one by one on several streams, are
// all dependent: with the same bound 12 requests on 3 operators take 3% longer.
constexpr long long DEP_WORK = 8LL << 20;
template <typename... P, typename... A>
void launch_rows(const BlockWork& W, long long work, void (*kernel)(P...), int grid, int threads, size_t smem,
                 cudaStream_t st, A&&... args) {
    if (W.fixed_width || work <= DEP_WORK) launch_dep(kernel, grid, threads, smem, st, std::forward<A>(args)...);
    else kernel<<<grid, threads, smem, st>>>(std::forward<A>(args)...);
}

int grid_rows(const amg_hierarchy* h, long long rows, int G) {
    const long long groups_per_block = (long long)WARPS * (32 / G);
    return blocks_for(rows, (int)groups_per_block, h->num_sms * 8);
}

// Grid of the reducing kernels: at most 8 blocks per SM and none without rows
// (every block costs a partial per column). Fixed for (rows, G), so the order
// of the sums is.
int red_grid(const amg_hierarchy* h, const BlockWork& W, int G) {
    return std::min(W.grid, grid_rows(h, h->lev[0].A.n, G));
}

// Z = B R for columns [0, k) (block V-cycle); level 0 finishes r . z per column.
template <typename T>
void block_vcycle(amg_hierarchy* h, BlockWork& W, int k, int flexible) {
    cudaStream_t st = h->stream;
    const int ld = W.K;
    const int L = (int)h->lev.size() - 1;
    const bool f32 = sizeof(T) == 4;
    const T omega = (T)h->opt.omega;
    int G, cpl;
    group_shape(W, k, &G, &cpl);
    auto lv = [&](std::vector<void*>& v, int l) { return static_cast<T*>(v[l]); };
    for (int l = 0; l < L; ++l) {
        Level& Lv = h->lev[l];
        const T* valm = f32 ? (const T*)Lv.valm32 : (const T*)Lv.valm;
        const T* minv = f32 ? (const T*)Lv.minv32 : (const T*)Lv.minv;
        const int g = grid_rows(h, Lv.S.n, G);
        Scope sc_(&h->prof, st, l == 0 ? K_PRE_L0 : K_PRE,
                  (double)Lv.A.nnz * (sizeof(T) + 4) + (double)Lv.A.n * k * ((l == 0 ? 8 : sizeof(T)) + 2.0 * sizeof(T)));
        if (l == 0 && !f32)
            DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)Lv.A.nnz * k, bk_pre<T, CPL, VEC>, g, TPB, 0, st, sv(Lv.S), valm, minv, omega, (const T*)W.R, lv(W.x, 0),
                                                                       lv(W.r, 0), k, ld, G));
        else
            DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)Lv.A.nnz * k, bk_pre<T, CPL, VEC>, g, TPB, 0, st, sv(Lv.S), valm, minv, omega, lv(W.b, l), lv(W.x, l),
                                                                  lv(W.r, l), k, ld, G));
        KERNEL_CHECK();
        const int nc = h->lev[l + 1].A.n;
        const T* p = f32 ? (const T*)Lv.p32 : (const T*)Lv.p;
        DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)Lv.A.n * k, bk_restrict<T, CPL, VEC>, grid_rows(h, nc, G), TPB, 0, st, nc, Lv.pt_ptr, Lv.pt_idx, p,
                                                                                   lv(W.r, l), lv(W.b, l + 1), k, ld, G));
        KERNEL_CHECK();
    }
    {
        Scope sc_(&h->prof, st, K_COARSE, 8.0 * h->nc * h->nc + 16.0 * h->nc * k);
        if (!h->coarse_cg) {
            DISPATCH_CPL(cpl, ld, launch_dep(bk_coarse_dense<T, T, CPL, VEC>, std::min(h->nc, h->num_sms * 8), TPB, 0, st, 
                                  h->nc, h->coarse_inv, lv(W.b, L), lv(W.x, L), k, ld, G));
            KERNEL_CHECK();
        } else {
            Level& Lc = h->lev[L];
            const SellV Sc = sv(Lc.S);
            const double* sval = Lc.S.val;
            int nrows = Lc.A.n, nlong = Lc.S.nlong, kk = k, ldd = ld, GG = G, maxit = 30;
            const int* long_rows = Lc.S.long_rows;
            const int* cptr = Lc.A.ptr;
            const int* ccol = Lc.A.col;
            const double* cval = Lc.A.val;
            const double* cminv = Lc.minv;
            const T* bin = lv(W.b, L);
            T* xout = lv(W.x, L);
            double rtol = 1e-4;
            unsigned* bar = reinterpret_cast<unsigned*>(W.cctl);
            int* err = W.cctl + 1;
            CUDA_CHECK(cudaMemsetAsync(W.cctl, 0, sizeof(int) * 4, st));
            void* args[] = {(void*)&Sc, (void*)&sval, &nrows, &nlong, (void*)&long_rows, (void*)&cptr, (void*)&ccol,
                            (void*)&cval, (void*)&cminv, (void*)&bin, (void*)&xout, &kk, &ldd, &GG, &W.cw[0],
                            &W.cw[1], &W.cw[2], &W.cw[3], &W.cw[4], &W.cpart, &bar, &err, &maxit, &rtol};
            const void* fn = nullptr;
            DISPATCH_CPL(cpl, ld, fn = (const void*)bk_coarse_cg<T, T, CPL, VEC>);
            CUDA_CHECK(cudaLaunchCooperativeKernel(fn, dim3(h->num_sms), dim3(CC_TPB), args,
                                                   sizeof(double) * CC_TPB * cpl, st));
            KERNEL_CHECK();
        }
    }
    for (int l = L - 1; l >= 0; --l) {
        Level& Lv = h->lev[l];
        const T* apv = f32 ? (const T*)Lv.AP.val32 : (const T*)Lv.AP.val;
        const T* minv = f32 ? (const T*)Lv.minv32 : (const T*)Lv.minv;
        const T* p = f32 ? (const T*)Lv.p32 : (const T*)Lv.p;
        const T* e = l + 1 == L ? lv(W.x, L) : lv(W.y, l + 1);
        const int g = grid_rows(h, Lv.AP.n, G);
        Scope sc_(&h->prof, st, l == 0 ? K_POST_L0 : K_POST,
                  (double)Lv.ap_nnz * (sizeof(T) + 4) + (double)Lv.A.n * k * (4.0 * sizeof(T) + 8));
        if (l > 0)
            DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)Lv.ap_nnz * k, bk_post<T, T, CPL, false, VEC>, g, TPB, 0, st, 
                                  sv(Lv.AP), apv, minv, omega, Lv.agg, p, e, lv(W.x, l), lv(W.r, l), nullptr, nullptr,
                                  lv(W.y, l), k, ld, G, W.partial, W.ticket, W.sc, flexible));
        else
            DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)Lv.ap_nnz * k, bk_post<T, T, CPL, true, VEC>, red_grid(h, W, G), TPB, 0, st, 
                                  sv(Lv.AP), apv, minv, omega, Lv.agg, p, e, lv(W.x, 0), lv(W.r, 0), W.R,
                                  flexible ? W.Q : nullptr, (T*)W.Z, k, ld, G, W.partial, W.ticket, W.sc, flexible));
        KERNEL_CHECK();
    }
}

// Lanes per row of the block V-cycle (G; each lane carries ceil(K/G)
// columns, at most 8): the candidates are timed on one V-cycle of all K
// columns, on zeroed work vectors, and the fastest is cached by shape.
void block_autotune(amg_hierarchy* h, BlockWork& W) {
    const bool f32 = h->opt.precision == AMG_FP32_VCYCLE;
    const int V = f32 ? 4 : 8;
    const Level& L0 = h->lev[0];
    const std::string key = tune_key("block", V, L0.A.n, L0.A.nnz, (long long)h->lev.size(), W.K, h->num_sms);
    int best = 0;
    if (!tune_get(key, &best)) {
        cudaStream_t st = h->stream;
        for (size_t l = 0; l < h->lev.size(); ++l) {
            const size_t m = (size_t)h->lev[l].A.n * W.K * V;
            for (void* v : {W.b[l], W.x[l], W.r[l], W.y[l]}) CUDA_CHECK(cudaMemsetAsync(v, 0, m, st));
        }
        const size_t m0 = (size_t)L0.A.n * W.K * 8;
        for (double* v : {W.R, W.Z, W.Q}) CUDA_CHECK(cudaMemsetAsync(v, 0, m0, st));
        const bool prof_on = h->prof.on;
        h->prof.on = false;
        double tbest = 1e30;
        try {
            for (int G = std::min(32, pow2_at_least(W.K)); G >= 1; G /= 2) {
                if (pow2_at_least((W.K + G - 1) / G) > 8) break;
                W.tuned_G = G;
                const double t = time_launches(st, [&]() {
                    if (f32) block_vcycle<float>(h, W, W.K, 0);
                    else block_vcycle<double>(h, W, W.K, 0);
                }, 2);
                if (t < tbest) {
                    tbest = t;
                    best = G;
                }
            }
        } catch (...) {
            h->prof.on = prof_on;
            W.tuned_G = 0;
            throw;
        }
        h->prof.on = prof_on;
        CUDA_CHECK(cudaMemsetAsync(W.sc.mode, 0, sizeof(int) * W.K, st));
        CUDA_CHECK(cudaMemsetAsync(W.sc.iters, 0, sizeof(int) * W.K, st));
        CUDA_CHECK(cudaStreamSynchronize(st));
        tune_put(key, best);
    }
    W.tuned_G = best;
}

void copy_state_async(amg_hierarchy* h, BlockWork& W) {
    cudaStream_t st = h->stream;
    CUDA_CHECK(cudaMemcpyAsync(W.mode_host, W.sc.mode, sizeof(int) * W.K, cudaMemcpyDeviceToHost, st));
    CUDA_CHECK(cudaMemcpyAsync(W.iters_host, W.sc.iters, sizeof(int) * W.K, cudaMemcpyDeviceToHost, st));
    CUDA_CHECK(cudaMemcpyAsync(W.rr_host, W.sc.rr, sizeof(double) * W.K, cudaMemcpyDeviceToHost, st));
    CUDA_CHECK(cudaMemcpyAsync(W.bb_host, W.sc.bb, sizeof(double) * W.K, cudaMemcpyDeviceToHost, st));
}

}  // namespace

BlockWork& block_ensure(amg_hierarchy* h, int K, bool fixed_width) {
    if (h->blk && h->blk->K == K && h->blk->fixed_width == fixed_width) return *h->blk;
    if (K < 1 || K > MAXK) AMG_THROW(AMG_ERR_TOO_LARGE, "block solves take 1..%d columns", MAXK);
    if (h->opt.pre != 1 || h->opt.post != 1) AMG_THROW(AMG_ERR_ARG, "block solves use 1+1 smoothing sweeps");
    if (h->lev.size() < 2) AMG_THROW(AMG_ERR_ARG, "block solves need at least two levels");
    if (!h->seg0.empty()) AMG_THROW(AMG_ERR_ARG, "block solves take a hierarchy of one system");
    if (h->opt.cycle > 0 || h->opt.smooth_p) AMG_THROW(AMG_ERR_ARG, "block solves use the unsmoothed V-cycle");
    if (h->blk) {
        CUDA_CHECK(cudaStreamSynchronize(h->stream));
        delete h->blk;
        h->blk = nullptr;
    }
    // the hierarchy gets the workspace when it is whole: one that an allocation
    // ended would be taken for it by the next call of the same width
    std::unique_ptr<BlockWork> own(new BlockWork);
    BlockWork* W = own.get();
    W->mem.stream = h->stream;
    W->K = K;
    W->fixed_width = fixed_width;
    const bool f32 = h->opt.precision == AMG_FP32_VCYCLE;
    W->vec_cols = f32 ? 4 : 2;
    const size_t V = f32 ? 4 : 8;
    for (auto& L : h->lev) {
        const size_t m = (size_t)L.A.n * K;
        W->b.push_back(W->mem.alloc<char>(m * V));
        W->x.push_back(W->mem.alloc<char>(m * V));
        W->r.push_back(W->mem.alloc<char>(m * V));
        W->y.push_back(W->mem.alloc<char>(m * V));
    }
    const size_t m0 = (size_t)h->lev[0].A.n * K;
    W->R = W->mem.alloc<double>(m0);
    W->Z = W->mem.alloc<double>(m0);
    W->P = W->mem.alloc<double>(m0);
    W->Q = W->mem.alloc<double>(m0);
    W->T = W->mem.alloc<double>(m0);
    W->sc.mode = W->mem.alloc<int>(K);
    W->sc.iters = W->mem.alloc<int>(K);
    W->sc.rho = W->mem.alloc<double>(K);
    W->sc.alpha = W->mem.alloc<double>(K);
    W->sc.beta = W->mem.alloc<double>(K);
    W->sc.pq = W->mem.alloc<double>(K);
    W->sc.rr = W->mem.alloc<double>(K);
    W->sc.bb = W->mem.alloc<double>(K);
    W->sc.rtol = W->mem.alloc<double>(K);
    W->grid = h->num_sms * 8;
    const int teams = (W->grid + CS_TEAM - 1) / CS_TEAM;
    W->partial = W->mem.alloc<double>((size_t)(W->grid + teams) * 2 * K);
    W->ticket = W->mem.alloc<unsigned>(1 + teams);
    CUDA_CHECK(cudaMemsetAsync(W->ticket, 0, sizeof(unsigned) * (1 + teams), h->stream));
    CUDA_CHECK(cudaMemsetAsync(W->sc.mode, 0, sizeof(int) * K, h->stream));
    CUDA_CHECK(cudaMemsetAsync(W->sc.iters, 0, sizeof(int) * K, h->stream));
    CUDA_CHECK(cudaHostAlloc(&W->mode_host, sizeof(int) * K, cudaHostAllocDefault));
    CUDA_CHECK(cudaHostAlloc(&W->iters_host, sizeof(int) * K, cudaHostAllocDefault));
    CUDA_CHECK(cudaHostAlloc(&W->rr_host, sizeof(double) * K, cudaHostAllocDefault));
    CUDA_CHECK(cudaHostAlloc(&W->bb_host, sizeof(double) * K, cudaHostAllocDefault));
    for (int c = 0; c < K; ++c) W->mode_host[c] = COL_IDLE;
    if (h->coarse_cg) {
        for (int v = 0; v < 5; ++v) W->cw[v] = W->mem.alloc<double>((size_t)h->nc * K);
        W->cpart = W->mem.alloc<double>((size_t)h->num_sms * K * 4);
        W->cctl = W->mem.alloc<int>(4);
        int per_sm = 0;
        CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bk_coarse_cg<double, double, 8, true>, CC_TPB,
                                                                 sizeof(double) * CC_TPB * 8));
        if (per_sm < 1) AMG_THROW(AMG_ERR_CUDA, "multi-column coarsest CG kernel cannot be resident");
    }
    if (h->opt.autotune && !fixed_width) block_autotune(h, *W);
    h->blk = own.release();
    return *h->blk;
}

size_t block_bytes_per_column(const amg_hierarchy* h) {
    const size_t V = h->opt.precision == AMG_FP32_VCYCLE ? 4 : 8;
    size_t rows = 0;
    for (auto& L : h->lev) rows += (size_t)L.A.n;
    return rows * 4 * V + (size_t)h->lev[0].A.n * 5 * 8;
}

// Level 0's float copy of R (FP32 V-cycle), else null.
static float* r32_of(amg_hierarchy* h) {
    return h->opt.precision == AMG_FP32_VCYCLE ? static_cast<float*>(h->blk->b[0]) : nullptr;
}

// INIT columns among [0, k): residual of X, then START (or DONE for b = 0,
// whose X column is zeroed). Launches only.
void block_init_launch(amg_hierarchy* h, const double* B, double* X, int k) {
    BlockWork& W = *h->blk;
    cudaStream_t st = h->stream;
    int G, cpl;
    group_shape(W, k, &G, &cpl);
    Level& L0 = h->lev[0];
    DISPATCH_CPL(cpl, W.K, launch_rows(W, (long long)L0.A.nnz * k, bk_residual<CPL, VEC>, red_grid(h, W, G), TPB, 0, st, sv(L0.S), L0.S.val, X, B, W.R, r32_of(h), k, W.K, G,
                                                             W.partial, W.ticket, W.sc, 0));
    KERNEL_CHECK();
    bk_zero_cols<<<blocks_for((long long)L0.A.n * k, TPB, h->num_sms * 8), TPB, 0, st>>>(L0.A.n, X, k, W.K, W.sc.mode,
                                                                                      W.sc.bb);
    KERNEL_CHECK();
}

namespace {

// The kernels of one step of columns [0, k): with `any_active` the CG half
// (p and q from the last step's z, x and r updates), then the V-cycle.
void block_step_kernels(amg_hierarchy* h, double* X, int k, bool any_active) {
    BlockWork& W = *h->blk;
    cudaStream_t st = h->stream;
    const int ld = W.K;
    const int flexible = h->opt.krylov == 1;
    int G, cpl;
    group_shape(W, k, &G, &cpl);
    Level& L0 = h->lev[0];
    const int n = L0.A.n;
    const double nnz = (double)L0.A.nnz;
    const bool f32 = h->opt.precision == AMG_FP32_VCYCLE;
    if (any_active) {
        {
            Scope sc_(&h->prof, st, K_SPMV_DOT, 12.0 * nnz + (f32 ? 36.0 : 40.0) * n * k);
            if (f32 && L0.A.max_row > SPLIT_WIDE)
                DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)L0.A.nnz * k, bk_direction<float, CPL, VEC, true>, red_grid(h, W, G), TPB, 0, st,
                                          sv(L0.S), L0.S.val, (const float*)W.Z, W.P, W.Q, k, ld, G, W.partial,
                                          W.ticket, W.sc));
            else if (f32)
                DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)L0.A.nnz * k, bk_direction<float, CPL, VEC, false>, red_grid(h, W, G), TPB, 0, st,
                                          sv(L0.S), L0.S.val, (const float*)W.Z, W.P, W.Q, k, ld, G, W.partial,
                                          W.ticket, W.sc));
            else
                DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)L0.A.nnz * k, bk_direction<double, CPL, VEC, false>, red_grid(h, W, G), TPB, 0, st, 
                                          sv(L0.S), L0.S.val, W.Z, W.P, W.Q, k, ld, G, W.partial, W.ticket, W.sc));
            KERNEL_CHECK();
        }
        {
            Scope sc_(&h->prof, st, K_UPDATE_XR, (f32 ? 52.0 : 48.0) * n * k);
            DISPATCH_CPL(cpl, ld, launch_rows(W, (long long)n * k, bk_update_xr<CPL, VEC>, red_grid(h, W, G), TPB, 0, st, n, W.P, W.Q, X, W.R, r32_of(h), k, ld, G,
                                                                      W.partial, W.ticket, W.sc));
            KERNEL_CHECK();
        }
    }
    if (f32) block_vcycle<float>(h, W, k, flexible);
    else block_vcycle<double>(h, W, k, flexible);
}

bool any_active_column(const BlockWork& W, int k) {
    for (int c = 0; c < k; ++c)
        if (W.mode_host[c] == COL_ACTIVE) return true;
    return false;
}

// The same step as one CUDA graph launch: the step's kernels are captured
// once per (active columns or not) on a private stream (the caller's may be
// the legacy default stream, which cannot capture) and replayed on the
// hierarchy's stream. Used while profiling is off and the coarsest level is
// dense (the coarsest CG is a cooperative launch).
void block_step_graph(amg_hierarchy* h, double* X, int k) {
    BlockWork& W = *h->blk;
    if (W.gk != k || W.gX != X) {
        for (auto& g : W.gstep)
            if (g) {
                CUDA_CHECK(cudaGraphExecDestroy(g));
                g = nullptr;
            }
        W.gk = k;
        W.gX = X;
    }
    const bool act = any_active_column(W, k);
    cudaGraphExec_t& ge = W.gstep[act ? 1 : 0];
    if (!ge) {
        cudaStream_t st = h->stream;
        cudaStream_t cs = nullptr;
        CUDA_CHECK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        h->stream = cs;
        cudaGraph_t graph = nullptr;
        try {
            CUDA_CHECK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
            const long long before = launch_counter().load();
            try {
                block_step_kernels(h, X, k, act);
                W.gkernels[act ? 1 : 0] = launch_counter().load() - before;
            } catch (...) {
                cudaStreamEndCapture(cs, &graph);
                if (graph) cudaGraphDestroy(graph);
                throw;
            }
            CUDA_CHECK(cudaStreamEndCapture(cs, &graph));
            CUDA_CHECK(cudaGraphInstantiate(&ge, graph, 0));
            CUDA_CHECK(cudaGraphDestroy(graph));
        } catch (...) {
            h->stream = st;
            cudaStreamDestroy(cs);
            throw;
        }
        h->stream = st;
        CUDA_CHECK(cudaStreamDestroy(cs));
    }
    CUDA_CHECK(cudaGraphLaunch(ge, h->stream));
    launch_counter().fetch_add(W.gkernels[act ? 1 : 0], std::memory_order_relaxed);
    copy_state_async(h, W);
}

}  // namespace

// One step of columns [0, k) (see the file comment), then an asynchronous
// copy of the column states to the host mirrors. Launches only.
void block_step_launch(amg_hierarchy* h, const double* B, double* X, int k) {
    (void)B;
    BlockWork& W = *h->blk;
    block_step_kernels(h, X, k, any_active_column(W, k));
    copy_state_async(h, W);
}

// After a synchronised step: true residual of the CHECK columns (DONE or
// restart). Returns whether anything was launched.
bool block_check_launch(amg_hierarchy* h, const double* B, double* X, int k) {
    BlockWork& W = *h->blk;
    bool any_check = false;
    for (int c = 0; c < k; ++c) any_check |= W.mode_host[c] == COL_CHECK;
    if (!any_check) return false;
    int G, cpl;
    group_shape(W, k, &G, &cpl);
    Level& L0 = h->lev[0];
    const double nnz = (double)L0.A.nnz;
    Scope sc_(&h->prof, h->stream, K_RESIDUAL, 12.0 * nnz + 24.0 * L0.A.n * k);
    DISPATCH_CPL(cpl, W.K, launch_rows(W, (long long)L0.A.nnz * k, bk_residual<CPL, VEC>, red_grid(h, W, G), TPB, 0, h->stream, sv(L0.S), L0.S.val, X, B, W.R, r32_of(h), k,
                                                                    W.K, G, W.partial, W.ticket, W.sc, 1));
    KERNEL_CHECK();
    copy_state_async(h, W);
    return true;
}

void block_report_launch(amg_hierarchy* h, const double* B, const double* X, int k) {
    BlockWork& W = *h->blk;
    int G, cpl;
    group_shape(W, k, &G, &cpl);
    Level& L0 = h->lev[0];
    DISPATCH_CPL(cpl, W.K, launch_rows(W, (long long)L0.A.nnz * k, bk_residual<CPL, VEC>, red_grid(h, W, G), TPB, 0, h->stream, sv(L0.S), L0.S.val, X, B, W.T, nullptr, k, W.K,
                                                                    G, W.partial, W.ticket, W.sc, 2));
    KERNEL_CHECK();
    copy_state_async(h, W);
}

void block_set_columns(amg_hierarchy* h, int c0, int cnt, int mode, double rtol) {
    BlockWork& W = *h->blk;
    std::vector<int> md(cnt, mode);
    std::vector<double> rt(cnt, rtol);
    std::vector<int> zi(cnt, 0);
    CUDA_CHECK(cudaMemcpyAsync(W.sc.mode + c0, md.data(), sizeof(int) * cnt, cudaMemcpyHostToDevice, h->stream));
    CUDA_CHECK(cudaMemcpyAsync(W.sc.rtol + c0, rt.data(), sizeof(double) * cnt, cudaMemcpyHostToDevice, h->stream));
    CUDA_CHECK(cudaMemcpyAsync(W.sc.iters + c0, zi.data(), sizeof(int) * cnt, cudaMemcpyHostToDevice, h->stream));
    // host buffers are pageable: make sure they are consumed before they go out of scope
    CUDA_CHECK(cudaStreamSynchronize(h->stream));
    for (int c = c0; c < c0 + cnt; ++c) W.mode_host[c] = mode;
}

static amg_status solve_columns(amg_hierarchy* h, int k, const double* B, double* X, double rtol, int maxit,
                                amg_solve_info* infos) {
    auto t0 = std::chrono::steady_clock::now();
    BlockWork& W = block_ensure(h, k, false);
    block_set_columns(h, 0, k, COL_INIT, rtol);
    block_init_launch(h, B, X, k);
    copy_state_async(h, W);
    CUDA_CHECK(cudaStreamSynchronize(h->stream));
    int steps = 0;
    const bool graphs = !h->prof.on && !h->coarse_cg;
    for (;;) {
        bool live = false;
        int maxi = 0;
        for (int c = 0; c < k; ++c) {
            live |= W.mode_host[c] == COL_START || W.mode_host[c] == COL_ACTIVE;
            maxi = std::max(maxi, W.iters_host[c]);
        }
        if (!live || maxi >= maxit || ++steps > 4 * maxit + 16) break;
        if (graphs) block_step_graph(h, X, k);
        else block_step_launch(h, B, X, k);
        CUDA_CHECK(cudaStreamSynchronize(h->stream));
        if (block_check_launch(h, B, X, k)) CUDA_CHECK(cudaStreamSynchronize(h->stream));
    }
    block_report_launch(h, B, X, k);
    CUDA_CHECK(cudaStreamSynchronize(h->stream));
    h->prof.flush();
    const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    amg_status status = AMG_OK;
    for (int c = 0; c < k; ++c) {
        const int md = W.mode_host[c];
        const double nb = std::sqrt(W.bb_host[c]);
        const double tr = nb > 0.0 ? std::sqrt(W.rr_host[c]) / nb : 0.0;
        if (md == COL_FAILED) status = AMG_ERR_BREAKDOWN;
        else if (md != COL_DONE && status == AMG_OK) status = AMG_NOT_CONVERGED;
        if (infos) {
            infos[c].iterations = W.iters_host[c];
            infos[c].restarts = 0;
            infos[c].relres = tr;
            infos[c].true_relres = tr;
            infos[c].solve_ms = ms;
        }
    }
    return status;
}

// The kernels load two doubles of B and X at once: blocks that start off a
// 16-byte boundary are solved in copies.
amg_status solve_batch(amg_hierarchy* h, int k, const double* B, double* X, double rtol, int maxit,
                       amg_solve_info* infos) {
    if (((reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(X)) & 15) == 0 || k > MAXK)
        return solve_columns(h, k, B, X, rtol, maxit, infos);
    const size_t count = (size_t)h->lev[0].A.n * k;
    DevArena mem;
    mem.stream = h->stream;
    double* Bc = mem.alloc<double>(count);
    double* Xc = mem.alloc<double>(count);
    CUDA_CHECK(cudaMemcpyAsync(Bc, B, sizeof(double) * count, cudaMemcpyDeviceToDevice, h->stream));
    CUDA_CHECK(cudaMemcpyAsync(Xc, X, sizeof(double) * count, cudaMemcpyDeviceToDevice, h->stream));
    const amg_status status = solve_columns(h, k, Bc, Xc, rtol, maxit, infos);
    CUDA_CHECK(cudaMemcpyAsync(X, Xc, sizeof(double) * count, cudaMemcpyDeviceToDevice, h->stream));
    CUDA_CHECK(cudaStreamSynchronize(h->stream));
    return status;
}

void block_free(amg_hierarchy* h) {
    delete h->blk;
    h->blk = nullptr;
}

void block_scatter_request(amg_hierarchy* h, const double* src, int k, const int* slots, double* dst) {
    SlotList sl;
    sl.n = k;
    for (int j = 0; j < k; ++j) sl.slot[j] = slots[j];
    const int n = h->lev[0].A.n;
    bk_scatter_slots<<<blocks_for((long long)n * k, TPB, h->num_sms * 8), TPB, 0, h->stream>>>(n, src, h->blk->K, dst,
                                                                                            sl);
    KERNEL_CHECK();
}

void block_gather_column(amg_hierarchy* h, const double* src, int slot, double* dst, int k, int j) {
    const int n = h->lev[0].A.n;
    bk_gather_slot<<<blocks_for(n, TPB, h->num_sms * 4), TPB, 0, h->stream>>>(n, src, h->blk->K, slot, dst, k, j);
    KERNEL_CHECK();
}

}  // namespace amg
