// Step 1 of Sec. 4: binning of the sample onto the grid.
//
// Linear binning (the multilinear rule the paper takes from Wand 1994):
//   inside iff lo_k <= x_k <= hi_k on every axis (the grid range contains
//   the data); t_k = (x_k - lo_k) * (1 / delta_k) (FP64, each operation
//   rounded separately, no contraction; within two ulps of the quotient),
//   clamped to M_k - 1 because the rounding of delta_k can push a point at
//   hi_k just past it
//   l_k = floor(t_k), clamped to M_k - 2 on the upper edge; f_k = t_k - l_k
//   corner l + b receives prod_k (b_k ? f_k : 1 - f_k), product in axis order.
// Simple binning: weight 1 at l_k = floor(t_k + 1/2), with t_k the quotient
// (x_k - lo_k) / delta_k itself, so that the cells match the oracle's bit for
// bit.
//
// The sample is read once: the same pass takes the moments that the
// normal-scale start needs (its FP64 work hides behind the atomics).  Its
// counts go to a histogram of its own in each block's shared memory where the
// grid fits, else to global atomics in L2.
//
// FP32 counts are accumulated in 64-bit fixed point (each weight rounded to
// a multiple of 2^-K, K = 32 for samples below 2^31 points): integer sums do
// not depend on the order of the atomic additions, so the counts, and every
// objective value computed from them, are the same from run to run.  Their
// corner weights are FP32 products of the FP64 fractions rounded to FP32: a
// weight's relative error of a few 2^-24 matches the FP32 rounding of the
// count itself.  FP64 counts use FP64 weights and FP64 atomics.
#include <cmath>
#include <cstring>
#include <type_traits>

#include "devutil.cuh"
#include "engine.cuh"

namespace kdefft {

// ------------------------------------------------------------ one point
// Order-preserving integer of a double: a < b as doubles iff key(a) < key(b)
// for ordered values; NaN lies beyond both infinities.
__host__ __device__ __forceinline__ long long order_key(long long bits) {
    return bits ^ ((bits >> 63) & 0x7fffffffffffffffLL);
}

void bin_axes(const GridDesc& g, BinAxes& ax) {
    std::memset(&ax, 0, sizeof(ax));
    unsigned int s = 1;
    for (int k = g.d - 1; k >= 0; --k) {
        ax.lo[k] = g.lo[k];
        ax.delta[k] = g.delta[k];
        ax.inv[k] = 1.0 / g.delta[k];
        // a bound at zero admits both of its signs
        const double lo = g.lo[k] == 0.0 ? -0.0 : g.lo[k], hi = g.hi[k] == 0.0 ? 0.0 : g.hi[k];
        long long b;
        std::memcpy(&b, &lo, 8);
        ax.klo[k] = order_key(b);
        std::memcpy(&b, &hi, 8);
        ax.khi[k] = order_key(b);
        ax.top[k] = (int)g.M[k] - 2;
        ax.stride[k] = s;
        s *= (unsigned int)g.M[k];
    }
}

// FP64 arithmetic is what a point costs on this part (2 lanes a cycle and SM,
// 64 for integer operations), so only t = (x - lo) * (1 / delta) is FP64: the
// bounds are integer comparisons, and cell and fraction come from t's bits.
// t is within two ulps of the oracle's (x - lo) / delta, so a point moves to
// the next cell only within two ulps of a node, where its weight there is
// ~1e-16.  x is inside iff lo <= x <= hi on every axis (NaN is not).
__device__ __forceinline__ bool inside(double x, long long klo, long long khi) {
    const long long key = order_key(__double_as_longlong(x));
    return key >= klo && key <= khi;
}

// v 2^e rounded once to FP32 (ties to even), for results of zero or from 2^-94
// up.  The leading bit goes to the top, what falls below the upper 32 bits
// leaves a one in the lowest of them (32 bits round to 24 as the 64 would),
// and the scale is exact.  The conversion instructions from and to 64-bit
// integers run at the FP64 rate here, so each costs as much as a product in
// FP64, which is what the pass is bound by: with them (d + 2^d a point) 1e7
// points on 512^2 take 363 us instead of 250, 1e6 on 128^3 103 instead of 75,
// 1e6 on 48^4 142 instead of 119.
__device__ __forceinline__ float scaled_f32(unsigned long long v, int e) {
    const unsigned int hi = (unsigned int)(v >> 32);
    const int n = hi ? __clz(hi) : 32 + __clz((unsigned int)v);
    v <<= n & 63;   // v = 0 has n = 64 and stays zero
    const unsigned int top = (unsigned int)(v >> 32) | ((unsigned int)v != 0u ? 1u : 0u);
    return __uint2float_rn(top) * __int_as_float((159 - n + e) << 23);
}

// w 2^K rounded to an integer (ties to even), w in [0, 1] and qs = 2^K <= 2^32:
// a 32-bit conversion, which stops at 2^32 - 1, and one more for 2^32
__device__ __forceinline__ unsigned long long fixed_weight(float w, float qs) {
    const float v = w * qs;
    return (unsigned long long)__float2uint_rn(v) + (v >= 4294967296.f ? 1ULL : 0ULL);
}

// A fixed-point weight added to a histogram in shared memory by two 32-bit
// additions, the carry from the low word's own sum (integer sums: any order
// gives the same bits).  A 64-bit addition retries where lanes meet on a cell,
// so that concentrated samples were slow: 4e6 points, all of them or half of
// them in one cell, 1-D on 700 nodes 487 and 272 us (75 and 76 this way; 80 ->
// 76 spread over the grid), sorted ones 215 (74), 2-D on 100^2 681 and 367 (126).
__device__ __forceinline__ void add_shared(unsigned long long* p, unsigned long long w) {
    unsigned int* q = reinterpret_cast<unsigned int*>(p);   // low word first
    const unsigned int lo = (unsigned int)w, old = atomicAdd(q, lo);
    const unsigned int hi = (unsigned int)(w >> 32) + (old + lo < lo ? 1u : 0u);
    if (hi) atomicAdd(q + 1, hi);
}

// Cell l = min(floor(t), M - 2) and fraction t - l (1 where t reaches M - 1,
// which the rounding of delta can push past it) of t >= 0, below 2^31: t is
// m 2^-sh with a 53-bit m, so the cell is m >> sh and the fraction the bits
// below, one rounding from FP32 (t < 2^-74 gives a fraction below 2^-73
// instead of its own, and a weight of zero either way).  A step below 2^-1024
// or past the largest double has no finite reciprocal, and t is then infinite
// or NaN (sh < 22): such a point lies at M - 1, as fmin(t, M - 1) has it.
__device__ __forceinline__ int cell_f32(double t, int top, float& f) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(t);
    const unsigned long long m = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
    const int sh = min(1075 - (int)((b >> 52) & 0x7ff), 126);   // the sign of -0 does not matter
    const int s = min(max(sh, 22), 63);
    int l = (int)(m >> s);
    f = scaled_f32(m << (64 - s), s - 64 - max(sh, 22));   // s >= 22: the cell's bits leave at the top
    if (l > top || sh < 22) {
        l = top;
        f = 1.f;
    }
    return l;
}
// the same with the fraction in FP64 (t + 2^52 rounded down holds floor(t))
__device__ __forceinline__ int cell_f64(double t, int top, double& f) {
    const double u = __dadd_rd(t, 4503599627370496.0);
    int l = (int)__double_as_longlong(u);
    f = __dsub_rn(t, __dsub_rn(u, 4503599627370496.0));
    if (l > top || (__double2hiint(t) & 0x7fffffff) >= 0x41e00000) {   // (t infinite or NaN)
        l = top;
        f = 1.0;
    }
    return l;
}

// Nearest node floor(min(t, M - 1) + 1/2) with t the quotient (x - lo) / delta
// itself.  t * (1 / delta) is within two ulps of it: the division is only
// needed within 2^-30 of a tie (and where there is no finite 1 / delta).
__device__ __forceinline__ int nearest(double x, double lo, double delta, double inv, int top) {
    const double y = __dsub_rn(x, lo);
    double t = __dmul_rn(y, inv);
    const double h = __dadd_rn(t, 0.5), u = __dadd_rd(h, 4503599627370496.0);
    const double r = __dsub_rn(h, __dsub_rn(u, 4503599627370496.0));   // in [0, 1)
    int l = (int)__double_as_longlong(u);
    if (!(r >= 1e-9 && r <= 1.0 - 1e-9)) {   // (NaN too)
        t = fmin(__ddiv_rn(y, delta), (double)(top + 1));
        l = (int)floor(__dadd_rn(t, 0.5));
    }
    return min(l, top + 1);
}

// ------------------------------------------------------------ the pass
// Points i0 + threadIdx.x, + stride, .. below n: their counts into `counts`
// (kind 0: fixed point, kind 1: FP64, kind 2: whole points), and the block's
// sums of x - s and (x - s)(x - s)^T to part.  SHARED: `counts` is a histogram
// in shared memory.
//
// A linear-binned point is 2^d 64-bit atomic additions to scattered cells,
// and what L2 is limited by is the 32-byte sectors they touch (58 G/s on
// 128^3 with a point per lane).  So a warp spreads its 32 points over lane
// pairs, half of them at a time, and a pair adds the two neighbours along the
// last axis with one instruction: three times out of four they share a sector.
// What is left is FP64: 2 d operations to locate a point and 2 d + d (d + 1) / 2
// for its moments, about 85 % of the FP64 pipe's time for d = 2; on 48^4 the
// atomics bound it again.  Binning and moments with their
// launches, against a thread per point with run-time dimensions, FP64
// comparisons and floor, and a second pass for the moments: 1e7 points on
// 512^2 250 us (866), 1e6 on 128^3 75 us (206), 1e6 on 48^4 119 us (336);
// FP64 counts, 1e6 on 256^2 97 us (161).
template <int D, int KIND, bool SHARED, typename acc>
__device__ __forceinline__ void bin_pass(const double* __restrict__ X, long long n, long long i0, long long stride,
                                         const BinAxes& ax, const double* __restrict__ shift, acc* counts,
                                         unsigned long long* __restrict__ outside, double qscale,
                                         double* __restrict__ part) {
    constexpr int NV = D + D * (D + 1) / 2;
    constexpr int NP = NV <= 2 ? 2 : NV <= 8 ? 8 : 16;   // sums padded to a power of two
    const int lane = threadIdx.x & 31;
    const float qs = (float)qscale;   // 2^K, exact
    const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    double sum[NP];
#pragma unroll
    for (int v = 0; v < NP; ++v) sum[v] = 0.0;
    unsigned int nout = 0;
    auto load = [&](long long i, double* x) {
        if constexpr (D % 2 == 0) {
            if (vec) {
#pragma unroll
                for (int k = 0; k < D; k += 2) {
                    const double2 v = *reinterpret_cast<const double2*>(X + i * D + k);
                    x[k] = v.x;
                    x[k + 1] = v.y;
                }
                return;
            }
        }
#pragma unroll
        for (int k = 0; k < D; ++k) x[k] = X[i * D + k];
    };
    double xn[D];
    long long i = i0 + threadIdx.x;
    if (i < n) load(i, xn);
    for (; i - lane < n; i += stride) {   // a warp's lanes leave together
        const bool have = i < n;
        double x[D];
#pragma unroll
        for (int k = 0; k < D; ++k) x[k] = xn[k];
        if (i + stride < n) load(i + stride, xn);   // the next point is on its way meanwhile
        bool in = have;
        if (have) {
#pragma unroll
            for (int k = 0; k < D; ++k) in = in && inside(x[k], ax.klo[k], ax.khi[k]);
            if (!in) ++nout;
        }
        unsigned int base = 0;
        if constexpr (KIND == 2) {
            if (in) {
#pragma unroll
                for (int k = 0; k < D; ++k)
                    base += (unsigned int)nearest(x[k], ax.lo[k], ax.delta[k], ax.inv[k], ax.top[k]) * ax.stride[k];
                atomicAdd(counts + base, acc(1));
            }
        } else {
            using real = typename std::conditional<KIND == 0, float, double>::type;
            real f[D];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const double t = in ? __dmul_rn(__dsub_rn(x[k], ax.lo[k]), ax.inv[k]) : 0.0;
                if constexpr (KIND == 0)
                    base += (unsigned int)cell_f32(t, ax.top[k], f[k]) * ax.stride[k];
                else
                    base += (unsigned int)cell_f64(t, ax.top[k], f[k]) * ax.stride[k];
            }
            if (!in) base = 0xffffffffu;   // no cell: the grid has at most 2^31
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int src = half * 16 + (lane >> 1);
                const unsigned int b = __shfl_sync(0xffffffffu, base, src);
                real ff[D], gg[D];
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    ff[k] = __shfl_sync(0xffffffffu, f[k], src);
                    if constexpr (KIND == 0)
                        gg[k] = 1.f - ff[k];
                    else
                        gg[k] = __dsub_rn(1.0, ff[k]);
                }
                if (b == 0xffffffffu) continue;
                const real last = (lane & 1) ? ff[D - 1] : gg[D - 1];
#pragma unroll
                for (int c = 0; c < (1 << (D - 1)); ++c) {
                    unsigned int idx = b + (lane & 1);
                    real w = real(1);
#pragma unroll
                    for (int k = 0; k < D - 1; ++k) {
                        if ((c >> k) & 1) idx += ax.stride[k];
                        const real v = ((c >> k) & 1) ? ff[k] : gg[k];
                        if constexpr (KIND == 0)
                            w = k == 0 ? v : w * v;
                        else
                            w = k == 0 ? v : __dmul_rn(w, v);
                    }
                    if constexpr (KIND == 0) {
                        w = D == 1 ? last : w * last;
                        if constexpr (SHARED)
                            add_shared(counts + idx, fixed_weight(w, qs));
                        else
                            atomicAdd(counts + idx, (acc)fixed_weight(w, qs));
                    } else {
                        w = D == 1 ? last : __dmul_rn(w, last);
                        atomicAdd(counts + idx, (acc)w);
                    }
                }
            }
        }
        if (have) {   // moments: every point, inside or not
#pragma unroll
            for (int k = 0; k < D; ++k) x[k] -= shift[k];
#pragma unroll
            for (int k = 0; k < D; ++k) sum[k] += x[k];
            int v = D;
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
                for (int b = a; b < D; ++b) sum[v++] += x[a] * x[b];
        }
    }
    nout = __reduce_add_sync(0xffffffffu, nout);
    if (nout && lane == 0) atomicAdd(outside, (unsigned long long)nout);
    // Sums over the warp, for all values together: at each step a lane keeps
    // half of its values and adds the other lane's share of them, which takes
    // about as many FP64 additions as there are values instead of five for
    // each.  The pairs added are those of a shuffle-down tree, so the bits
    // are its bits; the eight warps are then added in order.
    int held = NP, first = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (held > 1) {
            const bool upper = (lane & o) != 0;
            held >>= 1;
#pragma unroll
            for (int v = 0; v < NP / 2; ++v) {
                if (v < held) {
                    const double keep = upper ? sum[v + held] : sum[v];
                    const double give = upper ? sum[v] : sum[v + held];
                    sum[v] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            if (upper) first += held;
        } else {
            sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
        }
    }
    __shared__ double red[8][NP];
    constexpr int LOW = 32 / NP;   // lanes that hold the same value
    if ((lane & (LOW - 1)) == 0) red[threadIdx.x >> 5][first] = sum[0];
    __syncthreads();
    constexpr int NF = D + D * D;
    if (threadIdx.x < NF) {
        int v = threadIdx.x;
        if (v >= D) {   // the full product matrix from its upper triangle
            const int p = (v - D) / D, q = (v - D) % D, a = p < q ? p : q, b = p < q ? q : p;
            v = D + a * D - a * (a - 1) / 2 + (b - a);
        }
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w][v];
        part[threadIdx.x] = t;   // block partial; summed in block order by the host
    }
}

template <int D, int KIND, typename acc>
__global__ void __launch_bounds__(256) k_bin(const double* __restrict__ X, long long n,
                                             const __grid_constant__ BinAxes ax, const __grid_constant__ Shift sh,
                                             acc* __restrict__ counts, unsigned int smem_cells,
                                             unsigned long long* __restrict__ outside, double qscale,
                                             double* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    acc* hist = reinterpret_cast<acc*>(smem_raw);
    for (unsigned int c = threadIdx.x; c < smem_cells; c += blockDim.x) hist[c] = acc(0);
    if (smem_cells) __syncthreads();
    const long long i0 = (long long)blockIdx.x * blockDim.x, stride = (long long)gridDim.x * blockDim.x;
    double* out = part + (size_t)blockIdx.x * (D + D * D);
    if (smem_cells)
        bin_pass<D, KIND, true, acc>(X, n, i0, stride, ax, sh.s, hist, outside, qscale, out);
    else
        bin_pass<D, KIND, false, acc>(X, n, i0, stride, ax, sh.s, counts, outside, qscale, out);
    if (smem_cells) {
        __syncthreads();
        for (unsigned int c = threadIdx.x; c < smem_cells; c += blockDim.x) {
            const acc v = hist[c];
            if (v != acc(0)) atomicAdd(counts + c, v);
        }
    }
}

__global__ void k_f32_to_f64(const float* __restrict__ src, double* __restrict__ dst, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (double)src[i];
}

cudaError_t launch_f32_to_f64(const float* src, double* dst, long long n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long b = (n + 255) / 256;
    if (b > 4096) b = 4096;
    k_f32_to_f64<<<(int)b, 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

// Fixed point to FP32, four cells a thread (16-byte loads and stores; both
// arrays are 16-byte aligned): one correctly rounded conversion and an exact
// product with a power of two.
__device__ __forceinline__ void fix_cells(const unsigned long long* __restrict__ src, float* __restrict__ dst,
                                          long long c, long long n, int e) {
    if (c + 4 <= n) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(src + c);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(src + c + 2);
        *reinterpret_cast<float4*>(dst + c) = make_float4(scaled_f32(a.x, e), scaled_f32(a.y, e),
                                                          scaled_f32(b.x, e), scaled_f32(b.y, e));
    } else {
        for (; c < n; ++c) dst[c] = scaled_f32(src[c], e);
    }
}

__global__ void __launch_bounds__(256) k_fix_to_f32(const unsigned long long* __restrict__ src,
                                                    float* __restrict__ dst, long long n, int e,
                                                    const unsigned long long* __restrict__ outside,
                                                    unsigned long long* __restrict__ outside_copy) {
    for (long long c = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x); c < n;
         c += 4LL * gridDim.x * blockDim.x)
        fix_cells(src, dst, c, n, e);
    if (blockIdx.x == 0 && threadIdx.x == 0) *outside_copy = *outside;
}

cudaError_t launch_fix_to_f32(const unsigned long long* src, float* dst, long long n, double unit,
                              const unsigned long long* outside, unsigned long long* outside_copy, int nsm,
                              cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const long long b = (n + 1023) / 1024, cap = (long long)nsm * 8;
    k_fix_to_f32<<<(unsigned)(b < cap ? b : cap), 256, 0, st>>>(src, dst, n, std::ilogb(unit), outside, outside_copy);
    return cudaGetLastError();
}

template <typename real>
__global__ void k_int_to_real(const int* __restrict__ src, real* __restrict__ dst, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (real)src[i];
}

template <typename real>
cudaError_t launch_int_to_real(const int* src, real* dst, long long n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long b = (n + 255) / 256;
    if (b > 4096) b = 4096;
    k_int_to_real<real><<<(int)b, 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

// Counts that fit in kBinSmem (two blocks an SM) go to a histogram per block.
// Against global atomics for these it is never slower (a pass over 1000 points
// on 100^2 35 against 37 us with its launches, 2e6 points 103 against 145 us),
// and where many points share few cells it takes the contention out of L2
// (8e6 points on 512 nodes 161 against 2224 us).
constexpr int kBinSmem = 96 * 1024;

// blocks of a binning pass: at most two per SM (the moments' block partials,
// which the host adds in block order, keep their number and their points)
int bin_blocks(long long n, int nsm) {
    long long b = (n + 255) / 256;
    const long long cap = 2LL * nsm;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

template <int D, int KIND, typename acc>
static cudaError_t bin_go(const double* X, long long n, const BinAxes& ax, const Shift& sh, acc* counts,
                          long long ncells, unsigned long long* outside, double qscale, double* part, int nsm,
                          cudaStream_t st) {
    const int grid = bin_blocks(n, nsm);
    const long long bytes = (long long)sizeof(acc) * ncells;
    const bool smem = bytes <= kBinSmem;
    k_bin<D, KIND, acc><<<grid, 256, smem ? (size_t)bytes : 0, st>>>(X, n, ax, sh, counts, smem ? (unsigned)ncells : 0u,
                                                                     outside, qscale, part);
    return cudaGetLastError();
}

template <int KIND, typename acc>
static cudaError_t bin_d(const double* X, long long n, const GridDesc& g, const Shift& sh, acc* counts,
                         long long ncells, unsigned long long* outside, double qscale, double* part, int nsm,
                         cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    BinAxes ax;
    bin_axes(g, ax);
    switch (g.d) {
        case 1: return bin_go<1, KIND, acc>(X, n, ax, sh, counts, ncells, outside, qscale, part, nsm, st);
        case 2: return bin_go<2, KIND, acc>(X, n, ax, sh, counts, ncells, outside, qscale, part, nsm, st);
        case 3: return bin_go<3, KIND, acc>(X, n, ax, sh, counts, ncells, outside, qscale, part, nsm, st);
        case 4: return bin_go<4, KIND, acc>(X, n, ax, sh, counts, ncells, outside, qscale, part, nsm, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_bin_fixed(const double* X, long long n, const GridDesc& g, const Shift& sh,
                             unsigned long long* counts, long long ncells, unsigned long long* outside, double qscale,
                             double* part, int nsm, cudaStream_t st) {
    return bin_d<0, unsigned long long>(X, n, g, sh, counts, ncells, outside, qscale, part, nsm, st);
}
cudaError_t launch_bin_f64(const double* X, long long n, const GridDesc& g, const Shift& sh, double* counts,
                           long long ncells, unsigned long long* outside, double* part, int nsm, cudaStream_t st) {
    return bin_d<1, double>(X, n, g, sh, counts, ncells, outside, 1.0, part, nsm, st);
}
cudaError_t launch_bin_simple(const double* X, long long n, const GridDesc& g, const Shift& sh, int* counts,
                              long long ncells, unsigned long long* outside, double* part, int nsm, cudaStream_t st) {
    return bin_d<2, int>(X, n, g, sh, counts, ncells, outside, 1.0, part, nsm, st);
}

// ------------------------------------------------------------ batched binning
constexpr int kCellsPerBlock = 256 * 16;

template <int D>
__global__ void __launch_bounds__(256) k_bin_many(const BinJob* __restrict__ jobs, int njobs, double qscale) {
    const BinJob& jb = jobs[job_of_warp(njobs, blockIdx.x, [&](int k) { return jobs[k].blk0; })];
    const long long b = (long long)blockIdx.x - jb.blk0;
    bin_pass<D, 0, false, unsigned long long>(jb.X, jb.n, b * blockDim.x, (long long)jb.mblk * blockDim.x, jb.ax, jb.shift,
                                              jb.fix, jb.outside, qscale, jb.part + b * (D + D * D));
}

__global__ void __launch_bounds__(256) k_fix_many(const BinJob* __restrict__ jobs, int njobs, int e) {
    const BinJob& jb = jobs[job_of_warp(njobs, blockIdx.x, [&](int k) { return jobs[k].blk1; })];
    const long long c0 = ((long long)blockIdx.x - jb.blk1) * kCellsPerBlock;
    const long long c1 = c0 + kCellsPerBlock < jb.ncells ? c0 + kCellsPerBlock : jb.ncells;
#pragma unroll
    for (int r = 0; r < kCellsPerBlock / 1024; ++r) {
        const long long c = c0 + 4LL * (r * 256 + threadIdx.x);
        if (c < c1) fix_cells(jb.fix, jb.counts, c, c1, e);
    }
}

cudaError_t launch_bin_many(BinJob* jobs_h, BinJob* jobs_d, int n, int d, double qscale, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    long long b0 = 0, b1 = 0;
    for (int k = 0; k < n; ++k) {
        BinJob& jb = jobs_h[k];
        jb.blk0 = b0;
        jb.blk1 = b1;
        b0 += jb.mblk;
        b1 += (jb.ncells + kCellsPerBlock - 1) / kCellsPerBlock;
    }
    if (b0 <= 0 || b1 <= 0 || b0 > 0x7fffffffLL || b1 > 0x7fffffffLL) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemcpyAsync(jobs_d, jobs_h, sizeof(BinJob) * n, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    switch (d) {
        case 1: k_bin_many<1><<<(unsigned)b0, 256, 0, st>>>(jobs_d, n, qscale); break;
        case 2: k_bin_many<2><<<(unsigned)b0, 256, 0, st>>>(jobs_d, n, qscale); break;
        case 3: k_bin_many<3><<<(unsigned)b0, 256, 0, st>>>(jobs_d, n, qscale); break;
        case 4: k_bin_many<4><<<(unsigned)b0, 256, 0, st>>>(jobs_d, n, qscale); break;
        default: return cudaErrorInvalidValue;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_fix_many<<<(unsigned)b1, 256, 0, st>>>(jobs_d, n, -std::ilogb(qscale));
    return cudaGetLastError();
}

template <int D>
static cudaError_t prepare_bin_d() {
    const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_bin<D, 0, unsigned long long>, at, kBinSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_bin<D, 1, double>, at, kBinSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_bin<D, 2, int>, at, kBinSmem);
    return e;
}

cudaError_t prepare_binning() {
    cudaError_t e = prepare_bin_d<1>();
    if (e == cudaSuccess) e = prepare_bin_d<2>();
    if (e == cudaSuccess) e = prepare_bin_d<3>();
    if (e == cudaSuccess) e = prepare_bin_d<4>();
    return e;
}

template cudaError_t launch_int_to_real<float>(const int*, float*, long long, cudaStream_t);
template cudaError_t launch_int_to_real<double>(const int*, double*, long long, cudaStream_t);

}  // namespace kdefft
