// Lag-domain evaluation of the binned functionals (Eq. 25 with the sum over
// the lag done first) against the count autocorrelation (whose passes run
// in engine.cu with the other transforms).
//
// A work item is a group of kernels of one data set that share covariances
// and support; it yields, for each kernel, the sum over the half lag box of
// w_j k_j a_j, w_j in {0, 1, 2}.  Kernels come from the compile-time Hermite
// recurrence, sums are compensated FP32 pairs, or FP64.  The last block of an
// item to finish adds the item's tile sums in a fixed order, times n^-2.
#pragma once

#include <algorithm>
#include <type_traits>

#include "devutil.cuh"
#include "engine.cuh"

namespace kdefft {

// floor(n / v) for a 32-bit n from the invariant divisor's multiplier m and
// shifts (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994, unsigned case): t = mulhi(m, n), then
// (t + ((n - t) >> s1)) >> s2; exact for every 32-bit n.
__device__ __forceinline__ uint32_t inv_div(uint32_t n, uint32_t m, int sh) {
    const uint32_t t = __umulhi(m, n);
    return (t + ((n - t) >> (sh & 0xff))) >> (sh >> 8);
}

// ------------------------------------------------------------ forms of a group
// What a group's kernels are made of, at compile time:
//   NV >= 0   NV kernels of the Gaussian itself (Hermite index 0), then all
//             partials of order R in graded order (R = 0: none), each a
//             weighted sum over the covariances: LSCV and SCV values and
//             gradients (R = 2), psi_r (NV = 0, one covariance for R > 2)
//   NV = -1   two kernels (or one), each any sum of partials up to order R
// SG: covariances that may have weights (a FP64 group without weights on the
// third one has a kernel of its own, and psi_2, which has one covariance, too).
template <int D, int R, int NV, int SG>
struct LagForm {
    static constexpr bool dense = NV < 0;
    static constexpr int N = cx_binom(D + R, D);                          // Hermite values
    static constexpr int N0 = R > 0 ? cx_binom(D + R - 1, D) : 0;         // the first of order R
    static constexpr int NO = dense ? 2 : NV + (R > 0 ? N - N0 : 0);      // kernels
    static constexpr int NS = (!dense && R > 2) ? 1 : SG;                 // covariances
    static constexpr int at(int o) { return o < NV ? 0 : N0 + (o - NV); }
    // FP64 groups sum the Gaussian (if any) and each partial of order R per
    // covariance, and weigh the sums at the end
    static constexpr int V = NV > 0 ? 1 : 0;
    static constexpr int NI = V + (R > 0 ? N - N0 : 0);
    static constexpr int sum_of(int o) { return o < NV ? 0 : V + (o - NV); }
};
// values padded to whole warp reductions: 32s, then a power of two
__host__ __device__ constexpr int lag_chunk(int left) {
    int c = 1;
    while (c < left && c < 32) c *= 2;
    return c;
}
__host__ __device__ constexpr int lag_padded(int n) {
    int p = 0;
    while (p < n) p += lag_chunk(n - p);
    return p;
}

// Sums over a warp of C values a lane (a power of two up to 32), all together:
// at each step a lane keeps half of its values and adds the other lane's share
// of them, so that C values take about C additions instead of 5 C.  put(i, x)
// receives sum i on one lane.
template <int C, typename T, typename Add, typename Give, typename Put>
__device__ __forceinline__ void warp_sums(T* v, int lane, Add add, Give shfl, Put put) {
    int held = C, first = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (held > 1) {
            const bool upper = (lane & o) != 0;
            held >>= 1;
#pragma unroll
            for (int i = 0; i < C / 2; ++i)
                if (i < held) {
                    const T keep = upper ? v[i + held] : v[i], give = upper ? v[i] : v[i + held];
                    v[i] = add(keep, shfl(give, o));
                }
            if (upper) first += held;
        } else {
            v[0] = add(v[0], shfl(v[0], o));
        }
    }
    if ((lane & (32 / C - 1)) == 0) put(first, v[0]);
}
template <int BASE, int NO, typename T, typename Add, typename Give, typename Put>
__device__ __forceinline__ void warp_sums_all(T* v, int lane, Add add, Give shfl, Put put) {
    if constexpr (BASE < NO) {
        constexpr int C = lag_chunk(NO - BASE);
        warp_sums<C>(v + BASE, lane, add, shfl, [&](int i, T x) {
            if (BASE + i < NO) put(BASE + i, x);
        });
        warp_sums_all<BASE + C, NO>(v, lane, add, shfl, put);
    }
}

// ------------------------------------------------------------ lag evaluation
// Tiles [t0, t0 + ntiles) of the batch's tile list.  FP32: a tile per CTA
// (256 threads, thread t takes the tile's points t, t + 256, ...), one
// partial per tile and kernel.  FP64: a tile's 256 points are 8 warp slices of
// one point per thread; a CTA of blockDim threads takes blockDim / 32 slices
// of a tile, and each warp writes its slice's partials.  A thread's points, a
// warp's reduction and the order of the final sum are the same for every
// block size, so the results are too.
//
// Bound by the FP32 (FP64) pipes: an exponential and the Hermite recurrence per
// point and covariance, and a compensated addition per kernel.  So all kernels
// that share them are summed from one evaluation (psi_4 in three dimensions: 15
// kernels from 35 Hermite values, where pairs of kernels evaluated them 8
// times), covariances without a weight in the group are left out, and the warp
// reductions take a group's kernels together.  FP64 groups do without what is
// not a point's own: weights and normalisers apply to the sums of each
// covariance, and where only Gaussians are asked for, the quadratic form takes
// the products x_a x_b once for all covariances (SCV values of 5 bandwidths on
// 61 x 97 x 45 48 -> 42 us, values and gradients of 16 on 256^2 35 -> 31 us).
// Per launch, against pairs of kernels with the sums of their tiles in a launch
// of their own (4 to 6 us more): psi_4 of 256 bandwidths on 128^3 67 us (329),
// 512 data sets x 16 LSCV bandwidths with gradients 122 us (364), SCV with
// gradients in FP64, 16 bandwidths on 256^2, 31 us (145).
template <typename real, int D, int R, int NV, int SG>
__device__ __forceinline__ void lag_tiles(const LagJob<real>& jb) {
    using F = LagForm<D, R, NV, SG>;
    constexpr bool dbl = sizeof(real) == 8;
    constexpr bool late = dbl && !F::dense;   // weights at the end
    constexpr int NSUM = late ? F::NI * F::NS : F::NO;   // sums of a tile
    constexpr HTab<D, R> ht{};
    constexpr int N = F::N, NO = F::NO, NP = lag_padded(NSUM), NS = F::NS;
    constexpr int NW = F::dense ? 2 * MAXSIG * N : NO * MAXSIG;
    using Sum = typename std::conditional<dbl, double, DFloat>::type;
    __shared__ real Ws[NW];
    __shared__ __align__(8) LagItem<real> it;
    __shared__ Sum red[dbl ? 1 : 8][dbl ? 1 : NP];
    __shared__ double fin[256];
    constexpr int NX = (late && R == 0) ? D * (D + 1) / 2 : 1;
    __shared__ double quad[MAXSIG][NX];   // -x^T Sigma^-1 x / 2 on the products x_a x_b, a <= b
    __shared__ int lastone;
    static_assert(sizeof(LagItem<real>) % 8 == 0, "staged by 8-byte words");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpc = (int)(blockDim.x >> 5);               // warps (FP64: slices) per CTA
    const int per = dbl ? kLagSlices / wpc : 1;           // CTAs per tile
    const long long nunits = (long long)jb.ntiles * per;
    for (long long u = blockIdx.x; u < nunits; u += gridDim.x) {
        const int tix = jb.t0 + (int)(u / per);
        const int s0 = dbl ? (int)(u % per) * wpc : 0;   // first slice of this CTA
        const LagTile tl = jb.tiles[tix];
        const LagItem<real>& src = jb.items[tl.item];
        __syncthreads();   // the previous tile's readers of it / Ws are done
        {
            const unsigned long long* a = reinterpret_cast<const unsigned long long*>(&src);
            unsigned long long* b = reinterpret_cast<unsigned long long*>(&it);
            for (int t = threadIdx.x; t < (int)(sizeof(LagItem<real>) / 8); t += blockDim.x) b[t] = a[t];
            if constexpr (late && R == 0) {
                for (int t = threadIdx.x; t < MAXSIG * NX; t += blockDim.x) {
                    int k = t % NX, a0 = 0;
                    while (k >= D - a0) k -= D - a0++;
                    quad[t / NX][t % NX] = (k == 0 ? -0.5 : -1.0) * src.lam[t / NX][a0 * MAXD + a0 + k];
                }
            }
            const int nsig = src.nsig, w_off = src.w_off;
            for (int t = threadIdx.x; t < NW; t += blockDim.x) {
                if constexpr (F::dense) {   // [kernel][covariance][Hermite index]
                    const int h = t / (MAXSIG * N), s = (t / N) % MAXSIG, k = t % N;
                    Ws[t] = (s < nsig) ? jb.wpool[w_off + (h * nsig + s) * N + k] : real(0);
                } else {                    // [kernel][covariance]
                    const int o = t / MAXSIG, s = t % MAXSIG;
                    Ws[t] = (s < nsig) ? jb.wpool[w_off + o * nsig + s] : real(0);
                }
            }
        }
        __syncthreads();
        const int sigs = it.sigs;   // covariances with a weight
        Sum acc[NP];
#pragma unroll
        for (int o = 0; o < NP; ++o)
            if constexpr (dbl)
                acc[o] = 0.0;
            else
                acc[o] = DFloat{0.f, 0.f};
        const int n0 = it.L[0] + 1;
        const long long end = tl.first + tl.n;
        const int vstride = dbl ? 32 * kLagSlices : (int)blockDim.x;
        for (long long f = tl.first + s0 * 32 + threadIdx.x; f < end; f += vstride) {
            // the flat index splits into (j_0, .., j_{d-1}) by exact 32-bit
            // divisions (the engine takes half boxes below 2^32 points)
            int j[D];
            uint32_t g = (uint32_t)f;
#pragma unroll
            for (int k = 0; k < D - 1; ++k) {
                const uint32_t w = (k == 0) ? (uint32_t)n0 : (uint32_t)(2 * it.L[k] + 1);
                const uint32_t qv = inv_div(g, it.qm[k], it.qs[k]);
                j[k] = (int)(g - qv * w) - (k == 0 ? 0 : it.L[k]);
                g = qv;
            }
            j[D - 1] = (int)g - (D == 1 ? 0 : it.L[D - 1]);
            // half-space weight: 2 where the first nonzero coordinate is positive
            int wt = 1, decided = 0;
#pragma unroll
            for (int k = 0; k < D; ++k)
                if (!decided && j[k] != 0) {
                    wt = j[k] > 0 ? 2 : 0;
                    decided = 1;
                }
            if (wt == 0) continue;
            long long ai = 0;
#pragma unroll
            for (int k = D - 1; k >= 1; --k) ai = ai * (2 * it.A[k] + 1) + (j[k] + it.A[k]);
            ai = ai * (it.A[0] + 1) + j[0];
            const real wa = real(wt) * it.acorr[ai];
            real x[D];
#pragma unroll
            for (int k = 0; k < D; ++k) x[k] = it.delta[k] * (real)j[k];
            if constexpr (late) {
                double xx[NX];
                if constexpr (R == 0) {
                    int k = 0;
#pragma unroll
                    for (int a = 0; a < D; ++a)
#pragma unroll
                        for (int b = a; b < D; ++b) xx[k++] = x[a] * x[b];
                }
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    if ((sigs >> s) & 1) {
                        double z[D], q = 0.0;
                        if constexpr (R == 0) {
#pragma unroll
                            for (int k = 0; k < NX; ++k) q += quad[s][k] * xx[k];
                        } else {
#pragma unroll
                            for (int a = 0; a < D; ++a) {
                                double zz = 0.0;
#pragma unroll
                                for (int b = 0; b < D; ++b) zz += it.lam[s][a * MAXD + b] * x[b];
                                z[a] = zz;
                                q += x[a] * zz;
                            }
                            q *= -0.5;
                        }
                        const double we = wa * exp(q);
                        if constexpr (F::V > 0) acc[s] += we;
                        if constexpr (R > 0) {
                            double He[N];
                            He[0] = 1.0;
#pragma unroll
                            for (int t = 1; t < N; ++t) {
                                double w = z[ht.piv[t]] * He[ht.par[t]];
#pragma unroll
                                for (int r = 0; r < D; ++r)
                                    if (r < ht.nred[t])
                                        w -= double(ht.rc[t][r]) * it.lam[s][ht.piv[t] * MAXD + ht.rj[t][r]] *
                                             He[ht.ridx[t][r]];
                                He[t] = w;
                            }
#pragma unroll
                            for (int k = F::V; k < F::NI; ++k)
                                acc[k * NS + s] = fma(we, He[F::N0 + k - F::V], acc[k * NS + s]);
                        }
                    }
                }
            } else {
                real v[NO];
#pragma unroll
                for (int o = 0; o < NO; ++o) v[o] = real(0);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    if ((sigs >> s) & 1) {
                        real z[D];
                        real q = 0;
#pragma unroll
                        for (int a = 0; a < D; ++a) {
                            real zz = 0;
#pragma unroll
                            for (int b = 0; b < D; ++b) zz += it.lam[s][a * MAXD + b] * x[b];
                            z[a] = zz;
                            q += x[a] * zz;
                        }
                        const real e = it.nrm[s] * exp(real(-0.5) * q);
                        real He[N];
                        He[0] = real(1);
#pragma unroll
                        for (int t = 1; t < N; ++t) {
                            real w = z[ht.piv[t]] * He[ht.par[t]];
#pragma unroll
                            for (int r = 0; r < D; ++r)
                                if (r < ht.nred[t])
                                    w -= real(ht.rc[t][r]) * it.lam[s][ht.piv[t] * MAXD + ht.rj[t][r]] * He[ht.ridx[t][r]];
                            He[t] = w;
                        }
                        if constexpr (F::dense) {
                            real pa = 0, pb = 0;
#pragma unroll
                            for (int t = 0; t < N; ++t) {
                                pa += Ws[s * N + t] * He[t];
                                pb += Ws[(MAXSIG + s) * N + t] * He[t];
                            }
                            v[0] += e * pa;
                            v[1] += e * pb;
                        } else {
#pragma unroll
                            for (int o = 0; o < NO; ++o) v[o] = fma(e, Ws[o * MAXSIG + s] * He[F::at(o)], v[o]);
                        }
                    }
                }
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    if constexpr (dbl) {
                        acc[o] = fma(wa, v[o], acc[o]);
                    } else {   // two-sum of the pair and the unrounded product
                        const float s = fmaf(wa, v[o], acc[o].h);
                        const float b = s - acc[o].h;
                        acc[o].l += (acc[o].h - (s - b)) + fmaf(wa, v[o], -b);
                        acc[o].h = s;
                    }
                }
            }
        }
        double* part = jb.partial + it.part0 +
                       (long long)NSUM * ((long long)(tix - it.tile0) * (dbl ? kLagSlices : 1) + (dbl ? s0 + warp : 0));
        if constexpr (dbl) {
            warp_sums_all<0, NSUM>(
                acc, lane, [](double a, double b) { return a + b; },
                [](double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }, [&](int o, double x) { part[o] = x; });
        } else {
            warp_sums_all<0, NO>(
                acc, lane, [](DFloat a, DFloat b) { return df_add(a, b); },
                [](DFloat a, int o) {
                    return DFloat{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
                },
                [&](int o, DFloat x) { red[warp][o] = x; });
            __syncthreads();
            if (threadIdx.x < NO) {
                DFloat t = red[0][threadIdx.x];
                for (int w = 1; w < 8; ++w) t = df_add(t, red[w][threadIdx.x]);
                part[threadIdx.x] = (double)t.h + (double)t.l;
            }
        }
        // the item's last block adds its partials: 256 shares (whatever the
        // block's size) of every 256 / NQ-th slot, then a fixed tree
        if (dbl || threadIdx.x < NO) __threadfence();   // the threads that wrote them
        __syncthreads();
        if (threadIdx.x == 0)
            lastone = atomicAdd(jb.done + tl.item, 1u) == (unsigned)(it.ntile * per) - 1u;
        __syncthreads();
        if (!lastone) continue;
        __threadfence();
        constexpr int NQ = NSUM <= 1 ? 1 : NSUM <= 2 ? 2 : NSUM <= 4 ? 4 : NSUM <= 8 ? 8 : NSUM <= 16 ? 16
                           : NSUM <= 32 ? 32 : 64;
        static_assert(NSUM <= 64, "a share of the final sum per kernel");
        const int slots = it.ntile * (dbl ? kLagSlices : 1);
        const double* all = jb.partial + it.part0;
        for (int t = threadIdx.x; t < 256; t += blockDim.x) {
            const int o = t % NQ;
            double sum = 0.0;
            if (o < NSUM)
                for (int k = t / NQ; k < slots; k += 256 / NQ) sum += __ldcg(all + (long long)k * NSUM + o);
            fin[t] = sum;
        }
        __syncthreads();
        for (int h = 128; h >= NQ; h >>= 1) {
            for (int t = threadIdx.x; t < h; t += blockDim.x) fin[t] += fin[t + h];
            __syncthreads();
        }
        for (int o = threadIdx.x; o < NO; o += blockDim.x)
            if (o < it.nout) {
                double v = 0.0;
                if constexpr (late) {
                    for (int s = 0; s < NS; ++s)
                        if ((sigs >> s) & 1) v += (Ws[o * MAXSIG + s] * it.nrm[s]) * fin[F::sum_of(o) * NS + s];
                } else {
                    v = fin[o];
                }
                jb.out[it.out0 + o] = v * it.scale;
            }
    }
}

template <typename real, int D, int R, int NV, int SG>
__global__ void __launch_bounds__(256) k_lag(const __grid_constant__ LagJob<real> jb) {
    lag_tiles<real, D, R, NV, SG>(jb);
}

// FP32 groups with d <= 2 are held to 64 registers, four CTAs an SM (512 data
// sets x 16 bandwidths 122 us, against 148 with the compiler's 75); with d = 3
// the same cap (or three CTAs) is slower than the compiler's 126 (psi_4 with
// tiles of 1024 points 91 and 82 us against 78, SCV gradients 18 and 15 against
// 12).
template <typename real, int D, int R, int NV>
__global__ void __launch_bounds__(256, 4) k_lag_occ4(const __grid_constant__ LagJob<real> jb) {
    lag_tiles<real, D, R, NV, MAXSIG>(jb);
}

// dense forms instantiated for (d, R): FP32 d <= 2 up to R = 8, d = 3 up to 6,
// d = 4 up to 4; FP64 the same except d = 3 up to 4 (register budget of the
// Hermite table)
static int lag_rmax(int d, bool dbl) {
    switch (d) {
        case 1:
        case 2: return 8;
        case 3: return dbl ? 4 : 6;
        case 4: return 4;
        default: return -1;
    }
}

template <typename real, int D, int R, int NV>
static cudaError_t lag_go(const LagJob<real>& j, cudaStream_t st) {
    if constexpr (sizeof(real) == 4 && D <= 2 && NV >= 0)
        k_lag_occ4<real, D, R, NV><<<j.grid, j.block, 0, st>>>(j);
    else if (sizeof(real) == 8 && NV == 0 && R == 2 && j.covs == 1)   // (4-D: 48 us a call, 55 with two)
        k_lag<real, D, R, NV, (sizeof(real) == 8 && NV == 0 && R == 2) ? 1 : MAXSIG><<<j.grid, j.block, 0, st>>>(j);
    else if (sizeof(real) == 8 && NV >= 0 && R <= 2 && j.covs == 2)
        k_lag<real, D, R, NV, (sizeof(real) == 8 && NV >= 0 && R <= 2) ? 2 : MAXSIG><<<j.grid, j.block, 0, st>>>(j);
    else
        k_lag<real, D, R, NV, MAXSIG><<<j.grid, j.block, 0, st>>>(j);
    return cudaGetLastError();
}

template <typename real, int D>
static cudaError_t lag_d(int R, int nv, const LagJob<real>& j, cudaStream_t st) {
    constexpr bool dbl = sizeof(real) == 8;
    if (nv >= 0) {
        if (!lag_single_form(D, R, nv, 1)) return cudaErrorNotSupported;
        if (R == 4) return lag_go<real, D, 4, 0>(j, st);
        switch (nv) {
            case 0: return lag_go<real, D, 2, 0>(j, st);
            case 1: return R == 0 ? lag_go<real, D, 0, 1>(j, st) : lag_go<real, D, 2, 1>(j, st);
            default: return R == 0 ? lag_go<real, D, 0, 2>(j, st) : lag_go<real, D, 2, 2>(j, st);
        }
    }
    const int Re = (R + 1) & ~1;
    if (Re > lag_rmax(D, dbl)) return cudaErrorNotSupported;
    switch (Re) {
        case 0: return lag_go<real, D, 0, -1>(j, st);
        case 2: return lag_go<real, D, 2, -1>(j, st);
        case 4: return lag_go<real, D, 4, -1>(j, st);
        case 6:
            if constexpr (D <= 2 || (D == 3 && !dbl)) return lag_go<real, D, 6, -1>(j, st);
            return cudaErrorNotSupported;
        case 8:
            if constexpr (D <= 2) return lag_go<real, D, 8, -1>(j, st);
            return cudaErrorNotSupported;
        default: return cudaErrorNotSupported;
    }
}

template <typename real>
cudaError_t launch_lag(int d, int R, int nv, const LagJob<real>& j, cudaStream_t st) {
    if (j.ntiles <= 0) return cudaSuccess;
    if (j.grid < 1) return cudaErrorInvalidValue;
    const bool slices_ok = sizeof(real) == 8 && (j.block == 32 || j.block == 64 || j.block == 128);
    if (j.block != 256 && !slices_ok) return cudaErrorInvalidValue;
    switch (d) {
        case 1: return lag_d<real, 1>(R, nv, j, st);
        case 2: return lag_d<real, 2>(R, nv, j, st);
        case 3: return lag_d<real, 3>(R, nv, j, st);
        case 4: return lag_d<real, 4>(R, nv, j, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace kdefft
