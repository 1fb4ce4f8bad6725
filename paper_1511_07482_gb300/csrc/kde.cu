// The kernel density estimate on the grid and the cross term of the
// integrated squared error against a normal mixture, for the binned sample.
//
//   kde_table the stencil K_H(delta (.) l)
//   kde_tile  f_hat(g) = n^-1 sum_{|l_k| <= L_k} c_{g - l} K_H(delta (.) l) at
//             every grid node g (the binned estimator, the convolution that
//             Eqs. 19-24 evaluate through the FFT, truncated as in Eq. 26),
//             a tile of nodes per block, compensated FP32 sums written as
//             FP64.  The direct sum keeps the relative accuracy of small
//             values (and exact zeros beyond the support), which a transform
//             does not.
//   mix_dot   sum_g c_g sum_m w_m phi_{S_m}(x_g - mu_m) (FP64) for a batch of
//             mixtures.
#include "devutil.cuh"
#include "engine.cuh"

namespace kdefft {

// K_H(delta (.) l) for every stencil point l, last axis fastest, rounded from
// FP64 (the table has prod (2 L_k + 1) entries: 12 K to 60 K FP64 exponentials
// for a 3-D estimate, milliseconds on the host).
__global__ void __launch_bounds__(256) k_kde_table(KdeDesc g, KdeKernel kn, float* __restrict__ tab) {
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < g.nstencil;
         s += (long long)gridDim.x * blockDim.x) {
        long long r = s;
        double x[MAXD] = {0.0, 0.0, 0.0, 0.0};
        for (int k = g.d - 1; k >= 0; --k) {
            const int w = 2 * g.L[k] + 1;
            x[k] = g.delta[k] * (double)((int)(r % w) - g.L[k]);
            r /= w;
        }
        double q = 0.0;
        for (int a = 0; a < g.d; ++a)
            for (int b = 0; b < g.d; ++b) q += x[a] * kn.lam[a * MAXD + b] * x[b];
        tab[s] = (float)(kn.nrm * exp(-0.5 * q));
    }
}

// The estimate on a tile of 2 BY rows (axis d - 2) by BX * T nodes (axis
// d - 1) at one index of the outer axes; a thread has T consecutive nodes of
// two rows (packed pairs, BY rows apart), and KZ threads share each of them,
// every KZ-th stencil row theirs.
//
// It is bound by the FP32 pipes: a node takes prod (2 L_k + 1) terms c K (12 K
// to 60 K of them for a sample of 1e6 points on 128^3), four operations each:
//   s = fma(c, K, h);  l += fma(c, K, h - s);  h = s
// Where h >= c K (all terms are >= 0), h - s is exact and the second product
// sum is the rounding error of h + c K with the product itself unrounded, so
// that the pair h + l holds the sum to about 44 bits.  Where h is still
// smaller than the largest term that the next U taps can bring (the first
// rows of a stencil, the edge of a sample) the warp takes these taps with the
// seven operations of Knuth's two-sum, which needs no order.  Everything else
// is kept off the arithmetic's way: a block stages the counts of its tile and
// halo, paired as the nodes are, and the taps of up to CY x CX
// stencil columns in shared memory, a thread holds a window of T + U pairs in
// registers and takes U taps against it, and rows and windows without any
// counts (most of the box around a sample) are left out.  K_H is even, so the
// counts are read at g + l.
// 128^3 grid, sample of 1e6 points, 37 x 35 x 31 taps: 9.1 ms (406 ms for one
// node a thread with 64-bit indices and global loads), 21 x 25 x 25 taps 3.4
// ms (133 ms); 8e12 to 9e12 terms/s counting the ones left out, FP32 pipes 60 %
// busy.  Scalar operations instead of packed ones: 4.4 ms.  256^2, 77 x 69
// taps: 163 us (2203 us), 33 x 70 x 51, 11 x 21 x 13 taps: 205 us (2441 us).
constexpr int kKdeCY = 16, kKdeCX = 32, kKdeU = 4;

template <int T, int BX, int BY, int KZ>
__global__ void __launch_bounds__(BX* BY* KZ) k_kde_tile(const float* __restrict__ counts, KdeDesc g,
                                                         const float* __restrict__ ktab, double* __restrict__ out,
                                                         unsigned int ntx, unsigned int nty, long long ntile) {
    constexpr int NT = BX * BY * KZ, U = kKdeU;
    // pairs per staged row: 2 (mod 4), so that rows are 16-byte aligned and a
    // quarter warp's 16-byte loads (four threads of two rows, 32 bytes apart)
    // fall on distinct banks
    constexpr int PITCH = (BX * T + kKdeCX + 3) / 4 * 4 + 2;
    constexpr int ROWS = BY + kKdeCY - 1;              // staged pairs: rows r and r + BY
    static_assert(U % T == 0 && NT % 32 == 0 && (BX * BY) % 32 == 0, "tile shape");
    static_assert(BY == 1 || (BX == 8 && BY % 4 == 0), "lane order below");
    __shared__ __align__(16) float2 tin[ROWS * PITCH];
    __shared__ __align__(16) float2 tk[kKdeCY * kKdeCX];
    __shared__ float gtop[ROWS][BX + kKdeCX / T + 1];   // largest count of each T staged
    __shared__ float ktop[kKdeCY][kKdeCX / U];          // largest of each U taps
    __shared__ int nonzero[ROWS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tz = threadIdx.x / (BX * BY);
    int tx = threadIdx.x % BX, ty = 0;
    if constexpr (BY > 1) {   // a warp: 8 x 4 threads, each quarter 4 x 2 of them
        tx = (lane & 3) | ((lane >> 1) & 4);
        ty = ((warp * 4) % BY) + ((lane >> 2) & 1) + ((lane >> 3) & 2);
    }
    const int d = g.d;
    const int Mx = (int)g.M[d - 1], Lx = g.L[d - 1], Sx = 2 * Lx + 1;
    const int My = d >= 2 ? (int)g.M[d - 2] : 1, Ly = d >= 2 ? g.L[d - 2] : 0, Sy = 2 * Ly + 1;
    const int Mo1 = d >= 3 ? (int)g.M[d - 3] : 1, Lo1 = d >= 3 ? g.L[d - 3] : 0;   // inner outer axis
    const int Mo0 = d >= 4 ? (int)g.M[0] : 1, Lo0 = d >= 4 ? g.L[0] : 0;
    const int outer = Mo0 * Mo1;
    for (long long tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int x0 = (int)(tile % ntx) * (BX * T);
        const int y0 = (int)((tile / ntx) % nty) * (2 * BY);
        // outer indices from the middle outwards: the tiles with the most
        // counts around them start first
        const int oi = (int)(tile / ntx / nty);
        const int o = (oi & 1) ? (outer - 1) / 2 - (oi + 1) / 2 + (outer & 1 ? 0 : 1) : (outer - 1) / 2 + oi / 2 + (outer & 1 ? 0 : 1);
        const int o1 = o % Mo1, o0 = o / Mo1;
        f32x2 h[T], l[T];
#pragma unroll
        for (int i = 0; i < T; ++i) h[i] = l[i] = 0ull;
        const int a0 = max(-Lo0, -o0), b0 = min(Lo0, Mo0 - 1 - o0);
        const int a1 = max(-Lo1, -o1), b1 = min(Lo1, Mo1 - 1 - o1);
        for (int l0 = a0; l0 <= b0; ++l0)
            for (int l1 = a1; l1 <= b1; ++l1) {
                const float* slab = counts + ((long long)(o0 + l0) * Mo1 + (o1 + l1)) * My * Mx;
                const float* ks = ktab + ((long long)(l0 + Lo0) * (2 * Lo1 + 1) + (l1 + Lo1)) * Sy * Sx;
                // rows y0 + jy - Ly .. of the slab that some node of the tile reads
                const int jlo = max(0, Ly - (y0 + 2 * BY - 1)), jhi = min(Sy, Ly + My - y0);
                for (int jy = jlo; jy < jhi; jy += kKdeCY) {
                    const int ny = min(kKdeCY, jhi - jy);
                    for (int jx = 0; jx < Sx; jx += kKdeCX) {
                        const int nx = min(kKdeCX, Sx - jx);
                        const int nxp = (nx + U - 1) / U * U;   // taps rounded up, zeros past nx
                        const int ncol = BX * T + nxp;
                        if (x0 + jx - Lx >= Mx || x0 + jx - Lx + ncol <= 0) continue;   // off the grid: no counts
                        __syncthreads();   // the readers of the previous chunk are done
                        int mine = 0;
                        for (int r = warp; r < BY + ny - 1; r += NT / 32) {
                            const int y = y0 + jy - Ly + r;
                            const bool in0 = y >= 0 && y < My, in1 = y + BY >= 0 && y + BY < My;
                            const float* src = slab + (long long)y * Mx;
                            const float* src1 = src + (long long)BY * Mx;
                            int any = 0;
                            for (int c0 = 0; c0 < ncol; c0 += 32) {
                                const int c = c0 + lane, x = x0 + jx - Lx + c;
                                const bool inx = c < ncol && x >= 0 && x < Mx;
                                const float2 v = make_float2(in0 && inx ? src[x] : 0.f, in1 && inx ? src1[x] : 0.f);
                                if (c < ncol) tin[r * PITCH + c] = v;
                                float m = fmaxf(v.x, v.y);
#pragma unroll
                                for (int k = 1; k < T; k *= 2) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, k));
                                if (c < ncol && c % T == 0) gtop[r][c / T] = m;
                                any |= m != 0.f;
                            }
                            any = __any_sync(0xffffffffu, any);
                            if (lane == 0) nonzero[r] = any;
                            mine |= any;
                        }
                        for (int t0 = warp * 32; t0 < ny * nxp; t0 += NT) {
                            const int t = t0 + lane, r = t / nxp, c = t - r * nxp;
                            const float v = (r < ny && c < nx) ? ks[(long long)(jy + r) * Sx + jx + c] : 0.f;
                            if (r < ny) tk[r * kKdeCX + c] = make_float2(v, v);
                            float m = v;
#pragma unroll
                            for (int k = 1; k < U; k *= 2) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, k));
                            if (r < ny && c % U == 0) ktop[r][c / U] = m;
                        }
                        if (!__syncthreads_or(mine)) continue;
                        for (int r = tz; r < ny; r += KZ) {
                            const int row = ty + r;
                            if (!__any_sync(0xffffffffu, nonzero[row])) continue;
                            const f32x2* p = reinterpret_cast<const f32x2*>(tin + row * PITCH + tx * T);
                            const f32x2* kp = reinterpret_cast<const f32x2*>(tk + r * kKdeCX);
                            const float* gt = &gtop[row][tx];
                            auto smallest = [&]() {
                                float2 v = unpack2(h[0]);
                                float m = fminf(v.x, v.y);
#pragma unroll
                                for (int i = 1; i < T; ++i) {
                                    v = unpack2(h[i]);
                                    m = fminf(m, fminf(v.x, v.y));
                                }
                                return m;
                            };
                            float least = smallest();   // the sums only grow: a bound for the whole row
                            f32x2 w[T + U];
                            float last = gt[0];
#pragma unroll
                            for (int i = 0; i < T; ++i) w[i] = p[i];
#pragma unroll 2
                            for (int t = 0; t < nxp; t += U) {
                                f32x2 kk[U];
                                float top = last;
#pragma unroll
                                for (int i = 0; i < U; i += 2) {
                                    const ulonglong2 kv = *reinterpret_cast<const ulonglong2*>(kp + t + i);
                                    kk[i] = kv.x;
                                    kk[i + 1] = kv.y;
                                    if constexpr (T > 1) {
                                        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p + t + T + i);
                                        w[T + i] = v.x;
                                        w[T + i + 1] = v.y;
                                    } else {
                                        w[T + i] = p[t + T + i];
                                        w[T + i + 1] = p[t + T + i + 1];
                                    }
                                }
#pragma unroll
                                for (int i = 0; i < U / T; ++i) {
                                    last = gt[t / T + 1 + i];
                                    top = fmaxf(top, last);
                                }
                                if (__any_sync(0xffffffffu, top * ktop[r][t / U] > least)) {
#pragma unroll
                                    for (int u = 0; u < U; ++u)
#pragma unroll
                                        for (int i = 0; i < T; ++i) {
                                            const f32x2 s = fma2(w[u + i], kk[u], h[i]);
                                            const f32x2 b = sub2(h[i], s);   // minus what h gained
                                            l[i] = add2(l[i], add2(sub2(h[i], add2(s, b)), fma2(w[u + i], kk[u], b)));
                                            h[i] = s;
                                        }
                                    least = smallest();
                                } else if (__any_sync(0xffffffffu, top != 0.f)) {
#pragma unroll
                                    for (int u = 0; u < U; ++u)
#pragma unroll
                                        for (int i = 0; i < T; ++i) {
                                            const f32x2 s = fma2(w[u + i], kk[u], h[i]);
                                            l[i] = add2(l[i], fma2(w[u + i], kk[u], sub2(h[i], s)));
                                            h[i] = s;
                                        }
                                }
#pragma unroll
                                for (int i = 0; i < T; ++i) w[i] = w[U + i];
                            }
#pragma unroll
                            for (int i = 0; i < T; ++i) {   // the pair normalised, so that l stays small
                                const f32x2 s = add2(h[i], l[i]);
                                l[i] = sub2(l[i], sub2(s, h[i]));
                                h[i] = s;
                            }
                        }
                    }
                }
            }
        if constexpr (KZ > 1) {   // the KZ shares of a node, in order
            static_assert(sizeof(tin) >= sizeof(f32x2) * 2 * T * BX * BY * (KZ - 1), "shares fit the staged rows");
            f32x2* part = reinterpret_cast<f32x2*>(tin);
            __syncthreads();
            if (tz > 0)
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    f32x2* q = part + ((size_t)((tz - 1) * T + i) * 2) * (BX * BY) + ty * BX + tx;
                    q[0] = h[i];
                    q[BX * BY] = l[i];
                }
            __syncthreads();
            if (tz == 0)
                for (int z = 1; z < KZ; ++z)
#pragma unroll
                    for (int i = 0; i < T; ++i) {
                        const f32x2* q = part + ((size_t)((z - 1) * T + i) * 2) * (BX * BY) + ty * BX + tx;
                        const float2 ha = unpack2(h[i]), la = unpack2(l[i]), hb = unpack2(q[0]), lb = unpack2(q[BX * BY]);
                        const DFloat x = df_add({ha.x, la.x}, {hb.x, lb.x}), y = df_add({ha.y, la.y}, {hb.y, lb.y});
                        h[i] = pack2(x.h, y.h);
                        l[i] = pack2(x.l, y.l);
                    }
        }
        const int y = y0 + ty;
        if (tz == 0 && y < My) {
            double* dst = out + ((long long)o * My + y) * Mx + x0 + tx * T;
#pragma unroll
            for (int i = 0; i < T; ++i)
                if (x0 + tx * T + i < Mx) {
                    const float2 hv = unpack2(h[i]), lv = unpack2(l[i]);
                    dst[i] = ((double)hv.x + (double)lv.x) * g.inv_n;
                    if (y + BY < My) dst[(long long)BY * Mx + i] = ((double)hv.y + (double)lv.y) * g.inv_n;
                }
        }
    }
}

template <int T, int BX, int BY, int KZ>
static cudaError_t kde_go(const float* counts, const KdeDesc& g, const float* ktab, double* out, cudaStream_t st) {
    const long long Mx = g.M[g.d - 1], My = g.d >= 2 ? g.M[g.d - 2] : 1;
    const long long ntx = (Mx + BX * T - 1) / (BX * T), nty = (My + 2 * BY - 1) / (2 * BY);
    const long long ntile = ntx * nty * (g.ncells / (Mx * My));
    const unsigned grid = (unsigned)(ntile < (1LL << 20) ? ntile : (1LL << 20));
    k_kde_tile<T, BX, BY, KZ><<<grid, BX * BY * KZ, 0, st>>>(counts, g, ktab, out, (unsigned)ntx, (unsigned)nty, ntile);
    return cudaGetLastError();
}

cudaError_t launch_kde_table(const KdeDesc& g, const KdeKernel& kn, float* tab, cudaStream_t st) {
    const long long b = (g.nstencil + 255) / 256;
    k_kde_table<<<(unsigned)(b < 4096 ? b : 4096), 256, 0, st>>>(g, kn, tab);
    return cudaGetLastError();
}

cudaError_t launch_kde_grid(const float* counts, const KdeDesc& g, const float* ktab, double* out, int nsm,
                            cudaStream_t st) {
    if (g.ncells <= 0) return cudaSuccess;
    const long long Mx = g.M[g.d - 1], My = g.d >= 2 ? g.M[g.d - 2] : 1, outer = g.ncells / (Mx * My);
    if (g.d == 1) return kde_go<1, 32, 1, 1>(counts, g, ktab, out, st);
    // Nodes that a tile shape computes, its padding included, times the cost
    // of a term in it (loads a term grow as 1 / T), but no less than what four
    // blocks an SM compute meanwhile: wide tiles for large grids, a stencil
    // split over four warps and narrow tiles for small grids and short axes.
    auto cost = [&](int tx, int ty, double per) {
        const double padded = (double)((Mx + tx - 1) / tx * tx) * (double)((My + ty - 1) / ty * ty) * (double)outer;
        const double full = (double)nsm * 4.0 * tx * ty;
        return per * (padded > full ? padded : full);
    };
    const double wide = cost(32, 32, 1.0), split = cost(32, 8, 1.1), narrow = cost(16, 8, 1.4);
    if (wide <= split && wide <= narrow) return kde_go<4, 8, 16, 1>(counts, g, ktab, out, st);
    if (split <= narrow) return kde_go<4, 8, 4, 4>(counts, g, ktab, out, st);
    return kde_go<2, 8, 4, 4>(counts, g, ktab, out, st);
}

// sum_g c_g sum_m w_m phi_{S_m}(x_g - mu_m) for many mixtures (one per
// bandwidth), nb blocks each.  Bound by the FP64 pipe (an exponential and a
// quadratic form per component and cell with counts, about 30 operations), so
// all mixtures are one launch that fills the SMs, and lanes are not spent on
// cells without counts (two thirds of the box around a sample, and more than
// half of the lanes of the warps that have any): a block queues the cells with
// counts of its 32 segments of 8 a round and takes 256 of them at a time.  Of
// every nb segments a block has one, a different one each time: in a fixed
// order its segments lie in the same columns, and blocks (and with them the
// SMs, whose blocks differ by multiples of nb) had up to eight times the work
// of others.
// The mixture's last block adds its nb partials in block order.
// 32 bandwidths, three components, a 101^2 grid: 36 us (55 us with a thread per
// cell; 512 us in 32 launches, with an upload, a copy back and a host wait each).
template <int D>
__global__ void __launch_bounds__(256) k_mix_dot(const __grid_constant__ MixJob jb) {
    constexpr int NQ = D * (D + 1) / 2;
    __shared__ double mu[kMixMax][D], quad[kMixMax][NQ], amp[kMixMax];
    __shared__ unsigned int qcell[512];
    __shared__ float qcount[512];
    __shared__ int nwarp[8];
    __shared__ double red[8];
    __shared__ int lastone;
    const KdeDesc& g = jb.g;
    const int h = blockIdx.x / jb.nb, b = blockIdx.x % jb.nb, K = jb.ncomp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const MixComp* comps = jb.comps + (long long)h * K;
    for (int m = threadIdx.x; m < K; m += blockDim.x) {
        for (int k = 0; k < D; ++k) mu[m][k] = comps[m].mu[k];
        int v = 0;   // -z^T lam z / 2 on the upper triangle
        for (int i = 0; i < D; ++i)
            for (int k = i; k < D; ++k)
                quad[m][v++] = -0.5 * (i == k ? comps[m].lam[i * MAXD + i]
                                              : comps[m].lam[i * MAXD + k] + comps[m].lam[k * MAXD + i]);
        amp[m] = comps[m].w * comps[m].nrm;
    }
    double acc = 0.0;
    auto take = [&](unsigned int cell, float cv) {
        double x[D];
#pragma unroll
        for (int k = D - 1; k >= 0; --k) {
            const unsigned int M = (unsigned int)g.M[k], r = cell / M;
            x[k] = g.lo[k] + g.delta[k] * (double)(int)(cell - r * M);
            cell = r;
        }
        double f = 0.0;
        for (int m = 0; m < K; ++m) {
            double z[D], q = 0.0;
#pragma unroll
            for (int k = 0; k < D; ++k) z[k] = x[k] - mu[m][k];
            int v = 0;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                double t = 0.0;
#pragma unroll
                for (int k = i; k < D; ++k) t += quad[m][v++] * z[k];
                q += z[i] * t;
            }
            f += amp[m] * exp(q);
        }
        acc += (double)cv * f;
    };
    const int seg = threadIdx.x >> 3;
    const long long step = 32LL * jb.nb, nseg = (g.ncells + 7) / 8;
    const long long mine = (long long)seg * jb.nb + (b + (long long)seg * (jb.nb * 5LL / 8)) % jb.nb;
    int held = 0;   // queued cells, below 256 between rounds
    for (long long s0 = 0; s0 < nseg; s0 += step) {
        const long long cell = (s0 + mine) * 8 + (lane & 7);
        const float cv = cell < g.ncells ? jb.counts[cell] : 0.f;
        const unsigned int any = __ballot_sync(0xffffffffu, cv != 0.f);
        if (lane == 0) nwarp[warp] = __popc(any);
        __syncthreads();   // also: the tables are written, the last round's queue is moved
        int at = held;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const int n = nwarp[w];
            if (w < warp) at += n;
            held += n;
        }
        if (cv != 0.f) {
            at += __popc(any & ((1u << lane) - 1u));
            qcell[at] = (unsigned int)cell;
            qcount[at] = cv;
        }
        __syncthreads();
        if (held >= 256) {
            take(qcell[threadIdx.x], qcount[threadIdx.x]);
            held -= 256;
            __syncthreads();
            if (threadIdx.x < held) {
                qcell[threadIdx.x] = qcell[256 + threadIdx.x];
                qcount[threadIdx.x] = qcount[256 + threadIdx.x];
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < held) take(qcell[threadIdx.x], qcount[threadIdx.x]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        jb.partial[(long long)h * jb.nb + b] = t;
        __threadfence();
        lastone = atomicAdd(jb.done + h, 1u) == (unsigned)jb.nb - 1u;
    }
    __syncthreads();
    if (!lastone || threadIdx.x >= 32) return;
    __threadfence();
    double t = 0.0;   // lane l takes the partials l, l + 32, .., then a fixed tree
    for (int k = threadIdx.x; k < jb.nb; k += 32) t += __ldcg(jb.partial + (long long)h * jb.nb + k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) jb.out[h] = t;
}

cudaError_t launch_mix_dot(const MixJob& j, int nH, cudaStream_t st) {
    if (nH <= 0) return cudaSuccess;
    const long long blocks = (long long)j.nb * nH;
    if (j.ncomp < 1 || j.ncomp > kMixMax || j.nb < 1 || blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    switch (j.g.d) {
        case 1: k_mix_dot<1><<<(unsigned)blocks, 256, 0, st>>>(j); break;
        case 2: k_mix_dot<2><<<(unsigned)blocks, 256, 0, st>>>(j); break;
        case 3: k_mix_dot<3><<<(unsigned)blocks, 256, 0, st>>>(j); break;
        case 4: k_mix_dot<4><<<(unsigned)blocks, 256, 0, st>>>(j); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace kdefft
