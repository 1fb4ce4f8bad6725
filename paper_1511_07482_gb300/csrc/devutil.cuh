// Device helpers shared by the kernel files (engine.cu, lag.cu): compensated
// FP32 accumulation, block reductions to FP64, and the compile-time
// multivariate Hermite recurrence.  Internal; not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

namespace kdefft {

// ---- accumulation.  FP64 arithmetic is slow on this part, so FP32 sums
// carry an error term (two-sum / double-float): the pair (h, l) holds the
// sum to about u^2 relative, and it becomes FP64 once per block.
struct DFloat {
    float h, l;
};
__device__ __forceinline__ DFloat df_two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ DFloat df_add(DFloat a, DFloat b) {
    const DFloat s = df_two_sum(a.h, b.h);
    const float e = s.l + (a.l + b.l);
    const float h = s.h + e;
    return {h, e - (h - s.h)};
}
// a b for FP32 a, b as an unevaluated pair: exact (the fused multiply-add
// gives the product's rounding error)
__device__ __forceinline__ DFloat df_prod(float a, float b) {
    const float p = a * b;
    return DFloat{p, fmaf(a, b, -p)};
}
// (a.h + a.l)(b.h + b.l) to a few units of 2^-44 relative
__device__ __forceinline__ DFloat df_mul(DFloat a, DFloat b) {
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)));
    const float s = p + e;
    return DFloat{s, e - (s - p)};
}
// (a.h + a.l) b for an FP32 b
__device__ __forceinline__ DFloat df_mulf(DFloat a, float b) {
    const float p = a.h * b;
    const float e = fmaf(a.l, b, fmaf(a.h, b, -p));
    const float s = p + e;
    return DFloat{s, e - (s - p)};
}
__device__ __forceinline__ void df_acc(DFloat& a, float x) {
    const DFloat s = df_two_sum(a.h, x);
    const float e = s.l + a.l;
    a.h = s.h + e;
    a.l = e - (a.h - s.h);
}

// ---- an FP32 pair x = h + l with |l| <= ulp(h) / 2 as an arithmetic type
// (about 44 significant bits), so that templated transforms can run on the
// FP32 pipes where FP64 would be slow.  Sums renormalise through two-sum,
// products through the fused multiply-add's exact rounding error; both keep
// the error a few units of 2^-44 of the operands' magnitudes, which is what
// a transform's error bound needs.  Constants come from double literals,
// split at compile time.
struct dflt {
    float h, l;
    __host__ __device__ constexpr dflt() : h(0.f), l(0.f) {}
    __host__ __device__ constexpr dflt(float a, float b) : h(a), l(b) {}
    __host__ __device__ constexpr explicit dflt(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
};
__device__ __forceinline__ dflt operator+(dflt a, dflt b) {
    const float s = a.h + b.h;
    const float bb = s - a.h;
    const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
    const float h = s + e;
    return dflt(h, e - (h - s));
}
__device__ __forceinline__ dflt operator-(dflt a) { return dflt(-a.h, -a.l); }
__device__ __forceinline__ dflt operator-(dflt a, dflt b) { return a + (-b); }
__device__ __forceinline__ dflt operator*(dflt a, dflt b) {
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)));
    const float h = p + e;
    return dflt(h, e - (h - p));
}
__device__ __forceinline__ double to_double(dflt a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double to_double(double a) { return a; }
// Two FP32 values in a 64-bit register pair and the packed operations on
// them (both halves rounded as the scalar operations round): the FP32 pipes
// take a packed instruction in two cycles, so arithmetic that fills them
// leaves every other issue slot to loads and control.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// a - b: one rounding, as the subtraction's
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pack2(-1.f, -1.f), a); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 swap2(f32x2 a) {
    const float2 v = unpack2(a);
    return pack2(v.y, v.x);
}

// Complex FP32 pair, of double2's size: h holds the leading parts of (x, y), l
// the remainders, so that both components take each operation together (the
// sequences are dflt's, so are the bits).
struct __align__(16) dcplx {
    f32x2 h, l;
};
__device__ __forceinline__ dcplx cadd(dcplx a, dcplx b) {
    const f32x2 s = add2(a.h, b.h);
    const f32x2 bb = sub2(s, a.h);
    const f32x2 e = add2(add2(sub2(a.h, sub2(s, bb)), sub2(b.h, bb)), add2(a.l, b.l));
    const f32x2 h = add2(s, e);
    return dcplx{h, sub2(e, sub2(h, s))};
}
__device__ __forceinline__ dcplx csub(dcplx a, dcplx b) {
    const f32x2 s = sub2(a.h, b.h);
    const f32x2 bb = sub2(s, a.h);
    const f32x2 e = add2(sub2(sub2(a.h, sub2(s, bb)), add2(b.h, bb)), sub2(a.l, b.l));
    const f32x2 h = add2(s, e);
    return dcplx{h, sub2(e, sub2(h, s))};
}
// component-wise product (a.x b.x, a.y b.y)
__device__ __forceinline__ dcplx pmul(dcplx a, dcplx b) {
    const f32x2 p = mul2(a.h, b.h);
    const f32x2 e = fma2(a.h, b.l, fma2(a.l, b.h, fma2(a.h, b.h, neg2(p))));
    const f32x2 h = add2(p, e);
    return dcplx{h, sub2(e, sub2(h, p))};
}
__device__ __forceinline__ dcplx cmul(dcplx a, dcplx b) {   // a (x of b) + i a (y of b)
    const float2 bh = unpack2(b.h), bl = unpack2(b.l);
    return cadd(pmul(a, dcplx{pack2(bh.x, bh.x), pack2(bl.x, bl.x)}),
                pmul(dcplx{swap2(a.h), swap2(a.l)}, dcplx{pack2(-bh.y, bh.y), pack2(-bl.y, bl.y)}));
}
__device__ __forceinline__ dcplx cconj(dcplx a) {
    return dcplx{a.h ^ 0x8000000000000000ull, a.l ^ 0x8000000000000000ull};
}
__device__ __forceinline__ dcplx cmi(dcplx a) { return cconj(dcplx{swap2(a.h), swap2(a.l)}); }   // -i a
__device__ __forceinline__ dcplx cscale(dflt s, dcplx a) {
    return pmul(dcplx{pack2(s.h, s.h), pack2(s.l, s.l)}, a);
}
__device__ __forceinline__ dcplx chalf(dcplx a) {
    return dcplx{mul2(a.h, pack2(0.5f, 0.5f)), mul2(a.l, pack2(0.5f, 0.5f))};
}
__device__ __forceinline__ dflt re(dcplx a) { return dflt(unpack2(a.h).x, unpack2(a.l).x); }
__device__ __forceinline__ dflt im(dcplx a) { return dflt(unpack2(a.h).y, unpack2(a.l).y); }
__device__ __forceinline__ dcplx cmake(dflt x, dflt y) { return dcplx{pack2(x.h, y.h), pack2(x.l, y.l)}; }
__device__ __forceinline__ dflt cnorm2(dcplx a) {
    const dcplx q = pmul(a, a);
    return re(q) + im(q);
}
__device__ __forceinline__ bool czero(dcplx a) { return (a.h & 0x7fffffff7fffffffull) == 0; }   // (l is zero where h is)
// the same names for double2
__device__ __forceinline__ double2 cconj(double2 a) { return double2{a.x, -a.y}; }
__device__ __forceinline__ double2 chalf(double2 a) { return double2{0.5 * a.x, 0.5 * a.y}; }
__device__ __forceinline__ double re(double2 a) { return a.x; }
__device__ __forceinline__ double im(double2 a) { return a.y; }
__device__ __forceinline__ double2 cmake(double x, double y) { return double2{x, y}; }

// The job whose block range holds block b, from the jobs' first blocks
// (ascending, first(0) = 0): every warp searches for itself, 32 places at a
// time (two rounds for 1024 jobs instead of ten dependent loads).
template <typename F>
__device__ __forceinline__ int job_of_warp(int n, long long b, F&& first) {
    const int lane = threadIdx.x & 31;
    int lo = 0, len = n;
    while (len > 1) {
        const int step = (len + 31) >> 5;
        const int at = lane * step;
        const bool before = at < len && first(lo + at) <= b;
        const int k = __popc(__ballot_sync(0xffffffffu, before)) - 1;
        lo += k * step;
        len = min(step, len - k * step);
    }
    return lo;
}

// per-thread accumulator of the spectral sums: DFloat in FP32 mode, double in FP64 mode
template <typename real>
struct SumAcc;
template <>
struct SumAcc<float> {
    DFloat a{0.f, 0.f}, b{0.f, 0.f};
    __device__ __forceinline__ void add(float x, float y) {
        df_acc(a, x);
        df_acc(b, y);
    }
};
template <>
struct SumAcc<double> {
    double a = 0.0, b = 0.0;
    __device__ __forceinline__ void add(double x, double y) {
        a += x;
        b += y;
    }
};

// block sum of a SumAcc; thread 0 receives the two totals as doubles.
// Contains __syncthreads (call from uniform control flow).
__device__ __forceinline__ void block_reduce_acc(const SumAcc<float>& s, double* out2) {
    __shared__ DFloat red[2][32];
    DFloat a = s.a, b = s.b;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        DFloat ta{__shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.l, o)};
        DFloat tb{__shfl_down_sync(0xffffffffu, b.h, o), __shfl_down_sync(0xffffffffu, b.l, o)};
        a = df_add(a, ta);
        b = df_add(b, tb);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        red[0][w] = a;
        red[1][w] = b;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = (l < nw) ? red[0][l] : DFloat{0.f, 0.f};
        b = (l < nw) ? red[1][l] : DFloat{0.f, 0.f};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            DFloat ta{__shfl_down_sync(0xffffffffu, a.h, o), __shfl_down_sync(0xffffffffu, a.l, o)};
            DFloat tb{__shfl_down_sync(0xffffffffu, b.h, o), __shfl_down_sync(0xffffffffu, b.l, o)};
            a = df_add(a, ta);
            b = df_add(b, tb);
        }
        if (l == 0) {
            out2[0] = (double)a.h + (double)a.l;
            out2[1] = (double)b.h + (double)b.l;
        }
    }
    __syncthreads();
}
template <typename real>
__device__ void block_reduce2(double a, double b, double* out2) {
    __shared__ double red[2][32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        red[0][w] = a;
        red[1][w] = b;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = (l < nw) ? red[0][l] : 0.0;
        b = (l < nw) ? red[1][l] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
        if (l == 0) {
            out2[0] = a;
            out2[1] = b;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void block_reduce_acc(const SumAcc<double>& s, double* out2) {
    block_reduce2<double>(s.a, s.b, out2);
}

// ------------------------------------------------------------ compile-time Hermite recurrence
// The same graded enumeration and recurrence as the constant-memory table,
// generated at compile time for fixed (D, R) so that the polynomials live in
// registers and every index is a constant.
constexpr int cx_binom(int n, int k) {
    long long c = 1;
    for (int i = 1; i <= k; ++i) c = c * (n - k + i) / i;
    return (int)c;
}

template <int D, int R>
struct HTab {
    static constexpr int N = cx_binom(D + R, D);
    int al[N][D];
    int piv[N];
    int par[N];
    int nred[N];
    int rj[N][D];
    int rc[N][D];
    int ridx[N][D];
    constexpr int index_of(const int* a) const {
        for (int t = 0; t < N; ++t) {
            bool eq = true;
            for (int k = 0; k < D; ++k) eq = eq && (al[t][k] == a[k]);
            if (eq) return t;
        }
        return -1;
    }
    constexpr HTab() : al(), piv(), par(), nred(), rj(), rc(), ridx() {
        int n = 0;
        for (int o = 0; o <= R; ++o) {
            // all alpha with |alpha| = o, alpha_0 descending, then alpha_1, ...
            int a[D] = {};
            a[0] = o;
            for (;;) {
                int used = 0;
                for (int k = 0; k < D - 1; ++k) used += a[k];
                a[D - 1] = o - used;
                if (a[D - 1] >= 0) {
                    for (int k = 0; k < D; ++k) al[n][k] = a[k];
                    ++n;
                }
                int k = D - 2;
                for (; k >= 0; --k)
                    if (a[k] > 0) break;
                if (k < 0) break;
                a[k]--;
                int pre = 0;
                for (int m = 0; m <= k; ++m) pre += a[m];
                if (k + 1 <= D - 2) {
                    a[k + 1] = o - pre;
                    for (int m = k + 2; m <= D - 2; ++m) a[m] = 0;
                }
            }
        }
        for (int t = 1; t < N; ++t) {
            int p = 0;
            while (al[t][p] == 0) ++p;
            int beta[D] = {};
            for (int k = 0; k < D; ++k) beta[k] = al[t][k];
            beta[p] -= 1;
            piv[t] = p;
            par[t] = index_of(beta);
            for (int j = 0; j < D; ++j)
                if (beta[j] > 0) {
                    int g[D] = {};
                    for (int k = 0; k < D; ++k) g[k] = beta[k];
                    g[j] -= 1;
                    rj[t][nred[t]] = j;
                    rc[t][nred[t]] = beta[j];
                    ridx[t][nred[t]] = index_of(g);
                    nred[t]++;
                }
        }
    }
};

}  // namespace kdefft
