// Finalisation of a stage, device code: from the stage kernel's moment partials to the
// macroscopic fields, the next stage's cell records, the wall densities and the residual.
//
// A CTA of 128 threads finalises C cells at a time (C = 4, 8, 16 or 32, by the cells of the
// batch) in four phases with a barrier between them:
//   sums     13 moments of each cell over the velocity chunks, (moment, cell) pairs over the
//            threads, even and odd chunks apart;
//   state    four lanes per cell, one per axis: the rest state's moments about u_r added,
//            n, u, P, T, q (Eq. qdef);
//   terms    warps 0 and 1: the half-range coefficients b_l of both signs (FP64); warp 2: the
//            x and y coefficients a_l; warp 3: profiles, 1/tau and the record's scalars;
//   nodes    the per-node factors sum_l c_l basis_l over the cell's lanes, and R_SCALE.
//
// What bounds it: an FP64 warp instruction holds its scheduler's FP64 unit for about 76
// cycles whatever the number of active lanes, so a cell's time is the number of FP64
// instructions in sequence on one scheduler.  Hence the split of a cell over the CTA's four
// warps, which sit on the SM's four schedulers; the roles rotate with the block index so that
// the FP64-heavy ones do not meet on one scheduler.  With FP32 storage everything but the
// half-range coefficients (they cancel by up to 1e7 at order 6) and the scalars of warp 3 is
// double-float arithmetic: FP32 pairs of about 48 bits, a few cycles per instruction, far
// below the FP32 rounding of the partials that enter.  Against the same code in FP64 (and the
// wall flux of the stage kernel, which is double-float too) the errors of profiles and states
// against 64 bits are equal to four digits on each of 61 batches (both models, 3 to 64 nodes per
// half range, orders 3 to 6, Kn 0.02 to 100); the profiles differ by 2e-15.
// Measured, us per step (three launches; before: one thread per cell, or one warp per cell up
// to 608 cells, all but the node sums in FP64): one C2 channel 88 -> 43, the 20 table runs 98
// -> 47, 64 x C2 157 -> 71, 256 x C2 190 -> 139, 32 x C3 282 -> 92, the sweep 240 -> 116, the
// low-Mach runs (FP64) 89 -> 55.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "lbs_internal.h"
#include "pdl.cuh"

namespace lbs {

template <typename T> struct Acc { typedef double type; };
template <> struct Acc<float> { typedef float type; };

template <typename T>
__device__ __forceinline__ T ld(const void* p, int i) { return static_cast<const T*>(p)[i]; }

// 1 / x in FP64 for a finite normal x: the hardware's approximate reciprocal, which reads the
// upper 32 bits of x and sets those of the result (20 bits of mantissa each: a relative error
// of some 2^-20), and two Newton steps r <- r + r (1 - x r), each squaring the relative error:
// about 2^-40, then below the rounding; correct to an ulp in four FMAs, where the IEEE division
// takes about ten FP64 instructions.
static __device__ __forceinline__ double rcp_newton(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = fma(r, fma(-x, r, 1.0), r);
    return fma(r, fma(-x, r, 1.0), r);
}
// 1 / sqrt(x) likewise (a start of some 2^-20 too): r <- r + r (1 - x r^2) / 2, the relative error e
// becomes 3/2 e^2
static __device__ __forceinline__ double rsqrt_newton(double x)
{
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double h = 0.5 * x;
    r = fma(r, fma(-h * r, r, 0.5), r);
    return fma(r, fma(-h * r, r, 0.5), r);
}

// ---- packed FP32 (two lanes of f32x2 per instruction, each element rounded exactly as
// the scalar operation) ----------------------------------------------------------------
#define LBS_OP2(name, op)                                                                       \
    static __device__ __forceinline__ float2 name(float2 a, float2 b)                           \
    {                                                                                           \
        float2 d;                                                                               \
        asm("{.reg .b64 ra, rb, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n " op    \
            " rd, ra, rb;\n mov.b64 {%0, %1}, rd;\n}"                                           \
            : "=f"(d.x), "=f"(d.y)                                                              \
            : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                          \
        return d;                                                                               \
    }
LBS_OP2(add2, "add.rn.f32x2")
LBS_OP2(sub2, "sub.rn.f32x2")
LBS_OP2(mul2, "mul.rn.f32x2")
#undef LBS_OP2
static __device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{.reg .b64 ra, rb, rc, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rb, {%4, %5};\n mov.b64 rc, {%6, %7};\n"
        " fma.rn.f32x2 rd, ra, rb, rc;\n mov.b64 {%0, %1}, rd;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
static __device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }

// ---- the arithmetic of the cell state: FP64 for FP64 storage, double-float for FP32 -------
// Double-float: an FP32 pair hi + lo, |lo| <= ulp(hi) / 2, by error-free transforms (Knuth's
// TwoSum, the FMA form of TwoProduct, a Fast2Sum renormalisation).  Products feeding a sum
// use the _rn intrinsics, which the compiler does not contract.
struct DF {
    float hi, lo;
};
static __device__ __forceinline__ DF df_fast2(float s, float t)
{
    const float h = s + t;
    return DF{h, t - (h - s)};
}
static __device__ __forceinline__ DF df_of(double x)
{
    const float h = __double2float_rn(x);
    return DF{h, __double2float_rn(x - double(h))};
}
static __device__ __forceinline__ DF df_sum(DF S, float p, float e)  // S + p + e, |e| << |p|
{
    const float s = S.hi + p, bb = s - S.hi;
    const float t = (S.hi - (s - bb)) + (p - bb);  // TwoSum(S.hi, p)
    return df_fast2(s, t + (S.lo + e));
}

static __device__ __forceinline__ double r_add(double a, double b) { return a + b; }
static __device__ __forceinline__ double r_sub(double a, double b) { return a - b; }
static __device__ __forceinline__ double r_mul(double a, double b) { return a * b; }
static __device__ __forceinline__ double r_fma(double a, double b, double c) { return fma(a, b, c); }
static __device__ __forceinline__ double r_neg(double a) { return -a; }
static __device__ __forceinline__ double r_twice(double a) { return a + a; }
static __device__ __forceinline__ double r_half(double a) { return 0.5 * a; }
static __device__ __forceinline__ double r_inv(double a) { return rcp_newton(a); }
static __device__ __forceinline__ double r_double(double a) { return a; }
static __device__ __forceinline__ bool r_finite(double a) { return isfinite(a); }
static __device__ __forceinline__ bool r_positive(double a) { return __double2hiint(a) > 0; }
static __device__ __forceinline__ double r_shfl(double a, int lane) { return __shfl_sync(0xffffffffu, a, lane); }
static __device__ __forceinline__ double r_shfl_xor(double a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }

static __device__ __forceinline__ DF r_add(DF a, DF b) { return df_sum(a, b.hi, b.lo); }
static __device__ __forceinline__ DF r_sub(DF a, DF b) { return df_sum(a, -b.hi, -b.lo); }
static __device__ __forceinline__ DF r_mul(DF a, DF b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    return df_fast2(p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p))));
}
static __device__ __forceinline__ DF r_fma(DF a, DF b, DF c)
{
    const float p = __fmul_rn(a.hi, b.hi);
    return df_sum(c, p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p))));
}
static __device__ __forceinline__ DF r_neg(DF a) { return DF{-a.hi, -a.lo}; }
static __device__ __forceinline__ DF r_twice(DF a) { return DF{a.hi + a.hi, a.lo + a.lo}; }
static __device__ __forceinline__ DF r_half(DF a) { return DF{0.5f * a.hi, 0.5f * a.lo}; }
static __device__ __forceinline__ DF r_inv(DF a)
{
    const float y = __frcp_rn(a.hi);
    const float e = fmaf(-a.lo, y, fmaf(-a.hi, y, 1.f));  // 1 - a y, about 2^-24
    return df_fast2(y, __fmul_rn(y, fmaf(e, e, e)));       // y (1 + e + e^2)
}
static __device__ __forceinline__ double r_double(DF a) { return double(a.hi) + double(a.lo); }
static __device__ __forceinline__ bool r_finite(DF a) { return isfinite(a.hi) && isfinite(a.lo); }
static __device__ __forceinline__ bool r_positive(DF a) { return a.hi > 0.f; }
static __device__ __forceinline__ DF r_shfl(DF a, int lane)
{
    return DF{__shfl_sync(0xffffffffu, a.hi, lane), __shfl_sync(0xffffffffu, a.lo, lane)};
}
static __device__ __forceinline__ DF r_shfl_xor(DF a, int m)
{
    return DF{__shfl_xor_sync(0xffffffffu, a.hi, m), __shfl_xor_sync(0xffffffffu, a.lo, m)};
}

template <typename T> struct Real;
template <> struct Real<double> {
    typedef double type;
    static __device__ __forceinline__ double of(double a) { return a; }
    static __device__ __forceinline__ double from(double a) { return a; }  // of an FP64 value
    static __device__ __forceinline__ double round(double a) { return a; }
    // the basis tables and the rest state's moments in this arithmetic
    typedef double basis;
    static __device__ __forceinline__ const double* Hx(const InstDev& I) { return I.Hx; }
    static __device__ __forceinline__ const double* Hy(const InstDev& I) { return I.Hy; }
    static __device__ __forceinline__ const double* Pz(const InstDev& I) { return I.Pz; }
    static __device__ __forceinline__ double rest(const InstDev& I, int a) { return I.mrest[a]; }
    // a coefficient of both half ranges of z (x and y: the first alone, the second zero)
    static __device__ __forceinline__ double unit() { return 1.0; }
    typedef double2 pair;
    static __device__ __forceinline__ pair one(double a) { return make_double2(a, 0.0); }
    static __device__ __forceinline__ void put(pair& p, int s, double a) { (s ? p.y : p.x) = a; }
    static __device__ __forceinline__ double sumw(const InstDev& I, int a) { return I.sumw[a]; }
};
template <> struct Real<float> {
    typedef DF type;
    static __device__ __forceinline__ DF of(float a) { return DF{a, 0.f}; }
    static __device__ __forceinline__ DF from(double a) { return df_of(a); }
    static __device__ __forceinline__ float round(DF a) { return a.hi; }
    typedef float2 basis;
    static __device__ __forceinline__ const float2* Hx(const InstDev& I) { return I.Hx2; }
    static __device__ __forceinline__ const float2* Hy(const InstDev& I) { return I.Hy2; }
    static __device__ __forceinline__ const float2* Pz(const InstDev& I) { return I.Pz2; }
    static __device__ __forceinline__ DF rest(const InstDev& I, int a) { return DF{I.mrest2[a][0], I.mrest2[a][1]}; }
    static __device__ __forceinline__ float2 unit() { return make_float2(1.f, 0.f); }
    typedef float4 pair;  // (hi, hi, lo, lo)
    static __device__ __forceinline__ pair one(DF a) { return make_float4(a.hi, 0.f, a.lo, 0.f); }
    static __device__ __forceinline__ void put(pair& p, int s, DF a)
    {
        float* q = reinterpret_cast<float*>(&p);
        q[s] = a.hi;
        q[2 + s] = a.lo;
    }
    static __device__ __forceinline__ DF sumw(const InstDev& I, int a) { return DF{I.sumw2[a][0], I.sumw2[a][1]}; }
};

// Sums of products for a pair of nodes (both half ranges of z) at once.  FP32 storage: FP32
// products and sums with their rounding errors (TwoProduct, TwoSum) gathered in a second FP32
// sum, packed two lanes per instruction: 12 instructions per term for both nodes, about 2^-47
// of the largest term.  The negative of each product serves both transforms, which spares the
// packed negation the instruction set lacks.
template <typename T> struct PairSum;
template <> struct PairSum<float> {
    float2 s, e;
    __device__ __forceinline__ PairSum() : s(make_float2(0.f, 0.f)), e(make_float2(0.f, 0.f)) {}
    __device__ __forceinline__ void add(float2 np, float2 err)  // s - np + err
    {
        const float2 t = sub2(s, np), b = sub2(t, s);
        e = add2(e, add2(sub2(sub2(s, sub2(t, b)), add2(np, b)), err));
        s = t;
    }
    __device__ __forceinline__ void term(const float4& c, float2 h)
    {
        const float2 hx = splat(h.x), hi = make_float2(c.x, c.y), np = mul2(make_float2(-c.x, -c.y), hx);
        add(np, fma2(make_float2(c.z, c.w), hx, fma2(hi, splat(h.y), fma2(hi, hx, np))));
    }
    __device__ __forceinline__ void weighted(float w, float2 v)
    {
        const float2 np = mul2(splat(-w), v);
        add(np, fma2(splat(w), v, np));
    }
    __device__ __forceinline__ float2 value() const { return add2(s, e); }
    __device__ __forceinline__ DF total() const { return df_sum(df_fast2(s.x, e.x), s.y, e.y); }
};
template <> struct PairSum<double> {
    double2 s;
    __device__ __forceinline__ PairSum() : s(make_double2(0.0, 0.0)) {}
    __device__ __forceinline__ void term(const double2& c, double h)
    {
        s.x = fma(c.x, h, s.x);
        s.y = fma(c.y, h, s.y);
    }
    __device__ __forceinline__ void weighted(double w, double2 v)
    {
        s.x = fma(w, v.x, s.x);
        s.y = fma(w, v.y, s.y);
    }
    __device__ __forceinline__ double2 value() const { return s; }
    __device__ __forceinline__ double total() const { return s.x + s.y; }
};

// shared memory of the C cells a CTA finalises
template <typename T, int C>
struct FinShared {
    typedef typename Real<T>::type R;
    R mom[2][kNMom][C];            // moment sums over the even and the odd chunks
    R n[C], in[C], u[3][C], T_[C], q[3][C];  // the record's state (a neutral one where it is bad)
    R prof[14][C];                 // the profiles, as computed
    typename Real<T>::pair c[3][kMaxN + 1][C];  // coefficients of x, y (term 0 zero), z
    int bad[C];
};

// exp(-t) and sum_n (-t)^n / (n! (2n + 1)) (the Maclaurin series of erf(x) sqrt(pi) / (2 x) at
// t = x^2, Abramowitz & Stegun 7.1.5) to degree 7: below 2^-7 the omitted terms are under
// 2^-56 / 8! = 4e-22 of the sums
struct SmallSeries {
    double e[8], f[8];
    constexpr SmallSeries() : e(), f()
    {
        double fact = 1.0;
        for (int n = 0; n < 8; ++n) {
            if (n > 0) fact *= n;
            e[n] = (n % 2 ? -1.0 : 1.0) / fact;
            f[n] = e[n] / (2 * n + 1);
        }
    }
};

// Moments M_k = int_0^inf p^k g(p; u, T) dp, k = 0 .. K, of the drifting Maxwellian on a half
// line: M_0 = erfc(-u / sqrt(2T)) / 2, M_1 = u M_0 + T g(0), M_{k+1} = u M_k + k T M_{k-1};
// *dev0 = M_0 - 1/2.  In Couette flow the wall-normal drift is small: where every lane's
// t = u^2 / (2T) is below 2^-7 (|u| < 0.125 sqrt T) two short series replace erfc and exp.
template <int NB>
__device__ __forceinline__ void half_line_moments(double u, double T_, int K, double (&M)[NB + 1], double* dev0)
{
    const double r = rsqrt_newton(T_), x = u * (r * 0.70710678118654752440), t = x * x;
    double ex, dev;
    if (__all_sync(0xffffffffu, t < 0x1p-7)) {
        constexpr SmallSeries S;
        double p = S.f[7];
        ex = S.e[7];
#pragma unroll
        for (int n = 6; n >= 0; --n) {
            p = fma(p, t, S.f[n]);
            ex = fma(ex, t, S.e[n]);
        }
        dev = x * (p * 0.56418958354775628695);  // erf(x) / 2; 1 / sqrt(pi)
        M[0] = 0.5 + dev;
    } else {
        const double e = erfc_nonneg(fabs(x));
        M[0] = x >= 0.0 ? 1.0 - 0.5 * e : 0.5 * e;
        dev = M[0] - 0.5;
        ex = exp(-t);
    }
    *dev0 = dev;
    const double g0 = ex * (r * 0.39894228040143267794);  // g(0), 1 / sqrt(2 pi)
    M[1] = fma(u, M[0], T_ * g0);
#pragma unroll
    for (int k = 1; k < NB; ++k) M[k + 1] = k < K ? fma(u, M[k], (k * T_) * M[k - 1]) : 0.0;
}

// A node of x or y, or a pair of nodes of z: its basis row, weight and axis
template <typename T, int NB>
struct Node {
    typename Real<T>::basis h[NB + 1];
    T w;
    int ax;
    __device__ __forceinline__ Node() : w(T(0)), ax(0)
    {
#pragma unroll
        for (int l = 0; l <= NB; ++l) h[l] = typename Real<T>::basis();
    }
    __device__ __forceinline__ int order(const InstDev& I) const { return ax == 0 ? I.Nx : ax == 1 ? I.Ny : I.Nzq; }
    __device__ __forceinline__ void load(const InstDev& I, int r)
    {
        typedef Real<T> RT;
        const int Qx = I.Qx, Qy = I.Qy;
        if (r >= Qx + Qy + I.Qz) return;
        ax = r < Qx ? 0 : r < Qx + Qy ? 1 : 2;
        const int N = order(I), k = ax == 0 ? r : ax == 1 ? r - Qx : r - Qx - Qy;
        const typename RT::basis* row = (ax == 0 ? RT::Hx(I) : ax == 1 ? RT::Hy(I) : RT::Pz(I)) + k * (N + 1);
#pragma unroll
        for (int l = 0; l <= NB; ++l)
            if (l <= N) h[l] = row[l];
        w = ld<T>(ax == 0 ? I.wx : ax == 1 ? I.wy : I.wz, k);
    }
};

// ---- terms and nodes of the record: cells c0 .. c0 + nc - 1, their state in sm; node: this
// thread's first one, loaded (it does not depend on the state); PROF: also the profiles and W
template <typename T, int NB, int C, bool PROF>
__device__ __forceinline__ void record_cells(const InstDev& I, int c0, int nc, FinShared<T, C>& sm, int vt,
                                             Node<T, NB> node)
{
    typedef Real<T> RT;
    typedef typename RT::type R;
    constexpr int L = kThreads / C;  // lanes of a cell in the node phase
    const int warp = vt >> 5, lane = vt & 31;
    const int Qx = I.Qx, Qz = I.Qz, G = Qx + I.Qy + Qz;
    const int cell = vt / L, j = vt % L;
    if (warp < 2) {
        // z: with few cells 16 lanes per cell, lane l - 1 of each sign forming row l of the
        // polynomials' coefficients times the moments; else a lane per (cell, sign) and all rows
        const int K = I.Nzq;
        const double* A = I.half_poly;  // [kMaxN + 1][kMaxN + 1], monic coefficients of pi_l
        double M[NB + 1], dev;
        if constexpr (C <= 4) {
            const int zc = (vt >> 4) & (C - 1), s = (vt >> 3) & 1, l = (vt & 7) + 1;
            double row[NB + 1];
#pragma unroll
            for (int k = 0; k <= NB; ++k) row[k] = A[l * (kMaxN + 1) + k];
            const double u = r_double(sm.u[2][zc]);
            half_line_moments<NB>(s ? -u : u, r_double(sm.T_[zc]), K, M, &dev);
            double b = 0.0;
#pragma unroll
            for (int k = NB; k >= 0; --k) b = fma(row[k], M[k], b);
            if (l <= K) RT::put(sm.c[2][l][zc], s, RT::from(b));
            if (l == 1) RT::put(sm.c[2][0][zc], s, RT::from(dev));
        } else if ((vt & ~31) < 2 * C) {
            const int zc = vt % C, s = (vt / C) & 1;
            const double u = r_double(sm.u[2][zc]);
            half_line_moments<NB>(s ? -u : u, r_double(sm.T_[zc]), K, M, &dev);
            RT::put(sm.c[2][0][zc], s, RT::from(dev));
#pragma unroll
            for (int l = 1; l <= NB; ++l)
                if (l <= K) {
                    double b = M[l];
#pragma unroll
                    for (int k = l - 1; k >= 0; --k) b = fma(A[l * (kMaxN + 1) + k], M[k], b);
                    RT::put(sm.c[2][l][zc], s, RT::from(b));
                }
        }
    } else if (warp == 2) {
        // x and y: a_0 = 1 (not used: the factors are deviations from 1), a_1 = u,
        // a_{l+1} = u a_l + l (T - 1) a_{l-1}
        for (int e = lane; e < 2 * C; e += 32) {
            const int ax = e / C, xc = e % C, N = ax ? I.Ny : I.Nx;
            const R u = sm.u[ax][xc], t1 = r_sub(sm.T_[xc], RT::of(T(1)));
            R p = RT::of(T(1)), q = u, lt = t1;
            sm.c[ax][0][xc] = RT::one(RT::of(T(0)));
            if (I.reduced && ax) {  // the factors of phi and chi: 1 and T
                sm.c[1][1][xc] = RT::one(t1);
                continue;
            }
#pragma unroll
            for (int l = 1; l <= NB; ++l)
                if (l <= N) {
                    sm.c[ax][l][xc] = RT::one(q);
                    const R nx = r_fma(u, q, r_mul(lt, p));
                    p = q;
                    q = nx;
                    lt = r_add(lt, t1);
                }
        }
    } else {
        // the profiles, and the record's scalars
        const int Nz = I.Nz;
        for (int e = lane; PROF && e < 14 * C; e += 32) {
            const int row = e / C, xc = e % C;
            if (xc >= nc) continue;
            const double v = r_double(sm.prof[row][xc]);
            I.prof[(size_t)row * Nz + c0 + xc] = v;
            const int wi = row == 0 ? 0 : row == 1 ? 1 : row == 4 ? 2 : -1;  // W = n, u_x, T
            if (wi >= 0) I.Wnew[wi * Nz + c0 + xc] = v;
        }
        if (lane < C && lane < nc) {
            T* rec = static_cast<T*>(I.rec) + (size_t)(c0 + lane) * I.rec_stride;
            const double n = r_double(sm.n[lane]), Tc = r_double(sm.T_[lane]), iT = rcp_newton(Tc);
            rec[R_N] = RT::round(sm.n[lane]);
            rec[R_T] = RT::round(sm.T_[lane]);
            rec[R_UX] = RT::round(sm.u[0][lane]);
            rec[R_UY] = RT::round(sm.u[1][lane]);
            rec[R_UZ] = RT::round(sm.u[2][lane]);
            rec[R_QX] = RT::round(sm.q[0][lane]);
            rec[R_QY] = RT::round(sm.q[1][lane]);
            rec[R_QZ] = RT::round(sm.q[2][lane]);
            rec[R_ITAU] = T(inv_relax_time(I.visc_law, I.iKn, I.visc_param, I.isuth, n, Tc, iT));
            rec[R_CS] = T((1.0 - I.Pr) * r_double(sm.in[lane]) * iT * iT);
            rec[R_I5T] = T(0.2 * iT);
            if (sm.bad[lane]) atomicOr(I.status, STATUS_NONFINITE);
        }
    }
    __syncthreads();

    // nodes: v = sum_l c_l basis_l, rounded once; the weighted sums over the stored values,
    // per axis, so that R_SCALE makes the discrete equilibrium carry exactly n
    const bool live = cell < nc;
    T* rec = static_cast<T*>(I.rec) + (size_t)(c0 + (live ? cell : 0)) * I.rec_stride;
    R s[4];  // x, y, z, unused
#pragma unroll
    for (int a = 0; a < 4; ++a) s[a] = RT::of(T(0));
    PairSum<T> ws;  // of the current axis (a thread's nodes come in axis order)
    int cur = node.ax;
    for (int r = j; r < G; r += L) {
        Node<T, NB> next;
        next.load(I, r + L);
        const int ax = node.ax, N = node.order(I);
        if (ax != cur) {
            (cur == 0 ? s[0] : s[1]) = ws.total();
            ws = PairSum<T>();
            cur = ax;
        }
        PairSum<T> g;
        if (I.reduced && ax == 1) {
            if (r > Qx) g.term(sm.c[1][1][cell], RT::unit());
        } else {
#pragma unroll
            for (int l = 0; l <= NB; ++l)
                if (l <= N) g.term(sm.c[ax][l][cell], node.h[l]);
        }
        const auto v = g.value();
        if (live) {
            rec[R_DX + r] = v.x;
            if (ax == 2) rec[R_DX + r + Qz] = v.y;
        }
        ws.weighted(node.w, v);
        node = next;
    }
    (cur == 0 ? s[0] : cur == 1 ? s[1] : s[2]) = ws.total();
    // the cell's lanes: scatter the four sums over lane pairs L/2 and L/4 apart, then add up
    const bool hi = j & (L / 2), hi2 = j & (L / 4);
    R a0 = r_add(hi ? s[2] : s[0], r_shfl_xor(hi ? s[0] : s[2], L / 2));
    R a1 = r_add(hi ? s[3] : s[1], r_shfl_xor(hi ? s[1] : s[3], L / 2));
    a0 = r_add(hi2 ? a1 : a0, r_shfl_xor(hi2 ? a0 : a1, L / 4));
#pragma unroll
    for (int o = L / 8; o > 0; o >>= 1) a0 = r_add(a0, r_shfl_xor(a0, o));
    const int g0 = lane & ~(L - 1);  // lane 0 of the cell's group
    const R sx = r_add(RT::sumw(I, 0), r_shfl(a0, g0));
    const R sy = I.reduced ? RT::of(T(1)) : r_add(RT::sumw(I, 1), r_shfl(a0, g0 + L / 4));
    const R sz = r_add(RT::sumw(I, 2), r_shfl(a0, g0 + L / 2));
    if (live && j == 0) {
        const R sc = r_mul(sm.n[cell], r_inv(r_mul(r_mul(sx, sy), sz)));
        rec[R_SCALE1] = RT::round(r_sub(sc, RT::of(T(1))));
    }
}

// the thread index with the warps' roles rotated
static __device__ __forceinline__ int rotated(int rot) { return (threadIdx.x + 32 * rot) & (kThreads - 1); }

// ---- one group of cells c0 .. c0 + nc - 1 (nc <= C), all 128 threads of the CTA -------------
template <typename T, int NB, int C>
__device__ __forceinline__ void finalize_group(const InstDev& I, int c0, int nc, int stage, FinShared<T, C>& sm,
                                               int rot, const Node<T, NB>& node)
{
    typedef Real<T> RT;
    typedef typename RT::type R;
    typedef typename Acc<T>::type A;
    const int vt = rotated(rot);
    const int Nz = I.Nz, nch = I.nchunks;
    // sums over the chunks, in order within the even and the odd ones (the same order whatever
    // C is); loads past L1: other CTAs wrote the partials
    const A* part = static_cast<const A*>(I.partial);
    {
        constexpr int per = kThreads / C;  // (moment, parity) slots at a time
        const int c = vt % C, cell = c0 + min(c, nc - 1);
        for (int e = vt / C; e < 2 * 16; e += per) {
            const int a = e & 15, par = e >> 4;
            if (a >= kNMom) continue;
            R sum = RT::of(T(0));
            for (int k = par; k < nch; k += 16) {
                A p[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    p[i] = k + 2 * i < nch ? __ldcg(part + ((size_t)(k + 2 * i) * kNMom + a) * Nz + cell) : A(0);
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (k + 2 * i < nch) sum = r_add(sum, RT::of(p[i]));
            }
            sm.mom[par][a][c] = sum;
        }
    }
    __syncthreads();
    // state: lanes 4 c + axis (the fourth lane repeats axis z); the warps this covers run it
    // whole (their spare lanes repeat cells), so that the shuffles are convergent
    if ((vt & ~31) < 4 * C) {
        const int c = (vt >> 2) & (C - 1), a = min(vt & 3, 2), base = vt & 28;  // base: lane of axis x
        const int b = a == 2 ? 0 : a + 1, d = a == 0 ? 2 : a - 1;              // the other two axes
        const int ab = a == 0 ? 7 : a == 1 ? 9 : 8, ad = d == 0 ? 7 : d == 1 ? 9 : 8;  // pairs (a, b), (d, a)
        const int cell = c0 + min(c, nc - 1);
        const T* rc = static_cast<const T*>(I.rec) + (size_t)cell * I.rec_stride;
        // the velocity the stage kernel took its moments about: the record's u (0 for the
        // analysis pass)
        const T za = stage > 0 ? rc[R_UX + a] : T(0), zb = stage > 0 ? rc[R_UX + b] : T(0),
                zd = stage > 0 ? rc[R_UX + d] : T(0);
        const R ua = RT::of(za), ub = RT::of(zb), ud = RT::of(zd);
        const R na = r_neg(ua), nb = r_neg(ub);
        auto m = [&](int i) { return r_add(sm.mom[0][i][c], sm.mom[1][i][c]); };
        const R r0 = RT::rest(I, 0), r1a = RT::rest(I, 1 + a), r1b = RT::rest(I, 1 + b);
        const R r2aa = RT::rest(I, 4 + a), r2ab = RT::rest(I, ab), r2ad = RT::rest(I, ad);
        // the rest state's moments about u_r: R1_a = r1_a - u_a r0, R2_ab = r2_ab - u_a r1_b -
        // u_b R1_a, R3_a = r3_a - 2 u.r2_a + u^2 r1_a - u_a tr R2
        const R R1 = r_fma(na, r0, r1a);
        const R R2aa = r_fma(na, r_add(r1a, R1), r2aa), R2ab = r_fma(nb, R1, r_fma(na, r1b, r2ab));
        const R uu = r_fma(ua, ua, r_fma(ub, ub, r_mul(ud, ud)));
        const R trR = r_add(R2aa, r_add(r_shfl(R2aa, base + b), r_shfl(R2aa, base + d)));
        const R dot = r_fma(ua, r2aa, r_fma(ub, r2ab, r_mul(ud, r2ad)));
        const R R3 = r_fma(na, trR, r_fma(uu, r1a, r_sub(RT::rest(I, 10 + a), r_twice(dot))));
        // moments of the whole distribution about u_r
        const R M0 = r_add(m(0), r0), M1 = r_add(m(1 + a), R1), M2aa = r_add(m(4 + a), R2aa),
                M2ab = r_add(m(ab), R2ab), M3 = r_add(m(10 + a), R3);
        const R in = r_inv(M0);
        const R xa = r_mul(M1, in), xb = r_shfl(xa, base + b), xd = r_shfl(xa, base + d);  // the mean of p - u_r
        const R ma = r_neg(M1), M2ad = r_shfl(M2ab, base + d);
        const R Paa = r_fma(ma, xa, M2aa), Pab = r_fma(ma, xb, M2ab);
        const R trP = r_add(Paa, r_add(r_shfl(Paa, base + b), r_shfl(Paa, base + d)));
        const R Tc = r_mul(r_mul(trP, in), RT::from(1.0 / 3.0));
        const R xx = r_fma(xa, xa, r_fma(xb, xb, r_mul(xd, xd)));
        const R xm = r_fma(xa, M2aa, r_fma(xb, M2ab, r_mul(xd, M2ad)));
        // q_a = 1/2 sum |xi|^2 xi_a f about the mean
        const R qa = r_half(r_fma(r_neg(xa), trP, r_fma(xx, M1, r_sub(M3, r_twice(xm)))));
        const R va = r_add(ua, xa);
        const unsigned fin = __ballot_sync(0xffffffffu, r_finite(va) && r_finite(qa) && r_finite(Paa) && r_finite(Pab));
        const bool ok = ((fin >> base) & 7u) == 7u;  // every profile value finite
        const bool state = ok && r_finite(M0) && r_finite(Tc) && r_positive(M0) && r_positive(Tc);
        if (vt < 4 * C) {
            // profiles n, u, T, q, P_xx, P_yy, P_zz, P_xy, P_xz, P_yz
            sm.prof[1 + a][c] = va;
            sm.prof[5 + a][c] = qa;
            sm.prof[8 + a][c] = Paa;
            sm.prof[a == 0 ? 11 : a == 1 ? 13 : 12][c] = Pab;
            // a non-finite or non-positive state: the record of a neutral one, and the flag
            sm.u[a][c] = state ? va : RT::of(T(0));
            sm.q[a][c] = state ? qa : RT::of(T(0));
            if (a == 0) {
                sm.prof[0][c] = M0;
                sm.prof[4][c] = Tc;
                sm.n[c] = state ? M0 : RT::of(T(1));
                sm.in[c] = state ? in : RT::of(T(1));
                sm.T_[c] = state ? Tc : RT::of(T(1));
                sm.bad[c] = !state;
            }
        }
    }
    __syncthreads();
    launch_dependents();
    record_cells<T, NB, C, true>(I, c0, nc, sm, vt, node);
}

// the fused finalisation: the cells of a z-tile, four at a time; sm is the stage CTA's dynamic
// shared memory, which stage_smem makes at least this large
template <typename T>
__device__ __noinline__ void finalize_tile(const InstDev& I, int z0, int zn, int stage, FinShared<T, 4>& sm)
{
    for (int c = 0; c < zn; c += 4) {
        Node<T, kMaxN> node;
        node.load(I, threadIdx.x & 31);  // a cell's 32 lanes; the roles rotate by whole warps
        finalize_group<T, kMaxN, 4>(I, z0 + c, min(4, zn - c), stage, sm, (c >> 2) & 3, node);
        __syncthreads();
    }
}

// records from given macroscopic profiles macro[8][Nz] = n, ux, uy, uz, T, qx, qy, qz (four
// cells per block of 128 threads)
template <typename T>
__global__ void __launch_bounds__(kThreads) records_from_macro(const InstDev* __restrict__ insts, int inst,
                                                               const double* __restrict__ macro)
{
    typedef Real<T> RT;
    __shared__ FinShared<T, 4> sm;
    const InstDev& I = insts[inst];
    const int Nz = I.Nz, c0 = blockIdx.x * 4, nc = min(4, Nz - c0);
    if (threadIdx.x < 4) {
        const int c = threadIdx.x;
        double v[8];
        bool ok = true;
        for (int a = 0; a < 8; ++a) {
            v[a] = macro[a * Nz + c0 + min(c, nc - 1)];
            ok &= isfinite(v[a]);
        }
        ok &= v[0] > 0.0 && v[4] > 0.0;
        sm.n[c] = RT::from(ok ? v[0] : 1.0);
        sm.in[c] = RT::from(ok ? 1.0 / v[0] : 1.0);
        sm.T_[c] = RT::from(ok ? v[4] : 1.0);
        for (int a = 0; a < 3; ++a) {
            sm.u[a][c] = RT::from(ok ? v[1 + a] : 0.0);
            sm.q[a][c] = RT::from(ok ? v[5 + a] : 0.0);
        }
        sm.bad[c] = !ok;
    }
    __syncthreads();
    Node<T, kMaxN> node;
    node.load(I, threadIdx.x & 31);
    record_cells<T, kMaxN, 4, false>(I, c0, nc, sm, threadIdx.x, node);
}

// The instance descriptor copied into shared memory by the whole block at once: its
// fields (pointers, orders, wall sums) are then one shared load away instead of an
// L2 round trip each at first use -- in the stage kernel's prologue (pointer, then
// table, then value) and inside the finalisation's FP64 chains.
static __device__ __forceinline__ const InstDev& stage_descriptor(const InstDev* g, InstDev* s)
{
    static_assert(sizeof(InstDev) % 8 == 0, "descriptor copied in 8-byte words");
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(g);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(s);
    for (int e = threadIdx.x; e < (int)(sizeof(InstDev) / 8); e += blockDim.x) dst[e] = src[e];
    __syncthreads();
    return *s;
}

// Warp reduce-scatter of 8 values: lanes 4 i .. 4 i + 3 end with the warp's total of value i
// (9 additions per lane instead of 40 for 8 butterflies)
static __device__ __forceinline__ double reduce_scatter8(double (&v)[8], int lane)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool hi = lane & 16;
        v[i] = (hi ? v[i + 4] : v[i]) + __shfl_xor_sync(0xffffffffu, hi ? v[i] : v[i + 4], 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool hi = lane & 8;
        v[i] = (hi ? v[i + 2] : v[i]) + __shfl_xor_sync(0xffffffffu, hi ? v[i] : v[i + 2], 8);
    }
    {
        const bool hi = lane & 4;
        v[0] = (hi ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 4);
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// One instance (a whole CTA of 128 threads): wall densities n_w from the outgoing wall fluxes
// (zero net mass flux, Appendix); after stage 3 the residual, the step count and
// retirement; after the analysis pass W_old = W.  red: 8 * 4 shared doubles.
static __device__ __noinline__ void finalize_instance(const InstDev& I, int stage, double* red)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, Nz = I.Nz;
    // v: the two wall fluxes; the residual's sums ||W_new - W_old||^2, ||W_old||^2 for n, u_x, T
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.0;
    for (int c = t; c < I.nchunks; c += kThreads) {
        v[0] += __ldcg(I.flux_part + 2 * c);
        v[1] += __ldcg(I.flux_part + 2 * c + 1);
    }
    double tot;
    if (stage == 3) {
        for (int s = t; s < Nz; s += kThreads) {
            double wn[3], wo[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                wn[a] = __ldcg(I.Wnew + a * Nz + s);
                wo[a] = I.Wold[a * Nz + s];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double e = wn[a] - wo[a];
                v[2 + 2 * a] = fma(e, e, v[2 + 2 * a]);
                v[3 + 2 * a] = fma(wo[a], wo[a], v[3 + 2 * a]);
                I.Wold[a * Nz + s] = wn[a];
            }
        }
        tot = reduce_scatter8(v, lane);
    } else {
        const bool hi = lane & 16;
        tot = (hi ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if (stage == 0)
            for (int e = t; e < 3 * Nz; e += kThreads) I.Wold[e] = __ldcg(I.Wnew + e);
    }
    const int per = stage == 3 ? 4 : 16;  // lanes that hold one total
    if (lane % per == 0) red[warp * 8 + lane / per] = tot;
    __syncthreads();
    if (warp != 0) return;
    // lane i < 8: value i over the warps
    const int i = lane & 7;
    double x = 0.0;
    if (stage == 3 || i < 2)
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) x += red[w * 8 + i];
    if (lane < 2) {  // the partials sum w p_z over the deviations: add the rest state's flux
        const double nw = -((lane ? I.frest_top : I.frest_bot) + x) * (lane ? I.iDtop : I.iDbot);
        I.nw->d[2 * lane] = nw - 1.0;
        I.nw->d[2 * lane + 1] = nw;
        I.nw->f[2 * lane] = float(nw - 1.0);
        I.nw->f[2 * lane + 1] = float(nw);
        if (!isfinite(nw)) atomicOr(I.status, STATUS_NONFINITE);
    }
    if (stage == 3) {
        const double den = __shfl_down_sync(0xffffffffu, x, 1);  // for lanes 2, 4, 6
        // the velocity on the wall speed where u_x is smaller
        const double floor_ = i == 4 ? I.res_uscale : 1e-30;
        double r = x / fmax(den, floor_ * floor_);
        r = fmax(fmax(0.0, __shfl_sync(0xffffffffu, r, 2)),
                 fmax(__shfl_sync(0xffffffffu, r, 4), __shfl_sync(0xffffffffu, r, 6)));
        if (lane == 0) {
            const double R = sqrt(r);
            *I.res = R;
            *I.steps += 1;
            *I.cur ^= 1;  // the new state was written over the stage-1 increment
            if (I.tol > 0.0 && R < I.tol) *I.active = 0;
        }
    }
}

}  // namespace lbs
