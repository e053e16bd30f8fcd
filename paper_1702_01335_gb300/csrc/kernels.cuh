// Device code of one RK-3 stage of the mixed-quadrature Shakhov scheme (kernels.cuh).
// Included by kernels.cu (finalisation, seeding, launchers) and by the four
// stage_*.cu translation units, each of which instantiates the stage kernel for
// one storage type and velocity model so that they compile in parallel.
//
// Per stage (Eq. rk3 around Eq. L_def):
//   stage_kernel     one CTA per tile = (instance, z-range of <= 64 cells,
//                    velocity chunk of 128*V velocities).  The rows of F_in
//                    the tile needs (its cells and a 3-cell halo each side) and
//                    its rows of F_l are staged into shared memory by TMA bulk
//                    copies (one cp.async.bulk per row, one mbarrier).  While
//                    they land, the CTA evaluates the per-axis factors of the
//                    truncated Hermite equilibrium (Sec. III) of its cells.
//                    Ghost rows are then built in shared memory: outgoing
//                    populations by the quadratic extrapolation of the
//                    Appendix, incoming ones as n_w times the wall equilibrium;
//                    below a half channel's centre line, cells 0..2 at the
//                    mirrored velocity (bounce-back, Appendix).
//                    Each thread marches through the z-range in the upwind
//                    direction of its V velocities, carrying the differences of
//                    the WENO-5 stencil from one interface to the next (the pair
//                    layout keeps a window of six values): interface fluxes (Eqs.
//                    weno5_flux - weno_sigma, Table weno), the divergence of
//                    Eq. (flux), relaxation to n G_x G_y G_z (1 + S) and the
//                    Shu-Osher combine; it stores F_out and accumulates the raw
//                    moments of F_out (in FP32 within the CTA and stored per
//                    chunk in FP32 in FP32 mode; in FP64 in FP64 mode).  Tiles
//                    that end at a wall also reduce the outgoing WENO flux of
//                    F_out through the wall (double-float within the chunk in FP32
//                    mode).
//   finalisation     (finalize.cuh) per cell: the sum of the chunks' partials, n, u, P, T, q
//                    (Eq. qdef), tau, and the cell record of the next stage; per
//                    instance: the wall densities n_w (zero net mass
//                    flux, Appendix) and, after the third stage, the residual.
//                    Either a launch of its own (finalize_cells in kernels.cu), or folded
//                    into the stage kernel (fuse = 1: the CTA that ends last among the
//                    chunks of a z-tile does its cells, threadfence tickets).
//
// Template parameter RED: the reduced phi / chi model of Sec. III (j = 0 phi,
// j = 1 chi on a two-node transverse axis), otherwise the full 3D velocity set.
//
// Storage: F[s][k] for interior cells s = 0..Nz-1 (no ghost rows), velocity
// k = ((sg*Qz + m)*Qx + i)*Qy + j fastest, holding f_k / w_k.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "finalize.cuh"
#include "lbs_internal.h"

namespace lbs {

// ---- PTX helpers: mbarrier and bulk global -> shared copies ------------------
static __device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
static __device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
static __device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
static __device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
static __device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
static __device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes)  // into L2
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
static __device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// WENO-5 reconstruction of five upwind-ordered values (no advection factor), as the
// correction to the upwind cell's value v2: weno5 = v2 + weno5_corr.  The candidate
// reconstructions are c_q = v2 + e_q / 6 with e_q made of the differences d_j = v_j - v2
// (Eq. weno5_flux), and the smoothness indicators are written in the same differences
// (Eq. weno_sigma), so the correction carries the precision of the differences, not of
// v2, and the divergence of Eq. (flux) can be formed as a difference of cell values plus
// a difference of corrections.
//
// FP64 form.  The FP64 pipe bounds the FP64 stage kernel (an FP64 instruction holds a
// scheduler's unit about 76 cycles), so the form counts instructions.  The normalised
// weights of Eq. (weno5_omega), g_q / sigma_q^2 over their sum, are multiplied through by
// (sigma_1 sigma_2 sigma_3)^2: W_1 = (sigma_2 sigma_3)^2 and so on, one reciprocal of the
// sum instead of five divisions.  The sigma are scaled to [0, 2) by the power of two of the
// largest (its exponent bits, integer instructions; exact) so that no product leaves the
// range, and floored at 2^-250 of it: two or three vanishing indicators then take the limits
// of Table (weno), and a sigma above 2^-197 of the largest (differences above 1e-30 of the
// largest: everything FP64 values resolve) is not changed by the floor.  A non-finite sigma
// gives a non-finite result.  About 48 FP64 instructions instead of about 100.
// Measured, 2 steps of 16 x C2 with profiles and checkpoint: 9.09 -> 6.50 ms; 16 steps of the
// four low-Mach runs: 3.03 -> 2.45 ms; outputs within 2e-15 of the division form's.
template <typename T>
__device__ __forceinline__ T weno5_corr(T v0, T v1, T v2, T v3, T v4)
{
    const T d0 = v0 - v2, d1 = v1 - v2, d3 = v3 - v2, d4 = v4 - v2;
    const T a1 = fma(-2.0, d1, d0), b1 = fma(-4.0, d1, d0);  // v0-2v1+v2, v0-4v1+3v2
    const T a2 = d1 + d3, b2 = d1 - d3;                      // v1-2v2+v3, v1-v3
    const T a3 = fma(-2.0, d3, d4), b3 = fma(-4.0, d3, d4);  // v2-2v3+v4, 3v2-4v3+v4
    const T K = 13.0 / 3.0;                                  // 4 sigma = 13/3 a^2 + b^2
    const T q1 = fma(K * a1, a1, b1 * b1), q2 = fma(K * a2, a2, b2 * b2), q3 = fma(K * a3, a3, b3 * b3);
    const int top = max(__double2hiint(q1), max(__double2hiint(q2), __double2hiint(q3)));  // sigma >= 0
    const T s = __hiloint2double(0x7FE00000 - (top & 0x7FF00000), 0);
    const T floor_ = 0x1p-250;
    const T s1 = fma(q1, s, floor_), s2 = fma(q2, s, floor_), s3 = fma(q3, s, floor_);
    const T p1 = s2 * s3, p2 = s1 * s3, p3 = s1 * s2;
    const T w1 = p1 * p1, w2 = 6.0 * p2 * p2, w3 = 3.0 * p3 * p3;  // 10 g_q W_q
    // e_q / 2: d0 - 7/2 d1, d3 - d1 / 2, 5/2 d3 - d4 / 2
    const T e1 = fma(-3.5, d1, d0), e2 = fma(-0.5, d1, d3), e3 = fma(2.5, d3, -0.5 * d4);
    const T num = fma(w1, e1, fma(w2, e2, w3 * e3));
    return num * rcp_newton(fma(3.0, w1, 3.0 * (w2 + w3)));  // (sum w e_q / 6) / sum w
}

static __device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// FP32 form, the same stencils in constant-light operations (the multiples 2, 4, 5, 7 of
// the differences built by additions; two constants in all, which the packed form below
// keeps in registers): 4 sigma_q = 13/3 a_q^2 + b_q^2 and the ideal weights scaled by 10
// to (1, 6, 3), common factors that cancel in the normalised weights.  (4 sigma_q)^2 is
// floored at 1.6e-36 (sigma_q^2 at 1e-37; branch free, hardware reciprocals): as
// sigma_q -> 0 the floor gives exactly the limits of Table (weno), and it changes nothing
// while sigma_q^2 > 1e-30, i.e. for differences above the FP32 resolution of O(1)
// normalised populations.  The rounded weights only multiply the small corrections e_q.
constexpr float kWenoK = 13.f / 3.f, kWenoFloor = 1.6e-36f;
template <>
__device__ __forceinline__ float weno5_corr<float>(float v0, float v1, float v2, float v3, float v4)
{
    const float d0 = v0 - v2, d1 = v1 - v2, d3 = v3 - v2, d4 = v4 - v2;
    const float t = d1 + d1, u = d3 + d3;
    const float a1 = d0 - t, b1 = a1 - t;    // v0-2v1+v2, v0-4v1+3v2
    const float a2 = d1 + d3, b2 = d1 - d3;  // v1-2v2+v3, v1-v3
    const float a3 = d4 - u, b3 = a3 - u;    // v2-2v3+v4, 3v2-4v3+v4
    const float e1 = (a1 + b1) - d1;         // 6 (c1 - v2) = 2 d0 - 7 d1
    const float e2 = u - d1;                 // 6 (c2 - v2) = 2 d3 - d1
    const float e3 = (u + d3) - a3;          // 6 (c3 - v2) = 5 d3 - d4
    const float s1 = fmaf(kWenoK, a1 * a1, b1 * b1);
    const float s2 = fmaf(kWenoK, a2 * a2, b2 * b2);
    const float s3 = fmaf(kWenoK, a3 * a3, b3 * b3);
    const float w1 = rcp_approx(fmaf(s1, s1, kWenoFloor));
    const float w2 = 6.f * rcp_approx(fmaf(s2, s2, kWenoFloor));
    const float w3 = 3.f * rcp_approx(fmaf(s3, s3, kWenoFloor));
    const float inv = rcp_approx(6.f * ((w1 + w2) + w3));
    return fmaf(w1, e1, fmaf(w2, e2, w3 * e3)) * inv;
}

// weno5_corr<float> for two velocities at once (the same operations, element by element;
// the reciprocals and the multiplications by the scaled ideal weights stay scalar): about
// half the issued arithmetic of two scalar calls
static __device__ __forceinline__ float2 weno5_corr2(float2 v0, float2 v1, float2 v2, float2 v3, float2 v4)
{
    const float2 d0 = sub2(v0, v2), d1 = sub2(v1, v2), d3 = sub2(v3, v2), d4 = sub2(v4, v2);
    const float2 t = add2(d1, d1), u = add2(d3, d3);
    const float2 a1 = sub2(d0, t), b1 = sub2(a1, t);
    const float2 a2 = add2(d1, d3), b2 = sub2(d1, d3);
    const float2 a3 = sub2(d4, u), b3 = sub2(a3, u);
    const float2 e1 = sub2(add2(a1, b1), d1), e2 = sub2(u, d1), e3 = sub2(add2(u, d3), a3);
    const float2 K = splat(kWenoK), F = splat(kWenoFloor);
    const float2 s1 = fma2(K, mul2(a1, a1), mul2(b1, b1));
    const float2 s2 = fma2(K, mul2(a2, a2), mul2(b2, b2));
    const float2 s3 = fma2(K, mul2(a3, a3), mul2(b3, b3));
    const float2 q1 = fma2(s1, s1, F), q2 = fma2(s2, s2, F), q3 = fma2(s3, s3, F);
    const float2 w1 = make_float2(rcp_approx(q1.x), rcp_approx(q1.y));
    const float2 w2 = make_float2(6.f * rcp_approx(q2.x), 6.f * rcp_approx(q2.y));
    const float2 w3 = make_float2(3.f * rcp_approx(q3.x), 3.f * rcp_approx(q3.y));
    const float2 sw = add2(add2(w1, w2), w3);
    const float2 inv = make_float2(rcp_approx(6.f * sw.x), rcp_approx(6.f * sw.y));
    return mul2(fma2(w1, e1, fma2(w2, e2, mul2(w3, e3))), inv);
}

// ---- two velocities of either storage type: float2 by the packed instructions above,
// double2 component by component (the compiler merges equal components)
static __device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
static __device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
static __device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
static __device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
static __device__ __forceinline__ double2 splat(double a) { return make_double2(a, a); }
// and single velocities of either type by the same names
#define LBS_SCALAR(T)                                                                  \
    static __device__ __forceinline__ T add2(T a, T b) { return a + b; }               \
    static __device__ __forceinline__ T sub2(T a, T b) { return a - b; }               \
    static __device__ __forceinline__ T mul2(T a, T b) { return a * b; }               \
    static __device__ __forceinline__ T fma2(T a, T b, T c) { return fma(a, b, c); }
LBS_SCALAR(float)
LBS_SCALAR(double)
#undef LBS_SCALAR
template <typename P> struct Constant {
    static __device__ __forceinline__ P of(double a) { return P(a); }
};
template <> struct Constant<float2> {
    static __device__ __forceinline__ float2 of(double a) { return splat(float(a)); }
};
template <> struct Constant<double2> {
    static __device__ __forceinline__ double2 of(double a) { return splat(a); }
};
template <typename T> struct Two;
template <> struct Two<float> { typedef float2 type; };
template <> struct Two<double> { typedef double2 type; };

// WENO-5 correction from differences that the march carries from one interface to the next.
// With D12 = v2 - v1, D23 = v3 - v2 and the second differences A_j = v_{j-1} - 2 v_j + v_{j+1}
// (and K A_j^2, K = 13/3) the indicators are 4 sigma_1 = K A_1^2 + (A_1 + 2 D12)^2,
// 4 sigma_2 = K A_2^2 + (D12 + D23)^2, 4 sigma_3 = K A_3^2 + (A_3 - 2 D23)^2.  A_1 and A_2 of
// one interface are A_2 and A_3 of the one before, so a step forms one first and one second
// difference instead of four differences and six combinations: 12 instructions less.
// The candidates (e_q as in weno5_corr) are e_1 / 3 = D12 + 2/3 A_1, 2 e_2 = 2 (2 D23 + D12),
// e_3 = 3 D23 - A_3, which carry the ideal weights 1 : 6 : 3 in them; with W_q = 1 / (4 sigma_q)^2
// twice the correction is (W_1 e_1 / 3 + 2 W_2 (2 D23 + D12) + W_3 e_3) / (W_1 + 3 (2 W_2 + W_3)).
// The march carries twice the corrections (their difference enters by an FMA): six scalar
// multiplications less per pair of velocities than weights and sum scaled one by one.
// Measured, stage kernels per step: 256 x C2 960 -> 944 us, 32 x C3 943 -> 927, the sweep 362 ->
// 357; in FP64, where a multiplication costs most, 16 x C2 2013 -> 1914.
// The second differences are held negated, for the packed instructions have no negation.
template <typename P>
struct Carried {
    P v3, d12, d23, n1, k1, k2, n2;  // v3 the newest cell value; n = -A, k = K A^2
};
// from the 4 sigma_q and the candidates e_1 / 3, (2 D23 + D12), e_3: twice the correction
static __device__ __forceinline__ float2 carried_weights(float2 s1, float2 s2, float2 s3, float2 e1, float2 e2,
                                                         float2 e3)
{
    const float2 F = splat(kWenoFloor);
    const float2 q1 = fma2(s1, s1, F), q2 = fma2(s2, s2, F), q3 = fma2(s3, s3, F);
    const float2 w1 = make_float2(rcp_approx(q1.x), rcp_approx(q1.y));
    const float2 w2 = make_float2(rcp_approx(q2.x), rcp_approx(q2.y));
    const float2 w3 = make_float2(rcp_approx(q3.x), rcp_approx(q3.y));
    const float2 w22 = add2(w2, w2), sw = fma2(splat(3.f), add2(w22, w3), w1);
    const float2 inv = make_float2(rcp_approx(sw.x), rcp_approx(sw.y));
    return mul2(fma2(w1, e1, fma2(w22, e2, mul2(w3, e3))), inv);
}
static __device__ __forceinline__ float carried_weights(float s1, float s2, float s3, float e1, float e2, float e3)
{
    const float w1 = rcp_approx(fmaf(s1, s1, kWenoFloor));
    const float w2 = rcp_approx(fmaf(s2, s2, kWenoFloor));
    const float w3 = rcp_approx(fmaf(s3, s3, kWenoFloor));
    const float w22 = w2 + w2;
    return fmaf(w1, e1, fmaf(w22, e2, w3 * e3)) * rcp_approx(fmaf(3.f, w22 + w3, w1));
}
static __device__ __forceinline__ double carried_weights(double q1, double q2, double q3, double e1, double e2,
                                                         double e3)
{
    const int top = max(__double2hiint(q1), max(__double2hiint(q2), __double2hiint(q3)));  // sigma >= 0
    const double s = __hiloint2double(0x7FE00000 - (top & 0x7FF00000), 0), floor_ = 0x1p-250;
    const double s1 = fma(q1, s, floor_), s2 = fma(q2, s, floor_), s3 = fma(q3, s, floor_);
    const double p1 = s2 * s3, p2 = s1 * s3, p3 = s1 * s2;
    const double w1 = p1 * p1, w22 = 2.0 * p2 * p2, w3 = p3 * p3;
    return fma(w1, e1, fma(w22, e2, w3 * e3)) * rcp_newton(fma(3.0, w22 + w3, w1));
}
static __device__ __forceinline__ double2 carried_weights(double2 s1, double2 s2, double2 s3, double2 e1, double2 e2,
                                                          double2 e3)
{
    return make_double2(carried_weights(s1.x, s2.x, s3.x, e1.x, e2.x, e3.x),
                        carried_weights(s1.y, s2.y, s3.y, e1.y, e2.y, e3.y));
}
// twice the correction of the interface ahead of v2 for the new value v4; advances the differences
template <typename P>
static __device__ __forceinline__ P carried_corr(Carried<P>& w, P v4)
{
    typedef Constant<P> C;
    const P d34 = sub2(v4, w.v3), n3 = sub2(w.d23, d34), k3 = mul2(mul2(C::of(13.0 / 3.0), n3), n3);
    const P b1 = fma2(C::of(-2.0), w.d12, w.n1), b2 = add2(w.d12, w.d23), b3 = fma2(C::of(2.0), w.d23, n3);
    const P e1 = fma2(C::of(-2.0 / 3.0), w.n1, w.d12), e2 = fma2(C::of(2.0), w.d23, w.d12);
    const P e3 = fma2(C::of(3.0), w.d23, n3);
    const P c = carried_weights(fma2(b1, b1, w.k1), fma2(b2, b2, w.k2), fma2(b3, b3, k3), e1, e2, e3);
    w.v3 = v4;
    w.d12 = w.d23;
    w.d23 = d34;
    w.n1 = w.n2;
    w.n2 = n3;
    w.k1 = w.k2;
    w.k2 = k3;
    return c;
}
// the state before the first of them, from the values v0 .. v3 of its stencil
template <typename P>
static __device__ __forceinline__ Carried<P> carried_start(P v0, P v1, P v2, P v3)
{
    const P K = Constant<P>::of(13.0 / 3.0);
    Carried<P> w;
    w.v3 = v3;
    w.d12 = sub2(v2, v1);
    w.d23 = sub2(v3, v2);
    w.n1 = sub2(sub2(v1, v0), w.d12);
    w.n2 = sub2(w.d12, w.d23);
    w.k1 = mul2(mul2(K, w.n1), w.n1);
    w.k2 = mul2(mul2(K, w.n2), w.n2);
    return w;
}

template <typename T>
__device__ __forceinline__ T weno5(T v0, T v1, T v2, T v3, T v4)
{
    return v2 + weno5_corr<T>(v0, v1, v2, v3, v4);
}

// The warp's sum of a double-float or FP64 value, in every lane
template <typename R>
static __device__ __forceinline__ R warp_sum(R v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = r_add(v, r_shfl_xor(v, o));
    return v;
}
// Block-wide FP64 sum (all threads get the result); deterministic order.
static __device__ double block_sum(double v, double* red)
{
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < nw; ++i) s += red[i];
    __syncthreads();
    return s;
}

// Warp reduce-scatter of 16 values: afterwards lane l holds the warp total of
// value m(l) = 8 b4 + 4 b3 + 2 b2 + b1 (b = bits of l); lanes l, l^1 agree.
// 16 shuffles per lane instead of 16 x 5 for 16 separate butterflies.
template <typename A>
__device__ __forceinline__ A reduce_scatter16(A (&v)[16], int lane)
{
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool hi = lane & 16;
        const A send = hi ? v[i] : v[i + 8], keep = hi ? v[i + 8] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool hi = lane & 8;
        const A send = hi ? v[i] : v[i + 4], keep = hi ? v[i + 4] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool hi = lane & 4;
        const A send = hi ? v[i] : v[i + 2], keep = hi ? v[i + 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool hi = lane & 2;
        const A send = hi ? v[0] : v[1], keep = hi ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// The warp totals of 13 FP32 values per lane (q[3].y .. w unused) through 2 KB of shared memory:
// each lane writes its values as four 16-byte words, then lane 4 s + g sums word g of lanes
// s, s + 8, s + 16, s + 24 (packed adds) and a reduce-scatter over s finishes.  Word w of lane
// l sits at w ^ (l / 2 mod 4), which keeps both directions free of bank conflicts.  29
// instructions instead of the 62 of reduce_scatter16.  Returns the total of value
// 4 g + 2 b4 + b3 (g = lane mod 4, b = bits of the lane); lanes l, l ^ 4 agree.
static __device__ __forceinline__ float warp_totals13(const float4 (&q)[4], float4* buf, int lane)
{
    float4* row = buf + lane * 4;
    const int x = (lane >> 1) & 3;
    __syncwarp();  // the previous cell's reads are done
#pragma unroll
    for (int w = 0; w < 4; ++w) row[w ^ x] = q[w];
    __syncwarp();
    const int g = lane & 3, s = lane >> 2;
    const float4* col = buf + s * 4 + (g ^ ((s >> 1) & 3));  // rows s + 8 i have the same swizzle
    const float4 a = col[0], b = col[32], c = col[64], d = col[96];
    const float2 t0 = add2(add2(make_float2(a.x, a.y), make_float2(b.x, b.y)),
                           add2(make_float2(c.x, c.y), make_float2(d.x, d.y)));
    const float2 t1 = add2(add2(make_float2(a.z, a.w), make_float2(b.z, b.w)),
                           add2(make_float2(c.z, c.w), make_float2(d.z, d.w)));
    const bool h4 = lane & 16, h3 = lane & 8;
    const float2 keep = h4 ? t1 : t0, send = h4 ? t0 : t1;
    const float2 u = add2(keep, make_float2(__shfl_xor_sync(0xffffffffu, send.x, 16),
                                            __shfl_xor_sync(0xffffffffu, send.y, 16)));
    float v = (h3 ? u.y : u.x) + __shfl_xor_sync(0xffffffffu, h3 ? u.x : u.y, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 4);
}

// shared-memory layout of a stage CTA (offsets in bytes): the staged rows of the
// step's start state d (cells z0-3 .. z0+zn+2) and the cell records (by bulk copy), the
// per-axis factors of this chunk's nodes, 1/dz, and the per-warp moment sums.  The stage
// input's increment (stages 2 and 3) is read from global memory during the march.
struct StageSmem {
    size_t fin, rec, g, idz, red, sc, total;
};
// values per cell of the factor region: one per node of x, of y and of the chunk's z nodes, or
// (grouped layout) y's, then x's and z's, FP32 ones twice; a multiple of four either way
__host__ __device__ inline int factor_stride(int Qx, int Qy, int nzm, bool grouped, int esize)
{
    return (Qy + (Qx + nzm) * (grouped && esize == 4 ? 2 : 1) + 3) & ~3;
}
// scalars per cell of the grouped layout: u, q, (1 - Pr)/(n T^2), 1/(5T), and -1/tau and 1/dz
// times the stage's share of dt
enum { S_UX = 0, S_UY, S_UZ, S_QX, S_QY, S_QZ, S_CS, S_I5T, S_NITAU, S_IDZ, S_COUNT };
__host__ __device__ inline size_t pad16(size_t b) { return (b + 15) & ~size_t(15); }
__host__ __device__ inline StageSmem stage_smem(int zn, int KC, int G, int esize, int asize, int rstride,
                                                    bool grouped, int zsplit)
{
    StageSmem L;
    size_t o = 0;
    L.fin = o; o += (size_t)(zn + 6) * KC * esize;
    // grouped layout, FP32: the warps' moment scratch takes the records' place after the
    // factors have been formed from them
    const size_t scratch = grouped && esize == 4 ? (size_t)kThreads * 16 * 4 : 0, rec = (size_t)zn * rstride * esize;
    L.rec = o; o += rec > scratch ? rec : scratch;
    L.g = o; o += pad16((size_t)zn * G * esize);
    L.idz = o; o += pad16((size_t)zn * esize);
    L.red = o; o += (size_t)zn * (kThreads / 32 / zsplit) * 16 * asize;
    L.sc = o; o += grouped ? (size_t)zn * S_COUNT * 8 : 0;  // 80 bytes a cell in either type
    // the folded-in finalisation's cell group lies over all of it: the 32 columns of a three-cell
    // FP64 tile at two to four velocities are shorter (3200 bytes against 3312)
    const size_t fin = esize == 4 ? sizeof(FinShared<float, 4>) : sizeof(FinShared<double, 4>);
    L.total = o > fin ? o : fin;
    return L;
}

// ---- the FP32 state's rounding residual --------------------------------------
// The state d is stored as hi (FP32) plus lo, |lo| <= ulp(hi) / 2, kept as a 16-bit
// integer q = round(lo / ulp(hi) * 2^15).  The RK increment of a step near the steady
// state is far below ulp(hi); added to hi alone it would be rounded away and the state
// would stall at a distance of about eps_32 / (lambda dt) from the steady state
// (lambda the decay rate of its slowest mode).  With lo the increment accumulates in
// lo until it carries into hi; what is lost is below 2^-16 ulp(hi) per step.
// ulp(hi) = 2^(E - 150) for the biased exponent E of a normal hi, so
// lo / ulp(hi) * 2^15 = lo * 2^(165 - E), a power of two built in the exponent field
// from the masked exponent bits of hi (E clamped below at 38; the decoding scale
// 2^(E - 165) is then zero: a hi below 2^-88 keeps no residual).
// Both without int/float conversion instructions: for |x| < 2^22, fma(lo, s, 1.5 2^23)
// holds round-to-nearest-even(lo s) in its low mantissa bits (s is a power of two, so the
// product is exact and rounded once, as __float2int_rn rounds it), and 2^23 + u is exact
// for a 16-bit u, so q = float bits of (2^23 + 2^15 + q) minus (2^23 + 2^15).
static __device__ __forceinline__ unsigned lo_bits(float lo, float hi)  // q in the low 16 bits
{
    const unsigned m = max(__float_as_uint(hi) & 0x7f800000u, 38u << 23);
    const float s = __uint_as_float((292u << 23) - m);  // 2^(165 - E)
    return __float_as_uint(fmaf(lo, s, 12582912.0f));
}
static __device__ __forceinline__ unsigned short lo_encode(float lo, float hi)
{
    return static_cast<unsigned short>(lo_bits(lo, hi));
}
static __device__ __forceinline__ unsigned lo_encode2(float2 lo, float2 hi)  // two residuals, x low
{
    return __byte_perm(lo_bits(lo.x, hi.x), lo_bits(lo.y, hi.y), 0x5410);
}
static __device__ __forceinline__ float lo_decode(unsigned q16, float hi)  // q in the low 16 bits
{
    const unsigned m = max(__float_as_uint(hi) & 0x7f800000u, 38u << 23);
    const float s = __uint_as_float(m - (38u << 23));  // 2^(E - 165), zero for E = 38
    const float q = __uint_as_float((q16 & 0xffffu) ^ 0x4B008000u) - 8421376.0f;  // the int16 q
    return q * s;
}

// ----------------------------------------------------------------------------
// stage_kernel<T, V, STAGE, RED>: STAGE 1..3 are the RK stages; STAGE 0 only
// analyses F0 (moments and wall fluxes) without writing F.  RED selects the
// phi / chi model (Sec. III, Eqs. boltz_red, sred_def): j = 0 is phi, j = 1 chi.
// ----------------------------------------------------------------------------
// n / d for 0 <= n < 2^15 and 2 <= d < 2^14 from m = ceil(2^32 / d) (the error m d - 2^32 < d
// times n stays below 2^32); m = 0 stands for d = 1
static __device__ __forceinline__ int div_small(int n, unsigned m) { return m ? __umulhi(n, m) : n; }
// the walls' extrapolation weights and densities in the storage type
static __device__ __forceinline__ const Walls<float>& wall_weights(const InstDev& I, float) { return I.walls2; }
static __device__ __forceinline__ const Walls<double>& wall_weights(const InstDev& I, double) { return I.walls; }
static __device__ __forceinline__ const float* stored_nw(const InstDev& I, float) { return I.nw->f; }
static __device__ __forceinline__ const double* stored_nw(const InstDev& I, double) { return I.nw->d; }

template <typename T, bool PACK> struct PackedAs { typedef T type; };
template <> struct PackedAs<float, true> { typedef float2 type; };

// Minimum resident CTAs per SM requested from the register allocator: the
// per-velocity registers grow with V; the rarely taken finalisation
// path may spill instead of lowering occupancy.
template <typename T, int V, int ZW> struct MinBlocks {
    // FP32 at V = 4 fits 128 registers (four CTAs, sixteen warps per SM); FP64 values take
    // two registers each and keep three.  The small batches of ZW = 4 take what registers
    // they can use.
    static constexpr int value = ZW == 4 ? (V == 1 ? 4 : 2)
                                 : V == 1 ? (sizeof(T) == 4 ? 7 : 5)
                                 : V == 2 ? (sizeof(T) == 4 ? 6 : 4)
                                          : sizeof(T) == 4 ? 4 : 3;
};

// GRP (V = 4, full model, Qy a multiple of 4 in every instance): a thread's four velocities
// are adjacent, so they share the x and the z node.
// ZW = 4: the CTA's warps share 32 V velocities and split the tile's cells between them, for
// batches too small to fill the GPU otherwise: a warp marches a quarter of the cells (one of a
// four-cell tile), so a tile takes a quarter of the steps.  Rows, records and factors are
// staged once for the four.
// Measured, us per step: one C1 channel in FP64 102 -> 63, the low-Mach runs 107 -> 88, one C2
// channel in FP64 285 -> 225.
template <typename T, int V, int STAGE, bool RED, bool GRP, int ZW>
__global__ void __launch_bounds__(kThreads, MinBlocks<T, V, ZW>::value)
stage_kernel(const InstDev* __restrict__ insts, const Tile* __restrict__ tiles, int fuse)
{
    typedef typename Acc<T>::type A;
    constexpr bool kLo = sizeof(T) == 4;  // FP32 storage keeps the rounding residual of d
    constexpr bool kD = STAGE >= 2;       // the stage input is d + an increment
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ double wall_red[8 * (kThreads / 32)];
    __shared__ InstDev sI;
    typedef typename Real<T>::type R;
    const Tile tile = tiles[blockIdx.x];
    const InstDev& I = stage_descriptor(insts + tile.inst, &sI);

    const int Nz = I.Nz, Q = I.Q, Qx = I.Qx, Qy = I.Qy, Qz = I.Qz, QxQy = I.QxQy;
    const int z0 = tile.z0, zn = tile.zn;            // cells z0 .. z0+zn-1 (0-based)
    constexpr int NT = kThreads / ZW, KC = NT * V;   // threads along the velocities
    // chunks never straddle p_z = 0: this chunk's velocities share the sign of p_z
    const int Qh = Q >> 1, sgc = tile.chunk >= I.nchh;
    const int k0 = sgc * Qh + (tile.chunk - sgc * I.nchh) * KC;
    const int kend = min((sgc + 1) * Qh, k0 + KC), kn = kend - k0;
    const int zm_lo = div_small(k0, I.mQxQy), zm_hi = div_small(kend - 1, I.mQxQy), nzm = zm_hi - zm_lo + 1;
    const int G = factor_stride(Qx, Qy, nzm, GRP, sizeof(T));  // per-cell factors held in smem
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ctid = ZW == 1 ? tid : lane, zw = ZW == 1 ? 0 : warp;
    // this warp's part of the tile: cells zb .. zb + zc - 1
    const int zb = zn * zw / ZW, zc = zn * (zw + 1) / ZW - zb;

    const int rstride = I.rec_stride;
    const StageSmem L = stage_smem(zn, KC, G, sizeof(T), sizeof(A), rstride, GRP, ZW);
    T* Fs = reinterpret_cast<T*>(smem_raw + L.fin);   // d rows: cells z0-3 .. z0+zn+2
    T* recs = reinterpret_cast<T*>(smem_raw + L.rec); // records of cells z0 .. z0+zn-1
    T* gsm = reinterpret_cast<T*>(smem_raw + L.g);
    T* idzs = reinterpret_cast<T*>(smem_raw + L.idz);
    A* red = reinterpret_cast<A*>(smem_raw + L.red);  // per-warp moment sums
    T* scs = reinterpret_cast<T*>(smem_raw + L.sc);   // grouped layout: the cells' scalars

    const int s_lo = max(0, z0 - 3), s_hi = min(Nz - 1, z0 + zn + 2);
    const T* Rg = static_cast<const T*>(I.rec) + (size_t)z0 * rstride;
    const size_t rec_bytes = (size_t)zn * rstride * sizeof(T);

    // ---- 1. stage the input rows and the cell records by TMA bulk copies: warp 0 waits for
    //         the predecessor and issues them while the other warps load the constants below
    //         (all before the wait, 256 x C2 took 1121 us of stage kernels per step instead
    //         of 1061)
    if (warp == 0) {
        wait_predecessor();
        const int act = *I.active, c1 = *I.cur;  // both loads in flight
        if (tid == 0 && I.bulk && act != 0) {
            const T* H = static_cast<const T*>(c1 ? I.F1 : I.F0);
            mbar_init(&bar, 1);
            fence_barrier_init();
            const uint32_t bytes = kn * sizeof(T);
            uint32_t total = bytes * (s_hi - s_lo + 1);
            if (STAGE > 0) total += rec_bytes;
            mbar_expect_tx(&bar, total);
            for (int s = s_lo; s <= s_hi; ++s)
                bulk_g2s(Fs + (size_t)(s - z0 + 3) * KC, H + (size_t)s * Q + k0, bytes, &bar);
            if (STAGE > 0) bulk_g2s(recs, Rg, rec_bytes, &bar);  // records are 16-byte multiples
        }
        // The tile's increments and residuals into L2: the march reads them one step ahead (about
        // a microsecond with four CTAs per SM), which covers L2's latency but not HBM's.  For
        // FP32 batches larger than L2 (I.prefetch; FP64 is bound by its arithmetic).  Measured, us
        // per step: 256 x C2 1048.7 -> 1045.0, 32 x C3 992.6 -> 987.6, the sweep (64 instances)
        // 432 -> 427.8, 60 phi / chi channels of 16 x (2 x 60) nodes and 150 cells 739.6 -> 729.5;
        // 40 channels of 720 velocities and 200 cells, which fit L2, 186.7 -> 188.1.
        if constexpr (kD && kLo && V == 4) {
            if (I.prefetch && act != 0) {
                const T* D = static_cast<const T*>(STAGE == 3 ? I.F2 : c1 ? I.F0 : I.F1);
                for (int s = s_lo + lane; s <= s_hi; s += 32) bulk_prefetch(D + (size_t)s * Q + k0, kn * sizeof(T));
                if constexpr (STAGE == 3) {
                    const unsigned short* lo = I.L0 + (size_t)z0 * Q + k0;
                    if (((reinterpret_cast<uintptr_t>(lo) & 15) | (Q & 7) | (kn & 7)) == 0)
                        for (int s = lane; s < zn; s += 32) bulk_prefetch(lo + (size_t)s * Q, kn * 2);
                }
            }
        }
    }

    // per-velocity constants: p (and |p_z| for the fluxes), the weight w and |p|^2 for the
    // moments (formed from them per cell: fewer registers than 13 weighted monomials)
    // FP32 with an even V: the thread's velocities are adjacent pairs (2 tid, 2 tid + 1,
    // 2 tid + 2 kThreads, ...), so that a pair is one 64-bit word in memory and one
    // operand of the packed FP32 instructions; else tid + v kThreads.  voff(v) is v's
    // offset from the thread's first velocity tbase.
    // Grouped layout: the four velocities 4 tid .. 4 tid + 3.
    constexpr bool kPair = sizeof(T) == 4 && V % 2 == 0;
    const int tbase = GRP ? 4 * ctid : kPair ? 2 * ctid : ctid;
    auto voff = [](int v) { return GRP ? v : kPair ? (v & 1) + (v >> 1) * 2 * NT : v * NT; };
    int ii[V], jj[V], zz[V], kl[V];
    T px[V], py[V], pz[V], apz[V];
    A wv[V], yv[V], p2v[V], wm[V];  // weight; p_y for the moments; |p|^2; w of the mass flux
    bool ok[V], chi[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        kl[v] = tbase + voff(v);
        ok[v] = kl[v] < kn;
        const int kc = ok[v] ? k0 + kl[v] : kend - 1;
        // (grouped: kn is a multiple of 4, so v = 0 stands for all four but for the y node; past
        // the chunk the y nodes still lie inside the table)
        const int ky = div_small(kc, I.mQy);  // kc / Qy
        zz[v] = GRP && v ? zz[0] : div_small(kc, I.mQxQy);
        ii[v] = GRP && v ? ii[0] : ky - zz[v] * Qx;
        jj[v] = GRP ? (v ? jj[0] + v : (kc - ky * Qy) & ~3) : kc - ky * Qy;
        const int sg = zz[v] >= Qz, m = zz[v] - sg * Qz;
        px[v] = GRP && v ? px[0] : ld<T>(I.px, ii[v]);
        py[v] = ld<T>(I.py, jj[v]);
        const T x = GRP && v ? apz[0] : ld<T>(I.xi, m);
        pz[v] = sg ? -x : x;
        apz[v] = x;
        wv[v] = ok[v] ? A(ld<T>(I.wx, ii[v]) * ld<T>(I.wy, jj[v]) * ld<T>(I.wz, m)) : A(0);
        const A X = px[v], Y = py[v], Z = pz[v];
        yv[v] = Y;
        p2v[v] = X * X + Y * Y + Z * Z;
        chi[v] = RED && jj[v] == 1;
        wm[v] = chi[v] ? A(0) : wv[v];
        if (RED) {
            // p_y = 0 on both fields.  chi = int p_y^2 f dp_y carries the p_y^2 moments:
            // sum chi -> sum p_y^2 f, sum p_a chi -> sum p_y^2 p_a f (a = x, z), nothing else.
            // py[v] then holds -(the Shakhov offset of Eq. sred_def): -4/5 for phi, -2/5 for chi.
            py[v] = jj[v] ? T(-0.4) : T(-0.8);
        }
    }
    if (STAGE > 0 && !GRP)
        for (int c = tid; c < zn; c += kThreads) idzs[c] = ld<T>(I.inv_dz, z0 + c);
    if (warp != 0) wait_predecessor();
    // from here on: what other kernels write
    const int act = *I.active, cur = *I.cur;  // cur: which of F0 / F1 holds the step's start state
    if (act == 0) return;

    // Buffers (Eq. rk3 in increment form, F_l the step's start state d):
    //   stage 1: d1 = dt L[F_l]                  -> the other of F0 / F1
    //   stage 2: d2 = (d1 + dt L[F_l + d1]) / 4  -> F2
    //   stage 3: F_l + 2/3 (d2 + dt L[F_l + d2]) -> the other of F0 / F1 (over d1)
    const T* Hg = static_cast<const T*>(cur ? I.F1 : I.F0);
    T* Og = static_cast<T*>(cur ? I.F0 : I.F1);
    // the stage input's increment (stages 2, 3) is read from global memory, one march step
    // ahead.  Not through the read-only path: the CTA may start while the launch that writes
    // the increment still runs (wait_predecessor), and only ordinary loads are then coherent.
    const T* Dg = STAGE == 2 ? Og : static_cast<const T*>(I.F2);
    T* Fout = STAGE == 2 ? static_cast<T*>(I.F2) : Og;
    // rows that are not 16-byte aligned: plain loads
    if (!I.bulk) {
        for (int s = s_lo; s <= s_hi; ++s)
            for (int kl = tid; kl < kn; kl += kThreads) Fs[(size_t)(s - z0 + 3) * KC + kl] = Hg[(size_t)s * Q + k0 + kl];
        if (STAGE > 0)
            for (int e = tid; e < zn * rstride; e += kThreads) recs[e] = Rg[e];
    }
    __syncthreads();  // the barrier's initialisation

    // ---- 3. wait for the copies (bounded).  A CTA whose wait runs out flags the
    //         instance (STATUS_TIMEOUT), then waits a further bounded time for its copies
    //         in flight to land before it leaves, so that none writes shared memory after
    //         the CTA is gone; if that wait runs out too the CTA leaves regardless.
    int late = 0;
    if (I.bulk) {
        for (uint32_t spins = 0;; ++spins) {
            if (spins >= I.wait_limit) { late = 1; break; }
            if (mbar_try_wait(&bar, 0)) break;
        }
    }
    if (__syncthreads_or(late)) {
        if (tid == 0) atomicOr(I.status, STATUS_TIMEOUT);
        uint32_t spins = 0;
        while (!mbar_try_wait(&bar, 0) && ++spins < kDrainLimit) {
        }
        return;
    }

    // ---- 4a. per-cell factors of the truncated Hermite equilibrium (Sec. III) for this
    //          chunk's nodes, as deviations from 1, from the staged records:
    //          dx[i] with R_SCALE applied (R_SCALE (1 + dx) - 1), dy[j], dz[zm]
    if constexpr (GRP && STAGE > 0) {
        // [y][x][z], FP32's x and z values twice (a pair register without moves), and the
        // cell's scalars likewise
        const T dtc = T(I.dt) * (STAGE == 1 ? T(1) : STAGE == 2 ? T(0.25) : T(2.0 / 3.0));
        const int nf = Qy + Qx + nzm + S_COUNT;
        constexpr int dup = sizeof(T) == 4 ? 2 : 1;
        for (int c = warp; c < zn; c += kThreads / 32)  // a warp per cell
        for (int r = lane; r < nf; r += 32) {
            const T* rc = recs + (size_t)c * rstride;
            T g, *to;
            if (r < Qy) {
                gsm[(size_t)c * G + r] = rc[R_DX + Qx + r];  // dy
                continue;
            } else if (r < Qy + Qx) {
                const T s1 = rc[R_SCALE1];
                g = s1 + (T(1) + s1) * rc[R_DX + r - Qy];
                to = gsm + (size_t)c * G + Qy + dup * (r - Qy);
            } else if (r < Qy + Qx + nzm) {
                g = rc[R_DX + r + zm_lo];  // dz[zm]
                to = gsm + (size_t)c * G + Qy + dup * (r - Qy);
            } else {
                const int q = r - (Qy + Qx + nzm);
                // the record holds u at R_UX .., q at R_QX .., 1/tau, cS, 1/(5T)
                g = q < S_QX ? rc[R_UX + q]
                    : q < S_CS ? rc[R_QX + q - S_QX]
                    : q == S_CS ? rc[R_CS]
                    : q == S_I5T ? rc[R_I5T]
                    : q == S_NITAU ? -rc[R_ITAU] * dtc
                                   : ld<T>(I.inv_dz, z0 + c) * dtc;
                to = scs + (c * S_COUNT + q) * dup;
            }
            to[0] = g;
            if (dup == 2) to[1] = g;
        }
    } else if (STAGE > 0) {
        for (int c = warp; c < zn; c += kThreads / 32) {  // a warp per cell
            const T* rc = recs + (size_t)c * rstride;
            const T s1 = rc[R_SCALE1];
            for (int r = lane; r < Qx + Qy + nzm; r += 32) {
                T g;
                if (r < Qx) g = s1 + (T(1) + s1) * rc[R_DX + r];
                else if (r < Qx + Qy) g = rc[R_DX + r];                  // dy[r - Qx]
                else g = rc[R_DX + Qx + Qy + zm_lo + r - Qx - Qy];       // dz[zm]
                gsm[c * G + r] = g;
            }
        }
    }

    // ---- 4b. ghost rows (each thread fills only its own columns).  A ghost row holds
    //          the whole stage-input value d (+ increment); a cell's row holds d.
    const int rbase = 3 - z0;  // smem row of cell s is s + rbase
    const auto& ext_top = wall_weights(I, T(0)).top;
    const auto& ext_bot = wall_weights(I, T(0)).bot;
    const T* nwt = stored_nw(I, T(0));  // n_w - 1 and n_w of the bottom wall, then of the top one
    auto rowval = [&](int row, int col) -> T {  // the stage input of a cell's row
        return kD ? Fs[(size_t)row * KC + col] + __ldca(Dg + (size_t)(row - rbase) * Q + k0 + col)
                  : Fs[(size_t)row * KC + col];
    };
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if (!ok[v] || zw != 0) continue;  // columns past the chunk end hold no data
        T* col = Fs + kl[v];
        if (z0 < 3 && I.half) {  // bounce-back on the centre line: ghost -1-s holds cell s
            // at the mirrored velocity (p_z, p_x reversed: other half range, node Qx-1-i;
            // the Gauss nodes are sorted, so p_x[Qx-1-i] = -p_x[i]).  It lies in the other
            // sign's chunk, so it comes from the stage input in global memory.
            const int zm = zz[v] + (sgc ? -Qz : Qz);
            const int kmir = (zm * Qx + (Qx - 1 - ii[v])) * Qy + jj[v];
            for (int s = 0; s < 3; ++s)
                if (-1 - s + rbase >= 0)
                    col[(size_t)(-1 - s + rbase) * KC] =
                        kD ? Hg[(size_t)s * Q + kmir] + Dg[(size_t)s * Q + kmir] : Hg[(size_t)s * Q + kmir];
        } else if (z0 < 3) {
            if (!sgc) {  // incoming at the bottom wall: n_w times the wall equilibrium, minus 1
                const T ax = ld<T>(I.gwx_bot, ii[v]), ay = ld<T>(I.gwy, jj[v]), az = ld<T>(I.gwz, zz[v]);
                const T a = ax + ay + ax * ay, b = a + az + a * az;
                const T g = nwt[0] + nwt[1] * b;
                for (int s = -3; s <= -1; ++s)
                    if (s + rbase >= 0) col[(size_t)(s + rbase) * KC] = g;
            } else {      // outgoing: quadratic extrapolation (Appendix)
                const T f1 = rowval(0 + rbase, kl[v]), f2 = rowval(1 + rbase, kl[v]), f3 = rowval(2 + rbase, kl[v]);
                const T g0 = ext_bot[0][0] * f1 + ext_bot[0][1] * f2 + ext_bot[0][2] * f3;
                const T g1 = ext_bot[1][0] * g0 + ext_bot[1][1] * f1 + ext_bot[1][2] * f2;
                if (-1 + rbase >= 0) col[(size_t)(-1 + rbase) * KC] = g0;
                if (-2 + rbase >= 0) col[(size_t)(-2 + rbase) * KC] = g1;
                if (-3 + rbase >= 0) col[(size_t)(-3 + rbase) * KC] = g1;  // never read for p_z < 0
            }
        }
        if (z0 + zn + 3 > Nz) {
            const int smax = z0 + zn + 2;
            if (sgc) {
                const T ax = ld<T>(I.gwx_top, ii[v]), ay = ld<T>(I.gwy, jj[v]), az = ld<T>(I.gwz, zz[v]);
                const T a = ax + ay + ax * ay, b = a + az + a * az;
                const T g = nwt[2] + nwt[3] * b;
                for (int s = Nz; s <= Nz + 2; ++s)
                    if (s <= smax) col[(size_t)(s + rbase) * KC] = g;
            } else {
                const T f1 = rowval(Nz - 1 + rbase, kl[v]), f2 = rowval(Nz - 2 + rbase, kl[v]),
                        f3 = rowval(Nz - 3 + rbase, kl[v]);
                const T g0 = ext_top[0][0] * f1 + ext_top[0][1] * f2 + ext_top[0][2] * f3;
                const T g1 = ext_top[1][0] * g0 + ext_top[1][1] * f1 + ext_top[1][2] * f2;
                if (Nz <= smax) col[(size_t)(Nz + rbase) * KC] = g0;
                if (Nz + 1 <= smax) col[(size_t)(Nz + 1 + rbase) * KC] = g1;
                if (Nz + 2 <= smax) col[(size_t)(Nz + 2 + rbase) * KC] = g1;  // never read for p_z > 0
            }
        }
    }

    __syncthreads();  // per-cell factors complete

    if constexpr (GRP) {
        // ---- 5 (grouped layout). The march of the scalar section below with four adjacent
        // velocities per thread, as two pairs.  They share the x and the z node, so what depends
        // on those alone -- xi_x, xi_z, their squares, the products with q, the target's x and z
        // factors, the advection factor -- is formed once per cell, and the moments are the
        // powers 0 .. 3 of xi_y summed over the four, combined with the shared xi_x and xi_z
        // afterwards.  A row, an increment, an output of the thread is one 128-bit word (FP64:
        // two).  The WENO differences are carried (carried_corr), so no window of values shifts.
        // Measured, stage kernels per step against the pair march (FP32) and the scalar march
        // (FP64): 256 x C2 1061 -> 987 us, 32 x C3 1049 -> 962, the sweep 405 -> 375; 16 x C2
        // in FP64 3063 -> 2004 us (2365 at the same 12-cell tiles); now 944, 926, 357 and 1914
        // with the weights of carried_weights and the prefetch above.  Instructions per update of
        // the three FP32 stages: 112 / 137 / 155 -> 85 / 99 / 120; bound by latency at four CTAs
        // per SM (2.0 to 2.2 instructions per cycle of 4), then issue.
        typedef typename Two<T>::type P;
        struct alignas(16) Quad { P p[2]; };
        auto quad = [](const T* q) -> Quad {  // 16-byte aligned
            Quad r;
            if constexpr (sizeof(T) == 4) {
                const float4 v = *reinterpret_cast<const float4*>(q);
                r.p[0] = make_float2(v.x, v.y);
                r.p[1] = make_float2(v.z, v.w);
            } else {
                r.p[0] = *reinterpret_cast<const double2*>(q);
                r.p[1] = *reinterpret_cast<const double2*>(q + 2);
            }
            return r;
        };
        auto quad_g = [](const T* q) -> Quad {
            Quad r;
            if constexpr (sizeof(T) == 4) {
                const float4 v = __ldca(reinterpret_cast<const float4*>(q));
                r.p[0] = make_float2(v.x, v.y);
                r.p[1] = make_float2(v.z, v.w);
            } else {
                r.p[0] = __ldca(reinterpret_cast<const double2*>(q));
                r.p[1] = __ldca(reinterpret_cast<const double2*>(q + 2));
            }
            return r;
        };
        auto dup = [](const T* q) -> P {  // a value stored for both lanes
            if constexpr (sizeof(T) == 4) return *reinterpret_cast<const float2*>(q);
            else return splat(*q);
        };
        constexpr int kDup = sizeof(T) == 4 ? 2 : 1;
        // FP32: two steps per iteration, after which the carried values are back in their
        // registers (20 moves per step less)
        constexpr int kUnroll = sizeof(T) == 4 ? 2 : 1;
        const P zero = splat(T(0));
        const bool in = ok[0] && zc > 0;  // (ZW = 4: a three-cell tile leaves a warp without cells)
        const P PX = splat(px[0]), PZ = splat(pz[0]), NAPZ = splat(-apz[0]);
        P PY[2], WV[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            PY[p].x = py[2 * p];
            PY[p].y = py[2 * p + 1];
            WV[p].x = wv[2 * p];
            WV[p].y = wv[2 * p + 1];
        }
        const int sdir = sgc ? -1 : 1;
        const long rstep = sdir * (long)KC, ostep = sdir * (long)Q;
        const int zw0 = sgc ? z0 + zb + zc + 2 : z0 + zb - 3;  // the cell of march row 0
        const T* rp = Fs + (size_t)(sgc ? zb + zc + 5 : zb) * KC + tbase;  // march row r: rp + r rstep
        const T* dcol = Dg + k0 + tbase;
        auto inc_row = [&](int s) -> Quad {  // the increments of cell s (zero for a ghost row)
            Quad q;
            q.p[0] = q.p[1] = zero;
            if (kD && in && (unsigned)s < (unsigned)Nz) q = quad_g(dcol + (long)s * Q);
            return q;
        };
        // rows 0 .. 4 (the cell's three upwind neighbours, the cell, the next one) give the
        // differences and the correction of the interface behind the first cell
        Carried<P> w[2];
        P CM[2];
        {
            Quad r[5];
#pragma unroll
            for (int d = 0; d < 5; ++d) {
                r[d] = quad(rp + d * rstep);
                const Quad q = inc_row(zw0 + d * sdir);
#pragma unroll
                for (int p = 0; p < 2; ++p) r[d].p[p] = kD ? add2(r[d].p[p], q.p[p]) : r[d].p[p];
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                w[p] = carried_start(r[0].p[p], r[1].p[p], r[2].p[p], r[3].p[p]);
                CM[p] = carried_corr(w[p], r[4].p[p]);
            }
        }
        // the next row: its shared-memory part is read and its increments are added a step ahead
        int sn = zw0 + 5 * sdir;
        Quad NV = quad(rp + 5 * rstep);
        {
            const Quad q = inc_row(sn);
#pragma unroll
            for (int p = 0; p < 2; ++p) NV.p[p] = kD ? add2(NV.p[p], q.p[p]) : NV.p[p];
        }
        sn += sdir;
        Quad DN = inc_row(sn);
        const size_t orow0 = (size_t)(sgc ? z0 + zb + zc - 1 : z0 + zb) * Q + k0 + tbase;
        T* outp = Fout + orow0;
        const T* dop = kD ? Dg + orow0 : nullptr;
        unsigned short* lop = kLo && STAGE == 3 ? I.L0 + orow0 : nullptr;
        const T* dnp = dcol + (long)sn * Q;  // increments of the row after the next one
        Quad DIN;
        DIN.p[0] = DIN.p[1] = zero;
        if (kD && in) DIN = quad_g(dop);
        uint2 LQN = make_uint2(0u, 0u);
        if (kLo && STAGE == 3 && in) LQN = __ldcg(reinterpret_cast<const uint2*>(lop));
        const int gy = jj[0], gx = Qy + kDup * ii[0], gz = Qy + kDup * (Qx + zz[0] - zm_lo);
#pragma unroll(kUnroll)
        for (int c = 0; c < zc; ++c) {
            const int cc = zb + (sgc ? zc - 1 - c : c);
            const T* gc = gsm + (size_t)cc * G;
            const T* sc = scs + cc * (S_COUNT * kDup);
            const uint2 LQ = LQN;
            const Quad DI = DIN;
            const Quad own = quad(Fs + (size_t)(cc + 3) * KC + tbase);  // d of the cell
            Quad nx = NV;                                               // the row two ahead
            if (c + 1 < zc) {
                NV = quad(rp + (c + 6) * rstep);
#pragma unroll
                for (int p = 0; p < 2; ++p) NV.p[p] = kD ? add2(NV.p[p], DN.p[p]) : NV.p[p];
                if (kLo && STAGE == 3 && in) LQN = __ldcg(reinterpret_cast<const uint2*>(lop + ostep));
                if (kD) {
                    if (in) DIN = quad_g(dop + ostep);
                    sn += sdir;
                    dnp += ostep;
                    DN.p[0] = DN.p[1] = zero;
                    if (in && (unsigned)sn < (unsigned)Nz) DN = quad_g(dnp);
                }
            }
            P X = PX, Z = PZ, XZ2, XQ, GXZ, S1, Y[2], out[2];
            P UY, QY, CS, I5T, NIT;
            if (STAGE > 0) {
                X = sub2(PX, dup(sc + kDup * S_UX));
                Z = sub2(PZ, dup(sc + kDup * S_UZ));
                UY = dup(sc + kDup * S_UY);
                QY = dup(sc + kDup * S_QY);
                CS = dup(sc + kDup * S_CS);
                I5T = dup(sc + kDup * S_I5T);
                NIT = dup(sc + kDup * S_NITAU);
                XQ = fma2(Z, dup(sc + kDup * S_QZ), mul2(X, dup(sc + kDup * S_QX)));
                S1 = mul2(NAPZ, dup(sc + kDup * S_IDZ));
                const P DX = dup(gc + gx), DZ = dup(gc + gz);
                GXZ = fma2(DX, DZ, add2(DX, DZ));
            }
            XZ2 = fma2(Z, Z, mul2(X, X));
            const Quad DY = STAGE > 0 ? quad(gc + gy) : own;
            Quad st;
            P A0, A1, A2, A3;  // sums of w f xi_y^a over the thread's velocities, two lanes
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const P h = own.p[p];
                out[p] = h;
                Y[p] = PY[p];
                if (STAGE > 0) {
                    // the target's deviation from 1, (1 + dx)(1 + dz)(1 + dy)(1 + S) - 1
                    Y[p] = sub2(PY[p], UY);
                    const P p2 = fma2(Y[p], Y[p], XZ2), xq = fma2(Y[p], QY, XQ);
                    const P S = mul2(mul2(CS, fma2(p2, I5T, splat(T(-1)))), xq);
                    const P b = fma2(GXZ, DY.p[p], add2(GXZ, DY.p[p]));
                    const P tgt = fma2(b, S, add2(b, S));
                    // the departure from the target from its parts (see the scalar march)
                    const P dinc = DI.p[p];
                    P dep = sub2(h, tgt), lo = zero;
                    if (STAGE >= 2) dep = add2(dep, dinc);
                    if constexpr (kLo && STAGE == 3) {
                        const unsigned q = p ? LQ.y : LQ.x;
                        lo = make_float2(lo_decode(q, h.x), lo_decode(q >> 16, h.y));
                        dep = add2(dep, lo);
                    }
                    // Eq. (flux) and the relaxation, both scaled by the stage's share of dt
                    const P d12 = w[p].d12;  // this cell minus the upwind one
                    const P cp = carried_corr(w[p], nx.p[p]);
                    const P div = fma2(splat(T(0.5)), sub2(cp, CM[p]), d12);
                    CM[p] = cp;
                    P inc = fma2(dep, NIT, mul2(S1, div));
                    if (STAGE == 2) inc = fma2(splat(T(0.25)), dinc, inc);
                    if (STAGE == 3) inc = fma2(splat(T(2.0 / 3.0)), dinc, inc);
                    if (STAGE < 3) {
                        st.p[p] = inc;
                        out[p] = add2(h, inc);
                    } else if constexpr (kLo) {
                        const P t = add2(lo, inc), h2 = add2(h, t), lo2 = sub2(t, sub2(h2, h));
                        if (in) __stcg(reinterpret_cast<unsigned*>(lop) + p, lo_encode2(lo2, h2));
                        st.p[p] = out[p] = h2;
                    } else {
                        st.p[p] = out[p] = add2(h, inc);
                    }
                }
                // w f times the powers of xi_y; columns past the chunk hold no data
                const P o = in ? mul2(out[p], WV[p]) : zero;
                const P o1 = mul2(o, Y[p]), o2 = mul2(o1, Y[p]);
                A0 = p ? add2(A0, o) : o;
                A1 = p ? add2(A1, o1) : o1;
                A2 = p ? add2(A2, o2) : o2;
                A3 = p ? fma2(o2, Y[p], A3) : mul2(o2, Y[p]);
            }
            if (STAGE > 0 && in) {
                if constexpr (sizeof(T) == 4) {
                    __stcg(reinterpret_cast<float4*>(outp),
                           make_float4(st.p[0].x, st.p[0].y, st.p[1].x, st.p[1].y));
                } else {
                    __stcg(reinterpret_cast<double2*>(outp), st.p[0]);
                    __stcg(reinterpret_cast<double2*>(outp) + 1, st.p[1]);
                }
            }
            // the 13 moments about the record's u: 1, xi_a, xi_a xi_b, |xi|^2 xi_a
            const A x = X.x, z = Z.x, xz2 = XZ2.x;
            const A a0 = A0.x + A0.y, a1 = A1.x + A1.y, a2 = A2.x + A2.y, a3 = A3.x + A3.y;
            const A m1 = a0 * x, m3 = a0 * z, e = xz2 * a0 + a2;  // e: |xi|^2
            A* rd = red + ((size_t)cc * (kThreads / 32 / ZW) + (ZW == 1 ? warp : 0)) * 16;
            if constexpr (sizeof(T) == 4) {
                const float4 q[4] = {make_float4(a0, m1, a1, m3), make_float4(m1 * x, a2, m3 * z, a1 * x),
                                     make_float4(m3 * x, a1 * z, e * x, xz2 * a1 + a3),
                                     make_float4(e * z, 0.f, 0.f, 0.f)};
                const float tot = warp_totals13(q, reinterpret_cast<float4*>(recs) + warp * 128, lane);
                if ((lane & 4) == 0) rd[4 * (lane & 3) + 2 * (lane >> 4) + ((lane >> 3) & 1)] = tot;
            } else {
                A acc[16] = {a0, m1, a1, m3, m1 * x, a2, m3 * z, a1 * x, m3 * x, a1 * z, e * x, xz2 * a1 + a3, e * z,
                             A(0), A(0), A(0)};
                const A tot = reduce_scatter16<A>(acc, lane);
                const int m = (lane >> 4 & 1) * 8 + (lane >> 3 & 1) * 4 + (lane >> 2 & 1) * 2 + (lane >> 1 & 1);
                if ((lane & 1) == 0) rd[m] = tot;
            }
            outp += ostep;
            if (kD) dop += ostep;
            if (kLo && STAGE == 3) lop += ostep;
        }
    } else if constexpr (kPair && !RED) {
        // ---- 5 (FP32, full model). The march of section 5 below with the thread's
        // velocities as adjacent pairs: the same operations, two velocities per packed
        // FP32 instruction; rows, increments and outputs move as 64-bit pairs and the two
        // 16-bit residuals of a pair as one 32-bit word.  Q / 2 is even (the host's
        // condition for this layout), so a chunk start k0 and its length kn are even, a
        // pair lies wholly inside or wholly past the chunk, and every pair address is
        // 8-byte aligned.
        constexpr int NP = V / 2;
        const long rstep2 = sgc ? -(long)(KC / 2) : (long)(KC / 2);  // a row, in pairs
        const float2* rp2 = reinterpret_cast<const float2*>(Fs + (sgc ? (size_t)(zn + 5) * KC : 0)) + tid;
        const int sdir = sgc ? -1 : 1;
        const int zw0 = sgc ? z0 + zn + 2 : z0 - 3;  // the cell of window row 0 at step 0
        const float* Dgf = reinterpret_cast<const float*>(Dg);
        // the increments of the cell of a window row (zero for a ghost row)
        auto inc_row2 = [&](int s, float2(&out)[NP]) {
            const bool in = kD && (unsigned)s < (unsigned)Nz;
            const float2* q = reinterpret_cast<const float2*>(Dgf + (long)s * Q + k0) + tid;
#pragma unroll
            for (int p = 0; p < NP; ++p) out[p] = in && ok[2 * p] ? __ldca(q + p * kThreads) : make_float2(0.f, 0.f);
        };
        float2 PX[NP], PY[NP], PZ[NP], NAPZ[NP], WV[NP];  // per pair: p, -|p_z|, weights
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            PX[p] = make_float2(px[2 * p], px[2 * p + 1]);
            PY[p] = make_float2(py[2 * p], py[2 * p + 1]);
            PZ[p] = make_float2(pz[2 * p], pz[2 * p + 1]);
            NAPZ[p] = make_float2(-apz[2 * p], -apz[2 * p + 1]);
            WV[p] = make_float2(wv[2 * p], wv[2 * p + 1]);
        }
        float2 W[NP][6], CM[NP], DN[NP], DIN[NP];
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            inc_row2(zw0 + d * sdir, DN);
#pragma unroll
            for (int p = 0; p < NP; ++p) W[p][d] = add2(rp2[d * rstep2 + p * kThreads], DN[p]);
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) CM[p] = weno5_corr2(W[p][0], W[p][1], W[p][2], W[p][3], W[p][4]);
        int sn = zw0 + 6 * sdir;
        inc_row2(sn, DN);
        // the increments' row of cell sn as a running offset in pairs (one add per march
        // step instead of the row's product; a pointer is formed only inside the channel)
        const float2* dbase = reinterpret_cast<const float2*>(Dgf + k0) + tid;
        long doff = (long)sn * (Q / 2);
        const long dstep = sdir * (long)(Q / 2);
        const float2 DT = splat(float(I.dt));
        const long ostep2 = sgc ? -(long)(Q / 2) : (long)(Q / 2);
        const size_t orow0 = (size_t)(sgc ? z0 + zn - 1 : z0) * Q + k0 + tbase;
        float2* outp = reinterpret_cast<float2*>(reinterpret_cast<float*>(Fout) + orow0);
        const float2* dop = kD ? reinterpret_cast<const float2*>(Dgf + orow0) : nullptr;
        unsigned* lop = kLo && STAGE == 3 ? reinterpret_cast<unsigned*>(I.L0 + orow0) : nullptr;
        unsigned LQN[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            LQN[p] = kLo && STAGE == 3 && ok[2 * p] ? __ldcg(lop + p * kThreads) : 0u;
            DIN[p] = kD && ok[2 * p] ? __ldca(dop + p * kThreads) : make_float2(0.f, 0.f);
        }
        // stage 1 unrolled by two steps (the window's shift halves; 80 vs 86 us on 64 x C2);
        // stages 2 and 3, with their increment and residual streams, lose by unrolling
#pragma unroll(STAGE == 1 ? 2 : 1)
        for (int c = 0; c < zn; ++c) {
            unsigned LQC[NP];
            float2 DC[NP], DIC[NP];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                LQC[p] = LQN[p];
                if (kLo && STAGE == 3 && ok[2 * p] && c + 1 < zn) LQN[p] = __ldcg(lop + ostep2 + p * kThreads);
                DIC[p] = DIN[p];
                if (kD && ok[2 * p] && c + 1 < zn) DIN[p] = __ldca(dop + ostep2 + p * kThreads);
                DC[p] = DN[p];
            }
            if (kD && c + 1 < zn) {
                sn += sdir;
                doff += dstep;
                const bool in = (unsigned)sn < (unsigned)Nz;
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    DN[p] = in && ok[2 * p] ? __ldca(dbase + doff + p * kThreads) : make_float2(0.f, 0.f);
            }
            const int cc = sgc ? zn - 1 - c : c;
            const float* sc = reinterpret_cast<const float*>(recs) + (size_t)cc * rstride;
            const float* gc = reinterpret_cast<const float*>(gsm) + cc * G;
            const float2* rn2 = rp2 + (c + 6) * rstep2;
            const float2* own2 = reinterpret_cast<const float2*>(Fs + (size_t)(cc + 3) * KC) + tid;
            float2 UX, UY, UZ, QX, QY, QZ, NITAU, CS, I5T, IDZ;
            if (STAGE > 0) {
                UX = splat(sc[R_UX]); UY = splat(sc[R_UY]); UZ = splat(sc[R_UZ]);
                QX = splat(sc[R_QX]); QY = splat(sc[R_QY]); QZ = splat(sc[R_QZ]);
                NITAU = splat(-sc[R_ITAU]); CS = splat(sc[R_CS]); I5T = splat(sc[R_I5T]);
                IDZ = splat(float(idzs[cc]));
            }
            float2 S2[kNMom];  // the thread's moment sums, one lane per velocity of a pair
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const int v0 = 2 * p, v1 = v0 + 1;
                const float2 f = W[p][3];
                float2 out = f, X = PX[p], Y = PY[p], Z = PZ[p], P2;
                if (STAGE > 0) {
                    const float2 cp = weno5_corr2(W[p][1], W[p][2], W[p][3], W[p][4], W[p][5]);
                    // the Shakhov target's deviation from 1, (1 + dx)(1 + dy)(1 + dz)(1 + S) - 1
                    X = sub2(PX[p], UX);
                    Y = sub2(PY[p], UY);
                    Z = sub2(PZ[p], UZ);
                    P2 = fma2(Z, Z, fma2(Y, Y, mul2(X, X)));
                    const float2 xq = fma2(Z, QZ, fma2(Y, QY, mul2(X, QX)));
                    const float2 S = mul2(mul2(CS, fma2(P2, I5T, splat(-1.f))), xq);
                    const float2 DXf = make_float2(gc[ii[v0]], gc[ii[v1]]);
                    const float2 DYf = make_float2(gc[Qx + jj[v0]], gc[Qx + jj[v1]]);
                    const float2 DZf = make_float2(gc[Qx + Qy + zz[v0] - zm_lo], gc[Qx + Qy + zz[v1] - zm_lo]);
                    const float2 a = fma2(DXf, DYf, add2(DXf, DYf));
                    const float2 b = fma2(a, DZf, add2(a, DZf));
                    const float2 tgt = fma2(b, S, add2(b, S));
                    // the departure from the target from its parts (see section 5)
                    float2 h = f, dinc = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
                    if (STAGE >= 2) {
                        h = own2[p * kThreads];
                        dinc = DIC[p];
                    }
                    if constexpr (kLo && STAGE == 3)
                        lo = make_float2(lo_decode(LQC[p], h.x), lo_decode(LQC[p] >> 16, h.y));
                    const float2 dep = STAGE >= 2 ? add2(add2(sub2(h, tgt), dinc), lo) : sub2(f, tgt);
                    // Eq. (flux) and the relaxation: -|p_z| div / dz - dep / tau
                    const float2 div = add2(sub2(W[p][3], W[p][2]), sub2(cp, CM[p]));
                    const float2 Lv = fma2(dep, NITAU, mul2(mul2(NAPZ[p], div), IDZ));
                    float2 st;
                    if (STAGE == 1) {
                        st = mul2(DT, Lv);
                        out = add2(f, st);
                    } else if (STAGE == 2) {
                        st = mul2(splat(0.25f), fma2(DT, Lv, dinc));
                        out = add2(h, st);
                    } else {
                        const float2 inc = mul2(splat(float(2.0 / 3.0)), fma2(DT, Lv, dinc));
                        if constexpr (kLo) {
                            const float2 t = add2(lo, inc);
                            const float2 h2 = add2(h, t);
                            const float2 lo2 = sub2(t, sub2(h2, h));
                            if (ok[v0]) __stcg(lop + p * kThreads, lo_encode2(lo2, h2));
                            st = h2;
                        } else {
                            st = add2(h, inc);
                        }
                        out = st;
                    }
                    if (ok[v0]) __stcg(outp + p * kThreads, st);
                    CM[p] = cp;
                } else {
                    P2 = fma2(Z, Z, fma2(Y, Y, mul2(X, X)));
                }
#pragma unroll
                for (int d = 0; d < 5; ++d) W[p][d] = W[p][d + 1];
                W[p][5] = kD ? add2(rn2[p * kThreads], DC[p]) : rn2[p * kThreads];
                // the moments about the record's u (section 5): w f times 1, xi_a,
                // xi_a xi_b, |xi|^2 xi_a; pairs past the chunk contribute zero
                const float2 o = ok[v0] ? mul2(out, WV[p]) : make_float2(0.f, 0.f);
                const float2 oX = mul2(o, X), oY = mul2(o, Y), oZ = mul2(o, Z), oP = mul2(o, P2);
                if (p == 0) {
                    S2[0] = o; S2[1] = oX; S2[2] = oY; S2[3] = oZ;
                    S2[4] = mul2(oX, X); S2[5] = mul2(oY, Y); S2[6] = mul2(oZ, Z);
                    S2[7] = mul2(oX, Y); S2[8] = mul2(oX, Z); S2[9] = mul2(oY, Z);
                    S2[10] = mul2(oP, X); S2[11] = mul2(oP, Y); S2[12] = mul2(oP, Z);
                } else {
                    S2[0] = add2(S2[0], o); S2[1] = add2(S2[1], oX); S2[2] = add2(S2[2], oY);
                    S2[3] = add2(S2[3], oZ);
                    S2[4] = fma2(oX, X, S2[4]); S2[5] = fma2(oY, Y, S2[5]); S2[6] = fma2(oZ, Z, S2[6]);
                    S2[7] = fma2(oX, Y, S2[7]); S2[8] = fma2(oX, Z, S2[8]); S2[9] = fma2(oY, Z, S2[9]);
                    S2[10] = fma2(oP, X, S2[10]); S2[11] = fma2(oP, Y, S2[11]); S2[12] = fma2(oP, Z, S2[12]);
                }
            }
            float acc[16];
#pragma unroll
            for (int a = 0; a < kNMom; ++a) acc[a] = S2[a].x + S2[a].y;
#pragma unroll
            for (int a = kNMom; a < 16; ++a) acc[a] = 0.f;
            const float tot = reduce_scatter16<float>(acc, lane);
            const int m = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
            if ((lane & 1) == 0) red[((size_t)cc * (kThreads / 32) + warp) * 16 + m] = tot;
            outp += ostep2;
            if (kD) dop += ostep2;
            if (kLo && STAGE == 3) lop += ostep2;
        }
    } else {
    // ---- 5. march through the z-range in the upwind direction of the chunk: up
    // (p_z > 0) from z0, down (p_z < 0) from z0+zn-1.  At march step c the register
    // window holds the cells s-3 .. s+2 seen from upwind (s+3 .. s-2 going down), so
    // both directions use one stencil: the flux through the interface ahead is
    // |p_z| (w3 + its correction), the one behind was formed at the previous step, and the
    // divergence of Eq. (flux) is (ahead - behind) / dz for the signed p_z either way.
    const long rstep = sgc ? -(long)KC : (long)KC;
    const T* rp = Fs + (size_t)(sgc ? zb + zc + 5 : zb) * KC;  // window row d at step c: rp + (c + d) rstep
    // stages 2, 3: the increment of the cell of each window row, read from global memory
    // (this launch does not write it).  Window row cd at step c
    // holds cell zw0 + (c + cd) sdir; a ghost row (a cell outside 0 .. Nz-1) takes zero,
    // its shared-memory value being the whole stage input.  Thread-based pointers: the
    // thread's velocity v sits at + voff(v).
    const int sdir = sgc ? -1 : 1;
    const int zw0 = sgc ? z0 + zb + zc + 2 : z0 + zb - 3;
    const T* dq = Dg + k0 + tbase;
    auto inc_row = [&](int s, T(&out)[V]) {
        const bool in = kD && (unsigned)s < (unsigned)Nz;
        const T* p = dq + (long)s * Q;
#pragma unroll
        for (int v = 0; v < V; ++v) out[v] = in && ok[v] ? __ldca(p + voff(v)) : T(0);
    };
    // WENO differences carried from interface to interface (carried_corr), two velocities per
    // packed instruction where the storage is FP32 and V even.  Window rows 0 .. 4 (the cell's
    // three upwind neighbours, the cell, the next one) start them and give the correction
    // behind the first cell (its flux is |p_z| (w2 + cm)); nv is the row two ahead.
    constexpr bool kPack = sizeof(T) == 4 && V % 2 == 0;
    constexpr int NP = kPack ? V / 2 : V;
    typedef typename PackedAs<T, kPack>::type P;
    auto pack = [](const T(&a)[V], int p) -> P {
        if constexpr (kPack) return make_float2(a[2 * p], a[2 * p + 1]);
        else return a[p];
    };
    auto lane_of = [](const P(&a)[NP], int v) -> T {
        if constexpr (kPack) return v & 1 ? a[v >> 1].y : a[v >> 1].x;
        else return a[v];
    };
    Carried<P> w[NP];
    P cm[NP], nv[NP];
    T dn[V];
    {
        P r[6][NP];
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            inc_row(zw0 + d * sdir, dn);
            T x[V];
#pragma unroll
            for (int v = 0; v < V; ++v) x[v] = kD ? rp[d * rstep + kl[v]] + dn[v] : rp[d * rstep + kl[v]];
#pragma unroll
            for (int p = 0; p < NP; ++p) r[d][p] = pack(x, p);
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            w[p] = carried_start(r[0][p], r[1][p], r[2][p], r[3][p]);
            cm[p] = carried_corr(w[p], r[4][p]);
            nv[p] = r[5][p];
        }
    }
    int sn = zw0 + 6 * sdir;  // the cell of the row the next step loads
    inc_row(sn, dn);
    const T dt = T(I.dt);
    const long ostep = sgc ? -(long)Q : (long)Q;
    const size_t orow0 = (size_t)(sgc ? z0 + zb + zc - 1 : z0 + zb) * Q + k0 + tbase;  // the first cell, thread's column
    T* outp = Fout + orow0;
    const T* dop = kD ? Dg + orow0 : nullptr;  // the increment of the cell
    unsigned short* lop = kLo && STAGE == 3 ? I.L0 + orow0 : nullptr;
    // stage 3 (FP32): the residuals of the next cell are loaded one march step ahead, so
    // that their global-memory latency overlaps a step's arithmetic
    // the increments of the next cell (stages 2, 3) likewise
    unsigned short lqn[V];
    T din[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        lqn[v] = kLo && STAGE == 3 && ok[v] && zc > 0 ? __ldcg(lop + voff(v)) : 0;
        din[v] = kD && ok[v] && zc > 0 ? __ldca(dop + voff(v)) : T(0);  // zc = 0: a warp without cells
    }
#pragma unroll 1  // unrolling the z-march only adds instruction-cache misses
    for (int c = 0; c < zc; ++c) {
        unsigned short lqc[V];
        T dc[V], dic[V];  // increments of the window row this step loads and of the cell
#pragma unroll
        for (int v = 0; v < V; ++v) {
            lqc[v] = lqn[v];
            if (kLo && STAGE == 3 && ok[v] && c + 1 < zc) lqn[v] = __ldcg(lop + ostep + voff(v));
            dic[v] = din[v];
            if (kD && ok[v] && c + 1 < zc) din[v] = __ldca(dop + ostep + voff(v));
            dc[v] = dn[v];
        }
        if (kD && c + 1 < zc) {
            sn += sdir;
            inc_row(sn, dn);
        }
        const int cc = zb + (sgc ? zc - 1 - c : c);  // the cell within the tile
        const T* sc = recs + (size_t)cc * rstride;
        const T* gc = gsm + cc * G;
        const T* rn = rp + (c + 6) * rstep;
        const T* own = Fs + (size_t)(cc + 3) * KC;  // the cell's row of d
        T ux = 0, uy = 0, uz = 0, i5T = 0, qx = 0, qy = 0, qz = 0, itau = 0, cS = 0, idz = 0;
        if (STAGE > 0) {
            ux = sc[R_UX]; uy = sc[R_UY]; uz = sc[R_UZ];
            qx = sc[R_QX]; qy = sc[R_QY]; qz = sc[R_QZ];
            itau = sc[R_ITAU]; cS = sc[R_CS]; i5T = sc[R_I5T]; idz = idzs[cc];
        }
        // the corrections of the interfaces ahead, the cell minus the upwind one, and the next row
        P cp2[NP], d12[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            d12[p] = w[p].d12;
            cp2[p] = STAGE > 0 ? carried_corr(w[p], nv[p]) : cm[p];
        }
        {
            T x[V];
#pragma unroll
            for (int v = 0; v < V; ++v) x[v] = kD ? rn[kl[v]] + dc[v] : rn[kl[v]];
#pragma unroll
            for (int p = 0; p < NP; ++p) nv[p] = pack(x, p);
        }
        // ---- per velocity: the update, its store, and the moment variables
        A ov[V], mx[V], my[V], mz[V], m2[V];  // value; the monomials' factors (p or p - u_r); |.|^2
#pragma unroll
        for (int v = 0; v < V; ++v) {
            const unsigned short lq = lqc[v];
            const T h = own[kl[v]];
            T out = h;  // the value whose moments are taken
            T ex = 0, ey = 0, ez = 0, xi2 = 0;  // xi = p - u of the cell's record
            if (STAGE > 0) {
                const T cp = lane_of(cp2, v);
                // Shakhov target n Gx Gy Gz (1 + S), S = cS (xi^2/(5T) - 1) xi.q; in the
                // phi / chi model (Eq. sred_def) S = cS ((xi_x^2 + xi_z^2)/(5T) - 4/5 or 2/5) xi.q
                // with u_y = q_y = 0, and Gy = 1 (phi) or T (chi) from the record
                T S;
                ex = px[v] - ux;
                ez = pz[v] - uz;
                if (RED) {
                    xi2 = ex * ex + ez * ez;
                    S = cS * (xi2 * i5T + py[v]) * (ex * qx + ez * qz);
                } else {
                    ey = py[v] - uy;
                    xi2 = ex * ex + ey * ey + ez * ez;
                    const T xq = ex * qx + ey * qy + ez * qz;
                    S = cS * (xi2 * i5T - T(1)) * xq;
                }
                // the target's deviation from 1: (1 + dx)(1 + dy)(1 + dz)(1 + S) - 1
                const T dx = gc[ii[v]], dy = gc[Qx + jj[v]], dz = gc[Qx + Qy + zz[v] - zm_lo];
                const T a = dx + dy + dx * dy, b = a + dz + a * dz, tgt = b + S + b * S;
                // the departure from the target, f - tgt: from the cell's d, increment and
                // (stage 3, FP32) residual separately, (d - tgt) + increment + residual,
                // so that its rounding is relative to the departure, which in the
                // collision-dominated regime is much smaller than f itself
                const T dinc = STAGE >= 2 ? dic[v] : T(0);
                T lo = T(0);
                if constexpr (kLo && STAGE == 3) lo = lo_decode(lq, h);
                const T dep = STAGE >= 2 ? ((h - tgt) + dinc) + lo : h - tgt;
                // Eq. (flux): (|p_z| (w3 + cp) - |p_z| (w2 + cm)) / dz, formed from the
                // difference of the two upwind cells and of the two corrections (cp and cm are twice those), so that
                // its rounding is relative to the divergence rather than to d.  The
                // advection and relaxation increments nearly cancel near a steady state:
                // combine them first.
                const T Lv = -apz[v] * (lane_of(d12, v) + T(0.5) * (cp - lane_of(cm, v))) * idz - dep * itau;
                T st;  // the value stored
                if (STAGE == 1) {
                    st = dt * Lv;
                    out = h + st;
                } else if (STAGE == 2) {
                    st = T(0.25) * (dinc + dt * Lv);
                    out = h + st;
                } else {
                    // Shu-Osher combine in increment form: F_l + 2/3 (d2 + dt L), added to the
                    // state with its rounding residual carried (FP32)
                    const T inc = T(2.0 / 3.0) * (dinc + dt * Lv);
                    if constexpr (kLo) {
                        const T t = lo + inc;
                        const T h2 = h + t;
                        const T lo2 = t - (h2 - h);
                        if (ok[v]) __stcg(lop + voff(v), lo_encode(lo2, h2));
                        st = h2;
                    } else {
                        st = h + inc;
                    }
                    out = st;
                }
                if (ok[v]) __stcg(outp + voff(v), st);
            }
            // the moments: of psi(p - u_r) about the velocity u_r of the cell's record
            // (stage 0, which has no record: of psi(p)), so that the third moments are
            // close to the heat flux itself instead of its sum with terms of size u |p|^2
            // that cancel it (160-fold in config C1), and the Shakhov factor's xi and
            // |xi|^2 serve as the monomials' factors; the finalisation adds the rest
            // state's moments about u_r.  Columns past the chunk hold no data (their
            // shared memory is never written) and contribute zero.
            ov[v] = ok[v] ? A(out) * wv[v] : A(0);
            if (STAGE > 0) {
                mx[v] = A(ex); my[v] = A(ey); mz[v] = A(ez); m2[v] = A(xi2);
            } else {
                mx[v] = A(px[v]); my[v] = yv[v]; mz[v] = A(pz[v]); m2[v] = p2v[v];
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) cm[p] = cp2[p];
        // ---- the 13 weighted monomials summed over the thread's velocities: w f times
        // 1, p_a, p_a p_b, |p|^2 p_a (RED: chi carries the p_y^2 parts: sum chi, sum chi p_x,
        // sum chi p_z)
        A acc[16];
#pragma unroll
        for (int a = kNMom; a < 16; ++a) acc[a] = A(0);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            A t[kNMom];
            const A o = ov[v], X = mx[v], Y = my[v], Z = mz[v], P = m2[v];
            if (RED) {  // phi: p_y = 0; chi: the p_y^2 parts
                const A oc = chi[v] ? o : A(0), op = o - oc;
                const A oX = op * X, oZ = op * Z, r3 = op * P + oc;
                t[0] = op; t[1] = oX; t[2] = A(0); t[3] = oZ;
                t[4] = oX * X; t[5] = oc; t[6] = oZ * Z; t[7] = A(0); t[8] = oX * Z;
                t[9] = A(0); t[10] = r3 * X; t[11] = A(0); t[12] = r3 * Z;
            } else {
                const A oX = o * X, oY = o * Y, oZ = o * Z, oP = o * P;
                t[0] = o; t[1] = oX; t[2] = oY; t[3] = oZ;
                t[4] = oX * X; t[5] = oY * Y; t[6] = oZ * Z;
                t[7] = oX * Y; t[8] = oX * Z; t[9] = oY * Z;
                t[10] = oP * X; t[11] = oP * Y; t[12] = oP * Z;
            }
#pragma unroll
            for (int a = 0; a < kNMom; ++a) acc[a] = v == 0 ? t[a] : acc[a] + t[a];
        }
        const A tot = reduce_scatter16<A>(acc, lane);
        const int m = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
        if ((lane & 1) == 0) red[((size_t)cc * (kThreads / 32 / ZW) + (ZW == 1 ? warp : 0)) * 16 + m] = tot;
        outp += ostep;
        if (kD) dop += ostep;
        if (kLo && STAGE == 3) lop += ostep;
    }
    }  // the scalar march
    launch_dependents();
    __syncthreads();
    // the chunk's partial of each cell: the warps' sums added and stored in the
    // accumulation type (FP32 storage: no FP64 instruction here; the finalisation sums
    // the chunks exactly enough in double-float)
    for (int e = tid; e < zn * kNMom; e += kThreads) {
        const int c = e / kNMom, a = e - c * kNMom;
        constexpr int nw = kThreads / 32 / ZW;  // warps that share a cell
        A s = red[(size_t)c * nw * 16 + a];
#pragma unroll
        for (int q = 1; q < nw; ++q) s += red[((size_t)c * nw + q) * 16 + a];
        static_cast<A*>(I.partial)[((size_t)tile.chunk * kNMom + a) * Nz + z0 + c] = s;
    }

    // ---- 6. outgoing WENO flux of the stage output through the wall interfaces (for
    // n_w), as a sum over the deviations (the rest state's flux is added by the
    // finalisation).  The outputs are read back (ZW = 4: other warps wrote some): the new d after
    // stage 3, d + the increment after stages 1 and 2 (STAGE 0: its input rows).
    auto outval = [&](int v, int cell) -> T {
        const T* row = Fs + (size_t)(cell + rbase) * KC;
        if (STAGE == 0) return row[kl[v]];
        const T o = __ldcg(Fout + (size_t)cell * Q + k0 + kl[v]);
        return STAGE == 3 ? o : row[kl[v]] + o;
    };
    // The sums: exact products (double-float with FP32 storage: no FP64 instruction, which here
    // held the wall tiles' schedulers for some 2000 cycles; 64 x C2 339 -> 311 us per step), a
    // warp's and the CTA's sum in the same arithmetic, one FP64 value per chunk.
    R fl[2] = {Real<T>::of(T(0)), Real<T>::of(T(0))};  // bottom, top
    if (z0 == 0 && sgc && !I.half && zw == 0) {  // p_z < 0 leaves through s = -1/2; no wall below a half channel
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (ok[v]) {
                const T f1 = outval(v, 0), f2 = outval(v, 1), f3 = outval(v, 2);
                const T g0 = ext_bot[0][0] * f1 + ext_bot[0][1] * f2 + ext_bot[0][2] * f3;
                const T g1 = ext_bot[1][0] * g0 + ext_bot[1][1] * f1 + ext_bot[1][2] * f2;
                fl[0] = r_add(fl[0], r_mul(Real<T>::of(T(wm[v])), Real<T>::of(pz[v] * weno5<T>(f3, f2, f1, g0, g1))));
            }
    }
    if (z0 + zn == Nz && !sgc && zw == 0) {  // top: p_z > 0 leaves through s = Nz - 1/2
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (ok[v]) {
                const T f1 = outval(v, Nz - 1), f2 = outval(v, Nz - 2), f3 = outval(v, Nz - 3);
                const T g0 = ext_top[0][0] * f1 + ext_top[0][1] * f2 + ext_top[0][2] * f3;
                const T g1 = ext_top[1][0] * g0 + ext_top[1][1] * f1 + ext_top[1][2] * f2;
                fl[1] = r_add(fl[1], r_mul(Real<T>::of(T(wm[v])), Real<T>::of(pz[v] * weno5<T>(f3, f2, f1, g0, g1))));
            }
    }
    if (z0 == 0 || z0 + zn == Nz) {
        R* fr = reinterpret_cast<R*>(wall_red);
        const int side = z0 == 0 && (sgc || z0 + zn != Nz) ? 0 : 1;  // the one this chunk can leave through
        const R s = warp_sum(side ? fl[1] : fl[0]);
        if (lane == 0) fr[warp] = s;
        __syncthreads();
        if (tid == 0) {
            const double f = r_double(r_add(r_add(fr[0], fr[1]), r_add(fr[2], fr[3])));
            if (z0 == 0) I.flux_part[tile.chunk * 2 + 0] = side == 0 ? f : 0.0;
            if (z0 + zn == Nz) I.flux_part[tile.chunk * 2 + 1] = side == 1 ? f : 0.0;
        }
    }

    // ---- 7. (fuse != 0) finalisation without extra launches (threadfence tickets): the CTA
    // that finishes last among the chunks of this z-tile finalises the tile's
    // cells; the one that finalises the instance's last z-tile does the walls
    // and the residual.  Counters are reset by their last user.
    if (!fuse) return;  // finalize_cells follows as a separate launch
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(I.zcount + tile.zt, 1) == I.nchunks - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    finalize_tile<T>(I, z0, zn, STAGE, *reinterpret_cast<FinShared<T, 4>*>(smem_raw));  // the rows are done with
    if (tid == 0) I.zcount[tile.zt] = 0;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(I.icount, 1) == I.nzt - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (tid == 0) *I.icount = 0;
    finalize_instance(I, STAGE, wall_red);
}

// ---- host-side launch of one stage-kernel instantiation ----------------------
template <typename T, int V, int STAGE, bool RED, bool GRP, int ZW>
static cudaError_t launch_stage_t(const InstDev* d_inst, const Tile* d_tiles, int ntiles, size_t smem,
                                  int fuse, bool early, cudaStream_t st)
{
    auto kfn = stage_kernel<T, V, STAGE, RED, GRP, ZW>;
    if (smem > 40 * 1024) {  // with the static arrays above the default limit of 48 KB
        cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ntiles);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;  // stage_starts_early
    return cudaLaunchKernelEx(&cfg, kfn, d_inst, d_tiles, fuse);
}

template <typename T, int V, bool RED, bool GRP = false, int ZW = 1>
static cudaError_t launch_stage_r(int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                  bool early, cudaStream_t st)
{
    switch (stage) {
        case 0: return launch_stage_t<T, V, 0, RED, GRP, ZW>(d, t, n, smem, fuse, early, st);
        case 1: return launch_stage_t<T, V, 1, RED, GRP, ZW>(d, t, n, smem, fuse, early, st);
        case 2: return launch_stage_t<T, V, 2, RED, GRP, ZW>(d, t, n, smem, fuse, early, st);
        default: return launch_stage_t<T, V, 3, RED, GRP, ZW>(d, t, n, smem, fuse, early, st);
    }
}

template <typename T, bool RED>
static cudaError_t launch_stage_m(int V /* a layout: stage_layout in api.cu */, int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                  bool early, cudaStream_t st)
{
    if constexpr (!RED) {
        if (V == (4 | kGrouped)) return launch_stage_r<T, 4, false, true>(stage, d, t, n, smem, fuse, early, st);
        if constexpr (sizeof(T) == 8)
            if (V == (4 | kGrouped | kZSplit))
                return launch_stage_r<T, 4, false, true, 4>(stage, d, t, n, smem, fuse, early, st);
    }
    if constexpr (sizeof(T) == 8)
        if (V == (1 | kZSplit)) return launch_stage_r<T, 1, RED, false, 4>(stage, d, t, n, smem, fuse, early, st);
    if (V == 1) return launch_stage_r<T, 1, RED>(stage, d, t, n, smem, fuse, early, st);
    if (V == 2) return launch_stage_r<T, 2, RED>(stage, d, t, n, smem, fuse, early, st);
    return launch_stage_r<T, 4, RED>(stage, d, t, n, smem, fuse, early, st);
}

// per (storage type, model) launchers of the stage kernel, one translation unit each
cudaError_t launch_stage_f32_full(int V, int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                  bool early, cudaStream_t st);
cudaError_t launch_stage_f32_red(int V, int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                 bool early, cudaStream_t st);
cudaError_t launch_stage_f64_full(int V, int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                  bool early, cudaStream_t st);
cudaError_t launch_stage_f64_red(int V, int stage, const InstDev* d, const Tile* t, int n, size_t smem, int fuse,
                                 bool early, cudaStream_t st);

}  // namespace lbs
