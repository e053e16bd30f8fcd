// Internal definitions shared by the host set-up and the CUDA kernels.
#pragma once

#if __has_include(<vector_types.h>)
#include <vector_types.h>  // float2 (also for the host-only translation units)
#else
struct float2;  // host code built without the CUDA headers holds only pointers to it
#endif

#include <cmath>
#include <cstddef>
#include <vector>

#if defined(__CUDACC__)
#define LBS_HD __host__ __device__ __forceinline__
#else
#define LBS_HD inline
#endif

namespace lbs {

constexpr int kMaxQ1D = 100;    // nodes per axis (per sign on z): the largest order of the paper
constexpr int kMaxN = 8;        // equilibrium expansion order
constexpr int kNMom = 13;       // raw moments accumulated per cell
constexpr int kRecHead = 12;    // scalars at the head of a cell record
constexpr int kThreads = 128;   // threads of a stage CTA
constexpr int kMaxZT = 64;      // cells of a z-tile
// flags of the launchers' layout next to its velocities per thread (1, 2, 4)
constexpr int kGrouped = 8;     // four adjacent velocities of one x and z node per thread
constexpr int kZSplit = 16;     // the CTA's warps split the tile's cells
inline int layout_columns(int layout) { return (layout & 7) * (layout & kZSplit ? kThreads / 4 : kThreads); }

// whether a tiling's finalisation is folded into the stage kernel (api.cu has the reason)
constexpr int kFoldCells = 8;
inline bool fold_finalisation(int fuse, int ZT) { return fuse == 1 && ZT <= kFoldCells; }

enum { QUAD_FULL = 0, QUAD_HALF = 1 };

// Cell record (storage type T): n, ux, uy, uz, T, qx, qy, qz, 1/tau,
// (1 - Pr)/(n T^2), 1/(5T), R_SCALE - 1 where R_SCALE = n / (discrete weighted sums of
// the per-axis factors); then the per-node factors of the truncated equilibrium as
// deviations from the rest state's factor 1 (the populations are stored as deviations
// from the rest state too): dx[Qx] = Gx / w - 1 (before R_SCALE), dy[Qy], dz[2 Qz]
// (p_z > 0 nodes, then p_z < 0).  The finalisation sums them in FP64 (FP64 storage) or
// double-float (FP32 storage) and rounds once to the storage type.  Records are rec_stride
// values apart.
enum { R_N = 0, R_UX, R_UY, R_UZ, R_T, R_QX, R_QY, R_QZ, R_ITAU, R_CS, R_I5T, R_SCALE1 };
constexpr int R_DX = kRecHead;
// record length of an instance, rounded up to 16 bytes in either storage type
inline int rec_stride_of(int Qx, int Qy, int Qz) { return (kRecHead + Qx + Qy + 2 * Qz + 3) & ~3; }

// Weights of the ghost values' extrapolation: ghost Nz+1 <- (Nz, Nz-1, Nz-2), Nz+2 <-
// (Nz+1, Nz, Nz-1) above, ghost 0 <- (1, 2, 3), -1 <- (0, 1, 2) below
template <typename T>
struct Walls {
    T top[2][3], bot[2][3];
};
// n_w - 1 and n_w of the bottom wall, then of the top one, in FP64 and rounded to FP32
struct WallDensity {
    double d[4];
    float f[4];
};

// Everything a kernel needs to know about one instance (lives in device memory).
struct InstDev {
    int Nz, Qx, Qy, Qz, Q, QxQy;
    int Nx, Ny, Nzq;              // per-axis expansion orders
    int nchunks, bulk;            // bulk: rows are 16-byte aligned, stage them with TMA bulk copies
    int nchh;                     // chunks per half range of p_z (chunk c has p_z < 0 iff c >= nchh)
    int half;                     // 1: half channel, bounce-back ghosts below cell 0 (no bottom wall)
    int reduced;                  // 1: the phi / chi model (Qy = 2: j = 0 phi, j = 1 chi; p_y unused)
    int visc_law;
    double Kn, visc_param, Pr, dt, tol;
    double res_uscale;            // the residual's velocity scale max(|u_w| sqrt(Nz), 1e-30)
    double iKn, isuth;            // 1 / Kn; Sutherland: 1 / (1 + S)
    double iDtop, iDbot;          // 1 / the sum over incoming velocities of w p_z Gw (n_w = 1)
    int rec_stride;               // values per cell record
    double mrest[kNMom];          // raw moments of the rest state f = w (the stored weights and
                                  // nodes): the partials hold sums over the deviations only
    float mrest2[kNMom][2];       // the same as FP32 (hi, lo) pairs
    double frest_bot, frest_top;  // outgoing wall flux of the rest state (sum w p_z over the
                                  // velocities leaving through each wall)
    unsigned wait_limit;          // spins of the bounded wait for the bulk copies
    Walls<double> walls;
    Walls<float> walls2;          // the same rounded to FP32
    unsigned mQy, mQxQy;          // ceil(2^32 / d) for div_small, 0 for d = 1
    int prefetch;                 // the batch's buffers exceed the L2: tiles fetch their increments ahead
    // tables
    const double *Hx, *Hy, *Pz;   // FP64, [Q_a][N_a + 1] basis values He_l/l!, pi_l/h_l
    const float2 *Hx2, *Hy2, *Pz2;  // the same as FP32 (hi, lo) pairs, hi + lo = the FP64 value
                                    // to 2^-48 (FP32 storage: the records' node sums)
    double sumw[3];                 // sums of the stored weights of x, y, z (z: over both half ranges)
    float sumw2[3][2];              // the same as FP32 (hi, lo) pairs
    const double* half_poly;        // [kMaxN + 1][kMaxN + 1]: row l the coefficients of the monic pi_l
    // storage-typed tables (float or double)
    const void *px, *py, *xi, *wx, *wy, *wz;
    const void *gwx_top, *gwx_bot, *gwy, *gwz;  // wall equilibria per axis (Q_x, Q_x, Q_y, 2Q_z),
                                                 // deviations from 1 of the normalised factors
    const void *inv_dz;                          // [Nz]
    // state and work.  The state is d = f / w - 1 (deviation of the normalised populations
    // from the rest Maxwellian), [Nz][Q].  F0 and F1 take turns: *cur = 0 means F0 holds d
    // and F1 the stage-1 increment d1 = F1 - F_l; *cur = 1 the reverse.  F2 holds the
    // stage-2 increment d2 = F2 - F_l.  Stage 3 writes the new d over the stage-1
    // increment (no longer needed) and flips *cur, so no stage writes what another CTA
    // of the same launch still reads.  FP32 storage keeps the rounding residual of d in
    // L0 (16-bit fixed point in units of 2^-15 ulp(d), see lo_encode).
    void *F0, *F1, *F2;
    unsigned short *L0;           // [Nz][Q], FP32 storage only
    int *cur;                     // [1]
    long state_at;                // values of the instances before this one (whole-batch states)
    void *rec;                    // [Nz][rec_stride]
    void *partial;                // [nchunks][kNMom][Nz] in the accumulation type (FP32 sums of FP32 storage)
    double *flux_part;            // [nchunks][2]: bottom, top outgoing flux
    WallDensity *nw;              // [1]
    double *prof;                 // [14][Nz]
    double *Wold, *Wnew;          // [3][Nz]: n, u_x, T
    double *res;                  // [1]
    long long *steps;             // [1]
    int *active;                  // [1]
    int *zcount;                  // [nzt] chunks of a z-tile finished this stage (ticket counters)
    int *icount;                  // [1] z-tiles of the instance finalised this stage
    int nzt;                      // z-tiles of the current tiling
    int *status;                  // [1]: bit 0 non-finite / non-positive n, T; bit 1 a bounded
                                  // wait for the bulk copies ran out
};

enum { STATUS_NONFINITE = 1, STATUS_TIMEOUT = 2 };
constexpr unsigned kWaitLimit = 1u << 26;   // default spins of the bounded wait (~seconds)
constexpr unsigned kDrainLimit = 1u << 28;  // spins granted to copies still in flight after a timeout

struct Tile { int inst, z0, zn, chunk, zt; };

// ---- equilibrium coefficients of the walls, at set-up ----

// a_l = int g(p; u, T) He_l(p) dp: a_0 = 1, a_1 = u, a_{l+1} = u a_l + l (T - 1) a_{l-1}
// (from int g p He_l = u a_l + T l a_{l-1} and He_{l+1} = p He_l - l He_{l-1}).
inline void full_coeffs(double u, double T, int N, double* a)
{
    a[0] = 1.0;
    a[1] = u;  // read only when N >= 1
    for (int l = 1; l < N; ++l) a[l + 1] = u * a[l] + l * (T - 1.0) * a[l - 1];
}

// b_l = int_0^inf g(p; u, T) pi_l(p) dp for the monic half-range polynomials,
// by the modified-moment recurrence J_{l+1,k} = J_{l,k+1} - alpha_l J_{l,k} -
// beta_l J_{l-1,k} started from the half-line Gaussian moments
// J_{0,k} = M_k: M_0 = erfc(-u/sqrt(2T))/2, M_1 = u M_0 + T g(0),
// M_{k+1} = u M_k + k T M_{k-1}.
LBS_HD void half_coeffs(double u, double T, int N, const double* alpha, const double* beta,
                        double* b)
{
    double J[kMaxN + 1][kMaxN + 1];  // J[l][k] is needed for k <= N - l only
    const int K = N;
    const double g0 = exp(-u * u / (2.0 * T)) * (1.0 / sqrt(2.0 * M_PI * T));
    J[0][0] = 0.5 * erfc(-u / sqrt(2.0 * T));
    if (K >= 1) J[0][1] = u * J[0][0] + T * g0;
    for (int k = 1; k < K; ++k) J[0][k + 1] = u * J[0][k] + k * T * J[0][k - 1];
    for (int l = 0; l < N; ++l)
        for (int k = 0; k + l + 1 <= K; ++k)
            J[l + 1][k] = J[l][k + 1] - alpha[l] * J[l][k] - (l > 0 ? beta[l] * J[l - 1][k] : 0.0);
    for (int l = 0; l <= N; ++l) b[l] = J[l][0];
}

// erfc(x) for x >= 0.  For x < 1/2 from the Maclaurin series of erf,
//   erf(x) = (2 / sqrt(pi)) sum_n (-1)^n x^(2n+1) / (n! (2n+1))
// (Abramowitz & Stegun 7.1.5), 14 terms in Horner form in x^2: the last omitted
// term is below 3e-18 of erf(1/2), and erfc = 1 - erf lies in [0.47, 1] there, so
// the result is accurate to rounding.  That is a chain of 14 FMAs instead of the
// library's much longer evaluation.  It sits on the critical path of every cell
// record; in Couette flow the wall-normal drift u_z, hence x, is small.  Larger x
// use erfc itself.
struct ErfSeries {
    double c[14];
    constexpr ErfSeries() : c()
    {
        double fact = 1.0;
        for (int n = 0; n < 14; ++n) {
            if (n > 0) fact *= n;
            c[n] = (n % 2 ? -1.0 : 1.0) * 1.1283791670955125739 / (fact * (2 * n + 1));  // 2 / sqrt(pi)
        }
    }
};
LBS_HD double erfc_nonneg(double x)
{
    if (x >= 0.5) return erfc(x);
    constexpr ErfSeries S;
    const double t = x * x;
    double p = S.c[13];
#pragma unroll
    for (int n = 12; n >= 0; --n) p = fma(p, t, S.c[n]);
    return 1.0 - x * p;
}

// Macroscopic state of a cell from its 13 raw moments (FP64): n, u, the central
// second moments P_ab = sum p_a p_b f - n u_a u_b, T = tr P / (3n) and the heat flux
// q_a = 1/2 sum |xi|^2 xi_a f with xi = p - u (Eq. qdef), expanded in raw moments.
struct CellState {
    double n, in, u[3], T, q[3], P[6];  // P: xx, yy, zz, xy, xz, yz
};
LBS_HD void cell_state(const double* mom, CellState& c)
{
    const double n = mom[0], in = 1.0 / n;
    c.n = n;
    c.in = in;
    c.u[0] = mom[1] * in; c.u[1] = mom[2] * in; c.u[2] = mom[3] * in;
    const double* u = c.u;
    c.P[0] = mom[4] - n * u[0] * u[0]; c.P[1] = mom[5] - n * u[1] * u[1];
    c.P[2] = mom[6] - n * u[2] * u[2]; c.P[3] = mom[7] - n * u[0] * u[1];
    c.P[4] = mom[8] - n * u[0] * u[2]; c.P[5] = mom[9] - n * u[1] * u[2];
    c.T = (c.P[0] + c.P[1] + c.P[2]) * (1.0 / 3.0) * in;
    const double M2[3][3] = {{mom[4], mom[7], mom[8]}, {mom[7], mom[5], mom[9]}, {mom[8], mom[9], mom[6]}};
    const double tr = mom[4] + mom[5] + mom[6];
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const double um = u[0] * mom[1] + u[1] * mom[2] + u[2] * mom[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double uM2 = u[0] * M2[0][a] + u[1] * M2[1][a] + u[2] * M2[2][a];
        c.q[a] = 0.5 * (mom[10 + a] - u[a] * tr - 2.0 * uM2 + 2.0 * u[a] * um + uu * mom[1 + a] - uu * u[a] * n);
    }
}

// 1 / tau from 1 / n, 1 / T, 1 / Kn and (Sutherland) 1 / (1 + S), without a
// division: power law n T^(1 - omega) / Kn, Sutherland n (T + S) / (Kn sqrt(T) (1 + S))
LBS_HD double inv_relax_time(int law, double iKn, double param, double isuth, double n, double T, double iT)
{
    if (law == 0) {
        if (param == 1.0) return n * iKn;
        if (param == 0.5) return n * iKn * sqrt(T);
        return n * iKn * pow(T, 1.0 - param);
    }
    return n * (T + param) * iKn * isuth * sqrt(iT);
}

// relaxation time: power law tau = Kn T^(omega-1)/n, Sutherland tau = Kn sqrt(T)(1+S)/(n(T+S))
LBS_HD double relax_time(int law, double Kn, double param, double n, double T)
{
    if (law == 0) {
        // the hard-sphere and Maxwell-molecule exponents without a general pow
        if (param == 1.0) return Kn / n;
        if (param == 0.5) return Kn / (n * sqrt(T));
        return Kn * pow(T, param - 1.0) / n;
    }
    return Kn * sqrt(T) * (1.0 + param) / (n * (T + param));
}

// ---- whether a stage kernel starts while the finalisation before it still runs ----
// Started early (as a programmatic dependent), the stage kernel saves 1 us, but its CTAs go to the
// SMs that the finalisation's blocks have left room on and stay there.  Where the batch is one
// wave, the finalisation sits on many SMs and an SM can take more CTAs than its even share, they
// pile up, and in FP64, which is bound by an SM's FP64 units, the fullest SM sets the time: ten
// half channels of 5 x 3 x 11 nodes and 45 cells at V = 4 and eight cells 668 us per step before
// there were early starts, 1009 with one, 404 without.  Hence, in FP64, none where the finalisation
// holds a quarter of the 152 SMs, both together outnumber the SMs, and an SM could take a third
// more than its share.  Of 510 measured FP64 tilings (17 batches, V = 1, 2, 4, 3 to 64 cells, split
// or not) none is slower by the rule than with early starts throughout, 63 are faster by 3% to 65%.
// FP32, bound by latency, gains by early starts (one C2 channel 53 -> 48 us per step).
inline bool stage_starts_early(bool fp32, long ctas, long fit, long fin_blocks)
{
    const long share = (ctas + 151) / 152;
    return fp32 || 4 * fin_blocks < 152 || ctas + fin_blocks <= 152 || 4 * share > 3 * fit;
}

// ---- the destination of lbs_get_state's gathering launch ----
// A kernel needs the solver's device to be the current one and writes wherever it is told; a
// copy runs whatever device is current and refuses what is not memory.  So the launch takes
// memory of the solver's own device while that is current, in an allocation that holds the
// whole state, and everything else goes through the copies.
struct GatherTarget {
    int device = -1;   // the device whose memory it is, -1 otherwise (host, managed, unknown)
    int current = -1;  // the calling thread's device
    size_t bytes = 0;  // from the destination to the end of its allocation
};
inline bool gather_allowed(const GatherTarget& t, int solver_device, size_t state_bytes)
{
    return t.device == solver_device && t.current == solver_device && state_bytes <= t.bytes;
}

// ---- access to a handle for entry points defined outside api.cu ----
struct HandleView {
    const InstDev* d_inst;   // device array of descriptors
    InstDev inst;            // host copy of the selected instance's descriptor
    int fp32, device;
    void* stream;            // cudaStream_t
};
// fills *out for instance inst of handle h (an lbs_handle); returns 0 or an lbs_status
int handle_view(void* h, int inst, HandleView* out);
// records msg as the calling thread's last error and returns status
int record_error(int status, const char* msg);

// ---- host helpers (quadrature.cpp) ----
void recurrence(int kind, int n, std::vector<double>& alpha, std::vector<double>& beta);
int gauss_rule(int kind, int Q, double* nodes, double* weights);
void hermite_basis(const double* p, int Q, int N, double* out);
void half_basis(const double* xi, int Q, int N, const std::vector<double>& a,
                const std::vector<double>& b, double* out);

}  // namespace lbs
