// Warm-start network: a 3-layer perceptron (n_in -> H -> H -> n_out, GELU) that
// maps the parameters of a Couette problem to its steady profiles.  Matrix
// products run on the tensor cores in BF16 with FP32 accumulation
// (mma.sync.m16n8k16): every product operand is rounded to BF16 when it is
// staged into shared memory; biases, GELU, the loss, the gradients' elementwise
// parts and Adam are FP32, with FP32 master weights and BF16 working copies.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lbs.h"
#include "lbs_internal.h"
#include "pdl.cuh"

namespace lbs {
namespace mlp {

// ---- GEMM tiles: C(m, n) = sum_k A(m, k) B(k, n) -------------------------------------------
// A CTA of four warps computes a TILE x TILE block of C.  The products here are small (the
// network of the warm start: at most 256 x 512 x 256 per minibatch), so what bounds a launch is
// latency, not the tensor cores: a whole slice of K (256 values with 32 x 32 tiles, 128 with
// 64 x 64) is staged at once -- one round trip to L2 and one barrier per slice instead of one
// per 16 -- and small tiles spread a product over many SMs.  The 64 x 64 tiles take over where
// a product has more than kSmallTiles 32 x 32 tiles, four per SM: there the larger tile's reuse
// pays.  Measured, 32 against 64, host call of the 6 -> 256 -> 256 -> 512 network: forward at 1000 rows
// 39.8 / 46.9 us, 2000 rows 50.1 / 48.2, 8192 rows 91 / 81, 65536 rows 513 / 393; loss and
// gradients at 1000 rows 96 / 112 us; 1024-wide hidden layers at 1024 rows 291 / 193 us.  The
// weight gradients are a product of their own for this: at 65536 rows they keep the small
// tiles (128 of them; 3178 against 4921 us in all).
// Operands are rounded to BF16 as they are staged, in their own order: a k-contiguous operand
// as [row][k], a row-contiguous one (the transposed products of the backward pass) as [k][row],
// which ldmatrix transposes on the way to the fragments; 16-byte loads where the addresses
// allow.  Every output accumulates its k in steps of 16 in ascending order
// (mma.sync.m16n8k16), so the results do not depend on the tile.
// Measured on the 6 -> 256 -> 256 -> 512 network against 64 x 64 tiles staged 16 deep with separate
// elementwise and column-sum kernels: four minibatches of 250 rows with Adam and the
// parameters copied back 1285 -> 335 us, 2000 rows forward 84 -> 49 us (host calls; the
// kernels of a minibatch about 330 -> 45 us).
constexpr int kThreadsMlp = 128;
constexpr long kSmallTiles = 608;
template <int TILE> struct TileSize {
    static constexpr int TK = 8192 / TILE;             // staged slice of K
    // values of a staged operand in either order
    static constexpr int kOperand = TILE * (TK + 8) > TK * (TILE + 8) ? TILE * (TK + 8) : TK * (TILE + 8);
};

// one operand: element (r, k) is p[r ld + k] (KC: k contiguous) or p[k ld + r]
template <typename T>
struct Operand {
    const T* p;
    long ld;
    int rows;
};

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ __nv_bfloat16 to_b(float v) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ __nv_bfloat16 to_b(__nv_bfloat16 v) { return v; }

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// Staging of rows r0 .. r0 + TILE - 1, k0 .. k0 + kc - 1 (kc a multiple of 16) as BF16, zero
// beyond the operand.  fetch issues every load of the slice into registers (one round trip),
// put rounds and stores them; an operand whose rows are not whole 16-byte words is read by put
// itself.  sums: the thread's FP32 sums over k of its rows r (row-contiguous FP32 operands).
template <int TILE, bool KC, typename T>
struct Stager {
    static constexpr int TK = TileSize<TILE>::TK, VEC = 16 / (int)sizeof(T), LD = KC ? TK + 8 : TILE + 8;
    static constexpr int N = TILE * TK / VEC / kThreadsMlp;       // words per thread
    static constexpr int per = (KC ? TK : TILE) / VEC;            // words along the contiguous direction
    static constexpr int step = kThreadsMlp / per;                // rows (k) between a thread's words
    static_assert(kThreadsMlp % per == 0, "a thread keeps its place in the contiguous direction");
    union Word {
        uint4 w;
        T v[VEC];
    };
    Word x[N];
    bool vec;

    __device__ __forceinline__ void fetch(const Operand<T>& o, int r0, int k0, int K, int kc)
    {
        vec = o.ld % VEC == 0 && reinterpret_cast<uintptr_t>(o.p) % 16 == 0 && (!KC || kc > 16);
        if (!vec) return;
        const int c = (threadIdx.x % per) * VEC, s0 = threadIdx.x / per;
        const int left = KC ? K - (k0 + c) : o.rows - (r0 + c);  // values from here in the contiguous direction
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int s = s0 + i * step;  // row (KC) or k
            x[i].w = make_uint4(0u, 0u, 0u, 0u);
            const bool in = KC ? r0 + s < o.rows : s < kc && k0 + s < K;
            const T* src = o.p + (KC ? (long)(r0 + s) * o.ld + k0 + c : (long)(k0 + s) * o.ld + r0 + c);
            if (in && left >= VEC) x[i].w = *reinterpret_cast<const uint4*>(src);
            else if (in)
                for (int q = 0; q < VEC; ++q)
                    if (q < left) x[i].v[q] = src[q];
        }
    }
    __device__ __forceinline__ void put(const Operand<T>& o, int r0, int k0, int K, int kc, __nv_bfloat16* s,
                                        float* sums) const
    {
        const int tid = threadIdx.x;
        if (vec) {
            const int c = (tid % per) * VEC, s0 = tid / per;
            if (KC && c >= kc) return;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (!KC && s0 + i * step >= kc) break;
                __nv_bfloat16* d = s + (s0 + i * step) * LD + c;
#pragma unroll
                for (int q = 0; q < VEC; q += 2)
                    *reinterpret_cast<__nv_bfloat162*>(d + q) = __nv_bfloat162(to_b(x[i].v[q]), to_b(x[i].v[q + 1]));
                if (!KC && sums)
#pragma unroll
                    for (int q = 0; q < VEC; ++q) sums[q % 4] += to_f(x[i].v[q]);  // FP32: four rows
            }
        } else if (KC) {
#pragma unroll 4
            for (int e = tid; e < TILE * kc; e += kThreadsMlp) {
                const int r = e / kc, k = e - r * kc;
                const bool in = r0 + r < o.rows && k0 + k < K;
                s[r * LD + k] = to_b(in ? o.p[(long)(r0 + r) * o.ld + k0 + k] : T(0.f));
            }
        } else {
            constexpr int q4 = TILE / 4;  // the same rows per thread as FP32 words
            const int r = (tid % q4) * 4;
#pragma unroll 4
            for (int k = tid / q4; k < kc; k += kThreadsMlp / q4)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const bool in = r0 + r + i < o.rows && k0 + k < K;
                    const T v = in ? o.p[(long)(k0 + k) * o.ld + r0 + r + i] : T(0.f);
                    if (sums) sums[i] += to_f(v);
                    s[k * LD + r + i] = to_b(v);
                }
        }
    }
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p, bool trans)
{
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p));
    if (trans)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a)
                     : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(a)
                     : "memory");
}

// what becomes of C(m, n)
enum { EPI_STORE = 0, EPI_BIAS = 1, EPI_BIAS_GELU = 2, EPI_MSE = 3, EPI_GELU_GRAD = 4 };
struct Epilogue {
    float* C;           // the result (BIAS_GELU: z; MSE: dy), row length ldc
    long ldc;
    const float* bias;  // BIAS, BIAS_GELU, MSE
    float* H;           // BIAS_GELU: gelu(z)
    const float* aux;   // MSE: the targets; GELU_GRAD: z (C = acc gelu'(z))
    float scale;        // MSE: 1 / (B n_out)
    double* loss;       // MSE: sum of squared errors
    float* colsum;      // row sums of A over k (the bias gradients), or null
};

template <int TILE, typename TA, typename TB, bool AK, bool BK, int EPI>
__device__ __forceinline__ void gemm_tile(const Operand<TA>& A, const Operand<TB>& B, int K, const Epilogue& ep,
                                          int mt, int nt, __nv_bfloat16* As, __nv_bfloat16* Bs)
{
    constexpr int TK = TileSize<TILE>::TK, LDA = AK ? TK + 8 : TILE + 8, LDB = BK ? TK + 8 : TILE + 8;
    constexpr int WT = TILE / 2, MI = WT / 16, NI = WT / 16;  // warp tile, its 16-row and 16-column blocks
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = mt * TILE, n0 = nt * TILE, wm = (warp >> 1) * WT, wn = (warp & 1) * WT;
    float acc[MI][2 * NI][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NI; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
    const bool with_sums = !AK && sizeof(TA) == 4 && ep.colsum && nt == 0;
    float sums[4] = {0.f, 0.f, 0.f, 0.f};
    Stager<TILE, AK, TA> sa;
    Stager<TILE, BK, TB> sb;
    auto slice = [&](int k0) { return min(TK, (K - k0 + 15) & ~15); };
    sa.fetch(A, m0, 0, K, slice(0));
    sb.fetch(B, n0, 0, K, slice(0));
    for (int k0 = 0; k0 < K; k0 += TK) {
        const int kc = slice(k0);
        if (k0) __syncthreads();  // the previous slice has been read
        sa.put(A, m0, k0, K, kc, As, with_sums ? sums : nullptr);
        sb.put(B, n0, k0, K, kc, Bs, nullptr);
        __syncthreads();
        if (k0 + TK < K) {  // the next slice's loads run behind this slice's products
            sa.fetch(A, m0, k0 + TK, K, slice(k0 + TK));
            sb.fetch(B, n0, k0 + TK, K, slice(k0 + TK));
        }
#pragma unroll 2
        for (int k = 0; k < kc; k += 16) {
            uint32_t a[MI][4], b[NI][4];
#pragma unroll
            for (int i = 0; i < MI; ++i) {
                const int r = wm + 16 * i;
                ldsm4(a[i], AK ? As + (r + (lane & 15)) * LDA + k + (lane >> 4) * 8
                               : As + (k + (lane >> 4) * 8 + (lane & 7)) * LDA + r + ((lane >> 3) & 1) * 8,
                      !AK);
            }
#pragma unroll
            for (int j = 0; j < NI; ++j) {
                const int c = wn + 16 * j;
                ldsm4(b[j], BK ? Bs + (c + (lane >> 4) * 8 + (lane & 7)) * LDB + k + ((lane >> 3) & 1) * 8
                               : Bs + (k + ((lane >> 3) & 1) * 8 + (lane & 7)) * LDB + c + (lane >> 4) * 8,
                      !BK);
            }
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < 2 * NI; ++j)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                        "{%8,%9}, {%0,%1,%2,%3};"
                        : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
                        : "r"(a[i][0]), "r"(a[i][1]), "r"(a[i][2]), "r"(a[i][3]), "r"(b[j >> 1][(j & 1) * 2]),
                          "r"(b[j >> 1][(j & 1) * 2 + 1]));
        }
    }
    launch_dependents();
    const int g = lane >> 2, t = lane & 3, M = A.rows, N = B.rows;
    double err = 0.0;
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NI; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = m0 + wm + 16 * i + g + (r >= 2 ? 8 : 0), n = n0 + wn + 8 * j + 2 * t + (r & 1);
                if (m >= M || n >= N) continue;
                const long e = m * ep.ldc + n;
                float v = acc[i][j][r];
                if (EPI == EPI_BIAS || EPI == EPI_BIAS_GELU || EPI == EPI_MSE) v += ep.bias[n];
                if (EPI == EPI_MSE) {  // dy = 2 (y - t) / (B n_out)
                    const float d = v - ep.aux[e];
                    ep.C[e] = 2.f * d * ep.scale;
                    err += double(d) * double(d);
                } else if (EPI == EPI_GELU_GRAD) {
                    ep.C[e] = v * gelu_grad(ep.aux[e]);
                } else {
                    ep.C[e] = v;
                    if (EPI == EPI_BIAS_GELU) ep.H[e] = gelu(v);
                }
            }
    if (EPI == EPI_MSE) {
        double* red = reinterpret_cast<double*>(As);
        for (int o = 16; o > 0; o >>= 1) err += __shfl_xor_sync(0xffffffffu, err, o);
        __syncthreads();  // the operands have been read
        if (lane == 0) red[warp] = err;
        __syncthreads();
        if (tid == 0) atomicAdd(ep.loss, (red[0] + red[1]) + (red[2] + red[3]));
    }
    if constexpr (!AK && sizeof(TA) == 4) {
        if (with_sums) {  // the same for the whole CTA
            constexpr int per = TILE / 4, rows = kThreadsMlp / per;
            float* red = reinterpret_cast<float*>(As);  // [rows][TILE]
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 4; ++i) red[(tid / per) * TILE + (tid % per) * 4 + i] = sums[i];
            __syncthreads();
            if (tid < TILE && m0 + tid < M) {
                float s = 0.f;
#pragma unroll
                for (int q = 0; q < rows; ++q) s += red[q * TILE + tid];
                ep.colsum[m0 + tid] = s;
            }
        }
    }
}

__device__ __forceinline__ int tiles_of(int n, int TILE) { return (n + TILE - 1) / TILE; }

// the forward products (both operands k-contiguous); *zero, if given, is cleared for the loss
// that a later launch sums
template <int TILE, int EPI>
__global__ void __launch_bounds__(kThreadsMlp) forward_gemm(Operand<float> A, Operand<__nv_bfloat16> B, int K,
                                                            Epilogue ep, double* zero)
{
    __shared__ __align__(16) __nv_bfloat16 As[TileSize<TILE>::kOperand], Bs[TileSize<TILE>::kOperand];
    wait_predecessor();
    if (zero && blockIdx.x == 0 && threadIdx.x == 0) *zero = 0.0;
    const int nt = tiles_of(B.rows, TILE);
    gemm_tile<TILE, float, __nv_bfloat16, true, true, EPI>(A, B, K, ep, blockIdx.x / nt, blockIdx.x % nt,
                                                                  As, Bs);
}

// A layer's backward products in one launch, which both need the layer's dz [B][n] only:
// blocks below nW form dW = dz^T h (and the bias gradients, dz's column sums), the others the
// layer below's dz = (dz W) gelu'(z)
template <int TW, int TD>
__global__ void __launch_bounds__(kThreadsMlp) backward_gemm(Operand<float> dzT, Operand<float> h, int batch,
                                                             Epilogue epW, int nW, Operand<float> dz,
                                                             Operand<__nv_bfloat16> W, int n, Epilogue epD)
{
    constexpr int kOperand = TW == 32 || TD == 32 ? TileSize<32>::kOperand : TileSize<64>::kOperand;
    static_assert(TileSize<32>::kOperand >= TileSize<64>::kOperand, "the larger one");
    __shared__ __align__(16) __nv_bfloat16 As[kOperand], Bs[kOperand];
    wait_predecessor();
    const int b = blockIdx.x;
    if (b < nW) {
        const int nt = tiles_of(h.rows, TW);
        gemm_tile<TW, float, float, false, false, EPI_STORE>(dzT, h, batch, epW, b / nt, b % nt, As,
                                                                      Bs);
    } else {
        const int nt = tiles_of(W.rows, TD);
        gemm_tile<TD, float, __nv_bfloat16, true, false, EPI_GELU_GRAD>(dz, W, n, epD, (b - nW) / nt,
                                                                         (b - nW) % nt, As, Bs);
    }
}

// Adam (bias corrected) on the FP32 masters, then refresh the BF16 weight copies.  g is no
// __restrict__: the kernel starts while its predecessor still writes the gradients, and loads of
// memory promised constant could go through the read-only path or above the wait.
__global__ void adam(float* __restrict__ p, const float* g, float* __restrict__ m,
                     float* __restrict__ v, long n, float lr, float b1, float b2, float eps, float c1, float c2,
                     __nv_bfloat16* __restrict__ pb, const unsigned char* __restrict__ is_w)
{
    wait_predecessor();
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
        const float gg = g[e];
        const float mm = b1 * m[e] + (1.f - b1) * gg;
        const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
        m[e] = mm;
        v[e] = vv;
        const float w = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
        p[e] = w;
        if (is_w[e]) pb[e] = __float2bfloat16_rn(w);
    }
}

__global__ void to_bf16(const float* __restrict__ p, __nv_bfloat16* __restrict__ pb, long n)
{
    for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
        pb[e] = __float2bfloat16_rn(p[e]);
}

}  // namespace mlp
}  // namespace lbs

using namespace lbs;
using namespace lbs::mlp;

struct lbs_mlp {
    int I, H, O, maxB;
    long nW1, nb1, nW2, nb2, nW3, nb3, P;
    long oW1, ob1, oW2, ob2, oW3, ob3;  // offsets into the packed parameter vector
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    unsigned char* mem = nullptr;
    float *p, *g, *m, *v;                 // [P] masters, gradients, Adam moments
    __nv_bfloat16* pb;                    // [P] BF16 copies (weights; biases unused)
    unsigned char* is_w;                  // [P] 1 where the entry is a weight
    float *z1, *h1, *z2, *h2, *dy, *dh, *dz;  // activations and gradients (dh, dz: dz2, dz1), max batch
    double* loss;
    long step = 0;
};

#define MCK(call)                                                                              \
    do {                                                                                       \
        cudaError_t e_ = (call);                                                               \
        if (e_ != cudaSuccess)                                                                 \
            return static_cast<lbs_status>(record_error(LBS_ERR_CUDA, cudaGetErrorString(e_))); \
    } while (0)

static lbs_status merr(lbs_status s, const char* m) { return static_cast<lbs_status>(record_error(s, m)); }

static int blocks(long n) { return (int)std::min<long>((n + 255) / 256, 4096); }
static long tiles(long m, long n, long TILE) { return ((m + TILE - 1) / TILE) * ((n + TILE - 1) / TILE); }

// launch with programmatic dependence on the stream's previous kernel (every kernel of a
// training step waits before it touches memory)
template <typename... P, typename... Q>
static cudaError_t launch(void (*kernel)(P...), long grid, int block, cudaStream_t st, Q... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int EPI>
static cudaError_t forward_layer(lbs_mlp* h, const float* x, int B, int K, long oW, int N, const Epilogue& ep,
                                 double* zero = nullptr)
{
    const Operand<float> A = {x, K, B};
    const Operand<__nv_bfloat16> W = {h->pb + oW, K, N};
    if (tiles(B, N, 32) <= kSmallTiles)
        return launch(forward_gemm<32, EPI>, tiles(B, N, 32), kThreadsMlp, h->stream, A, W, K, ep, zero);
    return launch(forward_gemm<64, EPI>, tiles(B, N, 64), kThreadsMlp, h->stream, A, W, K, ep, zero);
}

// dW [n][m] = dz^T a and db = column sums of dz, for dz [B][n] and the layer's input a [B][m];
// with W [n][m]: also dz_below [B][m] = (dz W) gelu'(z_below)
static cudaError_t backward_layer(lbs_mlp* h, const float* dz, const float* a, int B, int n, int m, long oW, long ob,
                                  float* dz_below, const float* z_below)
{
    const Operand<float> dzT = {dz, n, n}, act = {a, m, m}, d = {dz, n, B};
    const Operand<__nv_bfloat16> W = {h->pb + oW, m, m};
    Epilogue epW = {}, epD = {};
    epW.C = h->g + oW;
    epW.ldc = m;
    epW.colsum = h->g + ob;
    epD.C = dz_below;
    epD.ldc = m;
    epD.aux = z_below;
    const bool sW = tiles(n, m, 32) <= kSmallTiles, sD = !dz_below || tiles(B, m, 32) <= kSmallTiles;
    const long nW = tiles(n, m, sW ? 32 : 64), nD = dz_below ? tiles(B, m, sD ? 32 : 64) : 0;
    auto go = [&](auto kernel) {
        return launch(kernel, nW + nD, kThreadsMlp, h->stream, dzT, act, B, epW, (int)nW, d, W, n, epD);
    };
    return sW ? (sD ? go(backward_gemm<32, 32>) : go(backward_gemm<32, 64>))
              : (sD ? go(backward_gemm<64, 32>) : go(backward_gemm<64, 64>));
}

// the two hidden layers for a batch already on the device; zero: cleared on the way
static lbs_status hidden_layers(lbs_mlp* h, const float* x, int B, double* zero)
{
    Epilogue ep = {};
    ep.C = h->z1;
    ep.H = h->h1;
    ep.ldc = h->H;
    ep.bias = h->p + h->ob1;
    MCK(forward_layer<EPI_BIAS_GELU>(h, x, B, h->I, h->oW1, h->H, ep, zero));
    ep.C = h->z2;
    ep.H = h->h2;
    ep.bias = h->p + h->ob2;
    MCK(forward_layer<EPI_BIAS_GELU>(h, h->h1, B, h->H, h->oW2, h->H, ep));
    return LBS_OK;
}

extern "C" {

lbs_status lbs_mlp_create(lbs_mlp_handle* out, int n_in, int n_hidden, int n_out, int max_batch, void* stream)
{
    if (!out || n_in < 1 || n_hidden < 1 || n_out < 1 || max_batch < 1 || n_in > 4096 || n_hidden > 4096 ||
        n_out > 4096 || max_batch > (1 << 20))
        return merr(LBS_ERR_ARG, "network sizes must lie in 1..4096 and the batch in 1..2^20");
    lbs_mlp* h = new lbs_mlp();
    h->I = n_in; h->H = n_hidden; h->O = n_out; h->maxB = max_batch;
    h->nW1 = (long)n_hidden * n_in; h->nb1 = n_hidden;
    h->nW2 = (long)n_hidden * n_hidden; h->nb2 = n_hidden;
    h->nW3 = (long)n_out * n_hidden; h->nb3 = n_out;
    h->oW1 = 0; h->ob1 = h->oW1 + h->nW1; h->oW2 = h->ob1 + h->nb1; h->ob2 = h->oW2 + h->nW2;
    h->oW3 = h->ob2 + h->nb2; h->ob3 = h->oW3 + h->nW3; h->P = h->ob3 + h->nb3;
    if (stream) {
        h->stream = static_cast<cudaStream_t>(stream);
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete h;
            return merr(LBS_ERR_CUDA, "cudaStreamCreate failed");
        }
        h->own_stream = true;
    }
    const long P = h->P, BH = (long)max_batch * n_hidden, BO = (long)max_batch * n_out;
    size_t bytes = 4 * P * 4 + 2 * P + P + (6 * BH + BO) * 4 + 8 + 16 * 16;  // + alignment slack
    void* mem = nullptr;
    if (cudaMalloc(&mem, bytes) != cudaSuccess) {
        if (h->own_stream) cudaStreamDestroy(h->stream);
        delete h;
        return merr(LBS_ERR_CUDA, "cudaMalloc of the network's buffers failed");
    }
    h->mem = static_cast<unsigned char*>(mem);
    size_t o = 0;
    auto take = [&](size_t n) { size_t r = o; o = (o + n + 15) & ~size_t(15); return h->mem + r; };
    h->p = reinterpret_cast<float*>(take(P * 4));
    h->g = reinterpret_cast<float*>(take(P * 4));
    h->m = reinterpret_cast<float*>(take(P * 4));
    h->v = reinterpret_cast<float*>(take(P * 4));
    h->pb = reinterpret_cast<__nv_bfloat16*>(take(P * 2));
    h->is_w = take(P);
    h->z1 = reinterpret_cast<float*>(take(BH * 4));
    h->h1 = reinterpret_cast<float*>(take(BH * 4));
    h->z2 = reinterpret_cast<float*>(take(BH * 4));
    h->h2 = reinterpret_cast<float*>(take(BH * 4));
    h->dy = reinterpret_cast<float*>(take(BO * 4));
    h->dh = reinterpret_cast<float*>(take(BH * 4));
    h->dz = reinterpret_cast<float*>(take(BH * 4));
    h->loss = reinterpret_cast<double*>(take(8));
    std::vector<unsigned char> isw(P, 0);
    for (long e = h->oW1; e < h->oW1 + h->nW1; ++e) isw[e] = 1;
    for (long e = h->oW2; e < h->oW2 + h->nW2; ++e) isw[e] = 1;
    for (long e = h->oW3; e < h->oW3 + h->nW3; ++e) isw[e] = 1;
    cudaError_t e1 = cudaMemcpyAsync(h->is_w, isw.data(), P, cudaMemcpyHostToDevice, h->stream);
    cudaError_t e2 = cudaMemsetAsync(h->mem, 0, 4 * P * 4, h->stream);
    cudaError_t e3 = cudaStreamSynchronize(h->stream);
    if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess) {
        lbs_mlp_destroy(h);
        return merr(LBS_ERR_CUDA, "initialising the network's buffers failed");
    }
    *out = h;
    return LBS_OK;
}

lbs_status lbs_mlp_destroy(lbs_mlp_handle h)
{
    if (!h) return LBS_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    if (h->mem) cudaFree(h->mem);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
    return LBS_OK;
}

lbs_status lbs_mlp_num_params(lbs_mlp_handle h, long* out)
{
    if (!h || !out) return merr(LBS_ERR_ARG, "invalid handle or null output");
    *out = h->P;
    return LBS_OK;
}

lbs_status lbs_mlp_set_params(lbs_mlp_handle h, const float* host_params)
{
    if (!h || !host_params) return merr(LBS_ERR_ARG, "invalid handle or null parameters");
    for (long e = 0; e < h->P; ++e)
        if (!std::isfinite(host_params[e])) return merr(LBS_ERR_NONFINITE, "parameter not finite");
    MCK(cudaMemcpyAsync(h->p, host_params, h->P * 4, cudaMemcpyHostToDevice, h->stream));
    MCK(cudaMemsetAsync(h->m, 0, h->P * 4, h->stream));
    MCK(cudaMemsetAsync(h->v, 0, h->P * 4, h->stream));
    to_bf16<<<blocks(h->P), 256, 0, h->stream>>>(h->p, h->pb, h->P);
    MCK(cudaGetLastError());
    MCK(cudaStreamSynchronize(h->stream));
    h->step = 0;
    return LBS_OK;
}

lbs_status lbs_mlp_get_params(lbs_mlp_handle h, float* host_params)
{
    if (!h || !host_params) return merr(LBS_ERR_ARG, "invalid handle or null output");
    MCK(cudaMemcpyAsync(host_params, h->p, h->P * 4, cudaMemcpyDeviceToHost, h->stream));
    MCK(cudaStreamSynchronize(h->stream));
    return LBS_OK;
}

lbs_status lbs_mlp_forward(lbs_mlp_handle h, const float* x_dev, int B, float* y_dev)
{
    if (!h || !x_dev || !y_dev || B < 1 || B > h->maxB) return merr(LBS_ERR_ARG, "invalid arguments or batch too large");
    const lbs_status s = hidden_layers(h, x_dev, B, nullptr);
    if (s != LBS_OK) return s;
    Epilogue ep = {};
    ep.C = y_dev;
    ep.ldc = h->O;
    ep.bias = h->p + h->ob3;
    MCK(forward_layer<EPI_BIAS>(h, h->h2, B, h->H, h->oW3, h->O, ep));
    return LBS_OK;
}

lbs_status lbs_mlp_loss_grad(lbs_mlp_handle h, const float* x_dev, const float* t_dev, int B, double* loss_out,
                             float* grad_host)
{
    if (!h || !x_dev || !t_dev || B < 1 || B > h->maxB) return merr(LBS_ERR_ARG, "invalid arguments or batch too large");
    const lbs_status s = hidden_layers(h, x_dev, B, h->loss);
    if (s != LBS_OK) return s;
    const int I = h->I, H = h->H, O = h->O;
    cudaStream_t st = h->stream;
    const long BO = (long)B * O;
    // the output layer with the loss and its gradient dy
    Epilogue ep = {};
    ep.C = h->dy;
    ep.ldc = O;
    ep.bias = h->p + h->ob3;
    ep.aux = t_dev;
    ep.scale = 1.f / float(BO);
    ep.loss = h->loss;
    MCK(forward_layer<EPI_MSE>(h, h->h2, B, H, h->oW3, O, ep));
    // layer 3: dW3 = dy^T h2, db3, dz2 = (dy W3) gelu'(z2); layer 2 likewise; layer 1: dW1, db1
    MCK(backward_layer(h, h->dy, h->h2, B, O, H, h->oW3, h->ob3, h->dh, h->z2));
    MCK(backward_layer(h, h->dh, h->h1, B, H, H, h->oW2, h->ob2, h->dz, h->z1));
    MCK(backward_layer(h, h->dz, x_dev, B, H, I, h->oW1, h->ob1, nullptr, nullptr));
    if (loss_out || grad_host) {
        double L = 0.0;
        MCK(cudaMemcpyAsync(&L, h->loss, 8, cudaMemcpyDeviceToHost, st));
        if (grad_host) MCK(cudaMemcpyAsync(grad_host, h->g, h->P * 4, cudaMemcpyDeviceToHost, st));
        MCK(cudaStreamSynchronize(st));
        if (loss_out) *loss_out = L / double(BO);
    }
    return LBS_OK;
}

lbs_status lbs_mlp_adam(lbs_mlp_handle h, float lr, float beta1, float beta2, float eps)
{
    if (!h || !(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
        return merr(LBS_ERR_ARG, "Adam needs lr > 0, 0 <= beta < 1, eps > 0");
    h->step += 1;
    const float c1 = 1.f - powf(beta1, float(h->step)), c2 = 1.f - powf(beta2, float(h->step));
    MCK(launch(adam, blocks(h->P), 256, h->stream, h->p, h->g, h->m, h->v, h->P, lr, beta1, beta2, eps, c1, c2, h->pb,
               h->is_w));
    return LBS_OK;
}

lbs_status lbs_mlp_get_stream(lbs_mlp_handle h, void** out)
{
    if (!h || !out) return merr(LBS_ERR_ARG, "invalid handle or null output");
    *out = static_cast<void*>(h->stream);
    return LBS_OK;
}

}  // extern "C"
