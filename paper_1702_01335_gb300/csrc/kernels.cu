// Finalisation and seeding kernels and the launchers of every kernel of the
// scheme (the device code shared with the stage kernel is in kernels.cuh; the
// stage kernel's instantiations are in the stage_*.cu translation units).
#include "kernels.cuh"

namespace lbs {

// ---- separate finalisation launches (used when the stage kernel does not fuse them): C
// cells per block of 128 threads, blockIdx.y the instance.  NB bounds the expansion orders of
// the batch (the unrolled coefficient loops run to NB, not to the largest order kMaxN).
template <typename T, int NB, int C>
__global__ void __launch_bounds__(kThreads) finalize_cells(const InstDev* __restrict__ insts, int stage)
{
    __shared__ FinShared<T, C> sm;
    __shared__ double red[8 * (kThreads / 32)];
    __shared__ int last;
    __shared__ InstDev sI;
    const InstDev& I = stage_descriptor(insts + blockIdx.y, &sI);
    const int nblk = (I.Nz + C - 1) / C, c0 = blockIdx.x * C, rot = (blockIdx.x + blockIdx.y) & 3;
    Node<T, NB> node;
    node.load(I, rotated(rot) % (kThreads / C));
    wait_predecessor();
    if (blockIdx.x >= nblk || *I.active == 0) return;
    finalize_group<T, NB, C>(I, c0, min(C, I.Nz - c0), stage, sm, rot, node);
    // the instance's last block to finish (threadfence ticket) forms n_w and, after
    // stage 3, the residual; the counter is reset by its last user
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(I.icount, 1) == nblk - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) *I.icount = 0;
    finalize_instance(I, stage, red);
}

// ---- seed a cell from its record: d_k = f_k / w_k - 1 = R_SCALE Gx Gy Gz (1 + S) - 1,
// formed from the factors' deviations as in the stage kernel; the rounding residual
// (FP32 storage) starts at zero.  Written into whichever buffer holds the state.
template <typename T>
__global__ void __launch_bounds__(128) seed_cells(const InstDev* __restrict__ insts, int inst)
{
    const InstDev& I = insts[inst];
    const int cell = blockIdx.x;
    const T* rc = static_cast<const T*>(I.rec) + (size_t)cell * I.rec_stride;
    T* F = static_cast<T*>(*I.cur ? I.F1 : I.F0) + (size_t)cell * I.Q;
    for (int k = threadIdx.x; k < I.Q; k += blockDim.x) {
        const int j = k % I.Qy, i = (k / I.Qy) % I.Qx, zm = k / I.QxQy;
        const int sg = zm >= I.Qz, m = zm - sg * I.Qz;
        const T gx = rc[R_SCALE1] + (T(1) + rc[R_SCALE1]) * rc[R_DX + i];
        const T gy = rc[R_DX + I.Qx + j], gz = rc[R_DX + I.Qx + I.Qy + zm];
        const T x = ld<T>(I.xi, m);
        const T ex = ld<T>(I.px, i) - rc[R_UX], ey = ld<T>(I.py, j) - rc[R_UY], ez = (sg ? -x : x) - rc[R_UZ];
        const T S = I.reduced ? rc[R_CS] * ((ex * ex + ez * ez) * rc[R_I5T] - (j ? T(0.4) : T(0.8))) *
                                    (ex * rc[R_QX] + ez * rc[R_QZ])
                              : rc[R_CS] * ((ex * ex + ey * ey + ez * ez) * rc[R_I5T] - T(1)) *
                    (ex * rc[R_QX] + ey * rc[R_QY] + ez * rc[R_QZ]);
        const T a = gx + gy + gx * gy, b = a + gz + a * gz;
        F[k] = b + S + b * S;
        if (I.L0) I.L0[(size_t)cell * I.Q + k] = 0;
    }
}

// ---- seed a cell with the free-molecular state of the channel: each velocity carries the
// discrete equilibrium of the wall it left (Appendix, with n_w = 1: p_z > 0 the bottom
// wall, p_z < 0 the top wall; the incoming ghosts' formula), then the cell is rescaled to
// unit density.  The collisionless limit of Couette flow between diffuse walls; a start
// for strongly rarefied instances.  One block per cell; residual 0.
template <typename T>
__global__ void __launch_bounds__(128) seed_free_molecular(const InstDev* __restrict__ insts, int inst)
{
    __shared__ double red[kThreads / 32];
    const InstDev& I = insts[inst];
    const int cell = blockIdx.x;
    T* F = static_cast<T*>(*I.cur ? I.F1 : I.F0) + (size_t)cell * I.Q;
    double m = 0.0;  // the cell's density sum w (1 + d), phi's alone in the reduced model
    for (int k = threadIdx.x; k < I.Q; k += blockDim.x) {
        const int j = k % I.Qy, i = (k / I.Qy) % I.Qx, zm = k / I.QxQy;
        const int sg = zm >= I.Qz, mz = zm - sg * I.Qz;
        const T ax = ld<T>(sg ? I.gwx_top : I.gwx_bot, i), ay = ld<T>(I.gwy, j), az = ld<T>(I.gwz, zm);
        const T a = ax + ay + ax * ay, b = a + az + a * az;
        F[k] = b;
        if (!(I.reduced && j == 1))
            m += double(ld<T>(I.wx, i)) * double(ld<T>(I.wy, j)) * double(ld<T>(I.wz, mz)) * (1.0 + double(b));
    }
    m = block_sum(m, red);
    const T c = T(1.0 / m - 1.0);  // (1 + d) / m - 1 = d + c (1 + d)
    for (int k = threadIdx.x; k < I.Q; k += blockDim.x) {
        const T d = F[k];
        F[k] = d + c * (T(1) + d);
        if (I.L0) I.L0[(size_t)cell * I.Q + k] = 0;
    }
}

// The eight profile rows that lbs_moments reports (n, u_x, T, q_x, q_z, P_xx, P_xz, P_zz:
// rows 0, 1, 4, 5, 7, 8, 12, 10 of the [14][Nz] profiles, one nibble each) of every
// instance, packed [8][Nz] per instance in instance order, so that a whole-batch read is
// one device-to-host copy.  The profiles sit back to back (14 Nz doubles per instance),
// so an instance's offset in out is 8/14 of its offset in prof_all.  Block (b, r) copies
// row r of instance b.
__global__ void __launch_bounds__(128) gather_moment_rows(const InstDev* __restrict__ insts,
                                                          const double* __restrict__ prof_all,
                                                          double* __restrict__ out)
{
    const InstDev& I = insts[blockIdx.x];
    const int r = blockIdx.y, row = (0xAC875410u >> (4 * r)) & 0xFu;
    const long before = (long)(I.prof - prof_all) / 14;  // cells of the instances before b
    const double* __restrict__ src = I.prof + (long)row * I.Nz;
    double* __restrict__ dst = out + 8 * before + (long)r * I.Nz;
    for (int c = threadIdx.x; c < I.Nz; c += blockDim.x) dst[c] = src[c];
}

// 16 bytes at an even address from the two aligned words that hold them: m the offset into a
static __device__ __forceinline__ uint4 word_at(const uint4& a, const uint4& b, int m)
{
    const unsigned r = (m & 2) * 8;
    auto four = [r](unsigned x0, unsigned x1, unsigned x2, unsigned x3, unsigned x4) {
        return make_uint4(__funnelshift_r(x0, x1, r), __funnelshift_r(x1, x2, r), __funnelshift_r(x2, x3, r),
                          __funnelshift_r(x3, x4, r));
    };
    switch (m >> 2) {
        case 0: return four(a.x, a.y, a.z, a.w, b.x);
        case 1: return four(a.y, a.z, a.w, b.x, b.y);
        case 2: return four(a.z, a.w, b.x, b.y, b.z);
        default: return four(a.w, b.x, b.y, b.z, b.w);
    }
}
// n bytes from src to dst by a warp, all even.  Aligned 16-byte stores; where src and dst lie
// differently in their words, a word is put together from the two of the source that hold it.
// Both hold bytes of the copy, so nothing is read outside the source's 16-byte words.
static __device__ __forceinline__ void copy_bytes(unsigned char* dst, const unsigned char* src, size_t n, int lane)
{
    const size_t to_word = (16 - (reinterpret_cast<uintptr_t>(dst) & 15)) & 15, head = to_word < n ? to_word : n;
    const size_t words = (n - head) / 16, tail = head + 16 * words;
    auto two_bytes = [&](size_t at) {
        *reinterpret_cast<unsigned short*>(dst + at) = *reinterpret_cast<const unsigned short*>(src + at);
    };
    if (2 * lane < head) two_bytes(2 * lane);
    if (tail + 2 * lane < n) two_bytes(tail + 2 * lane);
    uint4* d = reinterpret_cast<uint4*>(dst + head);
    const int m = reinterpret_cast<uintptr_t>(src + head) & 15;
    const uint4* s = reinterpret_cast<const uint4*>(src + head - m);
    for (size_t w = lane; w < words; w += 128) {
        uint4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (w + 32 * i < words) {
                a[i] = __ldcs(s + w + 32 * i);
                if (m) b[i] = __ldcs(s + w + 32 * i + 1);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (w + 32 * i < words) __stcs(d + w + 32 * i, m ? word_at(a[i], b[i], m) : a[i]);
    }
}

// The state of instances b0 .. b0 + n - 1 (at: values before b0, total: theirs) to device memory in
// lbs_get_state's layout: every d, then (FP32) every residual.  Each warp takes `per` values of
// the whole, whatever the instances' sizes, and finds the instance they begin in and its
// buffers on the device.  Bound by memory from some 10 MB on, by latency below.
// Measured, host call in us, against blocks shared out by instance with 2-byte units off 16 bytes
// (and against copies): FP32, one 39 MB instance and 99 small ones 66 -> 34 (45), the same to an
// address 8 off 16 bytes 817 -> 41 (53), one 47 MB state 8 off 188 -> 44 (54), one of odd size 2 off
// 194 -> 44 (78), four of 11 MB and odd size 77 -> 35 (103); FP64, 12 MB 8 off 35 -> 19 (29).
__global__ void __launch_bounds__(256) gather_states(const InstDev* __restrict__ insts, int b0, int n, long at,
                                                     long total, long per, unsigned char* dst, int esize)
{
    const int lane = threadIdx.x & 31;
    long v = (blockIdx.x * (long)(blockDim.x / 32) + threadIdx.x / 32) * per;
    const long end = v + per < total ? v + per : total;
    if (v >= end) return;
    // the last instance that begins at or before v: 32 candidates per step
    int b = 0;
    for (int len = n; len > 1;) {
        const int step = (len + 31) / 32, c = lane * step;
        const bool before = c < len && insts[b0 + b + c].state_at - at <= v;
        const int k = __popc(__ballot_sync(0xffffffffu, before)) - 1;  // candidate 0 always is
        b += k * step;
        len = len - k * step < step ? len - k * step : step;
    }
    for (; v < end; ++b) {
        const InstDev& I = insts[b0 + b];
        const long i0 = I.state_at - at, i1 = i0 + (long)I.Nz * I.Q, e = end < i1 ? end : i1;
        const unsigned char* F = static_cast<const unsigned char*>(*I.cur ? I.F1 : I.F0);
        copy_bytes(dst + v * esize, F + (v - i0) * esize, (size_t)(e - v) * esize, lane);
        if (I.L0)
            copy_bytes(dst + total * esize + v * 2, reinterpret_cast<const unsigned char*>(I.L0 + (v - i0)),
                       (size_t)(e - v) * 2, lane);
        v = e;
    }
}

// ---- host launchers ---------------------------------------------------------
cudaError_t launch_gather_states(const InstDev* d_inst, int b0, int n, long at, long total, void* dst, int esize,
                                 cudaStream_t st)
{
    // values of a warp: 128 (an FP32 word per lane), up to 512 while eight warps per SM take them all,
    // then as many more as one wave of 64 warps per SM needs.  Host call in us at 512 / 128 from the
    // start: one C1 channel in FP64 12.3 / 11.6, the low-Mach runs 13.2 / 12.1, 20 table runs
    // 13.6 / 14.8, eight C2 channels 15.3 / 17.9.
    const long few = (total - 1) / (128L * 8 * 152) + 1, many = (total - 1) / (512L * 64 * 152) + 1;
    const long per = few < 4 ? 128 * few : 512 * many, warps = (total + per - 1) / per;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((warps + 7) / 8));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    // the launch's own status: the last error may be an earlier call's (a refused copy's)
    return cudaLaunchKernelEx(&cfg, gather_states, d_inst, b0, n, at, total, per, static_cast<unsigned char*>(dst),
                              esize);
}
cudaError_t launch_gather_moments(const InstDev* d_inst, int ninst, const double* prof_all, double* out,
                                  cudaStream_t st)
{
    gather_moment_rows<<<dim3(ninst, 8), 128, 0, st>>>(d_inst, prof_all, out);
    return cudaGetLastError();
}

size_t stage_smem_bytes(int fp32, int V, int zn, int Qx, int Qy, int nzm, int rstride)
{
    const bool grouped = V & kGrouped;
    const int KC = layout_columns(V), G = factor_stride(Qx, Qy, nzm, grouped, fp32 ? 4 : 8);
    // element and accumulator sizes from the kernel's own types, so that the host's
    // dynamic shared-memory size always covers the kernel's layout
    return stage_smem(zn, KC, G, fp32 ? (int)sizeof(float) : (int)sizeof(double),
                      fp32 ? (int)sizeof(Acc<float>::type) : (int)sizeof(Acc<double>::type), rstride, grouped,
                      V & kZSplit ? 4 : 1)
        .total;
}

// stage CTAs per SM that the register allocator is asked for (shared memory may allow fewer)
int stage_min_ctas(int fp32, int layout)
{
    const int v = layout & 7;
    if (layout & kZSplit) return v == 1 ? MinBlocks<double, 1, 4>::value : MinBlocks<double, 4, 4>::value;
    if (fp32) return v == 1 ? MinBlocks<float, 1, 1>::value : v == 2 ? MinBlocks<float, 2, 1>::value : MinBlocks<float, 4, 1>::value;
    return v == 1 ? MinBlocks<double, 1, 1>::value : v == 2 ? MinBlocks<double, 2, 1>::value : MinBlocks<double, 4, 1>::value;
}

// Finalisation launches carry the device's highest priority: when the batch's halves step
// on two streams, the block scheduler then dispatches one half's finalisation blocks as soon
// as the other half's stage CTAs free room on an SM, instead of after all of them.  (The
// attribute is kept by CUDA-graph capture.)
static int highest_priority()
{
    int least = 0, greatest = 0;
    cudaDeviceGetStreamPriorityRange(&least, &greatest);
    return greatest;
}
template <typename K>
static cudaError_t launch_first(K kernel, dim3 g, dim3 b, cudaStream_t st, const InstDev* d_inst, int stage)
{
    static const int prio = highest_priority();
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributePriority;
    at[0].val.priority = prio;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, d_inst, stage);
}

template <typename T, int C>
static cudaError_t launch_finalize_t(int stage, const InstDev* d_inst, int ninst, int maxNz, int nb, cudaStream_t st)
{
    const dim3 g((maxNz + C - 1) / C, ninst), b(kThreads);
    if (nb <= 4) return launch_first(finalize_cells<T, 4, C>, g, b, st, d_inst, stage);
    if (nb <= 6) return launch_first(finalize_cells<T, 6, C>, g, b, st, d_inst, stage);
    return launch_first(finalize_cells<T, kMaxN, C>, g, b, st, d_inst, stage);
}

template <int C>
static cudaError_t launch_finalize_c(int fp32, int stage, const InstDev* d_inst, int ninst, int maxNz, int nb,
                                     cudaStream_t st)
{
    return fp32 ? launch_finalize_t<float, C>(stage, d_inst, ninst, maxNz, nb, st)
                : launch_finalize_t<double, C>(stage, d_inst, ninst, maxNz, nb, st);
}

// the stage kernel alone
cudaError_t launch_stage_only(int fp32, int red, int V, int stage, const InstDev* d_inst, const Tile* d_tiles,
                              int ntiles, size_t smem, int fuse, bool early, cudaStream_t st)
{
    if (ntiles <= 0) return cudaSuccess;  // a split half whose instances have all retired
    if (fp32)
        return red ? launch_stage_f32_red(V, stage, d_inst, d_tiles, ntiles, smem, fuse, early, st)
                   : launch_stage_f32_full(V, stage, d_inst, d_tiles, ntiles, smem, fuse, early, st);
    return red ? launch_stage_f64_red(V, stage, d_inst, d_tiles, ntiles, smem, fuse, early, st)
               : launch_stage_f64_full(V, stage, d_inst, d_tiles, ntiles, smem, fuse, early, st);
}

// the separate finalisation launches of an unfused stage
cudaError_t launch_finalize(int fp32, int stage, const InstDev* d_inst, int ninst, int maxNz, int fin_cells,
                            int nb, cudaStream_t st)
{
    switch (fin_cells) {
        case 4: return launch_finalize_c<4>(fp32, stage, d_inst, ninst, maxNz, nb, st);
        case 8: return launch_finalize_c<8>(fp32, stage, d_inst, ninst, maxNz, nb, st);
        case 16: return launch_finalize_c<16>(fp32, stage, d_inst, ninst, maxNz, nb, st);
        default: return launch_finalize_c<32>(fp32, stage, d_inst, ninst, maxNz, nb, st);
    }
}

// one RK stage (stage 1..3) or the analysis pass (stage 0); without fusion the
// finalisation follows as two more launches
cudaError_t launch_stage(int fp32, int red, int V, int stage, const InstDev* d_inst, const Tile* d_tiles,
                         int ntiles, size_t smem, int fuse, bool early, int ninst, int maxNz, int fin_cells, int nb,
                         cudaStream_t st)
{
    cudaError_t e = launch_stage_only(fp32, red, V, stage, d_inst, d_tiles, ntiles, smem, fuse, early, st);
    if (e != cudaSuccess || fuse) return e;
    return launch_finalize(fp32, stage, d_inst, ninst, maxNz, fin_cells, nb, st);
}

cudaError_t launch_seed_free_molecular(int fp32, const InstDev* d_inst, int inst, int Nz, cudaStream_t st)
{
    if (fp32) seed_free_molecular<float><<<Nz, 128, 0, st>>>(d_inst, inst);
    else seed_free_molecular<double><<<Nz, 128, 0, st>>>(d_inst, inst);
    return cudaGetLastError();
}

cudaError_t launch_seed(int fp32, const InstDev* d_inst, int inst, int Nz, const double* d_macro,
                        cudaStream_t st)
{
    const int g = (Nz + 3) / 4;
    if (fp32) records_from_macro<float><<<g, kThreads, 0, st>>>(d_inst, inst, d_macro);
    else records_from_macro<double><<<g, kThreads, 0, st>>>(d_inst, inst, d_macro);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (fp32) seed_cells<float><<<Nz, 128, 0, st>>>(d_inst, inst);
    else seed_cells<double><<<Nz, 128, 0, st>>>(d_inst, inst);
    return cudaGetLastError();
}

}  // namespace lbs
