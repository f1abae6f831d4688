// Passes of the far-field cycle with the column transform split between them.
//
// A column of N = R M pixels needs two factors, an R-point one over the rows
// n1 + M n2 (n2 < R) and an M-point one over n1.  A row-pass block that holds
// the R rows n1 + M n2 of one n1 does the first factor itself after its row
// transforms, and the backward row pass undoes it before its own, so that the
// column pass is left with one M-point codelet, the projection and one M-point
// codelet on values that a single thread loads and stores: no shared memory,
// no barrier, no twiddles, and whole rows of the stack and of the intensities per
// warp.  The arithmetic of every value is that of the passes in kernels_reg.cuh.
//
// The work stack of a frame is [n1][k2][kx]: block n1 of a row pass owns R N
// contiguous values, and the thread (k2, kx) of the column pass finds its M
// values n1 (and its M intensities, rows k2 + R k1) at id + n1 R N, id = k2 N + kx.
//
// Measured at 256^2, alone, per 62 frames (kernels_reg.cuh -> here): column pass 26.9
// -> 13.9 us (from two transposes and three barriers to none: 64 % issue active, the
// projection's arithmetic now half of it), forward row pass 20.8 -> 21.3, backward
// 20.7 -> 22.6 with the column factor added, near-field column pass 19.1 -> 10.7,
// line-search column pass 49 -> 27.  In the cycle: 4000 frames, DM 3.41 -> 3.22 ms; near field,
// 500 frames, 716 -> 630 us; gradient of 1000 frames 755 -> 685 us; two CG steps
// 3.60 -> 2.85 ms; three-mode CG step of 150 frames 944 -> 854 us.  The passes of
// kernels_reg.cuh keep the other sizes and, at 256^2, the stack order that the
// tensor-core, tensor-copy and persistent forms and ptx_llk_static work in.
#pragma once
#include "kernels_reg.cuh"

namespace ptx {

// Sizes whose line search takes them: 128^2 gains there (CG step of 900 frames 424 ->
// 389 us), though not in its other passes (use_split, kernels_reg.cuh).
template <int N>
__host__ __device__ constexpr bool use_split_ls() {
    return N >= 128;
}
template <int N>
struct SplitShape {
    static constexpr int R = Plan<N>::R, M = Plan<N>::M, P = reg_pitch<N>();
    static constexpr int I1 = (R * M + kThreads - 1) / kThreads;  // row first-factor items of a thread (and column items)
    static constexpr int I2 = (R * R + kThreads - 1) / kThreads;  // row second-factor items
    static constexpr int TC = R * reg_cols<N>();                  // threads of the column pass: N / C blocks per frame
    // a row's threads in one warp for both factors: the transpose between them needs no block barrier
    static constexpr bool kWarpRows = R == M && 32 % R == 0 && (R * R) % kThreads == 0;
    // (blocks per SM: forward row pass with 3 / 4 / 5: DM cycle 3282 / 3220 / 3196 us; column
    // pass with 3 / 4 / 5, the last spilling: 3278 / 3220 / 3502)
    static constexpr int RowBlocks = M > 16 ? 2 : 5;
    static constexpr int ColBlocks = M > 16 ? 2 : 4;
};
// sizes whose near-field passes are split too: k_row_proj_s keeps its rows in a warp
template <int N>
__host__ __device__ constexpr bool use_split_nf() {
    return use_split<N>() && SplitShape<N>::kWarpRows;
}
template <int N>
__device__ __forceinline__ void split_row_sync() {
    if constexpr (SplitShape<N>::kWarpRows)
        __syncwarp();
    else
        __syncthreads();
}

// Forward: rows n1 + M n2 of one frame and mode, row transforms, first factor of
// the column transform with its twiddles.  grid (M, frames in batch x K)
template <int N, bool kDM>
__global__ void __launch_bounds__(kThreads, SplitShape<N>::RowBlocks) k_row_fwd_s(ProbArgs a, int j0) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    const int K = a.K, n1b = blockIdx.x;
    const int b = blockIdx.y / K, k = blockIdx.y - b * K, j = j0 + b;
    const int2 p = a.pos[j];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S::I1; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < R * M) {
            const int line = w / M, n1 = w - line * M, y = n1b + M * line;
            const float2* pr = a.probe + ((size_t)k * N + y) * N + n1;
            const float2* ob = a.obj + (size_t)(p.x + y) * a.Wo + p.y + n1;
            float2 q[kDM ? R : 1];
            if constexpr (kDM) {
                const float2* ps = a.psi + (((size_t)j * K + k) * N + y) * N + n1;
                const uint64_t ef = policy_evict_first();
#pragma unroll
                for (int n2 = 0; n2 < R; ++n2) q[n2] = ld_hint(ps + M * n2, ef);
            }
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = cmul(__ldg(pr + M * n2), ob[M * n2]);
            if constexpr (kDM) {
#pragma unroll
                for (int n2 = 0; n2 < R; ++n2) v[n2] = make_float2(2.f * v[n2].x - q[n2].x, 2.f * v[n2].y - q[n2].y);
            }
            Dft<R, -1>::run(v);
            float2* o = buf + line * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, -1>(tw, k2, n1));
        }
    }
    split_row_sync<N>();
#define PTX_DST (a.spec + ((size_t)blockIdx.y * M + n1b) * R * N)
#include "body_split_tail.inc"
#undef PTX_DST
}

// k_col_s for a warp with a thread whose LLK is not finite, again from and back to the work
// stack (which still holds the values): with the scaled quotients, and without the
// background's sums, which are in already.  It takes what it needs from the kernel's
// parameters, so that k_col_s keeps no register for it.
template <int N, bool kBg>
__device__ __noinline__ float col_bright_s(const ProbArgs& a, int j0, int mode) {
    constexpr int M = Plan<N>::M, RN = Plan<N>::R * N;
    const int id = blockIdx.x * SplitShape<N>::TC + threadIdx.x;
    const float* ib = a.iobs + (size_t)(j0 + blockIdx.y) * N * N + id;
    float2* spec = a.spec + (size_t)blockIdx.y * N * N + id;
    float io[M];
    float2 u[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        io[k1] = ib[k1 * RN];
        u[k1] = spec[k1 * RN];
    }
    Dft<M, -1>::run(u);
    const float llk = project_pixels<N, kBg, true>(u, io, a.mbits_s[id], mode, kBg ? a.bg + id : nullptr, nullptr, false);
    if (mode != COL_LLK) {
        Dft<M, +1>::run(u);
#pragma unroll
        for (int n1 = 0; n1 < M; ++n1) spec[n1 * RN] = u[n1];
    }
    return llk;
}

// Column pass, one mode: second factor, projection and LLK (or the gradient's
// weights), second factor of the inverse.  grid (N / C, frames in batch)
template <int N, bool kBg, bool kCycle>
__global__ void __launch_bounds__(SplitShape<N>::TC, SplitShape<N>::ColBlocks * kThreads / SplitShape<N>::TC)
    k_col_s(const __grid_constant__ ProbArgs a, int j0, int mode_arg) {
    const int mode = kCycle ? (int)COL_PROJECT : mode_arg;
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, RN = R * N;
    __shared__ double red_s[S::TC / 32];
    pdl_launch_dependents();
    const int id = blockIdx.x * S::TC + threadIdx.x;
    const int j = j0 + blockIdx.y;
    const float* ib = a.iobs + (size_t)j * N * N + id;
    float io[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) io[k1] = __ldcs(ib + k1 * RN);
    const uint32_t mbits = a.mbits_s[id];
    float2* spec = a.spec + (size_t)blockIdx.y * N * N + id;
    // the forward row pass that wrote the work stack may still be running
    pdl_wait();
    const uint64_t el = policy_evict_last();
    float2 u[M];
#pragma unroll
    for (int n1 = 0; n1 < M; ++n1) u[n1] = ld_hint(spec + n1 * RN, el);
    Dft<M, -1>::run(u);
    float llk = project_pixels<N, kBg, false>(u, io, mbits, mode, kBg ? a.bg + id : nullptr, a.bg_acc + id,
                                              a.bg_acc != nullptr);
    if (__all_sync(0xffffffffu, llk < kInf)) {
        if (mode != COL_LLK) {
            Dft<M, +1>::run(u);
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) st_hint(spec + n1 * RN, u[n1], el);
        }
    } else {  // bright pixels without a model
        llk = col_bright_s<N, kBg>(a, j0, mode);
    }
    const double tot = block_sum_pos<S::TC>(llk, red_s);
    if (threadIdx.x == 0) a.llk_part[(size_t)j * gridDim.x + blockIdx.x] = tot;
}

// Column pass for K > 1 modes: the thread sums |X^_k|^2 of its pixels over the
// modes, then transforms each mode again from the stack and applies the common
// factor: a second M-point codelet per value instead of a write and a read of
// X^_k.  grid (N / C, frames in batch)
template <int N, bool kCycle>
__global__ void __launch_bounds__(SplitShape<N>::TC, SplitShape<N>::ColBlocks * kThreads / SplitShape<N>::TC)
    k_col_modes_s(ProbArgs a, int j0, int mode_arg) {
    const int mode = kCycle ? (int)COL_PROJECT : mode_arg;
    const float* bgp = kCycle ? nullptr : a.bg;
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, RN = R * N;
    __shared__ double red_s[S::TC / 32];
    pdl_launch_dependents();
    const int K = a.K;
    const int id = blockIdx.x * S::TC + threadIdx.x;
    const int j = j0 + blockIdx.y;
    const uint32_t mbits = a.mbits_s[id];
    float2* spec = a.spec + (size_t)blockIdx.y * K * N * N + id;
    const uint64_t el = policy_evict_last();
    float f[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) f[k1] = 0.f;
    pdl_wait();
    for (int k = 0; k < K; ++k) {
        float2 u[M];
#pragma unroll
        for (int n1 = 0; n1 < M; ++n1) u[n1] = ld_hint(spec + (size_t)k * N * N + n1 * RN, el);
        Dft<M, -1>::run(u);
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) f[k1] += cnorm(u[k1]);
    }
    constexpr float invN2 = 1.0f / float(N * N);
    const float* ib = a.iobs + (size_t)j * N * N + id;
    QuadAdd<M> bg_sum(a.bg_acc + id, RN);
    float llk = 0.f;  // the terms are >= 0: a plain float sum of a thread's pixels
    float io_r[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) io_r[k1] = __ldcs(ib + k1 * RN);
    by_brightness(io_r, [&](auto bright) {
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) {
            const bool masked = (mbits >> k1) & 1u;
            const float io = io_r[k1];
            float ic = f[k1] * invN2;
            if (bgp) {
                const int pix = id + k1 * RN;
                ic += __ldg(bgp + pix);
                if (a.bg_acc) bg_sum.put(k1, masked ? 0.f : quotient(io, ic));
            }
            if (mode == COL_PROJECT) {
                float ratio;
                const float term = llk_term_ratio<bright.value>(ic, io, ratio);
                if (!masked) llk += term;
                f[k1] = masked ? 0.f : (ratio - 1.0f) * invN2;
            } else {
                if (!masked) llk += llk_term_fast<bright.value>(ic, io);
                f[k1] = masked ? 0.f : 2.0f * (1.0f - io_over_ic(io, ic)) * invN2;
            }
        }
    });
    if (mode != COL_LLK) {
        for (int k = 0; k < K; ++k) {
            float2 u[M];
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) u[n1] = ld_hint(spec + (size_t)k * N * N + n1 * RN, el);
            Dft<M, -1>::run(u);
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) u[k1] = cscale(u[k1], f[k1]);
            Dft<M, +1>::run(u);
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) st_hint(spec + (size_t)k * N * N + n1 * RN, u[n1], el);
        }
    }
    const double tot = block_sum_pos<S::TC>(llk, red_s);
    if (threadIdx.x == 0) a.llk_part[(size_t)j * gridDim.x + blockIdx.x] = tot;
}

// Near field: column pass of the propagator (k_col_nf's arithmetic), h or
// conj(h) between the second factors.  grid (N / C, frames in batch)
template <int N, int DIR>
__global__ void __launch_bounds__(SplitShape<N>::TC, SplitShape<N>::ColBlocks * kThreads / SplitShape<N>::TC)
    k_col_nf_s(ProbArgs a) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, RN = R * N;
    pdl_launch_dependents();
    const int id = blockIdx.x * S::TC + threadIdx.x;
    const int k2 = id / N, kx = id - k2 * N;
    float2* spec = a.spec + (size_t)blockIdx.y * N * N + id;
    float2 tx = a.nf_t[kx];
    if constexpr (DIR < 0) tx.y = -tx.y;
    constexpr float invN2 = 1.0f / float(N * N);
    pdl_wait();
    const uint64_t el = policy_evict_last();
    float2 u[M];
#pragma unroll
    for (int n1 = 0; n1 < M; ++n1) u[n1] = ld_hint(spec + n1 * RN, el);
    Dft<M, -1>::run(u);
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        float2 ty = __ldg(a.nf_t + k2 + R * k1);
        if constexpr (DIR < 0) ty.y = -ty.y;
        u[k1] = cscale(cmul(u[k1], cmul(ty, tx)), invN2);
    }
    Dft<M, +1>::run(u);
#pragma unroll
    for (int n1 = 0; n1 < M; ++n1) st_hint(spec + n1 * RN, u[n1], el);
}

// Near field: the rows n1b + M l at the detector (k_row_proj's arithmetic) between
// the propagators' first column factors: inverse column factor, inverse rows,
// projection and LLK, forward rows, forward column factor.  grid (M, frames in batch)
template <int N, bool kCycle>
__global__ void __launch_bounds__(kThreads, SplitShape<N>::ColBlocks) k_row_proj_s(ProbArgs a, int j0, int llk_only_arg) {
    const int llk_only = kCycle ? 0 : llk_only_arg;
    const float* bgp = kCycle ? nullptr : a.bg;
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    static_assert(S::kWarpRows && S::I2 == 1 && S::I1 == 1, "one item per thread, rows within a warp");
    extern __shared__ __align__(16) float2 sm[];
    __shared__ double red_s[kThreads / 32];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    const int n1b = blockIdx.x, j = j0 + blockIdx.y;
    const int line = threadIdx.x / R, t = threadIdx.x - line * R;  // R == M: the same row in both factors
    const int y = n1b + M * line;
    float2* spec = a.spec + ((size_t)blockIdx.y * M + n1b) * R * N;
    float io[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) io[k1] = __ldcs(a.iobs + ((size_t)j * N + y) * N + t + R * k1);
    __syncthreads();
    pdl_wait();
    {
        const int kx = threadIdx.x;
        const uint64_t el = policy_evict_last();
        float2 v[R];
#pragma unroll
        for (int k2 = 0; k2 < R; ++k2) v[k2] = ld_hint(spec + k2 * N + kx, el);
#pragma unroll
        for (int k2 = 1; k2 < R; ++k2) v[k2] = cmul(v[k2], tw_get<N, +1>(tw, k2, n1b));
        Dft<R, +1>::run(v);
#pragma unroll
        for (int l = 0; l < R; ++l) buf[l * P + kx] = v[l];
    }
    __syncthreads();
    float2* o = buf + line * P;
    float2 v[R];
#pragma unroll
    for (int n2 = 0; n2 < R; ++n2) v[n2] = o[t + M * n2];
    __syncwarp();
    Dft<R, +1>::run(v);
    o[t] = v[0];
#pragma unroll
    for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1) + t] = cmul(v[k2], tw_get<N, +1>(tw, k2, t));
    __syncwarp();
    float2 u[M];
#pragma unroll
    for (int n1 = 0; n1 < M; ++n1) u[n1] = o[t * (M + 1) + n1];
    __syncwarp();
    Dft<M, +1>::run(u);  // the detector wave at x = t + R k1
    float llk = 0.f;  // the terms are >= 0: a plain float sum of a thread's pixels
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        const int pix = y * N + t + R * k1;
        float ic = cnorm(u[k1]);
        const bool masked = a.mask[pix] != 0;
        if (bgp) {  // incoherent background in the detector plane
            ic += __ldg(bgp + pix);
            if (a.bg_acc && !masked) atomicAdd(a.bg_acc + pix, quotient(io[k1], ic));
        }
        if (!masked) llk += llk_term_fast<true>(ic, io[k1]);
        const float f = masked ? 0.f : amp_ratio(io[k1], ic) - 1.0f;
        u[k1] = cscale(u[k1], f);
    }
    const double tot = block_sum_double<kThreads>((double)llk, red_s);
    if (threadIdx.x == 0) a.llk_part[(size_t)j * gridDim.x + blockIdx.x] = tot;
    if (llk_only) return;
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) o[t + R * k1] = u[k1];
    __syncwarp();
#pragma unroll
    for (int n2 = 0; n2 < R; ++n2) v[n2] = o[t + M * n2];
    __syncwarp();
    Dft<R, -1>::run(v);
    o[t] = v[0];
#pragma unroll
    for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1) + t] = cmul(v[k2], tw_get<N, -1>(tw, k2, t));
    __syncwarp();
#define PTX_DST spec
#include "body_split_tail.inc"
#undef PTX_DST
}

// Line search (k_row_fwd_ls_r's waves): grid (M, frames in batch, waves x K)
template <int N>
__global__ void __launch_bounds__(kThreads, SplitShape<N>::RowBlocks) k_row_fwd_ls_s(ProbArgs a, int j0) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    const int n1b = blockIdx.x, b = blockIdx.y;
    const int wave = blockIdx.z / a.K, k = blockIdx.z - wave * a.K;
    const LsWave w0 = ls_wave(a, wave);
    const int2 p = a.pos[j0 + b];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S::I1; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < R * M) {
            const int line = w / M, n1 = w - line * M, y = n1b + M * line;
            const size_t pi = ((size_t)k * N + y) * N + n1;
            const size_t oi = (size_t)(p.x + y) * a.Wo + p.y + n1;
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = cmul(__ldg(w0.p + pi + M * n2), __ldg(w0.o + oi + M * n2));
            if (w0.p2) {
#pragma unroll
                for (int n2 = 0; n2 < R; ++n2) v[n2] = cadd(v[n2], cmul(__ldg(w0.p2 + pi + M * n2), __ldg(w0.o2 + oi + M * n2)));
            }
            Dft<R, -1>::run(v);
            float2* o = buf + line * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, -1>(tw, k2, n1));
        }
    }
    split_row_sync<N>();
#define PTX_DST (a.spec + ((((size_t)b * gridDim.z + blockIdx.z) * M) + n1b) * R * N)
#include "body_split_tail.inc"
#undef PTX_DST
}

// Line search, column pass (k_col_ls_r's sums): second factors of every wave of
// the thread's pixels.  grid (N / C, frames in batch)
template <int N, bool kModes, bool kThree>
__global__ void __launch_bounds__(SplitShape<N>::TC, (ls_min_blocks<N, kModes, kThree>() * kThreads + SplitShape<N>::TC - 1) /
                                                         SplitShape<N>::TC)
    k_col_ls_s(ProbArgs a, int j0) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, RN = R * N, kWaves = kThree ? 3 : 2;
    __shared__ double red_s[2][S::TC];
    pdl_launch_dependents();
    const int K = kModes ? a.K : 1;
    const int id = blockIdx.x * S::TC + threadIdx.x;
    const int j = j0 + blockIdx.y;
    constexpr float invN2 = 1.0f / float(N * N);
    const float2* spec = a.spec + (size_t)blockIdx.y * K * kWaves * N * N + id;
    const float* io_p = a.iobs + (size_t)j * N * N + id;
    const uint32_t mbits = a.mbits_s[id];
    float2 A[M], B[M];
    float ic_s[kModes ? M : 1], di_s[kModes ? M : 1], d2_s[kModes || kThree ? M : 1];
    if constexpr (kModes) {
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) ic_s[k1] = di_s[k1] = d2_s[k1] = 0.f;
    }
    auto wave = [&](float2* v, const float2* w) {
#pragma unroll
        for (int n1 = 0; n1 < M; ++n1) v[n1] = __ldcs(w + n1 * RN);
    };
    // the intensities come from HBM and are needed last: into L2 meanwhile
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) asm volatile("prefetch.global.L2 [%0];" ::"l"(io_p + k1 * RN));
    }
    pdl_wait();
    for (int k = 0; k < K; ++k) {
        const float2* wa = spec + (size_t)k * N * N;  // wave w of mode k: (w K + k) N^2
        const float2* wb = wa + (size_t)K * N * N;
        const float2* wc = wb + (size_t)K * N * N;
        wave(A, wa);
        wave(B, kThree ? wc : wb);
        Dft<M, -1>::run(A);
        Dft<M, -1>::run(B);
        if constexpr (kThree) {
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) {
                const float t = 4.f * (A[k1].x * B[k1].x + A[k1].y * B[k1].y) * invN2;
                if constexpr (kModes)
                    d2_s[k1] += t;
                else
                    d2_s[k1] = t;
            }
            wave(B, wb);
            Dft<M, -1>::run(B);
        }
        if constexpr (kModes) {
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) {
                ic_s[k1] += cnorm(A[k1]) * invN2;
                di_s[k1] += 2.f * (A[k1].x * B[k1].x + A[k1].y * B[k1].y) * invN2;
                d2_s[k1] += 2.f * cnorm(B[k1]) * invN2;
            }
        }
    }
    KahanF l1, l2;  // per-pixel terms in single precision, compensated sums
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        float ic, di, dd;
        if constexpr (kModes) {
            ic = ic_s[k1];
            di = di_s[k1];
            dd = d2_s[k1];
        } else {
            ic = cnorm(A[k1]) * invN2;
            di = 2.f * (A[k1].x * B[k1].x + A[k1].y * B[k1].y) * invN2;
            dd = 2.f * cnorm(B[k1]) * invN2;
            if constexpr (kThree) dd = d2_s[k1] + dd;
        }
        if ((mbits >> k1) & 1u) continue;
        ic += a.bg ? __ldg(a.bg + id + k1 * RN) : 0.f;
        const float io = fmaxf(__ldcs(io_p + k1 * RN), 0.f);
        float w1, q;  // I_o dI^2 / I_c^2 = I_o q^2
        ls_weights<kModes>(io, ic, di, w1, q);
        l1.add(w1 * di);
        l2.add(fmaf(w1, dd, io * q * q));
    }
    block_sum_pair<S::TC>(l1.value(), l2.value(), red_s, a.ls_part + 2 * ((size_t)j * gridDim.x + blockIdx.x));
}

// Backward: first factor of the inverse column transform, row transforms, then
// Psi' and the probe sums (or the gradient) as in the backward row pass of
// kernels_reg.cuh.  grid (M, G K); blockIdx.y = slot * K + mode
// The object rows are staged by the thread (M < R) or the warp that uses them.
// DM cycle / gradient of 900 frames, kernels_reg.cuh -> split passes: 160^2 391 -> 373 /
// 300 -> 276 us, 192^2 520 -> 496 / 413 -> 368, 224^2 711 -> 698 / 579 -> 525.
template <int N, int kForm>
__global__ void __launch_bounds__(kThreads, 2) k_row_bwd_s(ProbArgs a, int j0, int nb, int mode_arg, int upd_obj_arg,
                                                           int upd_probe_arg) {
    const int mode = kForm == 1 ? (int)BWD_DM : kForm >= 2 ? (int)BWD_GRAD : mode_arg;
    const int upd_probe = kForm == 1 || kForm == 3 ? 1 : kForm == 2 ? 0 : upd_probe_arg;
    const int upd_obj = kForm >= 2 ? 1 : upd_obj_arg;
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    constexpr bool kWarp = S::kWarpRows;
    static_assert(R * R == kThreads && M <= R && N <= kThreads, "one item per thread");
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* stage = sm + N;          // [R][N] next frame's values (cp.async)
    float2* ostage = stage + R * N;  // next frame's object values: [R][N], or [M][thread] (cp.async)
    float2* buf = ostage + M * kThreads;
    load_twiddles<N>(tw);
    const int K = a.K, n1b = blockIdx.x, t = threadIdx.x;
    const int slot = blockIdx.y / K, k = blockIdx.y - slot * K;
    const int G = gridDim.y / K;
    const bool acc_p = upd_probe != 0, acc_o = upd_obj != 0;
    const bool stage_obj = mode != BWD_GRAD || acc_p;
    const int line = t / R, k2t = t - line * R;  // second factor: pixels k2t + R k1 of row `line`
    const int l1 = t / M, n1 = t - l1 * M;       // first factor (t < R M): row l1, elements n1 + M i
    const int y = n1b + M * line;
    auto prefetch_spec = [&](int b) {
        const float2* src = a.spec + (((size_t)b * K + k) * M + n1b) * R * N;
        const uint64_t ef = policy_evict_first();  // the stack's last read
#pragma unroll
        for (int i = 0; i < (R * N / 2 + kThreads - 1) / kThreads; ++i) {
            const int e = 2 * (t + i * kThreads);
            if (R * N / 2 % kThreads == 0 || e < R * N) cp_async16_hint(stage + e, src + e, ef);
        }
        cp_async_commit();
    };
    auto prefetch_obj = [&](int b) {
        if (stage_obj) {
            const int2 q = a.pos[j0 + b];
            if constexpr (kWarp) {  // the rows of this warp's lines (8-byte aligned only)
                constexpr int kLines = 32 / R;
#pragma unroll
                for (int l = 0; l < kLines; ++l) {
                    const int row = (t >> 5) * kLines + l;
                    const float2* src = a.obj + (size_t)(q.x + n1b + M * row) * a.Wo + q.y + (t & 31);
                    float2* dst = ostage + row * N + (t & 31);
#pragma unroll
                    for (int i = 0; i < N / 32; ++i) cp_async8(dst + 32 * i, src + 32 * i);
                }
            } else {
                const float2* src = a.obj + (size_t)(q.x + y) * a.Wo + q.y + k2t;
#pragma unroll
                for (int k1 = 0; k1 < M; ++k1) cp_async8(ostage + k1 * kThreads + t, src + R * k1);
            }
        }
        cp_async_commit();
    };
    pdl_launch_dependents();
    if (slot < nb) prefetch_obj(slot);
    pdl_wait();
    if (slot < nb) prefetch_spec(slot);
    float2 np_r[M], pr_r[M];
    float dp_r[M];
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        np_r[k1] = make_float2(0.f, 0.f);
        dp_r[k1] = 0.f;
        pr_r[k1] = __ldg(a.probe + ((size_t)k * N + y) * N + k2t + R * k1);
    }
    for (int b = slot; b < nb; b += G) {
        const int j = j0 + b;
        const int2 p = a.pos[j];
        cp_async_wait_all();
        __syncthreads();
        if (N == kThreads || t < N) {  // columns: thread kx, first factor of the inverse over k2 -> rows n1b + M l
            float2 v[R];
            v[0] = stage[t];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) v[k2] = cmul(stage[k2 * N + t], tw_get<N, +1>(tw, k2, n1b));
            Dft<R, +1>::run(v);
#pragma unroll
            for (int l = 0; l < R; ++l) buf[l * P + t] = v[l];
        }
        __syncthreads();
        if (b + G < nb) prefetch_spec(b + G);  // the stage is free again
        {
            float2 v[R];
            const bool on = kWarp || t < R * M;
            if (on) {
#pragma unroll
                for (int n2 = 0; n2 < R; ++n2) v[n2] = buf[l1 * P + n1 + M * n2];
            }
            split_row_sync<N>();
            if (on) {
                Dft<R, +1>::run(v);
                float2* o = buf + l1 * P + n1;
                o[0] = v[0];
#pragma unroll
                for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, +1>(tw, k2, n1));
            }
        }
        split_row_sync<N>();
        float2 u[M];
#pragma unroll
        for (int i = 0; i < M; ++i) u[i] = buf[line * P + k2t * (M + 1) + i];
        Dft<M, +1>::run(u);
        const size_t orow = (size_t)(p.x + y) * a.Wo + p.y + k2t;
        float2* ps = (mode != BWD_GRAD) ? a.psi + (((size_t)j * K + k) * N + y) * N + k2t : nullptr;
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) {
            const float2 obv = !stage_obj ? make_float2(0.f, 0.f)
                                          : (kWarp ? ostage[line * N + k2t + R * k1] : ostage[k1 * kThreads + t]);
            float2 wv;
            if (mode == BWD_GRAD) {
                wv = u[k1];
                if (acc_o) {
                    const float2 c = cconjmul(pr_r[k1], wv);
                    red_add_v2(a.grad_obj + orow + R * k1, c.x, c.y);
                }
            } else {
                wv = cadd(cmul(pr_r[k1], obv), u[k1]);
                __stcs(ps + R * k1, wv);
            }
            if (acc_p) {
                const float2 c = cconjmul(obv, wv);
                np_r[k1].x += c.x;
                np_r[k1].y += c.y;
                dp_r[k1] += cnorm(obv);
            }
        }
        if constexpr (kWarp) __syncwarp();
        if (b + G < nb) prefetch_obj(b + G);  // the object values are free again
    }
    if (acc_p) {
        const size_t pidx = ((size_t)k * N + y) * N + k2t;
#pragma unroll
        for (int k1 = 0; k1 < M; ++k1) {
            if (mode == BWD_GRAD)
                red_add_v2(a.grad_probe + pidx + R * k1, np_r[k1].x, np_r[k1].y);
            else
                red_add_v4(a.acc_probe + pidx + R * k1, np_r[k1].x, np_r[k1].y, dp_r[k1], 0.f);
        }
    }
}

// Sixteen 32-bit words per thread of a warp in tensor memory (the warp's lanes of its
// quarter, columns from addr on).  A load and its wait are one statement, so that
// nothing that uses the values can be moved in between.
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const float* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(addr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
        "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
        "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
        "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// The same for the sizes whose second factor is larger than the first (M > R = 16):
// two items of a thread per step (a column of 16 values; 16 pixels of a row), one
// M-point codelet in between.  The probe sums of a thread's 32 pixels are 96 words:
// in registers they would leave one block per SM, so they live in tensor memory (two
// blocks share its 512 columns), which a warp reads and writes at its own lanes
// without touching the shared-memory pipe that the transposes load.  Three-mode
// 512^2 frames, per 19 frames alone: 118 us (kernels_reg.cuh), 131 with one block of 512
// threads and register sums, 92 so; DM cycles with all split passes, kernels_reg.cuh ->
// here: 300 x 512^2 of three modes 3.89 -> 3.65 ms, 150 x 512^2 680 -> 620 us, 200 x 448^2
// 750 -> 650, 300 x 384^2 815 -> 700, AP of 203 x 400^2 with a background 717 -> 640.  (At
// 256^2 the 48 words fit the registers beside staged loads: 22.6 us per 62 frames
// there, 27 this way with three blocks per SM, more with four.)  grid (M, G K)
constexpr uint32_t kBwdTmemCols = 256;
template <int N, int kForm>
__global__ void __launch_bounds__(kThreads, 2) k_row_bwd_s2(ProbArgs a, int j0, int nb, int mode_arg, int upd_obj_arg,
                                                            int upd_probe_arg) {
    const int mode = kForm == 1 ? (int)BWD_DM : kForm >= 2 ? (int)BWD_GRAD : mode_arg;
    const int upd_probe = kForm == 1 || kForm == 3 ? 1 : kForm == 2 ? 0 : upd_probe_arg;
    const int upd_obj = kForm >= 2 ? 1 : upd_obj_arg;
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P, I = S::I1;
    static_assert(R == 16 && BwdShape<N>::kSwap && BwdShape<N>::R == M, "the M-point factor first, 16 pixels per item");
    static_assert(kThreads == R * R && I == 2 && 2 * 3 * 16 * I <= (int)kBwdTmemCols, "two warps per quarter of tensor memory");
    extern __shared__ __align__(16) float2 sm[];
    __shared__ uint32_t tmem_slot;
    float2* tw = sm;
    float2* buf = sm + N;
    const int K = a.K, n1b = blockIdx.x, t = threadIdx.x, warp = t >> 5;
    const int slot = blockIdx.y / K, k = blockIdx.y - slot * K;
    const int G = gridDim.y / K;
    const bool acc_p = upd_probe != 0, acc_o = upd_obj != 0;
    load_twiddles<N>(tw);
    uint32_t acc = 0;  // this thread's words: [item][Re N_P, Im N_P, D_P][16 pixels]
    if (acc_p) {
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             (uint32_t)__cvta_generic_to_shared(&tmem_slot)),
                         "r"(kBwdTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        acc = tmem_slot + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * 48u * I;
        const float zero[16] = {};
#pragma unroll
        for (int q = 0; q < 3 * I; ++q) tmem_st16(acc + 16 * q, zero);
        tmem_wait_st();
    } else {
        __syncthreads();
    }
    // (only now: a dependent pass that waits with tensor memory of its own must not
    // be able to take what a block of this one still needs)
    pdl_launch_dependents();
    pdl_wait();
    const uint64_t ef = policy_evict_first();  // the stack's last read
    for (int b = slot; b < nb; b += G) {
        const int j = j0 + b;
        const int2 p = a.pos[j];
        const float2* src = a.spec + (((size_t)b * K + k) * M + n1b) * R * N;
        {  // columns: first factor of the inverse over k2 -> rows n1b + M l
            float2 v[I][R];
#pragma unroll
            for (int i = 0; i < I; ++i) {
                const int kx = t + i * kThreads;
#pragma unroll
                for (int k2 = 0; k2 < R; ++k2)
                    v[i][k2] = kx < N ? ld_hint(src + k2 * N + kx, ef) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < I; ++i) {
#pragma unroll
                for (int k2 = 1; k2 < R; ++k2) v[i][k2] = cmul(v[i][k2], tw_get<N, +1>(tw, k2, n1b));
                Dft<R, +1>::run(v[i]);
            }
            __syncthreads();  // the previous frame's rows have been read
#pragma unroll
            for (int i = 0; i < I; ++i) {
                const int kx = t + i * kThreads;
                if (kx < N) {
#pragma unroll
                    for (int l = 0; l < R; ++l) buf[l * P + kx] = v[i][l];
                }
            }
        }
        __syncthreads();
        {  // rows: first factor, row t / R (its sixteen threads are in one warp), elements t % R + R i
            const int n1 = t % R;
            float2* o = buf + t / R * P + n1;
            float2 v[M];
#pragma unroll
            for (int n2 = 0; n2 < M; ++n2) v[n2] = o[R * n2];
            __syncwarp();
            Dft<M, +1>::run(v);
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < M; ++k2) o[k2 * (R + 1)] = cmul(v[k2], tw_bwd<N>(tw, k2, n1));
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < I; ++i) {  // rows: second factor, pixels x0 + M k1 of row `line`
            const int w = t + i * kThreads;
            const bool on = w < N;
            float tx[R], ty[R], tn[R];
            if (on) {
                const int line = w / M, x0 = w - line * M, y = n1b + M * line;
                const float2* pr = a.probe + ((size_t)k * N + y) * N + x0;
                const size_t orow = (size_t)(p.x + y) * a.Wo + p.y + x0;
                float2* ps = (mode != BWD_GRAD) ? a.psi + (((size_t)j * K + k) * N + y) * N + x0 : nullptr;
                float2 ob[R];
                if (mode != BWD_GRAD || acc_p) {
#pragma unroll
                    for (int k1 = 0; k1 < R; ++k1) ob[k1] = a.obj[orow + M * k1];
                }
                float2 u[R];
#pragma unroll
                for (int n = 0; n < R; ++n) u[n] = buf[line * P + x0 * (R + 1) + n];
                Dft<R, +1>::run(u);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) {
                    const float2 prv = __ldg(pr + M * k1);
                    float2 wv;
                    if (mode == BWD_GRAD) {
                        wv = u[k1];
                        if (acc_o) {
                            const float2 c = cconjmul(prv, wv);
                            red_add_v2(a.grad_obj + orow + M * k1, c.x, c.y);
                        }
                    } else {
                        wv = cadd(cmul(prv, ob[k1]), u[k1]);
                        __stcs(ps + M * k1, wv);
                    }
                    if (acc_p) {
                        const float2 c = cconjmul(ob[k1], wv);
                        tx[k1] = c.x;
                        ty[k1] = c.y;
                        tn[k1] = cnorm(ob[k1]);
                    }
                }
            } else {
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) tx[k1] = ty[k1] = tn[k1] = 0.f;
            }
            if (acc_p) {  // (whole warps)
                __syncwarp();
                float v[16];
                const uint32_t at = acc + 48 * i;
                tmem_ld16(at, v);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) tx[k1] += v[k1];
                tmem_st16(at, tx);
                tmem_ld16(at + 16, v);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) ty[k1] += v[k1];
                tmem_st16(at + 16, ty);
                tmem_ld16(at + 32, v);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) tn[k1] += v[k1];
                tmem_st16(at + 32, tn);
            }
        }
        if (acc_p) tmem_wait_st();
    }
    if (acc_p) {
#pragma unroll
        for (int i = 0; i < I; ++i) {
            const int w = t + i * kThreads;
            float nx[16], ny[16], dn[16];
            tmem_ld16(acc + 48 * i, nx);
            tmem_ld16(acc + 48 * i + 16, ny);
            tmem_ld16(acc + 48 * i + 32, dn);
            if (w < N) {
                const int line = w / M, x0 = w - line * M, y = n1b + M * line;
                const size_t pidx = ((size_t)k * N + y) * N + x0;
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) {
                    if (mode == BWD_GRAD)
                        red_add_v2(a.grad_probe + pidx + M * k1, nx[k1], ny[k1]);
                    else
                        red_add_v4(a.acc_probe + pidx + M * k1, nx[k1], ny[k1], dn[k1], 0.f);
                }
            }
            __syncwarp();
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(kBwdTmemCols) : "memory");
        }
    }
}

template <int N>
size_t smem_row_fwd_s() { return sizeof(float2) * (N + (size_t)Plan<N>::R * reg_pitch<N>()); }
template <int N>
size_t smem_row_bwd_s() {
    constexpr size_t stages = Plan<N>::M > Plan<N>::R ? 0 : Plan<N>::R * N + Plan<N>::M * kThreads;
    return sizeof(float2) * (N + stages + Plan<N>::R * reg_pitch<N>());
}

template <int N>
void launch_row_fwd_s(const ProbArgs& a, int j0, int nb, int mode, cudaStream_t s, bool pdl) {
    const dim3 grid(Plan<N>::M, nb * a.K);
    launch_dep(mode == X_DM ? k_row_fwd_s<N, true> : k_row_fwd_s<N, false>, grid, smem_row_fwd_s<N>(), s, pdl, a, j0);
}
template <int N>
void launch_col_s(const ProbArgs& a, int j0, int nb, int mode, cudaStream_t s, bool pdl) {
    const dim3 grid(N / reg_cols<N>(), nb);
    auto k = a.K > 1 ? (mode == COL_PROJECT && !a.bg ? k_col_modes_s<N, true> : k_col_modes_s<N, false>)
             : a.bg  ? (mode == COL_PROJECT ? k_col_s<N, true, true> : k_col_s<N, true, false>)
                     : (mode == COL_PROJECT ? k_col_s<N, false, true> : k_col_s<N, false, false>);
    launch_dep<SplitShape<N>::TC>(k, grid, 0, s, pdl, a, j0, mode);
}
// The cycle's form (Psi' and probe sums), the gradient of the object and of both
// parts have instantiations of their own (kForm 1, 2, 3), the rest takes its flags
// from the arguments (0).
template <int N, int kForm>
void launch_row_bwd_form(const ProbArgs& a, int j0, int nb, int G, int mode, int upd_obj, int upd_probe, cudaStream_t s,
                         bool pdl) {
    const dim3 grid(Plan<N>::M, G * a.K);
    if constexpr (Plan<N>::M > Plan<N>::R)
        launch_dep(k_row_bwd_s2<N, kForm>, grid, smem_row_bwd_s<N>(), s, pdl, a, j0, nb, mode, upd_obj, upd_probe);
    else
        launch_dep(k_row_bwd_s<N, kForm>, grid, smem_row_bwd_s<N>(), s, pdl, a, j0, nb, mode, upd_obj, upd_probe);
}
template <int N>
void launch_row_bwd_s(const ProbArgs& a, int j0, int nb, int G, int mode, int upd_obj, int upd_probe, cudaStream_t s,
                      bool pdl) {
    auto f = mode != BWD_GRAD ? (upd_probe ? &launch_row_bwd_form<N, 1> : &launch_row_bwd_form<N, 0>)
             : !upd_obj       ? &launch_row_bwd_form<N, 0>
                              : (upd_probe ? &launch_row_bwd_form<N, 3> : &launch_row_bwd_form<N, 2>);
    f(a, j0, nb, G, mode, upd_obj, upd_probe, s, pdl);
}

// Near field (pdl: as for the passes above) and line search.
template <int N>
void launch_col_nf_s(const ProbArgs& a, int nb, int dir, cudaStream_t s, bool pdl) {
    launch_dep<SplitShape<N>::TC>(dir < 0 ? k_col_nf_s<N, -1> : k_col_nf_s<N, +1>, dim3(N / reg_cols<N>(), nb), 0, s, pdl,
                                  a);
}
template <int N>
void launch_row_proj_s(const ProbArgs& a, int j0, int nb, int llk_only, cudaStream_t s, bool pdl) {
    launch_dep(!llk_only && !a.bg ? k_row_proj_s<N, true> : k_row_proj_s<N, false>, dim3(Plan<N>::M, nb), smem_row_fwd_s<N>(),
               s, pdl, a, j0, llk_only);
}
template <int N>
void launch_row_fwd_ls_s(const ProbArgs& a, int j0, int nb, int pdl, cudaStream_t s) {
    launch_dep(k_row_fwd_ls_s<N>, dim3(Plan<N>::M, nb, ls_waves(a.dir_obj, a.dir_probe) * a.K), smem_row_fwd_s<N>(), s,
               pdl != 0, a, j0);
}
template <int N>
void launch_col_ls_s(const ProbArgs& a, int j0, int nb, int pdl, cudaStream_t s) {
    const bool three = ls_waves(a.dir_obj, a.dir_probe) == 3;
    auto k = a.K == 1 ? (three ? k_col_ls_s<N, false, true> : k_col_ls_s<N, false, false>)
                      : (three ? k_col_ls_s<N, true, true> : k_col_ls_s<N, true, false>);
    launch_dep<SplitShape<N>::TC>(k, dim3(N / reg_cols<N>(), nb), 0, s, pdl != 0, a, j0);
}

template <class F>
cudaError_t split_attrs(F f) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}
template <int N>
cudaError_t set_attrs_split() {
    cudaError_t e;
    if constexpr (use_split_ls<N>())
        if ((e = split_attrs(k_row_fwd_ls_s<N>))) return e;
    if constexpr (use_split<N>()) {
        if ((e = split_attrs(k_row_fwd_s<N, false>))) return e;
        if ((e = split_attrs(k_row_fwd_s<N, true>))) return e;
        if constexpr (use_split_nf<N>()) {
            if ((e = split_attrs(k_row_proj_s<N, false>))) return e;
            if ((e = split_attrs(k_row_proj_s<N, true>))) return e;
        }
        if constexpr (Plan<N>::M > Plan<N>::R) {
            if ((e = split_attrs(k_row_bwd_s2<N, 0>))) return e;
            if ((e = split_attrs(k_row_bwd_s2<N, 1>))) return e;
            if ((e = split_attrs(k_row_bwd_s2<N, 3>))) return e;
            return split_attrs(k_row_bwd_s2<N, 2>);
        } else {
            if ((e = split_attrs(k_row_bwd_s<N, 0>))) return e;
            if ((e = split_attrs(k_row_bwd_s<N, 1>))) return e;
            if ((e = split_attrs(k_row_bwd_s<N, 3>))) return e;
            return split_attrs(k_row_bwd_s<N, 2>);
        }
    }
    return cudaSuccess;
}

}  // namespace ptx
