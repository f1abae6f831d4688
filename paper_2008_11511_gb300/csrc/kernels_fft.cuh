// Plain orthonormal 2D FFT of frames in place (FT / IFT operators) with the
// register-resident line transforms of kernels_reg.cuh.
//
// Bound: each frame has to be read and written once in HBM (16 B per pixel).
//   * Frames that fit one block (N <= 64: 32 KB) are transformed whole in shared
//     memory: one pass.
//   * Larger frames take a row pass and a column pass over chunks small enough
//     that the column pass finds its input in L2 (kFftChunkBytes): the row pass
//     reads with evict-first (nothing else needs the old values) and writes with
//     evict-last, the column pass reads it back from L2 and streams it out.
// Both passes of a chunk are programmatic dependents of the launch before: a
// block loads its lines before it waits, the row pass because its chunk is not
// touched by any earlier launch of the call, the column pass nothing.
// 1024 frames of 256^2: 482 -> 312 us (3.4 TB/s of the 16 B per pixel; the start
// took both passes through shared memory in natural order, at HBM each).  Whole
// frames in a cluster of 8 or 16 blocks, the transpose through distributed shared
// memory, took 354 - 450 us: that exchange sustains 3.2 - 4.2 TB/s.
#pragma once
#include "kernels_split.cuh"

namespace ptx {

template <int N>
constexpr bool fft_split() { return use_split<N>() && Plan<N>::M > Plan<N>::R; }
template <int N>
constexpr bool fft_whole() { return Plan<N>::M > 1 && RegShape<N>::L == N; }

// grid (N / L, frames): rows [x L, x L + L) of a frame
template <int N, int DIR>
__global__ void __launch_bounds__(kThreads, RegShape<N>::MinBlocks) k_fft_rows_r(float2* data) {
    using S = RegShape<N>;
    constexpr int R = S::R, M = S::M, L = S::L, P = S::P;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    float2* base = data + ((size_t)blockIdx.y * N + (size_t)blockIdx.x * L) * N;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S::I1; ++i) {
        const int w = row_item<N, M>(i);
        if (w < L * M) {
            const int line = w / M, n1 = w - line * M;
            const float2* src = base + line * N + n1;
            const uint64_t ef = policy_evict_first();
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = ld_hint(src + M * n2, ef);
            Dft<R, DIR>::run(v);
            float2* o = buf + line * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, DIR>(tw, k2, n1));
        }
    }
    row_sync<N>();
    pdl_wait();
#pragma unroll
    for (int i = 0; i < S::I2; ++i) {
        const int w = row_item<N, R>(i);
        if (w < L * R) {
            const int line = w / R, k2 = w - line * R;
            const float2* src = buf + line * P + k2 * (M + 1);
            float2 u[M];
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) u[n1] = src[n1];
            Dft<M, DIR>::run(u);
            float2* dst = base + line * N + k2;
            const uint64_t el = policy_evict_last();
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) st_hint(dst + R * k1, u[k1], el);
        }
    }
}

// grid (N / C, frames): columns [x C, x C + C) of a frame, scaled by 1 / N
template <int N, int DIR>
__global__ void __launch_bounds__(kThreads, RegShape<N>::MinBlocks) k_fft_cols_r(float2* data) {
    using S = RegShape<N>;
    constexpr int R = S::R, M = S::M, C = S::C, P = S::P;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    float2* base = data + (size_t)blockIdx.y * N * N + (size_t)blockIdx.x * C;
    __syncthreads();
    pdl_wait();
    constexpr float invN = 1.0f / float(N);
#pragma unroll
    for (int i = 0; i < S::CI1; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < C * M) {
            const int n1 = w / C, c = w - n1 * C;
            const uint64_t ef = policy_evict_first();
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = ld_hint(base + (size_t)(n1 + M * n2) * N + c, ef);
            Dft<R, DIR>::run(v);
            float2* o = buf + c * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, DIR>(tw, k2, n1));
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S::CI2; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < C * R) {
            const int k2 = w / C, c = w - k2 * C;
            const float2* src = buf + c * P + k2 * (M + 1);
            float2 u[M];
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) u[n1] = src[n1];
            Dft<M, DIR>::run(u);
            const uint64_t ef = policy_evict_first();
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) st_hint(base + (size_t)(k2 + R * k1) * N + c, cscale(u[k1], invN), ef);
        }
    }
}

// The same with the column transform split between the passes (kernels_split.cuh),
// where the second factor is the larger one: the column pass then has no idle
// threads in its first factor and no transpose.  200 frames of 512^2 288 -> 260 us,
// 300 of 400^2 315 -> 278, 400 of 384^2 356 -> 313; at 256^2 305 against 309 for 1024
// frames but 16.5 against 14.7 for 40, so it keeps the passes above.  Rows n1 + M l of a frame: row transforms, then the
// first factor of the columns, back into the same rows (value k2 in row n1 + M k2).
// grid (M, frames)
template <int N, int DIR>
__global__ void __launch_bounds__(kThreads, SplitShape<N>::RowBlocks) k_fft_rows_s(float2* data) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    pdl_launch_dependents();
    load_twiddles<N>(tw);
    const int n1b = blockIdx.x;
    float2* base = data + (size_t)blockIdx.y * N * N;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S::I1; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < R * M) {
            const int line = w / M, n1 = w - line * M;
            const float2* src = base + (size_t)(n1b + M * line) * N + n1;
            const uint64_t ef = policy_evict_first();
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = ld_hint(src + M * n2, ef);
            Dft<R, DIR>::run(v);
            float2* o = buf + line * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, DIR>(tw, k2, n1));
        }
    }
    split_row_sync<N>();
    float2 u[S::I2][M];
#pragma unroll
    for (int i = 0; i < S::I2; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < R * R) {
            const int line = w / R, k2 = w - line * R;
            const float2* src = buf + line * P + k2 * (M + 1);
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) u[i][n1] = src[n1];
            Dft<M, DIR>::run(u[i]);
        }
    }
    split_row_sync<N>();
#pragma unroll
    for (int i = 0; i < S::I2; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < R * R) {
            const int line = w / R, k2 = w - line * R;
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) buf[line * P + k2 + R * k1] = u[i][k1];
        }
    }
    __syncthreads();
    pdl_wait();
#pragma unroll
    for (int i = 0; i < S::I1; ++i) {
        const int kx = threadIdx.x + i * kThreads;
        if (kx < N) {
            float2 v[R];
#pragma unroll
            for (int l = 0; l < R; ++l) v[l] = buf[l * P + kx];
            Dft<R, DIR>::run(v);
            const uint64_t el = policy_evict_last();
            st_hint(base + (size_t)n1b * N + kx, v[0], el);
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2)
                st_hint(base + (size_t)(n1b + M * k2) * N + kx, cmul(v[k2], tw_get<N, DIR>(tw, k2, n1b)), el);
        }
    }
}

// Columns [x C, x C + C) of a frame: thread (k2, c) finds its M values in rows
// n1 + M k2 and leaves the results in rows k2 + R k1, so the block, which owns its
// columns, reads all of them before it writes.  grid (N / C, frames)
template <int N, int DIR>
__global__ void __launch_bounds__(SplitShape<N>::TC, SplitShape<N>::ColBlocks) k_fft_cols_s(float2* data) {
    using S = SplitShape<N>;
    constexpr int R = S::R, M = S::M, C = reg_cols<N>();
    pdl_launch_dependents();
    const int k2 = threadIdx.x / C, c = threadIdx.x - k2 * C;
    float2* base = data + (size_t)blockIdx.y * N * N + (size_t)blockIdx.x * C + c;
    pdl_wait();
    const uint64_t ef = policy_evict_first();
    float2 u[M];
#pragma unroll
    for (int n1 = 0; n1 < M; ++n1) u[n1] = ld_hint(base + (size_t)(n1 + M * k2) * N, ef);
    Dft<M, DIR>::run(u);
    __syncthreads();
    constexpr float invN = 1.0f / float(N);
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) st_hint(base + (size_t)(k2 + R * k1) * N, cscale(u[k1], invN), ef);
}

// grid (frames): one whole frame per block
template <int N, int DIR>
__global__ void __launch_bounds__(kThreads, 4) k_fft_frame_r(float2* data) {
    using S = RegShape<N>;
    constexpr int R = S::R, M = S::M, P = S::P;
    constexpr int I1 = (N * M + kThreads - 1) / kThreads, I2 = (N * R + kThreads - 1) / kThreads;
    extern __shared__ __align__(16) float2 sm[];
    float2* tw = sm;
    float2* buf = sm + N;
    load_twiddles<N>(tw);
    float2* base = data + (size_t)blockIdx.x * N * N;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I1; ++i) {  // rows, first factor
        const int w = threadIdx.x + i * kThreads;
        if (w < N * M) {
            const int line = w / M, n1 = w - line * M;
            float2 v[R];
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[n2] = __ldcs(base + line * N + n1 + M * n2);
            Dft<R, DIR>::run(v);
            float2* o = buf + line * P + n1;
            o[0] = v[0];
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) o[k2 * (M + 1)] = cmul(v[k2], tw_get<N, DIR>(tw, k2, n1));
        }
    }
    __syncthreads();
    float2 u[I2][M];
#pragma unroll
    for (int i = 0; i < I2; ++i) {  // rows, second factor
        const int w = threadIdx.x + i * kThreads;
        if (w < N * R) {
            const int line = w / R, k2 = w - line * R;
            const float2* src = buf + line * P + k2 * (M + 1);
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) u[i][n1] = src[n1];
            Dft<M, DIR>::run(u[i]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I2; ++i) {  // back in natural order for the columns
        const int w = threadIdx.x + i * kThreads;
        if (w < N * R) {
            const int line = w / R, k2 = w - line * R;
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) buf[line * P + k2 + R * k1] = u[i][k1];
        }
    }
    __syncthreads();
    float2 v[I1][R];
#pragma unroll
    for (int i = 0; i < I1; ++i) {  // columns, first factor
        const int w = threadIdx.x + i * kThreads;
        if (w < N * M) {
            const int n1 = w / N, c = w - n1 * N;
#pragma unroll
            for (int n2 = 0; n2 < R; ++n2) v[i][n2] = buf[(n1 + M * n2) * P + c];
            Dft<R, DIR>::run(v[i]);
#pragma unroll
            for (int k2 = 1; k2 < R; ++k2) v[i][k2] = cmul(v[i][k2], tw_get<N, DIR>(tw, k2, n1));
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < I1; ++i) {
        const int w = threadIdx.x + i * kThreads;
        if (w < N * M) {
            const int n1 = w / N, c = w - n1 * N;
#pragma unroll
            for (int k2 = 0; k2 < R; ++k2) buf[(k2 * M + n1) * P + c] = v[i][k2];
        }
    }
    __syncthreads();
    constexpr float invN = 1.0f / float(N);
#pragma unroll
    for (int i = 0; i < I2; ++i) {  // columns, second factor
        const int w = threadIdx.x + i * kThreads;
        if (w < N * R) {
            const int k2 = w / N, c = w - k2 * N;
            float2 t[M];
#pragma unroll
            for (int n1 = 0; n1 < M; ++n1) t[n1] = buf[(k2 * M + n1) * P + c];
            Dft<M, DIR>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) __stcs(base + (k2 + R * k1) * N + c, cscale(t[k1], invN));
        }
    }
}

// Bytes of frames per chunk of the two-pass form.  Small chunks leave the last
// wave of each launch nearly empty (1024 frames of 256^2: 8 MB 665 us, 16 MB 352,
// 32 MB 317, 48 MB 315, 64 MB 311); larger ones fall out of the 129 MB L2.
constexpr size_t kFftChunkBytes = (size_t)64 << 20;

template <int N, int DIR>
void launch_fft2_r(float2* data, int nframes, cudaStream_t s) {
    using S = RegShape<N>;
    if constexpr (fft_whole<N>()) {
        k_fft_frame_r<N, DIR><<<nframes, kThreads, sizeof(float2) * (N + (size_t)N * S::P), s>>>(data);
    } else {
        const size_t per = (size_t)N * N * sizeof(float2);
        const int chunk = (int)(kFftChunkBytes / per);
        for (int f = 0; f < nframes; f += chunk) {
            const int n = nframes - f < chunk ? nframes - f : chunk;
            float2* d = data + (size_t)f * N * N;
            // the first launch of the call follows whatever the stream holds: plain
            if constexpr (fft_split<N>()) {
                launch_dep(k_fft_rows_s<N, DIR>, dim3(Plan<N>::M, n), smem_row_fwd_s<N>(), s, f > 0, d);
                launch_dep(k_fft_cols_s<N, DIR>, dim3(N / S::C, n), 0, s, true, d);
            } else {
                launch_dep(k_fft_rows_r<N, DIR>, dim3(N / S::L, n), sizeof(float2) * (N + (size_t)S::L * S::P), s, f > 0, d);
                launch_dep(k_fft_cols_r<N, DIR>, dim3(N / S::C, n), sizeof(float2) * (N + (size_t)S::C * S::P), s, true, d);
            }
        }
    }
}

template <int N, class F>
cudaError_t fft_attrs(F f) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}
template <int N>
cudaError_t set_attrs_fft() {
    cudaError_t e;
    if constexpr (fft_whole<N>()) {
        if ((e = fft_attrs<N>(k_fft_frame_r<N, -1>))) return e;
        return fft_attrs<N>(k_fft_frame_r<N, +1>);
    } else if constexpr (fft_split<N>()) {
        if ((e = fft_attrs<N>(k_fft_rows_s<N, -1>))) return e;
        return fft_attrs<N>(k_fft_rows_s<N, +1>);
    } else {
        if ((e = fft_attrs<N>(k_fft_rows_r<N, -1>))) return e;
        if ((e = fft_attrs<N>(k_fft_rows_r<N, +1>))) return e;
        if ((e = fft_attrs<N>(k_fft_cols_r<N, -1>))) return e;
        return fft_attrs<N>(k_fft_cols_r<N, +1>);
    }
}

}  // namespace ptx
