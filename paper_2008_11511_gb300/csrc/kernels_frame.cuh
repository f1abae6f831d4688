// The whole cycle of a small frame in one block (N <= 64, one mode, far field,
// no background): ObjProbe2Psi, both FFT directions with the projection and the
// LLK in between, Psi' and the probe sums, without the work stack.
//
// Bound: a frame of 64^2 is 32 KB and fits one block's shared memory, so the
// three passes' launches and their trips through L2 only add latency: a scan of
// 100 frames leaves one block per SM, whose time is its chain of loads,
// codelets and barriers.  N R threads hold one codelet each (8 pixels), every
// transpose is in place (a column's second factor rewrites exactly the rows it
// read) or within a warp.  Two blocks of 512 threads per SM at 64^2.  The cycles take
// it while every frame has a block of its own (100 frames of 64^2, five AP cycles,
// 180 -> 170 us), whose probe terms go straight to the accumulators; the LLK's blocks
// loop over more frames than that: 6000 frames 163 (three passes) -> 131 us.
#pragma once
#include "kernels_reg.cuh"

namespace ptx {

template <int N>
__host__ __device__ constexpr bool frame_whole() { return Plan<N>::M > 1 && RegShape<N>::L == N; }
template <int N>
__host__ __device__ constexpr int frame_threads() { return N * Plan<N>::R; }

enum FrameForm : int { FRAME_PHI = 0, FRAME_DM = 1, FRAME_LLK = 2 };

// The thread's pixels k = 0 .. M - 1 of a column (rows cn + R k of the detector), whose
// terms are in the rows of col: their LLK (returned) and, but for FRAME_LLK, the
// first factor of the inverse transform in u.
template <int N, int kForm, bool kBright>
__device__ __forceinline__ float project_frame(const float2* col, float2* u, const float* io, uint32_t mbits) {
    constexpr int M = Plan<N>::M, P = reg_pitch<N>();
    constexpr float invN2 = 1.0f / float(N * N);
#pragma unroll
    for (int i = 0; i < M; ++i) u[i] = col[i * P];
    Dft<M, -1>::run(u);
    float llk = 0.f;  // the terms are >= 0: a plain float sum of a thread's pixels
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const float ic = cnorm(u[i]) * invN2;
        const bool masked = (mbits >> i) & 1u;
        float ratio;
        const float term = llk_term_ratio<kBright>(ic, io[i], ratio);
        if (!masked) llk += term;
        if constexpr (kForm != FRAME_LLK) u[i] = cscale(u[i], masked ? 0.f : (ratio - 1.0f) * invN2);
    }
    if constexpr (kForm != FRAME_LLK) Dft<M, +1>::run(u);
    return llk;
}
template <int N>
__device__ __forceinline__ void frame_put(float2* col, const float2* u, const float2* tw, int cn) {
    constexpr int M = Plan<N>::M, P = reg_pitch<N>();
    col[0] = u[0];
#pragma unroll
    for (int i = 1; i < M; ++i) col[i * P] = cmul(u[i], tw_get<N, +1>(tw, cn, i));
}
// Both with the scaled quotients, for a thread whose sum is not finite in frame j.
template <int N, int kForm>
__device__ __noinline__ float frame_bright(const ProbArgs& a, int j) {
    constexpr int R = Plan<N>::R, M = Plan<N>::M, P = reg_pitch<N>();
    extern __shared__ __align__(16) float2 sm[];
    const int cn = threadIdx.x / N, c = threadIdx.x - cn * N;
    float2* col = sm + N + cn * M * P + c;
    float io[M];
    float2 u[M];
    uint32_t mbits = 0u;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        io[i] = a.iobs[((size_t)j * N + cn + R * i) * N + c];
        mbits |= (a.mask[(cn + R * i) * N + c] != 0) ? (1u << i) : 0u;
    }
    const float llk = project_frame<N, kForm, true>(col, u, io, mbits);
    if constexpr (kForm != FRAME_LLK) frame_put<N>(col, u, sm, cn);
    return llk;
}

// grid (blocks): block x handles frame x, FRAME_LLK also x + gridDim.x, ...
template <int N, int kForm>
__global__ void __launch_bounds__(frame_threads<N>(), N >= 64 ? 2 : 4)
    k_frame_r(const __grid_constant__ ProbArgs a, int upd_probe) {
    constexpr int R = Plan<N>::R, M = Plan<N>::M, P = reg_pitch<N>(), T = frame_threads<N>();
    constexpr bool kWarp = R == M && 32 % R == 0;  // a row's threads are in one warp in both factors
    extern __shared__ __align__(16) float2 sm[];
    __shared__ double red_s[T / 32];
    float2* tw = sm;
    float2* buf = sm + N;
    load_twiddles<N>(tw);
    const int t = threadIdx.x;
    // the thread's items: first factor of a row (lf, nf), second factor of a row (ls, ks),
    // either factor of a column (c, cn)
    const bool f = t < N * M;                    // first-factor items (all threads when R == M)
    const int lf = t / M, nf = t - lf * M;       // row lf, elements nf + M i
    const int ls = t / R, ks = t - ls * R;       // row ls, elements ks + R i
    const int cn = t / N, c = t - cn * N;        // column c, index cn of either factor
    auto sync_row = [] {
        if constexpr (kWarp)
            __syncwarp();
        else
            __syncthreads();
    };
    uint32_t mbits = 0u;  // rows cn + R i of column c
#pragma unroll
    for (int i = 0; i < M; ++i) mbits |= (a.mask[(cn + R * i) * N + c] != 0) ? (1u << i) : 0u;
    __syncthreads();
    for (int j = blockIdx.x; j < a.J; j += gridDim.x) {
        const int2 p = a.pos[j];
        const float2* obj = a.obj + (size_t)p.x * a.Wo + p.y;
        float2* psi = a.psi + (size_t)j * N * N;
        float io[M];
#pragma unroll
        for (int i = 0; i < M; ++i) io[i] = __ldcs(a.iobs + ((size_t)j * N + cn + R * i) * N + c);
        float2 v[R], u[M];
        // rows, first factor
        if (f) {
            float2 q[kForm == FRAME_DM ? R : 1];
            if constexpr (kForm == FRAME_DM) {
#pragma unroll
                for (int i = 0; i < R; ++i) q[i] = __ldcs(psi + lf * N + nf + M * i);
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                v[i] = cmul(__ldg(a.probe + lf * N + nf + M * i), obj[(size_t)lf * a.Wo + nf + M * i]);
            if constexpr (kForm == FRAME_DM) {
#pragma unroll
                for (int i = 0; i < R; ++i) v[i] = make_float2(2.f * v[i].x - q[i].x, 2.f * v[i].y - q[i].y);
            }
            Dft<R, -1>::run(v);
            float2* o = buf + lf * P + nf;
            o[0] = v[0];
#pragma unroll
            for (int i = 1; i < R; ++i) o[i * (M + 1)] = cmul(v[i], tw_get<N, -1>(tw, i, nf));
        }
        sync_row();
        // rows, second factor, back in natural order
#pragma unroll
        for (int i = 0; i < M; ++i) u[i] = buf[ls * P + ks * (M + 1) + i];
        Dft<M, -1>::run(u);
        sync_row();
#pragma unroll
        for (int i = 0; i < M; ++i) buf[ls * P + ks + R * i] = u[i];
        __syncthreads();
        // columns, first factor: rows cn + M i, rewritten as rows cn + M k
        if (f) {
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = buf[(cn + M * i) * P + c];
            Dft<R, -1>::run(v);
            buf[cn * P + c] = v[0];
#pragma unroll
            for (int i = 1; i < R; ++i) buf[(cn + M * i) * P + c] = cmul(v[i], tw_get<N, -1>(tw, i, cn));
        }
        __syncthreads();
        // columns, second factor: rows cn M + i hold the terms of ky = cn + R k; projection and LLK,
        // first factor of the inverse over k, into the rows just read
        float llk = project_frame<N, kForm, false>(buf + cn * M * P + c, u, io, mbits);
        if (!(llk < kInf))  // bright pixels without a model
            llk = frame_bright<N, kForm>(a, j);
        else if constexpr (kForm != FRAME_LLK)
            frame_put<N>(buf + cn * M * P + c, u, tw, cn);
        const double tot = block_sum_pos<T>(llk, red_s);  // also the barrier of the exchange
        if (t == 0) a.llk_part[j] = tot;
        if constexpr (kForm == FRAME_LLK) {
            __syncthreads();
            continue;
        } else {
            // columns, second factor of the inverse: rows M k + cn become rows cn + M k
            if (f) {
#pragma unroll
                for (int i = 0; i < R; ++i) v[i] = buf[(i * M + cn) * P + c];
                Dft<R, +1>::run(v);
#pragma unroll
                for (int i = 0; i < R; ++i) buf[(cn + M * i) * P + c] = v[i];
            }
            __syncthreads();
            // inverse rows
            if (f) {
#pragma unroll
                for (int i = 0; i < R; ++i) v[i] = buf[lf * P + nf + M * i];
            }
            sync_row();
            if (f) {
                Dft<R, +1>::run(v);
                float2* o = buf + lf * P + nf;
                o[0] = v[0];
#pragma unroll
                for (int i = 1; i < R; ++i) o[i * (M + 1)] = cmul(v[i], tw_get<N, +1>(tw, i, nf));
            }
            sync_row();
#pragma unroll
            for (int i = 0; i < M; ++i) u[i] = buf[ls * P + ks * (M + 1) + i];
            Dft<M, +1>::run(u);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const int x = ks + R * i;
                const float2 prv = __ldg(a.probe + ls * N + x), obv = obj[(size_t)ls * a.Wo + x];
                const float2 w = cadd(cmul(prv, obv), u[i]);
                __stcs(psi + ls * N + x, w);
                if (upd_probe) {
                    const float2 s = cconjmul(obv, w);
                    red_add_v4(a.acc_probe + ls * N + x, s.x, s.y, cnorm(obv), 0.f);
                }
            }
            return;
        }
    }
}

template <int N>
size_t smem_frame_r() { return sizeof(float2) * (N + (size_t)N * reg_pitch<N>()); }

// form: FrameForm; all frames of the problem (but for FRAME_LLK no more than frame_blocks(N))
template <int N>
void launch_frame(const ProbArgs& a, int form, int upd_probe, cudaStream_t s) {
    if constexpr (frame_whole<N>()) {
        const int grid = form != FRAME_LLK || a.J < frame_blocks(N) ? a.J : frame_blocks(N);
        auto k = form == FRAME_DM    ? k_frame_r<N, FRAME_DM>
                 : form == FRAME_LLK ? k_frame_r<N, FRAME_LLK>
                                     : k_frame_r<N, FRAME_PHI>;
        k<<<grid, frame_threads<N>(), smem_frame_r<N>(), s>>>(a, upd_probe);
    }
}
template <int N>
cudaError_t set_attrs_frame() {
    if constexpr (frame_whole<N>()) {
        cudaError_t e = cudaSuccess;
        for (auto k : {k_frame_r<N, FRAME_PHI>, k_frame_r<N, FRAME_DM>, k_frame_r<N, FRAME_LLK>}) {
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024))) return e;
            if ((e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared)))
                return e;
        }
    }
    return cudaSuccess;
}

}  // namespace ptx
