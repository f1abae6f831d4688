// Normalisation, denominator maxima and FP64 log-likelihood reductions
// (second half of Psi2ObjProbe and the LLK operator's final sum).
#include "kernels.cuh"

namespace ptx {

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// max D_O and max D_P over the accumulators (both >= 0, so their bit patterns
// order like unsigned integers).
// Object numerator and denominator gathered per object tile from the stored
// exit waves and the (already updated) probe:
//   N_O(r) = sum_j sum_k conj(P_k(r - r_j)) Psi'_jk(r - r_j),  D_O(r) = sum_j sum_k |P_k(r - r_j)|^2
// over the frames whose patch contains r, in ascending j.  Each pixel is
// owned by one thread, so the accumulator is written without atomics.
__global__ void __launch_bounds__(256) k_obj_gather(ProbArgs a, TileLists tl, int fuse_max) {
    constexpr int TW = kObjTileW, TH = kObjTileH;
    constexpr int RS = 256 / TW;          // rows covered by the block's threads at once
    constexpr int Q = TW * TH / 256;      // pixels per thread (at most): rows wy + RS q of column x
    const int Qr = TW * tl.th / 256;      // this tile height's
    const int t = blockIdx.x;
    const int tid = tl.tile_ids[t];
    const int ty = tid / tl.ntx, tx = tid - ty * tl.ntx;
    const int wy = threadIdx.x / TW;
    const int x = tx * TW + threadIdx.x % TW;
    const int N = a.N, K = a.K;
    float2 n[Q];
    float d[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        n[q] = make_float2(0.f, 0.f);
        d[q] = 0.f;
    }
    const int f0 = tl.tile_ptr[t], f1 = tl.tile_ptr[t + 1];
    const int y0 = ty * tl.th + wy;
    // F frames per step: all their loads are issued before any is used, so each
    // thread keeps up to 2 F Q loads in flight (the loop is latency-bound otherwise)
    constexpr int F = 4;
    for (int f = f0; f < f1; f += F) {
        float2 pr[F][Q], ps[F][Q];
        bool ok[F][Q];
        for (int k = 0; k < K; ++k) {
#pragma unroll
            for (int u = 0; u < F; ++u) {
                const int fi = f + u;
                const int j = fi < f1 ? tl.tile_frames[fi] : 0;
                const int2 p = a.pos[j];
                const int px = x - p.y;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int py = y0 + RS * q - p.x;
                    ok[u][q] = q < Qr && fi < f1 && px >= 0 && px < N && py >= 0 && py < N;
                    const size_t off = ok[u][q] ? ((size_t)k * N + py) * N + px : 0;
                    pr[u][q] = ok[u][q] ? __ldg(a.probe + off) : make_float2(0.f, 0.f);
                    ps[u][q] = ok[u][q] ? __ldcs(a.psi + (size_t)j * K * N * N + off) : make_float2(0.f, 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < F; ++u)
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float2 c = cconjmul(pr[u][q], ps[u][q]);
                    n[q].x += c.x;
                    n[q].y += c.y;
                    d[q] = fmaf(pr[u][q].x, pr[u][q].x, fmaf(pr[u][q].y, pr[u][q].y, d[q]));
                }
        }
    }
    float dmax = 0.f;
    if (x < a.Wo) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int y = y0 + RS * q;
            if (q < Qr && y < a.Ho) {
                a.acc_obj[(size_t)y * a.Wo + x] = make_float4(n[q].x, n[q].y, d[q], 0.f);
                dmax = fmaxf(dmax, d[q]);
            }
        }
    }
    // max D_O for the inertia term, when the normalisation follows directly
    // (D_O >= 0, so float bits order like unsigned integers; tiles met by no
    // frame keep D_O = 0)
    if (fuse_max) {
        dmax = warp_max(dmax);
        if ((threadIdx.x & 31) == 0 && dmax > 0.f) atomicMax(&a.maxbits[0], __float_as_uint(dmax));
    }
}

__global__ void k_den_max(ProbArgs a, int upd_obj, int upd_probe) {
    float mo = 0.f, mp = 0.f;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (upd_obj) {
        const size_t n = (size_t)a.Ho * a.Wo;
        for (size_t i = i0; i < n; i += stride) mo = fmaxf(mo, a.acc_obj[i].z);
    }
    if (upd_probe) {
        const size_t n = (size_t)a.N * a.N;
        for (size_t i = i0; i < n; i += stride) mp = fmaxf(mp, a.acc_probe[i].z);
    }
    mo = warp_max(mo);
    mp = warp_max(mp);
    if ((threadIdx.x & 31) == 0) {
        if (mo > 0.f) atomicMax(&a.maxbits[0], __float_as_uint(mo));
        if (mp > 0.f) atomicMax(&a.maxbits[1], __float_as_uint(mp));
    }
}

// O <- (N_O + d_O O) / (D_O + d_O), d_O = alpha_obj max D_O (unchanged where the
// denominator is 0); the same for each probe mode with D_P; accumulators cleared,
// and by the last block the maxima, which every block has read by then (a memset
// node per cycle for them took 5 us of a 30 us cycle).  A block takes its ticket
// once all its threads have read the maxima, before its first store: a fence
// behind the stores would wait for them (cycle of 100 x 64^2: 27.0 -> 28.8 us).  The
// first pixel's loads go out before that barrier.
__global__ void k_normalise(ProbArgs a, float alpha_obj, float alpha_probe, int upd_obj, int upd_probe) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t no = upd_obj ? (size_t)a.Ho * a.Wo : 0, np = upd_probe ? (size_t)a.K * a.N * a.N : 0;
    const float d_o = upd_obj ? alpha_obj * __uint_as_float(a.maxbits[0]) : 0.f;
    const float d_p = upd_probe ? alpha_probe * __uint_as_float(a.maxbits[1]) : 0.f;
    float4 v;
    float2 o;
    auto load = [&](const float4* acc, const float2* x, size_t i) {
        v = acc[i];
        o = x[i];
    };
    if (i0 < no) load(a.acc_obj, a.obj, i0);
    __syncthreads();
    unsigned ticket = 0;
    if (threadIdx.x == 0) {
        __threadfence();  // the block's reads of the maxima come before its ticket
        ticket = atomicAdd(&a.maxbits[2], 1u);
    }
    auto store = [&](float4* acc, float2* x, size_t i, float d) {
        const float den = v.z + d;
        if (den > 0.f) x[i] = make_float2((v.x + d * o.x) / den, (v.y + d * o.y) / den);
        acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    for (size_t i = i0; i < no;) {
        store(a.acc_obj, a.obj, i, d_o);
        i += stride;
        if (i < no) load(a.acc_obj, a.obj, i);
    }
    for (size_t i = i0; i < np; i += stride) {
        load(a.acc_probe, a.probe, i);
        store(a.acc_probe, a.probe, i, d_p);
    }
    if (threadIdx.x == 0 && ticket == gridDim.x - 1) {
        __threadfence();  // every block's reads come before these stores
        if (upd_obj) a.maxbits[0] = 0u;
        if (upd_probe) a.maxbits[1] = 0u;
        a.maxbits[2] = 0u;
    }
}

// The probe's max D_P and normalisation in one launch, for probes that one
// cluster of kProbeCtas blocks holds in registers (K N^2 <= kProbeMax pixels): each
// thread keeps its pixels' accumulators, the blocks' maxima meet through
// distributed shared memory.  A block may only touch another's shared memory once
// that block has started, which nothing but a cluster barrier says: every thread
// arrives at entry and waits just before the stores, with the loads of the
// accumulators in between.  Replaces k_den_max and k_normalise, two launches
// of 3 to 4 us that each wait for the one before (64^2: 4.0 us, 128^2: 6.5 us in
// one; at 256^2 eight blocks take 14 us, the two launches 9).
constexpr int kProbeCtas = 8, kProbeThreads = 512;
static_assert(kProbeMax == 4 * kProbeCtas * kProbeThreads, "four pixels per thread at most");
template <int Q>
__global__ void __cluster_dims__(kProbeCtas, 1, 1) __launch_bounds__(kProbeThreads)
    k_probe_norm(ProbArgs a, float alpha_probe) {
    __shared__ float red[kProbeThreads / 32];
    __shared__ float maxima[kProbeCtas];  // every block's, written by the others
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int n1 = a.N * a.N, n = a.K * n1;
    const int i0 = blockIdx.x * kProbeThreads + threadIdx.x;
    constexpr int kStep = kProbeCtas * kProbeThreads;
    float4 v[Q];
    float mx = 0.f;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int i = i0 + q * kStep;
        v[q] = i < n ? a.acc_probe[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < n1) mx = fmaxf(mx, v[q].z);  // D_P is the same for every mode
    }
    mx = warp_max(mx);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every block has started
    if (threadIdx.x < kProbeCtas) {
        float b = 0.f;
#pragma unroll
        for (int w = 0; w < kProbeThreads / 32; ++w) b = fmaxf(b, red[w]);
        const unsigned local = (unsigned)__cvta_generic_to_shared(&maxima[blockIdx.x]);
        unsigned remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(b) : "memory");
    }
    __syncwarp();
    // (after this barrier no block touches another's shared memory)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    float m = 0.f;
#pragma unroll
    for (int c = 0; c < kProbeCtas; ++c) m = fmaxf(m, maxima[c]);
    const float d = alpha_probe * m;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int i = i0 + q * kStep;
        if (i >= n) continue;
        const float den = v[q].z + d;
        if (den > 0.f) {
            const float2 o = a.probe[i];
            a.probe[i] = make_float2((v[q].x + d * o.x) / den, (v[q].y + d * o.y) / den);
        }
        a.acc_probe[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

void launch_probe_norm(const ProbArgs& a, float alpha_probe, cudaStream_t s) {
    const int q = (a.K * a.N * a.N + kProbeCtas * kProbeThreads - 1) / (kProbeCtas * kProbeThreads);
    if (q <= 1)
        k_probe_norm<1><<<kProbeCtas, kProbeThreads, 0, s>>>(a, alpha_probe);
    else
        k_probe_norm<4><<<kProbeCtas, kProbeThreads, 0, s>>>(a, alpha_probe);
}

__device__ double block_reduce_llk(const double* part, size_t n) {
    __shared__ double red[32];
    double s = 0.0;
    for (size_t i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x < 32) {
        r = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    return r;
}

// Sum over blocks: block b adds the contiguous chunk b of n values into l2[b]; the
// last block to finish adds l2[0 .. gridDim.x) in index order, so the result does
// not depend on the blocks' timing.  True in the last block (all threads), whose
// thread 0 has the sum in r; the caller resets the ticket.
__device__ bool sum_last_block(const double* part, size_t n, double* l2, unsigned* ticket, double& r) {
    __shared__ bool is_last;
    const size_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const size_t b0 = (size_t)blockIdx.x * chunk;
    const size_t nb = b0 < n ? (n - b0 < chunk ? n - b0 : chunk) : 0;
    const double s = block_reduce_llk(part + b0, nb);
    if (threadIdx.x == 0) {
        l2[blockIdx.x] = s;
        __threadfence();
        is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    r = block_reduce_llk(l2, gridDim.x);
    return true;
}

// The LLK of one call (1000 x 256^2: one block 11.4 us, 64 blocks 5.7).
__global__ void k_llk_sum(Ctl* ctl, ProbArgs a, int nparts_per_frame, double* out) {
    double r;
    if (!sum_last_block(a.llk_part, (size_t)a.J * nparts_per_frame, ctl->l2, &ctl->ticket, r)) return;
    if (threadIdx.x == 0) {
        *out = r;
        ctl->ticket = 0u;
    }
}

// The same in one block, for ptx_llk_static, which has no control block.
__global__ void k_llk_reduce(ProbArgs a, int nparts_per_frame, double* out) {
    double r = block_reduce_llk(a.llk_part, (size_t)a.J * nparts_per_frame);
    if (threadIdx.x == 0) *out = r;
}

// The cycle's LLK, entered at the control block's cycle.
__global__ void k_cycle_end(Ctl* ctl, ProbArgs a, int p, int nparts_per_frame, int last_problem) {
    double r;
    if (!sum_last_block(a.llk_part, (size_t)a.J * nparts_per_frame, ctl->l2, &ctl->ticket, r)) return;
    if (threadIdx.x == 0) {
        if (ctl->llk_out) ctl->llk_out[(size_t)ctl->cycle * ctl->nprob + p] = r;
        ctl->ticket = 0u;
        if (last_problem) ctl->cycle += 1;
    }
}

// Background update of an AP cycle: B <- B * (1/J) sum_j I_o / (I_c + B) on
// unmasked pixels, then the sums are cleared for the next cycle.
__global__ void k_bg_update(float* bg, float* acc, const uint8_t* mask, int n, float inv_j) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (!mask[i]) bg[i] *= acc[i] * inv_j;
        acc[i] = 0.f;
    }
}

// Self-test of the bounded-wait failure path: one thread waits for a
// shared-memory flag that nothing sets, at most limit_ns of the global timer
// (and at most 2^31 SM clocks), then records the give-up in err_flag as the
// tensor-copy waits do.  The wait always ends.
__global__ void k_wait_selftest(int* err_flag, unsigned long long limit_ns) {
    __shared__ volatile int never;
    never = 0;
    __syncthreads();
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    const long long c0 = clock64();
    while (!never) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > limit_ns || clock64() - c0 > (1ll << 31)) {
            if (err_flag) {
                *(volatile int*)err_flag = 1;
                __threadfence_system();
            }
            return;
        }
    }
}

// FP32 FMA throughput probe: every thread runs `iters` rounds of 16 independent
// FMA chains (32 flop per round), enough independent work per warp to keep the
// FMA pipes issuing every cycle.  The chains' sum goes to sink[thread] so that
// nothing is dropped by the compiler; a, b keep the values bounded.
__global__ void __launch_bounds__(256) k_fma_peak(float* __restrict__ sink, int iters, float a, float b) {
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = (float)(threadIdx.x + i) * 1e-3f;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = fmaf(x[i], a, b);
    }
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) t += x[i];
    sink[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = t;
}

// Photon counts (uint16) to the float32 intensities the passes read: 8 counts
// (16 bytes) per thread and step, exact (every uint16 is a float32 integer).
__global__ void k_counts_to_float(const uint16_t* __restrict__ src, float* __restrict__ dst, size_t n) {
    const size_t n8 = n / 8;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += stride) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(src) + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float4 lo, hi;
        lo.x = (float)(w[0] & 0xffffu); lo.y = (float)(w[0] >> 16);
        lo.z = (float)(w[1] & 0xffffu); lo.w = (float)(w[1] >> 16);
        hi.x = (float)(w[2] & 0xffffu); hi.y = (float)(w[2] >> 16);
        hi.z = (float)(w[3] & 0xffffu); hi.w = (float)(w[3] >> 16);
        float4* d = reinterpret_cast<float4*>(dst) + 2 * i;
        __stcs(d, lo);  // streaming stores: the intensities are read a cycle later,
        __stcs(d + 1, hi);  // they should not push the work stack out of L2
    }
    // the tail (n not a multiple of 8)
    for (size_t i = 8 * n8 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) dst[i] = (float)src[i];
}

// One-byte counts to float32: 16 counts (16 bytes) per thread and step.
__global__ void k_counts8_to_float(const uint8_t* __restrict__ src, float* __restrict__ dst, size_t n) {
    const size_t n16 = n / 16;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += stride) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(src) + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float4* d = reinterpret_cast<float4*>(dst) + 4 * i;
#pragma unroll
        for (int q = 0; q < 4; ++q)  // streaming stores, as in k_counts_to_float
            __stcs(d + q, make_float4((float)(w[q] & 0xffu), (float)((w[q] >> 8) & 0xffu),
                                      (float)((w[q] >> 16) & 0xffu), (float)(w[q] >> 24)));
    }
    // the tail (n not a multiple of 16)
    for (size_t i = 16 * n16 + (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) dst[i] = (float)src[i];
}

// The escapes of the one-byte form: dst[index[k]] = value[k] for the indices
// inside the n elements of dst (others are skipped).
__global__ void k_counts8_escapes(const uint32_t* __restrict__ index, const uint16_t* __restrict__ value,
                                  float* __restrict__ dst, size_t n_esc, size_t n) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_esc; k += stride) {
        const uint32_t i = index[k];
        if (i < n) dst[i] = (float)value[k];
    }
}

__global__ void k_set_ctl(Ctl* ctl, double* llk_out, int nprob) {
    ctl->llk_out = llk_out;
    ctl->cycle = 0;
    ctl->ticket = 0u;
    ctl->nprob = nprob;
    ctl->err = 0;
}

}  // namespace ptx

namespace ptx {

// A float as a double by its bits: the conversion instruction shares the FP64
// pipe (a few lanes per clock) with the products it feeds.  Exact for zero and
// normal values; others take the instruction.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
    if (e == 0x7f800000u || (e == 0u && (b << 1) != 0u)) return (double)x;
    const unsigned hi = (b & 0x80000000u) | (e == 0u ? 0u : ((b & 0x7fffffffu) >> 3) + 0x38000000u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// <G,G> and <G,Gp> over the object and probe parts into cg[0], cg[1]: FP64 sums
// per block into cg_part, added in index order by the last block (so the result
// does not depend on scheduling).  <Gp,Gp> is the <G,G> of the step that made Gp
// (cg[kCgPrev], 0 after a restart) and goes to cg[2].  kCgBlocks blocks of 256 threads.
// Bound: FP64 throughput.  1536^2 object: 68 us with conversions, three products and
// a launch of its own (6 us) for the blocks' sums, 45 us now.
__global__ void k_cg_dots(CgArgs c) {
    double gg = 0.0, ggp = 0.0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t tot = c.n_obj + c.n_probe;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += stride) {
        const bool o = i < c.n_obj;
        const size_t k = o ? i : i - c.n_obj;
        const float2 g = o ? c.g_obj[k] : c.g_probe[k];
        const float2 q = o ? c.gp_obj[k] : c.gp_probe[k];
        const double gx = widen(g.x), gy = widen(g.y);
        gg = fma(gx, gx, fma(gy, gy, gg));
        ggp = fma(gx, widen(q.x), fma(gy, widen(q.y), ggp));
    }
    __shared__ double red_s[2][256];
    __shared__ bool is_last;
    block_sum_pair<256>(gg, ggp, red_s, c.cg_part + 2 * blockIdx.x);
    __syncthreads();
    unsigned* ticket = reinterpret_cast<unsigned*>(c.cg + kCgTicket);
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double v0 = 0.0, v1 = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) {
        v0 += c.cg_part[2 * b];
        v1 += c.cg_part[2 * b + 1];
    }
    __syncthreads();
    block_sum_pair<256>(v0, v1, red_s, c.cg);
    __syncthreads();
    if (threadIdx.x == 0) {
        c.cg[2] = c.cg[kCgPrev];
        *ticket = 0u;
    }
}

// Polak-Ribiere: beta = max(0, (<G,G> - <G,Gp>) / <Gp,Gp>) (0 without a previous
// gradient); D <- -G + beta D; Gp <- G.
__global__ void k_cg_direction(CgArgs c) {
    const double den = c.cg[2];
    const double beta = den > 0.0 ? fmax(0.0, (c.cg[0] - c.cg[1]) / den) : 0.0;
    const float b = (float)beta;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t tot = c.n_obj + c.n_probe;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += stride) {
        const bool o = i < c.n_obj;
        const size_t k = o ? i : i - c.n_obj;
        float2* g = o ? c.g_obj + k : c.g_probe + k;
        float2* gp = o ? c.gp_obj + k : c.gp_probe + k;
        float2* d = o ? c.d_obj + k : c.d_probe + k;
        const float2 gv = *g;
        const float2 dv = *d;
        *d = make_float2(fmaf(b, dv.x, -gv.x), fmaf(b, dv.y, -gv.y));
        *gp = gv;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) c.cg[kCgPrev] = c.cg[0];  // <Gp,Gp> of the next step
}

// alpha = -L'(0) / L''(0) (0 when L''(0) <= 0); O += alpha D_O, P += alpha D_P.
__global__ void k_cg_step(CgArgs c, float2* obj, float2* probe) {
    const double l1 = c.cg[3], l2 = c.cg[4];
    const float alpha = l2 > 0.0 ? (float)(-l1 / l2) : 0.f;
    if (blockIdx.x == 0 && threadIdx.x == 0) c.cg[5] = l2 > 0.0 ? -l1 / l2 : 0.0;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t tot = c.n_obj + c.n_probe;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += stride) {
        const bool o = i < c.n_obj;
        const size_t k = o ? i : i - c.n_obj;
        float2* z = o ? obj + k : probe + k;
        const float2 d = o ? c.d_obj[k] : c.d_probe[k];
        const float2 v = *z;
        *z = make_float2(fmaf(alpha, d.x, v.x), fmaf(alpha, d.y, v.y));
    }
}

// Sum of the line-search partials (pairs) in a fixed order: out[0] = L'(0), out[1]
// = L''(0); per block of kLsBlocks into scratch, then by the last block (one block
// for 16000 pairs 15.4 us, kLsBlocks 6.5 us).
__global__ void k_ls_reduce(const double* part, size_t nparts, double* scratch, unsigned* ticket, double* out) {
    __shared__ double red_s[2][256];
    __shared__ bool is_last;
    const size_t chunk = (nparts + gridDim.x - 1) / gridDim.x;
    const size_t b0 = (size_t)blockIdx.x * chunk, b1 = b0 + chunk < nparts ? b0 + chunk : nparts;
    double v0 = 0.0, v1 = 0.0;
    for (size_t i = b0 + threadIdx.x; i < b1; i += 256) {
        const double2 v = reinterpret_cast<const double2*>(part)[i];
        v0 += v.x;
        v1 += v.y;
    }
    block_sum_pair<256>(v0, v1, red_s, scratch + 2 * blockIdx.x);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    v0 = v1 = 0.0;
    if (threadIdx.x < gridDim.x) {
        v0 = scratch[2 * threadIdx.x];
        v1 = scratch[2 * threadIdx.x + 1];
    }
    block_sum_pair<256>(v0, v1, red_s, out);
    if (threadIdx.x == 0) *ticket = 0u;
}

}  // namespace ptx
