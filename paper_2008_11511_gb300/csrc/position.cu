// Position refinement (Psi2PosShift): per frame the first-order least-squares
// shift between the model exit wave Phi_j = P O[r_j] and the projected wave
// Psi_j left by the last AP / DM cycle.  With chi = Psi_j - Phi_j and
// G_a = P dO/da (a = y, x; central differences of the object, one-sided on its
// edges), the 2 x 2 normal equations
//   [<G_y,G_y> <G_y,G_x>; <G_x,G_y> <G_x,G_x>] d = [<G_y,chi>; <G_x,chi>],
// <u,v> = sum over modes and pixels of Re(conj(u) v), give d = (d_y, d_x).
// A frame whose gradient norm <G_y,G_y> + <G_x,G_x> is below filter_ratio
// times the mean over frames (or whose system is singular) keeps its position.
#include "kernels.cuh"

namespace ptx {

namespace {
constexpr int kPosRows = 16;  // rows each thread walks down
// pairs of adjacent columns, and rows of such pairs a block of 256 threads holds
__host__ __device__ inline int pos_groups(int N) { return 256 / (N / 2); }
}  // namespace

int pos_bands(int N) {
    const int rows = pos_groups(N) * kPosRows;
    return (N + rows - 1) / rows;
}

// grid (J, bands): a block sums the five products of its rows of frame j over
// all modes and writes them to part[(j * bands + band) * 5 + q] (FP64).
//
// Bound: the exit waves are read once from HBM, everything else comes from L2
// and L1.  A thread owns two adjacent columns and walks down kPosRows rows with
// the object rows y - 1, y, y + 1 of its columns in registers, so each object
// pixel is loaded for its own row only (and twice for the neighbours'
// columns), the probe and the exit wave by 16-byte loads, and no index is
// divided inside the loop.  With |G|^2 = |P|^2 |dO|^2 and Re(conj(P dO) chi) =
// Re(conj(dO) w), w = sum_k conj(P_k) chi_k, a mode costs two complex products and
// |P|^2 instead of three products and five sums.  (chi = Psi - P O comes first: in
// conj(P) Psi - |P|^2 O the rounding of two large products remains where Psi is
// near P O.)
// A thread's sums stay in FP32, with compensation (plain ones would be longer than
// the 8 N / 256 pixels that a thread added before), the block's are FP64.
// Sixteen rows per thread re-read 2 halo rows in 18 (8 rows: 2 in 10), and four
// blocks per SM leave the registers for four rows of loads in flight.
// 1000 frames of 256^2, all three launches: 1108 -> 215 us (before: every product
// from global memory, FP64 shuffles in every warp, one block for all the solves);
// 203 with plain sums of 16 pixels and the large products, at errors against 64 bits
// of 6.5 to 7.8e-7 over 64^2 to 512^2 instead of 5.4 to 6.5e-7, as before.
template <bool kOneMode>
__global__ void __launch_bounds__(256, kOneMode ? 4 : 3) k_pos_sums(ProbArgs a, double* part) {
    __shared__ float part_s[5][256];
    const int N = a.N, K = a.K;
    const int j = blockIdx.x, band = blockIdx.y;
    const int pairs = N / 2, groups = pos_groups(N);
    const int grp = threadIdx.x / pairs, x = 2 * (threadIdx.x - grp * pairs);
    const int y_first = (band * groups + grp) * kPosRows;
    KahanF s[5];  // yy, yx, xx, y.chi, x.chi
    if (grp < groups && y_first < N) {
        const int2 p = a.pos[j];
        const int c = p.y + x;                                       // object columns c, c + 1
        const int cl = c > 0 ? c - 1 : c, cr = c + 2 < a.Wo ? c + 2 : c + 1;  // their outer neighbours
        const float sx0 = c > 0 ? 0.5f : 1.0f, sx1 = c + 2 < a.Wo ? 0.5f : 1.0f;
        const int r = p.x + y_first;
        const float2* row = a.obj + (size_t)r * a.Wo;
        const float2* up = r > 0 ? row - a.Wo : row;
        float2 m0 = up[c], m1 = up[c + 1];                            // row y - 1 (clamped)
        float2 ol = row[cl], o0 = row[c], o1 = row[c + 1], oh = row[cr];  // row y
        const size_t f0 = (size_t)y_first * N + x;
        const float2* psi = a.psi + (size_t)j * K * N * N + f0;
        const float2* pr = a.probe + f0;
        const int rows = min(kPosRows, N - y_first);
#pragma unroll 4
        for (int i = 0; i < rows; ++i) {
            const bool last = r + i + 1 >= a.Ho, first = r + i == 0;
            const float2* down = last ? row : row + a.Wo;
            const float2 nl = down[cl], n0 = down[c], n1 = down[c + 1], nh = down[cr];
            const float sy = (last || first) ? 1.0f : 0.5f;
            float p0 = 0.f, p1 = 0.f;
            float2 w0 = make_float2(0.f, 0.f), w1 = w0;
#pragma unroll 1
            for (int k = 0; k < (kOneMode ? 1 : K); ++k) {
                const size_t o = (size_t)k * N * N + (size_t)i * N;
                const float4 q = __ldg(reinterpret_cast<const float4*>(pr + o));
                const float4 v = __ldcs(reinterpret_cast<const float4*>(psi + o));
                const float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
                const float2 chi0 = csub(make_float2(v.x, v.y), cmul(q0, o0));
                const float2 chi1 = csub(make_float2(v.z, v.w), cmul(q1, o1));
                p0 = fmaf(q.x, q.x, fmaf(q.y, q.y, p0));
                p1 = fmaf(q.z, q.z, fmaf(q.w, q.w, p1));
                w0 = cadd(w0, cconjmul(q0, chi0));
                w1 = cadd(w1, cconjmul(q1, chi1));
            }
            const float2 gy0 = cscale(csub(n0, m0), sy), gx0 = cscale(csub(o1, ol), sx0);
            const float2 gy1 = cscale(csub(n1, m1), sy), gx1 = cscale(csub(oh, o0), sx1);
            s[0].add(fmaf(p0, cnorm(gy0), p1 * cnorm(gy1)));
            s[1].add(fmaf(p0, fmaf(gy0.x, gx0.x, gy0.y * gx0.y), p1 * fmaf(gy1.x, gx1.x, gy1.y * gx1.y)));
            s[2].add(fmaf(p0, cnorm(gx0), p1 * cnorm(gx1)));
            s[3].add(fmaf(gy0.x, w0.x, fmaf(gy0.y, w0.y, fmaf(gy1.x, w1.x, gy1.y * w1.y))));
            s[4].add(fmaf(gx0.x, w0.x, fmaf(gx0.y, w0.y, fmaf(gx1.x, w1.x, gx1.y * w1.y))));
            m0 = o0; m1 = o1;
            ol = nl; o0 = n0; o1 = n1; oh = nh;
            row = down;
        }
    }
    // FP64 across the threads: warp q < 5 adds product q of all of them (one
    // FP64 addition per value; shuffling FP64 sums in every warp took 100 us
    // more at 1000 x 256^2, FP64 throughput being a few lanes per clock)
#pragma unroll
    for (int q = 0; q < 5; ++q) part_s[q][threadIdx.x] = s[q].s;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 5) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < 8; ++i) v += (double)part_s[warp][lane + 32 * i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) part[((size_t)j * gridDim.y + band) * 5 + warp] = v;
    }
}

// One warp per frame adds the frame's bands (in a fixed order) into the first
// band's five entries.  Apart from the solve so that the frames' bands are read
// by the whole GPU.
__global__ void __launch_bounds__(256) k_pos_frame(double* part, int J, int bands) {
    const int j = (int)((blockIdx.x * 256u + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (j >= J) return;
    double* f = part + (size_t)j * bands * 5;
    double m[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < bands; b += 32)
        for (int q = 0; q < 5; ++q) m[q] += f[b * 5 + q];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m[q] += __shfl_down_sync(0xffffffffu, m[q], o);
    }
    __syncwarp();
    if (lane == 0)
        for (int q = 0; q < 5; ++q) f[q] = m[q];
}

// Block b solves frames 256 b .. 256 b + 255.  Every block adds all the frames'
// norms itself, in the same order (the mean decides which frames are filtered):
// J doubles from L2 cost less than a launch in between, and the FP64 divisions of
// the solves, which one block alone would queue for 20 us at J = 1000, spread out.
__global__ void __launch_bounds__(256) k_pos_solve(const double* part, int J, int bands, float filter_ratio,
                                                    float* shifts) {
    __shared__ double red[32];
    double nsum = 0.0;
    for (int j = threadIdx.x; j < J; j += blockDim.x) {
        const double* m = part + (size_t)j * bands * 5;
        nsum += m[0] + m[2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nsum += __shfl_down_sync(0xffffffffu, nsum, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = nsum;
    __syncthreads();
    double total = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) total += red[w];
    const double mean = total / (double)J;
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j < J) {
        const double* m = part + (size_t)j * bands * 5;
        const double norm = m[0] + m[2];
        const double det = m[0] * m[2] - m[1] * m[1];
        float dy = 0.f, dx = 0.f;
        if (norm >= (double)filter_ratio * mean && det > 1e-12 * norm * norm) {
            dy = (float)((m[2] * m[3] - m[1] * m[4]) / det);
            dx = (float)((m[0] * m[4] - m[1] * m[3]) / det);
        }
        shifts[2 * j] = dy;
        shifts[2 * j + 1] = dx;
    }
}

void launch_position_shifts(const ProbArgs& a, double* part, float filter_ratio, float* shifts, cudaStream_t s) {
    const int bands = pos_bands(a.N);
    if (a.K == 1)
        k_pos_sums<true><<<dim3(a.J, bands), 256, 0, s>>>(a, part);
    else
        k_pos_sums<false><<<dim3(a.J, bands), 256, 0, s>>>(a, part);
    if (bands > 1) k_pos_frame<<<(a.J + 7) / 8, 256, 0, s>>>(part, a.J, bands);
    k_pos_solve<<<(a.J + 255) / 256, 256, 0, s>>>(part, a.J, bands, filter_ratio, shifts);
}

}  // namespace ptx
