// fft_planes.cuh -- the x and y transforms of one z-plane of a real N x N x N volume, as the
// CG loop's operators use them (Toeplitz apply: rows and columns padded to L = 2N;
// preconditioner: L = N).
//
// A block takes a plane.  Two real rows make one complex transform (row a + i row b), so
// the plane costs N / 2 row transforms; the pair's outputs stay in shared memory as one
// spectrum of L points, and the two rows' half spectra (H = L / 2 + 1 columns) are
// separated as the column transform loads them.  The inverse goes the same way back:
// columns first, then two Hermitian rows as one complex transform.  Rows and columns go
// in the fewest batches that fit the exchange buffer beside the plane.  The kernels are
// bound by the latency of their phases, so a block has as many threads as a batch has
// items: splitting a plane over a cluster of 2 to 4 blocks (columns exchanged through
// distributed shared memory) measured no faster at any N (N = 64: 44.4 us a plain CG
// iteration against 40.3), half the threads slower (N = 128: 163 us a preconditioned
// iteration against 154).
#pragma once
#include <cuda_runtime.h>

#include "fft.cuh"
#include "pdl.cuh"

namespace firm {

// Sum of n partial sums by one warp, in a fixed order; valid in every lane.  The kernel that
// needs a reduction's result sums the blocks' partials itself (every block the same way):
// cheaper than a last-block pass at the end of the kernel that formed them (2 to 4 us).
__device__ __forceinline__ double partial_sum(const double* red, int n, int stride = 1) {
    double v = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) v += __ldcg(&red[i * stride]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int L, int N> struct PlaneCfg {
    static constexpr int L1 = Split<L>::L1, L2 = Split<L>::L2;
    static constexpr int H = L / 2 + 1, NP = N / 2;
    static constexpr int kBudget = 224 * 1024 / (int)sizeof(float2);
    static constexpr int kPlane = N * H;                                    // plane buffer (complex)
    static constexpr int kRowElems = L1 * (L2 + 1);
    static constexpr int rb0 = (kBudget - kPlane) / kRowElems < NP ? (kBudget - kPlane) / kRowElems : NP;
    static constexpr int RB = (NP + (NP + rb0 - 1) / rb0 - 1) / ((NP + rb0 - 1) / rb0);   // row pairs a batch
    static constexpr int cb0 = (kBudget - kPlane) / L < H ? (kBudget - kPlane) / L : H;
    static constexpr int CB = (H + (H + cb0 - 1) / cb0 - 1) / ((H + cb0 - 1) / cb0);      // columns a batch
    static constexpr int kX = smem_elems<L, false>(RB) > smem_elems<L, true>(CB) ? smem_elems<L, false>(RB)
                                                                                 : smem_elems<L, true>(CB);
    static constexpr size_t kSmem = sizeof(float2) * (kPlane + kX);
    static constexpr int kItems = (RB > CB ? RB : CB) * (L1 > L2 ? L1 : L2);
    static constexpr int kThreads = kItems < 1024 ? (kItems + 31) / 32 * 32 : 1024;
};

// Forward: row pairs (op.load(p, n) gives sample n of rows 2p and 2p + 1, op.post(p, n, v)
// runs after a pair's loads), then columns into out[k2][k1].  S: kSmem bytes.
template <int L, int N, class Op>
__device__ __forceinline__ void plane_forward(Op& op, float2* out, const float2* __restrict__ tw, float2* S) {
    using P = PlaneCfg<L, N>;
    constexpr int H = P::H, NP = P::NP, M = NP * H;
    float2* plane = S;                       // [pair][k1], k1 < H; then [pair][L - k1]
    float2* X = S + P::kPlane;
    for (int r0 = 0; r0 < NP; r0 += P::RB) {
        const int nl = min(P::RB, NP - r0);
        auto ld = [&](int line, int n) { return op.load(r0 + line, n); };
        auto post = [&](int line, int n, float2 v) { op.post(r0 + line, n, v); };
        auto st = [&](int line, int k, float2 v) { plane[(r0 + line) * H + (k < H ? k : M + L - k)] = v; };
        fft_step1_post<L, -1, false>(nl, ld, post, X, tw);
        __syncthreads();
        fft_step2<L, -1, false>(nl, st, X);
        __syncthreads();
    }
    for (int b0 = 0; b0 < H; b0 += P::CB) {
        const int nl = min(P::CB, H - b0);
        auto ld = [&](int line, int n) {
            if (n >= N) return make_float2(0.0f, 0.0f);
            const int k = b0 + line;
            const float2* a = plane + (n >> 1) * H + k;
            const float2 z = a[0];
            const float2 m = (k == 0 || k == L / 2) ? z : a[M];      // the spectrum at L - k
            return (n & 1) ? make_float2(0.5f * (z.y + m.y), -0.5f * (z.x - m.x))
                           : make_float2(0.5f * (z.x + m.x), 0.5f * (z.y - m.y));
        };
        auto st = [&](int line, int k, float2 v) { out[(size_t)k * H + b0 + line] = v; };
        block_fft<L, -1, true>(nl, ld, st, X, tw);
    }
}

// Inverse: columns of in[k2][k1], outputs y < N kept, then row pairs; op.pre(p, n) is
// fetched ahead of op.store(p, n, (row 2p, row 2p + 1), pre).
template <int L, int N, class Op>
__device__ __forceinline__ void plane_inverse(Op& op, const float2* in, const float2* __restrict__ tw,
                                              float2* S) {
    using P = PlaneCfg<L, N>;
    constexpr int H = P::H, NP = P::NP;
    float2* plane = S;                       // [y][k1]
    float2* X = S + P::kPlane;
    for (int b0 = 0; b0 < H; b0 += P::CB) {
        const int nl = min(P::CB, H - b0);
        auto ld = [&](int line, int n) { return in[(size_t)n * H + b0 + line]; };
        auto st = [&](int line, int k, float2 v) {
            if (k < N) plane[k * H + b0 + line] = v;
        };
        block_fft<L, +1, true>(nl, ld, st, X, tw);
    }
    for (int r0 = 0; r0 < NP; r0 += P::RB) {
        const int nl = min(P::RB, NP - r0);
        auto ld = [&](int line, int n) {
            const int k = n < H ? n : L - n;
            const float2* a = plane + 2 * (r0 + line) * H + k;
            float2 xa = a[0], xb = a[H];
            if (n == 0 || n == L / 2) xa.y = xb.y = 0.0f;      // real by symmetry
            return n < H ? make_float2(xa.x - xb.y, xa.y + xb.x) : make_float2(xa.x + xb.y, xb.x - xa.y);
        };
        auto pre = [&](int line, int n) { return op.pre(r0 + line, n); };
        auto st = [&](int line, int n, float2 v, decltype(op.pre(0, 0)) pv) { op.store(r0 + line, n, v, pv); };
        fft_step1<L, +1, false>(nl, ld, X, tw);
        __syncthreads();
        fft_step2_pre<L, +1, false>(nl, pre, st, X);
        __syncthreads();
    }
}

}  // namespace firm
