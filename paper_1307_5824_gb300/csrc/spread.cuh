// spread.cuh -- device helpers shared by the spreading and interpolation kernels
// (spread.cu, spread_mma.cu): point positions on the fine grid, window taps, the
// region of a brick and the kernels' arguments.
#pragma once
#include <cuda_runtime.h>

#include "firm_internal.h"

namespace firm {

// Position of sample k of an image along one axis of the fine grid, relative to the grid's
// centre, (G/N)(k1 u + k2 v) in units of 2^-23 cells rounded to nearest (6e-8 cells, below
// the FP32 rounding of the taps formed from it).  Integer arithmetic only: every kernel that
// calls this (binning, spreading, interpolation) gets identical cells.  ls = log2(G / N) <= 2;
// exact, since u = uh 2^16 + ul to the last bit.  In 32 bits (T = unsigned) the sum wraps at 512
// cells of the 4N grid (256 of the 2N grid): a multiple of the grid's period where G is a power
// of two, and on the other grids out of reach of every rotation; longer matrices there
// carry kGeomWide and take 64 bits.
constexpr int kFracBits = 23;
template <class T>
__device__ __forceinline__ T axis_pos(const ImgGeom& g, int d, int k1, int k2, int ls) {
    const T p = (T)k1 * (T)g.uh[d] + (T)k2 * (T)g.vh[d];
    const int q = k1 * (d == 0 ? g.ul[0] & 0xffff : g.ul[d]) + k2 * g.vl[d] + (1 << (17 - ls));
    return p + (T)(q >> 16);
}

// A cell I in [0, G) (periodic) and a fraction of q / 2^23 cells per axis.
struct PointPos {
    int I[3];
    uint32_t q[3];
    __device__ __forceinline__ float f(int d) const { return (float)q[d] * (1.0f / (float)(1 << kFracBits)); }
};

__device__ __forceinline__ PointPos point_pos(const ImgGeom& g, int32_t kk, int ls, int halfG, int G) {
    const int k1 = (int)(int16_t)(kk & 0xffff), k2 = kk >> 16;
    PointPos p;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int t = (int)axis_pos<unsigned>(g, d, k1, k2, ls) >> (2 - ls);
        p.I[d] = (t >> kFracBits) + halfG;
        p.q[d] = (uint32_t)t & ((1u << kFracBits) - 1u);
    }
    if (g.ul[0] & kGeomWide) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
            p.I[d] = (int)(axis_pos<long long>(g, d, k1, k2, ls) >> (2 - ls + kFracBits)) + halfG;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // |k1 u + k2 v| <= |k| <= N/2 (u, v: parts of a unit column of R) puts the cell in
        // [-1, G], and k_geom keeps longer ones within [-G, 2G): one wrap either way is the
        // periodic index
        if (p.I[d] >= G) p.I[d] -= G;
        else if (p.I[d] < 0) p.I[d] += G;
    }
    return p;
}

// ---------------------------------------------------------------------------
// Window taps and the region base of a point
// ---------------------------------------------------------------------------
template <int W>
__device__ __forceinline__ int tap_shift(float f) {
    // first tap offset u = c - (f - h) in [0, 1), h = 1/2 for odd W, 0 for even W
    constexpr float h = (W & 1) ? 0.5f : 0.0f;
    return (int)ceilf(f - h);
}

template <int W>
__device__ __forceinline__ void window_taps(const KbPoly& P, float f, float* w) {
    constexpr float h = (W & 1) ? 0.5f : 0.0f;
    const float t0 = f - h;
    const float z = 2.0f * (ceilf(t0) - t0) - 1.0f;
#pragma unroll
    for (int l = 0; l < W; ++l) {
        float acc = P.c[l][kKbDeg];
#pragma unroll
        for (int j = kKbDeg - 1; j >= 0; --j) acc = fmaf(acc, z, P.c[l][j]);
        w[l] = acc;
    }
}

// Dither of the kernel channel's fixed-point rounding: a value in [-1/2, 1/2) fixed by
// the point id (a 32-bit integer hash), added to every tap of the point before it is
// rounded to an integer.  Rounding to nearest drops every tap below half a unit, and
// the far taps of the window are that small: without the dither the kernel's sums come
// out biased low (~1e-6 relative, a smooth error that moves a 10-iteration CG volume by
// 1e-4 on the N=64 workload).  With it the rounding is unbiased, E[round(v + d)] = v
// for d uniform, and its error is white (a 1e-6 white error in Ker moves that volume by
// ~4e-7).
__device__ __forceinline__ float point_dither(uint32_t id) {
    uint32_t h = id * 2654435761u;
    h ^= h >> 15;
    h *= 2246822519u;
    h ^= h >> 13;
    return (float)(h >> 8) * (1.0f / 16777216.0f) - 0.5f;
}

// Rank (mod W) of this lane's point among the lanes of its warp with the same bank
// class (base mod 32; base < 0: no point).  Called by all 32 lanes.  Most warp steps of
// a round-robin piece hold 32 distinct classes: one OR-reduction of the class bits
// finds those, and only the others pay for the match.
template <int W>
__device__ __forceinline__ int class_rank(int base, int lane) {
    const bool pt = base >= 0;
    const unsigned bits = __reduce_or_sync(0xffffffffu, pt ? 1u << (base & 31) : 0u);
    const unsigned pts = __ballot_sync(0xffffffffu, pt);
    if (__popc(bits) == __popc(pts)) return 0;
    const unsigned same = __match_any_sync(0xffffffffu, pt ? (base & 31) : -1 - lane);
    const int r = __popc(same & ((1u << lane) - 1u));
    return r < W ? r : r % W;
}

// Bricks: 8 x 8 x BZ cells (BZ = kBrickZk for the kernel channel, 8 for A*b).
template <bool KC> struct Brick { static constexpr int BZ = KC ? kBrickZk : kBrick; };

// Index of the first tap of a point inside its brick's (8 + W) x (8 + W) x (BZ + W)
// region (x fastest), or -1 if the point is not inside the brick (never expected:
// binning uses the same code).
template <int W, int BZ>
__device__ __forceinline__ int region_base(const PointPos& p, int lo0, int lo1, int lo2) {
    constexpr int RG = kBrick + W;
    const int r0 = p.I[0] - lo0 + tap_shift<W>(p.f(0));
    const int r1 = p.I[1] - lo1 + tap_shift<W>(p.f(1));
    const int r2 = p.I[2] - lo2 + tap_shift<W>(p.f(2));
    if ((unsigned)r0 > (unsigned)kBrick || (unsigned)r1 > (unsigned)kBrick || (unsigned)r2 > (unsigned)BZ)
        return -1;
    return (r2 * RG + r1) * RG + r0;
}

struct SpreadArgs {
    const uint32_t* payload;
    const uint4* pts;         // tensor-core form: placed points (Workspace)
    const float2* pts_w;
    uint32_t* rec;            //   sorted records, their groups' classes, the items (Workspace)
    uint8_t* rec_cls;
    int4* rec_item;
    uint32_t rec_slots;
    int4* pass;
    const int4* work;
    int* counters;
    const ImgGeom* geom;
    const int32_t* htab;
    const int32_t* gid;
    const float* h2;          // kernel channel weights [group][t]
    const float2* samples_b;  // right-hand-side weights in scatter order
    const uint16_t* perm;     // per payload position: the point's index in scatter order
    double* grid;             // G^3 real, or G^3 complex interleaved (re, im)
    int G, halfG, nb, nH, n_ctf;
    int ls;                   // log2(G / N)
    int mma;                  // 1: binned for the tensor-core form (spread_mma.cu); in a batch 2: several passes
    float wmax_fixed;         // > 0: bound on |w| known in advance (no pre-pass)
    const float* wmax_item;   // fused form: per work item, the largest |h b| of its points
    KbPoly poly;
};

// Coordinate word of a placed point along one axis: first tap r (0..8, relative to the
// first cell of its brick that a tap can reach) << 28 | tap offset u = ceil(f - h) -
// (f - h) in [0, 1) with 23 bits << 5.  cell: cell within the brick, q: its fraction.
constexpr int kOffBits = 4, kUShift = 32 - kOffBits - kFracBits;
template <int W>
__device__ __forceinline__ uint32_t coord_word(int cell, uint32_t q) {
    constexpr uint32_t h = (W & 1) ? 1u << (kFracBits - 1) : 0u;
    const uint32_t up = q > h ? 1u : 0u;
    return ((uint32_t)cell + up) << (32 - kOffBits) | ((up << kFracBits) + h - q) << kUShift;
}

// Tensor-core form (spread_mma.cu); ch: 1 kernel channel, 2 A*b, 3 both.
cudaError_t launch_mma_passes(Plan& P);
cudaError_t launch_mma_sort(Plan& P, const SpreadArgs& a, int ch, int pass);
cudaError_t launch_spread_mma(Plan& P, const SpreadArgs& a, int ch);
cudaError_t launch_spread_mma_batch(int n, bool kc, int W, const SpreadArgs* desc, const int* item_off, int* queue,
                                    const KbPoly& poly, int num_sms, cudaStream_t s);

}  // namespace firm
