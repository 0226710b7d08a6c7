// spread_mma.cu -- type-1 NUFFT spreading (FIRM steps 2-3, Section 3.4; eq. kernel and
// eq. backprojection) as small dense contractions on the tensor cores.
//
// The W^3 taps of a point are an outer product of its three axis windows, so the points
// whose first tap lies in the same cell class -- 3 consecutive cells per axis at W = 6,
// whose windows all fit one 8 x 8 x 8 block of the fine grid -- add up to
//     block[(y, x)][z] += sum_p (wy_p[y] wx_p[x]) (w_p wz_p[z]),
// a 64 x 8 product with the points as the contraction index.
//   1. k_mma_sort: a block per work item (points of one 8^3 brick) sorts the points into
//      their 27 classes in shared memory, pads every class to groups of 16 and writes a
//      record per point: its position within the class's cells along each axis and its
//      scaled weights.
//   2. k_spread_mma: a warp takes groups of 16 records and runs mma.m16n8k16; the (y, x)
//      operand and the weighted z operand are formed in registers, in the fragment
//      layout.  Every factor is an fp16 pair hi + lo (22 bits), a product keeps
//      hi hi + hi lo + lo hi.  The tensor core's FP32 additions truncate to half a unit in
//      the last place, so it adds the 16 points of a group only and the groups are added
//      by rounded FP32 adds (sums through the tensor core over 128 points came out 6e-7 of
//      their value too small, Ker's error against 64 bits 5.3e-7; 1.2e-7 this way, for 1% of
//      the time).  A warp's sums over at most 128 points go to the brick's (8 + W)^3 int32
//      region (native shared atomics; one rounding per sum instead of one per tap), which
//      is added into the FP64 grid when the item ends.
// Why: a tap per shared-memory atomic (spread.cu) is bound by the atomics' issue rate,
// 648 per point with both channels; here a point costs 2.5 mma (64 x 8 cells of which 216
// are hit, three products, padding) and ~30 warp instructions in all, of which the window
// arithmetic is 12 and the fragments 14; the fp16 tensor pipe of mma.sync (measured 961
// products per clock and SM) is a quarter busy.  mma.sync and not tcgen05, because both
// operands are made by the threads that use them, already in registers.
// Measured at N = 128, 50,000 images, W = 6 (3.2e8 points), binning and spreading together
// against the bank-class form (with its weight gather): both channels 50.8 -> 27.4 ms, of
// which the contraction takes 15.0, kernel channel 23.8 -> 17.0 ms, A*b 34.0 -> 18.6 ms.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "dw.cuh"
#include "firm_internal.h"
#include "pdl.cuh"
#include "spread.cuh"

namespace firm {

constexpr int kMmaThreads = 256;
constexpr int kMmaWarps = kMmaThreads / 32;
constexpr int kSortThreads = 512;
constexpr int kRunGroups = 8;                     // groups summed in FP32 before a class goes to the region
// fp16 operands carry each axis window scaled by 2^kTapBits; the weights' scale is chosen
// so that the products come out in the region's integer units.
constexpr int kTapBits = 5;
constexpr float kTapScale = (float)(1 << kTapBits);
constexpr int kUnitBias = 1024;                   // of the exponents in an item's last word

// CH: 1 kernel channel, 2 A*b, 3 both (Ker, Re, Im).
template <int W, int CH> struct MmaCfg {
    // First taps per class: y and z windows fit 8 cells; x windows 8 cells at W = 6 (3 first
    // taps, 27 classes) and 16 at W = 7 (all 9 first taps: 2 per class and axis would make
    // 125 classes, too few points in each on the 4N grid; this way there are 25).
    static constexpr int XS = W == 6 ? 8 : 16;                        // x cells of a class
    static constexpr int kBases = 9 - W, kBasesX = XS + 1 - W > 9 ? 9 : XS + 1 - W;
    static constexpr int kPer = (kBrick + 1 + kBases - 1) / kBases;   // classes along y and z
    static constexpr int kPerX = (kBrick + 1 + kBasesX - 1) / kBasesX;
    static constexpr int kClasses = kPer * kPer * kPerX;
    // Region, with planes padded so that 4 planes x 8 cells of a flush meet 32 banks
    static constexpr int RG = kBrick + W, PS = (RG * RG - 4 + 15) / 16 * 16 + 4, RG3 = PS * RG;
    static constexpr int T = XS == 8 ? 4 : 8;                         // 16-row tiles of (y, x)
    static constexpr int kSlots = (kMmaChunk + kClasses * 15 + 15) / 16 * 16;   // most slots of an item
    // A group's record: x, y, z coordinate words [16], then weights [pair 8][CH][hi, lo],
    // each word the fp16 parts of the pair's two points.
    static constexpr int kRecWords = 16 * (3 + CH);
    static constexpr size_t kSortSmem = sizeof(int) * (size_t)(kSlots / 16) * kRecWords;
    // Staging of one warp: windows of 4 groups along x (2 at 8 cells) and y, of 2 along z,
    // each axis hi | lo of 8 pairs per cell.  Strides are 8 mod 32 words, so that the four
    // groups a warp stores together meet different banks.
    static constexpr int kXG = XS == 8 ? 2 : 4;
    static constexpr int kXWords = 16 * XS + 8, kYWords = 136, kZWords = 136;
    static constexpr int kWarpWords = kXG * kXWords + 4 * kYWords + 2 * kZWords;
    // staging | record buffers [warp][2][4 groups] | region
    static constexpr size_t kSmem =
        sizeof(int) * ((size_t)kMmaWarps * (kWarpWords + 8 * kRecWords) + (size_t)CH * RG3);
    static_assert(kClasses <= 32, "one warp scans the class histogram");
    static_assert(kClasses * 15 <= kMmaPad - 15, "record slots");
};

// Window polynomials of taps 0 .. (W - 1) / 2, scaled by kTapScale, every coefficient twice
// (two points' worth): kernel parameters, so that they are operands from constant memory.
struct MmaPoly {
    float2 c[(kMaxW + 1) / 2][kKbDeg + 1];
};

static MmaPoly mma_poly(const KbPoly& P, int W) {
    MmaPoly q{};
    for (int l = 0; l < (W + 1) / 2; ++l)
        for (int j = 0; j <= kKbDeg; ++j) q.c[l][j] = make_float2(P.c[l][j] * kTapScale, P.c[l][j] * kTapScale);
    return q;
}

__device__ __forceinline__ uint32_t h2u(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }
__device__ __forceinline__ __half2 u2h(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }

// (x, y) = hi + lo, hi and lo fp16 pairs: 22 bits, absolute floor 2^-25.  (Splitting FP32 factors for
// the tensor cores, and adding their sums outside them because they truncate: Ootomo & Yokota,
// "Recovering single precision accuracy from Tensor Cores while surpassing the FP32
// theoretical peak performance", 2022.)
__device__ __forceinline__ void split2(float2 v, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __float22half2_rn(v);
    const float2 f = __half22float2(h);
    hi = h2u(h);
    lo = h2u(__float22half2_rn(make_float2(v.x - f.x, v.y - f.y)));
}

// Product of two hi + lo pairs as hi + lo: the fp16 product, its exact error by FMA, and
// the cross terms (lo lo, 2^-22 of the product, dropped).
__device__ __forceinline__ void mul_split(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl, uint32_t& ph,
                                          uint32_t& pl) {
    const __half2 p = __hmul2(u2h(ah), u2h(bh));
    __half2 e = __hfma2(u2h(ah), u2h(bh), __hneg2(p));
    e = __hfma2(u2h(ah), u2h(bl), e);
    e = __hfma2(u2h(al), u2h(bh), e);
    ph = h2u(p);
    pl = h2u(e);
}

__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Window taps of two points along one axis, scaled by kTapScale, in the S slots of their
// class's cells: slot off + l holds tap l (off < BASES may differ between the points),
// the others 0.  c: the points' coordinate words.  hi[s], lo[s]: the two points' values
// as fp16 pairs.  Taps l and W - 1 - l are one polynomial at z and -z: even and odd parts
// are shared.
template <int W, int BASES, int S>
__device__ __forceinline__ void slot_taps(const MmaPoly& poly, uint2 c, uint32_t* hi, uint32_t* lo) {
    const int off0 = (int)(c.x >> (32 - kOffBits)), off1 = (int)(c.y >> (32 - kOffBits));
    // z = 2u - 1 from the 28-bit offset u: (u - 1/2) as a signed 32-bit fraction
    const float2 z = make_float2((float)(int)((c.x << kOffBits) ^ 0x80000000u) * (1.0f / 2147483648.0f),
                                 (float)(int)((c.y << kOffBits) ^ 0x80000000u) * (1.0f / 2147483648.0f));
    const float2 nz = make_float2(-z.x, -z.y);
    const float2 z2 = __fmul2_rn(z, z);
#pragma unroll
    for (int l = 0; l < (W + 1) / 2; ++l) {
        const float2* p = poly.c[l];
        const float2 ev = __ffma2_rn(__ffma2_rn(__ffma2_rn(p[6], z2, p[4]), z2, p[2]), z2, p[0]);
        const float2 od = __ffma2_rn(__ffma2_rn(__ffma2_rn(p[7], z2, p[5]), z2, p[3]), z2, p[1]);
        split2(__ffma2_rn(od, z, ev), hi[l], lo[l]);
        if (W - 1 - l != l) split2(__ffma2_rn(od, nz, ev), hi[W - 1 - l], lo[W - 1 - l]);
    }
#pragma unroll
    for (int s = W; s < S; ++s) { hi[s] = 0u; lo[s] = 0u; }
    // shift by `n` slots in each point's half where its condition holds; `top`: last tap's slot
    auto shift = [&](bool c0, bool c1, int n, int top) {
        const uint32_t sel = (c0 ? 0x0054u : 0x0010u) | (c1 ? 0x7600u : 0x3200u);
#pragma unroll
        for (int s = S - 1; s >= 0; --s) {
            if (s > top) continue;
            hi[s] = __byte_perm(hi[s], s >= n ? hi[s - n] : 0u, sel);
            lo[s] = __byte_perm(lo[s], s >= n ? lo[s - n] : 0u, sel);
        }
    };
    if (BASES <= 3) {
#pragma unroll
        for (int st = 1; st < BASES; ++st) shift(off0 >= st, off1 >= st, 1, W - 1 + st);
    } else {                                       // 0..8, by its bits (8 alone has bit 3)
        shift(off0 & 1, off1 & 1, 1, W);
        shift(off0 & 2, off1 & 2, 2, W + 2);
        shift(off0 & 4, off1 & 4, 4, W + 6);
        shift(off0 & 8, off1 & 8, 8, W + 7);
    }
}

// ---------------------------------------------------------------------------
// Sort
// ---------------------------------------------------------------------------
template <int W, int CH>
__global__ void __launch_bounds__(kSortThreads, 2) k_mma_sort(const SpreadArgs a, int pass) {
    pdl_wait();
    pdl_launch();
    using C = MmaCfg<W, CH>;
    constexpr int BASES = C::kBases, BX = C::kBasesX, RW = C::kRecWords, PT = kMmaChunk / kSortThreads;
    constexpr int kWarps = kSortThreads / 32;
    extern __shared__ __align__(16) uint32_t s_rec[];
    __shared__ int s_hist[32], s_off[32], s_total, s_item, s_base;
    __shared__ float2 s_red[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int4* const ps = a.pass + pass;
    const int first = ps[0].x, n_work = ps[1].x;
    const float* const im2 = reinterpret_cast<const float*>(a.pts_w);      // A*b alone: imaginary parts
    if (tid == 0) s_item = first + atomicAdd(&ps->y, 1);
    __syncthreads();
    int item = s_item;
    int4 wk = make_int4(0, 0, 0, 0);
    uint4 pt[PT];
    // an item's points are loaded while the block writes out the item before it
    auto fetch = [&]() {
        if (item >= n_work) return;
        wk = a.work[item];
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            const int i = u * kSortThreads + tid;
            if (i < wk.z) pt[u] = a.pts[wk.y + i];
        }
    };
    fetch();
    while (item < n_work) {
        if (tid < 32) s_hist[tid] = 0;
        __syncthreads();
        // rank of the points in their class (arbitrary order); largest |h b|
        int cr[PT];                                // class | rank << 8
        float wmax = 0.0f, wsum = 0.0f;
        if (CH >= 2) {
#pragma unroll
            for (int u = 0; u < PT; ++u) {
                const int i = u * kSortThreads + tid;
                if (i >= wk.z) continue;
                const float2 v = CH == 3 ? a.pts_w[wk.y + i]
                                         : make_float2(__uint_as_float(pt[u].w), im2[wk.y + i]);
                const float w = fmaxf(fabsf(v.x), fabsf(v.y));
                wmax = fmaxf(wmax, w);
                wsum += w;
            }
        }
        bool in = true;
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            if (u * kSortThreads + tid >= wk.z) continue;
            const uint32_t r[3] = {pt[u].x >> 28, pt[u].y >> 28, pt[u].z >> 28};
            in = in && r[0] <= (uint32_t)kBrick && r[1] <= (uint32_t)kBrick && r[2] <= (uint32_t)kBrick;
            const uint32_t k[3] = {min(r[0], (uint32_t)kBrick) / BX, min(r[1], (uint32_t)kBrick) / BASES,
                                   min(r[2], (uint32_t)kBrick) / BASES};
            cr[u] = (int)((k[2] * C::kPer + k[1]) * C::kPerX + k[0]);
            // the first tap's slot within the class's cells takes the place of r
            pt[u].x -= (k[0] * BX) << 28;
            pt[u].y -= (k[1] * BASES) << 28;
            pt[u].z -= (k[2] * BASES) << 28;
            cr[u] |= atomicAdd(&s_hist[cr[u]], 1) << 8;
        }
        if (!in) atomicOr(&a.counters[2], kFlagPoint);      // a point outside its brick: never expected, reported
        if (CH >= 2) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
                wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
            }
            if (lane == 0) s_red[warp] = make_float2(wmax, wsum);
        }
        __syncthreads();
        if (warp == 0) {
            const int pad = (s_hist[lane] + 15) & ~15;
            int v = pad;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            s_off[lane] = v - pad;
            if (lane == 31) {
                s_total = v;
                s_base = atomicAdd(&ps->z, v / 16);
            }
        }
        __syncthreads();
        if (tid == 0) s_item = first + atomicAdd(&ps->y, 1);               // the next item
        if (CH >= 2) {
            wmax = s_red[0].x;
            wsum = s_red[0].y;
#pragma unroll
            for (int i = 1; i < kWarps; ++i) {
                wmax = fmaxf(wmax, s_red[i].x);
                wsum += s_red[i].y;
            }
        }
        // the region's units 2^ek and 2^eb: a cell's sum (taps <= 1) stays within 2^30 of them,
        // bounded by n points of weight wmax, for A*b by the sum of its |weights| where that is
        // less (a third of n wmax as a rule); 2^-25 wmax at least keeps the scaled weights within fp16
        // (fmaxf passes over a NaN, the sum keeps it)
        if (CH >= 2 && tid == 0 && (wsum != wsum || isinf(wmax))) atomicOr(&a.counters[2], kFlagInput);
        const int lgn = max(32 - __clz(max(wk.z - 1, 1)), 5);
        int ek = 0, eb = 0, es = 1 << 20;
        if (CH != 2 && a.wmax_fixed > 0.0f) frexpf(a.wmax_fixed, &ek);
        if (CH >= 2 && wmax > 0.0f) frexpf(wmax, &eb);
        if (CH >= 2 && wsum < 3e38f) frexpf(wsum, &es);
        ek = max(ek, -112) + lgn - 30;             // the scales stay within FP32
        eb = max(eb, -112) + min(lgn, max(es - eb, 5)) - 30;
        const float Sk = ldexpf(1.0f, -3 * kTapBits - ek), Sb = ldexpf(1.0f, -3 * kTapBits - eb);
        auto put = [&](int pos, uint32_t c0, uint32_t c1, uint32_t c2, const float* w) {
            uint32_t* r = s_rec + (pos >> 4) * RW + (pos & 15);
            r[0] = c0;
            r[16] = c1;
            r[32] = c2;
            __half* h = reinterpret_cast<__half*>(s_rec + (pos >> 4) * RW + 48 + ((pos >> 1) & 7) * 2 * CH) + (pos & 1);
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                const __half hi = __float2half_rn(w[ch]);
                h[4 * ch] = hi;
                h[4 * ch + 2] = __float2half_rn(w[ch] - __half2float(hi));
            }
        };
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            const int i = u * kSortThreads + tid;
            if (i >= wk.z) continue;
            float w[CH];
            const float w0 = __uint_as_float(pt[u].w);
            if (CH == 2) {
                w[0] = w0 * Sb;
                w[CH - 1] = im2[wk.y + i] * Sb;
            } else {
                w[0] = w0 * Sk;
            }
            if (CH == 3) {
                const float2 v = a.pts_w[wk.y + i];
                w[CH - 2] = v.x * Sb;
                w[CH - 1] = v.y * Sb;
            }
            put(s_off[cr[u] & 255] + (cr[u] >> 8), pt[u].x, pt[u].y, pt[u].z, w);
        }
        const int total = s_total;
        const bool fits = (long long)s_base * 16 + total <= (long long)a.rec_slots;
        {   // sixteen threads per class: its padding slots (weight 0) and its groups' class
            const int k = tid >> 4, h = s_hist[k], off = s_off[k], end = (h + 15) & ~15;
            const float zero[CH] = {};
            if (h + (tid & 15) < end) put(off + h + (tid & 15), 0u, 0u, 0u, zero);
            if (fits)
                for (int g = tid & 15; g < end / 16; g += 16) a.rec_cls[s_base + off / 16 + g] = (uint8_t)k;
        }
        const int base = s_base;
        if (tid == 0) {
            if (!fits) atomicOr(&a.counters[2], kFlagPoint);
            a.rec_item[item] = make_int4(wk.x, base, fits ? total / 16 : 0, (ek + kUnitBias) | (eb + kUnitBias) << 16);
        }
        __syncthreads();
        item = s_item;
        fetch();
        if (fits) {
            uint4* out = reinterpret_cast<uint4*>(a.rec + (size_t)base * RW);
            const uint4* in4 = reinterpret_cast<const uint4*>(s_rec);
            for (int i = tid; i < total / 16 * (RW / 4); i += kSortThreads) out[i] = in4[i];
        }
    }
}

// ---------------------------------------------------------------------------
// Spread
// ---------------------------------------------------------------------------
// A class's sums into the brick's region (one rounding to the region's unit per cell).
template <int W, int CH>
__device__ __forceinline__ void flush_class(const float2 (&D)[MmaCfg<W, CH>::T][CH][2], int cls, int* lev1, int row, int c) {
    using C = MmaCfg<W, CH>;
    constexpr int RG = C::RG, PS = C::PS, RG3 = C::RG3, PER = C::kPer, PERX = C::kPerX;
    const int z0 = cls / (PER * PERX) * C::kBases, y0 = cls / PERX % PER * C::kBases, x0 = cls % PERX * C::kBasesX;
    int* dst = lev1 + (z0 + 2 * c) * PS + y0 * RG + x0 + row;
    if (C::XS == 8) {                              // rows: 8 x of y = 2t, 8 x of y = 2t + 1
#pragma unroll
        for (int t = 0; t < C::T; ++t)
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                int* d = dst + ch * RG3 + 2 * t * RG;
                atomicAdd(d, __float2int_rn(D[t][ch][0].x));
                atomicAdd(d + PS, __float2int_rn(D[t][ch][0].y));
                atomicAdd(d + RG, __float2int_rn(D[t][ch][1].x));
                atomicAdd(d + PS + RG, __float2int_rn(D[t][ch][1].y));
            }
    } else {                                       // rows: 16 x of y = t
        // a class with fewer than kBases first taps, and x cell 15, reach past the region
        // with sums that are zero
        const bool z1 = z0 + 2 * c + 1 < RG, x1 = row < RG - 8;
#pragma unroll
        for (int t = 0; t < C::T; ++t) {
            if (y0 + t >= RG) break;
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                int* d = dst + ch * RG3 + t * RG;
                atomicAdd(d, __float2int_rn(D[t][ch][0].x));
                if (z1) atomicAdd(d + PS, __float2int_rn(D[t][ch][0].y));
                if (x1) atomicAdd(d + 8, __float2int_rn(D[t][ch][1].x));
                if (x1 && z1) atomicAdd(d + PS + 8, __float2int_rn(D[t][ch][1].y));
            }
        }
    }
}

// `n` 16-byte chunks of records from global to shared memory, asynchronously.
__device__ __forceinline__ void copy_async(uint32_t* dst, const uint32_t* src, int n, int lane) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (int i = lane; i < n; i += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * i), "l"(src + 4 * i) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// One work item.  lev1 is zero on entry and on return; called by the whole block.
template <int W, int CH>
__device__ __forceinline__ void spread_item_mma(const SpreadArgs& a, const MmaPoly& poly, const int4 wk, int* lev1,
                                                uint32_t* wbuf) {
    using C = MmaCfg<W, CH>;
    constexpr int RG = C::RG, RG3 = C::RG3, BASES = C::kBases, RW = C::kRecWords, XS = C::XS, T = C::T;
    constexpr int XO = XS * 8;                     // hi -> lo distance of the x windows
    __shared__ uint8_t s_cls[C::kSlots / 16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_groups = wk.z;
    for (int i = tid; i < n_groups; i += kMmaThreads) s_cls[i] = a.rec_cls[wk.y + i];
    // every warp takes a run of consecutive groups, in its own buffers
    const int per = (n_groups + kMmaWarps - 1) / kMmaWarps;
    const int ga = min(n_groups, warp * per), gb = min(n_groups, ga + per);
    uint32_t* const xs = wbuf;
    uint32_t* const ys = xs + C::kXG * C::kXWords;
    uint32_t* const zs = ys + 4 * C::kYWords;
    uint32_t* const in = wbuf + C::kWarpWords;
    const uint32_t* const rec = a.rec + (size_t)wk.y * RW;
    copy_async(in, rec + (size_t)ga * RW, min(4, gb - ga) * (RW / 4), lane);
    __syncthreads();
    const int row = lane >> 2, c = lane & 3, sx = row & 4;
    int g = ga;
#pragma unroll 1
    while (g < gb) {
        const int cls = s_cls[g];
        int ge = g + 1;                            // end of this class's run
        while (ge < gb && ge < g + kRunGroups && s_cls[ge] == cls) ++ge;
        float2 D[T][CH][2];
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) D[t][ch][0] = D[t][ch][1] = make_float2(0.0f, 0.0f);
#pragma unroll 1
        for (; g < ge; ++g) {
            const int r = g - ga, gi = r & 1;
            const uint32_t* const cur = in + ((r >> 2) & 1) * 4 * RW;
            if (gi == 0) {                         // stage the windows of the next groups
                __syncwarp();
                if ((r & 2) == 0) {
                    copy_async(in + (((r >> 2) & 1) ^ 1) * 4 * RW, rec + (size_t)(g + 4) * RW,
                               max(0, min(4, gb - g - 4)) * (RW / 4), lane);
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    __syncwarp();
                    // y windows of 4 groups, a pair of points per lane: [pair][slot], halves of
                    // four slots swapped for pairs 4-7 (16-byte accesses)
                    const int pr = lane & 7, sw = pr >> 2;
                    if (lane < 8 * (gb - g)) {
                        uint32_t hi[8], lo[8];
                        slot_taps<W, BASES, 8>(
                            poly, *reinterpret_cast<const uint2*>(cur + (lane >> 3) * RW + 16 + 2 * pr), hi, lo);
                        uint4* y = reinterpret_cast<uint4*>(ys + (lane >> 3) * C::kYWords + pr * 8);
                        y[sw] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        y[sw ^ 1] = make_uint4(hi[4], hi[5], hi[6], hi[7]);
                        y[16 + sw] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        y[16 + (sw ^ 1)] = make_uint4(lo[4], lo[5], lo[6], lo[7]);
                        if (XS == 16) {            // x windows of 4 groups, layout as below
                            uint32_t xh[16], xl[16];
                            slot_taps<W, C::kBasesX, 16>(
                                poly, *reinterpret_cast<const uint2*>(cur + (lane >> 3) * RW + 2 * pr), xh, xl);
                            uint32_t* Gs = xs + (lane >> 3) * C::kXWords;
#pragma unroll
                            for (int s = 0; s < 16; ++s) {
                                Gs[s * 8 + (pr ^ (s & 4))] = xh[s];
                                Gs[XO + s * 8 + (pr ^ (s & 4))] = xl[s];
                            }
                        }
                    }
                }
                // x (lanes 0-15, unless staged above) and z (16-31) windows of 2 groups:
                // [slot][pair], the pair's bit 2 flipped for slots 4-7 of every 8 (a fragment
                // read then meets 32 different banks)
                const int l16 = lane & 15, ax = lane >> 4, pr = l16 & 7;
                if (l16 < 8 * (gb - g) && (XS == 8 || ax == 1)) {
                    uint32_t hi[8], lo[8];
                    slot_taps<W, BASES, 8>(poly, *reinterpret_cast<const uint2*>(
                                                       cur + ((r & 2) + (l16 >> 3)) * RW + 32 * ax + 2 * pr),
                                           hi, lo);
                    uint32_t* Gs = ax ? zs + (l16 >> 3) * C::kZWords : xs + (l16 >> 3) * C::kXWords;
#pragma unroll
                    for (int s = 0; s < 8; ++s) {
                        Gs[s * 8 + (pr ^ (s & 4))] = hi[s];
                        Gs[64 + s * 8 + (pr ^ (s & 4))] = lo[s];
                    }
                }
                __syncwarp();
            }
            // ---- contract: pairs c and c + 4 of the group are this lane's ----
            const int f0 = row * 8 + (c ^ sx), f1 = row * 8 + ((c + 4) ^ sx);
            // weighted z operand: B[k][n = z], k = points (2c, 2c + 1) and (2c + 8, 2c + 9)
            uint32_t bh[CH][2], bl[CH][2];
            const uint32_t* Z = zs + gi * C::kZWords;
            const uint32_t zh0 = Z[f0], zh1 = Z[f1], zl0 = Z[64 + f0], zl1 = Z[64 + f1];
            const uint2* w0 = reinterpret_cast<const uint2*>(cur + (r & 3) * RW + 48) + c * CH;
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                const uint2 wa = w0[ch], wb = w0[4 * CH + ch];
                mul_split(wa.x, wa.y, zh0, zl0, bh[ch][0], bl[ch][0]);
                mul_split(wb.x, wb.y, zh1, zl1, bh[ch][1], bl[ch][1]);
            }
            const uint32_t* X = xs + (r & (C::kXG - 1)) * C::kXWords;
            uint32_t xh[2][2], xl[2][2];           // [x = row, row + 8][pair]
#pragma unroll
            for (int q = 0; q < XS / 8; ++q) {
                xh[q][0] = X[64 * q + f0];
                xh[q][1] = X[64 * q + f1];
                xl[q][0] = X[XO + 64 * q + f0];
                xl[q][1] = X[XO + 64 * q + f1];
            }
            const uint4* y0 = reinterpret_cast<const uint4*>(ys + (r & 3) * C::kYWords + c * 8);
            const uint4* y1 = y0 + 8;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const uint4 yh0v = y0[half], yl0v = y0[16 + half], yh1v = y1[half ^ 1], yl1v = y1[16 + (half ^ 1)];
                const uint32_t yh0[4] = {yh0v.x, yh0v.y, yh0v.z, yh0v.w}, yl0[4] = {yl0v.x, yl0v.y, yl0v.z, yl0v.w};
                const uint32_t yh1[4] = {yh1v.x, yh1v.y, yh1v.z, yh1v.w}, yl1[4] = {yl1v.x, yl1v.y, yl1v.z, yl1v.w};
#pragma unroll
                for (int q = 0; q < T / 2; ++q) {
                    // operand rows: (x, y = 2t), (x, 2t + 1) at 8 x cells; (x, t), (x + 8, t) at 16
                    const int t = half * (T / 2) + q;
                    const int ya = XS == 8 ? 2 * q : q, yb = XS == 8 ? 2 * q + 1 : q, xb = XS == 8 ? 0 : 1;
                    uint32_t ah[4], al[4];
                    mul_split(xh[0][0], xl[0][0], yh0[ya], yl0[ya], ah[0], al[0]);
                    mul_split(xh[xb][0], xl[xb][0], yh0[yb], yl0[yb], ah[1], al[1]);
                    mul_split(xh[0][1], xl[0][1], yh1[ya], yl1[ya], ah[2], al[2]);
                    mul_split(xh[xb][1], xl[xb][1], yh1[yb], yl1[yb], ah[3], al[3]);
                    // the group's products from zero, small ones first, then one rounded add: the
                    // tensor core's own additions truncate
                    float E[CH][4] = {};
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) mma16816(E[ch], al, bh[ch][0], bh[ch][1]);
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) mma16816(E[ch], ah, bl[ch][0], bl[ch][1]);
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) mma16816(E[ch], ah, bh[ch][0], bh[ch][1]);
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            D[t][ch][k] = __fadd2_rn(D[t][ch][k], make_float2(E[ch][2 * k], E[ch][2 * k + 1]));
                }
            }
        }
        flush_class<W, CH>(D, cls, lev1, row, c);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    // ---- the region into the FP64 grid (periodic wrap), cleared: a thread per column ----
    const int ek = (wk.w & 0xffff) - kUnitBias, eb = (wk.w >> 16) - kUnitBias;
    double* gk = a.grid;
    double* gb_ = CH == 3 ? a.grid + (size_t)a.G * a.G * a.G : a.grid;
    if (tid < RG * RG) {
        const int ry = tid / RG, rx = tid - ry * RG;
        int gx = (wk.x % a.nb) * kBrick - W / 2 + rx, gy = ((wk.x / a.nb) % a.nb) * kBrick - W / 2 + ry;
        int gz = (wk.x / (a.nb * a.nb)) * kBrick - W / 2;
        gx += gx < 0 ? a.G : gx >= a.G ? -a.G : 0;
        gy += gy < 0 ? a.G : gy >= a.G ? -a.G : 0;
        gz += gz < 0 ? a.G : 0;
        const uint32_t col = (uint32_t)gy * a.G + gx, plane = (uint32_t)a.G * a.G;
#pragma unroll 2
        for (int rz = 0; rz < RG; ++rz) {
            const uint32_t cell = (uint32_t)gz * plane + col;
            if (++gz == a.G) gz = 0;
#pragma unroll
            for (int ch = 0; ch < CH; ++ch) {
                int* p = &lev1[ch * RG3 + rz * C::PS + tid];
                const int v = *p;
                if (v == 0) continue;
                *p = 0;
                if (CH != 2 && ch == 0) atomicAdd(&gk[cell], widen_scaled((float)v, ek));
                else atomicAdd(&gb_[2 * (size_t)cell + (CH == 3 ? ch - 1 : ch)], widen_scaled((float)v, eb));
            }
        }
    }
}

template <int W, int CH>
__global__ void __launch_bounds__(kMmaThreads, 2) k_spread_mma(const SpreadArgs a, const __grid_constant__ MmaPoly poly,
                                                                     int pass) {
    pdl_wait();
    pdl_launch();
    using C = MmaCfg<W, CH>;
    extern __shared__ __align__(16) int sm_mma[];
    __shared__ int s_item;
    int* const lev1 = sm_mma + kMmaWarps * (C::kWarpWords + 8 * C::kRecWords);
    uint32_t* const wbuf = reinterpret_cast<uint32_t*>(sm_mma) + (threadIdx.x >> 5) * (C::kWarpWords + 8 * C::kRecWords);
    for (int i = threadIdx.x; i < CH * C::RG3; i += kMmaThreads) lev1[i] = 0;
    int4* const ps = a.pass + pass;
    const int first = ps[0].x, n_work = ps[1].x;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = first + atomicAdd(&ps->w, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= n_work) break;
        spread_item_mma<W, CH>(a, poly, a.rec_item[item], lev1, wbuf);
    }
}

// The work items of several plans (those binned for this form) from one queue, as
// k_spread_batch.
template <int W, int CH>
__global__ void __launch_bounds__(kMmaThreads, 2) k_spread_mma_batch(const SpreadArgs* __restrict__ desc, int n,
                                                                     const int* __restrict__ item_off, int* queue,
                                                                     const __grid_constant__ MmaPoly poly) {
    using C = MmaCfg<W, CH>;
    extern __shared__ __align__(16) int sm_mma[];
    __shared__ int s_item, s_prob;
    int* const lev1 = sm_mma + kMmaWarps * (C::kWarpWords + 8 * C::kRecWords);
    uint32_t* const wbuf = reinterpret_cast<uint32_t*>(sm_mma) + (threadIdx.x >> 5) * (C::kWarpWords + 8 * C::kRecWords);
    for (int i = threadIdx.x; i < CH * C::RG3; i += kMmaThreads) lev1[i] = 0;
    const int total = item_off[n];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const int g = atomicAdd(queue, 1);
            int lo = 0, hi = n;                        // last p with item_off[p] <= g
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (item_off[mid] <= g) lo = mid; else hi = mid;
            }
            s_item = g;
            s_prob = lo;
        }
        __syncthreads();
        const int g = s_item;
        if (g >= total) break;
        const int pi = s_prob;
        const SpreadArgs& a = desc[pi];
        spread_item_mma<W, CH>(a, poly, a.rec_item[g - item_off[pi]], lev1, wbuf);
    }
}

template <int W, int CH>
static cudaError_t spread_mma_batch_w(int n, const SpreadArgs* desc, const int* item_off, int* queue,
                                      const KbPoly& poly, int num_sms, cudaStream_t s) {
    constexpr size_t smem = MmaCfg<W, CH>::kSmem;
    cudaError_t e =
        cudaFuncSetAttribute(k_spread_mma_batch<W, CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spread_mma_batch<W, CH>, kMmaThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    k_spread_mma_batch<W, CH><<<num_sms * per_sm, kMmaThreads, smem, s>>>(desc, n, item_off, queue, mma_poly(poly, W));
    return cudaGetLastError();
}

cudaError_t launch_spread_mma_batch(int n, bool kc, int W, const SpreadArgs* desc, const int* item_off, int* queue,
                                    const KbPoly& poly, int num_sms, cudaStream_t s) {
    if (W == 7)
        return kc ? spread_mma_batch_w<7, 1>(n, desc, item_off, queue, poly, num_sms, s)
                  : spread_mma_batch_w<7, 2>(n, desc, item_off, queue, poly, num_sms, s);
    return kc ? spread_mma_batch_w<6, 1>(n, desc, item_off, queue, poly, num_sms, s)
              : spread_mma_batch_w<6, 2>(n, desc, item_off, queue, poly, num_sms, s);
}

template <int W, int CH>
static cudaError_t spread_mma_w(Plan& P, const SpreadArgs& a, int pass) {
    constexpr size_t smem = MmaCfg<W, CH>::kSmem;
    cudaError_t e = cudaFuncSetAttribute(k_spread_mma<W, CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spread_mma<W, CH>, kMmaThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    launch_pdl(k_spread_mma<W, CH>, P.num_sms * per_sm, kMmaThreads, smem, P.stream, a, mma_poly(a.poly, W), pass);
    P.launches += 1;
    return cudaGetLastError();
}

template <int W, int CH>
static cudaError_t mma_sort_w(Plan& P, const SpreadArgs& a, int pass) {
    constexpr size_t smem = MmaCfg<W, CH>::kSortSmem;
    cudaError_t e = cudaFuncSetAttribute(k_mma_sort<W, CH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    launch_pdl(k_mma_sort<W, CH>, P.num_sms * 2, kSortThreads, smem, P.stream, a, pass);
    P.launches += 1;
    return cudaGetLastError();
}

// First item of every pass: the item before which `pass` buffers of slots are spoken for, with
// all padding (an item's points and slots before it follow from its number and start).
__global__ void k_mma_passes(const int4* work, const int* counters, int4* pass, int n) {
    pdl_wait();
    pdl_launch();
    const int p = threadIdx.x;
    if (p > n) return;
    const unsigned at = (unsigned)p * kMmaPassSlots;          // 37 passes at most: below 2^32
    int lo = 0, hi = counters[0];
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((unsigned)work[mid].y + (unsigned)mid * kMmaPad < at) lo = mid + 1;
        else hi = mid;
    }
    pass[p] = make_int4(p == n ? counters[0] : lo, 0, 0, 0);
}

cudaError_t launch_mma_passes(Plan& P) {
    static_assert(kMmaMaxPasses < 64 && (unsigned long long)kMmaMaxPasses * kMmaPassSlots < (1ull << 32), "pass offsets");
    P.launches += 1;
    return launch_pdl(k_mma_passes, 1, 64, 0, P.stream, P.ws.work, P.ws.counters, P.ws.pass, P.bin_passes);
}

cudaError_t launch_mma_sort(Plan& P, const SpreadArgs& a, int ch, int pass) {
    if (P.p.W == 7)
        return ch == 1   ? mma_sort_w<7, 1>(P, a, pass)
               : ch == 2 ? mma_sort_w<7, 2>(P, a, pass)
                         : cudaErrorInvalidValue;
    switch (ch) {
        case 1: return mma_sort_w<6, 1>(P, a, pass);
        case 2: return mma_sort_w<6, 2>(P, a, pass);
        case 3: return mma_sort_w<6, 3>(P, a, pass);
        default: return cudaErrorInvalidValue;
    }
}

static cudaError_t spread_pass(Plan& P, const SpreadArgs& a, int ch, int pass) {
    if (P.p.W == 7)
        return ch == 1   ? spread_mma_w<7, 1>(P, a, pass)
               : ch == 2 ? spread_mma_w<7, 2>(P, a, pass)
                         : cudaErrorInvalidValue;
    switch (ch) {
        case 1: return spread_mma_w<6, 1>(P, a, pass);
        case 2: return spread_mma_w<6, 2>(P, a, pass);
        case 3: return spread_mma_w<6, 3>(P, a, pass);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_spread_mma(Plan& P, const SpreadArgs& a, int ch) {
    if (P.bin_passes == 1) return spread_pass(P, a, ch, 0);      // sorted with the placement
    for (int p = 0; p < P.bin_passes; ++p) {
        cudaError_t e = launch_mma_sort(P, a, ch, p);
        if (e == cudaSuccess) e = spread_pass(P, a, ch, p);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace firm
