// Transpose operator X = H(theta)^T Y in gather form (sm_103a).
//
//   k_adj_tile   FP32, parallel beam: one CTA per 32 x 32 pixel tile, view
//                subset and group of KB sinograms, 2 x 2 pixels per thread
//   k_adj64      FP64, parallel beam: one CTA per 16 x 16 pixel tile, view
//                subset and group of KB sinograms, one pixel per thread
//   k_adj_small  both precisions, small images: one CTA per 16 x 2 pixels and
//                group of KB sinograms, one pixel and one of SPLIT view subsets
//                per thread
//
// For pixel (i, j) and view v the continuous bin coordinate of the pixel
// centre is beta = beta0 + j*c - i*s.  The rays that sampled the pixel in
// the forward rule are the bins b with |b - beta| < 1/w, and the forward
// interpolation gave each of them the weight w * (1 - |b - beta| * w) -- at
// most two bins, floor(beta) and floor(beta) + 1.  This is the residual step
// H^T (H u - b) of every MM-GKS iteration (Eq. (3.6), Alg. "Enlarge").
//
// beta is split into an FP64 tile anchor (once per tile and view) plus an
// in-tile offset, in integer fixed point in k_adj_tile and k_adj64: exact sums,
// and the cell and fraction come from shifts.  There the `segs` CTAs of a tile form one
// thread-block cluster; CTA s takes the views s, s + segs, ... of the frame
// and leaves its sums in its shared memory; the CTAs then add them through
// distributed shared memory in segment order, each for its share of the
// pixels.  No atomics, no partial images in global memory.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ct_device.cuh"
#include "ct_internal.cuh"

namespace ctgb {
namespace {

namespace cg = cooperative_groups;

// A tile's first bin from a 64-bit cell.  A view shifted far off the detector
// stays off it: cells beyond 32 bits are held short of their range (with room
// for the in-tile offset), not wrapped back onto the bins.
__device__ __forceinline__ int far_cell(long long cell)
{
    return (int)max(min(cell, 0x7fff0000LL), -0x7fff0000LL);
}

// ---------------------------------------------------------------------------
// FP32
// ---------------------------------------------------------------------------
constexpr int kAdjTile = 32;      // tile side
constexpr int kAdjWin = 52;       // staged bins per view: 31 (|c| + |s|) <= 43.9, the cells around it, alignment
constexpr int kAdjViewCap = 128;  // views whose tile constants are staged at a time
static_assert(kAdjFrac == 26 && kAdjWin <= 64, "a staged slot coordinate fits 32 bits");

struct AdjArgs {
    const ViewGeo *vg;
    const int *fstart, *fcount;
    const int *rowflag;        // [group][V]: the group's sinograms hold a non-finite value in this view
    int N, B, V, F, tps, Pq;
    const float *YI;           // interleaved sinograms (see launch_sino_layout)
    long long group_stride;    // floats between the groups of this launch
    int kbase, ngroups, kend;
    float *X;
    long long img_stride;      // F * N * N
    int segs;                  // CTAs per tile (view subsets) = cluster size
    const int *skip;
};

// Per (view, tile) constants.
struct __align__(16) AdjView {
    int C, S;       // staged slot coordinate of pixel (x, y): x * C + y * S + F, unsigned, kAdjFrac
    unsigned F;     // fractional bits
    float w;        // weight 1/|cos| or 1/|sin|
    float p0, p1;   // KB <= 2: 1 + w and 1 - 2 w; KB >= 4: |c| and |s|, the coordinates of a 2 x 2
                    // block's neighbours of the lowest corner
    float om;       // KB >= 4: |c| + |s| - 1, the opposite corner less one bin
    int quad;       // bit 0: c < 0, bit 1: s > 0 (which corner is lowest), bit 2: non-finite sinogram row
    int start;      // first staged bin
    int row;        // view
    float w2, c1;   // KB >= 4: w^2 and w - w^2
};

// Sums of a thread's 2 x 2 pixels (index 2 * y + x) for KB sinograms.
// KB <= 2: each pixel reads its own two bins, the kernel being bound by the
// issue rate; the sums of the two pixels of a row are packed.  KB >= 4: the
// block reads its four bins together (below).
template <int KB> struct AdjSums {
    f32x2 v[2][KB];
    __device__ void clear()
    {
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int k = 0; k < KB; ++k) v[c][k] = 0ull;
    }
    __device__ float get(int c, int k) const { return half2f(v[c >> 1][k], c & 1); }

    // One view; p: its slot 0.  Per pixel: the cell and the fraction g = 1 + e of
    // the coordinate (23 bits, straight into a mantissa), the two hat values
    // without their factor w as saturated multiply-adds (1 - e w and 1 - (1 - e) w
    // clamped to [0, 1]), and the factor once per pixel.
    __device__ __forceinline__ void view(const float *p, int px, int py, const AdjView &av)
    {
        const unsigned t0 = ((unsigned)(px * av.C + py * av.S) + av.F) >> (kAdjFrac - 23);
        const int dx = av.C >> (kAdjFrac - 23), dy = av.S >> (kAdjFrac - 23);
        const f32x2 ww = pack2(av.w, av.w);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            float h0[2], h1[2];
            const float *q[2];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const unsigned t = t0 + (x ? dx : 0) + (r ? dy : 0);
                const float g = __int_as_float((t & 0x7FFFFF) | 0x3F800000);
                h0[x] = __saturatef(fmaf(-g, av.w, av.p0));
                h1[x] = __saturatef(fmaf(g, av.w, av.p1));
                q[x] = p + (t >> 23) * KB;
            }
            const f32x2 H0 = pack2(h0[0], h0[1]), H1 = pack2(h1[0], h1[1]);
            if constexpr (KB == 1) {
                v[r][0] = fma2(ww, fma2(H1, pack2(q[0][1], q[1][1]), mul2(H0, pack2(q[0][0], q[1][0]))), v[r][0]);
            } else {
                const float2 a0 = *reinterpret_cast<const float2 *>(q[0]), a1 = *reinterpret_cast<const float2 *>(q[0] + 2);
                const float2 b0 = *reinterpret_cast<const float2 *>(q[1]), b1 = *reinterpret_cast<const float2 *>(q[1] + 2);
                v[r][0] = fma2(ww, fma2(H1, pack2(a1.x, b1.x), mul2(H0, pack2(a0.x, b0.x))), v[r][0]);
                v[r][1] = fma2(ww, fma2(H1, pack2(a1.y, b1.y), mul2(H0, pack2(a0.y, b0.y))), v[r][1]);
            }
        }
    }
};

// KB = 4 or 8: the sums of two sinograms packed in a register pair, so that one
// fma.rn.f32x2 serves both.  The KB values of a staged slot are stored as
// arrays of 4 so that the 16-byte loads of a quarter-warp, whose lanes read at
// most 8 consecutive slots, fall in distinct banks.
template <int KB> struct AdjSumsPacked {
    f32x2 v[4][KB / 2];
    __device__ void clear()
    {
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int k = 0; k < KB / 2; ++k) v[c][k] = 0ull;
    }
    __device__ float get(int c, int k) const
    {
        return half2f(v[c][k >> 1], k & 1);
    }
    __device__ __forceinline__ static void load(const float *p, int slot, f32x2 (&y)[KB / 2])
    {
#pragma unroll
        for (int g = 0; g < KB / 4; ++g) {
            const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(p + (g * kAdjWin + slot) * 4);
            y[2 * g] = u.x;
            y[2 * g + 1] = u.y;
        }
    }
    __device__ __forceinline__ void add(int c, float h, const f32x2 (&y)[KB / 2])
    {
        const f32x2 hh = pack2(h, h);
#pragma unroll
        for (int k = 0; k < KB / 2; ++k) v[c][k] = fma2(hh, y[k], v[c][k]);
    }

    // One view's contribution to the block.  e in [0, 1] is the fraction of
    // the lowest corner's coordinate in cell 0 (slot s0).  The corners lie at e,
    // e + a, e + b and e + a + b with a, b <= 1 <= a + b < 1.42, so the lowest
    // reads slots 0-1, its two neighbours 0-2 and the opposite corner 1-3; the
    // hat w max(0, 1 - |x| w) vanishes on the slots left out.  QX (QY): the lowest
    // corner is the right (lower) one.
    template <int QX, int QY>
    __device__ __forceinline__ void block(const float *p, int s0, float e, const AdjView &av)
    {
        constexpr int LO = 2 * QY + QX, NX = 2 * QY + 1 - QX, NY = 2 * (1 - QY) + QX, HI = 2 * (1 - QY) + 1 - QX;
        const float w = av.w, w2 = av.w2, c1 = av.c1, c2 = c1 - w2;
        auto below = [&](float x) { return fmaxf(0.0f, fmaf(-x, w2, w)); };          // slot x below the pixel
        auto above1 = [&](float x) { return fmaxf(0.0f, fmaf(x, w2, c1)); };         // slot 1 - x above it
        auto above2 = [&](float x) { return fmaxf(0.0f, fmaf(x, w2, c2)); };         // slot 2 - x above it
        const float ea = e + av.p0, eb = e + av.p1, em = e + av.om;
        f32x2 y[KB / 2];
        load(p, s0, y);
        add(LO, below(e), y);
        add(NX, below(ea), y);
        add(NY, below(eb), y);
        load(p, s0 + 1, y);
        add(LO, above1(e), y);
        add(NX, below(fabsf(ea - 1.0f)), y);
        add(NY, below(fabsf(eb - 1.0f)), y);
        add(HI, below(em), y);
        load(p, s0 + 2, y);
        add(NX, above2(ea), y);
        add(NY, above2(eb), y);
        add(HI, below(fabsf(em - 1.0f)), y);
        load(p, s0 + 3, y);
        add(HI, above2(em), y);
    }

    __device__ __forceinline__ void view(const float *p, int px, int py, const AdjView &av)
    {
        const unsigned t = (unsigned)(px * av.C + py * av.S) + av.F;  // the block's lowest corner
        const int s0 = (int)(t >> kAdjFrac);
        const float e = __int_as_float(((t >> (kAdjFrac - 23)) & 0x7FFFFF) | 0x3F800000) - 1.0f;
        switch (av.quad) {  // uniform
        case 0: block<0, 0>(p, s0, e, av); break;
        case 1: block<1, 0>(p, s0, e, av); break;
        case 2: block<0, 1>(p, s0, e, av); break;
        case 3: block<1, 1>(p, s0, e, av); break;
        default:
            // each corner reads its own two bins only: zero weights on other slots
            // would spread a non-finite sample (0 * inf) to pixels whose bins do
            // not hold it
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int dx = (c & 1) ^ (av.quad & 1), dy = (c >> 1) ^ ((av.quad >> 1) & 1);
                const float x = e + (dx ? av.p0 : 0.0f) + (dy ? av.p1 : 0.0f), w2 = av.w2;
                const float fl = floorf(x), f = x - fl;
                const int s = s0 + (int)fl;
                f32x2 y[KB / 2];
                load(p, s, y);
                add(c, fmaxf(0.0f, fmaf(-f, w2, av.w)), y);
                load(p, s + 1, y);
                add(c, fmaxf(0.0f, fmaf(-(1.0f - f), w2, av.w)), y);
            }
        }
    }
};
template <> struct AdjSums<4> : AdjSumsPacked<4> {};
template <> struct AdjSums<8> : AdjSumsPacked<8> {};

// Four floats at a shared-memory address of CTA `rank` of the cluster (its own included).
__device__ __forceinline__ float4 ld_cluster4(unsigned addr, int rank)
{
    unsigned r;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(r)
                 : "memory");
    return v;
}

// Views per staged block (two blocks in flight).
template <int KB> constexpr int adj_vb() { return KB >= 8 ? 8 : 16; }
template <int KB> constexpr size_t adj_smem(bool reduce)
{
    const size_t st = sizeof(float) * 2 * adj_vb<KB>() * KB * kAdjWin;
    const size_t red = sizeof(float) * KB * kAdjTile * kAdjTile;
    return reduce && red > st ? red : st;
}

// One CTA = 256 threads on a 32 x 32 tile of one frame, the views of one
// segment and KB sinograms.  The window of bins a tile reads of a view is
// staged in shared memory (KB values of a bin side by side, no bin stored
// twice), VB views at a time, the next block copied with cp.async while the
// current one is read.  A thread owns a 2 x 2 block: its four pixels read four
// slots together instead of eight taps, which halves the shared-memory
// wavefronts, the bound of the one-pixel form.  The lanes of a quarter-warp
// take 4 x 2 blocks, whose slots lie within 8 consecutive ones: no bank
// conflicts.  For one or two sinograms the issue rate is the bound instead
// (89 % issued), and the instructions per pixel and view decide: 16 with
// packed multiply-adds and saturated hats.  Measured against one pixel per
// thread reading pairs: 2048^2 / 120 views, one sinogram 530 -> 232 us; 512^2 /
// 360 views, four 230 -> 99; 16 frames of 256^2 / 1200 views, eight 413 -> 165;
// 256^2 / 180 views, eight 37 (staged pairs) -> 31.
template <int KB>
__global__ void __launch_bounds__(256, KB <= 2 ? 6 : 0) k_adj_tile(AdjArgs a)
{
    chain_wait();
    constexpr int VB = adj_vb<KB>();
    constexpr int VIEW = KB * kAdjWin;  // floats per staged view
    constexpr int NCH = VIEW / 4;       // 16-byte copies per staged view
    static_assert(VIEW % 4 == 0 && kAdjViewCap % VB == 0, "whole copies and blocks");
    extern __shared__ float4 adj_smem4[];
    float *sbuf = reinterpret_cast<float *>(adj_smem4);  // [2][VB][VIEW]
    __shared__ AdjView s_view[kAdjViewCap];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // block coordinates: a quarter-warp 4 x 2, a warp 8 x 4, the CTA 16 x 16
    const int bx = (warp & 1) * 8 + ((lane >> 3) & 1) * 4 + (lane & 3);
    const int by = (warp >> 1) * 4 + (lane >> 4) * 2 + ((lane >> 2) & 1);
    const int px = 2 * bx - kAdjTile / 2, py = 2 * by - kAdjTile / 2;  // relative to the anchor pixel
    const int tiles = a.tps * a.tps;
    const int segs = a.segs;
    const int total = a.ngroups * a.F * tiles * segs;
    const int N = a.N;
    if (a.skip && *a.skip) return;
    // The grid is a whole number of clusters and total a multiple of segs, so
    // the CTAs of a cluster take the segments of one tile in every iteration
    // and leave the loop together (the cluster barriers below are uniform).
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int seg = item % segs;  // = rank of the CTA in its cluster
        int t2 = item / segs;
        const int tile = t2 % tiles;
        t2 /= tiles;
        const int f = t2 % a.F;
        const int grp = t2 / a.F;
        const int i0 = (tile / a.tps) * kAdjTile, j0 = (tile % a.tps) * kAdjTile;
        const int k0 = a.kbase + grp * KB;
        const float *yg = a.YI + (size_t)grp * a.group_stride;
        const int vs = a.fstart[f], vc = a.fcount[f];
        const int nv = vc > seg ? (vc - seg + segs - 1) / segs : 0;  // this CTA's views: vs + seg + q * segs

        AdjSums<KB> acc;
        acc.clear();
        for (int cb = 0; cb < nv; cb += kAdjViewCap) {
            const int nc = min(kAdjViewCap, nv - cb);
            const int nblk = (nc + VB - 1) / VB;
            __syncthreads();  // the previous chunk (or item) is done with s_view and both buffers
            for (int q = tid; q < nc; q += blockDim.x) {
                const int v = vs + seg + (cb + q) * segs;
                const ViewGeo &g = a.vg[v];
                // bin coordinate of the anchor pixel, the only FP64 step per tile and view
                const double bt = g.beta0 + (double)(j0 + kAdjTile / 2) * g.c - (double)(i0 + kAdjTile / 2) * g.s;
                const long long fx = __double2ll_rn(bt * (double)(1 << kAdjFrac));
                const int ix = far_cell(fx >> kAdjFrac);
                const int frac = (int)(fx & ((1 << kAdjFrac) - 1));
                const float w = GeoT<float>::w(g);
                AdjView av;
                av.C = g.aC;
                av.S = -g.aS;
                av.w = w;
                if constexpr (KB >= 4) {
                    const float unit = 1.0f / (float)(1 << kAdjFrac);
                    av.p0 = (float)abs(av.C) * unit;
                    av.p1 = (float)abs(av.S) * unit;
                    av.om = (float)(abs(av.C) + abs(av.S) - (1 << kAdjFrac)) * unit;
                    av.w2 = w * w;
                    av.c1 = w - av.w2;
                } else {
                    av.p0 = 1.0f + w;
                    av.p1 = 1.0f - 2.0f * w;
                    av.om = 0.0f;
                }
                av.quad = (av.C < 0 ? 1 : 0) | (av.S < 0 ? 2 : 0) | (a.rowflag[(size_t)grp * a.V + v] ? 4 : 0);
                // lowest cell of the tile, one bin of margin, aligned for 16-byte copies
                constexpr int AL = KB >= 4 ? 1 : 4 / KB;
                const int lo =
                    ix - 1 + ((frac + min(-16 * av.C, 15 * av.C) + min(-16 * av.S, 15 * av.S)) >> kAdjFrac);
                av.start = lo & ~(AL - 1);
                av.F = ((unsigned)(ix - av.start) << kAdjFrac) + (unsigned)frac;
                // KB >= 4: the block's lowest corner, half a unit of the 23-bit fraction
                // added (it is rounded, not truncated)
                if constexpr (KB >= 4) av.F += (unsigned)(min(0, av.C) + min(0, av.S) + (1 << (kAdjFrac - 24)));
                av.row = v;
                s_view[q] = av;
            }
            __syncthreads();

            auto stage = [&](int blk, int buf) {
                const int nq = min(VB, nc - blk * VB);
                for (int u = tid; u < nq * NCH; u += 256) {
                    const int q = u / NCH, c = u % NCH;
                    const AdjView &av = s_view[blk * VB + q];
                    float *dst = sbuf + (size_t)buf * VB * VIEW + q * VIEW;
                    if constexpr (KB >= 4) {
                        constexpr int G = KB / 4;
                        const int slot = c / G, g = c % G, bin = av.start + slot;
                        const bool ok = bin >= 0 && bin < a.Pq;
                        cp_async16_zfill(dst + (g * kAdjWin + slot) * 4,
                                         ok ? yg + ((size_t)av.row * a.Pq + bin) * KB + 4 * g : yg, ok);
                    } else {
                        const int bin = av.start + c * (4 / KB);  // Pq is a multiple of 4
                        const bool ok = bin >= 0 && bin < a.Pq;
                        cp_async16_zfill(dst + 4 * c, ok ? yg + ((size_t)av.row * a.Pq + bin) * KB : yg, ok);
                    }
                }
            };

            stage(0, 0);
            cp_async_commit();
            for (int blk = 0; blk < nblk; ++blk) {
                cp_async_wait0();
                // block blk is visible to every thread, and every thread has finished
                // block blk - 1, whose buffer the next copies overwrite
                __syncthreads();
                if (blk + 1 < nblk) stage(blk + 1, (blk + 1) & 1);
                cp_async_commit();
                const int nq = min(VB, nc - blk * VB);
                const float *base = sbuf + (size_t)(blk & 1) * VB * VIEW;
                for (int q = 0; q < nq; ++q) {
                    const AdjView av = s_view[blk * VB + q];
                    acc.view(base + q * VIEW, px, py, av);
                }
            }
            cp_async_wait0();  // the last group is empty
        }
        float *red = sbuf;  // [KB][32][32], over the staging buffers
        __syncthreads();    // every warp is done with them
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            float *r = red + k * kAdjTile * kAdjTile + 2 * by * kAdjTile + 2 * bx;
            *reinterpret_cast<float2 *>(r) = make_float2(acc.get(0, k), acc.get(1, k));
            *reinterpret_cast<float2 *>(r + kAdjTile) = make_float2(acc.get(2, k), acc.get(3, k));
        }
        cg::cluster_group cl = cg::this_cluster();
        if (segs > 1) cl.sync();
        else __syncthreads();
        // this CTA's share of the pixels, the segments added in order; W pixels of a
        // row at a time (wide groups have as many values to add as a few views take
        // time: 256^2, 22 views, 8 sinograms: 12.9 us with one at
        // a time, 11.1 so; 180 views 30.9 and 29.8)
        constexpr int W = KB >= 4 ? 4 : 1;
        constexpr int OUT = KB * kAdjTile * kAdjTile / W;
#pragma unroll 1
        for (int u = OUT / 32 * seg / segs * 32 + tid; u < OUT / 32 * (seg + 1) / segs * 32; u += 256) {
            float s[W];
            if constexpr (W == 4) {
                const unsigned at = (unsigned)__cvta_generic_to_shared(red + 4 * u);
#pragma unroll
                for (int q0 = 0; q0 < kMaxSegs; q0 += 4) {  // four segments' loads in flight
                    if (q0 >= segs) break;
                    float4 part[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) part[q] = ld_cluster4(at, min(q0 + q, segs - 1));
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q0 + q >= segs) break;
                        const float e[4] = {part[q].x, part[q].y, part[q].z, part[q].w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) s[c] = q0 + q == 0 ? e[c] : s[c] + e[c];
                    }
                }
            } else if (segs == 1) {
                s[0] = red[u];
            } else {
                float part[kMaxSegs];  // all loads in flight
#pragma unroll
                for (int q = 0; q < kMaxSegs; ++q) part[q] = q < segs ? *cl.map_shared_rank(red + u, q) : 0.0f;
                s[0] = part[0];
#pragma unroll
                for (int q = 1; q < kMaxSegs; ++q)
                    if (q < segs) s[0] += part[q];
            }
            const int k = W * u / (kAdjTile * kAdjTile), p = W * u % (kAdjTile * kAdjTile);
            const int i = i0 + p / kAdjTile, j = j0 + p % kAdjTile;
            if (i < N && k0 + k < a.kend) {
                float *x = a.X + (size_t)(k0 + k) * a.img_stride + (size_t)f * N * N + (size_t)i * N + j;
#pragma unroll
                for (int c = 0; c < W; ++c)
                    if (j + c < N) x[c] = s[c];
            }
        }
        if (segs > 1) cl.sync();  // the others keep their shared memory until it has been read
    }
}

// ---------------------------------------------------------------------------
// FP64
// ---------------------------------------------------------------------------
// FP64 instructions occupy a sub-partition's pipe for 64 cycles each on this
// part, so the kernel spends them on the products alone: two for the weights
// of a pixel and view, two per sinogram.  The bin coordinate, its cell and
// fraction and the clamping of the weights at zero are integer work.  255^2,
// 181 views, four sinograms: 508 -> 217 us, the FP64 pipe 94 % busy.
constexpr int kAdj64Frac = 56;
constexpr int kAdj64Cap = 128;

struct Adj64Args {
    const ViewGeo *vg;
    const int *fstart, *fcount;
    int N, B, F, tps, Pb;
    const double2 *YP;         // pair sinograms
    long long ysino_stride;    // pairs per batch element (V * Pb)
    int kbase, ngroups, kend;
    double *X;
    long long img_stride;
    int segs;
    const int *skip;
};

struct __align__(16) Adj64View {
    long long C, S, F;   // in-tile coordinate x * C - y * S + F
    double w2, wa, wb;   // weights max(0, wa - g w2) and max(0, wb + g w2), g = 1 + fraction
    int ix, row;
};

__device__ __forceinline__ double clamp0(double x)  // max(0, x) of a number, on the integer pipe
{
    return __double2hiint(x) < 0 ? 0.0 : x;
}

template <int KB>
__global__ void __launch_bounds__(256) k_adj64(Adj64Args a)
{
    chain_wait();
    __shared__ Adj64View s_view[kAdj64Cap];
    __shared__ double red[KB][256];
    const int tid = threadIdx.x;
    const int tx = tid & (kTile - 1), ty = tid / kTile;
    const int tiles = a.tps * a.tps;
    const int segs = a.segs;
    const int total = a.ngroups * a.F * tiles * segs;
    const int N = a.N;
    const double scale = (double)(1LL << kAdj64Frac);
    if (a.skip && *a.skip) return;
    for (int item = blockIdx.x; item < total; item += gridDim.x) {  // whole clusters, as in k_adj_tile
        const int seg = item % segs;
        int t2 = item / segs;
        const int tile = t2 % tiles;
        t2 /= tiles;
        const int f = t2 % a.F;
        const int grp = t2 / a.F;
        const int i0 = (tile / a.tps) * kTile, j0 = (tile % a.tps) * kTile;
        const int k0 = a.kbase + grp * KB;
        const double2 *yp = a.YP + (size_t)k0 * a.ysino_stride;
        const int vs = a.fstart[f], vc = a.fcount[f];
        const int nv = vc > seg ? (vc - seg + segs - 1) / segs : 0;
        double acc[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) acc[k] = 0.0;
        for (int cb = 0; cb < nv; cb += kAdj64Cap) {
            const int nc = min(kAdj64Cap, nv - cb);
            __syncthreads();
            for (int q = tid; q < nc; q += 256) {
                const int v = vs + seg + (cb + q) * segs;
                const ViewGeo &g = a.vg[v];
                const double bt = g.beta0 + (double)j0 * g.c - (double)i0 * g.s;
                const double fl = floor(bt);
                const double w = GeoT<double>::w(g);
                Adj64View av;
                av.C = __double2ll_rn(g.c * scale);
                av.S = __double2ll_rn(g.s * scale);
                av.F = __double2ll_rn((bt - fl) * scale);
                av.w2 = w * w;
                av.wa = w + av.w2;
                av.wb = w - 2.0 * av.w2;
                av.ix = far_cell((long long)fl) + 2;
                av.row = v * a.Pb;
                s_view[q] = av;
            }
            __syncthreads();
            constexpr int U = KB >= 4 ? 2 : 4;  // views whose loads are issued together
            for (int q = 0; q < nc; q += U) {
                double2 p[U][KB];
                double wa[U], wb[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const Adj64View &av = s_view[min(q + u, nc - 1)];
                    const long long t = (long long)tx * av.C - (long long)ty * av.S + av.F;
                    const int cell = (int)(t >> kAdj64Frac);
                    const double gf = __longlong_as_double(((t >> (kAdj64Frac - 52)) & 0xFFFFFFFFFFFFFLL) |
                                                           0x3FF0000000000000LL);
                    const bool on = q + u < nc;
                    wa[u] = on ? clamp0(fma(-gf, av.w2, av.wa)) : 0.0;  // bin floor(beta)
                    wb[u] = on ? clamp0(fma(gf, av.w2, av.wb)) : 0.0;   // bin floor(beta) + 1
                    const double2 *row = yp + av.row + min(max(av.ix + cell, 0), a.B + 2);
#pragma unroll
                    for (int k = 0; k < KB; ++k)
                        p[u][k] = on ? __ldg(row + (size_t)k * a.ysino_stride) : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (q + u < nc) {  // uniform
#pragma unroll
                        for (int k = 0; k < KB; ++k) acc[k] = fma(wa[u], p[u][k].x, fma(wb[u], p[u][k].y, acc[k]));
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < KB; ++k) red[k][tid] = acc[k];
        cg::cluster_group cl = cg::this_cluster();
        if (segs > 1) cl.sync();
        else __syncthreads();
        double *r0 = &red[0][0];
        constexpr int OUT = KB * 256;
#pragma unroll 1
        for (int u = OUT / 32 * seg / segs * 32 + tid; u < OUT / 32 * (seg + 1) / segs * 32; u += 256) {
            double s;
            if (segs == 1) {
                s = r0[u];
            } else {
                double part[kMaxSegs];
#pragma unroll
                for (int q = 0; q < kMaxSegs; ++q) part[q] = q < segs ? *cl.map_shared_rank(r0 + u, q) : 0.0;
                s = part[0];
#pragma unroll
                for (int q = 1; q < kMaxSegs; ++q)
                    if (q < segs) s += part[q];
            }
            const int k = u >> 8, p = u & 255;
            const int i = i0 + p / kTile, j = j0 + p % kTile;
            if (i < N && j < N && k0 + k < a.kend)
                a.X[(size_t)(k0 + k) * a.img_stride + (size_t)f * N * N + (size_t)i * N + j] = s;
        }
        if (segs > 1) cl.sync();
        else __syncthreads();  // red[] is rewritten by the next item
    }
}

// ---------------------------------------------------------------------------
// small images, both precisions
// ---------------------------------------------------------------------------
// Images of side up to kSmallN.  Every pixel sums its views in
// two (SPLIT) runs, one after the other, and a whole tile per CTA leaves most
// SMs idle (64^2, 90 views, one sinogram: 16 CTAs took 14 us in FP32 and 94 in
// FP64, bound by 16 SMs' FP64 pipes).  The shorter per-segment sums of the other
// kernels would not give the same bits, and a solve at these sizes repeats
// the product so often on so few pixels that its path follows the last bits.
// So a CTA owns 16 x 2 pixels, all its warps prepare the operands of the sums
// (the two weights and the two bins of each view) in shared memory, and SPLIT
// warps add them in order: 6.1 us in FP32, 16.4 in FP64.
// (More CTAs: 16 frames of 32^2, 10 views each, eight sinograms: 6.8 us before this form,
// 12.7 with it at 512 CTAs, 6.7 on the tiles; one sinogram 5.6, 7.2 and 5.2.)
constexpr int kSmallN = 64;
constexpr int kSmallRows = 2;
constexpr int kSmallCap = 128;   // views whose tile constants are staged at a time
constexpr int kSmallWarps = 16;
constexpr int kSmallViews = 32;  // views whose operands are in shared memory at a time

template <typename T> struct SmallArgs {
    const ViewGeo *vg;
    const int *fstart, *fcount;
    int N, B, F, tps, pitch;
    const T *Y;                // FP32: interleaved groups; FP64: pairs
    long long group_stride;    // FP32: elements between groups; FP64: pairs between sinograms
    int kbase, ngroups, kend;
    T *X;
    long long img_stride;
    const int *skip;
};

// floor(t) and t - floor(t), t small (the FP64 form without conversions: one
// addition rounded down leaves the integer in the low word)
__device__ __forceinline__ void small_split(float t, int &m, float &f) { floor_split(t, m, f); }
__device__ __forceinline__ void small_split(double t, int &m, double &f)
{
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    const double tr = __dadd_rd(t, magic);
    m = __double2loint(tr);
    f = __dsub_rn(t, __dsub_rn(tr, magic));
}
__device__ __forceinline__ float clamp0(float x) { return fmaxf(0.0f, x); }

template <typename T> struct __align__(16) Operands {
    T wa, y0, wb, y1;
};

template <typename T, int KB, int SPLIT>
__global__ void __launch_bounds__(32 * kSmallWarps) k_adj_small(SmallArgs<T> a)
{
    chain_wait();
    constexpr bool F32 = std::is_same<T, float>::value;
    constexpr int PER = kSmallViews / kSmallWarps;  // views a warp prepares
    __shared__ T s_c[kSmallCap], s_s[kSmallCap], s_w[kSmallCap], s_w1[kSmallCap], s_f[kSmallCap];
    __shared__ int2 s_idx[kSmallCap];  // (integer anchor, view)
    __shared__ Operands<T> s_op[kSmallViews][32];
    __shared__ T red[SPLIT][KB][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = lane & (kTile - 1);
    constexpr int kSub = kTile / kSmallRows;
    const int tiles = a.tps * a.tps;
    const int total = a.ngroups * a.F * tiles * kSub;
    const int N = a.N;
    if (a.skip && *a.skip) return;
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int sub = item % kSub;
        int t2 = item / kSub;
        const int tile = t2 % tiles;
        t2 /= tiles;
        const int f = t2 % a.F;
        const int grp = t2 / a.F;
        const int i0 = (tile / a.tps) * kTile, j0 = (tile % a.tps) * kTile;
        const int ty = sub * kSmallRows + lane / kTile;
        const T fx = (T)tx, fy = (T)ty;
        const int k0 = a.kbase + grp * KB;
        const int vs = a.fstart[f], vc = a.fcount[f];
        T acc[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) acc[k] = T(0);
        // (run p takes views p, p + SPLIT, ...: chunk and block sizes are multiples of SPLIT)
        for (int base = 0; base < vc; base += kSmallCap) {
            const int nv = min(kSmallCap, vc - base);
            __syncthreads();
            for (int q = threadIdx.x; q < nv; q += 32 * kSmallWarps) {
                const ViewGeo &g = a.vg[vs + base + q];
                const double bt = g.beta0 + (double)j0 * g.c - (double)i0 * g.s;
                const double fl = floor(bt);
                s_c[q] = (T)g.c;
                s_s[q] = (T)g.s;
                s_w[q] = GeoT<T>::w(g);
                s_w1[q] = T(1) - s_w[q];
                s_f[q] = (T)(bt - fl);
                s_idx[q] = make_int2(far_cell((long long)fl), vs + base + q);
            }
            __syncthreads();
            for (int blk = 0; blk < nv; blk += kSmallViews) {
                const int nb = min(kSmallViews, nv - blk);
                T wa[PER], wb[PER];
                int bin[PER];
#pragma unroll
                for (int u = 0; u < PER; ++u) {
                    const int q = blk + min(warp + u * kSmallWarps, nb - 1);
                    const T t = fma(fx, s_c[q], fma(-fy, s_s[q], s_f[q]));
                    int mm;
                    T fr;
                    small_split(t, mm, fr);
                    const T wv = s_w[q];
                    wa[u] = wv * clamp0(fma(-fr, wv, T(1)));   // bin floor(beta)
                    wb[u] = wv * clamp0(fma(fr, wv, s_w1[q]));  // bin floor(beta) + 1
                    bin[u] = s_idx[q].x + mm;
                }
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    Operands<T> op[PER];
#pragma unroll
                    for (int u = 0; u < PER; ++u) {
                        const int v = s_idx[blk + min(warp + u * kSmallWarps, nb - 1)].y, b = bin[u];
                        op[u].wa = wa[u];
                        op[u].wb = wb[u];
                        if constexpr (F32) {
                            const float *row =
                                a.Y + (size_t)grp * a.group_stride + ((long long)v * a.pitch + b) * KB + k;
                            op[u].y0 = (unsigned)b < (unsigned)a.B ? __ldg(row) : 0.0f;
                            op[u].y1 = (unsigned)(b + 1) < (unsigned)a.B ? __ldg(row + KB) : 0.0f;
                        } else {
                            const double2 p = __ldg(reinterpret_cast<const double2 *>(a.Y) +
                                                    (size_t)(k0 + k) * a.group_stride + (size_t)v * a.pitch +
                                                    min(max(b, -2), a.B) + 2);
                            op[u].y0 = p.x;
                            op[u].y1 = p.y;
                        }
                    }
                    if (blk > 0 || k > 0) __syncthreads();  // the previous operands have been added
#pragma unroll
                    for (int u = 0; u < PER; ++u)
                        if (warp + u * kSmallWarps < nb) s_op[warp + u * kSmallWarps][lane] = op[u];
                    __syncthreads();
                    if (warp < SPLIT) {
#pragma unroll 4
                        for (int q = warp; q < nb; q += SPLIT) {
                            const Operands<T> o = s_op[q][lane];
                            acc[k] = fma(o.wa, o.y0, fma(o.wb, o.y1, acc[k]));
                        }
                    }
                }
            }
        }
        if (warp < SPLIT) {
#pragma unroll
            for (int k = 0; k < KB; ++k) red[warp][k][lane] = acc[k];
        }
        __syncthreads();
        const int i = i0 + ty, j = j0 + tx;
        if (warp < KB && i < N && j < N && k0 + warp < a.kend) {
            T s = red[0][warp][lane];
#pragma unroll
            for (int q = 1; q < SPLIT; ++q) s += red[q][warp][lane];
            a.X[(size_t)(k0 + warp) * a.img_stride + (size_t)f * N * N + (size_t)i * N + j] = s;
        }
        __syncthreads();  // red is rewritten by the next item (which has no other barrier if its frame is empty)
    }
}

template <typename T, int KB> cudaError_t launch_small(const SmallArgs<T> &a, const Handle &h, int split)
{
    const long long items = (long long)a.ngroups * a.F * a.tps * a.tps * (kTile / kSmallRows);
    constexpr int NT = 32 * kSmallWarps;
    if (split > 2)
        launch_chained(k_adj_small<T, KB, 4>, persistent_grid(k_adj_small<T, KB, 4>, NT, 0, items, h.num_sms), NT, 0, h.stream, a);
    else
        launch_chained(k_adj_small<T, KB, 2>, persistent_grid(k_adj_small<T, KB, 2>, NT, 0, items, h.num_sms), NT, 0, h.stream, a);
    return cudaGetLastError();
}

template <typename T> cudaError_t launch_small(const SmallArgs<T> &a, const Handle &h, int width, int split)
{
    switch (width) {
    case 1: return launch_small<T, 1>(a, h, split);
    case 2: return launch_small<T, 2>(a, h, split);
    case 4: return launch_small<T, 4>(a, h, split);
    default: return launch_small<T, 8>(a, h, split);
    }
}

bool small_image(const Handle &h, int groups)
{
    const long long tps = (h.N + kTile - 1) / kTile;
    return h.N <= kSmallN && (long long)groups * h.F * tps * tps * (kTile / kSmallRows) <= 3LL * h.num_sms;
}

template <typename T> SmallArgs<T> small_args(const Handle &h, T *X, int k0, int groups, int kend, const int *skip)
{
    SmallArgs<T> a{};
    a.vg = h.d_views;
    a.fstart = h.d_fstart;
    a.fcount = h.d_fcount;
    a.N = h.N;
    a.B = h.B;
    a.F = h.F;
    a.tps = (h.N + kTile - 1) / kTile;
    a.kbase = k0;
    a.ngroups = groups;
    a.kend = kend;
    a.X = X;
    a.img_stride = (long long)h.F * h.N * h.N;
    a.skip = skip;
    return a;
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
cudaError_t adjoint32(const Handle &h, float *X, int batch, int kb, int split, int layout_batch, const int *skip)
{
    AdjArgs a{};
    a.vg = h.d_views;
    a.fstart = h.d_fstart;
    a.fcount = h.d_fcount;
    a.N = h.N;
    a.B = h.B;
    a.V = h.V;
    a.F = h.F;
    a.tps = (h.N + kAdjTile - 1) / kAdjTile;
    a.Pq = sino_pitch(h.B);
    a.X = X;
    a.img_stride = (long long)h.F * h.N * h.N;
    a.kend = batch;
    a.skip = skip;
    SinoGroup g[2];
    const int ng = sino_groups(layout_batch, kb, g);
    // (the form and the CTAs per tile follow the laid-out batch: the first sinograms
    // of a larger one get the bits they got in its own product)
    for (int q = 0; q < ng; ++q) {
        if (g[q].k0 >= batch) break;
        a.kbase = g[q].k0;
        a.ngroups = std::min(g[q].count, (batch - g[q].k0 + g[q].width - 1) / g[q].width);
        a.group_stride = (long long)h.V * a.Pq * g[q].width;
        a.YI = (const float *)h.d_yp + (size_t)g[q].k0 * h.V * a.Pq;
        a.rowflag = h.d_rowflag + (size_t)g[q].first * h.V;
        cudaError_t e;
        if (small_image(h, g[q].count)) {
            SmallArgs<float> b = small_args<float>(h, X, a.kbase, a.ngroups, batch, skip);
            b.Y = a.YI;
            b.pitch = a.Pq;
            b.group_stride = a.group_stride;
            e = launch_small<float>(b, h, g[q].width, split);
            if (e != cudaSuccess) return e;
            continue;
        }
        const int alone = g[q].width == 1 ? 20 : (g[q].width == 2 ? 12 : 0);  // views (see adj_cluster_size)
        a.segs = adj_segs(h, (long long)g[q].count * h.F * a.tps * a.tps, split, 8, alone);
        switch (g[q].width) {
        case 1: e = launch_cluster(k_adj_tile<1>, a, h, adj_smem<1>(true)); break;
        case 2: e = launch_cluster(k_adj_tile<2>, a, h, adj_smem<2>(true)); break;
        case 4: e = launch_cluster(k_adj_tile<4>, a, h, adj_smem<4>(true)); break;
        default: e = launch_cluster(k_adj_tile<8>, a, h, adj_smem<8>(true)); break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adjoint64(const Handle &h, double *X, int batch, int kb, int split, int layout_batch, const int *skip)
{
    Adj64Args a{};
    a.vg = h.d_views;
    a.fstart = h.d_fstart;
    a.fcount = h.d_fcount;
    a.N = h.N;
    a.B = h.B;
    a.F = h.F;
    a.tps = (h.N + kTile - 1) / kTile;
    a.Pb = h.Pb;
    a.YP = (const double2 *)h.d_yp;
    a.ysino_stride = (long long)h.V * h.Pb;
    a.X = X;
    a.img_stride = (long long)h.F * h.N * h.N;
    a.kend = batch;
    a.skip = skip;
    int k = 0;
    for (int width : {8, 4, 2, 1}) {  // the groups of the laid-out batch, as in adjoint32
        if (width > kb) continue;
        if (k >= batch) break;
        const int groups = (layout_batch - k) / width;
        if (groups == 0) continue;
        a.kbase = k;
        a.ngroups = std::min(groups, (batch - k + width - 1) / width);
        cudaError_t e;
        if (small_image(h, groups)) {
            SmallArgs<double> b = small_args<double>(h, X, k, a.ngroups, batch, skip);
            b.Y = (const double *)h.d_yp;
            b.pitch = h.Pb;
            b.group_stride = a.ysino_stride;
            e = launch_small<double>(b, h, width, split);
            if (e != cudaSuccess) return e;
            k += groups * width;
            continue;
        }
        a.segs = adj_segs(h, (long long)groups * h.F * a.tps * a.tps, split, 3);
        switch (width) {
        case 1: e = launch_cluster(k_adj64<1>, a, h, 0); break;
        case 2: e = launch_cluster(k_adj64<2>, a, h, 0); break;
        case 4: e = launch_cluster(k_adj64<4>, a, h, 0); break;
        default: e = launch_cluster(k_adj64<8>, a, h, 0); break;
        }
        if (e != cudaSuccess) return e;
        k += groups * width;
    }
    return cudaSuccess;
}

}  // namespace

int adj_kb(const Handle &h, int batch)
{
    if (h.precision || h.fan_D > 0.0) return h.tune.adj_kb;
    SinoGroup g[2];
    sino_groups(batch, h.tune.adj_kb, g);
    if (small_image(h, g[0].count)) return h.tune.adj_kb;  // the small form's sums are the same at any width
    const long long tps = (h.N + kAdjTile - 1) / kAdjTile;
    return adj_group_width(h.tune.adj_kb, batch, tps * tps, h.V, h.num_sms);
}

template <typename T>
cudaError_t launch_adjoint(const Handle &h, T *X, int batch, int kb, int split, int layout_batch, const int *skip)
{
    if (h.fan_D > 0.0) return launch_fan_adjoint<T>(h, X, batch, kb, split, layout_batch, skip);
    if constexpr (std::is_same<T, float>::value) return adjoint32(h, X, batch, kb, split, layout_batch, skip);
    else return adjoint64(h, X, batch, kb, split, layout_batch, skip);
}

template cudaError_t launch_adjoint<float>(const Handle &, float *, int, int, int, int, const int *);
template cudaError_t launch_adjoint<double>(const Handle &, double *, int, int, int, int, const int *);

}  // namespace ctgb
