// Fan-beam form of the Joseph operator (sm_103a).
//
// Geometry (the fan-beam CT of Sec. 6.2; the paper gives no distances, so
// they are a reading): a point source at distance D from the rotation
// centre and a flat detector rescaled to the line through the centre, on
// which bin b keeps the parallel-beam centre s_b = b - (B-1)/2 + delta_v.
// With e = (cos, sin) and t = (-sin, cos), the source is S = -D t, bin b is
// P_b = s_b e, and ray (v,b) has direction r = P_b - S = s_b e + D t.  As D
// grows the rays become the parallel-beam rays.
//
// Every ray is marched like a parallel-beam ray, but with its own line: rows
// when |r_x| <= |r_y| (x(y) = A + C y, C = r_x / r_y, A = P_x - P_y C),
// columns otherwise (y(x) = A + C x, C = r_y / r_x, A = P_y - P_x C), weight
// sqrt(1 + C^2).  In march coordinates q(r) = q_h + (r - h) qr with
// q_h = h + A (rows) or h - A (columns), qr = -C, carried in the same 64-bit
// fixed point as the parallel-beam lines.  The geometry turns rigidly with
// theta (dr/dtheta = (-r_y, r_x), dP_b/dtheta = s_b t), so
// dq/dtheta = g0 + r gr with gr = -dC/dtheta, g0 = +-dA/dtheta + h dC/dtheta,
// and dw/dtheta = C dC/dtheta / w.  An offset delta_v moves every bin centre
// along e (ds_b/ddelta = 1, the source stays): dq/ddelta = s0 + r sr with
// sr = -dC/ds, s0 = +-dA/ds + h dC/ds, and dw/ddelta = C dC/ds / w.
//
//   k_fan_table  per-ray table (fixed-point line, weight, derivative
//                constants, march range) and per-view record of the transpose
//                (FP32 constants, bin ranges of row- and column-marched rays)
//                from the view table, for the views rebuilt since
//   k_ray_fan    SPLIT warps (row segments) per 32 bins of one view: forward
//                (KB images), JVP, VJP and Gauss-Newton terms, each lane on
//                its own line
//   k_fan_sino   sinograms interleaved in blocks of 8 for the transpose
//   k_adj_fan_tile, k_adj_fan (FP32, FP64)
//                exact transpose in gather form: a pixel takes, per view,
//                the rays whose fixed-point sample at its row (row-marched
//                rays) or column (column-marched rays) falls in its
//                interpolation cell; the candidates come from the projective
//                inverse of the pixel's neighbourhood and are then tested
//                with the very values the forward uses, so the matrix
//                entries are those of the forward.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "ct_device.cuh"
#include "ct_internal.cuh"

namespace ctgb {
namespace {

template <typename T> struct __align__(16) FanRay {
    long long Qc, Qh;  // q(r) = (Qc + (2r - (N-1)) Qh) / 2^48
    T w, dw, g0, gr;   // weight, d w / d theta, dq/dtheta = g0 + r gr
    float rlo, rhi;    // march indices with -1 < q < N lie in [rlo, rhi] (two indices of margin)
    int mode;          // 0: rows of X, 1: rows of X^T (columns)
    int pad;
    T dws, s0, sr;     // d w / d delta, dq/ddelta = s0 + r sr
};

// The fields of a ray the transpose's candidate search reads, in a table of
// their own after the FanRay table (24 bytes a ray instead of 64: the search
// touches a few records per pixel and view, scattered over the whole table).
template <typename T> struct FanLine {
    long long Qc, Qh;
    T w;
};
template <typename T> __host__ __device__ inline FanLine<T> *fan_lines(void *rays, long long nrays)
{
    return reinterpret_cast<FanLine<T> *>(reinterpret_cast<unsigned char *>(rays) + nrays * sizeof(FanRay<T>));
}

// Per view: FP32 constants of the transpose's candidate search and the bin
// ranges of the two march axes (the ray direction turns monotonically with
// s_b over a fan narrower than 90 degrees, so the axis changes at most once:
// bins [0, split) march along mode0, bins [split, B) along the other axis).
struct __align__(16) FanView {
    float c, sn, sb0, iD;
    int mode0, split, gen, pad;
};

// One CTA per view: nothing when the view record it was built from is current
// (one generation stamp per view; a stamp per ray made every call read the
// whole table), else the view's rays and its record.
template <typename T>
__global__ void __launch_bounds__(128) k_fan_table(const ViewGeo *__restrict__ vg, int V, int B, int N, double D,
                                                   FanRay<T> *__restrict__ rays, FanLine<T> *__restrict__ lines,
                                                   FanView *__restrict__ views, const int *__restrict__ skip)
{
    chain_wait();
    if (skip && *skip) return;
    __shared__ int s_mode0, s_split;
    const double h = 0.5 * (N - 1);
    for (int v = blockIdx.x; v < V; v += gridDim.x) {
        const ViewGeo &g = vg[v];
        if (views[v].gen == g.gen) continue;  // uniform
        __syncthreads();  // every thread has read the stamp and the previous view's record is written
        if (threadIdx.x == 0) s_split = B;
        for (int b = threadIdx.x; b < B; b += blockDim.x) {
            const size_t idx = (size_t)v * B + b;
            const double c = g.c, sn = g.s, s = g.sb0d + (double)b;
            const double rx = s * c - D * sn, ry = s * sn + D * c;
            const double px = s * c, py = s * sn, dpx = -s * sn, dpy = s * c;
            double C, A, dC, dA, qh, g0, dCs, s0;
            int mode;
            if (fabs(rx) <= fabs(ry)) {
                mode = 0;
                C = rx / ry;
                A = px - py * C;
                dC = -(1.0 + C * C);
                dA = dpx - C * dpy - py * dC;
                qh = h + A;
                g0 = dA + h * dC;
                dCs = (c * ry - sn * rx) / (ry * ry);  // d/ds of C and A: P_b and r move by e
                s0 = (c - C * sn - py * dCs) + h * dCs;
            } else {
                mode = 1;
                C = ry / rx;
                A = py - px * C;
                dC = 1.0 + C * C;
                dA = dpy - C * dpx - px * dC;
                qh = h - A;
                g0 = -dA + h * dC;
                dCs = (sn * rx - c * ry) / (rx * rx);
                s0 = -(sn - C * c - px * dCs) + h * dCs;
            }
            const double qr = -C;
            const double w = sqrt(1.0 + C * C);
            FanRay<T> R;
            R.Qc = __double2ll_rn(qh * kFixScale);
            R.Qh = __double2ll_rn(qr * 0.5 * kFixScale);
            R.w = (T)w;
            R.dw = (T)(C * dC / w);
            R.g0 = (T)g0;
            R.gr = (T)(-dC);
            R.dws = (T)(C * dCs / w);
            R.s0 = (T)s0;
            R.sr = (T)(-dCs);
            R.mode = mode;
            R.pad = 0;
            if (fabs(qr) < 1e-12) {
                const bool in = qh > -1.0 && qh < (double)N;
                R.rlo = in ? 0.0f : (float)N;
                R.rhi = in ? (float)(N - 1) : -1.0f;
            } else {
                const double ra = h + (-1.0 - qh) / qr, rb = h + ((double)N - qh) / qr;
                R.rlo = (float)fmin(fmax(fmin(ra, rb) - 2.0, 0.0), (double)N);
                R.rhi = (float)fmax(fmin(fmax(ra, rb) + 2.0, (double)(N - 1)), -1.0);
            }
            rays[idx] = R;
            FanLine<T> L;
            L.Qc = R.Qc;
            L.Qh = R.Qh;
            L.w = R.w;
            lines[idx] = L;
            if (b == 0) s_mode0 = R.mode;
        }
        __syncthreads();
        for (int b = threadIdx.x; b < B; b += blockDim.x)  // the thread's own rays, written above
            if (rays[(size_t)v * B + b].mode != s_mode0) atomicMin(&s_split, b);
        __syncthreads();
        if (threadIdx.x == 0) {
            FanView f;
            f.c = (float)g.c;
            f.sn = (float)g.s;
            f.sb0 = (float)g.sb0d;
            f.iD = (float)(1.0 / D);
            f.mode0 = s_mode0;
            f.split = s_split;
            f.gen = g.gen;
            f.pad = 0;
            views[v] = f;
        }
    }
}

// One CTA = SPLIT warps on one work item: 32 consecutive bins of one view
// (and one batch group of KB images for the forward).  The warps march
// consecutive segments of the warp-union row range; their sums are added in
// segment order in shared memory and warp 0 writes the result.
template <typename T, int MODE, int KB, int SPLIT, bool OFFS>
__global__ void __launch_bounds__(32 * SPLIT) k_ray_fan(RayArgs<T> a, const FanRay<T> *__restrict__ rays)
{
    chain_wait();
    using P2 = pair_t<T>;
    constexpr bool F32 = std::is_same<T, float>::value;
    constexpr int NACC = (MODE == kFwd) ? KB : (OFFS ? 3 : 2);
    __shared__ T red[SPLIT > 1 ? SPLIT : 1][NACC][32];
    const int lane = threadIdx.x & 31;
    const int seg = threadIdx.x >> 5;
    const int N = a.N;
    const long long total = (long long)a.ngroups * a.V * a.nchunks;
    if (a.skip && *a.skip) return;
    for (long long item = blockIdx.x; item < total; item += gridDim.x) {  // CTA-uniform
        const int chunk = (int)(item % a.nchunks);
        const long long t = item / a.nchunks;
        const int v = (int)(t % a.V);
        const int grp = (int)(t / a.V);
        if (MODE == kGn && a.view_mask && a.view_mask[v] == 0) continue;  // CTA-uniform
        const int b = chunk * kChunk + lane;
        const bool active = b < a.B;
        const FanRay<T> R = rays[(size_t)v * a.B + (active ? b : a.B - 1)];
        const int k0 = a.kbase + grp * KB;
        int rlo = active ? (int)floorf(R.rlo) : N, rhi = active ? (int)ceilf(R.rhi) : -1;
        rlo = __reduce_min_sync(0xffffffffu, rlo);
        rhi = __reduce_max_sync(0xffffffffu, rhi);
        const int per = rhi >= rlo ? (rhi - rlo + SPLIT) / SPLIT : 0;
        const int r0 = rlo + seg * per, r1 = min(rhi, r0 + per - 1);
        T acc[NACC];
#pragma unroll
        for (int k = 0; k < NACC; ++k) acc[k] = T(0);
        const P2 *img = (R.mode ? a.PT : a.PX) + ((size_t)a.vg[v].frame * N + r0) * a.Pp + (size_t)k0 * a.pimg_stride;
        const long long dQ = 2 * R.Qh;
        long long Q = R.Qc + (long long)(2 * r0 - (N - 1)) * R.Qh;
        const unsigned pp = (unsigned)a.Pp, lim = (unsigned)(N + 2);
        constexpr int U = KB == 1 ? 8 : 4;  // (J^T of one image, 256^2 / 180 views: 26.2 us a call with 4, 21.4 with 8)
        // rows in blocks of U whose loads are all issued first; the last block's
        // missing rows read nothing and add exact zeros
        auto block = [&](auto whole, int r, int rows) {
            constexpr bool WHOLE = decltype(whole)::value;
            unsigned idx[U];
            T f[U];
            P2 p[U][KB];
            ray_cells<T, U, false>(Q, dQ, lim, idx, f);
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    if (WHOLE || u < rows) p[u][k] = __ldg(img + (idx[u] + u * pp) + (size_t)k * a.pimg_stride);
                    else p[u][k].x = p[u][k].y = T(0);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!F32 && !WHOLE && u >= rows) break;  // FP64 products are dear (uniform)
                const T fu = ray_frac<T, U>(Q, dQ, f, u);
                if constexpr (MODE == kFwd) {
                    const T omf = T(1) - fu;
#pragma unroll
                    for (int k = 0; k < KB; ++k) acc[k] = fma(omf, p[u][k].x, fma(fu, p[u][k].y, acc[k]));
                } else {
                    // acc[0] = sum of interpolated values, acc[1] = sum slope * dq/dtheta,
                    // acc[2] (offsets) = sum slope * dq/ddelta
                    const T d = p[u][0].y - p[u][0].x;
                    acc[0] += fma(fu, d, p[u][0].x);
                    acc[1] = fma(d, fma((T)(r + u), R.gr, R.g0), acc[1]);
                    if constexpr (OFFS) acc[NACC - 1] = fma(d, fma((T)(r + u), R.sr, R.s0), acc[NACC - 1]);
                }
            }
            img += (size_t)U * pp;
            Q += (long long)U * dQ;
        };
        int r = r0;
        for (; r + U - 1 <= r1; r += U) block(std::true_type(), r, U);
        if (r <= r1) block(std::false_type(), r, r1 - r + 1);
        if constexpr (SPLIT > 1) {
#pragma unroll
            for (int k = 0; k < NACC; ++k) red[seg][k][lane] = acc[k];
            __syncthreads();
            if (seg == 0) {
#pragma unroll
                for (int k = 0; k < NACC; ++k) {
                    T sum = red[0][k][lane];
#pragma unroll
                    for (int q = 1; q < SPLIT; ++q) sum += red[q][k][lane];
                    acc[k] = sum;
                }
            }
        }
        if (seg == 0) {
            if constexpr (MODE == kFwd) {
                if (active) {
#pragma unroll
                    for (int k = 0; k < KB; ++k)
                        a.Y[(size_t)(k0 + k) * a.sino_stride + (size_t)v * a.B + b] = R.w * acc[k];
                }
            } else {
                // one image per lane in the derivative modes: image k0 of the batch
                const size_t img = (size_t)k0, vb = (size_t)v * a.B + b;
                const T jt = fma(R.dw, acc[0], R.w * acc[1]);
                T jd = T(0);
                if constexpr (OFFS) jd = fma(R.dws, acc[0], R.w * acc[NACC - 1]);
                if constexpr (MODE == kJvp) {
                    if (active) {
                        T out = (T)a.dtheta[img * a.dir_stride + v] * jt;
                        if constexpr (OFFS) out = fma((T)a.ddelta[img * a.dir_stride + v], jd, out);
                        a.Y[img * a.sino_stride + vb] = out;
                    }
                } else if constexpr (MODE == kVjp) {
                    double pt = 0.0, pd = 0.0;
                    if (active) {
                        const T rr = a.R[img * a.r_stride + vb];
                        pt = (double)(rr * jt);
                        if constexpr (OFFS) pd = (double)(rr * jd);
                    }
                    double part[OFFS ? 2 : 1];
                    part[0] = pt;
                    if constexpr (OFFS) part[1] = pd;
                    constexpr int PER = OFFS ? 16 : 32;
                    const double sum = warp_sums(part, lane);
                    if (lane % PER == 0)
                        a.partial[img * a.part_stride + ((size_t)v * a.nchunks + chunk) * 4 + lane / PER] = sum;
                } else {  // kGn
                    double pg = 0.0, pj = 0.0, pf = 0.0, pr = 0.0;
                    if (active) {
                        const T hx = R.w * acc[0];
                        const T bb = a.R[img * a.r_stride + vb];
                        const T rr = hx - bb;
                        if (a.res) a.res[img * a.sino_stride + vb] = rr;
                        pg = (double)rr * (double)jt;
                        pj = (double)jt * (double)jt;
                        pf = (double)rr * (double)rr;
                        pr = fabs((double)rr) * (fabs((double)hx) + fabs((double)bb));
                    }
                    double part[4] = {pg, pj, pf, pr};
                    const double sum = warp_sums(part, lane);
                    if (lane % 8 == 0)
                        a.partial[img * a.part_stride + ((size_t)v * a.nchunks + chunk) * 4 + lane / 8] = sum;
                }
            }
        }
        if constexpr (SPLIT > 1) __syncthreads();  // red[] is reused by the next item
    }
}

// Detector coordinate of the point (x, y) for view (c, sn): the bin centre
// s of the ray through it, s = (x c + y sn) / (1 + (y c - x sn) / D).  Fast
// division: the candidate range keeps a margin of 0.05 bins.
__device__ __forceinline__ float fan_s(float x, float y, float c, float sn, float iD)
{
    return __fdividef(x * c + y * sn, 1.0f + (y * c - x * sn) * iD);
}

// YI[k / 8][v][b][k % 8] = Y[k][v][b] for k < nsino
template <typename T>
__global__ void k_fan_sino(const T *__restrict__ Y, T *__restrict__ YI, long long m, int nsino,
                           const int *__restrict__ skip)
{
    chain_wait();
    if (skip && *skip) return;
    const long long total = (long long)nsino * m;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(idx / m);
        const long long e = idx - (long long)k * m;
        YI[((long long)(k >> 3) * m + e) * 8 + (k & 7)] = Y[idx];
    }
}

// ---------------------------------------------------------------------------
// FP32 transpose
// ---------------------------------------------------------------------------
constexpr int kFanWin = 64;      // rays of a view staged at a time
constexpr int kFanVB = 4;        // views per staged block: one staged ray per thread
constexpr int kFanCap = 128;     // views whose tile constants are staged at a time
constexpr int kFanLow = kFracBits - 23;  // bits of a line's fraction below those of the forward's

struct FanTileArgs {
    const FanLine<float> *lines;
    const FanView *views;
    const int *fstart, *fcount;
    int N, B, F, tps;
    const float *YI;             // [k / 8][V][B][8]
    long long yi_stride;         // floats per block of 8 sinograms
    int kbase, ngroups, kend;
    float *X;
    long long img_stride;
    int segs;
    const int *skip;
};

struct __align__(16) FanTileView {
    float c, sn, sb0, iD;
    int mode0, split, start, count;  // rays [start, start + count) can touch the tile
    int v, pad[3];
};

// A ray near the tile: its coordinate at the tile's centre row (column, for
// column-marched rays) relative to the centre pixel and its slope, each as the
// part above the last kFanLow bits and those bits: all 48 bits of the line's
// fraction in 32-bit words, so that the sum at any row of the tile is exact.
struct __align__(16) FanTileRay {
    int ph, pl, sh, sl;
};

template <int KB> struct FanSums {
    float v[KB];
    __device__ void clear()
    {
#pragma unroll
        for (int k = 0; k < KB; ++k) v[k] = 0.0f;
    }
    __device__ float get(int k) const { return v[k]; }
    __device__ __forceinline__ void add(float w, const float *y)
    {
#pragma unroll
        for (int k = 0; k < KB; ++k) v[k] = fmaf(w, y[k], v[k]);
    }
};
template <int KB> struct FanSumsPacked {
    f32x2 v[KB / 2];
    __device__ void clear()
    {
#pragma unroll
        for (int k = 0; k < KB / 2; ++k) v[k] = 0ull;
    }
    __device__ float get(int k) const { return half2f(v[k >> 1], k & 1); }
    __device__ __forceinline__ void add(float w, const float *y)
    {
        const f32x2 ww = pack2(w, w);
#pragma unroll
        for (int g = 0; g < KB / 4; ++g) {
            const ulonglong2 u = *reinterpret_cast<const ulonglong2 *>(y + 4 * kFanWin * g);
            v[2 * g] = fma2(ww, u.x, v[2 * g]);
            v[2 * g + 1] = fma2(ww, u.y, v[2 * g + 1]);
        }
    }
};
template <> struct FanSums<4> : FanSumsPacked<4> {};
template <> struct FanSums<8> : FanSumsPacked<8> {};

// One CTA = one 16 x 16 pixel tile of one frame, one of `segs` view subsets
// and KB sinograms.  What bounds the transpose is the search: per pixel and
// view two projective bounds and two or three candidate rays, each tested with
// its own line.  With the rays' full-range lines read from global memory it
// took 250 instructions per warp and view, waiting on loads (152 us for 256^2 /
// 180 views, 8 sinograms).  Here the rays that can touch the tile (between the
// projections of the corners of its one-pixel neighbourhood) are staged once
// per tile and view with their lines relative to its centre, their sinogram
// bins beside them; the next block's lines are loaded and its bins copied while
// the current one is read: 99 us.  The staged lines keep every bit, so the
// cell, the fraction and the weight are the forward's own (with 25 bits of
// fraction kept instead of 48: 92 us, weights up to 2^-23 off).
template <int KB>
__global__ void __launch_bounds__(256) k_adj_fan_tile(FanTileArgs a)
{
    chain_wait();
    namespace cg = cooperative_groups;
    __shared__ FanTileView s_view[kFanCap];
    __shared__ FanTileRay s_ray[2][kFanVB][kFanWin];
    __shared__ float s_w[2][kFanVB][kFanWin];
    // (8 sinograms as two arrays of 4, so that a quarter-warp's 16-byte loads meet no bank twice)
    constexpr int W = KB >= 4 ? 4 : KB;
    __shared__ __align__(16) float s_y[2][kFanVB][KB / W][kFanWin][W];
    __shared__ int s_max;
    float *red = &s_y[0][0][0][0][0];  // [KB][256], after the views
    const int tid = threadIdx.x;
    const int tx = (tid & (kTile - 1)) - kTile / 2, ty = tid / kTile - kTile / 2;  // relative to the centre pixel
    const int tiles = a.tps * a.tps;
    const int segs = a.segs;
    const int total = a.ngroups * a.F * tiles * segs;
    const int N = a.N;
    const float h = 0.5f * (float)(N - 1);
    constexpr int one = 1 << (kFracBits - kFanLow), low = (1 << kFanLow) - 1;
    if (a.skip && *a.skip) return;
    for (int item = blockIdx.x; item < total; item += gridDim.x) {  // whole clusters
        const int seg = item % segs;
        int t2 = item / segs;
        const int tile = t2 % tiles;
        t2 /= tiles;
        const int f = t2 % a.F;
        const int grp = t2 / a.F;
        const int ic = (tile / a.tps) * kTile + kTile / 2, jc = (tile % a.tps) * kTile + kTile / 2;
        const int k0 = a.kbase + grp * KB;
        const float x = (float)(jc + tx) - h, y = h - (float)(ic + ty);
        const float *yg = a.YI + (size_t)(k0 >> 3) * a.yi_stride + (k0 & 7);
        const int vs = a.fstart[f], vc = a.fcount[f];
        const int nv = vc > seg ? (vc - seg + segs - 1) / segs : 0;
        FanSums<KB> acc;
        acc.clear();
        for (int cb = 0; cb < nv; cb += kFanCap) {
            const int nc = min(kFanCap, nv - cb);
            __syncthreads();
            if (tid == 0) s_max = 0;
            __syncthreads();
            for (int q = tid; q < nc; q += 256) {
                const int v = vs + seg + (cb + q) * segs;
                const FanView fv = a.views[v];
                FanTileView w;
                w.c = fv.c;
                w.sn = fv.sn;
                w.sb0 = fv.sb0;
                w.iD = fv.iD;
                w.mode0 = fv.mode0;
                w.split = fv.split;
                w.v = v;
                // (not beyond the image's own one-pixel neighbourhood, where the projection is regular)
                const float xl = (float)(jc - kTile / 2 - 1) - h, xr = (float)min(jc + kTile / 2, N) - h;
                const float yt = h - (float)(ic - kTile / 2 - 1), yb = h - (float)min(ic + kTile / 2, N);
                const float s1 = fan_s(xl, yt, fv.c, fv.sn, fv.iD), s2 = fan_s(xr, yt, fv.c, fv.sn, fv.iD);
                const float s3 = fan_s(xl, yb, fv.c, fv.sn, fv.iD), s4 = fan_s(xr, yb, fv.c, fv.sn, fv.iD);
                const int lo = max(0, (int)floorf(fminf(fminf(s1, s2), fminf(s3, s4)) - fv.sb0 - 0.1f));
                const int hi = min(a.B - 1, (int)ceilf(fmaxf(fmaxf(s1, s2), fmaxf(s3, s4)) - fv.sb0 + 0.1f));
                w.start = lo;
                w.count = max(0, hi - lo + 1);
                s_view[q] = w;
                if (w.count > 0) atomicMax(&s_max, (w.count + kFanWin - 1) / kFanWin);
            }
            __syncthreads();
            const int nwin = s_max;  // windows of kFanWin rays (one unless the tile is close to the source)
            const int nblk = (nc + kFanVB - 1) / kFanVB;
            // one staged ray per thread and block
            const int sq = tid / kFanWin, sr = tid % kFanWin;
            FanLine<float> line;
            bool have = false;
            auto fetch = [&](int u, int buf) {  // block u: window u / nblk of views (u % nblk) * kFanVB ...
                const int q = (u % nblk) * kFanVB + sq, off = (u / nblk) * kFanWin + sr;
                have = q < nc && off < s_view[min(q, nc - 1)].count;
                if (!have) return;
                const FanTileView &w = s_view[q];
                const size_t bin = (size_t)w.v * a.B + w.start + off;
                line = a.lines[bin];
                const float *src = yg + bin * 8;
                const unsigned dst = (unsigned)__cvta_generic_to_shared(&s_y[buf][sq][0][sr][0]);
                if constexpr (KB >= 4) {
#pragma unroll
                    for (int g = 0; g < KB / 4; ++g)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16 * kFanWin * g),
                                     "l"(src + 4 * g)
                                     : "memory");
                } else {
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(dst), "l"(src), "n"(4 * KB)
                                 : "memory");
                }
            };
            auto store = [&](int u, int buf) {
                if (!have) return;
                const FanTileView &w = s_view[(u % nblk) * kFanVB + sq];
                const int bin = w.start + (u / nblk) * kFanWin + sr;
                const int mode = bin < w.split ? w.mode0 : 1 - w.mode0;
                const int r = mode ? jc : ic, m = mode ? ic : jc;
                const long long Q = line.Qc + (long long)(2 * r - (N - 1)) * line.Qh - ((long long)m << kFracBits);
                // rays that pass the tile at a distance are held at 20 pixels, out of reach of its pixels
                const long long far = 20LL << kFracBits;
                const long long P = min(max(Q, -far), far), S = 2 * line.Qh;
                FanTileRay R;
                R.ph = (int)(P >> kFanLow);
                R.pl = (int)P & low;
                R.sh = (int)(S >> kFanLow);
                R.sl = (int)S & low;
                s_ray[buf][sq][sr] = R;
                s_w[buf][sq][sr] = line.w;
            };
            const int nu = nblk * nwin;
            if (nu > 0) fetch(0, 0);
            cp_async_commit();
            for (int u = 0; u < nu; ++u) {
                const int buf = u & 1;
                store(u, buf);
                cp_async_wait0();
                // block u is staged, and every thread has finished block u - 1
                __syncthreads();
                if (u + 1 < nu) fetch(u + 1, buf ^ 1);
                cp_async_commit();
                const int q0 = (u % nblk) * kFanVB, w0 = (u / nblk) * kFanWin;
                for (int qq = 0; qq < kFanVB && q0 + qq < nc; ++qq) {
                    const FanTileView &w = s_view[q0 + qq];
                    const int wlo = w.start + w0, whi = min(w.start + w.count, wlo + kFanWin);  // rays staged
                    if (wlo >= whi) continue;
                    const float num = fmaf(x, w.c, y * w.sn), den = fmaf(fmaf(y, w.c, -x * w.sn), w.iD, 1.0f);
                    const float cD = w.c * w.iD, sD = w.sn * w.iD;
                    // rays marched along rows that sample row i inside (x - 1, x + 1), then rays
                    // marched along columns that sample column j inside (y - 1, y + 1)
#pragma unroll
                    for (int pass = 0; pass < 2; ++pass) {
                        const int mlo = max(wlo, w.mode0 == pass ? 0 : w.split);
                        const int mhi = min(whi, w.mode0 == pass ? w.split : a.B);
                        if (mlo >= mhi) continue;  // uniform
                        const float dn = pass == 0 ? w.c : w.sn, dd = pass == 0 ? -sD : cD;
                        const float s1 = __fdividef(num - dn, den - dd), s2 = __fdividef(num + dn, den + dd);
                        // margin 0.05 bins: the FP32 detector coordinates are off by < 0.01 bins for N <= 4096
                        const int blo = max(mlo, (int)ceilf(fminf(s1, s2) - w.sb0 - 0.05f));
                        const int bhi = min(mhi - 1, (int)floorf(fmaxf(s1, s2) - w.sb0 + 0.05f));
                        const int along = pass == 0 ? ty : tx, across = (pass == 0 ? tx : ty) * one;
                        for (int b = blo; b <= bhi; ++b) {
                            const FanTileRay R = s_ray[buf][qq][b - wlo];
                            // the ray's coordinate relative to the pixel, rounded down to 23 bits of fraction:
                            // exact, as |pl + along * sl| < 2^29 and |ph + along * sh| < 2^29
                            const int t = R.ph + along * R.sh + ((R.pl + along * R.sl) >> kFanLow) - across;
                            if (abs(t) < one) {  // (at -1 pixel the weight is 0)
                                const float g = __int_as_float(abs(t) | 0x3F800000);  // 1 + distance
                                acc.add(s_w[buf][qq][b - wlo] * (2.0f - g), &s_y[buf][qq][0][b - wlo][0]);
                            }
                        }
                    }
                }
            }
            cp_async_wait0();  // the last group is empty
        }
        __syncthreads();  // every thread is done with the staged bins
#pragma unroll
        for (int k = 0; k < KB; ++k) red[k * 256 + tid] = acc.get(k);
        cg::cluster_group cl = cg::this_cluster();
        if (segs > 1) cl.sync();
        else __syncthreads();
        // this CTA's share of the pixels, the segments added in order
        constexpr int OUT = KB * 256;
#pragma unroll 1
        for (int u = OUT / 32 * seg / segs * 32 + tid; u < OUT / 32 * (seg + 1) / segs * 32; u += 256) {
            float s;
            if (segs == 1) {
                s = red[u];
            } else {
                float part[kMaxSegs];
#pragma unroll
                for (int q = 0; q < kMaxSegs; ++q) part[q] = q < segs ? *cl.map_shared_rank(red + u, q) : 0.0f;
                s = part[0];
#pragma unroll
                for (int q = 1; q < kMaxSegs; ++q)
                    if (q < segs) s += part[q];
            }
            const int k = u >> 8, p = u & 255;
            const int i = ic - kTile / 2 + p / kTile, j = jc - kTile / 2 + p % kTile;
            if (i < N && j < N && k0 + k < a.kend)
                a.X[(size_t)(k0 + k) * a.img_stride + (size_t)f * N * N + (size_t)i * N + j] = s;
        }
        if (segs > 1) cl.sync();
        else __syncthreads();
    }
}

struct AdjFanArgs {
    const int *fstart, *fcount;
    int N, B, F, tps, kbase, ngroups;
    long long ysino_stride, img_stride;
    const int *skip;
};

// The KB values of one bin in the interleaved layout (16-byte loads from groups of 2 on).
template <int KB> __device__ __forceinline__ void load_bin(const double *p, double (&out)[KB])
{
    if constexpr (KB % 2 == 0) {
#pragma unroll
        for (int q = 0; q < KB / 2; ++q) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(p) + q);
            out[2 * q] = v.x;
            out[2 * q + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < KB; ++k) out[k] = __ldg(p + k);
    }
}

// FP64: one CTA = one 16 x 16 pixel tile of one frame and KB sinograms, SPLIT
// thread groups of 256: group g of a pixel sums the views vs + g, vs + g +
// SPLIT, ... of its frame in order; the groups' sums are added in group
// order in shared memory.
template <int KB, int SPLIT>
__global__ void __launch_bounds__(256 * SPLIT) k_adj_fan(AdjFanArgs a, const FanLine<double> *__restrict__ rays,
                                                         const FanView *__restrict__ views,
                                                         const double *__restrict__ YI, double *__restrict__ X)
{
    chain_wait();
    __shared__ double red[SPLIT > 1 ? SPLIT - 1 : 1][KB][256];
    const int pix = threadIdx.x & 255, grp_v = threadIdx.x >> 8;
    const int tx = pix & (kTile - 1), ty = pix / kTile;
    const int N = a.N;
    const int tiles = a.tps * a.tps;
    const long long total = (long long)a.ngroups * a.F * tiles;
    const float h = 0.5f * (float)(N - 1);
    if (a.skip && *a.skip) return;
    for (long long item = blockIdx.x; item < total; item += gridDim.x) {  // CTA-uniform
        const int tile = (int)(item % tiles);
        const long long t2 = item / tiles;
        const int f = (int)(t2 % a.F);
        const int grp = (int)(t2 / a.F);
        const int i = (tile / a.tps) * kTile + ty, j = (tile % a.tps) * kTile + tx;
        const int k0 = a.kbase + grp * KB;
        const bool inside = i < N && j < N;
        const float x = (float)j - h, y = h - (float)i;
        const long long Qrow = (long long)(2 * i - (N - 1)), Qcol = (long long)(2 * j - (N - 1));
        double acc[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) acc[k] = 0.0;
        const int vs = a.fstart[f], vc = a.fcount[f];
        for (int v = vs + grp_v; inside && v < vs + vc; v += SPLIT) {
            const FanView fv = views[v];
            const FanLine<double> *rv = rays + (size_t)v * a.B;
            // the KB sinograms of this group at bin b: KB consecutive values (KB divides 8, and a
            // group starts at a multiple of its width)
            const double *yv = YI + ((size_t)(k0 >> 3) * a.ysino_stride + (size_t)v * a.B) * 8 + (k0 & 7);
            // rays marched along rows that sample row i inside (x - 1, x + 1), then
            // rays marched along columns that sample column j inside (y - 1, y + 1)
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
                const int mlo = fv.mode0 == pass ? 0 : fv.split;
                const int mhi = fv.mode0 == pass ? fv.split : a.B;  // bins [mlo, mhi) march along this axis
                if (mlo >= mhi) continue;
                const float s1 = pass == 0 ? fan_s(x - 1.0f, y, fv.c, fv.sn, fv.iD) : fan_s(x, y - 1.0f, fv.c, fv.sn, fv.iD);
                const float s2 = pass == 0 ? fan_s(x + 1.0f, y, fv.c, fv.sn, fv.iD) : fan_s(x, y + 1.0f, fv.c, fv.sn, fv.iD);
                // margin 0.05 bins: the FP32 detector coordinates are off by < 0.01 bins for N <= 4096
                const int blo = max(mlo, (int)floorf(fminf(s1, s2) - fv.sb0 - 0.05f));
                const int bhi = min(mhi - 1, (int)ceilf(fmaxf(s1, s2) - fv.sb0 + 0.05f));
                const long long Qr = pass == 0 ? Qrow : Qcol;
                const int me = pass == 0 ? j : i;
                for (int b = blo; b <= bhi; ++b) {
                    const long long Q = rv[b].Qc + Qr * rv[b].Qh;
                    const int cell = cell_of(Q);
                    if (cell != me && cell != me - 1) continue;
                    const double fr = frac_of(Q, 0.0);
                    const double wt = rv[b].w * (cell == me ? 1.0 - fr : fr);
                    double yk[KB];
                    load_bin<KB>(yv + (size_t)b * 8, yk);
#pragma unroll
                    for (int k = 0; k < KB; ++k) acc[k] = fma(wt, yk[k], acc[k]);
                }
            }
        }
        if constexpr (SPLIT > 1) {
            if (grp_v > 0) {
#pragma unroll
                for (int k = 0; k < KB; ++k) red[grp_v - 1][k][pix] = acc[k];
            }
            __syncthreads();
            if (grp_v == 0) {
#pragma unroll
                for (int k = 0; k < KB; ++k)
#pragma unroll
                    for (int q = 0; q < SPLIT - 1; ++q) acc[k] += red[q][k][pix];
            }
        }
        if (grp_v == 0 && inside) {
#pragma unroll
            for (int k = 0; k < KB; ++k)
                X[(size_t)(k0 + k) * a.img_stride + (size_t)f * N * N + (size_t)i * N + j] = acc[k];
        }
        if constexpr (SPLIT > 1) __syncthreads();  // red[] is reused by the next item
    }
}

template <typename T, int MODE, int KB, int SPLIT, bool OFFS = false>
cudaError_t run_fan(const Handle &h, const RayArgs<T> &a)
{
    auto kern = k_ray_fan<T, MODE, KB, SPLIT, OFFS>;
    const long long items = (long long)a.ngroups * a.V * a.nchunks;
    const int grid = persistent_grid(kern, 32 * SPLIT, 0, items, h.num_sms);
    launch_chained(kern, grid, 32 * SPLIT, 0, h.stream, a, (const FanRay<T> *)h.d_rays);
    return cudaGetLastError();
}

template <typename T, int MODE, int KB, bool OFFS = false>
cudaError_t run_fan_split(const Handle &h, const RayArgs<T> &a, int split)
{
    switch (split) {
    case 1: return run_fan<T, MODE, KB, 1, OFFS>(h, a);
    case 2: return run_fan<T, MODE, KB, 2, OFFS>(h, a);
    default: return run_fan<T, MODE, KB, 4, OFFS>(h, a);
    }
}

template <int KB, int SPLIT> cudaError_t run_adj_fan(const Handle &h, const AdjFanArgs &a, double *X)
{
    auto kern = k_adj_fan<KB, SPLIT>;
    const long long items = (long long)a.ngroups * a.F * a.tps * a.tps;
    const int grid = persistent_grid(kern, 256 * SPLIT, 0, items, h.num_sms);
    launch_chained(kern, grid, 256 * SPLIT, 0, h.stream, a, fan_lines<double>(h.d_rays, (long long)h.V * h.B),
                                             (const FanView *)h.d_fanview, (const double *)h.d_yi, X);
    return cudaGetLastError();
}

template <int KB> cudaError_t run_adj_fan_split(const Handle &h, const AdjFanArgs &a, double *X, int split)
{
    return split >= 4 ? run_adj_fan<KB, 4>(h, a, X)
                      : (split >= 2 ? run_adj_fan<KB, 2>(h, a, X) : run_adj_fan<KB, 1>(h, a, X));
}

}  // namespace

// bytes a ray takes in the handle's table: its FanRay and its FanLine
size_t fan_ray_bytes(int precision)
{
    return precision ? sizeof(FanRay<double>) + sizeof(FanLine<double>) : sizeof(FanRay<float>) + sizeof(FanLine<float>);
}
size_t fan_view_bytes() { return sizeof(FanView); }

cudaError_t launch_fan_rays(const Handle &h, const int *skip)
{
    const long long n = (long long)h.V * h.B;
    const int grid = std::min(h.V, 16 * h.num_sms);
    if (h.precision)
        launch_chained(k_fan_table<double>, grid, 128, 0, h.stream, h.d_views, h.V, h.B, h.N, h.fan_D, (FanRay<double> *)h.d_rays,
                                                        fan_lines<double>(h.d_rays, n), (FanView *)h.d_fanview, skip);
    else
        launch_chained(k_fan_table<float>, grid, 128, 0, h.stream, h.d_views, h.V, h.B, h.N, h.fan_D, (FanRay<float> *)h.d_rays,
                                                       fan_lines<float>(h.d_rays, n), (FanView *)h.d_fanview, skip);
    return cudaGetLastError();
}

// split: warps per work item (row segments), 1, 2 or 4 (larger values take 4);
// offs: the JVP / VJP also carry the offset derivatives
template <typename T>
cudaError_t run_fan_ray(const Handle &h, const RayArgs<T> &a, int mode, int kb, int split, bool offs)
{
    switch (mode) {
    case kFwd:
        switch (kb) {
        case 1: return run_fan_split<T, kFwd, 1>(h, a, split);
        case 2: return run_fan_split<T, kFwd, 2>(h, a, split);
        case 4: return run_fan_split<T, kFwd, 4>(h, a, split);
        default: return run_fan_split<T, kFwd, 8>(h, a, split);
        }
    case kJvp: return offs ? run_fan_split<T, kJvp, 1, true>(h, a, split) : run_fan_split<T, kJvp, 1>(h, a, split);
    case kVjp: return offs ? run_fan_split<T, kVjp, 1, true>(h, a, split) : run_fan_split<T, kVjp, 1>(h, a, split);
    default: return run_fan_split<T, kGn, 1>(h, a, split);
    }
}

// kb: sinograms per thread (the candidate search of a pixel and view is
// shared by them); split: thread groups per pixel (view subsets).
cudaError_t fan_adjoint32(const Handle &h, float *X, int batch, int kb, int split, int layout_batch, const int *skip)
{
    FanTileArgs a{};
    a.lines = fan_lines<float>(h.d_rays, (long long)h.V * h.B);
    a.views = (const FanView *)h.d_fanview;
    a.fstart = h.d_fstart;
    a.fcount = h.d_fcount;
    a.N = h.N;
    a.B = h.B;
    a.F = h.F;
    a.tps = (h.N + kTile - 1) / kTile;
    a.YI = (const float *)h.d_yi;
    a.yi_stride = 8LL * h.V * h.B;
    a.X = X;
    a.img_stride = (long long)h.F * h.N * h.N;
    a.kend = batch;
    a.skip = skip;
    int k = 0;
    for (int width : {8, 4, 2, 1}) {  // the groups of the laid-out batch
        if (width > kb) continue;
        if (k >= batch) break;
        const int groups = (layout_batch - k) / width;
        if (groups == 0) continue;
        a.kbase = k;
        a.ngroups = std::min(groups, (batch - k + width - 1) / width);
        a.segs = adj_segs(h, (long long)groups * h.F * a.tps * a.tps, split, 8);
        cudaError_t e;
        switch (width) {
        case 1: e = launch_cluster(k_adj_fan_tile<1>, a, h, 0); break;
        case 2: e = launch_cluster(k_adj_fan_tile<2>, a, h, 0); break;
        case 4: e = launch_cluster(k_adj_fan_tile<4>, a, h, 0); break;
        default: e = launch_cluster(k_adj_fan_tile<8>, a, h, 0); break;
        }
        if (e != cudaSuccess) return e;
        k += groups * width;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_fan_adjoint(const Handle &h, T *X, int batch, int kb, int split, int layout_batch, const int *skip)
{
    if constexpr (std::is_same<T, float>::value) {
        return fan_adjoint32(h, X, batch, kb, split, layout_batch, skip);
    } else {
        AdjFanArgs a{};
        a.fstart = h.d_fstart;
        a.fcount = h.d_fcount;
        a.N = h.N;
        a.B = h.B;
        a.F = h.F;
        a.tps = (h.N + kTile - 1) / kTile;
        a.ysino_stride = (long long)h.V * h.B;  // per block of 8 interleaved sinograms, in bins
        a.img_stride = (long long)h.F * h.N * h.N;
        a.skip = skip;
        int k = 0;
        for (int width : {8, 4, 2, 1}) {
            if (width > kb) continue;
            const int groups = (batch - k) / width;
            if (groups == 0) continue;
            a.kbase = k;
            a.ngroups = groups;
            cudaError_t e;
            switch (width) {
            case 1: e = run_adj_fan_split<1>(h, a, X, split); break;
            case 2: e = run_adj_fan_split<2>(h, a, X, split); break;
            case 4: e = run_adj_fan_split<4>(h, a, X, split); break;
            default: e = run_adj_fan_split<8>(h, a, X, split); break;
            }
            if (e != cudaSuccess) return e;
            k += groups * width;
        }
        return cudaSuccess;
    }
}

template <typename T> cudaError_t launch_fan_sino(const Handle &h, const T *Y, int nsino, const int *skip)
{
    const long long m = (long long)h.V * h.B;
    const long long total = (long long)nsino * m;
    const int grid = (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, 8LL * h.num_sms));
    launch_chained(k_fan_sino<T>, grid, 256, 0, h.stream, Y, (T *)h.d_yi, m, nsino, skip);
    return cudaGetLastError();
}

template cudaError_t launch_fan_sino<float>(const Handle &, const float *, int, const int *);
template cudaError_t launch_fan_sino<double>(const Handle &, const double *, int, const int *);
template cudaError_t run_fan_ray<float>(const Handle &, const RayArgs<float> &, int, int, int, bool);
template cudaError_t run_fan_ray<double>(const Handle &, const RayArgs<double> &, int, int, int, bool);
template cudaError_t launch_fan_adjoint<float>(const Handle &, float *, int, int, int, int, const int *);
template cudaError_t launch_fan_adjoint<double>(const Handle &, double *, int, int, int, int, const int *);

}  // namespace ctgb
