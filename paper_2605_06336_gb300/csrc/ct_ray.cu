// Ray-driven kernels of the angle-dependent Joseph operator (sm_103a).
//
//   k_view_prep   per-view constants from (theta, delta), FP64 -> fixed point,
//                 and the view order of the ray kernels
//   k_pairs_img   X -> pair layouts of X and X^T (zero padded)
//   k_pairs_sino, k_interleave_sino  Y -> the layout of the FP64 / FP32 transpose
//   k_ray         one warp per 32 consecutive rays of one view (optionally
//                 SPLIT warps per ray group, each marching a row segment):
//                   FWD  Y = H X for KB images at once
//                   JVP  dY = J_theta dtheta (+ J_delta ddelta)
//                   VJP  J_theta^T r (and J_delta^T r), per-view partials
//                   GN   residual, J^T r, |J_v|^2, f_v partials
//   k_finalize    per-view sums of the partials in a fixed order
//
// Forward model: Joseph rule on a parallel-beam geometry with per-view angle
// theta_v and detector offset delta_v (the CT operator of Sec. 6.2, with the
// per-parameter derivatives H_{p_i} u of Alg. "UPDATE-PARAM").
#include <cuda_runtime.h>

#include <type_traits>

#include <algorithm>
#include <cmath>

#include "ct_device.cuh"
#include "ct_internal.cuh"

namespace ctgb {
namespace {

// ---------------------------------------------------------------------------
// per-view setup
// ---------------------------------------------------------------------------
// Joseph axis: one sample per image row iff |cos theta| >= |sin theta|, i.e.
// iff theta mod pi lies in [0, pi/4] or [3pi/4, pi).  The test runs on theta
// itself with exact operations (fmod is exact, one rounded addition for a
// negative angle) against the doubles nearest pi, pi/4 and 3pi/4: it differs
// from the exact rule only within ~3e-16 rad of a diagonal, where comparing
// |cos| with |sin| would depend on the last bit of the sine and cosine.
__device__ __forceinline__ bool march_rows(double theta)
{
    const double pi = 3.14159265358979323846, q1 = 0.78539816339744830962, q3 = 2.35619449019234492885;
    double t = fmod(theta, pi);
    if (t < 0.0) t = __dadd_rn(t, pi);
    return t <= q1 || t >= q3;
}

// Rebuilds the constants of view v when its (theta, delta) changed since the
// last call; returns whether it did.
__device__ bool view_setup_one(int v, const double *__restrict__ theta, const double *__restrict__ delta,
                               const int *__restrict__ fov, int N, int B, ViewGeo *__restrict__ out,
                               int *__restrict__ flag)
{
    double th = theta[v];
    double dl = delta ? delta[v] : 0.0;
    ViewGeo *gp = out + v;
    if ((gp->flags & kValid) && __double_as_longlong(gp->th) == __double_as_longlong(th) &&
        __double_as_longlong(gp->dl) == __double_as_longlong(dl))
        return false;  // unchanged since the last call
    const double th_in = th, dl_in = dl;
    int bad = 0;
    if (!isfinite(th) || !isfinite(dl)) {
        *flag = 1;  // every writer stores the same value
        th = 0.0;
        dl = 0.0;
        bad = 1;
    }
    double s, c;
    sincos(th, &s, &c);
    const double h = 0.5 * (N - 1);
    const double sb0 = -0.5 * (B - 1) + dl;
    ViewGeo g;
    double q0, qb, qr;
    if (march_rows(th)) {  // one sample per image row
        const double ic = 1.0 / c;
        const double ic2 = ic * ic;
        g.mode = 0;
        qb = ic;
        qr = s * ic;
        q0 = (sb0 - h * s) * ic + h;
        g.w = (float)fabs(ic);
        g.dw = (float)(copysign(1.0, c) * s * ic2);
        g.gs = (float)(s * ic2);
        g.gh = (float)(-h * ic2);
        g.gr = (float)ic2;
    } else {  // one sample per image column (rows of X^T)
        const double is = 1.0 / s;
        const double is2 = is * is;
        g.mode = 1;
        qb = -is;
        qr = c * is;
        q0 = h - (sb0 + h * c) * is;
        g.w = (float)fabs(is);
        g.dw = (float)(-copysign(1.0, s) * c * is2);
        g.gs = (float)(c * is2);
        g.gh = (float)(h * is2);
        g.gr = (float)(-is2);
    }
    // Fixed-point line anchored at the image centre with an integer bin offset.
    const double n0 = floor(sb0);
    g.n0 = (int)n0;
    g.Qc = __double2ll_rn(h * kFixScale) + __double2ll_rn((sb0 - n0) * qb * kFixScale);
    g.Qb = __double2ll_rn(qb * kFixScale);
    g.Qh = __double2ll_rn(qr * 0.5 * kFixScale);
    g.qbf = (float)qb;
    g.sb0 = (float)sb0;
    g.sb0d = sb0;
    int flags = kValid;
    if (fabs(qr) < kAllRowsBelow) {
        flags |= kAllRows;
        g.alo = g.ahi = g.gam = 0.0f;
    } else {
        const double iqr = 1.0 / qr;
        g.alo = (float)((-1.0 - q0) * iqr);
        g.ahi = (float)(((double)N - q0) * iqr);
        g.gam = (float)(-qb * iqr);
    }
    g.flags = bad ? (flags & ~kValid) : flags;  // a bad view is rebuilt (and reported) every call
    g.beta0 = h * (s - c) - dl + 0.5 * (B - 1);
    g.c = c;
    g.s = s;
    g.aC = __double2int_rn(c * (double)(1 << kAdjFrac));
    g.aS = __double2int_rn(s * (double)(1 << kAdjFrac));
    g.th = th_in;
    g.dl = dl_in;
    g.frame = fov ? fov[v] : 0;
    g.gen = gp->gen + 1;
    *gp = g;
    return true;
}

// The view-table step of a call: the per-view constants of the views whose
// angle or offset changed, then the view order.  The order of the ray kernels
// sorts the views by frame, then by marching axis, then by ray slope qr (ties
// by index), so that consecutive entries read the same image and sweep nearly
// the same band of it; it is rebuilt only when a view changed.  Without an
// order buffer (nullable) only the constants are built.
//
// The constants are FP64: some hundred dependent operations of ~63 cycles a
// view, one warp per scheduler filling the pipe, so the step is spread over
// ceil(V / 256) CTAs and the last one to finish sorts.  In one CTA, ranking by
// counting, the layout kernel that carries the step waited for it when the
// angles were new: 120 us instead of 31 us at 1200 views (first call of a
// 16-frame block of 8 images: 585 us; 503 us spread).  Up to 256 views one CTA
// does it, as the arrival costs 0.6 us of every call (28.5 us instead of
// 27.9 us for a one-image block of 180 views, 128 views per CTA).
constexpr int kOrderMaxV = 4096;
constexpr int kOrderRankMaxV = 256;   // rank counting up to here, sorting above
constexpr int kPrepViews = 256;       // views per CTA of the view-table step, one per thread

// What the view-table step of an operator call needs; `on` = 0: no step.
struct ViewPrep {
    const double *theta, *delta;
    const int *fov;
    int V, N, B, on;  // on: CTAs of the step
    ViewGeo *vg;
    int *flag;           // flag[0]: bad input, flag[1]: arrivals of the step's CTAs (0 between calls)
    int *order;  // nullable: constants only
};

__device__ void build_order(const ViewPrep &p, unsigned long long *key);

// CTA `part` of the p.on CTAs of the view-table step (kPrepViews threads);
// key: shared memory of prep_smem bytes.  No CTA waits for another: each adds
// itself, and whether it rebuilt a view, to the arrival count, and the last
// one builds the order and clears the count.
__device__ void view_prep_block(const ViewPrep &p, int part, unsigned long long *key)
{
    __shared__ int s_build;
    int mine = 0;
    for (int v = part * kPrepViews + threadIdx.x; v < p.V; v += p.on * kPrepViews)
        mine |= view_setup_one(v, p.theta, p.delta, p.fov, p.N, p.B, p.vg, p.flag);
    mine = __syncthreads_or(mine);
    if (!p.order) return;
    if (p.on > 1) {
        if (threadIdx.x == 0) {
            const int add = mine ? 0x10001 : 1;
            __threadfence();
            const int all = atomicAdd(p.flag + 1, add) + add;
            const bool last = (all & 0xffff) == p.on;
            if (last) p.flag[1] = 0;
            s_build = last && (all >> 16);
            __threadfence();
        }
        __syncthreads();
        mine = s_build;
    }
    if (mine) build_order(p, key);
}

// The view order, by one CTA, from the current view records.
__device__ void build_order(const ViewPrep &p, unsigned long long *key)
{
    const int V = p.V;
    if (V > kOrderMaxV) {
        for (int i = threadIdx.x; i < V; i += blockDim.x) p.order[i] = i;
        return;
    }
    int P = V;
    if (V > kOrderRankMaxV)
        for (P = 2 * kOrderRankMaxV; P < V;) P *= 2;
    for (int i = threadIdx.x; i < P; i += blockDim.x)
        key[i] = i < V ? order_key(p.vg[i].frame, p.vg[i].mode, p.vg[i].Qh, i) : ~0ULL;
    __syncthreads();
    // Up to one view per thread the rank of a view counts the keys below it (V
    // steps); above, a bitonic sort: 1200 views in 66 steps of 4 exchanges a
    // thread instead of 5 x 1200 compares, 512 views in 45 instead of 2 x 512.
    if (V <= kOrderRankMaxV) {
        for (int i = threadIdx.x; i < V; i += blockDim.x) {
            const unsigned long long ki = key[i];
            int rank = 0;
            for (int j = 0; j < V; ++j) rank += key[j] < ki ? 1 : 0;
            p.order[rank] = i;
        }
        return;
    }
    for (int size = 2; size <= P; size *= 2) {
        for (int stride = size / 2; stride > 0; stride /= 2) {
            for (int t = threadIdx.x; t < P / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (stride - 1)), j = i + stride;
                const unsigned long long a = key[i], b = key[j];
                if ((a > b) == ((i & size) == 0)) {
                    key[i] = b;
                    key[j] = a;
                }
            }
            // exchanges over at most 32 stay within the 64 keys of a warp
            if (stride > 32 || (stride == 1 && size > 32))
                __syncthreads();
            else
                __syncwarp();
        }
    }
    for (int i = threadIdx.x; i < V; i += blockDim.x) p.order[i] = (int)(key[i] & 0xfff);
}

__global__ void __launch_bounds__(256) k_view_prep(ViewPrep p, const int *__restrict__ skip)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    if (skip && *skip) return;
    view_prep_block(p, blockIdx.x, prep_key);
}

// ---------------------------------------------------------------------------
// pair layouts
// ---------------------------------------------------------------------------
// PX[img][r][cp] = (X[r][c], X[r][c + 1]) and PT[img][c][rp] = (X[r][c],
// X[r + 1][c]) with cp = c + 2, rp = r + 2 and zero outside the image: the
// 33 x 33 elements of X from (r0, c0) on, both from -2 in steps of 32, hold a
// 32 x 32 tile of each, so that X is read once.  Bound by
// memory (2048^2, one image: 84 MB, 12.4 us at the copy rate): 35 us reading X
// once per orientation, 17.4 us so; 48 registers (5 CTAs an SM) instead of 64.
// With p.on, extra columns of CTAs are launched and their first p.on CTAs run
// the view-table step of the call (the two are independent).
template <typename T>
__global__ void __launch_bounds__(256, 5) k_pairs_img(const T *__restrict__ X, pair_t<T> *__restrict__ PX,
                                                   pair_t<T> *__restrict__ PT, int N, int Pp, int nimg, ViewPrep p,
                                                   const int *__restrict__ skip)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    if (skip && *skip) return;
    if (blockIdx.x >= (Pp + 31) / 32) {
        const int part = ((blockIdx.x - (Pp + 31) / 32) * gridDim.z + blockIdx.z) * gridDim.y + blockIdx.y;
        if (part < p.on) view_prep_block(p, part, prep_key);
        return;
    }
    __shared__ T t[33][33];  // t[i][j] = X[r0 + i][c0 + j]
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int r0 = blockIdx.y * 32 - 2, c0 = blockIdx.x * 32 - 2;
    for (int img = blockIdx.z; img < nimg; img += gridDim.z) {
        const T *src = X + (size_t)img * N * N;
        auto at = [&](int i, int j) {
            const int r = r0 + i, c = c0 + j;
            return (r >= 0 && r < N && c >= 0 && c < N) ? src[(size_t)r * N + c] : T(0);
        };
        T x[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) x[m] = at(ty + 8 * m, tx);
        const T edge = ty == 0 ? at(32, tx) : (ty == 1 ? at(tx, 32) : T(0));  // the corner (32, 32) is not used
        __syncthreads();  // the previous image's tile has been read
#pragma unroll
        for (int m = 0; m < 4; ++m) t[ty + 8 * m][tx] = x[m];
        if (ty == 0) t[32][tx] = edge;
        if (ty == 1) t[tx][32] = edge;
        __syncthreads();
        pair_t<T> *px = PX + (size_t)img * N * Pp;
        pair_t<T> *pt = PT + (size_t)img * N * Pp;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int i = ty + 8 * m;
            if (r0 + i >= 0 && r0 + i < N && c0 + tx + 2 < Pp) {
                pair_t<T> q;
                q.x = x[m];
                q.y = t[i][tx + 1];
                px[(size_t)(r0 + i) * Pp + c0 + tx + 2] = q;
            }
            if (c0 + i >= 0 && c0 + i < N && r0 + tx + 2 < Pp) {
                pair_t<T> q;
                q.x = t[tx][i];
                q.y = t[tx + 1][i];
                pt[(size_t)(c0 + i) * Pp + r0 + tx + 2] = q;
            }
        }
    }
}

constexpr size_t kInterleaveTile = sizeof(float) * 4 * 32 * 33;
static_assert(kInterleaveTile <= 48 * 1024 && sizeof(unsigned long long) * kOrderMaxV + sizeof(double) * 33 * 33 <= 47 * 1024,
              "tiles and keys fit the shared memory of a launch as they are");

// X -> interleaved images of X and X^T (FP32): each CTA reads a 32 x 32 tile
// of the images of one group, of one frame, from (r0, c0) on (both from -2 in
// steps of 32), once; a thread has the group's images at its elements side by
// side and writes them as one vector of w floats to the image of X, and
// through shared memory to that of X^T.  Bound by memory (16 frames of 256^2,
// 8 images: 100 MB, 15 us at the copy rate): 31 us with a CTA and a read of X
// per orientation, 20 us so.
// With p.on the last columns of CTAs carry the view-table step, as in k_pairs_img.
__global__ void __launch_bounds__(256, 5) k_interleave_img(const float *__restrict__ X, float *__restrict__ QX,
                                                           float *__restrict__ QT, int N, int Pp, int F, int K,
                                                           ViewPrep p, const int *__restrict__ skip)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    if (skip && *skip) return;
    if (blockIdx.x >= (Pp + 31) / 32) {
        const int part = ((blockIdx.x - (Pp + 31) / 32) * gridDim.z + blockIdx.z) * gridDim.y + blockIdx.y;
        if (part < p.on) view_prep_block(p, part, prep_key);
        return;
    }
    // t[j][i][e] = X_j[r0 + i][c0 + e], where the CTAs of the step have their keys: both
    // together would pass the 48 KB that a launch may use without asking the device
    float (*t)[32][33] = reinterpret_cast<float (*)[32][33]>(prep_key);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int r0 = blockIdx.y * 32 - 2, c0 = blockIdx.x * 32 - 2;
    const int n4 = K & ~3, rem = K - n4;
    const int ngroups = n4 / 4 + (rem >= 2 ? 1 : 0) + (rem & 1);
    for (int z = blockIdx.z; z < F * ngroups; z += gridDim.z) {
        const int gi = z / F, f = z - gi * F;
        int k0, w;
        interleave_group(gi < n4 / 4 ? 4 * gi : (gi == n4 / 4 && rem >= 2 ? n4 : K - 1), K, k0, w);
        float x[4][4];  // [m][j]
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float *src = X + ((size_t)(k0 + j) * F + f) * N * N;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int r = r0 + ty + 8 * m, c = c0 + tx;
                x[m][j] = (j < w && r >= 0 && r < N && c >= 0 && c < N) ? src[(size_t)r * N + c] : 0.0f;
            }
        }
        auto put = [&](float *Q, int row, int e, const float (&v)[4]) {
            if (row < 0 || row >= N || e >= Pp) return;
            float *q = Q + (size_t)k0 * F * N * Pp + (((size_t)f * N + row) * Pp + e) * w;
            if (w == 4)
                *reinterpret_cast<float4 *>(q) = make_float4(v[0], v[1], v[2], v[3]);
            else if (w == 2)
                *reinterpret_cast<float2 *>(q) = make_float2(v[0], v[1]);
            else
                *q = v[0];
        };
        __syncthreads();  // the previous group's tile has been read
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            put(QX, r0 + ty + 8 * m, c0 + tx + 2, x[m]);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < w) t[j][ty + 8 * m][tx] = x[m][j];
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = t[j][tx][ty + 8 * m];
            put(QT, c0 + ty + 8 * m, r0 + tx + 2, v);
        }
    }
}

// Pair images of the first nimg images of a batch of K from the interleaved
// ones of X, and (PT not null) those of X^T: pair e of a row is (element e,
// element e + 1), zero past the row end.  The first p.on CTAs run the
// view-table step of the call instead.
__global__ void k_interleaved_to_pairs(const float *__restrict__ QX, const float *__restrict__ QT,
                                       float2 *__restrict__ PX, float2 *__restrict__ PT, long long per, int Pp, int K,
                                       int nimg, ViewPrep p)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    const int nblk = gridDim.x - p.on, blk = blockIdx.x - p.on;
    if (blk < 0) {
        view_prep_block(p, blockIdx.x, prep_key);
        return;
    }
    const long long total = (long long)nimg * per;  // per: elements per image
    for (long long idx = blk * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)nblk * blockDim.x) {
        const int k = (int)(idx / per);
        const long long el = idx - k * per;
        const int e = (int)(el % Pp);
        int k0, w;
        interleave_group(k, K, k0, w);
        const size_t o = (size_t)k0 * per + (size_t)el * w + (k - k0);
        const bool last = e + 1 >= Pp;
        PX[idx] = make_float2(QX[o], last ? 0.0f : QX[o + w]);
        if (PT) PT[idx] = make_float2(QT[o], last ? 0.0f : QT[o + w]);
    }
}

// Pair images of X^T from those of X, by 33 x 33 elements as k_pairs_img.
__global__ void __launch_bounds__(256) k_transpose_pairs(const float2 *__restrict__ PX, float2 *__restrict__ PT, int N,
                                                         int Pp, int nimg)
{
    chain_wait();
    __shared__ float t[33][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int r0 = blockIdx.y * 32 - 2, c0 = blockIdx.x * 32;
    for (int img = blockIdx.z; img < nimg; img += gridDim.z) {
        const float2 *px = PX + (size_t)img * N * Pp;
        __syncthreads();  // the previous image's tile has been read
        for (int i = ty; i < 33; i += 8) {
            const int r = r0 + i, c = c0 + tx;
            t[i][tx] = (r >= 0 && r < N && c < N) ? px[(size_t)r * Pp + c + 2].x : 0.0f;
        }
        __syncthreads();
        for (int i = ty; i < 32; i += 8)
            if (c0 + i < N && r0 + tx + 2 < Pp)
                PT[((size_t)img * N + c0 + i) * Pp + r0 + tx + 2] = make_float2(t[tx][i], t[tx + 1][i]);
    }
}

// FP64: YP[row][bp] = (Y[row][bp - 2], Y[row][bp - 1]), zero outside [0, B).
// With p.on, the first p.on CTAs run the view-table step of the call instead.
__global__ void k_pairs_sino(const double *__restrict__ Y, double2 *__restrict__ YP, int B, int Pb, long long total,
                             ViewPrep p, const int *__restrict__ skip)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    if (skip && *skip) return;
    const int nblk = gridDim.x - p.on, blk = blockIdx.x - p.on;
    if (blk < 0) {
        view_prep_block(p, blockIdx.x, prep_key);
        return;
    }
    for (long long idx = blk * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)nblk * blockDim.x) {
        const long long row = idx / Pb;
        const int bp = (int)(idx - row * Pb);
        const int b0 = bp - 2, b1 = bp - 1;
        const double *y = Y + row * B;
        double2 p;
        p.x = (b0 >= 0 && b0 < B) ? y[b0] : 0.0;
        p.y = (b1 >= 0 && b1 < B) ? y[b1] : 0.0;
        YP[idx] = p;
    }
}

// One row of a group of W sinograms, `live` of them given: U bins of every
// sinogram in flight per thread.  The loads carry no condition (their
// addresses are clamped into the row, what lies outside is replaced by zero
// afterwards): with one around each the compiler kept them one after another.
template <int W, int U>
__device__ __forceinline__ int interleave_row(const float *__restrict__ in, float *__restrict__ out, long long pitch,
                                              int live, int B, int Pq)
{
    int bad = 0;
    for (int b0 = threadIdx.x; b0 < Pq; b0 += U * blockDim.x) {
        float y[U][W];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < W; ++k)
                y[u][k] = __ldg(in + min(k, live - 1) * pitch + min(b0 + u * (int)blockDim.x, B - 1));
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int b = b0 + u * blockDim.x;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                if (k >= live || b >= B) y[u][k] = 0.0f;
                bad |= !isfinite(y[u][k]);
            }
            if (b >= Pq) continue;
            float *o = out + (size_t)b * W;
            if constexpr (W == 1)
                *o = y[u][0];
            else if constexpr (W == 2)
                *reinterpret_cast<float2 *>(o) = make_float2(y[u][0], y[u][1]);
            else
#pragma unroll
                for (int k = 0; k < W; k += 4)
                    *reinterpret_cast<float4 *>(o + k) = make_float4(y[u][k], y[u][k + 1], y[u][k + 2], y[u][k + 3]);
        }
    }
    return bad;
}

// FP32: the interleaved sinograms of the transpose (ct_internal.cuh).  A CTA
// takes rows (group, view): each thread reads its bins of the group's
// sinograms (coalesced over the bins) and writes them side by side; the row's
// flag says whether it holds a non-finite value.  Bound by memory latency
// (1200 views x 363 bins, 8 sinograms, 28 MB, 4 us at the copy rate: 20 us with a
// condition around each load, 9 us so; 2901 bins, 120 views, one: 9.5 -> 4.6 us).
// With p.on, the first p.on CTAs run the view-table step of the call instead.
__global__ void __launch_bounds__(256, 5) k_interleave_sino(const float *__restrict__ Y, float *__restrict__ YI,
                                                            int *__restrict__ rowflag, int B, int Pq, int V,
                                                            int nsino, int kb, long long rows, ViewPrep p,
                                                            const int *__restrict__ skip)
{
    chain_wait();
    extern __shared__ unsigned long long prep_key[];
    if (skip && *skip) return;
    const int nblk = gridDim.x - p.on, blk = blockIdx.x - p.on;
    if (blk < 0) {
        view_prep_block(p, blockIdx.x, prep_key);
        return;
    }
    for (long long row = blk; row < rows; row += nblk) {
        const int grp = (int)(row / V), v = (int)(row - (long long)grp * V);
        const int k0 = grp * kb, live = min(kb, nsino - k0);
        int w = 1;
        while (w < live) w *= 2;
        float *out = YI + ((size_t)k0 * V + (size_t)v * w) * Pq;
        const float *in = Y + ((size_t)k0 * V + v) * B;
        const long long pitch = (long long)V * B;
        int bad = 0;
        switch (w) {
        case 1: bad = interleave_row<1, 8>(in, out, pitch, live, B, Pq); break;
        case 2: bad = interleave_row<2, 4>(in, out, pitch, live, B, Pq); break;
        case 4: bad = interleave_row<4, 4>(in, out, pitch, live, B, Pq); break;
        default: bad = interleave_row<8, 2>(in, out, pitch, live, B, Pq); break;
        }
        bad = __syncthreads_or(bad);
        if (threadIdx.x == 0) rowflag[row] = bad;
    }
}

// ---------------------------------------------------------------------------
// ray march
// ---------------------------------------------------------------------------
// One CTA = VW view slots x SPLIT row segments, all on the same 32-bin chunk.
// The view slots take VW consecutive entries of the view order (views sorted
// by marching axis and ray slope), so the warps of a CTA sweep nearly the
// same image band row by row and share it in L1.  SPLIT warps march
// consecutive row segments of the same rays and are combined in shared memory
// in a fixed order.
// Both taps of the KB images of an interleaved group at element e of a row
// (q points at element e): one vector load at e and one at e + 1 for each
// group of 4 images (gstride floats per image between the groups).
template <int KB>
__device__ __forceinline__ void taps_interleaved(const float *__restrict__ q, long long gstride, float2 (&p)[KB])
{
    if constexpr (KB >= 4) {
#pragma unroll
        for (int h = 0; h < KB / 4; ++h) {
            const float4 *e = reinterpret_cast<const float4 *>(q + (size_t)h * 4 * gstride);
            const float4 x = __ldg(e), y = __ldg(e + 1);
            p[4 * h + 0] = make_float2(x.x, y.x);
            p[4 * h + 1] = make_float2(x.y, y.y);
            p[4 * h + 2] = make_float2(x.z, y.z);
            p[4 * h + 3] = make_float2(x.w, y.w);
        }
    } else if constexpr (KB == 2) {
        const float2 *e = reinterpret_cast<const float2 *>(q);
        const float2 x = __ldg(e), y = __ldg(e + 1);
        p[0] = make_float2(x.x, y.x);
        p[1] = make_float2(x.y, y.y);
    } else {
        p[0] = make_float2(__ldg(q), __ldg(q + 1));
    }
}

// QL (FP32): the images come from the interleaved layout; the taps, the
// fractions and the order of the sums are those of the pair form, so both
// give the same bits.
template <typename T, int MODE, bool OFFS, int KB, int SPLIT, bool QL = false>
__global__ void __launch_bounds__(512) k_ray(RayArgs<T> a)
{
    chain_wait();
    using P2 = pair_t<T>;
    constexpr bool F32 = std::is_same<T, float>::value;
    constexpr int NACC = (MODE == kFwd) ? KB : 3 * KB;
    extern __shared__ unsigned char ray_smem[];
    T *red = reinterpret_cast<T *>(ray_smem);  // [VW][SPLIT][NACC][32], only when SPLIT > 1
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int seg = warp % SPLIT;
    const int slot = warp / SPLIT;
    const int VW = a.VW;
    const int N = a.N;
    const int ngv = (a.V + VW - 1) / VW;
    const int total = a.ngroups * ngv * a.nchunks;
    if (a.skip && *a.skip) return;
    for (int item = blockIdx.x; item < total; item += gridDim.x) {
        const int chunk = item % a.nchunks;
        const int t = item / a.nchunks;
        const int vgi = t % ngv;
        const int grp = t / ngv;
        const int pos = vgi * VW + slot;
        const int v = pos < a.V ? (a.order ? a.order[pos] : pos) : -1;
        const bool live = v >= 0 && !(MODE == kGn && a.view_mask && a.view_mask[v] == 0);  // warp-uniform
        const ViewGeo &g = a.vg[live ? v : 0];
        const int b = chunk * kChunk + lane;
        const bool active = live && b < a.B;
        const int k0 = a.kbase + grp * KB;
        T acc[NACC];
#pragma unroll
        for (int k = 0; k < NACC; ++k) acc[k] = T(0);
        if (live) {
            int rlo, rhi;
            warp_rows(g, b, b < a.B, N, rlo, rhi);
            const int len = rhi - rlo + 1;
            const int per = (len + SPLIT - 1) / SPLIT;
            const int r0 = rlo + seg * per;
            const int r1 = min(rhi, r0 + per - 1);
            long long Q = line_at(g, b, r0, N);
            const long long dQ = 2 * g.Qh;
            constexpr int QW = KB >= 4 ? 4 : KB;  // floats per element of the group's interleaved layout
            const unsigned pp = (unsigned)a.Pp, lim = (unsigned)(N + 2);
            const P2 *img = nullptr;
            const float *qimg = nullptr;
            if constexpr (QL)
                qimg = (g.mode ? a.QT : a.QX) + (size_t)k0 * a.qimg_stride + ((size_t)g.frame * N + r0) * pp * QW;
            else
                img = (g.mode ? a.PT : a.PX) + ((size_t)g.frame * N + r0) * pp + (size_t)k0 * a.pimg_stride;
            [[maybe_unused]] const T g0 = fma(GeoT<T>::sb(g, b), GeoT<T>::gs(g), GeoT<T>::gh(g, N));
            [[maybe_unused]] const T gr = GeoT<T>::gr(g);
            [[maybe_unused]] T rf = (T)r0;
            // Rows are processed in blocks of U: all loads of a block are issued
            // before any of them is used, so U*KB gathers are in flight per warp.
            // The rows past the segment's end in the last block read nothing and add
            // exact zeros (one more round trip to memory, where a row at a time
            // took one each).  16 rows for one FP32 image: 512^2 / 360 views, Gauss-Newton
            // terms 82.0 us with 8, 104 with 4, 76.8 with 16.
            constexpr int U = KB >= 4 ? 4 : (KB == 1 && F32 ? 16 : 8);
            auto block = [&](auto whole, int rows) {
                constexpr bool WHOLE = decltype(whole)::value;
                unsigned idx[U];
                T f[U];
                P2 p[U][KB];
                ray_cells<T, U, true>(Q, dQ, lim, idx, f);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (WHOLE || u < rows) {
                        if constexpr (QL) {
                            taps_interleaved<KB>(qimg + (size_t)(idx[u] + u * pp) * QW, a.qimg_stride, p[u]);
                        } else {
                            const P2 *row = img + (idx[u] + u * pp);
#pragma unroll
                            for (int k = 0; k < KB; ++k) p[u][k] = __ldg(row + (size_t)k * a.pimg_stride);
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < KB; ++k) p[u][k].x = p[u][k].y = T(0);
                    }
                }
                if constexpr (MODE == kFwd) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (!F32 && !WHOLE && u >= rows) break;  // FP64 products are dear (uniform)
                        const T omf = T(1) - f[u];
#pragma unroll
                        for (int k = 0; k < KB; ++k) acc[k] = fma(omf, p[u][k].x, fma(f[u], p[u][k].y, acc[k]));
                    }
                } else {
                    // per image k of the group: acc[3k] = sum of interpolated values,
                    // acc[3k+1] = sum slope * dq/dtheta, acc[3k+2] = sum of slopes
                    // (offset derivative); the line, cell and fraction serve all KB images
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (!F32 && !WHOLE && u >= rows) break;
                        const T dq = fma(rf + T(u), gr, g0);
#pragma unroll
                        for (int k = 0; k < KB; ++k) {
                            const T d = p[u][k].y - p[u][k].x;
                            acc[3 * k] += fma(f[u], d, p[u][k].x);
                            acc[3 * k + 1] = fma(d, dq, acc[3 * k + 1]);
                            if (OFFS) acc[3 * k + 2] += d;
                        }
                    }
                    rf += T(U);
                }
                if constexpr (QL) qimg += (size_t)U * pp * QW;
                else img += (size_t)U * pp;
                Q += (long long)U * dQ;
            };
            int r = r0;
            // (4 images a lane on pairs: the second block's loads start before the first's sums, or
            // a launch of few views waits for each: 256^2, 22 views, 8 images, 2 segments a ray
            // 37.0 us a call, 31.1 so; one whole ray per warp has warps enough, 49.5 and 64.3)
            constexpr int UNR = F32 && MODE == kFwd && KB == 4 && !QL && (SPLIT == 2 || SPLIT == 4) ? 2 : 1;
#pragma unroll UNR
            for (; r + U - 1 <= r1; r += U) block(std::true_type(), U);
            if (r <= r1) block(std::false_type(), r1 - r + 1);
        }
        if constexpr (SPLIT > 1) {
            T *mine = red + ((size_t)(slot * SPLIT + seg) * NACC) * 32;
#pragma unroll
            for (int k = 0; k < NACC; ++k) mine[k * 32 + lane] = acc[k];
            __syncthreads();
            if (seg == 0) {
                const T *base = red + ((size_t)slot * SPLIT * NACC) * 32;
#pragma unroll
                for (int k = 0; k < NACC; ++k) {
                    T s = base[k * 32 + lane];
#pragma unroll
                    for (int q = 1; q < SPLIT; ++q) s += base[(q * NACC + k) * 32 + lane];
                    acc[k] = s;
                }
            }
        }
        if (seg == 0 && live) ray_epilogue<T, MODE, OFFS, KB>(a, g, v, b, active, k0, chunk, lane, acc);
        if constexpr (SPLIT > 1) __syncthreads();  // red[] is reused by the next item
    }
}

// out_q[k][v] = scale_q * sum_c partial[k][v][c][q], summed in chunk order,
// for each of nimg images (partials part_stride doubles apart); with sum, one
// output per view summing the images in order (each image's chunks in order).
// One thread per output and quantity, the four quantities of a view side by
// side: an FP64 addition serves 8 views' four sums at once (it occupies the
// pipe for 64 cycles whatever the lanes do), where a warp per view with the
// sums carried by shuffles issued 36 for each view, and the loads of kFinAhead
// chunks are in flight (Gauss-Newton terms of 512^2 / 360 views: 95.5 -> 91.6
// us a call).
constexpr int kFinAhead = 24;
__global__ void __launch_bounds__(64) k_finalize(const double *__restrict__ partial, int V, int nchunks, int nimg,
                                                 long long part_stride, int sum, double *out0, double *out1,
                                                 double *out2, double scale2, double *out3,
                                                 const int *__restrict__ view_mask, const int *__restrict__ skip)
{
    chain_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int o = t >> 2, q = t & 3;
    const int nout = sum ? 1 : nimg;
    if (o >= V * nout || (skip && *skip)) return;
    const int v = o % V, kout = o / V;
    double *out = q == 0 ? out0 : (q == 1 ? out1 : (q == 2 ? out2 : out3));
    if (!out || (view_mask && view_mask[v] == 0)) return;
    double s = 0.0;  // sum over the images, each image's sum added in order
    const int klo = sum ? 0 : kout, khi = sum ? nimg : kout + 1;
    for (int k = klo; k < khi; ++k) {
        const double *p = partial + (size_t)k * part_stride + (size_t)v * nchunks * 4 + q;
        double x = 0.0;  // this image, chunks in order
        for (int c = 0; c < nchunks; c += kFinAhead) {
            double y[kFinAhead];
#pragma unroll
            for (int u = 0; u < kFinAhead; ++u) y[u] = c + u < nchunks ? p[4 * (c + u)] : 0.0;
#pragma unroll
            for (int u = 0; u < kFinAhead; ++u)
                if (c + u < nchunks) x += y[u];
        }
        s += x;
    }
    out[(size_t)kout * V + v] = q == 2 ? scale2 * s : s;
}

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
template <typename T> RayArgs<T> base_args(const Handle &h, ImgForm form = kPairImages)
{
    RayArgs<T> a{};
    a.vg = h.d_views;
    a.V = h.V;
    a.N = h.N;
    a.B = h.B;
    a.nchunks = h.nchunks;
    a.Pp = h.Pp;
    a.PX = (const pair_t<T> *)h.d_px;
    a.pimg_stride = h.img_elems();
    a.PT = form == kSidePairs ? a.PX + h.side_pairs * a.pimg_stride : (const pair_t<T> *)h.d_pt;
    a.kbase = 0;
    a.ngroups = 1;
    a.sino_stride = (long long)h.V * h.B;
    a.order = h.d_order;
    a.VW = 1;
    a.segs = 1;
    a.kend = 1 << 30;
    return a;
}

template <typename T, int MODE, bool OFFS, int KB, int SPLIT, bool QL = false>
cudaError_t run_ray(const Handle &h, const RayArgs<T> &a)
{
    auto kern = k_ray<T, MODE, OFFS, KB, SPLIT, QL>;
    constexpr int NACC = (MODE == kFwd) ? KB : 3 * KB;
    const int threads = 32 * SPLIT * a.VW;
    const size_t smem = SPLIT > 1 ? (size_t)a.VW * SPLIT * NACC * 32 * sizeof(T) : 0;
    const long long items = (long long)a.ngroups * ((a.V + a.VW - 1) / a.VW) * a.nchunks;
    const int grid = persistent_grid(kern, threads, smem, items, h.num_sms);
    launch_chained(kern, grid, threads, smem, h.stream, a);
    return cudaGetLastError();
}

template <typename T, int MODE, bool OFFS, int KB, bool QL = false>
cudaError_t run_ray_split(const Handle &h, const RayArgs<T> &a, int split)
{
    switch (split) {
    case 1: return run_ray<T, MODE, OFFS, KB, 1, QL>(h, a);
    case 2: return run_ray<T, MODE, OFFS, KB, 2, QL>(h, a);
    case 4: return run_ray<T, MODE, OFFS, KB, 4, QL>(h, a);
    default: return run_ray<T, MODE, OFFS, KB, 8, QL>(h, a);
    }
}

// FP32 with a staged shape runs the band kernel (ct_band.cu); every other
// case runs k_ray.
template <typename T, int MODE, bool OFFS, int KB>
cudaError_t run_ray_any(const Handle &h, const RayArgs<T> &a, int split, int stage)
{
    if (h.fan_D > 0.0) return run_fan_ray<T>(h, a, MODE, KB, split, OFFS);
    if constexpr (std::is_same<T, float>::value) {
        if (stage > 0 && band_shape_ok(MODE, KB, a.VW, stage)) return run_ray_band(h, a, MODE, OFFS, KB, stage);
    }
    return run_ray_split<T, MODE, OFFS, KB>(h, a, split);
}

template <typename T>
cudaError_t fwd_groups(const Handle &h, RayArgs<T> a, int kb, int split, int stage)
{
    switch (kb) {
    case 1: return run_ray_any<T, kFwd, false, 1>(h, a, split, stage);
    case 2: return run_ray_any<T, kFwd, false, 2>(h, a, split, stage);
    case 4: return run_ray_any<T, kFwd, false, 4>(h, a, split, stage);
    default: return run_ray_any<T, kFwd, false, 8>(h, a, split, stage);
    }
}

}  // namespace

namespace {

ViewPrep view_prep_args(const Handle &h, const double *theta, const double *delta)
{
    ViewPrep p{};
    p.theta = theta;
    p.delta = delta;
    p.fov = h.d_fov;
    p.V = h.V;
    p.N = h.N;
    p.B = h.B;
    p.on = theta ? std::min((h.V + kPrepViews - 1) / kPrepViews, 1024) : 0;
    p.vg = h.d_views;
    p.flag = h.d_flag;
    p.order = h.d_order;
    return p;
}

// Shared memory for the keys of the order: a power of two where they are sorted.
size_t prep_smem(const ViewPrep &p)
{
    if (!p.on || !p.order || p.V > kOrderMaxV) return 0;
    size_t keys = p.V;
    if (p.V > kOrderRankMaxV)
        for (keys = 2 * kOrderRankMaxV; keys < (size_t)p.V;) keys *= 2;
    return sizeof(unsigned long long) * keys;
}

// Columns of CTAs that an image layout launch adds for the step.
unsigned prep_columns(const ViewPrep &p, dim3 grid) { return (p.on + grid.y * grid.z - 1) / (grid.y * grid.z); }

}  // namespace

cudaError_t launch_view_setup(const Handle &h, const double *theta, const double *delta, const int *skip)
{
    const ViewPrep p = view_prep_args(h, theta, delta);
    launch_chained(k_view_prep, p.on, 256, prep_smem(p), h.stream, p, skip);
    if (h.fan_D > 0.0 && theta) {
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return launch_fan_rays(h, skip);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pairs_img(const Handle &h, const T *X, int nimg, const int *skip, const double *theta,
                             const double *delta)
{
    const ViewPrep p = view_prep_args(h, theta, delta);
    dim3 grid((h.Pp + 31) / 32, (h.Pp + 31) / 32, std::max(1, std::min(nimg, 65535)));
    grid.x += prep_columns(p, grid);
    launch_chained(k_pairs_img<T>, grid, 256, prep_smem(p), h.stream, X, (pair_t<T> *)h.d_px, (pair_t<T> *)h.d_pt, h.N, h.Pp,
                                                          nimg, p, skip);
    if (h.fan_D > 0.0 && theta) {
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        return launch_fan_rays(h, skip);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prep_forward(const Handle &h, const T *X, int nimg, const int *skip, const double *theta,
                                const double *delta)
{
    return launch_pairs_img<T>(h, X, nimg, skip, theta, delta);
}

cudaError_t launch_interleave_img(const Handle &h, const float *X, int batch, const double *theta,
                                  const double *delta, const int *skip)
{
    if (h.precision != 0 || h.fan_D > 0.0 || batch < 1 || batch > h.max_batch) return cudaErrorInvalidValue;
    const ViewPrep p = view_prep_args(h, theta, delta);
    const int n4 = batch & ~3, rem = batch - n4;
    const int ngroups = n4 / 4 + (rem >= 2 ? 1 : 0) + (rem & 1);
    dim3 grid((h.Pp + 31) / 32, (h.Pp + 31) / 32, std::max(1, std::min(h.F * ngroups, 65535)));
    grid.x += prep_columns(p, grid);
    launch_chained(k_interleave_img, grid, 256, std::max(prep_smem(p), kInterleaveTile), h.stream, X, h.qx(), h.qt(), h.N, h.Pp, h.F, batch, p, skip);
    return cudaGetLastError();
}

cudaError_t launch_interleaved_to_pairs(const Handle &h, int side, const double *theta, const double *delta)
{
    const int K = h.img_ready, nimg = side ? side : K;
    if (h.precision != 0 || h.fan_D > 0.0 || K < 1 || nimg > K || 2 * side > h.max_batch + 1)
        return cudaErrorInvalidValue;
    const long long per = h.img_elems(), total = nimg * per;
    const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)h.num_sms * 16);
    float2 *px = (float2 *)h.d_px;
    const ViewPrep p = view_prep_args(h, theta, delta);
    launch_chained(k_interleaved_to_pairs, blocks + p.on, 256, prep_smem(p), h.stream, h.qx(), h.qt(), px,
                   side ? px + side * per : nullptr, per, h.Pp, K, nimg, p);
    if (!side) {  // the pairs of X^T over the interleaved images, from those of X
        const dim3 grid((h.N + 31) / 32, (h.Pp + 31) / 32, std::min(K * h.F, 65535));
        launch_chained(k_transpose_pairs, grid, 256, 0, h.stream, px, (float2 *)h.d_pt, h.N, h.Pp, K * h.F);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sino_layout(const Handle &h, const T *Y, int nsino, int kb, const int *skip, const double *theta,
                               const double *delta)
{
    const ViewPrep p = view_prep_args(h, theta, delta);
    if (h.fan_D > 0.0) {
        // fan beam: the view-table step (when the angles come with the call) runs on its own
        if (p.on) {
            cudaError_t e = launch_view_setup(h, theta, delta, skip);
            if (e != cudaSuccess) return e;
        }
        return launch_fan_sino<T>(h, Y, nsino, skip);
    }
    if constexpr (std::is_same<T, float>::value) {
        SinoGroup g[2];
        const int ng = sino_groups(nsino, kb, g);
        const int groups = g[ng - 1].first + g[ng - 1].count;
        const long long rows = (long long)groups * h.V;
        const int blocks = (int)std::min<long long>(rows, (long long)h.num_sms * 16);
        launch_chained(k_interleave_sino, blocks + p.on, 256, prep_smem(p), h.stream, 
            Y, (float *)h.d_yp, h.d_rowflag, h.B, sino_pitch(h.B), h.V, nsino, kb, rows, p, skip);
    } else {
        const long long total = (long long)nsino * h.V * h.Pb;
        const int threads = 256;
        const long long blocks = std::min<long long>((total + threads - 1) / threads, (long long)h.num_sms * 16);
        launch_chained(k_pairs_sino, (int)std::max<long long>(1, blocks) + p.on, threads, prep_smem(p), h.stream, 
            Y, (double2 *)h.d_yp, h.B, h.Pb, total, p, skip);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_forward(const Handle &h, T *Y, int batch, int kb, int split, int vw, int stage, const int *skip,
                           bool interleaved, int layout_batch)
{
    RayArgs<T> a = base_args<T>(h);
    a.Y = Y;
    a.skip = skip;
    a.VW = vw;
    if (interleaved) {
        // The groups of the layout (a batch of layout_batch images: groups of 8 = two
        // interleaved groups of 4, or 4, then the remainder's 2 and 1) that hold one of
        // the first `batch` images; images past `batch` in the last of them are read
        // but not written.
        if constexpr (std::is_same<T, float>::value) {
            if (h.fan_D > 0.0 || layout_batch < batch || layout_batch > h.max_batch)
                return cudaErrorInvalidValue;
            a.QX = h.qx();
            a.QT = h.qt();
            a.qimg_stride = (long long)h.F * h.N * h.Pp;
            a.kend = batch;
            int k = 0;
            for (int width : {8, 4, 2, 1}) {
                if (width == 8 && kb < 8) continue;
                if (k >= batch) break;
                const int groups = std::min((layout_batch - k) / width, (batch - k + width - 1) / width);
                if (groups == 0) continue;
                a.kbase = k;
                a.ngroups = groups;
                cudaError_t e = width == 8   ? run_ray_split<float, kFwd, false, 8, true>(h, a, split)
                                : width == 4 ? run_ray_split<float, kFwd, false, 4, true>(h, a, split)
                                : width == 2 ? run_ray_split<float, kFwd, false, 2, true>(h, a, split)
                                             : run_ray_split<float, kFwd, false, 1, true>(h, a, split);
                if (e != cudaSuccess) return e;
                k += groups * width;
            }
            return cudaSuccess;
        } else {
            return cudaErrorInvalidValue;
        }
    }
    // band-staged FP32 march with `split` CTAs per ray: segment partials go to Y and d_segpart
    const bool band = std::is_same<T, float>::value && stage > 0 && band_shape_ok(kFwd, 1, vw, stage) &&
                      !(h.fan_D > 0.0);
    if (band && split > 1) {
        if (!h.d_segpart || split > 4) return cudaErrorInvalidValue;
        a.segs = split;
        a.fpart = (T *)h.d_segpart;
        a.fpart_stride = (long long)h.max_batch * h.V * h.B;
    }
    int k = 0;
    for (int width : {8, 4, 2, 1}) {
        if (width > kb) continue;
        const int groups = (batch - k) / width;
        if (groups == 0) continue;
        a.kbase = k;
        a.ngroups = groups;
        cudaError_t e = fwd_groups<T>(h, a, width, split, stage);
        if (e != cudaSuccess) return e;
        k += groups * width;
    }
    if constexpr (std::is_same<T, float>::value) {
        if (a.segs > 1) return launch_fwd_combine(h, Y, a.fpart, a.segs, a.fpart_stride, batch, skip);
    }
    return cudaSuccess;
}

// The derivative modes over `batch` images sharing the view table: groups of
// up to kb (1, 2 or 4) images per lane; the fan-beam and band-staged forms
// take one image per lane (their launches still cover the whole batch).
// kInterleaved (FP32, parallel beam, stage 0): the images are those of the
// interleaved layout of a batch of `batch`, read by its groups of 4, 2 and 1.
template <typename T, int MODE, bool OFFS>
cudaError_t der_groups(const Handle &h, RayArgs<T> a, int batch, int kb, int split, int stage, ImgForm form)
{
    if (form == kInterleaved) {
        if constexpr (std::is_same<T, float>::value) {
            if (h.fan_D > 0.0 || batch > h.max_batch) return cudaErrorInvalidValue;
            a.QX = h.qx();
            a.QT = h.qt();
            a.qimg_stride = (long long)h.F * h.N * h.Pp;
            int k = 0;
            for (int width : {4, 2, 1}) {
                const int groups = (batch - k) / width;
                if (groups == 0) continue;
                a.kbase = k;
                a.ngroups = groups;
                cudaError_t e = width == 4   ? run_ray_split<float, MODE, OFFS, 4, true>(h, a, split)
                                : width == 2 ? run_ray_split<float, MODE, OFFS, 2, true>(h, a, split)
                                             : run_ray_split<float, MODE, OFFS, 1, true>(h, a, split);
                if (e != cudaSuccess) return e;
                k += groups * width;
            }
            return cudaSuccess;
        } else {
            return cudaErrorInvalidValue;
        }
    }
    bool one = h.fan_D > 0.0;
    if constexpr (std::is_same<T, float>::value) one = one || (stage > 0 && band_shape_ok(MODE, 1, a.VW, stage));
    int k = 0;
    for (int width : {4, 2, 1}) {
        if (width > kb || (one && width > 1)) continue;
        const int groups = (batch - k) / width;
        if (groups == 0) continue;
        a.kbase = k;
        a.ngroups = groups;
        cudaError_t e;
        switch (width) {
        case 4: e = run_ray_any<T, MODE, OFFS, 4>(h, a, split, stage); break;
        case 2: e = run_ray_any<T, MODE, OFFS, 2>(h, a, split, stage); break;
        default: e = run_ray_any<T, MODE, OFFS, 1>(h, a, split, stage); break;
        }
        if (e != cudaSuccess) return e;
        k += groups * width;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_jvp(const Handle &h, const double *dtheta, const double *ddelta, T *dY, int split, int vw,
                       int stage, int batch, int kb, long long dir_stride, ImgForm form)
{
    RayArgs<T> a = base_args<T>(h, form);
    a.VW = vw;
    a.Y = dY;
    a.dtheta = dtheta;
    a.ddelta = ddelta;
    a.dir_stride = dir_stride;
    return ddelta ? der_groups<T, kJvp, true>(h, a, batch, kb, split, stage, form)
                  : der_groups<T, kJvp, false>(h, a, batch, kb, split, stage, form);
}

template <typename T>
cudaError_t launch_vjp(const Handle &h, const T *R, double *gtheta, double *gdelta, int split, int vw, int stage,
                       int batch, int kb, long long r_stride, int sum, ImgForm form)
{
    RayArgs<T> a = base_args<T>(h, form);
    a.VW = vw;
    a.R = R;
    a.r_stride = r_stride;
    a.partial = h.d_partial;
    a.part_stride = 4LL * h.V * h.nchunks;
    cudaError_t e = gdelta ? der_groups<T, kVjp, true>(h, a, batch, kb, split, stage, form)
                           : der_groups<T, kVjp, false>(h, a, batch, kb, split, stage, form);
    if (e != cudaSuccess) return e;
    const long long outs = (long long)h.V * (sum ? 1 : batch);
    launch_chained(k_finalize, (int)((4 * outs + 63) / 64), 64, 0, h.stream, h.d_partial, h.V, h.nchunks, batch, a.part_stride,
                                                            sum, gtheta, gdelta, nullptr, 1.0, nullptr, nullptr,
                                                            nullptr);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gn(const Handle &h, const T *bdata, T *res, double *grad, double *jnorm2, double *fval, int split,
                      int vw, int stage, const int *view_mask, const int *skip, int batch, int kb, double *rscale,
                      ImgForm form)
{
    RayArgs<T> a = base_args<T>(h, form);
    a.VW = vw;
    a.R = bdata;
    a.r_stride = (long long)h.V * h.B;
    a.res = res;
    a.partial = h.d_partial;
    a.part_stride = 4LL * h.V * h.nchunks;
    a.view_mask = view_mask;
    a.skip = skip;
    cudaError_t e = der_groups<T, kGn, false>(h, a, batch, kb, split, stage, form);
    if (e != cudaSuccess) return e;
    const long long outs = (long long)h.V * batch;
    launch_chained(k_finalize, (int)((4 * outs + 63) / 64), 64, 0, h.stream, h.d_partial, h.V, h.nchunks, batch, a.part_stride, 0,
                                                            grad, jnorm2, fval, 0.5, rscale, view_mask, skip);
    return cudaGetLastError();
}

#define CTGB_RAY_INSTANTIATE(T)                                                                             \
    template cudaError_t launch_pairs_img<T>(const Handle &, const T *, int, const int *, const double *,   \
                                             const double *);                                              \
    template cudaError_t launch_sino_layout<T>(const Handle &, const T *, int, int, const int *,            \
                                               const double *, const double *);                            \
    template cudaError_t launch_prep_forward<T>(const Handle &, const T *, int, const int *, const double *, \
                                                const double *);                                           \
    template cudaError_t launch_forward<T>(const Handle &, T *, int, int, int, int, int, const int *, bool, int); \
    template cudaError_t launch_jvp<T>(const Handle &, const double *, const double *, T *, int, int, int, int, \
                                       int, long long, ImgForm);                                          \
    template cudaError_t launch_vjp<T>(const Handle &, const T *, double *, double *, int, int, int, int, int, \
                                       long long, int, ImgForm);                                          \
    template cudaError_t launch_gn<T>(const Handle &, const T *, T *, double *, double *, double *, int,    \
                                      int, int, const int *, const int *, int, int, double *, ImgForm);

CTGB_RAY_INSTANTIATE(float)
CTGB_RAY_INSTANTIATE(double)

}  // namespace ctgb
