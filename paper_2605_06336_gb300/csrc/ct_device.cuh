// Device helpers shared by the kernel translation units.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "ct_internal.cuh"

namespace ctgb {

template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };
template <typename T> using pair_t = typename Pair<T>::type;

// Launches with programmatic stream serialization: a kernel may be scheduled
// while its predecessor in the stream drains, so the launch latency between two
// dependent kernels overlaps.  Every such kernel starts with chain_wait(),
// before any access to global memory and before any return: it waits until
// the predecessor has completed and its writes are visible (and, as that one
// waited too, everything before it).  One image of 256^2 / 180 views, H and
// H^T, four launches: 38.9 -> 29.6 us a pass.  No kernel triggers its successor
// before it ends: resident early, the successor's CTAs take the places of the
// predecessor's last ones (42.4 us with the trigger at entry).
// What this relies on: a kernel reads what its predecessor wrote also through
// read-only loads (__ldg, const __restrict__), whose data must not change while the
// kernel runs; these have to stay behind the wait.  The wait is volatile and clobbers
// memory, it is the first statement of every kernel, and each such load is
// under a condition or in a loop that comes after it, or volatile: a load that
// the compiler may move but not speculate has nowhere ahead of it to go.  A new
// kernel keeps to that, and none may signal its successor before its last write.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KA, typename... A>
inline cudaError_t launch_chained(void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                  A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KA>(args)...);
}

__device__ __forceinline__ int cell_of(long long Q) { return (int)(Q >> kFracBits); }

// Fraction q - floor(q) of a fixed-point value: the top 23 (or 48) of the 48
// fractional bits placed in the mantissa of 1.m, minus one.
__device__ __forceinline__ float frac_of(long long Q, float)
{
    const unsigned m = (unsigned)((unsigned long long)Q >> (kFracBits - 23)) & 0x7FFFFFu;
    return __uint_as_float(m | 0x3F800000u) - 1.0f;
}
__device__ __forceinline__ double frac_of(long long Q, double)
{
    const unsigned long long m = ((unsigned long long)Q & ((1ull << kFracBits) - 1ull)) << (52 - kFracBits);
    return __longlong_as_double((long long)(m | 0x3FF0000000000000ull)) - 1.0;
}

// Fixed-point q of ray b at march index r (see ct_internal.cuh).
__device__ __forceinline__ long long line_at(const ViewGeo &g, int b, int r, int N)
{
    return g.Qc + (long long)(b + g.n0) * g.Qb + (long long)(2 * r - (N - 1)) * g.Qh;
}

__device__ __forceinline__ double warp_sum(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Sums of NQ (a power of two) values over the warp, each by the tree of
// warp_sum: while more than one is left, the lanes at each level keep half of
// them and hand the other half over, so that four sums take 6
// additions a lane instead of 20 (an FP64 addition occupies the pipe for 64
// cycles; the same additions, so the same bits).  Lane l returns the sum of
// value l / (32 / NQ).
template <int NQ, int O = 16> __device__ __forceinline__ double warp_sums(double (&x)[NQ], int lane)
{
    if constexpr (O == 0) {
        return x[0];
    } else if constexpr (NQ > 1) {
        double h[NQ / 2];
        const bool up = lane & O;
#pragma unroll
        for (int i = 0; i < NQ / 2; ++i) {
            const double send = up ? x[i] : x[i + NQ / 2], keep = up ? x[i + NQ / 2] : x[i];
            h[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
        return warp_sums<NQ / 2, O / 2>(h, lane);
    } else {
        x[0] += __shfl_xor_sync(0xffffffffu, x[0], O);
        return warp_sums<1, O / 2>(x, lane);
    }
}

// floor(t) and t - floor(t) in [0, 1] for |t| < 2^22 without a conversion
// instruction: t - 1/2 is rounded to an integer by the 1.5 * 2^23 shift.
// When t is an integer the rounding may land on t - 1, giving f = 1, which
// the hat weights treat the same as f = 0 on the next cell.
__device__ __forceinline__ void floor_split(float t, int &m, float &f)
{
    const float magic = 12582912.0f;
    const float tr = __fadd_rn(__fsub_rn(t, 0.5f), magic);
    m = __float_as_int(tr) - 0x4B400000;
    f = __fsub_rn(t, __fsub_rn(tr, magic));
}

// Per-view derivative constants in the working precision.  The FP64 form
// recomputes them from (c, s) in double.
template <typename T> struct GeoT;
template <> struct GeoT<float> {
    __device__ static float w(const ViewGeo &g) { return g.w; }
    __device__ static float dw(const ViewGeo &g) { return g.dw; }
    __device__ static float gs(const ViewGeo &g) { return g.gs; }
    __device__ static float gh(const ViewGeo &g, int) { return g.gh; }
    __device__ static float gr(const ViewGeo &g) { return g.gr; }
    __device__ static float qb(const ViewGeo &g) { return g.qbf; }
    __device__ static float sb(const ViewGeo &g, int b) { return g.sb0 + (float)b; }
};
template <> struct GeoT<double> {
    __device__ static double w(const ViewGeo &g) { return g.mode ? 1.0 / fabs(g.s) : 1.0 / fabs(g.c); }
    __device__ static double dw(const ViewGeo &g)
    {
        return g.mode ? -copysign(1.0, g.s) * g.c / (g.s * g.s) : copysign(1.0, g.c) * g.s / (g.c * g.c);
    }
    __device__ static double gs(const ViewGeo &g) { return g.mode ? g.c / (g.s * g.s) : g.s / (g.c * g.c); }
    __device__ static double gh(const ViewGeo &g, int N)
    {
        const double h = 0.5 * (N - 1);
        return g.mode ? h / (g.s * g.s) : -h / (g.c * g.c);
    }
    __device__ static double gr(const ViewGeo &g) { return g.mode ? -1.0 / (g.s * g.s) : 1.0 / (g.c * g.c); }
    __device__ static double qb(const ViewGeo &g) { return g.mode ? -1.0 / g.s : 1.0 / g.c; }
    __device__ static double sb(const ViewGeo &g, int b) { return g.sb0d + (double)b; }
};

// ---------------------------------------------------------------------------
// ray march arguments (ct_ray.cu, ct_band.cu)
// ---------------------------------------------------------------------------
enum RayMode { kFwd = 0, kJvp = 1, kVjp = 2, kGn = 3 };

template <typename T> struct RayArgs {
    const ViewGeo *vg;
    int V, N, B, nchunks, Pp;
    const pair_t<T> *PX, *PT;
    long long pimg_stride;  // pairs per batch element (F * N * Pp)
    int kbase, ngroups;
    T *Y;                   // FWD: [batch][V*B]; JVP: dY
    long long sino_stride;
    const double *dtheta, *ddelta;
    long long dir_stride;   // JVP: doubles between the directions of consecutive images (0: one for all)
    const T *R;             // VJP: r; GN: data b
    T *res;                 // GN: residual (nullable)
    long long r_stride;     // VJP / GN: elements between the R of consecutive images (0: one for all)
    double *partial;        // VJP / GN: [image][view][chunk][4]
    long long part_stride;  // doubles between the partials of consecutive images (V * nchunks * 4)
    const int *view_mask;   // GN: views with mask 0 are skipped (nullable)
    const int *skip;        // whole launch is a no-op when *skip != 0 (nullable)
    const int *order;       // view order (nullable: identity)
    int VW;                 // view slots per CTA
    int segs;               // band-staged forward: row segments per ray, one CTA each (1: whole rays)
    T *fpart;               // segments 1..segs-1 of the band-staged forward (segment 0 goes to Y)
    long long fpart_stride; // elements per segment in fpart
    const float *QX, *QT;   // interleaved images (FP32 forward)
    long long qimg_stride;  // floats per image in the interleaved layout (F * N * Pp)
    int kend;               // FWD: images k >= kend of a group are not written (a batch below the
                            // interleaved layout's ends inside a group)
};

// Warp-uniform row range [rlo, rhi] covering every row where one of the
// warp's rays has -1 < q < N; rows added by the union or by the two-row
// margin read exact zeros.
__device__ __forceinline__ void warp_rows(const ViewGeo &g, int b, bool active, int N, int &rlo, int &rhi)
{
    if (g.flags & kAllRows) {
        rlo = 0;
        rhi = N - 1;
        return;
    }
    const float r1 = fmaf((float)b, g.gam, g.alo);
    const float r2 = fmaf((float)b, g.gam, g.ahi);
    const float lo = fminf(fmaxf(fminf(r1, r2) - 2.0f, 0.0f), (float)N);
    const float hi = fmaxf(fminf(fmaxf(r1, r2) + 2.0f, (float)(N - 1)), -1.0f);
    int l = (int)floorf(lo), u = (int)ceilf(hi);
    if (!active) {
        l = N;
        u = -1;
    }
    rlo = __reduce_min_sync(0xffffffffu, l);
    rhi = __reduce_max_sync(0xffffffffu, u);
}

// Element indices (cell + 2, clamped to the row's zero padding) and fractions
// of U consecutive rows from the exact line value Q at the first.  FP32: the
// rows are walked relative to the first one's cell with 55 fractional bits (the
// 48 of the line, shifted), so the high word holds the cell offset in its top
// 9 bits and the 23 bits of the fraction below them: one shift, one logic
// operation and one add-and-clamp a row, where the full-range line needs a
// two-word shift, two clamps and a second shift (the integer pipe was the bound
// of one image per lane: 74 % busy, now 58).  The same bits as cell_of and
// frac_of.  One image of 2048^2, 120 views: 362 -> 282 us; 256^2 / 180 views:
// 18.6 -> 16.3.  FP64 without FRAC: the indices alone; ray_frac gives a row's
// fraction when its sum is formed (an FP64 subtraction, not spent on the rows
// past a segment's end: the fan beam's choice, 130^2 / 180 views, J of 8 images
// 468 -> 399 us with the sums of those rows left out too; the parallel beam, whose
// segments end together, is faster with the fractions of a block formed ahead of
// its loads: 32^2 / 360 views, 4 images, forward 20.4 us against 24.7).
template <typename T, int U, bool FRAC>
__device__ __forceinline__ void ray_cells(long long Q, long long dQ, unsigned lim, unsigned (&idx)[U], T (&f)[U])
{
    if constexpr (std::is_same<T, float>::value) {
        static_assert(kFracBits == 48 && U <= 16, "cell offsets of a block fit 9 bits");
        const unsigned base = (unsigned)(cell_of(Q) + 2);
        const long long L0 = (long long)(((unsigned long long)Q << 16) >> 9), dL = dQ << 7;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int hi = (int)((L0 + (long long)u * dL) >> 32);
            // (a negative index is a large unsigned one)
            idx[u] = __viaddmin_u32((unsigned)(hi >> 23), base, lim);
            f[u] = __int_as_float((hi & 0x7FFFFF) | 0x3F800000) - 1.0f;
        }
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long Qu = Q + (long long)u * dQ;
            idx[u] = min((unsigned)(cell_of(Qu) + 2), lim);
            if constexpr (FRAC) f[u] = frac_of(Qu, T());
        }
    }
}
// Fraction of row u of the block.
template <typename T, int U>
__device__ __forceinline__ T ray_frac(long long Q, long long dQ, const T (&f)[U], int u)
{
    if constexpr (std::is_same<T, float>::value) return f[u];
    else return frac_of(Q + (long long)u * dQ, T());
}

// Per-ray output of a march: the forward stores w * sum for each image, the
// JVP stores the directional derivative, the VJP and Gauss-Newton modes write
// per-(view, chunk) partial sums reduced over the warp in a fixed order.
template <typename T, int MODE, bool OFFS, int KB>
__device__ __forceinline__ void ray_epilogue(const RayArgs<T> &a, const ViewGeo &g, int v, int b, bool active, int k0,
                                             int chunk, int lane, const T (&acc)[(MODE == kFwd) ? KB : 3 * KB])
{
    const T wv = GeoT<T>::w(g);
    if constexpr (MODE == kFwd) {
        if (active) {
#pragma unroll
            for (int k = 0; k < KB; ++k)
                if (k0 + k < a.kend) a.Y[(size_t)(k0 + k) * a.sino_stride + (size_t)v * a.B + b] = wv * acc[k];
        }
    } else {
        // image k of the group: acc[3k] interpolated sum, acc[3k+1] slope x dq/dtheta, acc[3k+2] slopes;
        // VJP / GN: NQ quantities per image, reduced over the warp together
        constexpr int NQ = MODE == kGn ? 4 : (OFFS ? 2 : 1);
        const size_t vb = (size_t)v * a.B + b;
        [[maybe_unused]] double part[KB * NQ];
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const size_t img = (size_t)(k0 + k);
            const T jt = fma(GeoT<T>::dw(g), acc[3 * k], wv * acc[3 * k + 1]);
            const T jd = wv * GeoT<T>::qb(g) * acc[3 * k + 2];
            if constexpr (MODE == kJvp) {
                if (active) {
                    T out = (T)a.dtheta[img * a.dir_stride + v] * jt;
                    if (OFFS) out = fma((T)a.ddelta[img * a.dir_stride + v], jd, out);
                    a.Y[img * a.sino_stride + vb] = out;
                }
            } else if constexpr (MODE == kVjp) {
                double pt = 0.0, pd = 0.0;
                if (active) {
                    const T r = a.R[img * a.r_stride + vb];
                    pt = (double)(r * jt);
                    if (OFFS) pd = (double)(r * jd);
                }
                part[k * NQ] = pt;
                if constexpr (OFFS) part[k * NQ + 1] = pd;
            } else {  // kGn
                // pr: the rounding scale |r| (|H x| + |b|) of the misfit (Armijo noise floor)
                double pg = 0.0, pj = 0.0, pf = 0.0, pr = 0.0;
                if (active) {
                    const T hx = wv * acc[3 * k];
                    const T bb = a.R[img * a.r_stride + vb];
                    const T rr = hx - bb;
                    if (a.res) a.res[img * a.sino_stride + vb] = rr;
                    pg = (double)rr * (double)jt;
                    pj = (double)jt * (double)jt;
                    pf = (double)rr * (double)rr;
                    pr = fabs((double)rr) * (fabs((double)hx) + fabs((double)bb));
                }
                part[k * NQ] = pg;
                part[k * NQ + 1] = pj;
                part[k * NQ + 2] = pf;
                part[k * NQ + 3] = pr;
            }
        }
        if constexpr (MODE != kJvp) {
            constexpr int PER = 32 / (KB * NQ);  // lanes holding one sum
            const double s = warp_sums(part, lane);
            if (lane % PER == 0) {
                const int q = lane / PER;
                a.partial[(size_t)(k0 + q / NQ) * a.part_stride + ((size_t)v * a.nchunks + chunk) * 4 + q % NQ] = s;
            }
        }
    }
}

// Band-staged FP32 ray march (ct_band.cu): the rows a CTA's rays cross are
// staged in shared memory block by block.  a.VW in {4, 8} view slots, rb in
// {4, 8} rows per staged block, kb in {1, 2, 4, 8} images (forward only).
// Results are bit-identical to k_ray with one row segment per ray.
bool band_shape_ok(int mode, int kb, int vw, int rb);
cudaError_t run_ray_band(const Handle &h, const RayArgs<float> &a, int mode, bool offs, int kb, int rb);
// Fan-beam ray march (ct_fan.cu) for the same arguments: mode kFwd (kb
// images), kJvp, kVjp (angle and, with offs, offset derivatives) or kGn
// (angle derivatives); split warps share a ray.
template <typename T>
cudaError_t run_fan_ray(const Handle &h, const RayArgs<T> &a, int mode, int kb, int split, bool offs);
// Y[k][v][b] = w_v * (Y + P_1 + ... + P_{segs-1}), summed in segment order.
cudaError_t launch_fwd_combine(const Handle &h, float *Y, const float *P, int segs, long long stride, int batch,
                               const int *skip);

// Resident CTAs per SM of a kernel at a launch shape, queried once per
// (kernel, threads, shared memory) and cached: the occupancy query is a host
// API call that would otherwise cost several microseconds per launch.
inline int resident_per_sm(const void *kernel, int threads, size_t smem)
{
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, size_t>, int> cache;
    const auto key = std::make_tuple(kernel, threads, smem);
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    std::lock_guard<std::mutex> lock(mu);
    cache[key] = per_sm;
    return per_sm;
}

// Grid of a work-item kernel: one CTA per item, so that the hardware hands
// items to SMs as CTAs finish (items differ in cost: chunks at the detector
// edge carry short rays).  Very large item counts are folded into a grid of
// 64 resident waves; the kernels loop over item += gridDim.x.
template <typename K>
inline int persistent_grid(K kernel, int threads, size_t smem, long long work_blocks, int num_sms)
{
    const int per_sm = resident_per_sm((const void *)kernel, threads, smem);
    const long long cap = 64LL * per_sm * num_sms;
    return (int)std::max<long long>(1, std::min(work_blocks, cap));
}

// ---------------------------------------------------------------------------
// transpose kernels (ct_backproject.cu, ct_fan.cu)
// ---------------------------------------------------------------------------
// CTAs per tile of a frame's views (adj_cluster_size in ct_internal.cuh)
inline int adj_segs(const Handle &h, long long tiles, int split, int fixed, int alone = 0)
{
    return adj_cluster_size(std::max(1, h.V / h.F), tiles, h.num_sms, split, fixed, alone);
}

// Launch of a transpose kernel: 256 threads, the a.segs CTAs of a tile one cluster.
template <typename A> inline cudaError_t launch_cluster(void (*kern)(A), const A &a, const Handle &h, size_t smem)
{
    if (smem > 48 * 1024) return cudaErrorInvalidValue;  // no kernel here needs more
    const long long items = (long long)a.ngroups * a.F * a.tps * a.tps * a.segs;
    int grid = persistent_grid(kern, 256, smem, items, h.num_sms);
    grid -= grid % a.segs;  // whole clusters (items is a multiple of segs, so grid >= segs)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.segs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

__device__ __forceinline__ void cp_async16_zfill(void *smem, const void *gmem, bool valid)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    const int bytes = valid ? 16 : 0;  // 0: the destination is zero-filled, the source is not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// Two floats in a register pair, for the packed multiply-adds (fma.rn.f32x2:
// one issue slot for two).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float half2f(f32x2 v, int i) { return __uint_as_float((unsigned)(v >> (32 * i))); }

}  // namespace ctgb
