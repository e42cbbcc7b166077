// vr_modes.cu -- the paper's other uses of the same ray march:
//   - maximum intensity projection (Section 3.3.1): the largest sample value
//     on each ray, shown through the colour map;
//   - the sigma-clipping transfer function (Section 4.5): a statistical
//     mini-map holds the mean and standard deviation of regions of the cube,
//     and each sample value is scaled by the statistics interpolated at its
//     position before the table lookup;
//   - the 3D spectrum tool (Section 4.4): the data profile along one pixel's
//     line of sight, at the renderer's sample positions.
// Same camera, clipping, sampling, brick layouts and work queue as
// vr_forward.cu.
#include "vr_modes.cuh"

#include <algorithm>
#include <cmath>

namespace vr {

// ---------------------------------------------------------------------------
// Maximum intensity projection
// ---------------------------------------------------------------------------

// Resident CTAs the register budget is sized for, and samples whose gathers
// are in flight ahead of the one compared: four CTAs and two samples for the
// texture layers (a 1080p view of the 1024^3 cube along x 1.49 -> 1.40 ms
// against five CTAs with one, two samples at five CTAs 1.59; a tilted 45-degree
// view of a 512^3 cube 517 -> 470 us), the compiler's choice and one for the
// brick layouts.
template <typename T> struct ModeMinBlocks { static constexpr int value = 0; };   // 0: no minimum
template <> struct ModeMinBlocks<TexLayers<float>> { static constexpr int value = 4; };
template <typename T> struct ModeDepth { static constexpr int value = 1; };
template <> struct ModeDepth<TexLayers<float>> { static constexpr int value = 2; };

// Largest interpolated value of the ray's samples (all of them: no early
// termination); the next samples' gathers are issued before the current one
// is compared (depth + 1 register sets in turn).
template <typename T, int LOG2B, int L, int D>
__device__ __forceinline__ float march_max(const VolDev &v, const ParamDev &p, const Ray &ray, bool active)
{
    float m = -INFINITY;
    int k = 0;
    Cell c0, c1, c2;
    Gathered<T, L> f0, f1, f2;
    auto fetch = [&](int q, Cell &c, Gathered<T, L> &f) {
        if (q >= ray.n) return;
        c = locate_t<T, LOG2B, L, false>(v, sample_pos(ray, q, p.step));
        fetch_corners<T, LOG2B, L>(v, c, f);
    };
    auto step = [&](const Cell &cur, const Gathered<T, L> &fc, Cell &nxt, Gathered<T, L> &fn) {
        fetch(k + D, nxt, fn);
        m = fmaxf(m, interp_corners(cur, fc));
        if (++k >= ray.n) active = false;
    };
    if (active) {
        fetch(0, c0, f0);
        if constexpr (D == 2) fetch(1, c1, f1);
    }
    while (__any_sync(kFull, active)) {
        if constexpr (D == 1) {
            // a vote for each step: with one for two, 16-bit views (30, over 35 to
            // 2000 MB of paired copies) ran at 0.88 to 1.06 of this speed, the
            // largest the slowest
            if (active) step(c0, f0, c1, f1);
            if (!__any_sync(kFull, active)) break;
            if (active) step(c1, f1, c0, f0);
        } else {
            if (active) step(c0, f0, c2, f2);
            if (active) step(c1, f1, c0, f0);
            if (active) step(c2, f2, c1, f1);
        }
    }
    return m;
}

// The same maximum with eight lanes to a ray (as march_group): each lane its
// own samples, then the group's largest, on every lane of the group.
template <typename T, int LOG2B, int L>
__device__ __forceinline__ float march_max_group(const VolDev &v, const ParamDev &p, const Ray &ray, bool hit)
{
    const int n = hit ? ray.n : 0;
    int k = (threadIdx.x & 31) / (32 / kGroup);
    float m = -INFINITY;
    Cell c0, c1;
    Gathered<T, L> f0, f1;
    auto fetch = [&](int q, Cell &c, Gathered<T, L> &f) {
        if (q >= n) return;
        c = locate_t<T, LOG2B, L, false>(v, sample_pos(ray, q, p.step));
        fetch_corners<T, LOG2B, L>(v, c, f);
    };
    auto step = [&](const Cell &cur, const Gathered<T, L> &fc, Cell &nxt, Gathered<T, L> &fn) {
        fetch(k + kGroup, nxt, fn);
        if (k < n) m = fmaxf(m, interp_corners(cur, fc));
        k += kGroup;
    };
    fetch(k, c0, f0);
    while (__any_sync(kFull, k < n)) {
        step(c0, f0, c1, f1);
        step(c1, f1, c0, f0);
    }
#pragma unroll
    for (int o = 32 / kGroup; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    return m;
}

// The pixel is the table entry of the largest value composited once over
// the background; a ray that misses the box shows the background.
template <typename T, int LOG2B, int L, bool GROUPS>
__global__ void __launch_bounds__(kModeThreads, ModeMinBlocks<T>::value) mip_kernel(VolDev v, CamDev c, ParamDev p, float4 *out,
                                                            uint32_t *nsamples, unsigned *counter, Tiles t)
{
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= t.ntiles) break;
        const LanePixel px = lane_pixel<GROUPS>(t, tile, c.W, c.H);
        Ray ray;
        const bool hit = px.march && setup_ray(c, v.nx, v.ny, v.nz, p.step, px.i, px.j, ray);
        float m;
        if constexpr (GROUPS) m = march_max_group<T, LOG2B, L>(v, p, ray, hit);
        else m = march_max<T, LOG2B, L, ModeDepth<T>::value>(v, p, ray, hit);
        if (!px.writes) continue;
        const long long at = (long long)px.j * c.W + px.i;
        float4 o = p.bg;
        if (hit) {
            TfPos tp;
            const float4 e = tf_lookup_l1(p, m, tp);
            const float a = e.w, t = 1.0f - e.w;
            o = make_float4(fmaf(a, e.x, t * p.bg.x), fmaf(a, e.y, t * p.bg.y), fmaf(a, e.z, t * p.bg.z),
                            fmaf(t, p.bg.w, a));
        }
        out[at] = o;
        if (nsamples) nsamples[at] = hit ? (uint32_t)ray.n : 0u;
    }
}

// ---------------------------------------------------------------------------
// Sigma clipping
// ---------------------------------------------------------------------------

// Device view of a mini-map: (mean, sd) per point, x fastest; point i of an
// axis sits at voxel (i + 1/2) region - 1/2.
struct MiniDev {
    const float2 *mm;
    int mx, my, mz;
    float rx, ry, rz;          // 1 / region size
    unsigned *status;          // the bounds-check build's report
};

// First point and weight of an axis (an axis of one point: that point, 0).
__device__ __forceinline__ void mini_axis(float p, float rinv, int m, int &i0, float &w)
{
    const float g = fmaf(p + 0.5f, rinv, -0.5f);
    i0 = max(min(max(__float2int_rd(g), 0), m - 2), 0);
    w = m < 2 ? 0.0f : fminf(fmaxf(g - (float)i0, 0.0f), 1.0f);
}

// The sample value in units of the local standard deviation above the local
// mean (trilinear on the mini-map at the sample's position; a standard
// deviation below 1e-30 counts as 1e-30).  The eight points around the last
// sample are kept in registers (each x edge as its first value and its
// difference): a ray stays in a mini-map cell for about a region's length,
// and the march is bound by instructions, of which the eight loads and their
// addresses were a fifth.  I: the type that holds the map's point numbers,
// long long from 2^31 points (regions of a voxel or two of a very large cube;
// in every kernel it cost 0.7 to 4%).
template <typename I> struct SigmaMap {
    MiniDev m;
    mutable I at = -1;                             // the kept cell's first point
    mutable float2 a[4], d[4];                     // edges (y0, z0), (y1, z0), (y0, z1), (y1, z1)
    __device__ __forceinline__ explicit SigmaMap(const MiniDev &md) : m(md) {}
    __device__ __forceinline__ float operator()(float v, const Cell &c) const
    {
        int x0, y0, z0;
        float wx, wy, wz;
        mini_axis((float)c.x0 + c.fx, m.rx, m.mx, x0, wx);
        mini_axis((float)c.y0 + c.fy, m.ry, m.my, y0, wy);
        mini_axis((float)c.z0 + c.fz, m.rz, m.mz, z0, wz);
        const I p = ((I)z0 * m.my + y0) * m.mx + x0;
        if (p != at) {
            at = p;
            const int dx = m.mx > 1 ? 1 : 0, dy = m.my > 1 ? m.mx : 0;
            const I dz = m.mz > 1 ? (I)m.mx * m.my : 0;
            if constexpr (kBoundsCheck) {
                const long long n = (long long)m.mx * m.my * m.mz;
                if (!index_ok(m.status, p, n) || !index_ok(m.status, (long long)p + dx + dy + dz, n)) {
                    at = -1;
                    return 0.0f;
                }
            }
            const float2 *b = m.mm + p;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 *e = b + ((q & 1) ? dy : 0) + ((q & 2) ? dz : 0);
                const float2 u = __ldg(e), w = __ldg(e + dx);
                a[q] = u;
                d[q] = make_float2(w.x - u.x, w.y - u.y);
            }
        }
        auto lerp = [](float a, float b, float w) { return fmaf(w, b - a, a); };
        float2 s[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = make_float2(fmaf(wx, d[q].x, a[q].x), fmaf(wx, d[q].y, a[q].y));
        const float mean = lerp(lerp(s[0].x, s[1].x, wy), lerp(s[2].x, s[3].x, wy), wz);
        const float sd = lerp(lerp(s[0].y, s[1].y, wy), lerp(s[2].y, s[3].y, wy), wz);
        return (v - mean) / fmaxf(sd, 1e-30f);
    }
};

// Six four-warp CTAs per SM (80 registers): with the kept mini-map cell the
// 1280 x 720 view of a 640 x 720 x 500 cube takes 0.76 ms at six, 0.98 at five
// and 1.07 at four (before: 1.02 ms at three eight-warp CTAs).
constexpr int kSigmaThreads = 128;

template <typename T, int LOG2B, int L, bool GROUPS, typename I>
__global__ void __launch_bounds__(kSigmaThreads, 6) sigma_kernel(VolDev v, CamDev c, ParamDev p, MiniDev m, float4 *out,
                                                              uint32_t *nsamples, unsigned *counter, Tiles t)
{
    if (GROUPS && left_to_lanes(t, p)) return;
    const int lane = threadIdx.x & 31;
    const SigmaMap<I> map(m);
    const float z = GROUPS || skips_transparent<T, SigmaMap<I>>() ? transparent_below(p) : 0.0f;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= t.ntiles) break;
        const LanePixel px = lane_pixel<GROUPS>(t, tile, c.W, c.H);
        Ray ray;
        const bool hit = px.march && setup_ray(c, v.nx, v.ny, v.nz, p.step, px.i, px.j, ray);
        Composite acc{0.0f, 0.0f, 0.0f, 1.0f};
        int used;
        if constexpr (GROUPS) used = march_group<T, LOG2B, L, kGroup, SigmaMap<I>>(v, p, ray, hit, acc, z, map);
        else used = march_ray<T, LOG2B, L, SigmaMap<I>>(v, p, ray, hit, acc, z, map);
        if (px.writes) write_pixel(p, acc, hit ? used : 0, out, nsamples, (long long)px.j * c.W + px.i);
    }
}

cudaError_t launch_mip(const VolDev &v, vr_dtype dt, const CamDev &c, const ParamDev &p, const Tiles &t, float4 *out,
                       uint32_t *nsamples, unsigned *counter, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    return visit_layout_tex(
        v, dt,
        [&](auto lay) {
            using Y = decltype(lay);
            auto fn = t.groups ? mip_kernel<typename Y::type, Y::log2b, Y::order, true>
                             : mip_kernel<typename Y::type, Y::log2b, Y::order, false>;
            fn<<<persistent_grid(fn, t.ntiles), kModeThreads, 0, s>>>(v, c, p, out, nsamples, counter, t);
            return cudaGetLastError();
        },
        cudaErrorInvalidValue);
}

cudaError_t launch_sigma(const VolDev &v, vr_dtype dt, const CamDev &c, const ParamDev &p, const Tiles &t,
                         const float *minimap,
                         const int region[3], float4 *out, uint32_t *nsamples, unsigned *counter, cudaStream_t s)
{
    MiniDev m;
    m.mm = reinterpret_cast<const float2 *>(minimap);
    m.mx = (v.nx + region[0] - 1) / region[0];
    m.my = (v.ny + region[1] - 1) / region[1];
    m.mz = (v.nz + region[2] - 1) / region[2];
    m.rx = (float)(1.0 / region[0]);
    m.ry = (float)(1.0 / region[1]);
    m.rz = (float)(1.0 / region[2]);
    m.status = v.status;
    const bool wide = (long long)m.mx * m.my * m.mz > 0x7fffffffLL;
    if (wide && t.groups) return cudaErrorInvalidValue;           // built with a ray to a lane only
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    return visit_layout_tex(
        v, dt,
        [&](auto lay) {
            using Y = decltype(lay);
            auto fn = wide     ? sigma_kernel<typename Y::type, Y::log2b, Y::order, false, long long>
                    : t.groups ? sigma_kernel<typename Y::type, Y::log2b, Y::order, true, int>
                               : sigma_kernel<typename Y::type, Y::log2b, Y::order, false, int>;
            fn<<<persistent_grid(fn, t.ntiles, kSigmaThreads), kSigmaThreads, 0, s>>>(v, c, p, m, out, nsamples, counter, t);
            if (t.by_table) {                     // both ways: one of the two finds nothing to do
                const Tiles q = lane_tiles(t);
                fn = sigma_kernel<typename Y::type, Y::log2b, Y::order, false, int>;
                fn<<<persistent_grid(fn, q.ntiles, kSigmaThreads), kSigmaThreads, 0, s>>>(v, c, p, m, out, nsamples, counter, q);
            }
            return cudaGetLastError();
        },
        cudaErrorInvalidValue);
}

// ---------------------------------------------------------------------------
// Statistical mini-map: mean and standard deviation of each region's voxels,
// one CTA per region.
//
// FP64 adds and fused multiply-adds run at two lanes per clock and SM here:
// two passes of them take 5.1 ms for a 768^3 float cube in regions of 32^3,
// where reading its bricks takes 0.33 ms; this takes 0.94 ms (1.8 with a NaN in
// every region, 2.1 where every region takes the second pass below), bound by
// FP32 instructions.  So a region is read once, and its sums of
// d = a - shift and of d^2 (shift: the region's first voxel) are kept as
// unevaluated sums of two floats, with the rounding errors of every
// subtraction, product and addition carried along (Knuth's two-sum and the
// fused product error): about 25 FP32 operations a voxel.  The low parts are
// plain FP32 sums, so the two are brought back to hi + lo with |lo| below half
// an ulp of hi after kRenorm values or a column of them.  The variance
// S2 / n - (S1 / n)^2 is formed in FP64 and loses what the shift is away from the
// mean: where (S1 / n)^2 exceeds 256 variances (a first voxel 16 deviations off,
// hardly ever but in outliers) a second pass has the mean found as its shift,
// and so do deviations whose squares leave the float range, scaled by a power of
// two.  Against 64 bits, restated on the CPU over noise, outliers up to 1e7 as
// the first voxel and quantised data in regions of up to 128^3: 2e-9 of the
// deviation at most (5e-8 with no renorm, 4e-6 without the second pass), where
// rounding the result to float is 6e-8.
// A region with a voxel that is not finite needs no sums; one above 2^21
// voxels, or whose differences overflow, takes two FP64 passes.
// ---------------------------------------------------------------------------

constexpr int kMiniThreads = 256;                  // 64 or 128 for regions of few voxels (region_sums: at most 8 warps)
constexpr long long kMiniMaxOnePass = 1LL << 21;
constexpr float kMiniMinFar = 1e-12f, kMiniMaxFar = 1e18f;        // largest deviations whose squares need no scale

__device__ __forceinline__ double block_sum(double x, double *red)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();                  // red[] may still be read by the previous call
    if (lane == 0) red[w] = x;
    __syncthreads();
    double t = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
    return t;
}

// Offset of one coordinate in the x-fastest bricks: the brick that owns it
// (the last voxel of an axis may sit in the apron of the last brick) and the
// place inside, in elements.
__device__ __forceinline__ long long axis_offset(int c, int log2b, int nb, long long brick_pitch, int pitch)
{
    const int b = min(c >> log2b, nb - 1);
    return b * brick_pitch + (long long)(c - (b << log2b)) * pitch;
}

// Voxel (x, y, z) of the x-fastest bricks.
template <typename T>
__device__ __forceinline__ float brick_voxel(const VolDev &v, int x, int y, int z)
{
    const int B1 = (1 << v.log2b) + 1;
    const long long e = axis_offset(x, v.log2b, v.nbx, v.stride, 1) +
                        axis_offset(y, v.log2b, v.nby, v.stride * v.nbx, B1) +
                        axis_offset(z, v.log2b, v.nbz, v.stride * v.nbx * v.nby, B1 * B1);
    return to_f(static_cast<const T *>(v.data)[e]);
}

// A sum kept as hi + lo, hi the rounded sum so far.
constexpr int kRenorm = 128;
struct TwoFloat {
    float hi = 0.0f, lo = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float s = __fadd_rn(hi, x), b = __fadd_rn(s, -hi);
        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -b)), __fadd_rn(x, -b)));
        hi = s;
    }
    __device__ __forceinline__ void renorm()
    {
        const float x = lo;
        lo = 0.0f;
        add(x);
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
    // the sum over the warp, on every lane
    __device__ __forceinline__ void warp_sum()
    {
        for (int o = 16; o > 0; o >>= 1) {
            const float h = __shfl_xor_sync(kFull, hi, o), l = __shfl_xor_sync(kFull, lo, o);
            add(h);
            lo = __fadd_rn(lo, l);
        }
    }
};

// A region of voxels [x0, x0 + lx) x [y0, y0 + ly) x [z0, z0 + lz).
struct Region {
    int x0, y0, z0, lx, ly, lz;
};

// Calls f(value) for every voxel of the region (each thread its own) and
// after(n) after at most n of a thread's, those of one (x, y).
template <typename T, typename F, typename G>
__device__ __forceinline__ void for_region(const VolDev &v, const Region &q, F &&f, G &&after)
{
    const T *data = static_cast<const T *>(v.data);
    const int B1 = (1 << v.log2b) + 1;
    // threads: 2^bx along x, then 2^by along y, the rest along z
    const int bx = min(q.lx > 1 ? 32 - __clz(q.lx - 1) : 0, 5);
    const int by = min(q.ly > 1 ? 32 - __clz(q.ly - 1) : 0, 31 - __clz((int)blockDim.x) - bx);
    const int tx = threadIdx.x & ((1 << bx) - 1), ty = (threadIdx.x >> bx) & ((1 << by) - 1);
    const int tz = threadIdx.x >> (bx + by), sz = (int)blockDim.x >> (bx + by);
    constexpr int U = 4;                                    // loads in flight
    for (int x = tx; x < q.lx; x += 1 << bx) {
        const long long ex = axis_offset(q.x0 + x, v.log2b, v.nbx, v.stride, 1);
        for (int y = ty; y < q.ly; y += 1 << by) {
            const T *row = data + ex + axis_offset(q.y0 + y, v.log2b, v.nby, v.stride * v.nbx, B1);
            for (int z = tz; z < q.lz; z += U * sz) {
                T raw[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (z + u * sz < q.lz)
                        raw[u] = row[axis_offset(q.z0 + z + u * sz, v.log2b, v.nbz, v.stride * v.nbx * v.nby, B1 * B1)];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (z + u * sz >= q.lz) break;
                    f(to_f(raw[u]));
                }
            }
            after(q.lz / sz + 1);
        }
    }
}

// Sums over the region of d = (a - shift) scale and d^2 (SCALED; else scale is
// 1), and the largest |d|, on every thread of the CTA.
struct RegionSums {
    double s1, s2;
    float far;
};

template <typename T, bool SCALED>
__device__ __forceinline__ RegionSums region_sums(const VolDev &v, const Region &q, float shift, float scale, double *red)
{
    TwoFloat s1, s2;
    float far = 0.0f;
    int run = 0;
    for_region<T>(
        v, q,
        [&](float a) {
            float d = __fadd_rn(a, -shift);
            const float b = __fadd_rn(d, -a);                                          // d + e = a - shift
            float e = __fadd_rn(__fadd_rn(a, -__fadd_rn(d, -b)), __fadd_rn(-shift, -b));
            if (SCALED) d = __fmul_rn(d, scale), e = __fmul_rn(e, scale);
            const float p = __fmul_rn(d, d);
            s1.add(d);
            s1.lo = __fadd_rn(s1.lo, e);
            s2.add(p);
            s2.lo = __fadd_rn(s2.lo, __fmaf_rn(__fadd_rn(d, d), e, __fmaf_rn(d, d, -p)));
            far = fmaxf(far, fabsf(d));
        },
        [&](int n) {
            if ((run += n) >= kRenorm) {
                s1.renorm();
                s2.renorm();
                run = 0;
            }
        });
    // over the warps in FP64 by the first of them (on every thread they would take
    // a fifth of a 32^3 region's time)
    s1.warp_sum();
    s2.warp_sum();
    for (int o = 16; o > 0; o >>= 1) far = fmaxf(far, __shfl_xor_sync(kFull, far, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = (int)(blockDim.x >> 5);
    double *far_of = red + 16;                    // red: 8 warps' s1, s2, far, and the three totals
    __syncthreads();                              // red[] may still be read by the previous call
    if (lane == 0) red[warp] = s1.value(), red[8 + warp] = s2.value(), far_of[warp] = (double)far;
    __syncthreads();
    if (warp == 0) {
        double x = lane < warps ? red[lane] : 0.0, y = lane < warps ? red[8 + lane] : 0.0;
        far = lane < warps ? (float)far_of[lane] : 0.0f;
        for (int o = 4; o > 0; o >>= 1) {
            x += __shfl_xor_sync(kFull, x, o);
            y += __shfl_xor_sync(kFull, y, o);
            far = fmaxf(far, __shfl_xor_sync(kFull, far, o));
        }
        if (lane == 0) red[24] = x, red[25] = y, red[26] = (double)far;
    }
    __syncthreads();
    RegionSums r;
    r.s1 = red[24];
    r.s2 = red[25];
    far = (float)red[26];
    r.far = far;
    return r;
}

// The region's mean and variance by two passes in FP64.
template <typename T>
__device__ double2 region_two_pass(const VolDev &v, const Region &q, double *red)
{
    const long long cnt = (long long)q.lx * q.ly * q.lz;
    double s = 0.0;
    for (long long e = threadIdx.x; e < cnt; e += blockDim.x) {
        const int x = (int)(e % q.lx), y = (int)((e / q.lx) % q.ly), z = (int)(e / ((long long)q.lx * q.ly));
        s += (double)brick_voxel<T>(v, q.x0 + x, q.y0 + y, q.z0 + z);
    }
    const double mean = block_sum(s, red) / (double)cnt;
    double ss = 0.0;
    for (long long e = threadIdx.x; e < cnt; e += blockDim.x) {
        const int x = (int)(e % q.lx), y = (int)((e / q.lx) % q.ly), z = (int)(e / ((long long)q.lx * q.ly));
        const double d = (double)brick_voxel<T>(v, q.x0 + x, q.y0 + y, q.z0 + z) - mean;
        ss += d * d;
    }
    return make_double2(mean, block_sum(ss, red) / (double)cnt);
}

// What the first pass's sums t about `shift` do not settle (see above).  A call of
// its own, so that its registers do not bound the first pass.
template <typename T>
__device__ __noinline__ double2 region_again(const VolDev &v, const Region &q, float shift, RegionSums t, double *red)
{
    const double n = (double)((long long)q.lx * q.ly * q.lz);
    if (isfinite(t.s1)) {                                       // so every voxel is finite
        shift = (float)((double)shift + t.s1 / n);
        const bool in_range = t.far >= kMiniMinFar && t.far <= kMiniMaxFar;
        const float scale = in_range ? 1.0f : ldexpf(1.0f, min(max(-ilogbf(t.far), -126), 126));
        t = region_sums<T, true>(v, q, shift, scale, red);
        if (isfinite(t.s1) && isfinite(t.s2)) {
            const double m = t.s1 / n, var = fmax(t.s2 / n - m * m, 0.0) / ((double)scale * (double)scale);
            return make_double2((double)shift + m / (double)scale, var);
        }
    } else {
        // NaN, or infinities of both signs: no mean; of one sign: that one; no deviation
        int kinds = 0;
        for_region<T>(v, q, [&](float a) { kinds |= a != a ? 3 : (a == INFINITY ? 1 : (a == -INFINITY ? 2 : 0)); },
                      [](int) {});
        const bool up = __syncthreads_or(kinds & 1), down = __syncthreads_or(kinds & 2);
        if (up || down) return make_double2(up && down ? (double)NAN : (up ? INFINITY : -INFINITY), (double)NAN);
    }
    return region_two_pass<T>(v, q, red);
}

// The region's mean and variance by the one-pass sums.
template <typename T>
__device__ __forceinline__ double2 region_one_pass(const VolDev &v, const Region &q, double *red)
{
    const float shift = brick_voxel<T>(v, q.x0, q.y0, q.z0);
    const RegionSums t = region_sums<T, false>(v, q, shift, 1.0f, red);
    const double n = (double)((long long)q.lx * q.ly * q.lz), m = t.s1 / n, var = t.s2 / n - m * m;
    const bool settled = t.far == 0.0f || (t.far >= kMiniMinFar && t.far <= kMiniMaxFar && m * m <= 256.0 * var);
    if (isfinite(t.s1) && settled) return make_double2((double)shift + m, fmax(var, 0.0));
    return region_again<T>(v, q, shift, t, red);
}

template <typename T>
__global__ void __launch_bounds__(kMiniThreads, 4) minimap_kernel(VolDev v, int rx, int ry, int rz, int mx, int my,
                                                               float2 *out)
{
    __shared__ double red[32];
    const long long at = blockIdx.x;
    const int i = (int)(at % mx), j = (int)((at / mx) % my), k = (int)(at / ((long long)mx * my));
    Region q;
    q.x0 = i * rx, q.y0 = j * ry, q.z0 = k * rz;
    q.lx = min(rx, v.nx - q.x0), q.ly = min(ry, v.ny - q.y0), q.lz = min(rz, v.nz - q.z0);
    const double2 r = (long long)q.lx * q.ly * q.lz <= kMiniMaxOnePass ? region_one_pass<T>(v, q, red)
                                                                       : region_two_pass<T>(v, q, red);
    if (threadIdx.x == 0) out[at] = make_float2((float)r.x, (float)sqrt(r.y));
}

cudaError_t launch_minimap(const VolDev &v, vr_dtype dt, const int region[3], float *dev_out, cudaStream_t s)
{
    const int mx = (v.nx + region[0] - 1) / region[0], my = (v.ny + region[1] - 1) / region[1],
              mz = (v.nz + region[2] - 1) / region[2];
    const long long n = (long long)mx * my * mz;
    if (n > 0x7fffffffLL) return cudaErrorInvalidValue;
    float2 *o = reinterpret_cast<float2 *>(dev_out);
    const long long cnt = (long long)region[0] * region[1] * region[2];
    const int threads = cnt <= 1024 ? 64 : (cnt <= 8192 ? 128 : kMiniThreads);
    switch (dt) {
    case VR_F32: minimap_kernel<float><<<(unsigned)n, threads, 0, s>>>(v, region[0], region[1], region[2], mx, my, o); break;
    case VR_F16: minimap_kernel<__half><<<(unsigned)n, threads, 0, s>>>(v, region[0], region[1], region[2], mx, my, o); break;
    case VR_BF16:
        minimap_kernel<__nv_bfloat16><<<(unsigned)n, threads, 0, s>>>(v, region[0], region[1], region[2], mx, my, o);
        break;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 3D spectrum tool: one thread per sample of pixel (i, j)'s ray.
// ---------------------------------------------------------------------------

template <typename T, int LOG2B>
__global__ void __launch_bounds__(256) profile_kernel(VolDev v, CamDev c, float step, int i, int j, float *values,
                                                       unsigned max_values, unsigned *count)
{
    Ray ray;
    const bool hit = setup_ray(c, v.nx, v.ny, v.nz, step, i, j, ray);
    const int n = hit ? ray.n : 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = (unsigned)n;
    const long long lim = min((long long)n, (long long)max_values);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < lim; k += (long long)gridDim.x * blockDim.x) {
        const Cell cell = locate<LOG2B, 0>(v, sample_pos(ray, (int)k, step));
        Gathered<T, 0> f;
        fetch_corners<T, LOG2B, 0>(v, cell, f);
        values[k] = interp_corners(cell, f);
    }
}

cudaError_t launch_profile(const VolDev &v, vr_dtype dt, const CamDev &c, float step, int i, int j, float *values,
                           unsigned max_values, unsigned *count, cudaStream_t s)
{
    const unsigned blocks = max(1u, min((max_values + 255u) / 256u, 4096u));
    const VolDev vb = v;       // the x-fastest bricks (order 0, plain)
#define VR_PROFILE(TT, LB) profile_kernel<TT, LB><<<blocks, 256, 0, s>>>(vb, c, step, i, j, values, max_values, count)
#define VR_PROFILE_DT(TT)                  \
    switch (v.log2b) {                     \
    case 4: VR_PROFILE(TT, 4); break;      \
    case 5: VR_PROFILE(TT, 5); break;      \
    default: VR_PROFILE(TT, 6); break;     \
    }
    switch (dt) {
    case VR_F32: VR_PROFILE_DT(float); break;
    case VR_F16: VR_PROFILE_DT(__half); break;
    case VR_BF16: VR_PROFILE_DT(__nv_bfloat16); break;
    }
#undef VR_PROFILE_DT
#undef VR_PROFILE
    return cudaGetLastError();
}

}  // namespace vr
