// vr_sortlast.cu -- sort-last rendering (Sections 3.2, 3.4): partial images of
// sub-boxes of cells, composited over one another in depth order.  Same
// camera, clipping, sampling, brick layouts and work queue as vr_forward.cu.
#include "vr_modes.cuh"

#include <algorithm>
#include <cmath>

namespace vr {

// ---------------------------------------------------------------------------
// Sort-last rendering (Sections 3.2 and 3.4): the samples of the whole
// volume's ray whose cell lies in a sub-box [lo, hi) of cells, composited
// into a partial image (premultiplied C, transmittance T, depth of the first
// sample); partial images composite over one another in depth order.
// ---------------------------------------------------------------------------

// As the plain forward (vr_forward.cu): four CTAs and two samples in flight for
// the texture layers, the compiler's choice and the march's own depth otherwise.
template <typename T> struct SubMinBlocks { static constexpr int value = 0; };
template <> struct SubMinBlocks<TexLayers<float>> { static constexpr int value = 4; };
template <typename T> struct SubDepth { static constexpr int value = Pipeline<T>::depth; };
template <> struct SubDepth<TexLayers<float>> { static constexpr int value = 2; };

// Ray parameters where the ray is inside [a, b] along one axis (intersected
// into [s0, s1]); false when it misses.
__device__ __forceinline__ bool slab_range(float q, float d, float a, float b, float &s0, float &s1)
{
    if (d == 0.0f) return q >= a && q <= b;
    const float inv = 1.0f / d;
    float t0 = (a - q) * inv, t1 = (b - q) * inv;
    if (t0 > t1) {
        const float t = t0;
        t0 = t1;
        t1 = t;
    }
    s0 = fmaxf(s0, t0);
    s1 = fminf(s1, t1);
    return s0 <= s1;
}

// Ray parameter of the eye (perspective) or of the image plane (orthographic)
// in the units of Ray: depths are reported from there, like the oracle's t.
__device__ __forceinline__ float eye_param(const CamDev &c, int i, int j)
{
    if (!c.persp) return -c.dist;
    const float hi = (float)i - 0.5f * (float)(c.W - 1);
    const float hj = (float)j - 0.5f * (float)(c.H - 1);
    const float wx = fmaf(hi, c.wa.x, fmaf(hj, c.wb.x, c.wf.x));
    const float wy = fmaf(hi, c.wa.y, fmaf(hj, c.wb.y, c.wf.y));
    const float wz = fmaf(hi, c.wa.z, fmaf(hj, c.wb.z, c.wf.z));
    return -c.dist * sqrtf(wx * wx + wy * wy + wz * wz);
}

// The samples of a ray whose cell lies in the sub-box.  Along one axis a
// sample's cell is clamp(floor(g), 0, n - 2), and the computed position g(k)
// is monotone in k (fmaf of a value monotone in k), so the cell is at least lo
// where g >= lo (everywhere if lo = 0), below hi where g < hi (everywhere if hi
// = n - 1): the samples form one run, whose ends a bisection finds with the
// positions the march itself computes.
struct SubBox {
    float3 lo, hi;             // -inf / +inf at the grid's own faces
    __device__ __forceinline__ bool entered(const float3 &g, const float3 &d) const
    {
        return (d.x < 0.0f ? g.x < hi.x : g.x >= lo.x) && (d.y < 0.0f ? g.y < hi.y : g.y >= lo.y) &&
               (d.z < 0.0f ? g.z < hi.z : g.z >= lo.z);
    }
    __device__ __forceinline__ bool left(const float3 &g, const float3 &d) const
    {
        return (d.x < 0.0f ? g.x < lo.x : g.x >= hi.x) || (d.y < 0.0f ? g.y < lo.y : g.y >= hi.y) ||
               (d.z < 0.0f ? g.z < lo.z : g.z >= hi.z);
    }
    // [first, end) of the samples 0 .. r.n - 1
    __device__ __forceinline__ int2 run(const Ray &r, float step) const
    {
        int a = 0, b = r.n;                          // first sample that has entered
        while (a < b) {
            const int m = (a + b) >> 1;
            if (entered(sample_pos(r, m, step), r.d)) b = m; else a = m + 1;
        }
        const int first = a;
        b = r.n;                                     // first sample from there that has left
        while (a < b) {
            const int m = (a + b) >> 1;
            if (left(sample_pos(r, m, step), r.d)) b = m; else a = m + 1;
        }
        return make_int2(first, a);
    }
};

// The samples of the run are marched as a whole render marches its rays (the
// same pipeline and register budget), without a test per sample: eight boxes
// of a 1080p view of the 1024^3 cube 4.18 -> 2.62 ms (the whole render of that
// view takes 1.5; the rest is each launch's tail and 400 MB of partial images).
template <typename T, int LOG2B, int L, bool GROUPS>
__global__ void __launch_bounds__(kModeThreads, SubMinBlocks<T>::value) subbox_kernel(
    VolDev v, CamDev c, ParamDev p, int3 lo, int3 hi, SubBox box, int3 gdim, float3 off, float4 *partial, float *depth,
    uint32_t *count, unsigned *counter, Tiles t)
{
    if (GROUPS && left_to_lanes(t, p)) return;
    const int lane = threadIdx.x & 31;
    const float z = GROUPS || skips_transparent<T, IdentityMap>() ? transparent_below(p) : 0.0f;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= t.ntiles) break;
        const LanePixel px = lane_pixel<GROUPS>(t, tile, c.W, c.H);
        Ray ray;
        // rays and samples of the whole grid (gdim voxels; the camera is in its
        // coordinates); the volume holds its voxels from off on
        bool active = px.march && setup_ray(c, gdim.x, gdim.y, gdim.z, p.step, px.i, px.j, ray);
        int2 run = make_int2(0, 0);
        if (active) {
            // a ray that misses the sub-box widened by one voxel has no sample in it
            float s0 = -INFINITY, s1 = INFINITY;
            if (slab_range(ray.q.x, ray.d.x, (float)lo.x - 1.0f, (float)hi.x + 1.0f, s0, s1) &&
                slab_range(ray.q.y, ray.d.y, (float)lo.y - 1.0f, (float)hi.y + 1.0f, s0, s1) &&
                slab_range(ray.q.z, ray.d.z, (float)lo.z - 1.0f, (float)hi.z + 1.0f, s0, s1))
                run = box.run(ray, p.step);
            active = run.x < run.y;
        }
        Composite acc{0.0f, 0.0f, 0.0f, 1.0f};
        ray.n = run.y;
        if constexpr (GROUPS)
            march_group<T, LOG2B, L, kGroup, IdentityMap, PartOfGrid>(v, p, ray, active, acc, z, IdentityMap(),
                                                                      PartOfGrid{off}, run.x);
        else
            march_ray<T, LOG2B, L, IdentityMap, SubDepth<T>::value, PartOfGrid>(v, p, ray, active, acc, z, IdentityMap(),
                                                                                PartOfGrid{off}, run.x);
        if (!px.writes) continue;
        const long long at = (long long)px.j * c.W + px.i;
        partial[at] = make_float4(acc.r, acc.g, acc.b, acc.T);
        depth[at] = active ? fmaf((float)run.x + 0.5f, p.step, ray.s_in) - eye_param(c, px.i, px.j) : INFINITY;
        if (count) count[at] = (uint32_t)(run.y - run.x);
    }
}

cudaError_t launch_subbox(const VolDev &v, vr_dtype dt, const CamDev &c, const ParamDev &p, const Tiles &t, const int lo[3],
                          const int hi[3], const int gdim[3], const int off[3], float4 *partial, float *depth,
                          uint32_t *count, unsigned *counter, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const int3 l3 = make_int3(lo[0], lo[1], lo[2]), h3 = make_int3(hi[0], hi[1], hi[2]);
    const int3 g3 = make_int3(gdim[0], gdim[1], gdim[2]);
    const float3 o3 = make_float3((float)off[0], (float)off[1], (float)off[2]);
    SubBox box;
    float *blo = &box.lo.x, *bhi = &box.hi.x;
    for (int a = 0; a < 3; ++a) {
        blo[a] = lo[a] <= 0 ? -INFINITY : (float)lo[a];
        bhi[a] = hi[a] >= gdim[a] - 1 ? INFINITY : (float)hi[a];
    }
    ParamDev q = p;
    q.t_stop = -INFINITY;                       // no early termination inside a sub-box
    return visit_layout_tex(
        v, dt,
        [&](auto lay) {
            using Y = decltype(lay);
            auto fn = t.groups ? subbox_kernel<typename Y::type, Y::log2b, Y::order, true>
                             : subbox_kernel<typename Y::type, Y::log2b, Y::order, false>;
            fn<<<persistent_grid(fn, t.ntiles), kModeThreads, 0, s>>>(v, c, q, l3, h3, box, g3, o3, partial, depth, count,
                                                                      counter, t);
            if (t.by_table) {                     // both ways: one of the two finds nothing to do
                const Tiles lt = lane_tiles(t);
                fn = subbox_kernel<typename Y::type, Y::log2b, Y::order, false>;
                fn<<<persistent_grid(fn, lt.ntiles), kModeThreads, 0, s>>>(v, c, q, l3, h3, box, g3, o3, partial, depth,
                                                                           count, counter, lt);
            }
            return cudaGetLastError();
        },
        cudaErrorInvalidValue);
}

// Over-composite of k partial images per pixel, ordered by depth (front
// first); the pixel is (C + T bg.rgb, 1 - T + T bg.a).
struct PartialList {
    const float4 *img[kMaxPartials];
    const float *depth[kMaxPartials];
};

__global__ void __launch_bounds__(256) composite_kernel(PartialList pl, int k, long long npx, float4 bg,
                                                         float4 *out)
{
    for (long long px = (long long)blockIdx.x * blockDim.x + threadIdx.x; px < npx;
         px += (long long)gridDim.x * blockDim.x) {
        float d[kMaxPartials];
        unsigned char ord[kMaxPartials];
        for (int q = 0; q < k; ++q) {
            d[q] = pl.depth[q][px];
            ord[q] = (unsigned char)q;
        }
        for (int q = 1; q < k; ++q)               // insertion sort by depth (stable)
            for (int r = q; r > 0 && d[ord[r]] < d[ord[r - 1]]; --r) {
                const unsigned char t = ord[r];
                ord[r] = ord[r - 1];
                ord[r - 1] = t;
            }
        float Cr = 0.0f, Cg = 0.0f, Cb = 0.0f, T = 1.0f;
        for (int q = 0; q < k; ++q) {
            const float4 s = pl.img[ord[q]][px];
            Cr = fmaf(T, s.x, Cr);
            Cg = fmaf(T, s.y, Cg);
            Cb = fmaf(T, s.z, Cb);
            T *= s.w;
        }
        out[px] = make_float4(fmaf(T, bg.x, Cr), fmaf(T, bg.y, Cg), fmaf(T, bg.z, Cb), fmaf(T, bg.w, 1.0f - T));
    }
}

cudaError_t launch_composite(int k, const float *const *partials, const float *const *depths, long long npx,
                             const float bg[4], float *out, cudaStream_t s)
{
    PartialList pl;
    for (int q = 0; q < k; ++q) {
        pl.img[q] = reinterpret_cast<const float4 *>(partials[q]);
        pl.depth[q] = depths[q];
    }
    const long long blocks = std::min<long long>((npx + 255) / 256, (long long)sm_count() * 16);
    composite_kernel<<<(unsigned)std::max<long long>(blocks, 1), 256, 0, s>>>(
        pl, k, npx, make_float4(bg[0], bg[1], bg[2], bg[3]), reinterpret_cast<float4 *>(out));
    return cudaGetLastError();
}

}  // namespace vr
