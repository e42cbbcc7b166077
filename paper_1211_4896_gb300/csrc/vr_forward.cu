// vr_forward.cu -- forward ray-casting kernels (Sections 3.3-3.4 and 4.4 of
// Hassan et al. 2012): per pixel, clip the ray to the box, sample at a
// constant step with trilinear interpolation, map each sample through the
// RGBA transfer function and composite front to back, stopping early once the
// accumulated opacity reaches the threshold.
//
// GB300 mapping: persistent warps, one 8x4 pixel tile per warp at a time (its
// lanes in 2x2 quads), pulled from a global atomic queue (load balance across uneven ray lengths
// and early termination); voxel gathers go through the read-only L1 path from
// bricks (+apron) so all eight corners of a cell are at constant offsets in
// one brick, with the next sample's gathers in flight while the current one
// is composited; a warp vote retires the tile once every lane's ray has
// finished; float4 image stores.
#include "vr_device.cuh"

#include <cstdlib>
#include <map>
#include <mutex>

namespace vr {

// Two-warp CTAs: warps do not depend on one another, and small CTAs hand an
// SM's slots on warp pair by warp pair at the end of a view (views that follow
// each other in a batch's graph: 16 uneven cubes 2.04 -> 1.89 ms against
// eight-warp CTAs).  Eight-warp CTAs for the paired copies, whose dense views
// are not graph nodes of their own as a rule: neighbouring tiles then share an
// SM's L1 (16-bit views with an opaque table 1 to 4% faster).
constexpr int kFwdThreads = 64;
template <typename T> struct FwdThreads { static constexpr int value = kFwdThreads; };
template <typename S> struct FwdThreads<Pair<S>> { static constexpr int value = 256; };
constexpr int kPerSm = 256 / kFwdThreads;            // CTAs that make eight warps

// Resident warps the register budget is sized for, and samples whose gathers
// are in flight ahead of the one composited: 32 warps (64 registers) for the
// texture layers, with two samples ahead (the eight 1080p views of the 1024^3
// cube 198.6 -> 209.3 Gsamples/s, against 40 warps at 48 registers with one;
// the batched kernel keeps the latter, 1% faster there), and for the paired
// copies; 24 for the other brick layouts, with the march's own depth.
template <typename T> struct FwdMinBlocks { static constexpr int value = 3 * kPerSm; };
template <> struct FwdMinBlocks<TexLayers<float>> { static constexpr int value = 4 * kPerSm; };
template <typename S> struct FwdMinBlocks<Pair<S>> { static constexpr int value = 4; };
template <typename T> struct FwdDepth { static constexpr int value = Pipeline<T>::depth; };
template <> struct FwdDepth<TexLayers<float>> { static constexpr int value = 2; };

template <typename T, int LOG2B, int L>
__global__ void __launch_bounds__(FwdThreads<T>::value, FwdMinBlocks<T>::value) fwd_kernel(VolDev v, CamDev c, ParamDev p, float4 *out,
                                                           uint32_t *nsamples, unsigned *counter, Tiles t)
{
    const int lane = threadIdx.x & 31;
    const float z = skips_transparent<T, IdentityMap>() ? transparent_below(p) : 0.0f;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= t.ntiles) break;
        const LanePixel px = lane_pixel<false>(t, tile, c.W, c.H);
        Ray ray;
        const bool hit = px.march && setup_ray(c, v.nx, v.ny, v.nz, p.step, px.i, px.j, ray);
        Composite acc{0.0f, 0.0f, 0.0f, 1.0f};
        const int used = march_ray<T, LOG2B, L, IdentityMap, FwdDepth<T>::value>(v, p, ray, hit, acc, z);
        if (px.writes) write_pixel(p, acc, hit ? used : 0, out, nsamples, (long long)px.j * c.W + px.i);
    }
}

// Eight lanes to a ray (march_group, kGroup), for two kinds of views:
//
// Sparse views (rays three or more voxels apart at the volume centre) that cover
// few pixels or look along the layout's rows (sparse_in_groups has the limits).
// Neighbouring rays share no sectors there, and with a ray to each lane the lines it fetched were evicted before its next
// samples came to use them: 59 DRAM bytes a sample against 17 compulsory, the
// march waiting on memory 12 of 13 issue slots.  Eight consecutive samples of
// a ray in one warp instruction use a line at once, and an eighth of the rays
// are in flight.  1080p-like views of big cubes, rays 6 voxels apart: 2048 x
// 2048 x 1024 float in 64^3 bricks 3.23 -> 2.33 ms, 1024 x 1024 x 700 float along
// z 618 -> 391 us, along x 851 -> 414, tilted with an opaque table 492 -> 330;
// float16 on blocked copies 685 -> 300 us.  Sixteen lanes gain 5-10% more
// where rays are long and transparent and lose 15% where they end after 50
// samples; two rounds of gathers in flight are the same trade.
//
// Views whose volume covers few pixels: with a ray to each lane they leave the
// SMs a few warps each, which wait out every gather's latency along the whole
// ray.  Against a ray to a lane (five cubes from 60^3 to 400 x 300 x 350, three
// directions, float and float16, step 0.7; slowest to fastest), by covered
// pixels: 2500: 1.8 to 3.4 times as fast with the benchmark's ramp, 1.5 to 1.9
// with an opaque table; 10 000: 1.8 to 3.0 and 1.2 to 1.7; 16 000: 1.6 to 3.8 and
// 0.9 to 1.8; 24 000: 1.3 to 3.5 and 0.75 to 1.6; 38 000: 1.2 to 3.8 and 0.6 to
// 1.5: an opaque table's samples are all handed over and composited, which costs
// more than the latency once an SM has a few tiles.  So views of up to 112
// covered pixels an SM march in groups (sigma clipping and sub-boxes, whose
// samples cost more and whose limits lie higher, up to 160; the maximum, which
// composites nothing, up to 256), and up to 256 an SM those whose table begins
// with transparent entries (sparse views: sparse_in_groups).
// Only the device has read the table, so these are launched both ways
// (Tiles::by_table): 2 to 3 us.  Both marches in one kernel cost each of them 10%
// to a factor of 4.
template <typename T, int LOG2B, int L>
__global__ void __launch_bounds__(kFwdThreads, 3 * kPerSm) fwd_group_kernel(VolDev v, CamDev c, ParamDev p, float4 *out,
                                                                uint32_t *nsamples, unsigned *counter, Tiles t)
{
    if (left_to_lanes(t, p)) return;
    const int lane = threadIdx.x & 31;
    const float z = transparent_below(p);
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= t.ntiles) break;
        const LanePixel px = lane_pixel<true>(t, tile, c.W, c.H);
        Ray ray;
        const bool hit = px.march && setup_ray(c, v.nx, v.ny, v.nz, p.step, px.i, px.j, ray);
        Composite acc{0.0f, 0.0f, 0.0f, 1.0f};
        const int used = march_group<T, LOG2B, L, kGroup>(v, p, ray, hit, acc, z);
        if (px.writes) write_pixel(p, acc, hit ? used : 0, out, nsamples, (long long)px.j * c.W + px.i);
    }
}

// Hardware-filter alternative: tex3D with cudaFilterModeLinear (texel
// centres at +0.5 in unnormalised coordinates).  Same camera, lookup and
// compositing; only the interpolation differs (8-bit fractional weights).
__global__ void __launch_bounds__(kFwdThreads) fwd_tex_kernel(cudaTextureObject_t tex, int nx, int ny, int nz,
                                                               CamDev c, ParamDev p, float4 *out,
                                                               uint32_t *nsamples, unsigned *counter,
                                                               int tiles_x, unsigned ntiles)
{
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned tile = 0;
        if (lane == 0) tile = atomicAdd(counter, 1u);
        tile = __shfl_sync(kFull, tile, 0);
        if (tile >= ntiles) break;
        const int2 at = tile_pixel(lane, 3);
        const int i = (int)(tile % tiles_x) * 8 + at.x;
        const int j = (int)(tile / tiles_x) * 4 + at.y;
        const bool inside = i < c.W && j < c.H;
        Ray ray;
        const bool hit = inside && setup_ray(c, nx, ny, nz, p.step, i, j, ray);
        Composite acc{0.0f, 0.0f, 0.0f, 1.0f};
        int k = 0;
        bool active = hit;
        while (__any_sync(kFull, active)) {
            if (active) {
                const float3 pos = sample_pos(ray, k, p.step);
                const float val = tex3D<float>(tex, pos.x + 0.5f, pos.y + 0.5f, pos.z + 0.5f);
                TfPos tp;
                const float4 e = tf_lookup_l1(p, val, tp);
                const float aT = e.w * acc.T;
                acc.r = fmaf(aT, e.x, acc.r);
                acc.g = fmaf(aT, e.y, acc.g);
                acc.b = fmaf(aT, e.z, acc.b);
                acc.T = fmaf(-e.w, acc.T, acc.T);
                ++k;
                if (k >= ray.n || acc.T <= p.t_stop) active = false;
            }
        }
        if (inside) write_pixel(p, acc, hit ? k : 0, out, nsamples, (long long)j * c.W + i);
    }
}

// ---------------------------------------------------------------------------
// Launch helpers
// ---------------------------------------------------------------------------

int occupancy_blocks(const void *fn, int threads, size_t smem)
{
    static std::mutex mu;
    static std::map<std::pair<const void *, size_t>, int> cache;
    std::lock_guard<std::mutex> g(mu);
    auto key = std::make_pair(fn, smem);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, smem) != cudaSuccess || nb < 1) nb = 1;
    cache[key] = nb;
    return nb;
}

// Resident CTAs per SM for the persistent forward grid: the occupancy limit,
// at most `cap` (0: none), or eight warps for each VR_FWD_CTAS_PER_SM when set
// (a tuning knob: fewer resident warps thrash the L1 and L2 less).
static int fwd_ctas_per_sm(const void *fn, int threads, int cap)
{
    const int occ = occupancy_blocks(fn, threads, 0);
    static const int env = [] {
        const char *s = std::getenv("VR_FWD_CTAS_PER_SM");
        return s ? std::atoi(s) : 0;
    }();
    const int want = env > 0 ? env * (256 / threads) : cap;
    return (want > 0 && want < occ) ? want : occ;
}

// CTAs per SM for the float brick layouts with a ray to each lane (dense views
// that cannot have texture layers): 24 warps, where each resident ray keeps its
// own cache lines live and more of them thrash L1 and L2.  The other layouts:
// the occupancy limit.
template <typename T> struct FwdCtaCap { static constexpr int value = 0; };
template <> struct FwdCtaCap<float> { static constexpr int value = 3 * kPerSm; };

static const char *layout_name(const VolDev &v)
{
    const char *names[4] = {"", " paired", " blocked", " texture layers"};
    return names[v.paired & 3];
}

// Persistent grid of `tiles` tiles: per_sm CTAs on each SM, no more than
// there are tiles for.
static unsigned fwd_grid(int per_sm, int threads, unsigned tiles)
{
    const unsigned warps = (unsigned)threads / 32, grid = (unsigned)(per_sm * sm_count()), useful = (tiles + warps - 1) / warps;
    return grid < useful ? grid : (useful ? useful : 1u);
}

// A view's kernel and its grid.
struct FwdLaunch {
    void (*fn)(VolDev, CamDev, ParamDev, float4 *, uint32_t *, unsigned *, Tiles) = nullptr;
    unsigned grid = 0;
    int threads = kFwdThreads;
};

template <typename T, int LOG2B, int L>
static FwdLaunch plan_fwd_t(const VolDev &v, const CamDev &c, const Tiles &t)
{
    FwdLaunch f;
    f.fn = fwd_group_kernel<T, LOG2B, L>;
    if constexpr (is_blocked<T>::value) {      // only sparse views read these, and they march in groups
        if (!t.groups) return FwdLaunch();
    } else {
        if (!t.groups) f.fn = fwd_kernel<T, LOG2B, L>, f.threads = FwdThreads<T>::value;
    }
    const int per_sm = t.groups ? occupancy_blocks((const void *)f.fn, f.threads, 0)
                                : fwd_ctas_per_sm((const void *)f.fn, f.threads, FwdCtaCap<T>::value);
    f.grid = fwd_grid(per_sm, f.threads, t.ntiles);
    log_line("forward %dx%d: layout order %d%s, %u tiles of %s rays, %d lane(s) to a ray, grid %u x %d threads (%d per SM)",
             c.W, c.H, v.order, layout_name(v), t.nmarch, t.groups ? "2x2" : "8x4", t.groups ? kGroup : 1, f.grid,
             f.threads, per_sm);
    return f;
}

static FwdLaunch plan_fwd(const VolDev &v, vr_dtype dt, const CamDev &c, const Tiles &t)
{
    return visit_layout_all(
        v, dt,
        [&](auto lay) {
            using Y = decltype(lay);
            return plan_fwd_t<typename Y::type, Y::log2b, Y::order>(v, c, t);
        },
        FwdLaunch());
}

cudaError_t launch_forward(const VolDev &v, vr_dtype dt, const CamDev &c, const ParamDev &p, const Tiles &t, float4 *out,
                           uint32_t *nsamples, unsigned *counter, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
    auto launch = [&](const Tiles &q) {
        const FwdLaunch f = plan_fwd(v, dt, c, q);
        if (!f.fn) return cudaErrorInvalidValue;
        f.fn<<<f.grid, f.threads, 0, s>>>(v, c, p, out, nsamples, counter, q);
        return cudaGetLastError();
    };
    if (e == cudaSuccess) e = launch(t);
    if (e == cudaSuccess && t.by_table) e = launch(lane_tiles(t));    // one of the two finds nothing to do
    return e;
}

// The same view as a kernel node after `reset`, which clears its counter.
cudaError_t add_forward_node(cudaGraph_t graph, cudaGraphNode_t reset, const VolDev &v, vr_dtype dt, const CamDev &c,
                             const ParamDev &p, const Tiles &t, float4 *out, uint32_t *nsamples, unsigned *counter)
{
    const FwdLaunch f = plan_fwd(v, dt, c, t);
    if (!f.fn) return cudaErrorInvalidValue;
    void *args[] = {const_cast<VolDev *>(&v), const_cast<CamDev *>(&c), const_cast<ParamDev *>(&p), &out, &nsamples,
                    &counter, const_cast<Tiles *>(&t)};
    cudaKernelNodeParams kp = {};
    kp.func = (void *)f.fn;
    kp.gridDim = dim3(f.grid);
    kp.blockDim = dim3(f.threads);
    kp.kernelParams = args;
    cudaGraphNode_t node = nullptr;
    return cudaGraphAddKernelNode(&node, graph, &reset, 1, &kp);
}

cudaError_t launch_forward_texture(const vr_volume *vol, const CamDev &c, const ParamDev &p, float4 *out,
                                   uint32_t *nsamples, unsigned *counter, cudaStream_t s)
{
    const int tiles_x = (c.W + 7) / 8, tiles_y = (c.H + 3) / 4;
    const unsigned ntiles = (unsigned)tiles_x * (unsigned)tiles_y;
    const int per_sm = occupancy_blocks((const void *)fwd_tex_kernel, kFwdThreads, 0);
    const unsigned grid = fwd_grid(per_sm, kFwdThreads, ntiles);
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    fwd_tex_kernel<<<grid, kFwdThreads, 0, s>>>(vol->tex, (int)vol->dims[0], (int)vol->dims[1], (int)vol->dims[2],
                                                c, p, out, nsamples, counter, tiles_x, ntiles);
    return cudaGetLastError();
}

}  // namespace vr
