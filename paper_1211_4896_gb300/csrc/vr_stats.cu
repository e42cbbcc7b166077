// vr_stats.cu -- global statistics of the resident cube (Sections 4.1-4.3):
// count, mean, standard deviation, minimum and maximum; a histogram; the
// exact median.  Each is a streaming pass over the x-fastest bricks (every
// voxel counted once: an apron element is skipped unless it is the cube's
// last layer), so the passes run at HBM bandwidth.  NULL (NaN) voxels are
// left out.
//
// Mean and deviation follow the paper's mixed precision (Section 4.2): short
// runs of values are summed in FP32, the runs with compensated FP32 sums,
// the threads' totals in FP64, all about a shift (the first voxel) to keep
// the squares small.  (FP64 arithmetic is slow on this part, so it stays out
// of the per-voxel loop.)  The median is the value of
// rank (n + 1) / 2, found by a radix select on order-preserving 32-bit keys
// instead of the paper's Torben bisection, which needs a pass per halving of
// the value range: the same rank in three counting passes (11, 11 and 10
// bits), or for large cubes in one pass that keeps the few keys near the
// median, bracketed by a sample.
#include "vr_device.cuh"

#include <cmath>

namespace vr {

constexpr int kStatThreads = 256;

// Calls f(value) for every non-NaN voxel of the bricks handed to this CTA
// (bricks blockIdx.x, blockIdx.x + gridDim.x, ...), and after() on every
// thread at least once for each U values of a thread (the calls line up across
// the CTA, so it may hold a barrier).  A thread keeps one (x, y) of a brick's
// layers and steps along z, so an element costs its load, one bound test and
// f; with 16-byte chunks, whose elements each had their place in the 17-wide
// rows worked out, the passes were bound by those instructions at a third of
// the copy bandwidth (moments of a 1024^3 float cube 1.95 -> 0.97 ms: its
// bricks at 74% of the copy bandwidth; 385^3 bfloat16 288 -> 73 us).  An element counts when it is a voxel of the cube and
// not an apron copy: the main part takes cells 0 .. B - 1 of x and y, and the
// last brick of an axis, whose apron may hold the cube's last layer, adds its
// two faces.
constexpr int U = 16;                        // loads in flight per thread
constexpr int kMaxFace = 65 * 65;            // values between two calls of after(), at most

template <typename T, int LOG2B, typename F, typename G>
__device__ __forceinline__ void for_each_voxel(const VolDev &v, F &&f, G &&after)
{
    constexpr int B = 1 << LOG2B, B1 = B + 1;
    constexpr int ROWS = kStatThreads / B, PARTS = B / ROWS;
    const int lx = threadIdx.x & (B - 1), ly0 = threadIdx.x >> LOG2B;
    // brick indices fit 32 bits (the volume limits keep nbx*nby*nbz < 2^31): 32-bit
    // division instead of the much slower 64-bit one
    const unsigned nbx = (unsigned)v.nbx, nbxy = (unsigned)v.nbx * (unsigned)v.nby;
    const unsigned nbricks = nbxy * (unsigned)v.nbz;
    for (unsigned brick = blockIdx.x; brick < nbricks; brick += gridDim.x) {
        const unsigned bz_ = brick / nbxy, rem = brick - bz_ * nbxy, by_ = rem / nbx;
        const int bx = (int)(rem - by_ * nbx), by = (int)by_, bz = (int)bz_;
        const int ex = min(B1, v.nx - bx * B) - ((bx < v.nbx - 1) ? 1 : 0);
        const int ey = min(B1, v.ny - by * B) - ((by < v.nby - 1) ? 1 : 0);
        const int ez = min(B1, v.nz - bz * B) - ((bz < v.nbz - 1) ? 1 : 0);
        const T *b = static_cast<const T *>(v.data) + (long long)brick * v.stride;
        for (int part = 0; part < PARTS; ++part) {
            const int ly = ly0 + part * ROWS;
            const T *col = b + ly * B1 + lx;
            const int end = lx < ex && ly < ey ? ez : 0;         // this thread's voxels along z
            for (int z = 0; z < ez; z += U) {
                T raw[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (z + u < end) raw[u] = __ldg(col + (z + u) * (B1 * B1));
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float a = to_f(raw[u]);
                    if (z + u < end && a == a) f(a);
                }
                after();
            }
        }
        if (ex > B) {
            for (int e = threadIdx.x; e < ey * ez; e += kStatThreads) {
                const int z = e / ey, y = e - z * ey;
                const float a = to_f(b[(z * B1 + y) * B1 + B]);
                if (a == a) f(a);
            }
            after();
        }
        if (ey > B) {
            const int wx = min(ex, B);
            for (int e = threadIdx.x; e < wx * ez; e += kStatThreads) {
                const int z = e / wx, x = e - z * wx;
                const float a = to_f(b[(z * B1 + B) * B1 + x]);
                if (a == a) f(a);
            }
            after();
        }
    }
}

__device__ __forceinline__ double warp_sum(double x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// ---------------------------------------------------------------------------
// Moments
// ---------------------------------------------------------------------------

struct MomentPartial {
    double n, s1, s2;
    float mn, mx;
};

// Compensated FP32 accumulation (Kahan): the running error of the sum is
// carried along, so per-thread totals keep about FP32 precision relative to
// the sum however many runs they add.
struct Kahan {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x)
    {
        const float y = x - c, t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

template <typename T, int LOG2B>
__global__ void __launch_bounds__(kStatThreads) moments_kernel(VolDev v, MomentPartial *part)
{
    // shift: the first voxel (every thread reads the same element), 0 if NULL
    const float s0 = to_f(static_cast<const T *>(v.data)[0]);
    const float shift = s0 == s0 ? s0 : 0.0f;
    unsigned cnt = 0;
    unsigned long long total = 0;
    Kahan k1, k2;
    float r1 = 0.0f, r2 = 0.0f, mn = INFINITY, mx = -INFINITY;
    for_each_voxel<T, LOG2B>(
        v,
        [&](float a) {
            const float d = a - shift;
            r1 += d;
            r2 = fmaf(d, d, r2);
            mn = fminf(mn, a);
            mx = fmaxf(mx, a);
            ++cnt;
        },
        [&] {                            // runs of about 16 values in plain FP32, the runs compensated
            k1.add(r1);
            k2.add(r2);
            r1 = r2 = 0.0f;
            total += cnt;
            cnt = 0;
        });
    double n = warp_sum((double)total);
    double s1 = warp_sum((double)k1.s - (double)k1.c);
    double s2 = warp_sum((double)k2.s - (double)k2.c);
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(kFull, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    }
    __shared__ MomentPartial w[kStatThreads / 32];
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) w[warp] = MomentPartial{n, s1, s2, mn, mx};
    __syncthreads();
    if (threadIdx.x == 0) {
        MomentPartial t = w[0];
        for (int q = 1; q < kStatThreads / 32; ++q) {
            t.n += w[q].n;
            t.s1 += w[q].s1;
            t.s2 += w[q].s2;
            t.mn = fminf(t.mn, w[q].mn);
            t.mx = fmaxf(t.mx, w[q].mx);
        }
        part[blockIdx.x] = t;
    }
}

// One CTA: the parts in a fixed order (deterministic).
template <typename T>
__global__ void __launch_bounds__(kStatThreads) moments_final(VolDev v, const MomentPartial *part, int nparts,
                                                                double *out)
{
    const float s0 = to_f(static_cast<const T *>(v.data)[0]);
    const double shift = s0 == s0 ? (double)s0 : 0.0;
    double n = 0.0, s1 = 0.0, s2 = 0.0;
    float mn = INFINITY, mx = -INFINITY;
    for (int q = threadIdx.x; q < nparts; q += kStatThreads) {
        n += part[q].n;
        s1 += part[q].s1;
        s2 += part[q].s2;
        mn = fminf(mn, part[q].mn);
        mx = fmaxf(mx, part[q].mx);
    }
    n = warp_sum(n);
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(kFull, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    }
    __shared__ MomentPartial w[kStatThreads / 32];
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = MomentPartial{n, s1, s2, mn, mx};
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int q = 1; q < kStatThreads / 32; ++q) {
        n += w[q].n;
        s1 += w[q].s1;
        s2 += w[q].s2;
        mn = fminf(mn, w[q].mn);
        mx = fmaxf(mx, w[q].mx);
    }
    const double m1 = n > 0.0 ? s1 / n : 0.0;
    out[0] = n;
    out[1] = n > 0.0 ? shift + m1 : NAN;
    out[2] = n > 0.0 ? sqrt(fmax(s2 / n - m1 * m1, 0.0)) : NAN;
    out[3] = n > 0.0 ? (double)mn : NAN;
    out[4] = n > 0.0 ? (double)mx : NAN;
}

// ---------------------------------------------------------------------------
// Histogram: per-CTA shared counters, added to the global counts at the end.
// Bin b of n covers [lo + b (hi - lo)/n, lo + (b+1) (hi - lo)/n), the top
// value hi in the last bin; the bin is decided by the FP64 expression of
// bin64.  When `fast` (the host has bounded the FP32 estimate's error below
// 0.02 bin widths) the bin is estimated in FP32 and decided again only within
// `band` (4x that bound) of an edge: by the edges' floats, where the caller
// has worked them out (bin64 never falls as the value grows, so the least
// float of each bin decides it), otherwise in FP64, whose divide takes a
// warp some 500 clocks on this part.
// ---------------------------------------------------------------------------

__device__ __forceinline__ int bin64(float a, double lo, double range, int nbins)
{
    return (int)floor(((double)a - lo) / range * (double)nbins);
}

// Keys that order like the values (no NaN).
__device__ __forceinline__ unsigned order_key(float a)
{
    const unsigned u = __float_as_uint(a);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_value(unsigned k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// edge[b], 1 <= b < nbins: the least of the floats in [flo, fhi] whose bin64 is
// b or more (above fhi if there is none).  bin64 never falls as the value
// grows, so a search over the floats' keys is exact: from the float nearest to
// the edge in doubling steps, then by bisection.  Nearly every edge takes two
// decisions; where an edge lies at or near zero the floats are far closer
// together than the FP64 expression can tell apart (for lo = -0.1, hi = 0.2 and
// 30 bins it puts everything from -6.9e-18 on into bin 10), and it takes up to
// 64.
__global__ void bin_edges_kernel(double lo, double hi, float flo, float fhi, int nbins, float *edge)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < 1 || b >= nbins) return;
    const double range = hi - lo;
    const unsigned first = order_key(flo), last = order_key(fhi);
    auto reaches = [&](unsigned k) { return bin64(key_value(k), lo, range, nbins) >= b; };
    const float near = (float)(lo + range * (double)b / (double)nbins);
    // below: a key that does not reach b (or first - 1); at: one that does (or last + 1)
    unsigned k = order_key(fminf(fmaxf(near, flo), fhi)), below = first - 1, at = last + 1;
    if (reaches(k)) {
        at = k;
        for (unsigned d = 1; at > first; d = min(d, 1u << 30) * 2) {
            k = at - first > d ? at - d : first;
            if (!reaches(k)) {
                below = k;
                break;
            }
            at = k;
        }
    } else {
        below = k;
        for (unsigned d = 1; below < last; d = min(d, 1u << 30) * 2) {
            k = last - below > d ? below + d : last;
            if (reaches(k)) {
                at = k;
                break;
            }
            below = k;
        }
    }
    while (at - below > 1) {
        k = below + (at - below) / 2;
        if (reaches(k)) at = k; else below = k;
    }
    edge[b] = key_value(at);
}

// With `copies` = 32 each lane of a warp counts into its own copy of the
// shared histogram (row stride nbins + 1, so equal bins of different lanes
// sit in different banks): lanes never contend on one counter.
template <typename T, int LOG2B, bool EDGES>
__global__ void __launch_bounds__(kStatThreads) histogram_kernel(VolDev v, double lo, double hi, float flo_in,
                                                                   float fhi_in, int nbins, int fast, float band,
                                                                   int copies, const float *__restrict__ edge,
                                                                   unsigned long long *counts)
{
    extern __shared__ unsigned sh[];
    const int pitch = nbins + 1;
    for (int b = threadIdx.x; b < copies * pitch; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    unsigned *mine = sh + (copies > 1 ? (threadIdx.x & 31) * pitch : 0);
    const float flo = (float)lo, fscale = (float)((double)nbins / (hi - lo));
    const double range = hi - lo;          // the FP64 decision: (a - lo) / (hi - lo) * nbins, in this order
    for_each_voxel<T, LOG2B>(v, [&](float a) {
        // flo_in / fhi_in: the least float >= lo and the greatest float <= hi, so
        // the FP32 test equals the FP64 one for every float a
        if (!(a >= flo_in && a <= fhi_in)) return;
        int b;
        if (EDGES || fast) {
            const float u = (a - flo) * fscale;
            b = (int)floorf(u);
            const float fr = u - floorf(u);
            if (fr < band || fr > 1.0f - band) {
                if constexpr (EDGES) {         // one of the two bins at the nearest edge
                    const int e = fr < band ? b : b + 1;
                    if (e >= 1 && e < nbins) b = a < __ldg(edge + e) ? e - 1 : e;
                } else {
                    b = bin64(a, lo, range, nbins);
                }
            }
        } else {
            b = bin64(a, lo, range, nbins);
        }
        b = min(max(b, 0), nbins - 1);
        atomicAdd(&mine[b], 1u);
    }, [] {});
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        unsigned long long t = 0;
        for (int q = 0; q < copies; ++q) t += sh[q * pitch + b];
        if (t) atomicAdd(&counts[b], t);
    }
}

// ---------------------------------------------------------------------------
// Median: radix select on keys that order like the values.
// ---------------------------------------------------------------------------

// How the digits of the median's key are found: by passes over all voxels, or
// over the list of keys that the collecting pass kept.
enum SelectMode { kSelectVoxels = 0, kSelectList = 1 };

struct SelectState {
    unsigned prefix;           // key bits fixed so far (high bits)
    int mode;                  // SelectMode of this call
    unsigned long long n;      // values counted (non-NaN)
    unsigned long long k;      // rank still to find among the values matching the prefix (1-based)
    // the collecting pass
    unsigned digit[2];         // top digits of the sample's two ranks
    unsigned long long rank[2], before[2];      // the ranks within those digits, and the sample's keys before them
    unsigned key_lo, key_hi;   // the bracket
    unsigned long long count;  // keys in the bracket (those beyond the list's capacity are not in it)
    unsigned long long below;  // keys under the bracket
};

__device__ __forceinline__ int digit_bits(int pass) { return pass == 2 ? 10 : 11; }
__device__ __forceinline__ int digit_shift(int pass) { return pass == 0 ? 21 : (pass == 1 ? 10 : 0); }

// Whether the bits above a pass's digit are those already selected.
__device__ __forceinline__ bool key_matches(unsigned key, unsigned prefix, int pass)
{
    const int top = digit_shift(pass) + digit_bits(pass);
    return top == 32 || (key >> top) == (prefix >> top);
}

template <typename T, int LOG2B>
__global__ void __launch_bounds__(kStatThreads) digit_hist_kernel(VolDev v, int pass, const SelectState *st,
                                                                    unsigned long long *hist)
{
    if (st->mode != kSelectVoxels) return;
    __shared__ unsigned sh[2048];
    const int shift = digit_shift(pass), nb = 1 << digit_bits(pass);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    const unsigned prefix = pass == 0 ? 0u : st->prefix;
    for_each_voxel<T, LOG2B>(v, [&](float a) {
        const unsigned key = order_key(a);
        if (key_matches(key, prefix, pass)) atomicAdd(&sh[(key >> shift) & (unsigned)(nb - 1)], 1u);
    }, [] {});
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        if (sh[b]) atomicAdd(&hist[b], (unsigned long long)sh[b]);
}

// Called by a whole CTA of kSelectThreads: the bin of hist[0, nb) (nb <= 2
// kSelectThreads) that holds rank k (1-based; k at most the total), and the
// number of values in the bins before it.  Returns the total; *bin and
// *before are valid on every thread.
constexpr int kSelectThreads = 1024;

__device__ unsigned long long find_rank(const unsigned long long *hist, int nb, unsigned long long k, int *bin,
                                        unsigned long long *before)
{
    __shared__ unsigned long long sums[32], s_before;
    __shared__ int s_bin;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b0 = 2 * threadIdx.x;
    const unsigned long long h0 = b0 < nb ? hist[b0] : 0ull, h1 = b0 + 1 < nb ? hist[b0 + 1] : 0ull;
    unsigned long long incl = h0 + h1;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();                   // the shared words may still be read by the previous call
    if (lane == 31) sums[warp] = incl;
    if (threadIdx.x == 0) s_bin = nb - 1, s_before = 0ull;
    __syncthreads();
    unsigned long long base = 0, total = 0;
    for (int q = 0; q < kSelectThreads / 32; ++q) {
        if (q < warp) base += sums[q];
        total += sums[q];
    }
    const unsigned long long at = base + incl - h0 - h1;         // values before bin b0
    if (k > at && k <= at + h0) s_bin = b0, s_before = at;
    else if (k > at + h0 && k <= at + h0 + h1) s_bin = b0 + 1, s_before = at + h0;
    __syncthreads();
    *bin = s_bin;
    *before = s_before;
    return total;
}

// One CTA: picks the digit that holds rank k, narrows the prefix and the
// rank, clears the histogram for the next pass; after the last pass writes
// the median (NaN without values).
__global__ void __launch_bounds__(kSelectThreads) select_digit_kernel(int pass, int mode, SelectState *st,
                                                                       unsigned long long *hist, double *median)
{
    if (st->mode != mode) return;
    const int nb = 1 << digit_bits(pass);
    int d = 0;
    unsigned long long below = 0, k = st->k, n = st->n;
    if (pass == 0 && mode == kSelectVoxels) {            // the voxels' count: from the histogram itself
        n = find_rank(hist, nb, 1, &d, &below);
        k = (n + 1) / 2;
    }
    const unsigned prefix = pass == 0 ? 0u : st->prefix;
    find_rank(hist, nb, k, &d, &below);
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) hist[b] = 0ull;
    if (threadIdx.x != 0) return;
    st->n = n;
    st->k = k - below;
    st->prefix = prefix | ((unsigned)d << digit_shift(pass));
    if (pass == 2) *median = n ? (double)key_value(st->prefix) : (double)NAN;
}

// ---------------------------------------------------------------------------
// Median of a large cube in one pass over its voxels: a stratified sample of
// 2^20 voxels (one in each of as many equal runs of bricks, at a hashed place
// in the brick) brackets the median between the keys of its ranks m/2 -+ 2
// sqrt(m) -- four standard deviations of the sample's rank of the median --
// and the pass counts the keys below the bracket and keeps those inside,
// about 0.4% of them, in a list; the digits are then found in the list.  The
// counts say whether the median is in the list; if not (a sample that misled,
// many equal values), the three passes over the voxels follow, whose kernels
// return at once otherwise.  1024^3 floats: 4.67 -> 1.37 ms.
// ---------------------------------------------------------------------------
constexpr int kSampleLog2 = 20;
constexpr unsigned kNoKey = 0xffffffffu;                 // (the key of a NaN)

template <typename T, int LOG2B>
__global__ void __launch_bounds__(kStatThreads) sample_kernel(VolDev v, unsigned *keys, unsigned long long *hist)
{
    __shared__ unsigned sh[2048];
    for (int b = threadIdx.x; b < 2048; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    constexpr int B = 1 << LOG2B, B1 = B + 1;
    const unsigned long long nbricks = (unsigned long long)v.nbx * v.nby * v.nbz;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < (1u << kSampleLog2); q += gridDim.x * blockDim.x) {
        const unsigned brick = (unsigned)((q * nbricks) >> kSampleLog2);
        unsigned h = q * 0x9E3779B1u;                    // Knuth's multiplicative hash
        h ^= h >> 15;
        h *= 0x9E3779B1u;
        const int lx = (h >> 8) & (B - 1), ly = (h >> 16) & (B - 1), lz = (h >> 24) & (B - 1);
        const int bx = (int)(brick % (unsigned)v.nbx), by = (int)(brick / (unsigned)v.nbx % (unsigned)v.nby),
                  bz = (int)(brick / ((unsigned)v.nbx * (unsigned)v.nby));
        unsigned key = kNoKey;
        if (bx * B + lx < v.nx && by * B + ly < v.ny && bz * B + lz < v.nz) {
            const float a = to_f(static_cast<const T *>(v.data)[(long long)brick * v.stride + (lz * B1 + ly) * B1 + lx]);
            if (a == a) key = order_key(a);
        }
        keys[q] = key;
        if (key != kNoKey) atomicAdd(&sh[key >> 21], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 2048; b += blockDim.x)
        if (sh[b]) atomicAdd(&hist[b], (unsigned long long)sh[b]);
}

// Second digits of the sample's keys whose top digit is that of rank r: hist[r].
__global__ void __launch_bounds__(kStatThreads) sample_hist_kernel(const unsigned *__restrict__ keys,
                                                                    const SelectState *st, unsigned long long *hist)
{
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < (1u << kSampleLog2); q += gridDim.x * blockDim.x) {
        const unsigned key = keys[q], d = key >> 21;
        if (key == kNoKey) continue;
        if (d == st->digit[0]) atomicAdd(&hist[(key >> 10) & 2047u], 1ull);
        if (d == st->digit[1]) atomicAdd(&hist[2048 + ((key >> 10) & 2047u)], 1ull);
    }
}

// One CTA: the digits of the sample's two ranks; after the second, the bracket,
// and whether it holds at most `limit` of the sample's keys (kSelectList: the
// voxels are collected).
__global__ void __launch_bounds__(kSelectThreads) sample_select_kernel(int pass, SelectState *st,
                                                                        unsigned long long *hist,
                                                                        unsigned long long limit)
{
    int d[2];
    unsigned long long before[2], rank[2];
    if (pass == 0) {
        const unsigned long long m = find_rank(hist, 2048, 1, &d[0], &before[0]);
        const unsigned long long w = (unsigned long long)(2.0f * sqrtf((float)m)) + 1ull, mid = (m + 1) / 2;
        rank[0] = mid > w ? mid - w : (m ? 1ull : 0ull);
        rank[1] = mid + w < m ? mid + w : m;
    } else {
        rank[0] = st->rank[0], rank[1] = st->rank[1];
    }
    for (int r = 0; r < 2; ++r) find_rank(hist + (pass ? r * 2048 : 0), 2048, rank[r], &d[r], &before[r]);
    const unsigned long long held = pass ? st->before[1] + before[1] + hist[2048 + d[1]] - st->before[0] - before[0] : 0ull;
    __syncthreads();
    for (int b = threadIdx.x; b < 2 * 2048; b += blockDim.x) hist[b] = 0ull;
    if (threadIdx.x != 0) return;
    for (int r = 0; r < 2; ++r) {
        if (pass == 0) {
            st->digit[r] = (unsigned)d[r];
            st->rank[r] = rank[r] - before[r];
            st->before[r] = before[r];
        } else {
            const unsigned key = (st->digit[r] << 21) | ((unsigned)d[r] << 10);
            if (r == 0) st->key_lo = key;
            else st->key_hi = key | 1023u;
        }
    }
    if (pass) st->mode = held <= limit ? kSelectList : kSelectVoxels;
}

// The pass over the voxels: count and below-bracket count of the non-NaN
// values, and the keys inside the bracket appended to list[0, cap) through a
// staging buffer in shared memory (one global counter update per flush).
constexpr int kStageFlush = 2048, kStageCap = kStageFlush + kMaxFace + 256;

template <typename T, int LOG2B>
__global__ void __launch_bounds__(kStatThreads) collect_kernel(VolDev v, SelectState *st, unsigned *list, unsigned cap)
{
    static_assert(kStatThreads * U <= kMaxFace, "the staging buffer holds a round of values");
    if (st->mode != kSelectList) return;
    __shared__ unsigned stage[kStageCap], staged;
    __shared__ unsigned long long base;
    if (threadIdx.x == 0) staged = 0u;
    __syncthreads();
    const unsigned lo = st->key_lo, width = st->key_hi - lo;
    unsigned long long n = 0, below = 0;
    unsigned n32 = 0, b32 = 0;
    auto flush = [&] {                     // called by the whole CTA after a barrier
        const unsigned c = staged;
        if (threadIdx.x == 0) base = atomicAdd(&st->count, (unsigned long long)c);
        __syncthreads();
        for (unsigned q = threadIdx.x; q < c; q += kStatThreads)
            if (base + q < cap) list[base + q] = stage[q];
        __syncthreads();
        if (threadIdx.x == 0) staged = 0u;
        __syncthreads();
    };
    for_each_voxel<T, LOG2B>(
        v,
        [&](float a) {
            const unsigned key = order_key(a);
            ++n32;
            b32 += key < lo;
            if (key - lo <= width) stage[atomicAdd(&staged, 1u)] = key;
        },
        [&] {
            n += n32;
            below += b32;
            n32 = b32 = 0;
            if (__syncthreads_or(staged > kStageFlush)) flush();
        });
    __syncthreads();
    if (staged) flush();
    for (int o = 16; o > 0; o >>= 1) {
        n += __shfl_xor_sync(kFull, n, o);
        below += __shfl_xor_sync(kFull, below, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&st->n, n);
        atomicAdd(&st->below, below);
    }
}

// Whether the median is in the list, and its rank there.
__global__ void list_begin_kernel(SelectState *st, unsigned cap)
{
    const unsigned long long k = (st->n + 1) / 2;
    if (st->mode == kSelectList && st->count <= cap && k > st->below && k <= st->below + st->count) {
        st->mode = kSelectList;
        st->k = k - st->below;
    } else {
        st->mode = kSelectVoxels;
    }
}

__global__ void __launch_bounds__(kStatThreads) list_hist_kernel(const unsigned *__restrict__ list, int pass,
                                                                  const SelectState *st, unsigned long long *hist)
{
    if (st->mode != kSelectList) return;
    __shared__ unsigned sh[2048];
    const int shift = digit_shift(pass), nb = 1 << digit_bits(pass);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) sh[b] = 0u;
    __syncthreads();
    const unsigned prefix = pass == 0 ? 0u : st->prefix, n = (unsigned)st->count;      // at most the list's capacity
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const unsigned key = list[q];
        if (key_matches(key, prefix, pass)) atomicAdd(&sh[(key >> shift) & (unsigned)(nb - 1)], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
        if (sh[b]) atomicAdd(&hist[b], (unsigned long long)sh[b]);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------

// One wave of resident CTAs (a second, shorter one would leave most SMs idle).
static unsigned stat_grid(const void *fn, long long nbricks, size_t smem = 0)
{
    const long long g = (long long)sm_count() * occupancy_blocks(fn, kStatThreads, smem);
    return (unsigned)(nbricks < g ? (nbricks > 0 ? nbricks : 1) : g);
}

template <typename F>
static cudaError_t by_storage(const VolDev &v, vr_dtype dt, F &&f)
{
    // the x-fastest bricks: element type = storage type, order 0
    return visit_layout(
        v, dt,
        [&](auto lay) {
            using Y = decltype(lay);
            if constexpr (Y::order == 0 && !is_pair<typename Y::type>::value)
                return f(lay);
            else
                return cudaErrorInvalidValue;
        },
        cudaErrorInvalidValue);
}

constexpr size_t kMaxParts = 152 * 8 * 4;              // CTAs of a pass
constexpr size_t kHistBytes = 2 * 2048 * sizeof(unsigned long long);

// Statistics scratch: the moments' parts, the digit histograms, the select
// state, the histogram's edges.
constexpr size_t kEdgeOffset = (sizeof(MomentPartial) * kMaxParts + kHistBytes + sizeof(SelectState) + 255) / 256 * 256;

size_t stats_scratch_bytes() { return kEdgeOffset + 16384 * sizeof(float); }

cudaError_t launch_moments(const VolDev &v, vr_dtype dt, void *scratch, double *out, cudaStream_t s)
{
    MomentPartial *part = static_cast<MomentPartial *>(scratch);
    return by_storage(v, dt, [&](auto lay) {
        using Y = decltype(lay);
        auto fn = moments_kernel<typename Y::type, Y::log2b>;
        const unsigned grid = stat_grid((const void *)fn, (long long)v.nbx * v.nby * v.nbz);
        if (grid > kMaxParts) return cudaErrorInvalidValue;
        fn<<<grid, kStatThreads, 0, s>>>(v, part);
        moments_final<typename Y::type><<<1, kStatThreads, 0, s>>>(v, part, (int)grid, out);
        return cudaGetLastError();
    });
}

// Voxels from which the histogram works its edges' floats out first: the
// launch takes about as long as the FP64 decisions of 8 million noise values
// over 256 bins (16-bit values, which fall on edges more often, take more).
constexpr long long kEdgesMinVoxels = 1LL << 23;
constexpr int kEdgeThreads = 32;          // one warp a CTA: spread over the SMs' FP64 units

// The error of the FP32 estimate of a bin, in bins: rounding of lo and of a - lo
// (each within one ulp of max(|lo|, |hi|)) times the scale, plus the scale's
// rounding.
static double estimate_error(double lo, double hi, int nbins)
{
    const double m = std::fmax(std::fabs(lo), std::fabs(hi));
    const double ulp = m > 0.0 ? std::ldexp(1.0, std::ilogb(m) - 23) : 0.0;
    return 2.0 * ulp * (double)nbins / (hi - lo) + 4.0 * 6e-8 * (double)nbins;
}

constexpr double kFastError = 0.02;       // bins: the estimate is used up to this error

bool histogram_wants_edges(long long nvox, double lo, double hi, int nbins)
{
    return nvox >= kEdgesMinVoxels && estimate_error(lo, hi, nbins) <= kFastError;
}

// scratch: the statistics scratch, or NULL (near an edge the bin is then
// decided in FP64).
cudaError_t launch_histogram(const VolDev &v, vr_dtype dt, double lo, double hi, int nbins, void *scratch,
                             unsigned long long *counts, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * (size_t)nbins, s);
    if (e != cudaSuccess) return e;
    const int copies = (size_t)32 * (nbins + 1) * sizeof(unsigned) <= 96 * 1024 ? 32 : 1;
    const size_t smem = sizeof(unsigned) * (size_t)copies * (nbins + 1);
    const double err = estimate_error(lo, hi, nbins);
    const int fast = err <= kFastError ? 1 : 0;
    const float band = (float)std::fmax(4.0 * err, 1e-3);       // decide again this close to an edge
    float flo_in = (float)lo, fhi_in = (float)hi;
    if ((double)flo_in < lo) flo_in = std::nextafterf(flo_in, INFINITY);
    if ((double)fhi_in > hi) fhi_in = std::nextafterf(fhi_in, -INFINITY);
    float *edge = nullptr;
    if (scratch && histogram_wants_edges((long long)v.nx * v.ny * v.nz, lo, hi, nbins)) {
        edge = reinterpret_cast<float *>(static_cast<unsigned char *>(scratch) + kEdgeOffset);
        bin_edges_kernel<<<(unsigned)((nbins + kEdgeThreads - 1) / kEdgeThreads), kEdgeThreads, 0, s>>>(lo, hi, flo_in,
                                                                                               fhi_in, nbins, edge);
    }
    return by_storage(v, dt, [&](auto lay) {
        using Y = decltype(lay);
        auto fn = edge ? histogram_kernel<typename Y::type, Y::log2b, true>
                       : histogram_kernel<typename Y::type, Y::log2b, false>;
        if (smem > 48 * 1024) {
            cudaError_t a = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (a != cudaSuccess) return a;
        }
        const unsigned grid = stat_grid((const void *)fn, (long long)v.nbx * v.nby * v.nbz, smem);
        fn<<<grid, kStatThreads, smem, s>>>(v, lo, hi, flo_in, fhi_in, nbins, fast, band, copies, edge, counts);
        return cudaGetLastError();
    });
}

// Voxels from which the collecting pass is used: below, the three short passes
// take less than its sample and list (2^25 voxels of 4 bytes: 20 us a pass).
constexpr long long kCollectMinVoxels = 1LL << 25;

// Bytes of the collecting pass's sample and list for a volume of n voxels (0:
// too small for it): the list takes n / 128 keys, twice what it should hold.
size_t median_list_bytes(long long n)
{
    return n < kCollectMinVoxels ? 0 : (size_t)((1LL << kSampleLog2) + n / 128) * sizeof(unsigned);
}

// list: median_list_bytes of scratch, or NULL (three passes over the voxels).
cudaError_t launch_median(const VolDev &v, vr_dtype dt, void *scratch, void *list, double *median, cudaStream_t s)
{
    unsigned char *base = static_cast<unsigned char *>(scratch) + sizeof(MomentPartial) * kMaxParts;
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(base);
    SelectState *st = reinterpret_cast<SelectState *>(base + kHistBytes);
    cudaError_t e = cudaMemsetAsync(base, 0, kHistBytes + sizeof(SelectState), s);
    if (e != cudaSuccess) return e;
    const long long nbricks = (long long)v.nbx * v.nby * v.nbz;
    return by_storage(v, dt, [&](auto lay) {
        using Y = decltype(lay);
        using T = typename Y::type;
        if (list) {
            unsigned *sample = static_cast<unsigned *>(list), *keys = sample + (1u << kSampleLog2);
            const unsigned cap = (unsigned)((long long)v.nx * v.ny * v.nz / 128);
            const unsigned grid = (unsigned)sm_count() * 4;
            // sample places inside the cube that stand for cap voxels
            const double cells = (double)nbricks * (double)(1LL << 3 * v.log2b);
            const auto limit = (unsigned long long)(std::fmin(1.0, (double)v.nx * v.ny * v.nz / cells) * (1 << kSampleLog2) / 128);
            sample_kernel<T, Y::log2b><<<grid, kStatThreads, 0, s>>>(v, sample, hist);
            sample_select_kernel<<<1, kSelectThreads, 0, s>>>(0, st, hist, 0);
            sample_hist_kernel<<<grid, kStatThreads, 0, s>>>(sample, st, hist);
            sample_select_kernel<<<1, kSelectThreads, 0, s>>>(1, st, hist, limit);
            auto fn = collect_kernel<T, Y::log2b>;
            fn<<<stat_grid((const void *)fn, nbricks), kStatThreads, 0, s>>>(v, st, keys, cap);
            list_begin_kernel<<<1, 1, 0, s>>>(st, cap);
            for (int pass = 0; pass < 3; ++pass) {
                list_hist_kernel<<<grid, kStatThreads, 0, s>>>(keys, pass, st, hist);
                select_digit_kernel<<<1, kSelectThreads, 0, s>>>(pass, kSelectList, st, hist, median);
            }
        }
        auto fn = digit_hist_kernel<T, Y::log2b>;
        const unsigned grid = stat_grid((const void *)fn, nbricks);
        for (int pass = 0; pass < 3; ++pass) {
            fn<<<grid, kStatThreads, 0, s>>>(v, pass, st, hist);
            select_digit_kernel<<<1, kSelectThreads, 0, s>>>(pass, kSelectVoxels, st, hist, median);
        }
        return cudaGetLastError();
    });
}

}  // namespace vr
