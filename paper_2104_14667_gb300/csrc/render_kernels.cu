// render_kernels.cu -- the display step: composite counts to overlap classes
// and colours (Fig. 1 caption: a blue saturation map where high overlap is
// high saturation, and the frequency of overlap classes), or depth sums to a
// mean depth.  Outputs are dense row-major, walked in units of four pixels
// (render_units.cuh).
#include <algorithm>

#include "overlap.cuh"
#include "render_units.cuh"

namespace cpt {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kHistCtasPerSm = 4;   // resident CTAs of the histogram render (64 registers, 41 KB of shared memory)
constexpr int kCtasPerSm = 16;      // grid cap of the others

// Bound by HBM (and L2) traffic: the plane once, every output once.  With the
// histogram every lane of a warp takes part in the folds of its counters
// (class_histogram.cuh; 16 pixels per lane and item), and the grid is one wave
// of resident CTAs, so that the hand-over of the totals per block stays short.
// The totals meet in a scratch that is zero between renders: cleared outputs
// would need an operation of their own before this one, between kernels that
// otherwise follow one another closely (509 x 516, two members out and two in:
// 35.3 us a pass with it, 29.5 without).  Without a scratch the totals go to
// the output, cleared by such an operation.
static_assert(kThreads == 256, "a thread hands over one class");
template <typename CountT, int kRows, bool kHist, int kUnits>
__global__ void __launch_bounds__(kThreads, kHist ? kHistCtasPerSm : 1)
render_counts_kernel(Plane p, ClassDivisor div, CountT *counts_out, uint8_t *bucket_out,
                     uint32_t *rgba_out, int vec, Lut lut, unsigned long long *hist_out, HistScratch *scratch) {
    __shared__ uint32_t table[256];
    __shared__ __align__(16) uint8_t s_hist[kHist ? kWarps * kHistWarpBytes : 16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *cnt = s_hist + (kHist ? warp * kHistWarpBytes : 0);
    uint8_t *row = kHist ? cnt + (lane / kHistLanesPerRow) * 256 : nullptr;
    const uint32_t key = (uint32_t)(lane / kHistLanesPerRow) << 2;
    uint32_t *tot = reinterpret_cast<uint32_t *>(cnt + kHistCounterBytes);
    for (int i = threadIdx.x; i < 256; i += blockDim.x) table[i] = lut.rgba[i];
    if (kHist)
        for (int i = threadIdx.x; i < kWarps * kHistWarpBytes / 16; i += blockDim.x)
            reinterpret_cast<uint4 *>(s_hist)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    await_previous();
    const CountT *plane = static_cast<const CountT *>(p.data);
    const int64_t total = (int64_t)p.width * p.height;
    constexpr int kItemPixels = 32 * kUnits * 4;
    int since_fold = 0;
    for (int64_t base = ((int64_t)blockIdx.x * kWarps + warp) * kItemPixels; base < total;
         base += (int64_t)gridDim.x * kWarps * kItemPixels) {
        if (kHist) {
            if (since_fold == kHistFoldItems) {
                hist_fold(cnt, tot, lane);
                since_fold = 0;
            }
            ++since_fold;
        }
        const int left = (int)min(total - base, (int64_t)kItemPixels);
        Unit<CountT> c[kUnits];
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
            const int at = 4 * (32 * k + lane);
            if (at < left) load_unit<CountT, kRows>(plane, p.pitch, p.width, base + at, left - at, c[k]);
        }
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
            const int at = 4 * (32 * k + lane);
            if (at >= left) break;
            uint32_t b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = overlap_class(c[k].get(j), div);
            store_unit(c[k], b, base + at, left - at, vec, counts_out, bucket_out, rgba_out, table, row, key);
        }
    }
    if (kHist) {
        hist_fold(cnt, tot, lane);
        __syncthreads();
        hist_emit_block(s_hist, kWarps, scratch ? scratch->bins : hist_out);
        if (!scratch) return;
        // the last CTA to get here hands the bins over and leaves them zero
        __shared__ int last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&scratch->arrived, 1u) == gridDim.x - 1;
        __syncthreads();
        if (last) {
            __threadfence();
            hist_out[threadIdx.x] = atomicExch(scratch->bins + threadIdx.x, 0ull);
            if (threadIdx.x == 0) scratch->arrived = 0u;
        }
    }
}

template <int kRows, int kUnits>
__global__ void __launch_bounds__(kThreads)
render_mean_kernel(Plane p, uint64_t n_members, float *mean_out, int vec) {
    const float *plane = static_cast<const float *>(p.data);
    const int64_t total = (int64_t)p.width * p.height;
    const float n = (float)n_members;
    constexpr int kItemPixels = 32 * kUnits * 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    await_previous();
    for (int64_t base = ((int64_t)blockIdx.x * kWarps + warp) * kItemPixels; base < total;
         base += (int64_t)gridDim.x * kWarps * kItemPixels) {
        const int left = (int)min(total - base, (int64_t)kItemPixels);
        Unit<float> c[kUnits];
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
            const int at = 4 * (32 * k + lane);
            if (at < left) load_unit<float, kRows>(plane, p.pitch, p.width, base + at, left - at, c[k]);
        }
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
            const int at = 4 * (32 * k + lane);
            if (at >= left) break;
#pragma unroll
            for (int j = 0; j < 4; ++j) c[k].v[j] = n_members == 0 ? 0.0f : c[k].v[j] / n;
            float *out = mean_out + base + at;
            if (vec && left - at >= 4)
                c[k].store(out);
            else
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < left - at) out[j] = c[k].v[j];
        }
    }
}

// A lane takes kUnits units at a time where that leaves two CTAs for every SM,
// else one: 66 x 550 in items of 512 pixels is nine CTAs, and a clear, fold
// and render took 26.8 us instead of 24.2.
bool small_raster(int64_t total, const DeviceCaps &caps) {
    return total < 2ll * caps.num_sms * kWarps * kItemPixels;
}

unsigned grid_for(int64_t total, int units, int ctas_per_sm, const DeviceCaps &caps) {
    const int64_t per_cta = (int64_t)kWarps * 32 * 4 * units;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + per_cta - 1) / per_cta, (int64_t)caps.num_sms * ctas_per_sm));
}

template <typename CountT, bool kHist, int kUnits>
void launch_counts(const Plane &p, const ClassDivisor &div, CountT *counts_out, uint8_t *bucket_out, uint32_t *rgba_out,
                   int vec, const Lut &lut, unsigned long long *hist_out, HistScratch *scratch, const DeviceCaps &caps,
                   cudaStream_t s) {
    const unsigned grid = grid_for((int64_t)p.width * p.height, kUnits, kHist ? kHistCtasPerSm : kCtasPerSm, caps);
    switch (plane_rows(p.pitch, p.width)) {
        case kRowsDense:
            launch_overlapped(render_counts_kernel<CountT, kRowsDense, kHist, kUnits>, grid, kThreads, 0, s, p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch);
            break;
        case kRowsOfFours:
            launch_overlapped(render_counts_kernel<CountT, kRowsOfFours, kHist, kUnits>, grid, kThreads, 0, s, p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch);
            break;
        default:
            launch_overlapped(render_counts_kernel<CountT, kRowsRagged, kHist, kUnits>, grid, kThreads, 0, s, p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch);
    }
}

// The classes or the 16-bit counts alone are few bytes a pixel: from this size
// on a lane takes eight units at a time (8192^2 classes 44.6 us with four, 39.4
// with eight, counts 49.3 and 43.9; 4096^2 13.0 and 12.2).
constexpr int64_t kManyPixels = 16ll << 20;

template <typename CountT, bool kHist>
cudaError_t render_counts_t(const Plane &p, uint64_t n_members, void *counts, uint8_t *bucket_out,
                            uint32_t *rgba_out, const Lut &lut, unsigned long long *hist_out, HistScratch *scratch,
                            const DeviceCaps &caps, cudaStream_t s) {
    const ClassDivisor div = class_divisor(n_members);
    CountT *counts_out = static_cast<CountT *>(counts);
    const int vec = reinterpret_cast<uintptr_t>(counts_out) % (4 * sizeof(CountT)) == 0 &&
                    reinterpret_cast<uintptr_t>(bucket_out) % 4 == 0 && reinterpret_cast<uintptr_t>(rgba_out) % 16 == 0;
    if (!kHist && sizeof(CountT) == 2 && !rgba_out && (!counts_out || !bucket_out) &&
        (int64_t)p.width * p.height >= kManyPixels)
        launch_counts<CountT, kHist, kHist ? kUnits : 2 * kUnits>(p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch, caps, s);
    else if (small_raster((int64_t)p.width * p.height, caps))
        launch_counts<CountT, kHist, 1>(p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch, caps, s);
    else
        launch_counts<CountT, kHist, kUnits>(p, div, counts_out, bucket_out, rgba_out, vec, lut, hist_out, scratch, caps, s);
    return cudaGetLastError();
}

template <int kUnits>
void launch_mean(const Plane &p, uint64_t n_members, float *mean_out, int vec, const DeviceCaps &caps, cudaStream_t s) {
    const unsigned grid = grid_for((int64_t)p.width * p.height, kUnits, kCtasPerSm, caps);
    switch (plane_rows(p.pitch, p.width)) {
        case kRowsDense: launch_overlapped(render_mean_kernel<kRowsDense, kUnits>, grid, kThreads, 0, s, p, n_members, mean_out, vec); break;
        case kRowsOfFours: launch_overlapped(render_mean_kernel<kRowsOfFours, kUnits>, grid, kThreads, 0, s, p, n_members, mean_out, vec); break;
        default: launch_overlapped(render_mean_kernel<kRowsRagged, kUnits>, grid, kThreads, 0, s, p, n_members, mean_out, vec);
    }
}

}  // namespace

cudaError_t launch_render_counts(const Plane &p, uint64_t n_members, void *counts_out,
                                 uint8_t *bucket_out, uint32_t *rgba_out, const Lut &lut,
                                 const DeviceCaps &caps, cudaStream_t s, uint64_t *hist_out, HistScratch *scratch) {
    const bool u16 = p.count_bits == 16;
    if (hist_out) {
        unsigned long long *h = reinterpret_cast<unsigned long long *>(hist_out);
        if (!scratch) {
            const cudaError_t e = cudaMemsetAsync(h, 0, 256 * sizeof(*h), s);
            if (e != cudaSuccess) return e;
        }
        return u16 ? render_counts_t<uint16_t, true>(p, n_members, counts_out, bucket_out, rgba_out, lut, h, scratch, caps, s)
                   : render_counts_t<uint32_t, true>(p, n_members, counts_out, bucket_out, rgba_out, lut, h, scratch, caps, s);
    }
    if (!counts_out && !bucket_out && !rgba_out) return cudaSuccess;
    return u16 ? render_counts_t<uint16_t, false>(p, n_members, counts_out, bucket_out, rgba_out, lut, nullptr, nullptr, caps, s)
               : render_counts_t<uint32_t, false>(p, n_members, counts_out, bucket_out, rgba_out, lut, nullptr, nullptr, caps, s);
}

cudaError_t launch_render_mean(const Plane &p, uint64_t n_members, float *mean_out,
                               const DeviceCaps &caps, cudaStream_t s) {
    if (!mean_out) return cudaSuccess;
    const int vec = reinterpret_cast<uintptr_t>(mean_out) % 16 == 0;
    if (small_raster((int64_t)p.width * p.height, caps))
        launch_mean<1>(p, n_members, mean_out, vec, caps, s);
    else
        launch_mean<kUnits>(p, n_members, mean_out, vec, caps, s);
    return cudaGetLastError();
}

}  // namespace cpt
