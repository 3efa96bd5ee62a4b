// oneshot.cu -- composite_oneshot_static: a one-shot composite of
// device-resident rasters that allocates nothing.
//
// Some callers cannot call cudaMalloc: an interactive viewer's per-frame
// render callback must not risk the implicit device synchronisation an
// allocation can bring, and a host application that owns all device memory
// through its own pool may forbid libraries from allocating at all.  This
// entry point is one kernel that folds the members and classifies, colours
// and stores the counts it holds: no composite plane, no scratch, nothing
// shared between calls.
#include <algorithm>

#include "composite.h"
#include "mask_load.cuh"
#include "overlap_class.cuh"

namespace {

constexpr int64_t kMaxPixels = CPT_ONESHOT_MAX_PIXELS;
constexpr int kThreads = 256;
constexpr int kPackedLimit = 255;   // members a packed byte counter can hold

// A CTA composites kThreads / kSlices 16-pixel groups: each slice of its
// threads folds a share of up to 255 members at a time into packed counters,
// which are added up in shared memory four pixels to a thread; the sums are
// classified, coloured and stored from registers.  For small rasters the
// launch and one or two memory latencies are all there is: 512 x 512 x 8 took
// 16.4 us as two clears, a fold and a render of a scratch plane.
template <int kSlices>
__global__ void __launch_bounds__(kThreads)
oneshot_kernel(cpt::RasterBatch b, int width, int height, int groups_per_row, int64_t groups, cpt::ClassDivisor div,
               uint32_t *counts_out, uint8_t *bucket_out, uint32_t *rgba_out, int vec, cpt::Lut lut) {
    constexpr int kGroups = kThreads / kSlices;
    constexpr int kWords = (4 * kGroups + kThreads - 1) / kThreads;   // four-pixel words per thread
    __shared__ uint4 part[kSlices][kGroups];
    __shared__ uint32_t table[256];
    for (int i = threadIdx.x; i < 256; i += kThreads) table[i] = lut.rgba[i];
    const int lane_group = threadIdx.x % kGroups, slice = threadIdx.x / kGroups;
    const int64_t g = (int64_t)blockIdx.x * kGroups + lane_group;
    const int y = (int)(g / groups_per_row);
    const int x0 = (int)(g - (int64_t)y * groups_per_row) * 16;
    const int valid = min(16, width - x0);
    const uint8_t *base = static_cast<const uint8_t *>(b.base);
    const uint8_t *q = base + (int64_t)y * b.row_pitch + x0;
    uint32_t c[kWords][4];
#pragma unroll
    for (int i = 0; i < kWords; ++i) c[i][0] = c[i][1] = c[i][2] = c[i][3] = 0u;
    for (int s0 = 0; s0 < b.n; s0 += kPackedLimit) {
        const int s1 = min(b.n, s0 + kPackedLimit);
        uint32_t k[4] = {0u, 0u, 0u, 0u};
        if (g < groups) {
            const int share = (s1 - s0 + kSlices - 1) / kSlices;
            const int m0 = min(s1, s0 + slice * share), m1 = min(s1, m0 + share);
            int f0, f1;
            cpt::safe_members(q, b.member_stride, base, cpt::batch_end(b, width, height), 16, 16, m0, m1, f0, f1);
            cpt::fold_masks<true>(q, b.member_stride, f0, f1, k);
            for (int m = f1; m < m1; ++m) cpt::add_group(k, cpt::load_group_bytes(q + (int64_t)m * b.member_stride, valid));
        }
        part[slice][lane_group] = make_uint4(k[0], k[1], k[2], k[3]);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kWords; ++i) {
            const int w = threadIdx.x + i * kThreads;
            if (w >= 4 * kGroups) break;
            uint32_t sum = 0;
#pragma unroll
            for (int s = 0; s < kSlices; ++s) sum += reinterpret_cast<const uint32_t *>(part[s])[w];
#pragma unroll
            for (int j = 0; j < 4; ++j) c[i][j] += (sum >> (8 * j)) & 0xFFu;
        }
        __syncthreads();
    }
    if (b.n <= 0) __syncthreads();   // the colour table
#pragma unroll
    for (int i = 0; i < kWords; ++i) {
        const int w = threadIdx.x + i * kThreads;
        const int64_t at = (int64_t)blockIdx.x * kGroups + w / 4;
        if (w >= 4 * kGroups || at >= groups) break;
        const int py = (int)(at / groups_per_row);
        const int px = (int)(at - (int64_t)py * groups_per_row) * 16 + (w % 4) * 4;
        if (px >= width) continue;
        const int64_t o = (int64_t)py * width + px;
        uint32_t cls[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cls[j] = cpt::overlap_class(c[i][j], div);
        if (vec) {
            if (counts_out) *reinterpret_cast<uint4 *>(counts_out + o) = make_uint4(c[i][0], c[i][1], c[i][2], c[i][3]);
            if (bucket_out)
                *reinterpret_cast<uint32_t *>(bucket_out + o) = cls[0] | (cls[1] << 8) | (cls[2] << 16) | (cls[3] << 24);
            if (rgba_out)
                *reinterpret_cast<uint4 *>(rgba_out + o) = make_uint4(table[cls[0]], table[cls[1]], table[cls[2]], table[cls[3]]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (px + j >= width) break;
                if (counts_out) counts_out[o + j] = c[i][j];
                if (bucket_out) bucket_out[o + j] = (uint8_t)cls[j];
                if (rgba_out) rgba_out[o + j] = table[cls[j]];
            }
        }
    }
}

int reject(int code, const char *message) {
    cpt::set_thread_error(message);
    return code;
}

// True when p is device (or managed) memory the current device can address
// as its own: the kernel reads and writes these pointers directly, so host
// memory or another GPU's memory must be turned away before any launch.
bool on_current_device(const void *p, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

template <int kSlices>
void launch(const cpt::RasterBatch &b, int width, int height, const cpt::ClassDivisor &div, uint32_t *counts, uint8_t *bucket,
            uint32_t *rgba, int vec, const cpt::Lut &lut, cudaStream_t s) {
    const int gpr = (width + 15) / 16;
    const int64_t groups = (int64_t)gpr * height;
    constexpr int64_t kGroups = kThreads / kSlices;
    oneshot_kernel<kSlices><<<(unsigned)((groups + kGroups - 1) / kGroups), kThreads, 0, s>>>(
        b, width, height, gpr, groups, div, counts, bucket, rgba, vec, lut);
}

}  // namespace

extern "C" int composite_oneshot_static(const void *members, int32_t n_members,
                                        int64_t member_stride_bytes, int32_t row_pitch_bytes,
                                        int32_t width, int32_t height, uint32_t *counts_out,
                                        uint8_t *bucket_out, uint8_t *rgba_out,
                                        const uint8_t *lut_rgba, void *cuda_stream) try {
    if (width <= 0 || height <= 0) return reject(CPT_EINVAL, "raster is empty");
    if (n_members < 0) return reject(CPT_EINVAL, "n_members < 0");
    const int64_t pitch_px = ((int64_t)width + 15) / 16 * 16;
    if (pitch_px * height > kMaxPixels)
        return reject(CPT_EINVAL, "raster too large: roundup(width, 16) * height must be at most "
                                  "CPT_ONESHOT_MAX_PIXELS (the size of the former static scratch)");
    if (n_members > 0) {
        if (!members) return reject(CPT_EINVAL, "members is NULL");
        if (row_pitch_bytes < width || member_stride_bytes < (int64_t)row_pitch_bytes * height)
            return reject(CPT_EINVAL, "row pitch or member stride too small");
        if ((reinterpret_cast<uintptr_t>(members) % 16) || (row_pitch_bytes % 16) || (member_stride_bytes % 16))
            return reject(CPT_EINVAL, "members, row pitch and member stride must be 16-byte aligned");
    }
    if ((reinterpret_cast<uintptr_t>(counts_out) % 4) || (reinterpret_cast<uintptr_t>(rgba_out) % 4))
        return reject(CPT_EINVAL, "counts_out and rgba_out must be 4-byte aligned");

    int dev = 0, num_sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return reject(CPT_ECUDA, cudaGetErrorString(e));
    if (n_members > 0 && !on_current_device(members, dev))
        return reject(CPT_EINVAL, "members must be device memory of the current device");
    const void *outs[3] = {counts_out, bucket_out, rgba_out};
    for (const void *o : outs)
        if (o && !on_current_device(o, dev))
            return reject(CPT_EINVAL, "outputs must be device memory of the current device");
    if (!counts_out && !bucket_out && !rgba_out) return CPT_OK;
    cpt::Lut lut;
    for (int b = 0; b < 256; ++b) {
        const uint8_t *t = lut_rgba ? lut_rgba + 4 * b : nullptr;
        const uint32_t r = t ? t[0] : 255u - b, g = t ? t[1] : 255u - b, bl = t ? t[2] : 255u, al = t ? t[3] : 255u;
        lut.rgba[b] = r | (g << 8) | (bl << 16) | (al << 24);
    }
    const cpt::RasterBatch b{members, member_stride_bytes, row_pitch_bytes, n_members};
    const cpt::ClassDivisor div = cpt::class_divisor((uint64_t)n_members);
    uint32_t *rgba = reinterpret_cast<uint32_t *>(rgba_out);
    // four pixels of a row are stored at once where every row of every output allows it
    const int vec = width % 4 == 0 && reinterpret_cast<uintptr_t>(counts_out) % 16 == 0 &&
                    reinterpret_cast<uintptr_t>(bucket_out) % 4 == 0 && reinterpret_cast<uintptr_t>(rgba_out) % 16 == 0;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // slices of at least eight members; more than four only while four leave
    // the chip less than a wave of threads, 32 while eight leave it less than an
    // eighth of one.  Measured, us a call (slices): 512^2 x 1 2.9 (2) 3.6 (1),
    // 2048^2 x 1 10.3 (1) 11.4 (2); 512^2 x 8 3.5 (2, 4) 4.5 (1); 2048^2 x 16
    // 19.6 (2) 24.0 (4); 512^2 x 32 3.8 (4) 4.6 (2); 2048^2 x 64 53 (2) 55 (4);
    // 64^2 x 64 3.1 (8) 3.8 (4); 256^2 x 64 3.3 (8) 4.0 (4); 512^2 x 64 4.6 (4)
    // 5.3 (8); 512^2 x 255 10.5 (8) 10.7 (4); 1024^2 x 255 51 (8) 54 (4); 64^2 x
    // 255 3.9 (32) 5.4 (8); 256^2 x 255 5.2 (16) 5.8 (8, 32); 100 x 80 x 128 3.0
    // (32) 4.1 (8); 400 x 192 x 128 4.2 (8) 5.0 (32)
    const int64_t groups = pitch_px / 16 * height, wave = 2048ll * num_sms;
    const int members_at_once = std::min(n_members, kPackedLimit);
    if (members_at_once >= 128 && groups * 64 < wave)
        launch<32>(b, width, height, div, counts_out, bucket_out, rgba, vec, lut, stream);
    else if (members_at_once >= 64 && groups * 4 < wave)
        launch<8>(b, width, height, div, counts_out, bucket_out, rgba, vec, lut, stream);
    else if (members_at_once >= 32)
        launch<4>(b, width, height, div, counts_out, bucket_out, rgba, vec, lut, stream);
    else
        launch<2>(b, width, height, div, counts_out, bucket_out, rgba, vec, lut, stream);
    e = cudaGetLastError();
    if (e != cudaSuccess) return reject(CPT_ECUDA, cudaGetErrorString(e));
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}
