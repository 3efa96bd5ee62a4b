// gather_kernels.cu -- copies into staging memory that a kernel makes better
// than the copy calls.
//
// The server's overflow upload: a cycle's distinct overflow rasters, scattered
// over the pinned host part, gathered into one device staging half by a single
// launch on the copy stream.  The kernel reads host memory through its device
// mapping over the host link, so one launch replaces one copy call per raster
// (a cycle moves about a thousand).
//
// Rasters at odd pitches or addresses into aligned staging rows: device rasters
// for the paths that need those (tensor maps, float arrays), pinned host
// rasters through their device mapping.
#include <algorithm>

#include "mask_load.cuh"

namespace cpt {
namespace {

constexpr int kThreads = 256;

// dst + i * stride <- src + ids[i] * stride, vecs_per_raster 16-byte vectors
// each; consecutive threads take consecutive vectors of one raster.
__global__ void __launch_bounds__(kThreads)
gather_rasters_kernel(uint8_t *dst, const uint8_t *src, const int32_t *ids, int n, int64_t stride,
                      int64_t vecs_per_raster) {
    const int64_t total = vecs_per_raster * n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / vecs_per_raster);
        const int64_t v = t - (int64_t)i * vecs_per_raster;
        const uint4 x = __ldcs(reinterpret_cast<const uint4 *>(src + (int64_t)ids[i] * stride) + v);
        reinterpret_cast<uint4 *>(dst + (int64_t)i * stride)[v] = x;
    }
}

// One 16-byte vector of a staging row per thread and member; blockIdx.y
// strides over the members.  Bound by HBM: two bytes moved per byte.
__global__ void __launch_bounds__(kThreads)
repitch_kernel(uint8_t *dst, int64_t dpitch, int64_t dmember, RasterBatch b, int64_t row, int height, int vecs_per_row) {
    const int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    if (t >= (int64_t)vecs_per_row * height) return;
    const int y = (int)(t / vecs_per_row);
    const int64_t x = (t - (int64_t)y * vecs_per_row) * 16;
    const int valid = (int)min((int64_t)16, row - x);
    const uint8_t *base = static_cast<const uint8_t *>(b.base);
    const uintptr_t lo = reinterpret_cast<uintptr_t>(base);
    const uintptr_t end = reinterpret_cast<uintptr_t>(batch_end(b, row, height));
    for (int m = blockIdx.y; m < b.n; m += gridDim.y) {
        const uint8_t *q = base + (int64_t)m * b.member_stride + (int64_t)y * b.row_pitch + x;
        const uint32_t shift = (uint32_t)reinterpret_cast<uintptr_t>(q) & 15u;
        const uintptr_t block = reinterpret_cast<uintptr_t>(q) - shift;
        uint4 v;
        if (block >= lo && block + 32 <= end) {
            const uint4 *at = reinterpret_cast<const uint4 *>(block);
            v = align_group(__ldg(at), __ldg(at + 1), shift);
            uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] &= 0xFFu * valid_byte_mask(i, valid);
            v = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
            v = load_group_bytes(q, valid);
        }
        *reinterpret_cast<uint4 *>(dst + (int64_t)m * dmember + (int64_t)y * dpitch + x) = v;
    }
}

}  // namespace

cudaError_t launch_repitch(void *dst, int64_t dpitch, int64_t dmember, const RasterBatch &b, int64_t row, int height,
                           cudaStream_t s) {
    if (b.n <= 0 || row <= 0 || height <= 0) return cudaSuccess;
    const int vecs = (int)((row + 15) / 16);
    const int64_t blocks = ((int64_t)vecs * height + kThreads - 1) / kThreads;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    repitch_kernel<<<dim3((unsigned)blocks, (unsigned)std::min(b.n, 65535)), kThreads, 0, s>>>(
        static_cast<uint8_t *>(dst), dpitch, dmember, b, row, height, vecs);
    return cudaGetLastError();
}

cudaError_t launch_gather_rasters(void *dst, const void *src, const int32_t *ids, int n, int64_t stride,
                                  int64_t raster_bytes, const DeviceCaps &caps, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t vecs = raster_bytes / 16;
    // two CTAs per SM: enough loads in flight for the link, and room left for
    // the compute kernels it overlaps
    const int64_t blocks = std::min<int64_t>((vecs * n + kThreads - 1) / kThreads, (int64_t)caps.num_sms * 2);
    gather_rasters_kernel<<<(unsigned)blocks, kThreads, 0, s>>>(
        static_cast<uint8_t *>(dst), static_cast<const uint8_t *>(src), ids, n, stride, vecs);
    return cudaGetLastError();
}

}  // namespace cpt
