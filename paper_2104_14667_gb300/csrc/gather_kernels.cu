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
#include <mutex>
#include <set>
#include <utility>

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

// The 16 bytes of member m's staging row y from byte x on, `valid` of them the
// row's.  [lo, end): the batch.
__device__ __forceinline__ void move_vector(uint8_t *dst, int64_t dpitch, int64_t dmember, const RasterBatch &b,
                                            const uint8_t *base, uintptr_t lo, uintptr_t end, int y, int64_t x, int valid,
                                            int m) {
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
    for (int m = blockIdx.y; m < b.n; m += gridDim.y)
        move_vector(dst, dpitch, dmember, b, base, lo, end, y, x, valid, m);
}

// The same by two CTAs per SM, for uploads over the host link beside a fold of
// the TMA path.  The fold's CTAs hold 140 KB of shared memory: they find a place
// only on an SM with threads to spare that runs at a large shared memory size,
// which this kernel therefore asks for too.  Without either, uploads and folds
// took turns (ms: a thread per vector / two CTAs per SM / and the larger size):
// 16 depths of 4090 x 1500 2.97 / 2.95 / 2.11, 32 of 4090 x 2048 8.33 / 8.19 /
// 5.61, 48 of 1001 x 3000 3.79 / 3.80 / 3.06, 16 masks of 504 x 1500 0.086 /
// 0.088 / 0.086; four CTAs per SM are too many for some (16 masks of 16001 x
// 1500 3.43, two 2.10).
constexpr int kBesideCtasPerSm = 2;

__global__ void __launch_bounds__(kThreads)
repitch_beside_kernel(uint8_t *dst, int64_t dpitch, int64_t dmember, RasterBatch b, int64_t row, int height, int vecs_per_row) {
    const int64_t vecs = (int64_t)vecs_per_row * height;
    const uint8_t *base = static_cast<const uint8_t *>(b.base);
    const uintptr_t lo = reinterpret_cast<uintptr_t>(base);
    const uintptr_t end = reinterpret_cast<uintptr_t>(batch_end(b, row, height));
    for (int m = blockIdx.y; m < b.n; m += gridDim.y)
        for (int64_t t = blockIdx.x * (int64_t)kThreads + threadIdx.x; t < vecs; t += (int64_t)gridDim.x * kThreads) {
            const int y = (int)(t / vecs_per_row);
            const int64_t x = (t - (int64_t)y * vecs_per_row) * 16;
            move_vector(dst, dpitch, dmember, b, base, lo, end, y, x, (int)min((int64_t)16, row - x), m);
        }
}

// Asks for the largest shared memory size for a kernel, once on each device.
cudaError_t prefer_shared(const void *kernel) {
    static std::mutex mu;
    static std::set<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({kernel, dev})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) done.insert({kernel, dev});
    return e;
}

}  // namespace

cudaError_t launch_repitch(void *dst, int64_t dpitch, int64_t dmember, const RasterBatch &b, int64_t row, int height,
                           bool leave_room, const DeviceCaps &caps, cudaStream_t s) {
    if (b.n <= 0 || row <= 0 || height <= 0) return cudaSuccess;
    const int vecs = (int)((row + 15) / 16);
    const int64_t blocks = ((int64_t)vecs * height + kThreads - 1) / kThreads;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    if (leave_room) {
        const cudaError_t e = prefer_shared(reinterpret_cast<const void *>(repitch_beside_kernel));
        if (e != cudaSuccess) return e;
        const int ctas = kBesideCtasPerSm * caps.num_sms;
        const int x = (int)std::min<int64_t>(blocks, ctas);
        const int y = std::max(1, std::min(b.n, ctas / x));
        repitch_beside_kernel<<<dim3((unsigned)x, (unsigned)y), kThreads, 0, s>>>(
            static_cast<uint8_t *>(dst), dpitch, dmember, b, row, height, vecs);
        return cudaGetLastError();
    }
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
