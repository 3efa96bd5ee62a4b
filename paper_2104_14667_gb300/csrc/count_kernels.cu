// count_kernels.cu -- the accumulation step (Fig. 3, step 4: fold member i
// into the composite) over the linear read path, mask bytes and float32
// depths, at any alignment.
//
// One thread owns one 16-byte group of a composite row (16 mask pixels, or
// 4 float32 depth pixels) and walks members of the batch, so every member
// byte is read once with 16-byte loads and the composite is read and written
// once per launch instead of once per member (the paper's kernel reads and
// writes the accumulator per member, Fig. 2 step 4).  Mask bytes are turned
// into per-byte ones and summed four to a 32-bit word, in slabs of at most
// 255 members so the packed byte counters cannot overflow.  Both kernels are
// bound by HBM (large batches) or by its latency (small ones): 4096^2 x 1024
// takes 2.32 ms, 7.4 TB/s.  Rasters at odd addresses or pitches used to be
// copied into staging slots first: 1501 x 1103 x 100 with clear and render
// 338 us, now 46.
#include <algorithm>

#include "mask_load.cuh"
#include "overlap.cuh"

namespace cpt {
namespace {

constexpr int kThreads = 256;
constexpr int kPackedLimit = 255;   // members a packed byte counter can hold

// Work unit = (member slab, 16-byte group); blockIdx.y is the slab.  The
// CTA's kSlices slices of 256 / kSlices threads each take a share of the
// slab's members for the same groups and add their packed counters up in
// shared memory, four pixels to a thread: small rasters then fill the chip
// without atomics.  With more than one slab the counts go into the composite
// by atomics.
template <typename CountT, bool kAligned, int kSlices>
__global__ void __launch_bounds__(kThreads)
count_linear_kernel(RasterBatch b, Plane p, int sign, int *flags, int64_t groups, int groups_per_row, int slab) {
    constexpr int kGroups = kThreads / kSlices;
    CountT *plane = static_cast<CountT *>(p.data);
    const int lane_group = threadIdx.x % kGroups;
    const int slice = threadIdx.x / kGroups;
    const int64_t g = (int64_t)blockIdx.x * kGroups + lane_group;
    uint32_t k[4] = {0u, 0u, 0u, 0u};
    int y = 0, x0 = 0;
    await_previous();   // every thread: a clear or render before may still be using the plane
    if (g < groups) {
        y = (int)(g / groups_per_row);
        x0 = (int)(g - (int64_t)y * groups_per_row) * 16;
        const int valid = min(16, p.width - x0);
        const int s0 = blockIdx.y * slab, s1 = min(b.n, s0 + slab);
        const int share = (s1 - s0 + kSlices - 1) / kSlices;
        const int m0 = min(s1, s0 + slice * share), m1 = min(s1, m0 + share);
        const uint8_t *base = static_cast<const uint8_t *>(b.base);
        const uint8_t *q = base + (int64_t)y * b.row_pitch + x0;
        int f0, f1;
        safe_members(q, b.member_stride, base, batch_end(b, p.width, p.height), 16, kAligned ? 16 : 32, m0, m1, f0, f1);
        fold_masks<kAligned>(q, b.member_stride, f0, f1, k);
        for (int m = m0; m < f0; ++m) add_group(k, load_group_bytes(q + (int64_t)m * b.member_stride, valid));
        for (int m = f1; m < m1; ++m) add_group(k, load_group_bytes(q + (int64_t)m * b.member_stride, valid));
        keep_valid(k, valid);
    }
    if constexpr (kSlices == 1) {
        if (g >= groups) return;
        uint32_t wide[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) wide[j] = 0;
        widen16(wide, k[0], k[1], k[2], k[3]);
        // the plane's pitch is a whole number of groups: all 16 counts are its own
        CountT *dst = plane + (int64_t)y * p.pitch + x0;
        if (gridDim.y == 1)
            apply_count_group<CountT>(dst, 16, wide, sign, flags);
        else
            atomic_count_group<CountT>(dst, wide, sign, flags);
    } else {
        __shared__ uint4 part[kSlices][kGroups];
        part[slice][lane_group] = make_uint4(k[0], k[1], k[2], k[3]);
        __syncthreads();
        // word w of the CTA's groups, four pixels, consecutive words to consecutive threads
        for (int w = threadIdx.x; w < 4 * kGroups; w += kThreads) {
            const int64_t at = (int64_t)blockIdx.x * kGroups + w / 4;
            if (at >= groups) break;
            uint32_t sum = 0;
#pragma unroll
            for (int s = 0; s < kSlices; ++s) sum += reinterpret_cast<const uint32_t *>(part[s])[w];
            const int py = (int)(at / groups_per_row);
            CountT *dst = plane + (int64_t)py * p.pitch + (int)(at - (int64_t)py * groups_per_row) * 16 + (w % 4) * 4;
            if (gridDim.y == 1)
                apply_count_word<CountT>(dst, sum, sign, flags);
            else
                atomic_count_word<CountT>(dst, sum, sign, flags);
        }
    }
}

// Depth sums: the same over float32 rasters, four pixels to a group, without
// slabs (no atomics on floats: a pixel's sum has one fixed order).  Depths
// are 4-byte aligned, so a shift is a whole number of words.  A batch of eight
// members is added as a tree, eight batches into a block and the blocks into
// the total: 1024 members meet about 30 roundings instead of 1024.  Against 64
// bits, several hundred unaligned members were 3.8e-7 off summed one by one,
// 8.7e-8 as the sums of staged chunks and are 6.4e-8 off this way, at the same
// speed (1856 x 2208 x 64: 149 us, 7.0 TB/s).
template <bool kAligned>
__device__ __forceinline__ void fold_depths(const uint8_t *q, int64_t stride, int m0, int m1, float (&acc)[4]) {
    q += (int64_t)m0 * stride;
    int left = m1 - m0;
    while (left > 0) {
        float block[4] = {0.f, 0.f, 0.f, 0.f};
        for (int batch = 0; batch < 8 && left > 0; ++batch, left -= 8) {
            float4 lo[8], hi[8];
            uint32_t shift[8];
#pragma unroll
            for (int j = 0; j < 8; ++j, q += stride) {
                lo[j] = hi[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                shift[j] = kAligned ? 0u : (uint32_t)reinterpret_cast<uintptr_t>(q) & 15u;
                const float4 *at = reinterpret_cast<const float4 *>(q - shift[j]);
                if (j < left) {
                    lo[j] = kAligned ? __ldcs(at) : __ldg(at);
                    if (!kAligned) hi[j] = __ldg(at + 1);
                }
            }
            float d[8][4];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float w[8] = {lo[j].x, lo[j].y, lo[j].z, lo[j].w, hi[j].x, hi[j].y, hi[j].z, hi[j].w};
                if constexpr (!kAligned) {
#pragma unroll
                    for (int i = 0; i < 6; ++i) w[i] = (shift[j] & 8u) ? w[i + 2] : w[i];
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = (shift[j] & 4u) ? w[i + 1] : w[i];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) d[j][i] = w[i];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                block[i] += ((d[0][i] + d[1][i]) + (d[2][i] + d[3][i])) + ((d[4][i] + d[5][i]) + (d[6][i] + d[7][i]));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] += block[i];
    }
}

template <bool kAligned, int kSlices>
__global__ void __launch_bounds__(kThreads)
depth_linear_kernel(RasterBatch b, Plane p, int sign, int64_t groups, int groups_per_row) {
    constexpr int kGroups = kThreads / kSlices;
    float *plane = static_cast<float *>(p.data);
    const int lane_group = threadIdx.x % kGroups;
    const int slice = threadIdx.x / kGroups;
    const int64_t g = (int64_t)blockIdx.x * kGroups + lane_group;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    int y = 0, x0 = 0, valid = 0;
    await_previous();
    if (g < groups) {
        y = (int)(g / groups_per_row);
        x0 = (int)(g - (int64_t)y * groups_per_row) * 4;
        valid = min(4, p.width - x0);
        const int share = (b.n + kSlices - 1) / kSlices;
        const int m0 = min(b.n, slice * share), m1 = min(b.n, m0 + share);
        const uint8_t *base = static_cast<const uint8_t *>(b.base);
        const uint8_t *q = base + (int64_t)y * b.row_pitch + x0 * 4;
        int f0, f1;
        safe_members(q, b.member_stride, base, batch_end(b, (int64_t)p.width * 4, p.height), 16, kAligned ? 16 : 32, m0, m1,
                     f0, f1);
        auto exact = [&](int m) {
            const float *d = reinterpret_cast<const float *>(q + (int64_t)m * b.member_stride);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < valid) acc[j] += d[j];
        };
        for (int m = m0; m < f0; ++m) exact(m);
        fold_depths<kAligned>(q, b.member_stride, f0, f1, acc);
        for (int m = f1; m < m1; ++m) exact(m);
    }
    if constexpr (kSlices > 1) {
        __shared__ float4 part[kSlices][kGroups];
        part[slice][lane_group] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        __syncthreads();
        if (slice > 0) return;
#pragma unroll
        for (int s = 1; s < kSlices; ++s) {
            const float4 v = part[s][lane_group];
            acc[0] += v.x;
            acc[1] += v.y;
            acc[2] += v.z;
            acc[3] += v.w;
        }
    }
    if (g < groups) apply_depth_group(plane + (int64_t)y * p.pitch + x0, valid, acc, sign);
}

bool batch_aligned(const RasterBatch &b) {
    return reinterpret_cast<uintptr_t>(b.base) % 16 == 0 && b.row_pitch % 16 == 0 && b.member_stride % 16 == 0;
}

constexpr int64_t kMaxSlabs = 65535;   // grid rows

// How a launch is cut: slices of a CTA, and member slabs (grid rows).  Slices
// of at least eight members, up to four -- neighbouring warps then read the
// same pixels of different members, which also suits the memory system -- and
// eight where four leave the chip less than one wave of threads.  A slab is a
// whole number of load batches per slice.  More slabs than the counters need
// only where even the slices leave less than a quarter of a wave, down to
// eight members per slice.  Measured (us; slices/slabs): 1856x2208x64 1/1 52,
// 1/8 85, 4/1 42, 8/1 44; 2048^2 x 256 1/4 168, 4/2 147 (7.3 TB/s); 4096^2 x
// 64 1/1 157, 1/2 190, 4/1 157; 512^2 x 255 1/8 16, 4/1 14, 8/1 10.7; 256^2 x
// 300 1/8 8.4, 8/2 5.5; 1024^2 x 16 1/1 5.9, 2/1 6.0; 109x105x614 1/8 18, 8/3
// 8.2, 8/8 5.5.  Unaligned: 1501x1103x100 1/1 42, 4/1 37; x400 1/2 149, 4/2 116.
struct CountSplit {
    int slices;
    int slab;
    int slabs;
};

CountSplit split_count(int64_t groups, int n, const DeviceCaps &caps) {
    const int64_t wave = (int64_t)caps.num_sms * 2048;
    int64_t slabs = (n + kPackedLimit - 1) / kPackedLimit;
    const int64_t members = (n + slabs - 1) / slabs;
    int slices = members >= 32 ? 4 : members >= 16 ? 2 : 1;
    if (members >= 64 && groups * 4 < wave) slices = 8;
    slabs = std::max(slabs, std::min<int64_t>(wave / (4 * groups * slices), n / (8 * slices)));
    slabs = std::max<int64_t>(1, std::min(slabs, kMaxSlabs));
    int slab = (int)((n + slabs - 1) / slabs);
    const int whole = (slab + 8 * slices - 1) / (8 * slices) * (8 * slices);
    if (slabs > 1 && whole <= kPackedLimit) slab = whole;
    return {slices, slab, (n + slab - 1) / slab};
}

// Slices of a depth launch: no slabs to fall back on, and a group is a
// quarter of the pixels, so only rasters of less than a third of a wave are
// split (us: 533x438x87 1 15.1, 2 11.6, 4 13.8; 476x239x71 1 8.8, 4 5.2;
// 1856x2208x64 1 148, 4 148; 3045x1992x16 1 72, 4 95).
int depth_slices(int64_t groups, int n, const DeviceCaps &caps) {
    const int64_t wave = (int64_t)caps.num_sms * 2048;
    int s = 1;
    while (s < 8 && n >= 16 * s && 3 * groups * s < wave) s *= 2;
    return s;
}

template <typename CountT, bool kAligned>
cudaError_t launch_count_t(const RasterBatch &b, const Plane &p, int sign, int *flags, const DeviceCaps &caps,
                           cudaStream_t s) {
    const int gpr = (p.width + 15) / 16;
    const int64_t groups = (int64_t)gpr * p.height;
    const CountSplit c = split_count(groups, b.n, caps);
    const int64_t per_cta = kThreads / c.slices;
    const int64_t blocks = (groups + per_cta - 1) / per_cta;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)blocks, (unsigned)c.slabs);
    switch (c.slices) {
        case 1: launch_overlapped(count_linear_kernel<CountT, kAligned, 1>, grid, kThreads, 0, s, b, p, sign, flags, groups, gpr, c.slab); break;
        case 2: launch_overlapped(count_linear_kernel<CountT, kAligned, 2>, grid, kThreads, 0, s, b, p, sign, flags, groups, gpr, c.slab); break;
        case 4: launch_overlapped(count_linear_kernel<CountT, kAligned, 4>, grid, kThreads, 0, s, b, p, sign, flags, groups, gpr, c.slab); break;
        default: launch_overlapped(count_linear_kernel<CountT, kAligned, 8>, grid, kThreads, 0, s, b, p, sign, flags, groups, gpr, c.slab); break;
    }
    return cudaGetLastError();
}

template <bool kAligned>
cudaError_t launch_depth_t(const RasterBatch &b, const Plane &p, int sign, const DeviceCaps &caps, cudaStream_t s) {
    const int gpr = (p.width + 3) / 4;
    const int64_t groups = (int64_t)gpr * p.height;
    const int slices = depth_slices(groups, b.n, caps);
    const int64_t per_cta = kThreads / slices;
    const int64_t blocks = (groups + per_cta - 1) / per_cta;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)blocks;
    switch (slices) {
        case 1: launch_overlapped(depth_linear_kernel<kAligned, 1>, grid, kThreads, 0, s, b, p, sign, groups, gpr); break;
        case 2: launch_overlapped(depth_linear_kernel<kAligned, 2>, grid, kThreads, 0, s, b, p, sign, groups, gpr); break;
        case 4: launch_overlapped(depth_linear_kernel<kAligned, 4>, grid, kThreads, 0, s, b, p, sign, groups, gpr); break;
        default: launch_overlapped(depth_linear_kernel<kAligned, 8>, grid, kThreads, 0, s, b, p, sign, groups, gpr); break;
    }
    return cudaGetLastError();
}

// From this size on two memsets are quicker than the kernel (134 MB 22.7 us
// either way, 196 MB 30.4 and 31.8, 268 MB 39.8 and 42.3).
constexpr int64_t kMemsetBytes = 144ll << 20;

// Counts (or sums) and device flags to zero, in one launch.
__global__ void __launch_bounds__(kThreads)
clear_plane_kernel(uint4 *data, int64_t words, int *flags) {
    await_previous();
    if (blockIdx.x == 0 && threadIdx.x < kFlagCount) flags[threadIdx.x] = 0;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < words; i += (int64_t)gridDim.x * kThreads)
        data[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace

cudaError_t launch_clear_plane(void *data, int64_t bytes, int *flags, const DeviceCaps &caps, cudaStream_t s) {
    if (bytes >= kMemsetBytes) {
        const cudaError_t e = cudaMemsetAsync(flags, 0, kFlagCount * sizeof(int), s);
        return e != cudaSuccess ? e : cudaMemsetAsync(data, 0, (size_t)bytes, s);
    }
    const int64_t words = bytes / 16;   // plane rows are whole 16-byte vectors
    const int64_t blocks = std::min<int64_t>((words + 4 * kThreads - 1) / (4 * kThreads), 8ll * caps.num_sms);
    launch_overlapped(clear_plane_kernel, (unsigned)std::max<int64_t>(1, blocks), kThreads, 0, s, static_cast<uint4 *>(data), words, flags);
    return cudaGetLastError();
}

cudaError_t launch_count_linear(const RasterBatch &b, const Plane &p, int sign, int *flags,
                                const DeviceCaps &caps, cudaStream_t s) {
    if (b.n <= 0 || p.width <= 0 || p.height <= 0) return cudaSuccess;
    const bool aligned = batch_aligned(b);
    // a launch holds kMaxSlabs slabs; batches beyond that take several
    constexpr int64_t kMost = kMaxSlabs * kPackedLimit;
    for (int64_t m0 = 0; m0 < b.n; m0 += kMost) {
        RasterBatch part = b;
        part.base = static_cast<const uint8_t *>(b.base) + m0 * b.member_stride;
        part.n = (int32_t)std::min<int64_t>(kMost, b.n - m0);
        const cudaError_t e =
            p.count_bits == 16 ? (aligned ? launch_count_t<uint16_t, true>(part, p, sign, flags, caps, s)
                                          : launch_count_t<uint16_t, false>(part, p, sign, flags, caps, s))
                               : (aligned ? launch_count_t<uint32_t, true>(part, p, sign, flags, caps, s)
                                          : launch_count_t<uint32_t, false>(part, p, sign, flags, caps, s));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_depth_linear(const RasterBatch &b, const Plane &p, int sign, int *,
                                const DeviceCaps &caps, cudaStream_t s) {
    if (b.n <= 0 || p.width <= 0 || p.height <= 0) return cudaSuccess;
    return batch_aligned(b) ? launch_depth_t<true>(b, p, sign, caps, s) : launch_depth_t<false>(b, p, sign, caps, s);
}

}  // namespace cpt
