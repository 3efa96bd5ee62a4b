// texture_kernels.cu -- the texture (image) read path: the accumulation
// step over members held as layers of a cudaArray, and the hand-written
// buffer-to-array conversion (Section 4's layout transform) through a
// surface object.
#include <algorithm>

#include "bit_count.cuh"
#include "mask_load.cuh"

namespace cpt {
namespace {

constexpr int kPackedLimit = 255;   // members a packed byte counter can hold

// Both texture-path kernels walk the layered array in 2-D tiles of texels
// rather than along rows: the array is stored in tiles of rows (block
// linear), and a CTA that covers a few texels of many rows reads and writes
// whole tiles.  Measured at 4096 x 4096 x 32 layers, alone on the GPU: the
// texture count moved 5.44 TB/s of member bytes with 4 x 32 tiles against
// 4.78 with a CTA per row, and the conversion 3.19 TB/s of source (6.4 TB/s
// of DRAM traffic, read plus write) with 16 x 8 tiles against 2.60 for a
// flat, row-ordered index.  Several layers per conversion thread were slower
// (1.8-2.4 TB/s): the stores, not the loads in flight, set the pace.
constexpr int kCountTileW = 4, kCountTileH = 32;
constexpr int kConvertTileW = 16, kConvertTileH = 8;
constexpr int kTileThreads = 128;
static_assert(kCountTileW * kCountTileH == kTileThreads && kConvertTileW * kConvertTileH == kTileThreads,
              "tiles fill a CTA");

// Texture path: member `layer` of the batch is layer `layer` of a layered
// cudaArray whose texels are 16 bytes (16 mask pixels).  Texels past the
// raster's right edge hold padding and are masked off.  One thread per texel
// column (x, y), over every layer.
template <typename CountT>
__global__ void __launch_bounds__(kTileThreads)
count_texture_kernel(cudaTextureObject_t tex, int n_layers, Plane p, int sign, int *flags, int groups_per_row) {
    const int gx = blockIdx.x * kCountTileW + (int)(threadIdx.x % kCountTileW);
    const int y = blockIdx.y * kCountTileH + (int)(threadIdx.x / kCountTileW);
    if (gx >= groups_per_row || y >= p.height) return;
    CountT *plane = static_cast<CountT *>(p.data);
    const int x0 = gx * 16;
    const int valid = min(16, p.width - x0);
    const uint32_t m0 = valid_byte_mask(0, valid), m1 = valid_byte_mask(1, valid);
    const uint32_t m2 = valid_byte_mask(2, valid), m3 = valid_byte_mask(3, valid);
    const float u = gx + 0.5f, v = y + 0.5f;
    uint32_t k0 = 0, k1 = 0, k2 = 0, k3 = 0;
#pragma unroll 8
    for (int layer = 0; layer < n_layers; ++layer) {
        const uint4 t = tex2DLayered<uint4>(tex, u, v, layer);
        k0 += nonzero_bytes(t.x) & m0;
        k1 += nonzero_bytes(t.y) & m1;
        k2 += nonzero_bytes(t.z) & m2;
        k3 += nonzero_bytes(t.w) & m3;
    }
    uint32_t wide[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) wide[j] = 0;
    widen16(wide, k0, k1, k2, k3);
    apply_count_group<CountT>(plane + (int64_t)y * p.pitch + x0, valid, wide, sign, flags);
}

__global__ void __launch_bounds__(kTileThreads)
depth_texture_kernel(cudaTextureObject_t tex, int n_layers, Plane p, int sign, int groups_per_row) {
    const int gx = blockIdx.x * kCountTileW + (int)(threadIdx.x % kCountTileW);
    const int y = blockIdx.y * kCountTileH + (int)(threadIdx.x / kCountTileW);
    if (gx >= groups_per_row || y >= p.height) return;
    float *plane = static_cast<float *>(p.data);
    const int x0 = gx * 4;
    const int valid = min(4, p.width - x0);
    const float u = gx + 0.5f, v = y + 0.5f;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int layer = 0; layer < n_layers; ++layer) {
        const float4 t = tex2DLayered<float4>(tex, u, v, layer);
        acc[0] += t.x;
        acc[1] += valid > 1 ? t.y : 0.f;
        acc[2] += valid > 2 ? t.z : 0.f;
        acc[3] += valid > 3 ? t.w : 0.f;
    }
    apply_depth_group(plane + (int64_t)y * p.pitch + x0, valid, acc, sign);
}

// Layout conversion by hand (the buffer-to-image transform of Section 4):
// one thread per 16-byte texel of one layer, a 16-byte streaming load from
// the linear raster and a surface store into the layered array, over a grid
// of (tile column, tile row, layer).
__global__ void __launch_bounds__(kTileThreads)
convert_to_array_kernel(const uint8_t *src, int64_t pitch, int64_t member_stride, cudaSurfaceObject_t surf,
                        int texels_per_row, int height) {
    const int x = blockIdx.x * kConvertTileW + (int)(threadIdx.x % kConvertTileW);
    const int y = blockIdx.y * kConvertTileH + (int)(threadIdx.x / kConvertTileW);
    const int layer = blockIdx.z;
    if (x >= texels_per_row || y >= height) return;
    const uint4 v = __ldcs(reinterpret_cast<const uint4 *>(src + layer * member_stride + (int64_t)y * pitch + x * 16));
    surf2DLayeredwrite(v, surf, x * 16, y, layer);
}

// ---- bit-packed arrays ---------------------------------------------------------
//
// With the conversion kernel the layers of a mask array hold one bit per
// pixel: a texel is two 32-pixel words.  A byte per pixel makes the path move
// three bytes per member byte (read, write into the array, fetch); a bit makes
// it 1.25, and the fold fetches an eighth of the texels.  2048^2 x 256
// resident: 620 us a pass with byte arrays, of which the array's own traffic
// was two thirds.
constexpr int kPackedTexelPx = 64;
constexpr int kPackLayers = 8;      // layers per conversion thread, all loads in flight
constexpr int kPackTileH = 8;
constexpr int kPackThreads = 32 * kPackTileH;
constexpr int kFoldTileW = 8, kFoldTileH = 8;   // an 8-byte texel: tiles of 64 bytes by rows, as above
constexpr int kFoldTexels = kFoldTileW * kFoldTileH;
constexpr int kFoldLayers = 255;    // members a bit-sliced counter can hold

// 16 mask bytes as 16 bits: each word's four 0/1 bytes meet in its top four
// bits (28 + 0, 21 + 8, 14 + 16, 7 + 24; no other product reaches them).
__device__ __forceinline__ uint32_t mask_bits(const uint4 &v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t bits = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) bits |= ((nonzero_bytes(w[i]) * 0x10204080u) >> 28) << (4 * i);
    return bits;
}

// Conversion: a lane reads the 16 bytes of 16 pixels, four lanes' bits make a
// texel.  `lanes` (4, 8, 16 or 32) lanes side by side cover a row piece, so
// that narrow rasters fill their warps with rows; blockIdx.z counts blocks of
// kPackLayers members.  Rasters of any alignment (kAligned: 16 bytes).
template <bool kAligned>
__global__ void __launch_bounds__(kPackThreads)
pack_to_array_kernel(RasterBatch b, int width, int height, int lanes, cudaSurfaceObject_t surf) {
    const int lane = threadIdx.x & 31;
    const int rows = 32 / lanes;
    const int x = (blockIdx.x * lanes + lane % lanes) * 16;
    const int y = (blockIdx.y * kPackTileH + (int)(threadIdx.x >> 5)) * rows + lane / lanes;
    const bool inside = x < width && y < height;
    const int valid = inside ? min(16, width - x) : 0;
    const uint8_t *base = static_cast<const uint8_t *>(b.base);
    const uint8_t *q = base + (int64_t)y * b.row_pitch + x;
    const uintptr_t lo = reinterpret_cast<uintptr_t>(base);
    const uintptr_t end = reinterpret_cast<uintptr_t>(batch_end(b, width, height));
    const int m0 = blockIdx.z * kPackLayers;
    uint4 v[kPackLayers];
#pragma unroll
    for (int k = 0; k < kPackLayers; ++k) {
        v[k] = make_uint4(0u, 0u, 0u, 0u);
        if (!inside || m0 + k >= b.n) continue;
        const uint8_t *r = q + (int64_t)(m0 + k) * b.member_stride;
        const uint32_t shift = kAligned ? 0u : (uint32_t)reinterpret_cast<uintptr_t>(r) & 15u;
        const uintptr_t block = reinterpret_cast<uintptr_t>(r) - shift;
        if (block >= lo && block + (kAligned ? 16 : 32) <= end) {
            const uint4 *at = reinterpret_cast<const uint4 *>(block);
            v[k] = kAligned ? __ldcs(at) : align_group(__ldg(at), __ldg(at + 1), shift);
        } else {
            v[k] = load_group_bytes(r, valid);
        }
    }
    const uint32_t keep = (1u << valid) - 1u;
#pragma unroll
    for (int k = 0; k < kPackLayers; ++k) {
        const uint32_t h = mask_bits(v[k]) & keep;
        const uint32_t word = h | (__shfl_down_sync(0xFFFFFFFFu, h, 1) << 16);   // in even lanes
        const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, word, 2);
        if (lane % 4 == 0 && inside && m0 + k < b.n)
            surf2DLayeredwrite(make_uint2(word, next), surf, x / kPackedTexelPx * 8, y, m0 + k);
    }
}

// The fold over bit-packed layers: one thread per texel and slice, 16 layers'
// texels in flight, the counts of its 64 pixels in carry-save accumulators.
// The slices of a CTA share the layers -- texels alone are few threads: 2048^2
// has 65536, and one slice took 42 us for 248 layers -- and add up their
// counts, two to a word, in shared memory, from where consecutive threads
// fold consecutive words into the composite.
template <typename CountT, int kSlices>
__global__ void __launch_bounds__(kFoldTexels * kSlices)
count_packed_texture_kernel(cudaTextureObject_t tex, int n_layers, Plane p, int sign, int *flags) {
    constexpr int kThreads = kFoldTexels * kSlices;
    constexpr int kWords = kPackedTexelPx / 2;
    // [slice][word][texel], padded so that neither order of access shares banks
    __shared__ uint32_t part[kSlices][kWords][kFoldTexels + 1];
    const int texel = threadIdx.x % kFoldTexels, slice = threadIdx.x / kFoldTexels;
    const int gx = blockIdx.x * kFoldTileW + texel % kFoldTileW;
    const int y = blockIdx.y * kFoldTileH + texel / kFoldTileW;
    const float u = gx + 0.5f, v = y + 0.5f;
    const int share = ((n_layers + kSlices - 1) / kSlices + 15) / 16 * 16;   // whole steps
    const int l0 = min(n_layers, slice * share), l1 = min(n_layers, l0 + share);
    BitCounter acc[2];
    if (gx * kPackedTexelPx < p.width && y < p.height) {
        for (int l = l0; l < l1; l += 16) {
            uint32_t w[2][16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                uint2 t = make_uint2(0u, 0u);
                if (l + k < l1) t = tex2DLayered<uint2>(tex, u, v, l + k);
                w[0][k] = t.x;
                w[1][k] = t.y;
            }
            bitcount_add16(acc[0], w[0]);
            bitcount_add16(acc[1], w[1]);
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        uint32_t pairs[16];
        bitcount_pairs(acc[j], pairs);
#pragma unroll
        for (int i = 0; i < 16; ++i) part[slice][16 * j + i][texel] = pairs[i];
    }
    __syncthreads();
    bool under = false;
    // eight words' counts are loaded before any is stored: one after another
    // each would wait for its own load
    constexpr int kAtOnce = 8;
    for (int i0 = threadIdx.x; i0 < kFoldTexels * kWords; i0 += kThreads * kAtOnce) {
        CountT *dst[kAtOnce];
        uint32_t d[kAtOnce], c[kAtOnce][2];
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
            const int i = i0 + j * kThreads;
            const int t = i / kWords, w = i % kWords;
            const int x = (blockIdx.x * kFoldTileW + t % kFoldTileW) * kPackedTexelPx + 2 * w;
            const int py = blockIdx.y * kFoldTileH + t / kFoldTileW;
            // pixel x + 1 is at most row padding, with no bits set
            dst[j] = x < p.width && py < p.height ? static_cast<CountT *>(p.data) + (int64_t)py * p.pitch + x : nullptr;
            if (!dst[j]) continue;
            d[j] = 0;
#pragma unroll
            for (int s = 0; s < kSlices; ++s) d[j] += part[s][w][t];   // at most 255 layers: no carry
            if constexpr (sizeof(CountT) == 2) {
                c[j][0] = *reinterpret_cast<const uint32_t *>(dst[j]);
            } else {
                const uint2 v = *reinterpret_cast<const uint2 *>(dst[j]);
                c[j][0] = v.x, c[j][1] = v.y;
            }
        }
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
            if (!dst[j]) continue;
            const uint32_t d0 = d[j] & 0xFFFFu, d1 = d[j] >> 16;
            uint32_t c0 = sizeof(CountT) == 2 ? c[j][0] & 0xFFFFu : c[j][0];
            uint32_t c1 = sizeof(CountT) == 2 ? c[j][0] >> 16 : c[j][1];
            under |= sign < 0 && (d0 > c0 || d1 > c1);
            c0 = sign > 0 ? c0 + d0 : c0 - d0;
            c1 = sign > 0 ? c1 + d1 : c1 - d1;
            if constexpr (sizeof(CountT) == 2)
                *reinterpret_cast<uint32_t *>(dst[j]) = (c0 & 0xFFFFu) | (c1 << 16);
            else
                *reinterpret_cast<uint2 *>(dst[j]) = make_uint2(c0, c1);
        }
    }
    if (under) flag_set(flags, kFlagUnderflow);
}

// Grid of (tile columns, tile rows[, layers]); false when a dimension is
// beyond the launch limits (never for arrays within the texture limits).
inline bool tile_grid(dim3 *g, int cols, int rows, int tw, int th, int layers) {
    *g = dim3((unsigned)((cols + tw - 1) / tw), (unsigned)((rows + th - 1) / th), (unsigned)layers);
    return g->y <= 65535 && g->z <= 65535;
}

}  // namespace

cudaError_t launch_count_texture(cudaTextureObject_t tex, int n_layers, const Plane &p, int sign,
                                 int *flags, const DeviceCaps &, cudaStream_t s) {
    const int gpr = (p.width + 15) / 16;
    if (n_layers <= 0 || p.height <= 0 || gpr == 0) return cudaSuccess;
    if (n_layers > kPackedLimit) return cudaErrorInvalidValue;
    dim3 grid;
    if (!tile_grid(&grid, gpr, p.height, kCountTileW, kCountTileH, 1)) return cudaErrorInvalidValue;
    if (p.count_bits == 16)
        count_texture_kernel<uint16_t><<<grid, kTileThreads, 0, s>>>(tex, n_layers, p, sign, flags, gpr);
    else
        count_texture_kernel<uint32_t><<<grid, kTileThreads, 0, s>>>(tex, n_layers, p, sign, flags, gpr);
    return cudaGetLastError();
}

cudaError_t launch_convert_to_array(const void *src, int64_t pitch, int64_t member_stride,
                                    cudaSurfaceObject_t surf, int texels_per_row, int height, int n_layers,
                                    cudaStream_t s) {
    if (texels_per_row <= 0 || height <= 0 || n_layers <= 0) return cudaSuccess;
    dim3 grid;
    if (!tile_grid(&grid, texels_per_row, height, kConvertTileW, kConvertTileH, n_layers)) return cudaErrorInvalidValue;
    convert_to_array_kernel<<<grid, kTileThreads, 0, s>>>(static_cast<const uint8_t *>(src), pitch, member_stride,
                                                          surf, texels_per_row, height);
    return cudaGetLastError();
}

int packed_texels(int width) { return (width + kPackedTexelPx - 1) / kPackedTexelPx; }

cudaError_t launch_pack_to_array(const RasterBatch &b, int width, int height, cudaSurfaceObject_t surf, cudaStream_t s) {
    if (b.n <= 0 || width <= 0 || height <= 0) return cudaSuccess;
    int lanes = 4;   // whole texels
    while (lanes < 32 && lanes * 16 < width) lanes *= 2;
    const int rows = kPackTileH * (32 / lanes);
    dim3 grid;
    if (!tile_grid(&grid, (width + 15) / 16, height, lanes, rows, (b.n + kPackLayers - 1) / kPackLayers))
        return cudaErrorInvalidValue;
    const bool aligned = reinterpret_cast<uintptr_t>(b.base) % 16 == 0 && b.row_pitch % 16 == 0 && b.member_stride % 16 == 0;
    if (aligned)
        pack_to_array_kernel<true><<<grid, kPackThreads, 0, s>>>(b, width, height, lanes, surf);
    else
        pack_to_array_kernel<false><<<grid, kPackThreads, 0, s>>>(b, width, height, lanes, surf);
    return cudaGetLastError();
}

cudaError_t launch_count_packed_texture(cudaTextureObject_t tex, int n_layers, const Plane &p, int sign, int *flags,
                                        const DeviceCaps &, cudaStream_t s) {
    if (n_layers <= 0 || p.height <= 0 || p.width <= 0) return cudaSuccess;
    if (n_layers > kFoldLayers) return cudaErrorInvalidValue;
    dim3 grid;
    if (!tile_grid(&grid, packed_texels(p.width), p.height, kFoldTileW, kFoldTileH, 1)) return cudaErrorInvalidValue;
    // four slices from two steps of layers on
    const bool u16 = p.count_bits == 16;
    if (n_layers > 16) {
        if (u16)
            count_packed_texture_kernel<uint16_t, 4><<<grid, 4 * kFoldTexels, 0, s>>>(tex, n_layers, p, sign, flags);
        else
            count_packed_texture_kernel<uint32_t, 4><<<grid, 4 * kFoldTexels, 0, s>>>(tex, n_layers, p, sign, flags);
    } else if (u16) {
        count_packed_texture_kernel<uint16_t, 1><<<grid, kFoldTexels, 0, s>>>(tex, n_layers, p, sign, flags);
    } else {
        count_packed_texture_kernel<uint32_t, 1><<<grid, kFoldTexels, 0, s>>>(tex, n_layers, p, sign, flags);
    }
    return cudaGetLastError();
}

cudaError_t launch_depth_texture(cudaTextureObject_t tex, int n_layers, const Plane &p, int sign,
                                 int *, const DeviceCaps &, cudaStream_t s) {
    const int gpr = (p.width + 3) / 4;
    if (n_layers <= 0 || p.height <= 0 || gpr == 0) return cudaSuccess;
    dim3 grid;
    if (!tile_grid(&grid, gpr, p.height, kCountTileW, kCountTileH, 1)) return cudaErrorInvalidValue;
    depth_texture_kernel<<<grid, kTileThreads, 0, s>>>(tex, n_layers, p, sign, gpr);
    return cudaGetLastError();
}

}  // namespace cpt
