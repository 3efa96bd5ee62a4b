// bits_kernels.cu -- the accumulation step over bit-packed masks (one bit
// per pixel) for layouts the bulk-copy kernel of tma_kernels.cu does not take:
// padded or unaligned rows, and pinned host memory read in place.
#include <algorithm>

#include "bit_count.cuh"
#include "mask_load.cuh"
#include "overlap.cuh"

namespace cpt {
namespace {

constexpr int kThreads = 256;
constexpr int kPackedLimit = 255;   // members a bit-sliced counter can hold

// How a lane reads its share of a member's row.
enum WordLoads {
    kPairs = 0,     // two words, rows 8-byte aligned: a warp reads 256 contiguous bytes per member
    kSingles = 1,   // one word, rows 4-byte aligned
    kShifted = 2    // one word at any byte address, cut out of the two aligned words that hold it
};

// Bit-packed masks (one bit per pixel, pixel x at bit x & 7 of byte x >> 3 of
// the row).  A thread owns one or two 32-pixel words of a composite row and
// keeps the slab's counts in BitCounters (carry-save accumulators, see
// bit_count.cuh), 16 members per step; the bits past a row's last pixel are
// counted along (they are row padding, or the next row's) and dropped from
// the counters at the end, and the counts leave the bit-sliced form through
// bitcount_pairs.  Bound by memory latency: the bytes in flight wait in
// registers.  Rows that are no multiple of 16 bytes used to be copied into
// staging slots first: 1856 x 2208 x 1024 (rows of 232 bytes, which the
// bulk-copy kernel now takes in place) 852 us with clear and render.
template <typename CountT, int kLoads>
__global__ void __launch_bounds__(kThreads, 4)
count_bits_kernel(RasterBatch b, Plane p, int sign, int *flags, int64_t units, int units_per_row,
                  int slab, int slabs) {
    constexpr int kWords = kLoads == kPairs ? 2 : 1;
    constexpr int kPix = 32 * kWords;
    CountT *plane = static_cast<CountT *>(p.data);
    const int64_t stride = b.member_stride;
    const uint8_t *base = static_cast<const uint8_t *>(b.base);
    const uint8_t *end = batch_end(b, (p.width + 7) / 8, p.height);
    await_previous();
    for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < units * slabs;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int sl = (int)(u / units);
        const int64_t g = u - (int64_t)sl * units;
        const int y = (int)(g / units_per_row);
        const int gx = (int)(g - (int64_t)y * units_per_row);
        const int x0 = gx * kPix;
        const int valid = min(kPix, p.width - x0);
        const int m0 = sl * slab;
        const int m1 = min(b.n, m0 + slab);
        const uint8_t *at = base + (int64_t)y * b.row_pitch + gx * 4 * kWords;
        int f0, f1;
        safe_members(at, stride, base, end, 4 * kWords, kLoads == kSingles ? 4 : 8, m0, m1, f0, f1);
        BitCounter acc[kWords];
        const uint8_t *q = at + (int64_t)f0 * stride;
        for (int left = f1 - f0; left > 0; left -= 16) {
            uint32_t w[kWords][16], hi[16], shift[16];
#pragma unroll
            for (int k = 0; k < 16; ++k, q += stride) {
                const uint8_t *r = q;
                if constexpr (kLoads == kPairs) {
                    uint2 v = make_uint2(0u, 0u);
                    if (k < left) v = __ldcs(reinterpret_cast<const uint2 *>(r));
                    w[0][k] = v.x;
                    w[1][k] = v.y;
                } else if constexpr (kLoads == kSingles) {
                    w[0][k] = k < left ? __ldcs(reinterpret_cast<const uint32_t *>(r)) : 0u;
                } else {
                    shift[k] = (uint32_t)reinterpret_cast<uintptr_t>(r) & 3u;
                    const uint32_t *block = reinterpret_cast<const uint32_t *>(r - shift[k]);
                    w[0][k] = k < left ? __ldg(block) : 0u;
                    hi[k] = k < left ? __ldg(block + 1) : 0u;
                }
            }
            if constexpr (kLoads == kShifted)
#pragma unroll
                for (int k = 0; k < 16; ++k) w[0][k] = __funnelshift_r(w[0][k], hi[k], 8u * shift[k]);
#pragma unroll
            for (int j = 0; j < kWords; ++j) bitcount_add16(acc[j], w[j]);
        }
        // the few members whose aligned loads would leave the batch, byte by byte
        auto exact = [&](int m) {
            const uint8_t *r = at + (int64_t)m * stride;
            const int nbytes = (valid + 7) / 8;
#pragma unroll
            for (int j = 0; j < kWords; ++j) {
                uint32_t w[16] = {0u};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * j + i < nbytes) w[0] |= (uint32_t)r[4 * j + i] << (8 * i);
                bitcount_add16(acc[j], w);
            }
        };
        for (int m = m0; m < f0; ++m) exact(m);
        for (int m = f1; m < m1; ++m) exact(m);
        CountT *dst = plane + (int64_t)y * p.pitch + x0;
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
            const int vj = valid - 32 * j;
            if (vj <= 0) break;
            if (vj < 32) bitcount_keep(acc[j], (1u << vj) - 1u);
            uint32_t pairs[16];
            bitcount_pairs(acc[j], pairs);
#pragma unroll
            for (int h = 0; h < 2; ++h) {           // two 16-pixel groups per word
                if (vj <= 16 * h) break;            // a half word past the plane's pitch
                if (slabs == 1)
                    apply_pair_group<CountT>(dst + 32 * j + 16 * h, 16, pairs + 8 * h, sign, flags);
                else
                    atomic_pair_group<CountT>(dst + 32 * j + 16 * h, pairs + 8 * h, sign, flags);
            }
        }
    }
}

template <typename CountT>
void launch_count_bits_t(int loads, unsigned grid, cudaStream_t s, const RasterBatch &b, const Plane &p, int sign, int *flags,
                         int64_t units, int per_row, int slab, int slabs) {
    if (loads == kPairs)
        launch_overlapped(count_bits_kernel<CountT, kPairs>, grid, kThreads, 0, s, b, p, sign, flags, units, per_row, slab, slabs);
    else if (loads == kSingles)
        launch_overlapped(count_bits_kernel<CountT, kSingles>, grid, kThreads, 0, s, b, p, sign, flags, units, per_row, slab, slabs);
    else
        launch_overlapped(count_bits_kernel<CountT, kShifted>, grid, kThreads, 0, s, b, p, sign, flags, units, per_row, slab, slabs);
}

inline int64_t blocks_for(int64_t groups) {
    int64_t blocks = (groups + kThreads - 1) / kThreads;
    return blocks < 1 ? 1 : (blocks > 0x7FFFFFFF ? 0x7FFFFFFF : blocks);
}

}  // namespace

cudaError_t launch_count_bits(const RasterBatch &b, const Plane &p, int sign, int *flags,
                              const DeviceCaps &caps, cudaStream_t s) {
    const int wpr = (p.width + 31) / 32;
    if (b.n <= 0 || wpr == 0 || p.height == 0) return cudaSuccess;
    // two words (8 bytes) per thread and member where every row start is 8-byte aligned
    const uint64_t places = reinterpret_cast<uintptr_t>(b.base) | (uint64_t)b.row_pitch | (uint64_t)b.member_stride;
    const int loads = wpr >= 2 && places % 8 == 0 ? kPairs : places % 4 == 0 ? kSingles : kShifted;
    const int per_row = loads == kPairs ? (wpr + 1) / 2 : wpr;
    const int64_t units = (int64_t)per_row * p.height;
    // member slabs of at most 255 (eight counter levels); more only to fill
    // about four waves of four 256-thread CTAs per SM, since every slab pays
    // the bit-sliced epilogue and its atomics
    const int64_t target_units = 4ll * caps.num_sms * 4 * kThreads;
    int64_t slabs = (b.n + kPackedLimit - 1) / kPackedLimit;
    const int64_t want = std::min<int64_t>((target_units + units - 1) / units, (b.n + 31) / 32);
    slabs = std::max<int64_t>(std::max<int64_t>(slabs, want), 1);
    const int slab = (int)((b.n + slabs - 1) / slabs);
    slabs = (b.n + slab - 1) / slab;
    const unsigned grid = (unsigned)blocks_for(units * slabs);
    if (p.count_bits == 16)
        launch_count_bits_t<uint16_t>(loads, grid, s, b, p, sign, flags, units, per_row, slab, (int)slabs);
    else
        launch_count_bits_t<uint32_t>(loads, grid, s, b, p, sign, flags, units, per_row, slab, (int)slabs);
    return cudaGetLastError();
}

}  // namespace cpt
