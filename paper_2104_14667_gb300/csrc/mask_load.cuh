// mask_load.cuh -- reading and folding the 16-byte groups of mask rasters,
// shared by the linear and the engine accumulation kernels.
#pragma once

#include "device_common.cuh"

namespace cpt {

// The first `valid` (1..15) bytes of a 16-byte aligned group, zero above
// them, by at most four naturally aligned loads: nothing past the valid bytes
// is touched.  For the one group of a batch whose 16 bytes may reach past the
// caller's memory (the right edge of a raster's last row).
__device__ __forceinline__ uint4 load_group_exact(const uint8_t *p, int valid) {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    int at = 0;
    if (valid & 8) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        w[0] = v.x;
        w[1] = v.y;
        at = 8;
    }
    uint32_t t = 0;
    if (valid & 4) {
        t = *reinterpret_cast<const uint32_t *>(p + at);
        if (at) w[2] = t; else w[0] = t;
        at += 4;
    }
    t = 0;
    if (valid & 2) t = *reinterpret_cast<const uint16_t *>(p + at);
    if (valid & 1) t |= (uint32_t)p[at + (valid & 2)] << (8 * (valid & 2));
    const int i = at >> 2;
    if (i == 0) w[0] = t;
    if (i == 1) w[1] = t;
    if (i == 2) w[2] = t;
    if (i == 3) w[3] = t;
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void add_group(uint32_t (&k)[4], const uint4 &v) {
    k[0] += nonzero_bytes(v.x);
    k[1] += nonzero_bytes(v.y);
    k[2] += nonzero_bytes(v.z);
    k[3] += nonzero_bytes(v.w);
}

// Drops the counters of the pixels past the raster's right edge, whose bytes
// were row padding.  Once per fold: a counter never carries into the next
// pixel's (at most 255 members), so the padding does no harm until then.
__device__ __forceinline__ void keep_valid(uint32_t (&k)[4], int valid) {
    if (valid < 16)
#pragma unroll
        for (int i = 0; i < 4; ++i) k[i] &= 0xFFu * valid_byte_mask(i, valid);
}

// Rasters at any byte address.  The 16 bytes at an address are cut out of
// the two aligned 16-byte blocks that hold them: the blocks of neighbouring
// lanes overlap, so the second load is answered by the L1 cache, and about 15
// operations shift the bytes into place -- half of the instruction issue that
// the memory rate leaves per group.

// The 16 bytes from byte `shift` (0..15) of the 32 bytes lo, hi.
__device__ __forceinline__ uint4 align_group(const uint4 &lo, const uint4 &hi, uint32_t shift) {
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = (shift & 8u) ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = (shift & 4u) ? w[i + 1] : w[i];
    const uint32_t bits = (shift & 3u) * 8u;
    return make_uint4(__funnelshift_r(w[0], w[1], bits), __funnelshift_r(w[1], w[2], bits),
                      __funnelshift_r(w[2], w[3], bits), __funnelshift_r(w[3], w[4], bits));
}

// The first `valid` (0..16) bytes at p, zero above them, one by one.
__device__ __forceinline__ uint4 load_group_bytes(const uint8_t *p, int valid) {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (j < valid) w[j / 4] |= (uint32_t)p[j] << (8 * (j % 4));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Narrows [m0, m1), the members a lane folds at offset `q` of member 0, to
// those whose aligned loads -- `extent` bytes from the multiple of `grain` at
// or below the address -- stay within the batch, bytes [lo, hi).  The members
// left out (a few, at the very first and last pixels) take exact loads.
__device__ __forceinline__ void safe_members(const uint8_t *q, int64_t stride, const uint8_t *lo, const uint8_t *hi,
                                             int grain, int extent, int m0, int m1, int &s0, int &s1) {
    auto block = [&](int m) { return (reinterpret_cast<uintptr_t>(q) + (uintptr_t)(m * stride)) & ~(uintptr_t)(grain - 1); };
    s0 = m0;
    s1 = m1;
    while (s0 < s1 && block(s0) < reinterpret_cast<uintptr_t>(lo)) ++s0;
    while (s1 > s0 && block(s1 - 1) + extent > reinterpret_cast<uintptr_t>(hi)) --s1;
}

// Folds the masks of members [m0, m1) at one group into the packed counters
// k.  q: the group in member 0.  Eight members' loads are in flight at a time
// (twice as many where a group takes two blocks), the last ones' too: with a
// remainder loop of single loads a batch of 4 members cost four memory
// latencies instead of one.  The pointer steps from load to load: offsets
// j * stride are kept in registers that the loads in flight then lack.
template <bool kAligned>
__device__ __forceinline__ void fold_masks(const uint8_t *q, int64_t stride, int m0, int m1, uint32_t (&k)[4]) {
    q += (int64_t)m0 * stride;
    int left = m1 - m0;
    if constexpr (kAligned) {
        for (; left >= 8; left -= 8) {
            uint4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j, q += stride) v[j] = __ldcs(reinterpret_cast<const uint4 *>(q));
#pragma unroll
            for (int j = 0; j < 8; ++j) add_group(k, v[j]);
        }
        if (left > 0) {
            uint4 v[7];
#pragma unroll
            for (int j = 0; j < 7; ++j, q += stride) {
                v[j] = make_uint4(0u, 0u, 0u, 0u);
                if (j < left) v[j] = __ldcs(reinterpret_cast<const uint4 *>(q));
            }
#pragma unroll
            for (int j = 0; j < 7; ++j) add_group(k, v[j]);
        }
    } else {
        constexpr int kBatch = 8;
        for (; left >= kBatch; left -= kBatch) {
            uint4 lo[kBatch], hi[kBatch];
            uint32_t shift[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j, q += stride) {
                shift[j] = (uint32_t)reinterpret_cast<uintptr_t>(q) & 15u;
                const uint4 *block = reinterpret_cast<const uint4 *>(q - shift[j]);
                lo[j] = __ldg(block);
                hi[j] = __ldg(block + 1);
            }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) add_group(k, align_group(lo[j], hi[j], shift[j]));
        }
        if (left > 0) {
            uint4 lo[kBatch - 1], hi[kBatch - 1];
            uint32_t shift[kBatch - 1];
#pragma unroll
            for (int j = 0; j < kBatch - 1; ++j, q += stride) {
                lo[j] = hi[j] = make_uint4(0u, 0u, 0u, 0u);
                shift[j] = (uint32_t)reinterpret_cast<uintptr_t>(q) & 15u;
                const uint4 *block = reinterpret_cast<const uint4 *>(q - shift[j]);
                if (j < left) {
                    lo[j] = __ldg(block);
                    hi[j] = __ldg(block + 1);
                }
            }
#pragma unroll
            for (int j = 0; j < kBatch - 1; ++j) add_group(k, align_group(lo[j], hi[j], shift[j]));
        }
    }
}

// One past the last byte of a batch of rasters of `row` bytes by `height` rows.
__device__ __forceinline__ const uint8_t *batch_end(const RasterBatch &b, int64_t row, int height) {
    return static_cast<const uint8_t *>(b.base) + (int64_t)(b.n - 1) * b.member_stride +
           (int64_t)(height - 1) * b.row_pitch + row;
}

}  // namespace cpt
