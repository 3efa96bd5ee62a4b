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

}  // namespace cpt
