// render_units.cuh -- the display step in units of four consecutive pixels of
// the dense outputs, shared by the plain and the engine render: reading a
// unit's counts from a padded plane, and storing its counts, classes and
// colours.
//
// A warp item is 32 x kUnits units, a unit per lane at a time: consecutive
// lanes store consecutive 16 bytes of colours, and a lane has kUnits loads in
// flight.  With 16 consecutive pixels per lane every store instruction touched
// 32 separate sectors, and rasters whose width is no multiple of 16 went
// pixel by pixel.  Measured, us: 1501 x 1103 with counts, classes and colours
// 16.2 -> 6.4; 1856 x 2208 with a histogram 16.0 -> 12.7, means 19.0 -> 10;
// the engine's 64 uneven planes (23 M pixels) 93 -> 41, at 7 bytes a
// pixel 3.9 TB/s.
#pragma once

#include "class_histogram.cuh"
#include "device_common.cuh"
#include "overlap_class.cuh"

namespace cpt {

constexpr int kUnits = 4;                  // units of a lane per warp item
constexpr int kItemPixels = 32 * kUnits * 4;

// Where the counts of output pixels come from.  The outputs are dense, the
// plane's rows are padded to 16 pixels.
enum PlaneRows {
    kRowsDense = 0,    // pitch == width: pixel i of the outputs is element i of the plane
    kRowsOfFours = 1,  // width a multiple of 4: a unit lies in one row
    kRowsRagged = 2    // any width
};

__host__ __device__ inline int plane_rows(int64_t pitch, int32_t width) {
    return pitch == width ? kRowsDense : width % 4 == 0 ? kRowsOfFours : kRowsRagged;
}

// A unit's four elements as they lie in memory: two 16-bit counts to a register.
template <typename T>
struct Unit {
    T v[4];
    __device__ __forceinline__ void load(const T *at) { *this = *reinterpret_cast<const Unit *>(at); }
    __device__ __forceinline__ void store(T *at) const { *reinterpret_cast<Unit *>(at) = *this; }
    __device__ __forceinline__ T get(int j) const { return v[j]; }
    __device__ __forceinline__ void set(int j, T x) { v[j] = x; }
    __device__ __forceinline__ void clear() { v[0] = v[1] = v[2] = v[3] = (T)0; }
};
template <>
struct Unit<uint16_t> {
    uint2 w;
    __device__ __forceinline__ void load(const uint16_t *at) { w = *reinterpret_cast<const uint2 *>(at); }
    __device__ __forceinline__ void store(uint16_t *at) const { *reinterpret_cast<uint2 *>(at) = w; }
    __device__ __forceinline__ uint32_t get(int j) const {
        const uint32_t x = j < 2 ? w.x : w.y;
        return j & 1 ? x >> 16 : x & 0xFFFFu;
    }
    __device__ __forceinline__ void set(int j, uint32_t x) { (j < 2 ? w.x : w.y) |= x << (16 * (j & 1)); }   // after clear
    __device__ __forceinline__ void clear() { w = make_uint2(0u, 0u); }
};
template <>
__device__ __forceinline__ void Unit<uint32_t>::load(const uint32_t *at) {
    const uint4 x = *reinterpret_cast<const uint4 *>(at);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
}
template <>
__device__ __forceinline__ void Unit<uint32_t>::store(uint32_t *at) const {
    *reinterpret_cast<uint4 *>(at) = make_uint4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ void Unit<float>::load(const float *at) {
    const float4 x = *reinterpret_cast<const float4 *>(at);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
}
template <>
__device__ __forceinline__ void Unit<float>::store(float *at) const {
    *reinterpret_cast<float4 *>(at) = make_float4(v[0], v[1], v[2], v[3]);
}

// The elements of output pixels i .. i+3, i a multiple of 4; zero from the
// `left`th on.
template <typename T, int kRows>
__device__ __forceinline__ void load_unit(const T *plane, int64_t pitch, int32_t width, int64_t i, int left, Unit<T> &u) {
    if constexpr (kRows == kRowsDense) {
        u.load(plane + i);
    } else {
        const int64_t y = i <= 0xFFFFFFFFll ? (int64_t)((uint32_t)i / (uint32_t)width) : i / width;
        int x = (int)(i - y * width);
        const T *row = plane + y * pitch;
        if constexpr (kRows == kRowsOfFours) {
            u.load(row + x);
        } else {
            u.clear();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j < left) u.set(j, row[x]);
                if (++x == width) {
                    x = 0;
                    row += pitch;
                }
            }
        }
    }
}

// Stores one unit's outputs (each may be NULL) and counts its classes b into
// the lane's histogram row, if it has one.  `left`: pixels from i to the last
// (of the item).
// vec: every output is aligned to four of its elements.
template <typename CountT>
__device__ __forceinline__ void store_unit(const Unit<CountT> &c, const uint32_t (&b)[4], int64_t i, int left, bool vec,
                                           CountT *counts_out, uint8_t *bucket_out, uint32_t *rgba_out,
                                           const uint32_t *table, uint8_t *row, uint32_t key) {
    if (vec && left >= 4) {
        if (counts_out) c.store(counts_out + i);
        if (bucket_out) *reinterpret_cast<uint32_t *>(bucket_out + i) = b[0] | (b[1] << 8) | (b[2] << 16) | (b[3] << 24);
        if (rgba_out)
            *reinterpret_cast<uint4 *>(rgba_out + i) = make_uint4(table[b[0]], table[b[1]], table[b[2]], table[b[3]]);
        if (row) hist_count_quarter(row, key, b[0], b[1], b[2], b[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= left) break;
            if (counts_out) counts_out[i + j] = (CountT)c.get(j);
            if (bucket_out) bucket_out[i + j] = (uint8_t)b[j];
            if (rgba_out) rgba_out[i + j] = table[b[j]];
            if (row) hist_add(row, key, b[j], 1u);
        }
    }
}

}  // namespace cpt
