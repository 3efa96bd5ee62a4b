// engine.cu -- the batched composite engine of include/composite_engine.h.
//
// A submit turns every op (add/remove a member set to one plane) into work
// items (op, member slab, steps of 16-pixel groups), numbered op after op,
// slab after slab, chunk after chunk.  One persistent launch of
// num_SMs x ctas_per_sm CTAs claims item numbers from a device counter; the
// op owning an item is found by binary search over the ops' first items.  A
// CTA folds its groups of one slab's members into packed byte counters
// (member i of the op read at base + idx(i) * stride, the slab's indices
// staged in shared memory) and adds the counts into the op's plane (uint32,
// or uint16 for a 16-bit plane): with L2 atomics, or with plain
// read-modify-writes when the plane's ops are single slabs folded one after
// another by the same items (split_ops).  The render launch deals warp-level
// (plane, 512 pixels) items round robin to its warps.  Consecutive items are
// neighbouring chunks of the same slab, so concurrently running CTAs read
// neighbouring bytes of the same members.
#include <algorithm>
#include <chrono>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include "composite_engine.h"
#include "bit_count.cuh"
#include "internal.cuh"
#include "mask_load.cuh"
#include "render_units.cuh"

namespace {

using cpt::DeviceCaps;
using cpt::Lut;

constexpr int kThreads = 256;          // threads per CTA = 16-pixel groups per tile
constexpr int kMaxPlanes = 1 << 16;
constexpr int kMaxSlab = 255;          // packed byte counters
constexpr int kUploadRing = 64;        // descriptor uploads in flight before the host waits
constexpr int kSplitMembers = 32;      // shortest slab that a launch short of items is cut into
constexpr int kSlices = 4;             // slices of a CTA's threads on items of kSliceMembers members or more
constexpr int kSliceMembers = 32;
constexpr int kResidentCtas = 4;       // CTAs per SM that the accumulate kernels' registers allow
// A launch of bit-packed ops that are mostly of several slabs, whose counts go
// into the plane by atomics, waits for those: five CTAs per SM (on 48 registers)
// hide more of them.  us, four / five: one plane of 4000 x 3000 x 600, 16-bit
// counts 708 / 584, 32-bit 728 / 606; single slabs are better off with four:
// eight planes of 1024^2 x 128, 32-bit 90 / 125.
constexpr int kDeepBitsCtas = 5;

struct OpDesc {
    const uint8_t *base;
    const int32_t *index;
    uint32_t *plane;
    int64_t stride;
    int64_t plane_pitch;   // elements
    int64_t item_start;
    int32_t pitch;
    int32_t n;
    int32_t width;
    int32_t height;
    int32_t groups_per_row;
    int32_t tiles;
    int32_t slab;
    int32_t sign;
    int32_t plane_id;
    int32_t steps;               // steps per item: each kThreads / slices groups (or words)
    int32_t slices;              // shares of a slab's members that the CTA's threads fold at once: 1 or 4
    int32_t exclusive;           // this chain is the only one on its plane, one slab: plain read-modify-write
    int32_t bits;                // bit-packed masks: a group is a 32-pixel word
    int32_t words_per_row;       // bits: ceil(width / 32)
    int32_t u16;                 // the plane holds uint16 counts (else uint32)
    int32_t chain;               // ops folded by this op's items: itself and the chain - 1 that follow it
};

// One render op: its output pixels in items of 512 (render_units.cuh).
struct RenderDesc {
    const void *plane;
    void *counts_out;
    uint8_t *bucket_out;
    uint32_t *rgba_out;
    int64_t item_start;
    int64_t pitch;         // of the plane, elements
    int64_t pixels;
    int32_t width;
    int32_t rows;          // cpt::PlaneRows
    int32_t vec;           // outputs aligned to four of their elements
    int32_t u16;           // the plane holds uint16 counts (else uint32)
    cpt::ClassDivisor div; // floor(255 c / n_members) by multiplication
    unsigned long long *hist;   // 256 class counts, zeroed before the launch, or NULL
};

// One plane of a batched clear: its bytes as 16-byte words, in items of
// 32 lanes x kClearWords words.
struct ClearDesc {
    uint4 *data;
    int64_t words;
    int64_t item_start;
    int32_t plane_id;
    int32_t pad;
};

constexpr int kSmemStarts = 2048;      // ops whose first items fit in shared memory
constexpr int kClearWords = 8;         // 16-byte words per lane per clear item
constexpr int kClearCtasPerSm = 4;
constexpr int kRenderCtasPerSm = 4;    // render launch: CTAs per SM, grid-stride over items
constexpr int kRenderHistCtasPerSm = 4;   // with histograms: 32 KB of counters per CTA

template <typename Desc>
__device__ __forceinline__ int find_desc(const Desc *d, int n, int64_t item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (d[mid].item_start <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The op owning `item`: binary search over the first items, in shared memory
// when the op list is short enough, else over the descriptors themselves.
template <typename Desc>
__device__ __forceinline__ int find_op(const Desc *d, int n, const uint32_t *starts, uint32_t item) {
    if (n > kSmemStarts) return find_desc(d, n, item);
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// First item of op i (from shared memory when the list fits there).
template <typename Desc>
__device__ __forceinline__ uint32_t op_start(const Desc *d, int n, const uint32_t *starts, int i) {
    return n <= kSmemStarts ? starts[i] : (uint32_t)d[i].item_start;
}

template <typename Desc>
__device__ __forceinline__ void load_starts(const Desc *d, int n, uint32_t *starts) {
    if (n <= kSmemStarts)
        for (int i = threadIdx.x; i < n; i += blockDim.x) starts[i] = (uint32_t)d[i].item_start;
}

// Adds the masks of `cnt` members at one 16-pixel group into the packed byte
// counters k.  `row` is the group's address in member 0 of the op, m0 the
// slab's first member; with an index list the slab's ids are in shared memory.
// Eight members' loads are in flight at a time, the last (< 8) of them too: a
// short slab costs one memory latency, where a remainder loop of single loads
// pays one for each of its members.  `exact`: the group's valid bytes when the
// rest of its 16 may lie past the caller's memory, else 0.  Bound by HBM: 64
// uneven requests (2.1 GB of masks, half of the widths ragged) take 0.53 ms
// with clear and render where ragged groups' byte loads made it 1.09 ms.
template <bool kGather>
__device__ __forceinline__ void fold_group(const uint8_t *row, int64_t stride, int m0, const int32_t *index, int cnt,
                                           int exact, uint32_t (&k)[4]) {
    if (exact != 0) {
#pragma unroll 4
        for (int i = 0; i < cnt; ++i)
            cpt::add_group(k, cpt::load_group_exact(row + (int64_t)(kGather ? index[i] : m0 + i) * stride, exact));
    } else if (!kGather) {
        cpt::fold_masks<true>(row, stride, m0, m0 + cnt, k);
    } else {
        int i = 0;
        for (; i + 8 <= cnt; i += 8) {
            uint4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __ldcs(reinterpret_cast<const uint4 *>(row + (int64_t)index[i + j] * stride));
#pragma unroll
            for (int j = 0; j < 8; ++j) cpt::add_group(k, v[j]);
        }
        if (i < cnt) {
            uint4 v[7];
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                v[j] = make_uint4(0u, 0u, 0u, 0u);
                if (i + j < cnt) v[j] = __ldcs(reinterpret_cast<const uint4 *>(row + (int64_t)index[i + j] * stride));
            }
#pragma unroll
            for (int j = 0; j < 7; ++j) cpt::add_group(k, v[j]);
        }
    }
}

// plane counts of a group (+|-)= the packed counters k
template <typename CountT>
__device__ __forceinline__ void apply_group(CountT *dst, const uint32_t (&k)[4], const OpDesc &op, int *flags) {
    uint32_t wide[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) wide[j] = 0;
    cpt::widen16(wide, k[0], k[1], k[2], k[3]);
    // the plane's pitch is a whole number of groups: all 16 counts are its own
    if (op.exclusive)
        cpt::apply_count_group<CountT>(dst, 16, wide, op.sign, flags + op.plane_id);
    else
        cpt::atomic_count_group<CountT>(dst, wide, op.sign, flags + op.plane_id);
}

// The same for one word of the packed counters, four pixels.
template <typename CountT>
__device__ __forceinline__ void apply_word(CountT *dst, uint32_t k, const OpDesc &op, int *flags) {
    if (op.exclusive)
        cpt::apply_count_word<CountT>(dst, k, op.sign, flags + op.plane_id);
    else
        cpt::atomic_count_word<CountT>(dst, k, op.sign, flags + op.plane_id);
}

// What a CTA shares while it works on an item: the slab's member ids, the
// slices' packed counters.
struct ItemShared {
    int32_t index[kMaxSlab + 1];
    uint4 part[kSlices][kThreads / kSlices];
};

// Row and first pixel of group (or word) g of rows of `per_row`.
__device__ __forceinline__ int row_of(int64_t g, int per_row) {
    return g <= 0xFFFFFFFFll ? (int)((uint32_t)g / (uint32_t)per_row) : (int)(g / per_row);
}

// The ids of op's slab from member m0 on into shared memory.
__device__ __forceinline__ void stage_index(const OpDesc &op, int m0, int cnt, int32_t *index) {
    for (int i = threadIdx.x; i < cnt; i += kThreads) index[i] = op.index[m0 + i];
    __syncthreads();
}

// One CTA item: (op, member slab, `steps` steps of groups), and after the
// op's own slab those of the ops chained to it (one slab each, the same plane
// and groups): each op in turn adds to or takes from the counts, by the same
// CTA alone.  With four slices a step is 64 groups whose members the slices
// share, their counters added up in shared memory four pixels to a thread;
// with one a thread folds its own group.
__device__ __forceinline__ void process_item(const OpDesc *head, uint32_t item, ItemShared &sh, int *flags) {
    const uint32_t local = item - (uint32_t)head->item_start;
    const int sl = (int)(local / (uint32_t)head->tiles);
    const int chunk = (int)(local - (uint32_t)sl * head->tiles);
    const int64_t groups = (int64_t)head->groups_per_row * head->height;
    const int slices = head->slices;
    const int span = kThreads / slices;
    const int lane_group = threadIdx.x % span, slice = threadIdx.x / span;
    const int64_t first = (int64_t)chunk * head->steps * span;
    const int64_t last = min(groups, first + (int64_t)head->steps * span);
    const int chain = head->chain;
    for (int link = 0; link < chain; ++link) {
        const OpDesc &op = head[link];
        const int m0 = sl * op.slab;
        const int cnt = min(op.n - m0, op.slab);
        const bool gather = op.index != nullptr;
        if (gather) stage_index(op, m0, cnt, sh.index);
        const int share = (cnt + slices - 1) / slices;
        const int i0 = min(cnt, slice * share);
        const int mine = min(cnt, i0 + share) - i0;
        for (int64_t base = first; base < last; base += span) {
            const int64_t g = base + lane_group;
            uint32_t k[4] = {0u, 0u, 0u, 0u};
            int64_t at = 0;
            if (g < last) {
                const int y = row_of(g, op.groups_per_row);
                const int x0 = (int)(g - (int64_t)y * op.groups_per_row) * 16;
                const int valid = min(16, op.width - x0);
                // rows are at least a whole number of groups apart, so only the last
                // row's right edge can end before its group does
                const int exact = valid < 16 && y == op.height - 1 ? valid : 0;
                const uint8_t *row = op.base + (int64_t)y * op.pitch + x0;
                if (gather)
                    fold_group<true>(row, op.stride, 0, sh.index + i0, mine, exact, k);
                else
                    fold_group<false>(row, op.stride, m0 + i0, nullptr, mine, exact, k);
                cpt::keep_valid(k, valid);
                at = (int64_t)y * op.plane_pitch + x0;
            }
            if (slices == 1) {
                if (g >= last) continue;
                if (op.u16)
                    apply_group<uint16_t>(reinterpret_cast<uint16_t *>(op.plane) + at, k, op, flags);
                else
                    apply_group<uint32_t>(op.plane + at, k, op, flags);
                continue;
            }
            sh.part[slice][lane_group] = make_uint4(k[0], k[1], k[2], k[3]);
            __syncthreads();
            const int64_t wg = base + threadIdx.x / 4;   // this thread's word of the step's 64 groups
            if (wg < last) {
                uint32_t sum = 0;
#pragma unroll
                for (int s = 0; s < kSlices; ++s) sum += reinterpret_cast<const uint32_t *>(sh.part[s])[threadIdx.x];
                const int y = row_of(wg, op.groups_per_row);
                const int64_t to = (int64_t)y * op.plane_pitch + (wg - (int64_t)y * op.groups_per_row) * 16 +
                                   (threadIdx.x % 4) * 4;
                if (op.u16)
                    apply_word<uint16_t>(reinterpret_cast<uint16_t *>(op.plane) + to, sum, op, flags);
                else
                    apply_word<uint32_t>(op.plane + to, sum, op, flags);
            }
            __syncthreads();
        }
        if (gather) __syncthreads();
    }
}

// A 32-pixel word of a bit row; `exact` (1..3) bytes of it when the rest may
// lie past the caller's memory, else 0.
__device__ __forceinline__ uint32_t load_word(const uint8_t *q, int exact) {
    if (exact == 0) return __ldcs(reinterpret_cast<const uint32_t *>(q));
    uint32_t v = 0;
    if (exact & 2) v = *reinterpret_cast<const uint16_t *>(q);
    if (exact & 1) v |= (uint32_t)q[exact & 2] << (8 * (exact & 2));
    return v;
}

// The same for bit-packed masks: a thread owns 32-pixel words and keeps their
// counts in carry-save accumulators (BitCounter), 16 members per step.  Bits
// past the raster's right edge are counted along and dropped from the
// bit-slices at the end.
__device__ __forceinline__ void process_bits_item(const OpDesc *head, uint32_t item, ItemShared &sh, int *flags) {
    const uint32_t local = item - (uint32_t)head->item_start;
    const int sl = (int)(local / (uint32_t)head->tiles);
    const int chunk = (int)(local - (uint32_t)sl * head->tiles);
    const int64_t words = (int64_t)head->words_per_row * head->height;
    const int64_t first = (int64_t)chunk * head->steps * kThreads;
    const int64_t last = min(words, first + (int64_t)head->steps * kThreads);
    const int chain = head->chain;
    const int32_t *index = sh.index;
    for (int link = 0; link < chain; ++link) {
        const OpDesc &op = head[link];
        const int m0 = sl * op.slab;
        const int cnt = min(op.n - m0, op.slab);
        const bool gather = op.index != nullptr;
        if (gather) stage_index(op, m0, cnt, sh.index);
        const int64_t stride = op.stride;
        for (int64_t g = first + threadIdx.x; g < last; g += kThreads) {
            const int y = row_of(g, op.words_per_row);
            const int gx = (int)(g - (int64_t)y * op.words_per_row);
            const int x0 = gx * 32;
            const int valid = min(32, op.width - x0);
            const int exact = valid <= 24 && y == op.height - 1 ? (valid + 7) / 8 : 0;
            const uint8_t *row = op.base + (int64_t)y * op.pitch + gx * 4;
            cpt::BitCounter acc;
            for (int i = 0; i < cnt; i += 16) {
                const int take = min(16, cnt - i);
                uint32_t w[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    w[k] = 0;
                    if (k < take) {
                        const int64_t mi = gather ? index[i + k] : (int64_t)(m0 + i + k);
                        w[k] = load_word(row + mi * stride, exact);
                    }
                }
                cpt::bitcount_add16(acc, w);
            }
            if (valid < 32) cpt::bitcount_keep(acc, (1u << valid) - 1u);
            const int64_t at = (int64_t)y * op.plane_pitch + x0;
            uint32_t pairs[16];
            cpt::bitcount_pairs(acc, pairs);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (valid <= 16 * h) break;   // a half word past the plane's pitch
                if (op.u16) {
                    uint16_t *dst = reinterpret_cast<uint16_t *>(op.plane) + at + 16 * h;
                    if (op.exclusive)
                        cpt::apply_pair_group<uint16_t>(dst, 16, pairs + 8 * h, op.sign, flags + op.plane_id);
                    else
                        cpt::atomic_pair_group<uint16_t>(dst, pairs + 8 * h, op.sign, flags + op.plane_id);
                } else {
                    uint32_t *dst = op.plane + at + 16 * h;
                    if (op.exclusive)
                        cpt::apply_pair_group<uint32_t>(dst, 16, pairs + 8 * h, op.sign, flags + op.plane_id);
                    else
                        cpt::atomic_pair_group<uint32_t>(dst, pairs + 8 * h, op.sign, flags + op.plane_id);
                }
            }
        }
        if (gather) __syncthreads();
    }
}

// The mask formats of a launch's ops.  Each has a kernel of its own: the bit
// counters' registers would otherwise be taken from the byte path, which had
// to spill.
enum Formats { kBytesOnly = 0, kBitsOnly = 1, kBothFormats = 2 };

template <int kFormats>
__device__ __forceinline__ void run_item(const OpDesc *head, uint32_t item, ItemShared &sh, int *flags) {
    if (kFormats == kBitsOnly || (kFormats == kBothFormats && head->bits))
        process_bits_item(head, item, sh, flags);
    else
        process_item(head, item, sh, flags);
}

// Persistent schedule: CTA b takes item b, then claims items from the counter
// (zero at launch) one ahead: thread 0 asks for the next while the CTA works
// on the current one, and uneven items balance across the GPU.
// At most four CTAs per SM are resident, on 64 registers: five on 48 spilled
// and were slower (64 uneven requests with clear and render: 421 against 400
// us).  Two or three of them leave room for a kernel on another stream.
template <int kFormats, int kCtas>
__global__ void __launch_bounds__(kThreads, kCtas)
engine_accumulate_kernel(const OpDesc *ops, int n_ops, uint32_t n_items, uint32_t *counter, int *flags) {
    __shared__ ItemShared sh;
    __shared__ uint32_t s_starts[kSmemStarts];
    __shared__ uint32_t s_item;
    load_starts(ops, n_ops, s_starts);
    __syncthreads();
    uint32_t item = blockIdx.x;
    while (item < n_items) {
        uint32_t next = 0;
        if (threadIdx.x == 0) next = gridDim.x + atomicAdd(counter, 1u);
        run_item<kFormats>(ops + find_op(ops, n_ops, s_starts, item), item, sh, flags);
        if (threadIdx.x == 0) s_item = next;
        __syncthreads();
        item = s_item;
        __syncthreads();
    }
}

// Grid schedule: a CTA per item; the hardware block scheduler balances them.
template <int kFormats, int kCtas>
__global__ void __launch_bounds__(kThreads, kCtas)
engine_accumulate_grid_kernel(const OpDesc *ops, int n_ops, int *flags) {
    __shared__ ItemShared sh;
    const uint32_t item = blockIdx.x;
    run_item<kFormats>(ops + find_desc(ops, n_ops, item), item, sh, flags);
}

// Clear of many planes in one launch (counts to zero, the planes' underflow
// flags too): warp-level items (plane, 32 x kClearWords words) dealt round
// robin.  A CUDA graph that clears its planes this way has one node for all
// of them instead of two memset nodes per plane, which run one after another.
__global__ void __launch_bounds__(kThreads)
engine_clear_kernel(const ClearDesc *ops, int n_ops, uint32_t n_items, int *flags) {
    __shared__ uint32_t s_starts[kSmemStarts];
    load_starts(ops, n_ops, s_starts);
    __syncthreads();
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < n_ops; i += blockDim.x)
            if (ops[i].plane_id >= 0) flags[ops[i].plane_id] = 0;   // -1: a histogram or a counter, no flag
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (kThreads / 32);
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t item = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); item < n_items; item += warps) {
        const ClearDesc op = ops[find_op(ops, n_ops, s_starts, item)];   // by value: the stores may alias
        const int64_t w0 = (int64_t)(item - (uint32_t)op.item_start) * (32 * kClearWords) + lane;
#pragma unroll
        for (int k = 0; k < kClearWords; ++k) {
            const int64_t wi = w0 + 32 * k;
            if (wi < op.words) op.data[wi] = zero;
        }
    }
}

// One warp item of a render op: every lane loads its units' counts, `between`
// runs while they are on their way, then the units are classified and stored.
// row: the lane's histogram counters, or NULL.  The row form and the class
// path (one multiply-high below 2^16 members, the general division above) are
// chosen per item, so that each keeps only its own values live.
template <typename CountT, bool kNarrow>
__device__ __forceinline__ void store_item(const RenderDesc &op, const cpt::Unit<CountT> (&c)[cpt::kUnits], int64_t base,
                                           int left, int lane, const uint32_t *table, uint8_t *row, uint32_t key) {
    CountT *counts_out = static_cast<CountT *>(op.counts_out);
#pragma unroll
    for (int k = 0; k < cpt::kUnits; ++k) {
        const int at = 4 * (32 * k + lane);
        if (at >= left) break;
        uint32_t b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            b[j] = kNarrow ? cpt::overlap_class_narrow(c[k].get(j), op.div) : cpt::overlap_class(c[k].get(j), op.div);
        cpt::store_unit(c[k], b, base + at, left - at, op.vec != 0, counts_out, op.bucket_out, op.rgba_out, table, row, key);
    }
}

template <typename CountT, int kRows>
__device__ __forceinline__ void load_item(const RenderDesc &op, int64_t base, int left, int lane,
                                          cpt::Unit<CountT> (&c)[cpt::kUnits]) {
    const CountT *plane = static_cast<const CountT *>(op.plane);
#pragma unroll
    for (int k = 0; k < cpt::kUnits; ++k) {
        const int at = 4 * (32 * k + lane);
        if (at < left) cpt::load_unit<CountT, kRows>(plane, op.pitch, op.width, base + at, left - at, c[k]);
    }
}

template <typename CountT, typename Between>
__device__ __forceinline__ void render_item(const RenderDesc &op, int64_t base, int lane, const uint32_t *table, uint8_t *row,
                                            uint32_t key, Between between) {
    const int left = (int)min(op.pixels - base, (int64_t)cpt::kItemPixels);
    cpt::Unit<CountT> c[cpt::kUnits];
    if (op.rows == cpt::kRowsDense)
        load_item<CountT, cpt::kRowsDense>(op, base, left, lane, c);
    else if (op.rows == cpt::kRowsOfFours)
        load_item<CountT, cpt::kRowsOfFours>(op, base, left, lane, c);
    else
        load_item<CountT, cpt::kRowsRagged>(op, base, left, lane, c);
    between();
    if (op.div.narrow)
        store_item<CountT, true>(op, c, base, left, lane, table, row, key);
    else
        store_item<CountT, false>(op, c, base, left, lane, table, row, key);
}

// A whole item of a flat op (is_flat), 16 consecutive pixels per lane: the
// classes alone are a byte a pixel, which a lane stores 16 at a time where units
// of four take a store and their checks each (4096^2 20.5 us, 16.4 this way).
template <bool kNarrow>
__device__ __forceinline__ void render_flat(const RenderDesc &op, const uint4 (&v)[2], uint8_t *out) {
    const uint32_t w[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
    uint32_t q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t c = j & 1 ? w[2 * k + j / 2] >> 16 : w[2 * k + j / 2] & 0xFFFFu;
            b[j] = kNarrow ? cpt::overlap_class_narrow(c, op.div) : cpt::overlap_class(c, op.div);
        }
        q[k] = b[0] | (b[1] << 8) | (b[2] << 16) | (b[3] << 24);
    }
    *reinterpret_cast<uint4 *>(out) = make_uint4(q[0], q[1], q[2], q[3]);
}

template <typename Between>
__device__ __forceinline__ void render_flat_item(const RenderDesc &op, int64_t base, int lane, Between between) {
    const int64_t at = base + 16 * lane;
    const uint4 *p = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(op.plane) + at);
    const uint4 v[2] = {p[0], p[1]};
    between();
    if (op.div.narrow)
        render_flat<true>(op, v, op.bucket_out + at);
    else
        render_flat<false>(op, v, op.bucket_out + at);
}

// Render: warp-level items (render op, 512 of its pixels) dealt round robin
// to every warp of the launch -- items are all the same size, so no counter is
// needed.  With histograms (kHist; 5 KB of dynamic shared memory per warp)
// every CTA takes one contiguous range of items instead, so that a warp's
// items span one or two ops and its totals go to global memory once or twice.
// kFlat: every op is flat.
template <bool kHist, bool kFlat>
__global__ void __launch_bounds__(kThreads, kHist ? kRenderHistCtasPerSm : kRenderCtasPerSm)
engine_render_kernel(const RenderDesc *__restrict__ ops, int n_ops, uint32_t n_items, Lut lut) {
    __shared__ uint32_t table[256];
    __shared__ uint32_t s_starts[kSmemStarts];
    extern __shared__ __align__(16) uint8_t s_hist[];
    const int lane = threadIdx.x & 31;
    uint8_t *cnt = s_hist + (kHist ? (threadIdx.x >> 5) * cpt::kHistWarpBytes : 0);
    uint8_t *row = cnt + (kHist ? (lane / cpt::kHistLanesPerRow) * 256 : 0);
    const uint32_t key = (uint32_t)(lane / cpt::kHistLanesPerRow) << 2;
    for (int i = threadIdx.x; i < 256; i += kThreads) table[i] = lut.rgba[i];
    if (kHist)
        for (int i = lane; i < cpt::kHistWarpBytes / 16; i += 32) reinterpret_cast<uint4 *>(cnt)[i] = make_uint4(0, 0, 0, 0);
    load_starts(ops, n_ops, s_starts);
    __syncthreads();
    unsigned long long *hist_at = nullptr;   // the histogram the warp's counts belong to
    uint32_t *tot = reinterpret_cast<uint32_t *>(cnt + cpt::kHistCounterBytes);
    int since_fold = 0;
    uint32_t first, last, stride;
    if (kHist) {
        const uint32_t per = (n_items + gridDim.x - 1) / gridDim.x;
        first = blockIdx.x * per + (threadIdx.x >> 5);
        last = min(n_items, (blockIdx.x + 1) * per);
        stride = kThreads / 32;
    } else {
        first = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
        last = n_items;
        stride = gridDim.x * (kThreads / 32);
    }
    // the op of the warp's current item: without histograms the next item's
    // op is looked up while the current item's counts are on their way; with
    // them (contiguous items, few op changes) only when an item passes the
    // current op's end
    int idx = first < last ? find_op(ops, n_ops, s_starts, first) : 0;
    uint32_t op_end = kHist && first < last && idx + 1 < n_ops ? op_start(ops, n_ops, s_starts, idx + 1) : n_items;
    for (uint32_t item = first; item < last; item += stride) {
        if (kHist && item >= op_end) {
            idx = find_op(ops, n_ops, s_starts, item);
            op_end = idx + 1 < n_ops ? op_start(ops, n_ops, s_starts, idx + 1) : n_items;
        }
        // restrict: the outputs are plain pointers, and without it every
        // store would force the descriptor's fields to be reloaded
        const RenderDesc &op = ops[idx];
        if (kHist) {
            if (op.hist != hist_at) {
                if (hist_at) {
                    cpt::hist_fold(cnt, tot, lane);
                    cpt::hist_emit(tot, hist_at, lane);
                }
                hist_at = op.hist;
                since_fold = 0;
            } else if (hist_at && since_fold == cpt::kHistFoldItems) {
                cpt::hist_fold(cnt, tot, lane);
                since_fold = 0;
            }
            ++since_fold;
        }
        const int64_t base = (int64_t)(item - (uint32_t)op.item_start) * cpt::kItemPixels;
        const uint32_t next = item + stride;
        int next_idx = idx;
        auto look_up = [&]() {
            if (!kHist && next < last && idx + 1 < n_ops && next >= op_start(ops, n_ops, s_starts, idx + 1))
                next_idx = find_op(ops, n_ops, s_starts, next);
        };
        uint8_t *count_into = kHist && hist_at ? row : nullptr;
        if (kFlat && op.pixels - base >= cpt::kItemPixels)
            render_flat_item(op, base, lane, look_up);
        else if (op.u16)
            render_item<uint16_t>(op, base, lane, table, count_into, key, look_up);
        else
            render_item<uint32_t>(op, base, lane, table, count_into, key, look_up);
        idx = next_idx;
    }
    if (kHist) {
        // the warps of a CTA mostly end on one plane: its totals then go out once
        // per CTA instead of once per warp (eight planes of 1024^2: 44 -> 26 us)
        __shared__ unsigned long long *s_at[kThreads / 32];
        if (hist_at) cpt::hist_fold(cnt, tot, lane);
        if (lane == 0) s_at[threadIdx.x >> 5] = hist_at;
        __syncthreads();
        unsigned long long *at = nullptr;
        bool one = true;
        for (int w = 0; w < kThreads / 32; ++w) {
            if (!s_at[w]) continue;   // no totals
            one = one && (!at || at == s_at[w]);
            at = s_at[w];
        }
        if (one) {
            if (at) cpt::hist_emit_block(s_hist, kThreads / 32, at);
        } else if (hist_at) {
            cpt::hist_emit(tot, hist_at, lane);
        }
    }
}

struct PlaneRec {
    int32_t width = 0, height = 0;
    int64_t pitch_px = 0;
    uint32_t *data = nullptr;    // uint16 counts when count_bits is 16
    int32_t count_bits = 32;
    int64_t n = 0;
    bool alive = false;
    bool poisoned = false;       // a submit failed after its launch may have begun
    int32_t listed = -1;         // split_ops: the plane's place in the list of the submit's planes

    size_t bytes() const { return (size_t)pitch_px * height * (count_bits / 8); }
    int64_t max_members() const { return count_bits == 16 ? 0xFFFFll : 0xFFFFFFFFll; }
};

// A device buffer of descriptors with its pinned host mirror.
struct Upload {
    void *d = nullptr;
    void *h = nullptr;
    size_t cap = 0;
    cudaEvent_t done = nullptr;      // the upload out of h finished (upload stream)
    cudaEvent_t consumed = nullptr;  // the launch that read d finished (engine stream)
    bool used = false;
};

// A staging buffer for ops on pinned host members.
struct StageSlot {
    uint8_t *d = nullptr;
    cudaEvent_t ready = nullptr;     // its upload finished (copy stream)
    cudaEvent_t consumed = nullptr;  // the launch that read it finished (engine stream)
    bool used = false;
};

constexpr int64_t kDefaultStageBytes = 256ll << 20;
constexpr int kDefaultItemMemberGroups = 512;

thread_local std::string g_engine_error;

}  // namespace

struct composite_engine {
    composite_engine_config cfg{};
    int device = 0;
    DeviceCaps caps{};
    cudaStream_t stream = nullptr;
    std::vector<PlaneRec> planes;
    int *d_flags = nullptr;
    int *h_flags = nullptr;
    Upload up_ops[kUploadRing], up_render[kUploadRing];
    int up_i = 0, rup_i = 0;
    cudaEvent_t done_ev = nullptr;
    Lut default_lut{};
    // captured graph
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t graph_exec = nullptr;
    void *graph_ops = nullptr;
    void *graph_rops = nullptr;
    void *graph_clears = nullptr;
    uint32_t *graph_counters = nullptr;
    std::vector<std::pair<int32_t, int64_t>> graph_n;   // plane -> N after a replay
    std::vector<int32_t> graph_planes;                  // every plane the graph touches
    cudaStream_t capture_stream = nullptr;              // private stream for graph capture
    // ops on pinned host members
    std::vector<StageSlot> stage;
    int64_t stage_bytes = 0;       // bytes per allocated staging buffer
    uint64_t stage_next = 0;
    cudaStream_t copy = nullptr;   // their uploads
    cudaEvent_t caller_ready = nullptr;
    std::string err;
};

namespace {

int efail(composite_engine *e, int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (e)
        e->err = buf;
    else
        g_engine_error = buf;
    return code;
}

int ecuda(composite_engine *e, cudaError_t err, const char *what) {
    return efail(e, err == cudaErrorMemoryAllocation ? CPT_ENOMEM : CPT_ECUDA, "%s: %s", what,
                 cudaGetErrorString(err));
}

#define ECK(e, call)                                      \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return ecuda(e, e_, #call); \
    } while (0)

int64_t etimeout(const composite_engine *e) { return e->cfg.wait_timeout_ms > 0 ? e->cfg.wait_timeout_ms : 10000; }

int ewait(composite_engine *e, cudaEvent_t ev) {
    const auto deadline = std::chrono::steady_clock::now() + std::chrono::milliseconds(etimeout(e));
    for (unsigned spin = 0;; ++spin) {
        const cudaError_t r = cudaEventQuery(ev);
        if (r == cudaSuccess) return CPT_OK;
        if (r != cudaErrorNotReady) return ecuda(e, r, "cudaEventQuery");
        if (std::chrono::steady_clock::now() > deadline)
            return efail(e, CPT_ETIMEOUT, "wait exceeded %lld ms", (long long)etimeout(e));
        if (spin < 200)
            std::this_thread::yield();
        else
            std::this_thread::sleep_for(std::chrono::microseconds(50));
    }
}

int drain(composite_engine *e) {
    ECK(e, cudaEventRecord(e->done_ev, e->stream));
    return ewait(e, e->done_ev);
}

Lut make_lut(const uint8_t *rgba) {
    Lut l;
    for (int b = 0; b < 256; ++b) {
        const uint32_t r = rgba ? rgba[4 * b] : 255u - b, g = rgba ? rgba[4 * b + 1] : 255u - b;
        const uint32_t bl = rgba ? rgba[4 * b + 2] : 255u, a = rgba ? rgba[4 * b + 3] : 255u;
        l.rgba[b] = r | (g << 8) | (bl << 16) | (a << 24);
    }
    return l;
}

// Bytes ahead of a submit's op descriptors: the item counter, zero.
constexpr size_t kCounterBytes = 16;

// Copies `bytes` of descriptors into the next slot of the upload ring
// and queues their upload, on the upload stream when the engine has one (so
// that small uploads follow the caller's own uploads in order instead of
// waiting behind them on a copy engine); returns the slot.  `head` zero bytes
// come first.  The caller records slot->consumed on the engine stream after the
// launch that reads it.
int upload(composite_engine *e, Upload *ring, int *idx, const void *src, size_t bytes, Upload **slot,
           cudaStream_t on = nullptr, size_t head = 0) {
    Upload &u = ring[*idx];
    *idx = (*idx + 1) % kUploadRing;
    bytes += head;
    if (u.used) {
        int rc = ewait(e, u.done);
        if (rc) return rc;
    }
    cudaStream_t us = on ? on : e->cfg.upload_stream ? static_cast<cudaStream_t>(e->cfg.upload_stream) : e->stream;
    if (u.cap < bytes) {
        if (u.d) cudaFree(u.d);
        if (u.h) cudaFreeHost(u.h);
        u.d = u.h = nullptr;
        u.cap = 0;
        const size_t cap = std::max<size_t>(bytes, 4096);
        ECK(e, cudaMalloc(&u.d, cap));
        ECK(e, cudaHostAlloc(&u.h, cap, cudaHostAllocDefault));
        u.cap = cap;
    }
    if (head) memset(u.h, 0, head);
    memcpy(static_cast<unsigned char *>(u.h) + head, src, bytes - head);
    if (us != e->stream && u.used) ECK(e, cudaStreamWaitEvent(us, u.consumed, 0));
    ECK(e, cudaMemcpyAsync(u.d, u.h, bytes, cudaMemcpyHostToDevice, us));
    ECK(e, cudaEventRecord(u.done, us));
    if (us != e->stream) ECK(e, cudaStreamWaitEvent(e->stream, u.done, 0));
    u.used = true;
    *slot = &u;
    return CPT_OK;
}

// Memory kind of an op's members as seen from `device`: 1 = pinned host,
// 0 = device (this device's, or managed), -1 = neither (pageable host, or
// another GPU's memory, which a kernel here cannot be assumed to reach).
int member_kind(const void *p, int device) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    if (a.type == cudaMemoryTypeManaged) return 0;
    if (a.type == cudaMemoryTypeDevice) return a.device == device ? 0 : -1;
    return a.type == cudaMemoryTypeHost ? 1 : -1;
}

// Whether a kernel on `device` may read or write p in place: this device's
// memory, managed memory, or pinned host memory mapped for the device.
bool device_reachable(const void *p, int device) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    if (a.type == cudaMemoryTypeDevice) return a.device == device;
    return a.type == cudaMemoryTypeHost && a.devicePointer != nullptr;
}

bool plane_ok(const composite_engine *e, int32_t p) {
    return p >= 0 && p < (int32_t)e->planes.size() && e->planes[p].alive;
}

// Cuts the ops into work items: their order, chains, slabs, tiles and first
// items; returns the number of items.
//
// Chains.  Short ops on one plane (a session's adds and removes) share their
// items: a lane folds one op after the other into its groups by plain
// read-modify-writes.  As separate ops they need an atomic for every count
// (or pair of 16-bit counts) of the plane, of which 32 lanes touch 32 sectors
// at a time.  A plane's ops chain when each is one slab, all have one mask
// format and they hold at most item_member_groups members together.
//
// Slices.  From kSliceMembers members on, a slab's members are shared by four
// slices of the CTA (see count_kernels.cu, where the split was measured).
//
// Parallelism.  A launch runs num_SMs x ctas_per_sm CTAs (at most four per
// SM).  Where its planes'
// groups alone do not give every CTA an item, chains and slabs of more than
// kSplitMembers members are cut into slabs of down to that many -- but not
// chains that both add and remove: folded in order, a member added and taken
// away in one submit never looks like an underflow.
// A thread's work on an item is at most item_member_groups (member, group)
// pairs, and less where the launch would otherwise have fewer than eight
// items per CTA.  Measured on eight sessions' adds and removes of about 26
// overflow rasters of 1024^2: 15 CTAs and 1.66 ms in items of 512 pairs; a
// whole served pass 2.88 ms with such items and atomics, 0.47 ms now.  Items
// of single warps (no slices) took 420 us for the 64 uneven requests' 2.0 GB
// of masks, items of CTAs take 350 (5.8 TB/s).
int64_t split_ops(composite_engine *e, std::vector<OpDesc> *descs) {
    const int64_t ctas = (int64_t)e->caps.num_sms * std::min(e->cfg.ctas_per_sm, kResidentCtas);
    const int cfg_slab = e->cfg.slab_members;
    auto slices_of = [](const OpDesc &d, int members) { return !d.bits && members >= kSliceMembers ? kSlices : 1; };
    auto steps_of = [](const OpDesc &d, int slices) {   // steps over the whole plane
        const int64_t span = kThreads / slices;
        return ((int64_t)(d.bits ? d.words_per_row : d.groups_per_row) * d.height + span - 1) / span;
    };
    struct PlaneOps {
        int64_t members = 0;
        int most = 0;           // members of its longest op
        int ops = 0;
        int32_t bits = -1;      // the ops' mask format, -2 when they differ
        bool single = true;     // every op is one slab
        bool adds = false, removes = false;
        bool chained = false;
        bool together = true;   // its ops follow one another in the list
        size_t last = 0;        // its last op in the list
    };
    // One entry per plane of the submit, not per plane of the engine: tables
    // over 60000 planes cost a submit of one small op 0.14 ms on the host.
    std::vector<PlaneOps> planes;
    planes.reserve(descs->size());
    for (const OpDesc &d : *descs) e->planes[d.plane_id].listed = -1;
    auto place = [e](const OpDesc &d) { return (size_t)e->planes[d.plane_id].listed; };
    int64_t steps_once = 0;      // steps of the planes' first ops
    int64_t thread_work = 0;     // (member, group) pairs per thread over all steps
    for (size_t i = 0; i < descs->size(); ++i) {
        const OpDesc &d = (*descs)[i];
        int32_t &listed = e->planes[d.plane_id].listed;
        if (listed < 0) {
            listed = (int32_t)planes.size();
            planes.emplace_back();
        }
        PlaneOps &p = planes[listed];
        p.together = p.together && (p.ops == 0 || p.last + 1 == i);
        p.last = i;
        if (p.ops++ == 0) {
            p.bits = d.bits;
            steps_once += steps_of(d, slices_of(d, d.n));
        } else if (p.bits != d.bits) {
            p.bits = -2;
        }
        p.members += d.n;
        p.single = p.single && d.n <= cfg_slab;
        (d.sign > 0 ? p.adds : p.removes) = true;
        p.most = std::max(p.most, d.n);
        thread_work += steps_of(d, 1) * d.n;
    }
    const bool fills = steps_once >= ctas;
    for (PlaneOps &p : planes)
        p.chained = p.ops > 0 && p.single && p.bits >= 0 && p.members <= std::max(cfg_slab, e->cfg.item_member_groups) &&
                    (fills || p.members <= kSplitMembers || (p.adds && p.removes));
    // a plane's chained ops one after another, at the place of its first
    bool in_order = true;
    for (const PlaneOps &p : planes) in_order = in_order && (p.together || !p.chained);
    if (!in_order) {
        constexpr size_t kNone = ~(size_t)0;
        std::vector<size_t> next(descs->size(), kNone);   // the op's successor in its chain
        std::vector<size_t> first(planes.size(), kNone), last(planes.size(), kNone);
        for (size_t i = 0; i < descs->size(); ++i) {
            const size_t at = place((*descs)[i]);
            if (first[at] == kNone)
                first[at] = i;
            else
                next[last[at]] = i;
            last[at] = i;
        }
        std::vector<OpDesc> order;
        order.reserve(descs->size());
        for (size_t i = 0; i < descs->size(); ++i) {
            const size_t at = place((*descs)[i]);
            if (!planes[at].chained)
                order.push_back((*descs)[i]);
            else if (first[at] == i)
                for (size_t j = i; j != kNone; j = next[j]) order.push_back((*descs)[j]);
        }
        descs->swap(order);
    }
    const int64_t target = std::min<int64_t>(e->cfg.item_member_groups, std::max<int64_t>(8, thread_work / (8 * ctas)));
    int64_t items = 0;
    for (size_t i = 0; i < descs->size();) {
        OpDesc &head = (*descs)[i];
        const PlaneOps &p = planes[place(head)];
        const int chain = p.chained ? p.ops : 1;
        int slab = cfg_slab;
        if (!p.chained && !fills && head.n > kSplitMembers) {
            const int64_t parts = (ctas + steps_once - 1) / steps_once;
            slab = (int)std::min<int64_t>(slab, std::max<int64_t>(kSplitMembers, (head.n + parts - 1) / parts));
        }
        head.slices = slices_of(head, p.chained ? p.most : std::min(head.n, slab));
        const int64_t per_thread = (p.chained ? p.members : std::min(head.n, slab)) / head.slices;
        const int64_t steps = steps_of(head, head.slices);
        head.steps = (int32_t)std::max<int64_t>(1, std::min<int64_t>(steps, target / std::max<int64_t>(1, per_thread)));
        head.tiles = (int32_t)((steps + head.steps - 1) / head.steps);
        head.slab = slab;
        head.chain = chain;
        head.exclusive = p.chained || (p.ops == 1 && head.n <= slab) ? 1 : 0;
        head.item_start = items;
        items += (int64_t)head.tiles * ((head.n + slab - 1) / slab);
        for (int link = 1; link < chain; ++link) {
            OpDesc &d = (*descs)[i + link];
            d.slab = slab;
            d.exclusive = 1;
            d.item_start = items;   // none of its own: the search for an item's op passes it by
        }
        i += chain;
    }
    return items;
}

// Validates ops and builds their descriptors.  n_after holds, per plane
// touched, the member count after the ops starting from `start` counts.
int plan_ops(composite_engine *e, const composite_op *ops, int32_t n_ops, std::vector<OpDesc> *descs,
             int64_t *n_items, std::vector<std::pair<int32_t, int64_t>> *n_after, bool from_zero,
             bool check_n = true) {
    if (n_ops < 0 || (n_ops > 0 && !ops)) return efail(e, CPT_EINVAL, "bad op list");
    descs->clear();
    n_after->clear();
    std::vector<int64_t> n(e->planes.size(), -1);
    for (int32_t i = 0; i < n_ops; ++i) {
        const composite_op &o = ops[i];
        if (!plane_ok(e, o.plane)) return efail(e, CPT_EINVAL, "op %d: no plane %d", i, o.plane);
        if (o.sign != 1 && o.sign != -1) return efail(e, CPT_EINVAL, "op %d: sign must be +1 or -1", i);
        if (o.n_members < 0) return efail(e, CPT_EINVAL, "op %d: n_members < 0", i);
        const PlaneRec &p = e->planes[o.plane];
        if (n[o.plane] < 0) n[o.plane] = from_zero ? 0 : p.n;
        n[o.plane] += (int64_t)o.sign * o.n_members;
        if (check_n && n[o.plane] < 0)
            return efail(e, CPT_EINVAL, "op %d: plane %d would hold fewer than 0 members", i, o.plane);
        if (check_n && n[o.plane] > p.max_members())
            return efail(e, CPT_EINVAL, "op %d: plane %d would exceed %lld members (%d-bit counts)", i, o.plane,
                         (long long)p.max_members(), p.count_bits);
        if (o.n_members == 0) continue;
        if (!o.members) return efail(e, CPT_EINVAL, "op %d: members is NULL", i);
        if ((reinterpret_cast<uintptr_t>(o.members) % 16) || (o.row_pitch_bytes % 16) || (o.member_stride_bytes % 16))
            return efail(e, CPT_EINVAL, "op %d: members, row pitch and stride must be 16-byte aligned", i);
        if (o.mask_format != CPT_MASK_BYTES && o.mask_format != CPT_MASK_BITS)
            return efail(e, CPT_EINVAL, "op %d: mask_format %d out of range", i, o.mask_format);
        const bool bits = o.mask_format == CPT_MASK_BITS;
        const int64_t row_bytes = bits ? ((int64_t)p.width + 7) / 8 : p.width;
        if (o.row_pitch_bytes < row_bytes || o.member_stride_bytes < (int64_t)o.row_pitch_bytes * p.height)
            return efail(e, CPT_EINVAL, "op %d: row pitch or member stride too small", i);
        OpDesc d{};
        d.base = static_cast<const uint8_t *>(o.members);
        d.index = o.member_index;
        d.plane = p.data;
        d.stride = o.member_stride_bytes;
        d.plane_pitch = p.pitch_px;
        d.pitch = o.row_pitch_bytes;
        d.n = o.n_members;
        d.width = p.width;
        d.height = p.height;
        d.groups_per_row = (int32_t)(p.pitch_px / 16);
        d.bits = bits ? 1 : 0;
        d.u16 = p.count_bits == 16 ? 1 : 0;
        d.words_per_row = (int32_t)(((int64_t)p.width + 31) / 32);
        d.sign = o.sign;
        d.plane_id = o.plane;
        d.chain = 1;
        descs->push_back(d);
    }
    const int64_t items = split_ops(e, descs);
    if (items >= (int64_t)1 << 31) return efail(e, CPT_EINVAL, "too many work items in one submit");
    for (size_t p = 0; p < n.size(); ++p)
        if (n[p] >= 0) n_after->push_back({(int32_t)p, n[p]});
    *n_items = items;
    return CPT_OK;
}

int plan_render(composite_engine *e, const composite_render_op *ops, int32_t n_ops, std::vector<RenderDesc> *descs,
                int64_t *n_items, const std::vector<std::pair<int32_t, int64_t>> *n_override) {
    if (n_ops < 0 || (n_ops > 0 && !ops)) return efail(e, CPT_EINVAL, "bad render list");
    descs->clear();
    int64_t items = 0;
    for (int32_t i = 0; i < n_ops; ++i) {
        const composite_render_op &o = ops[i];
        if (!plane_ok(e, o.plane)) return efail(e, CPT_EINVAL, "render %d: no plane %d", i, o.plane);
        const PlaneRec &p = e->planes[o.plane];
        if ((reinterpret_cast<uintptr_t>(o.counts_out) % (p.count_bits / 8)) || (reinterpret_cast<uintptr_t>(o.rgba_out) % 4))
            return efail(e, CPT_EINVAL, "render %d: counts_out must be aligned to its count type, rgba_out to 4 bytes", i);
        if (reinterpret_cast<uintptr_t>(o.histogram_out) % 16)
            return efail(e, CPT_EINVAL, "render %d: histogram_out must be 16-byte aligned", i);
        const void *outs[4] = {o.counts_out, o.bucket_out, o.rgba_out, o.histogram_out};
        for (const void *q : outs)
            if (q && !device_reachable(q, e->device))
                return efail(e, CPT_EINVAL, "render %d: outputs must be device memory of device %d (or mapped pinned "
                                            "host memory)", i, e->device);
        int64_t n = p.n;
        bool refolded = false;   // a captured graph clears and refolds the plane first
        if (n_override)
            for (const auto &pn : *n_override)
                if (pn.first == o.plane) {
                    n = pn.second;
                    refolded = true;
                }
        if (p.poisoned && !refolded)
            return efail(e, CPT_ESTATE, "render %d: plane %d: an earlier submit failed part-way; clear it", i, o.plane);
        RenderDesc d{};
        d.plane = p.data;
        d.counts_out = o.counts_out;
        d.bucket_out = o.bucket_out;
        d.rgba_out = reinterpret_cast<uint32_t *>(o.rgba_out);
        d.item_start = items;
        d.div = cpt::class_divisor((uint64_t)n);
        d.pitch = p.pitch_px;
        d.pixels = (int64_t)p.width * p.height;
        d.width = p.width;
        d.rows = cpt::plane_rows(p.pitch_px, p.width);
        d.vec = reinterpret_cast<uintptr_t>(o.counts_out) % (4 * (p.count_bits / 8)) == 0 &&
                reinterpret_cast<uintptr_t>(o.bucket_out) % 4 == 0 && reinterpret_cast<uintptr_t>(o.rgba_out) % 16 == 0;
        d.u16 = p.count_bits == 16 ? 1 : 0;
        d.hist = reinterpret_cast<unsigned long long *>(o.histogram_out);
        const int64_t tiles = (d.pixels + cpt::kItemPixels - 1) / cpt::kItemPixels;
        items += tiles;
        descs->push_back(d);
    }
    if (items >= (int64_t)1 << 31) return efail(e, CPT_EINVAL, "too many render items");
    *n_items = items;
    return CPT_OK;
}

unsigned persistent_grid(const composite_engine *e, int64_t items, int resident) {
    const int64_t cap = (int64_t)e->caps.num_sms * std::min(e->cfg.ctas_per_sm, resident);
    return (unsigned)std::max<int64_t>(1, std::min(cap, items));
}

template <int kFormats, int kCtas = kResidentCtas>
void launch_accumulate_t(composite_engine *e, const OpDesc *ops, int n_ops, int64_t n_items, uint32_t *counter) {
    const unsigned grid = persistent_grid(e, n_items, kCtas);
    const uint32_t items = (uint32_t)n_items;
    if (e->cfg.schedule == CPT_SCHEDULE_GRID)
        engine_accumulate_grid_kernel<kFormats, kCtas><<<items, kThreads, 0, e->stream>>>(ops, n_ops, e->d_flags);
    else
        engine_accumulate_kernel<kFormats, kCtas><<<grid, kThreads, 0, e->stream>>>(ops, n_ops, items, counter, e->d_flags);
}

// counter: a zeroed device word (persistent schedule).
int launch_accumulate(composite_engine *e, const void *d_ops, const std::vector<OpDesc> &descs, int64_t n_items,
                      uint32_t *counter) {
    bool bytes = false, bits = false;
    int64_t work = 0, deep = 0;   // (member, word) pairs of the bit ops, and of those in several slabs
    for (const OpDesc &d : descs) {
        (d.bits ? bits : bytes) = true;
        const int64_t pairs = (int64_t)d.n * d.words_per_row * d.height;
        work += pairs;
        if (d.n > d.slab) deep += pairs;
    }
    const OpDesc *ops = static_cast<const OpDesc *>(d_ops);
    const int n_ops = (int)descs.size();
    if (!bits)
        launch_accumulate_t<kBytesOnly>(e, ops, n_ops, n_items, counter);
    else if (!bytes && e->cfg.ctas_per_sm >= kDeepBitsCtas && 2 * deep > work)
        launch_accumulate_t<kBitsOnly, kDeepBitsCtas>(e, ops, n_ops, n_items, counter);
    else if (!bytes)
        launch_accumulate_t<kBitsOnly>(e, ops, n_ops, n_items, counter);
    else
        launch_accumulate_t<kBothFormats>(e, ops, n_ops, n_items, counter);
    ECK(e, cudaGetLastError());
    return CPT_OK;
}

int launch_uploaded(composite_engine *e, const std::vector<OpDesc> &descs, int64_t items, void *blob) {
    return launch_accumulate(e, static_cast<unsigned char *>(blob) + kCounterBytes, descs, items,
                             static_cast<uint32_t *>(blob));
}

// True when some render op asks for a class histogram.
bool any_histogram(const std::vector<RenderDesc> &descs) {
    for (const RenderDesc &d : descs)
        if (d.hist) return true;
    return false;
}

// Whether a render op asks for the classes alone, from a dense plane of 16-bit
// counts and to a 16-byte aligned output.
bool is_flat(const RenderDesc &d) {
    return d.u16 && d.rows == cpt::kRowsDense && d.bucket_out && !d.counts_out && !d.rgba_out && !d.hist &&
           reinterpret_cast<uintptr_t>(d.bucket_out) % 16 == 0;
}

// Clear entries (plane_id -1, no flag) for the histograms of a render, each
// 256 x uint64 = 128 16-byte words, one clear item.
void plan_histogram_clears(const std::vector<RenderDesc> &rdescs, std::vector<ClearDesc> *cdescs, int64_t *citems) {
    for (const RenderDesc &r : rdescs) {
        if (!r.hist) continue;
        ClearDesc d{};
        d.data = reinterpret_cast<uint4 *>(r.hist);
        d.words = 256 * sizeof(uint64_t) / 16;
        d.item_start = *citems;
        d.plane_id = -1;
        *citems += (d.words + 32 * kClearWords - 1) / (32 * kClearWords);
        cdescs->push_back(d);
    }
}

constexpr int kRenderHistSmem = (kThreads / 32) * cpt::kHistWarpBytes;   // dynamic: the warps' counters

// The histogram render's dynamic shared memory (40 KB, beside 9 KB static):
// allowed explicitly, and the largest carveout asked for, so that four such
// CTAs fit on an SM.
int prepare_render_kernels(composite_engine *e) {
    ECK(e, cudaFuncSetAttribute(engine_render_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kRenderHistSmem));
    ECK(e, cudaFuncSetAttribute(engine_render_kernel<true, false>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared));
    return CPT_OK;
}

int launch_render(composite_engine *e, const void *d_ops, const std::vector<RenderDesc> &descs, int64_t n_items,
                  const Lut &lut) {
    const int n_ops = (int)descs.size();
    const bool hist = any_histogram(descs);
    bool flat = true;
    for (const RenderDesc &d : descs) flat = flat && is_flat(d);
    const int64_t ctas = std::min<int64_t>((int64_t)e->caps.num_sms * (hist ? kRenderHistCtasPerSm : kRenderCtasPerSm),
                                           (n_items + kThreads / 32 - 1) / (kThreads / 32));
    const unsigned grid = (unsigned)std::max<int64_t>(1, ctas);
    if (hist)
        engine_render_kernel<true, false><<<grid, kThreads, kRenderHistSmem, e->stream>>>(
            static_cast<const RenderDesc *>(d_ops), n_ops, (uint32_t)n_items, lut);
    else if (flat)
        engine_render_kernel<false, true><<<grid, kThreads, 0, e->stream>>>(static_cast<const RenderDesc *>(d_ops), n_ops,
                                                                             (uint32_t)n_items, lut);
    else
        engine_render_kernel<false, false><<<grid, kThreads, 0, e->stream>>>(static_cast<const RenderDesc *>(d_ops), n_ops,
                                                                              (uint32_t)n_items, lut);
    ECK(e, cudaGetLastError());
    return CPT_OK;
}

int clear_plane(composite_engine *e, int32_t p) {
    PlaneRec &r = e->planes[p];
    ECK(e, cudaMemsetAsync(r.data, 0, r.bytes(), e->stream));
    ECK(e, cudaMemsetAsync(e->d_flags + p, 0, sizeof(int), e->stream));
    r.n = 0;
    r.poisoned = false;
    return CPT_OK;
}

// Descriptors of one clear launch over the listed planes (each once).
int plan_clears(composite_engine *e, const int32_t *planes, int32_t n, std::vector<ClearDesc> *descs,
                int64_t *n_items) {
    if (n < 0 || (n > 0 && !planes)) return efail(e, CPT_EINVAL, "bad plane list");
    descs->clear();
    std::vector<char> seen(e->planes.size(), 0);
    int64_t items = 0;
    for (int32_t i = 0; i < n; ++i) {
        const int32_t p = planes[i];
        if (!plane_ok(e, p)) return efail(e, CPT_EINVAL, "clear %d: no plane %d", i, p);
        if (seen[p]) continue;
        seen[p] = 1;
        const PlaneRec &r = e->planes[p];
        ClearDesc d{};
        d.data = reinterpret_cast<uint4 *>(r.data);
        d.words = (int64_t)(r.bytes() / 16);   // plane rows are whole 16-pixel groups
        d.item_start = items;
        d.plane_id = p;
        items += (d.words + 32 * kClearWords - 1) / (32 * kClearWords);
        descs->push_back(d);
    }
    if (items >= (int64_t)1 << 31) return efail(e, CPT_EINVAL, "too many clear items");
    *n_items = items;
    return CPT_OK;
}

int launch_clear(composite_engine *e, const void *d_ops, int n_ops, int64_t n_items) {
    const int64_t ctas = std::min<int64_t>((int64_t)e->caps.num_sms * kClearCtasPerSm,
                                           (n_items + kThreads / 32 - 1) / (kThreads / 32));
    engine_clear_kernel<<<(unsigned)std::max<int64_t>(1, ctas), kThreads, 0, e->stream>>>(
        static_cast<const ClearDesc *>(d_ops), n_ops, (uint32_t)n_items, e->d_flags);
    ECK(e, cudaGetLastError());
    return CPT_OK;
}

// Clears the listed planes in one launch (their counts, N and underflow and
// failure marks).
int clear_many(composite_engine *e, const int32_t *planes, int32_t n) {
    std::vector<ClearDesc> descs;
    int64_t items = 0;
    int rc = plan_clears(e, planes, n, &descs, &items);
    if (rc || descs.empty()) return rc;
    Upload *u = nullptr;
    rc = upload(e, e->up_render, &e->rup_i, descs.data(), descs.size() * sizeof(ClearDesc), &u);
    if (rc) return rc;
    rc = launch_clear(e, u->d, (int)descs.size(), items);
    if (rc) return rc;
    ECK(e, cudaEventRecord(u->consumed, e->stream));
    for (const ClearDesc &d : descs) {
        e->planes[d.plane_id].n = 0;
        e->planes[d.plane_id].poisoned = false;
    }
    return CPT_OK;
}

void free_stage(composite_engine *e) {
    for (StageSlot &s : e->stage) {
        if (s.d) cudaFree(s.d);
        if (s.ready) cudaEventDestroy(s.ready);
        if (s.consumed) cudaEventDestroy(s.consumed);
    }
    e->stage.clear();
    e->stage_bytes = 0;
    e->stage_next = 0;
}

// Staging buffers of the configured count and size, allocated at the first
// host op and again whenever the configuration changed (after the engine's
// queued work, which may still read the old ones).
int ensure_stage(composite_engine *e) {
    const int k = e->cfg.staging_buffers;
    const int64_t bytes = e->cfg.staging_bytes;
    if ((int)e->stage.size() == k && e->stage_bytes == bytes) return CPT_OK;
    int rc = drain(e);
    if (rc) return rc;
    free_stage(e);
    if (!e->copy) ECK(e, cudaStreamCreateWithFlags(&e->copy, cudaStreamNonBlocking));
    if (!e->caller_ready) ECK(e, cudaEventCreateWithFlags(&e->caller_ready, cudaEventDisableTiming));
    e->stage.resize(k);
    for (StageSlot &s : e->stage) {
        cudaError_t err = cudaMalloc(&s.d, (size_t)bytes);
        if (err == cudaSuccess) err = cudaEventCreateWithFlags(&s.ready, cudaEventDisableTiming);
        if (err == cudaSuccess) err = cudaEventCreateWithFlags(&s.consumed, cudaEventDisableTiming);
        if (err != cudaSuccess) {
            free_stage(e);
            return ecuda(e, err, "staging buffer allocation");
        }
    }
    e->stage_bytes = bytes;
    return CPT_OK;
}

// Launches the accumulate kernel over ops (already validated as a whole).
// desc_stream: where the descriptors are uploaded (NULL = the usual upload
// stream); the launch waits for them either way.
int launch_ops(composite_engine *e, const composite_op *ops, int32_t n_ops, bool *launched,
               cudaStream_t desc_stream = nullptr) {
    std::vector<OpDesc> descs;
    std::vector<std::pair<int32_t, int64_t>> n_after;
    int64_t items = 0;
    int rc = plan_ops(e, ops, n_ops, &descs, &items, &n_after, false, false);
    if (rc || items == 0) return rc;
    Upload *u = nullptr;
    rc = upload(e, e->up_ops, &e->up_i, descs.data(), descs.size() * sizeof(OpDesc), &u, desc_stream, kCounterBytes);
    if (rc) return rc;
    if (cpt::fault_injected("engine_submit")) return efail(e, CPT_ECUDA, "submit refused before its launch (injected)");
    *launched = true;   // from here on the launch may have begun
    rc = launch_uploaded(e, descs, items, u->d);
    if (rc) return rc;
    ECK(e, cudaEventRecord(u->consumed, e->stream));
    return CPT_OK;
}

// Ops on pinned host members: their rasters are packed, op after op, into
// staging buffers of stage_bytes; a full buffer is uploaded on the copy
// stream (after the launch that last read it) and folded by one accumulate
// launch on the engine stream (after the upload), so the upload of one
// buffer overlaps the fold of the previous one.
int stream_host_ops(composite_engine *e, const std::vector<composite_op> &hops, bool *launched) {
    int rc = ensure_stage(e);
    if (rc) return rc;
    // uploads start after the caller's earlier work on the engine stream
    ECK(e, cudaEventRecord(e->caller_ready, e->stream));
    ECK(e, cudaStreamWaitEvent(e->copy, e->caller_ready, 0));
    struct Run {
        size_t op;
        int32_t m0, cnt;
        int64_t offset;
    };
    std::vector<Run> runs;
    int64_t used = 0;
    int64_t chunk = 0;
    const int64_t inject_at = cpt::fault_injected_value("engine_chunk_fail");
    auto flush = [&]() -> int {
        if (runs.empty()) return CPT_OK;
        if (inject_at == chunk) return efail(e, CPT_ECUDA, "upload of staging chunk %lld refused (injected)", (long long)chunk);
        ++chunk;
        StageSlot &slot = e->stage[e->stage_next++ % e->stage.size()];
        if (slot.used) ECK(e, cudaStreamWaitEvent(e->copy, slot.consumed, 0));
        std::vector<composite_op> cops;
        cops.reserve(runs.size());
        for (const Run &r : runs) {
            const composite_op &o = hops[r.op];
            const int64_t rb = (int64_t)o.row_pitch_bytes * e->planes[o.plane].height;
            const uint8_t *src = static_cast<const uint8_t *>(o.members) + (int64_t)r.m0 * o.member_stride_bytes;
            if (o.member_stride_bytes == rb)
                ECK(e, cudaMemcpyAsync(slot.d + r.offset, src, (size_t)(r.cnt * rb), cudaMemcpyHostToDevice, e->copy));
            else
                ECK(e, cudaMemcpy2DAsync(slot.d + r.offset, (size_t)rb, src, (size_t)o.member_stride_bytes, (size_t)rb,
                                         (size_t)r.cnt, cudaMemcpyHostToDevice, e->copy));
            composite_op c = o;
            c.members = slot.d + r.offset;
            c.member_index = nullptr;
            c.n_members = r.cnt;
            c.member_stride_bytes = rb;
            cops.push_back(c);
        }
        ECK(e, cudaEventRecord(slot.ready, e->copy));
        ECK(e, cudaStreamWaitEvent(e->stream, slot.ready, 0));
        // the chunk's descriptors follow its rasters on the copy stream: on the
        // engine stream they would queue on a copy engine behind the next
        // chunk's rasters, and the fold would wait one upload longer
        int r = launch_ops(e, cops.data(), (int32_t)cops.size(), launched, e->copy);
        if (r) return r;
        ECK(e, cudaEventRecord(slot.consumed, e->stream));
        slot.used = true;
        runs.clear();
        used = 0;
        return CPT_OK;
    };
    for (size_t i = 0; i < hops.size(); ++i) {
        const composite_op &o = hops[i];
        const int64_t rb = (int64_t)o.row_pitch_bytes * e->planes[o.plane].height;
        for (int32_t m = 0; m < o.n_members;) {
            const int64_t fit = (e->stage_bytes - used) / rb;
            if (fit <= 0) {
                if ((rc = flush())) return rc;
                continue;
            }
            const int32_t take = (int32_t)std::min<int64_t>(fit, o.n_members - m);
            runs.push_back({i, m, take, used});
            used += take * rb;
            m += take;
        }
    }
    return flush();
}

int submit_internal(composite_engine *e, const composite_op *ops, int32_t n_ops) {
    const cpt::TraceRange range("composite_engine_submit");
    std::vector<OpDesc> descs;
    std::vector<std::pair<int32_t, int64_t>> n_after;
    int64_t items = 0;
    int rc = plan_ops(e, ops, n_ops, &descs, &items, &n_after, false);
    if (rc) return rc;
    for (const auto &pn : n_after)
        if (e->planes[pn.first].poisoned)
            return efail(e, CPT_ESTATE, "plane %d: an earlier submit failed part-way; clear it", pn.first);
    // device ops fold in one launch; ops on pinned host members stream
    std::vector<composite_op> dev_ops, host_ops;
    for (int32_t i = 0; i < n_ops; ++i) {
        const composite_op &o = ops[i];
        if (o.n_members == 0) continue;
        const int kind = member_kind(o.members, e->device);
        if (kind < 0)
            return efail(e, CPT_EINVAL, "op %d: members must be device memory of device %d or pinned host memory", i,
                         e->device);
        if (kind == 0) {
            if (o.member_index && !device_reachable(o.member_index, e->device))
                return efail(e, CPT_EINVAL, "op %d: member_index must be device memory of device %d", i, e->device);
            dev_ops.push_back(o);
            continue;
        }
        if (o.member_index) return efail(e, CPT_EINVAL, "op %d: an index list needs device members", i);
        if ((int64_t)o.row_pitch_bytes * e->planes[o.plane].height > e->cfg.staging_bytes)
            return efail(e, CPT_EINVAL, "op %d: a raster is larger than staging_bytes", i);
        host_ops.push_back(o);
    }
    bool launched = false;
    if (host_ops.empty()) {
        if (items > 0) {
            Upload *u = nullptr;
            rc = upload(e, e->up_ops, &e->up_i, descs.data(), descs.size() * sizeof(OpDesc), &u, nullptr, kCounterBytes);
            if (rc) return rc;   // nothing launched: every plane is as before
            if (cpt::fault_injected("engine_submit"))
                return efail(e, CPT_ECUDA, "submit refused before its launch (injected)");
            launched = true;
            rc = launch_uploaded(e, descs, items, u->d);
            if (!rc) {
                for (const auto &pn : n_after) e->planes[pn.first].n = pn.second;
                ECK(e, cudaEventRecord(u->consumed, e->stream));
                return CPT_OK;
            }
        }
    } else {
        rc = launch_ops(e, dev_ops.data(), (int32_t)dev_ops.size(), &launched);
        if (!rc) rc = stream_host_ops(e, host_ops, &launched);
    }
    if (rc) {
        // a launch may have begun: the planes of the submit hold an unknown
        // part of the ops until they are cleared
        if (launched)
            for (const auto &pn : n_after) e->planes[pn.first].poisoned = true;
        return rc;
    }
    for (const auto &pn : n_after) e->planes[pn.first].n = pn.second;
    return CPT_OK;
}

void destroy_graph(composite_engine *e) {
    if (e->graph_exec) cudaGraphExecDestroy(e->graph_exec);
    if (e->graph) cudaGraphDestroy(e->graph);
    if (e->graph_ops) cudaFree(e->graph_ops);
    if (e->graph_rops) cudaFree(e->graph_rops);
    if (e->graph_clears) cudaFree(e->graph_clears);
    if (e->graph_counters) cudaFree(e->graph_counters);
    e->graph_exec = nullptr;
    e->graph = nullptr;
    e->graph_ops = e->graph_rops = e->graph_clears = nullptr;
    e->graph_counters = nullptr;
    e->graph_n.clear();
    e->graph_planes.clear();
}

void destroy_engine(composite_engine *e) {
    destroy_graph(e);
    for (PlaneRec &p : e->planes)
        if (p.data) cudaFree(p.data);
    for (Upload *ring : {e->up_ops, e->up_render})
        for (int i = 0; i < kUploadRing; ++i) {
            if (ring[i].d) cudaFree(ring[i].d);
            if (ring[i].h) cudaFreeHost(ring[i].h);
            if (ring[i].done) cudaEventDestroy(ring[i].done);
            if (ring[i].consumed) cudaEventDestroy(ring[i].consumed);
        }
    if (e->d_flags) cudaFree(e->d_flags);
    if (e->h_flags) cudaFreeHost(e->h_flags);
    if (e->done_ev) cudaEventDestroy(e->done_ev);
    if (e->capture_stream) cudaStreamDestroy(e->capture_stream);
    free_stage(e);
    if (e->copy) cudaStreamDestroy(e->copy);
    if (e->caller_ready) cudaEventDestroy(e->caller_ready);
    delete e;
}

}  // namespace

extern "C" {

int composite_engine_default_config(composite_engine_config *cfg) try {
    if (!cfg) return CPT_EINVAL;
    memset(cfg, 0, sizeof *cfg);
    cfg->slab_members = 128;
    cfg->ctas_per_sm = 5;
    cfg->schedule = CPT_SCHEDULE_PERSISTENT;
    cfg->item_member_groups = kDefaultItemMemberGroups;
    cfg->staging_buffers = 2;
    cfg->staging_bytes = kDefaultStageBytes;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_begin(composite_engine **out, const composite_engine_config *cfg) try {
    g_engine_error.clear();
    if (!out) return efail(nullptr, CPT_EINVAL, "out is NULL");
    *out = nullptr;
    composite_engine_config c;
    composite_engine_default_config(&c);
    if (cfg) {
        c.cuda_stream = cfg->cuda_stream;
        c.wait_timeout_ms = cfg->wait_timeout_ms;
        if (cfg->slab_members) c.slab_members = cfg->slab_members;
        if (cfg->ctas_per_sm) c.ctas_per_sm = cfg->ctas_per_sm;
        c.schedule = cfg->schedule;
        c.upload_stream = cfg->upload_stream;
        if (cfg->item_member_groups) c.item_member_groups = cfg->item_member_groups;
        if (cfg->staging_buffers) c.staging_buffers = cfg->staging_buffers;
        if (cfg->staging_bytes) c.staging_bytes = cfg->staging_bytes;
    }
    if (c.schedule != CPT_SCHEDULE_PERSISTENT && c.schedule != CPT_SCHEDULE_GRID)
        return efail(nullptr, CPT_EINVAL, "schedule must be CPT_SCHEDULE_PERSISTENT or CPT_SCHEDULE_GRID");
    if (c.slab_members < 1 || c.slab_members > kMaxSlab) return efail(nullptr, CPT_EINVAL, "slab_members not in 1..255");
    if (c.ctas_per_sm < 1 || c.ctas_per_sm > 8) return efail(nullptr, CPT_EINVAL, "ctas_per_sm not in 1..8");
    if (c.wait_timeout_ms < 0) return efail(nullptr, CPT_EINVAL, "negative timeout");
    if (c.item_member_groups < 16 || c.item_member_groups > 8192)
        return efail(nullptr, CPT_EINVAL, "item_member_groups not in 16..8192");
    if (c.staging_buffers < 2 || c.staging_buffers > 8) return efail(nullptr, CPT_EINVAL, "staging_buffers not in 2..8");
    if (c.staging_bytes < (1ll << 20)) return efail(nullptr, CPT_EINVAL, "staging_bytes below 1 MiB");
    composite_engine *e = new composite_engine();
    e->cfg = c;
    auto setup = [&]() -> int {
        ECK(e, cudaGetDevice(&e->device));
        ECK(e, cudaDeviceGetAttribute(&e->caps.num_sms, cudaDevAttrMultiProcessorCount, e->device));
        e->stream = static_cast<cudaStream_t>(c.cuda_stream);   // NULL: the legacy default stream
        ECK(e, cudaMalloc(&e->d_flags, kMaxPlanes * sizeof(int)));
        ECK(e, cudaMemsetAsync(e->d_flags, 0, kMaxPlanes * sizeof(int), e->stream));
        ECK(e, cudaHostAlloc(&e->h_flags, kMaxPlanes * sizeof(int), cudaHostAllocDefault));
        ECK(e, cudaEventCreateWithFlags(&e->done_ev, cudaEventDisableTiming));
        for (Upload *ring : {e->up_ops, e->up_render})
            for (int i = 0; i < kUploadRing; ++i) {
                ECK(e, cudaEventCreateWithFlags(&ring[i].done, cudaEventDisableTiming));
                ECK(e, cudaEventCreateWithFlags(&ring[i].consumed, cudaEventDisableTiming));
            }
        e->default_lut = make_lut(nullptr);
        return prepare_render_kernels(e);
    };
    const int rc = setup();
    if (rc) {
        g_engine_error = e->err;
        destroy_engine(e);
        return rc;
    }
    *out = e;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_add_plane(composite_engine *e, int32_t width, int32_t height, int32_t *plane_out) try {
    return composite_engine_add_plane_bits(e, width, height, 32, plane_out);
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_add_plane_bits(composite_engine *e, int32_t width, int32_t height, int32_t count_bits,
                                    int32_t *plane_out) try {
    if (!e || !plane_out) return CPT_EINVAL;
    e->err.clear();
    if (width <= 0 || height <= 0) return efail(e, CPT_EINVAL, "plane %d x %d is empty", width, height);
    if (count_bits != 16 && count_bits != 32) return efail(e, CPT_EINVAL, "count_bits must be 16 or 32");
    if ((int)e->planes.size() >= kMaxPlanes) return efail(e, CPT_EINVAL, "at most %d planes", kMaxPlanes);
    PlaneRec r;
    r.width = width;
    r.height = height;
    r.pitch_px = ((int64_t)width + 15) / 16 * 16;
    r.count_bits = count_bits;
    if (cpt::fault_injected("engine_plane")) return efail(e, CPT_ENOMEM, "plane allocation refused (injected)");
    ECK(e, cudaMalloc(&r.data, r.bytes()));
    r.alive = true;
    e->planes.push_back(r);
    const int32_t id = (int32_t)e->planes.size() - 1;
    const int rc = clear_plane(e, id);
    if (rc) return rc;
    *plane_out = id;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_free_plane(composite_engine *e, int32_t plane) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    if (!plane_ok(e, plane)) return efail(e, CPT_EINVAL, "no plane %d", plane);
    int rc = drain(e);
    if (rc) return rc;
    cudaFree(e->planes[plane].data);
    e->planes[plane] = PlaneRec();
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_clear(composite_engine *e, int32_t plane) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    if (!plane_ok(e, plane)) return efail(e, CPT_EINVAL, "no plane %d", plane);
    return clear_plane(e, plane);
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_clear_many(composite_engine *e, const int32_t *planes, int32_t n_planes) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    return clear_many(e, planes, n_planes);
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_submit(composite_engine *e, const composite_op *ops, int32_t n_ops) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    return submit_internal(e, ops, n_ops);
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_render(composite_engine *e, const composite_render_op *ops, int32_t n_ops,
                            const uint8_t *lut_rgba) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    std::vector<RenderDesc> descs;
    int64_t items = 0;
    int rc = plan_render(e, ops, n_ops, &descs, &items, nullptr);
    if (rc || items == 0) return rc;
    const bool hist = any_histogram(descs);
    std::vector<ClearDesc> cdescs;
    int64_t citems = 0;
    if (hist) plan_histogram_clears(descs, &cdescs, &citems);
    // one upload: the histograms' clear entries, then the render descriptors
    std::vector<unsigned char> blob(cdescs.size() * sizeof(ClearDesc) + descs.size() * sizeof(RenderDesc));
    if (!cdescs.empty()) memcpy(blob.data(), cdescs.data(), cdescs.size() * sizeof(ClearDesc));
    memcpy(blob.data() + cdescs.size() * sizeof(ClearDesc), descs.data(), descs.size() * sizeof(RenderDesc));
    Upload *u = nullptr;
    rc = upload(e, e->up_render, &e->rup_i, blob.data(), blob.size(), &u);
    if (rc) return rc;
    if (citems > 0) {
        rc = launch_clear(e, u->d, (int)cdescs.size(), citems);
        if (rc) return rc;
    }
    rc = launch_render(e, static_cast<unsigned char *>(u->d) + cdescs.size() * sizeof(ClearDesc), descs, items,
                       lut_rgba ? make_lut(lut_rgba) : e->default_lut);
    if (rc) return rc;
    ECK(e, cudaEventRecord(u->consumed, e->stream));
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_member_count(const composite_engine *e, int32_t plane, int64_t *n_out) try {
    if (!e || !n_out || !plane_ok(e, plane)) return CPT_EINVAL;
    *n_out = e->planes[plane].n;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_sync(composite_engine *e, int32_t *bad_plane_out) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    if (bad_plane_out) *bad_plane_out = -1;
    const size_t n = e->planes.size();
    if (n) ECK(e, cudaMemcpyAsync(e->h_flags, e->d_flags, n * sizeof(int), cudaMemcpyDeviceToHost, e->stream));
    int rc = drain(e);
    if (rc) return rc;
    for (size_t p = 0; p < n; ++p)
        if (e->planes[p].alive && e->h_flags[p]) {
            if (bad_plane_out) *bad_plane_out = (int32_t)p;
            return efail(e, CPT_EUNDERFLOW, "plane %zu: a remove took away a member that was never added", p);
        }
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_capture(composite_engine *e, const composite_op *ops, int32_t n_ops,
                             const composite_render_op *rops, int32_t n_rops, const uint8_t *lut_rgba) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    std::vector<OpDesc> descs;
    std::vector<RenderDesc> rdescs;
    std::vector<std::pair<int32_t, int64_t>> n_after;
    int64_t items = 0, ritems = 0;
    int rc = plan_ops(e, ops, n_ops, &descs, &items, &n_after, true);
    if (rc) return rc;
    for (int32_t i = 0; i < n_ops; ++i) {
        if (ops[i].n_members == 0) continue;
        if (member_kind(ops[i].members, e->device) != 0)
            return efail(e, CPT_EINVAL, "op %d: a captured graph reads members of device %d only", i, e->device);
        if (ops[i].member_index && !device_reachable(ops[i].member_index, e->device))
            return efail(e, CPT_EINVAL, "op %d: member_index must be device memory of device %d", i, e->device);
    }
    rc = plan_render(e, rops, n_rops, &rdescs, &ritems, &n_after);
    if (rc) return rc;
    std::vector<int32_t> cleared;
    for (const auto &pn : n_after) cleared.push_back(pn.first);
    std::vector<ClearDesc> cdescs;
    int64_t citems = 0;
    rc = plan_clears(e, cleared.data(), (int32_t)cleared.size(), &cdescs, &citems);
    if (rc) return rc;
    plan_histogram_clears(rdescs, &cdescs, &citems);   // zeroed in the same clear node
    rc = drain(e);
    if (rc) return rc;
    destroy_graph(e);
    ECK(e, cudaMalloc(&e->graph_counters, kCounterBytes));
    if (items > 0) {   // the item counter too
        ClearDesc d{};
        d.data = reinterpret_cast<uint4 *>(e->graph_counters);
        d.words = kCounterBytes / 16;
        d.item_start = citems++;
        d.plane_id = -1;
        cdescs.push_back(d);
    }
    if (!cdescs.empty()) {
        ECK(e, cudaMalloc(&e->graph_clears, cdescs.size() * sizeof(ClearDesc)));
        ECK(e, cudaMemcpy(e->graph_clears, cdescs.data(), cdescs.size() * sizeof(ClearDesc), cudaMemcpyHostToDevice));
    }
    if (!descs.empty()) {
        ECK(e, cudaMalloc(&e->graph_ops, descs.size() * sizeof(OpDesc)));
        ECK(e, cudaMemcpy(e->graph_ops, descs.data(), descs.size() * sizeof(OpDesc), cudaMemcpyHostToDevice));
    }
    if (!rdescs.empty()) {
        ECK(e, cudaMalloc(&e->graph_rops, rdescs.size() * sizeof(RenderDesc)));
        ECK(e, cudaMemcpy(e->graph_rops, rdescs.data(), rdescs.size() * sizeof(RenderDesc), cudaMemcpyHostToDevice));
    }
    const Lut lut = lut_rgba ? make_lut(lut_rgba) : e->default_lut;
    // Capture happens on a private stream (the legacy default stream cannot
    // be captured); the graph is launched on the engine's stream.
    if (!e->capture_stream) ECK(e, cudaStreamCreateWithFlags(&e->capture_stream, cudaStreamNonBlocking));
    cudaStream_t engine_stream = e->stream;
    e->stream = e->capture_stream;
    struct Restore {
        composite_engine *e;
        cudaStream_t s;
        ~Restore() { e->stream = s; }
    } restore{e, engine_stream};
    ECK(e, cudaStreamBeginCapture(e->stream, cudaStreamCaptureModeThreadLocal));
    auto body = [&]() -> int {
        if (citems > 0) {   // every target plane and its flag in one node
            int r = launch_clear(e, e->graph_clears, (int)cdescs.size(), citems);
            if (r) return r;
        }
        if (items > 0) {
            int r = launch_accumulate(e, e->graph_ops, descs, items, e->graph_counters);
            if (r) return r;
        }
        if (ritems > 0) {
            int r = launch_render(e, e->graph_rops, rdescs, ritems, lut);
            if (r) return r;
        }
        return CPT_OK;
    };
    const int brc = body();
    cudaGraph_t g = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(e->stream, &g);
    if (brc) {
        if (g) cudaGraphDestroy(g);
        return brc;
    }
    if (ec != cudaSuccess) return ecuda(e, ec, "cudaStreamEndCapture");
    e->graph = g;
    ECK(e, cudaGraphInstantiate(&e->graph_exec, e->graph, 0));
    e->graph_n = n_after;
    for (const auto &pn : n_after) e->graph_planes.push_back(pn.first);
    for (int32_t i = 0; i < n_rops; ++i) e->graph_planes.push_back(rops[i].plane);
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_replay(composite_engine *e) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    if (!e->graph_exec) return efail(e, CPT_ESTATE, "nothing captured");
    for (const int32_t p : e->graph_planes)
        if (!plane_ok(e, p)) return efail(e, CPT_ESTATE, "a captured plane was freed");
    ECK(e, cudaGraphLaunch(e->graph_exec, e->stream));
    // the graph clears every plane it folds into before folding
    for (const auto &pn : e->graph_n) {
        e->planes[pn.first].n = pn.second;
        e->planes[pn.first].poisoned = false;
    }
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_tune(composite_engine *e, const composite_op *ops, int32_t n_ops, int32_t repeats,
                          int32_t *slab_out, int32_t *ctas_out) try {
    if (!e) return CPT_EINVAL;
    e->err.clear();
    if (repeats < 1) return efail(e, CPT_EINVAL, "repeats < 1");
    std::vector<OpDesc> descs;
    std::vector<std::pair<int32_t, int64_t>> n_after;
    int64_t items = 0;
    int rc = plan_ops(e, ops, n_ops, &descs, &items, &n_after, true);
    if (rc) return rc;
    bool any_host = false;
    for (int32_t i = 0; i < n_ops; ++i)
        if (ops[i].n_members > 0 && member_kind(ops[i].members, e->device) == 1) any_host = true;
    cudaEvent_t a = nullptr, b = nullptr;
    ECK(e, cudaEventCreate(&a));
    cudaError_t ce = cudaEventCreate(&b);
    if (ce != cudaSuccess) {
        cudaEventDestroy(a);
        return ecuda(e, ce, "cudaEventCreate");
    }
    std::vector<int32_t> cleared;
    for (const auto &pn : n_after) cleared.push_back(pn.first);
    auto run = [&]() -> int {
        const int r = clear_many(e, cleared.data(), (int32_t)cleared.size());
        return r ? r : submit_internal(e, ops, n_ops);
    };
    // Best of `repeats` timed runs (each after an untimed one) of the current
    // configuration, in ms; < 0 on error (rc set).
    auto time_config = [&]() -> float {
        float t_best = 1e30f;
        for (int r = 0; r < repeats; ++r) {
            if ((rc = run())) return -1.f;             // warm and measure alike: clear + submit
            if (cudaEventRecord(a, e->stream) != cudaSuccess) { rc = efail(e, CPT_ECUDA, "cudaEventRecord"); return -1.f; }
            if ((rc = run())) return -1.f;
            if (cudaEventRecord(b, e->stream) != cudaSuccess) { rc = efail(e, CPT_ECUDA, "cudaEventRecord"); return -1.f; }
            if ((rc = ewait(e, b))) return -1.f;
            float ms = 0;
            cudaEventElapsedTime(&ms, a, b);
            t_best = std::min(t_best, ms);
        }
        return t_best;
    };
    composite_engine_config best = e->cfg;
    float best_ms = 1e30f;
    auto consider = [&]() -> bool {
        const float ms = time_config();
        if (ms < 0) return false;
        if (ms < best_ms) {
            best_ms = ms;
            best = e->cfg;
        }
        return true;
    };
    // pass 1: slab depth x schedule (ctas_per_sm 0 stands for the grid schedule)
    static const int slabs[] = {32, 64, 128, 255};
    static const int ctas[] = {0, 3, 4, kDeepBitsCtas};
    bool any_bits = false;
    for (const OpDesc &d : descs) any_bits = any_bits || d.bits;
    const int ctas_before = e->cfg.ctas_per_sm;
    for (int sl : slabs)
        for (int c : ctas) {
            if (rc) break;
            if (c == kDeepBitsCtas && !any_bits) continue;   // would run as four
            e->cfg.slab_members = sl;
            e->cfg.schedule = c ? CPT_SCHEDULE_PERSISTENT : CPT_SCHEDULE_GRID;
            e->cfg.ctas_per_sm = c ? c : ctas_before;
            if (!consider()) break;
        }
    // pass 2: the work item's tile of groups
    static const int item_groups[] = {256, 512, 1024, 2048};
    if (!rc) {
        e->cfg = best;
        for (int g : item_groups) {
            e->cfg.item_member_groups = g;
            if (!consider()) break;
        }
    }
    // pass 3: staging buffers for host members
    static const int stage_counts[] = {2, 3, 4};
    static const int stage_mib[] = {64, 128, 256, 512};
    if (!rc && any_host) {
        int64_t largest = 0;
        for (int32_t i = 0; i < n_ops; ++i)
            largest = std::max<int64_t>(largest, (int64_t)ops[i].row_pitch_bytes * e->planes[ops[i].plane].height);
        e->cfg = best;
        for (int k : stage_counts)
            for (int mib : stage_mib) {
                if (rc || ((int64_t)mib << 20) < largest) continue;
                e->cfg.staging_buffers = k;
                e->cfg.staging_bytes = (int64_t)mib << 20;
                if (!consider()) break;
            }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    e->cfg = best;
    if (rc) return rc;
    rc = run();
    if (rc) return rc;
    if (slab_out) *slab_out = best.slab_members;
    if (ctas_out) *ctas_out = best.schedule == CPT_SCHEDULE_GRID ? 0 : best.ctas_per_sm;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_get_tuning(const composite_engine *e, int32_t *slab_out, int32_t *ctas_out) try {
    if (!e) return CPT_EINVAL;
    if (slab_out) *slab_out = e->cfg.slab_members;
    if (ctas_out) *ctas_out = e->cfg.schedule == CPT_SCHEDULE_GRID ? 0 : e->cfg.ctas_per_sm;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_get_config(const composite_engine *e, composite_engine_config *cfg_out) try {
    if (!e || !cfg_out) return CPT_EINVAL;
    *cfg_out = e->cfg;
    return CPT_OK;
} catch (...) {
    return cpt::abi_exception_status();
}

int composite_engine_end(composite_engine *e) try {
    if (!e) return CPT_OK;
    const int rc = drain(e);
    destroy_engine(e);
    return rc;
} catch (...) {
    return cpt::abi_exception_status();
}

const char *composite_engine_last_error(const composite_engine *e) try {
    return e ? e->err.c_str() : g_engine_error.c_str();
} catch (...) {
    return "internal error (exception)";
}

}  // extern "C"
