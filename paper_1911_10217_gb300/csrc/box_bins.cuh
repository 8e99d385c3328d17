// Occluder boxes with a table that tells which of them can meet a segment.
//
// Along each axis the boxes' extent, or the part of it where most of them
// begin and end (narrow_bins), is cut into uniform bins; for every bin j
// two bit masks over the boxes are kept: those that begin in bin j or before
// it, and those that end in bin j or after it. A box can meet a segment only
// if on every axis it begins no later than the segment's upper end and ends
// no earlier than its lower end, so the AND of six masks, picked by the bins
// of the segment's bounding box, holds every box that can; only those are
// tested. A bin is a monotone function of the coordinate (one rounded
// multiply-add, clamped), the same for boxes and segments, so no box whose
// interval meets the segment's is left out; a coordinate without an order
// (NaN) takes the bin that keeps every box.
//
// The table is rebuilt from the boxes by one block before every sampling
// launch (4.6 us; the boxes may change from call to call) and copied to
// shared memory by each of its blocks. In a sampling launch of few blocks and
// boxes, and in the energy sampler and the bounces, whose blocks stay and
// take many points, each block builds the table for itself.
// Against one run of the boxes sorted along x, which every segment searched
// and then walked through (and, in the energy sampler and the bounces, against
// every box): 12-scene batch equal, 1080p passes 424 -> 416 us, sky dome (128
// leaves, 2 samples) 668 -> 648, paths 570 -> 512, energy sampler 590 -> 392;
// the table took 3.8 us to build at that point (4.6 with narrow_bins), the sort 6.3 us.
#pragma once

#include <cuda_runtime.h>

#include "rll_device.cuh"

namespace rll {
namespace {

// Bins an axis, and 64-bit words a mask, for n boxes: the table is 1.5 KB at 64 boxes, 6 KB at 256
// and 12 KB at 1024 (where half as many bins keep it and the boxes within 48 KB).
__host__ __device__ constexpr int box_bins(int n) { return n <= 256 ? 32 : 16; }
__host__ __device__ constexpr int box_words(int n) { return (n + 63) / 64; }
static_assert(2 * box_words(256) == 8 && 2 * box_words(257) > 8, "build_box_table: 32 bins where it scans by warps");

// Layout of the table: (scale xyz, w) and (offset xyz, 0) as float4, w = 1 where a box has a minimum
// above its maximum, else 0; masks [6][bins][words] of 64 bits, axis k's begin masks at 2k and its end
// masks at 2k + 1; boxes [n] as float4 (min), (max).
__host__ __device__ constexpr size_t box_mask_bytes(int n) { return 48u * (size_t)box_bins(n) * (size_t)box_words(n); }
__host__ __device__ constexpr size_t box_table_bytes(int n) { return 32u + box_mask_bytes(n) + 32u * (size_t)n; }
constexpr size_t kMaxBoxTable = box_table_bytes(kMaxBoxes);
static_assert(box_table_bytes(256) < kMaxBoxTable && kMaxBoxTable % 16 == 0, "box table size");

// Bytes that hold the table of any number of boxes up to n, which box_table_bytes(n) does not: the
// bins halve above 256 boxes, where 257 take 12 096 bytes and 256 take 14 368.
__host__ __device__ constexpr size_t box_table_room(int n)
{
    return n > 256 && box_table_bytes(n) < box_table_bytes(256) ? box_table_bytes(256) : box_table_bytes(n);
}
constexpr bool box_table_room_holds()
{
    size_t most = 0;
    for (int n = 0; n <= kMaxBoxes; ++n) {
        most = box_table_bytes(n) > most ? box_table_bytes(n) : most;
        if (box_table_room(n) < most) return false;
    }
    return box_table_room(kMaxBoxes) == kMaxBoxTable;
}
static_assert(box_table_room_holds(), "a smaller table exceeds the room of a larger one");

// Bin of a coordinate whose scaled value is t: as a lower end (NaN: the first bin) or an upper end
// (NaN: the last).
__device__ __forceinline__ int box_bin_lo(float t, int bins)
{
    return (int)fminf(fmaxf(t, 0.0f), (float)(bins - 1));
}
__device__ __forceinline__ int box_bin_hi(float t, int bins)
{
    return (int)fmaxf(fminf(t, (float)(bins - 1)), 0.0f);
}

// A table in shared memory, of n boxes (n = 0: none, nothing is read).
struct BoxTable {
    const char* at;
    int n;

    __device__ __forceinline__ const float4* boxes() const
    {
        return reinterpret_cast<const float4*>(at + 32 + box_mask_bytes(n));
    }
    // A box has a minimum above its maximum.
    __device__ __forceinline__ bool swapped() const
    {
        return n > 0 && reinterpret_cast<const float4*>(at)[0].w != 0.0f;
    }
    // The boxes' largest extent along an axis (0: none, or no boxes).
    __device__ __forceinline__ float extent() const
    {
        if (n == 0) return 0.0f;
        const float4 sc = reinterpret_cast<const float4*>(at)[0];
        float e = 0.0f;
        if (sc.x > 0.0f) e = fmaxf(e, (float)box_bins(n) / sc.x);
        if (sc.y > 0.0f) e = fmaxf(e, (float)box_bins(n) / sc.y);
        if (sc.z > 0.0f) e = fmaxf(e, (float)box_bins(n) / sc.z);
        return e;
    }
    // Calls test(box index) for the boxes that can meet the axis-aligned box lo .. hi, in increasing
    // order of their index, until it returns true; whether it did.
    template <class Test>
    __device__ __forceinline__ bool any(float lo0, float lo1, float lo2, float hi0, float hi1, float hi2,
                                        Test test) const
    {
        if (n == 0) return false;
        const int bins = box_bins(n), words = box_words(n);
        const float4 sc = reinterpret_cast<const float4*>(at)[0], of = reinterpret_cast<const float4*>(at)[1];
        const unsigned long long* mask = reinterpret_cast<const unsigned long long*>(at + 32);
        const unsigned long long* b0 = mask + box_bin_hi(__fmaf_rn(hi0, sc.x, of.x), bins) * words;
        const unsigned long long* e0 = mask + (bins + box_bin_lo(__fmaf_rn(lo0, sc.x, of.x), bins)) * words;
        const unsigned long long* b1 = mask + (2 * bins + box_bin_hi(__fmaf_rn(hi1, sc.y, of.y), bins)) * words;
        const unsigned long long* e1 = mask + (3 * bins + box_bin_lo(__fmaf_rn(lo1, sc.y, of.y), bins)) * words;
        const unsigned long long* b2 = mask + (4 * bins + box_bin_hi(__fmaf_rn(hi2, sc.z, of.z), bins)) * words;
        const unsigned long long* e2 = mask + (5 * bins + box_bin_lo(__fmaf_rn(lo2, sc.z, of.z), bins)) * words;
        for (int w = 0; w < words; ++w) {
            unsigned long long m = b0[w] & e0[w] & b1[w] & e1[w] & b2[w] & e2[w];
            // the word's halves in turn: a 64-bit find-first and clear take twice the instructions, which
            // tells where most boxes are candidates (52 of 64 boxes in one spot of the room, 1080p:
            // sampling 457 -> 429 us, energy sampler 269 -> 241, bounces 239 -> 218; the walled room 320,
            // 88 -> 89 and 126 -> 120)
            uint32_t cur = (uint32_t)m, next = (uint32_t)(m >> 32);
            int first = 64 * w + 31;
            while (cur | next) {
                if (cur == 0u) {
                    cur = next;
                    next = 0u;
                    first += 32;
                }
                const uint32_t bit = cur & (0u - cur);
                if (test(first - __clz((int)bit))) return true;
                cur ^= bit;
            }
        }
        return false;
    }
};

// The ends of a box along axis k, lower and upper, also of one given the other way round (which the
// slab tests take like any other).
__device__ __forceinline__ float box_lower(const float* v, int k) { return v[3 + k] < v[k] ? v[3 + k] : v[k]; }
__device__ __forceinline__ float box_upper(const float* v, int k) { return v[3 + k] < v[k] ? v[k] : v[3 + k]; }

// Bins over a part of the extent, where few boxes stretch it (a ground slab, a distant wall): called by
// a warp for one axis, after every box has set its bit in the mask of the bin it begins in and in that
// of the bin it ends in (begins, ends: [bins][words]). Where a window of at most `most` bins holds at
// least 5/8 of the ends, the bins next to it none, and at most a quarter of all bins beside it any, the
// window is the bins' next range (ends beyond it are clamped, which keeps the masks right). Returns
// whether it is.
// Bins over the whole extent, where a ground slab of 100 times the room's size left one bin to the room,
// had lost the table's gain and more: 1080p, 64 boxes and that slab, by the loops that the table
// replaced / by bins over the whole extent / so: sampling 439 / 431 / 331 us, energy sampler 177 / 238 /
// 95, bounces 269 / 376 / 139; 1 024 boxes and the slab 2 500 / 3 643 / 2 006, 2 016 / 3 410 / 1 667 and
// 3 665 / 5 300 / 1 236. Boxes without such a one take one step, which finds nothing (1080p passes equal).
__device__ __forceinline__ bool narrow_bins(const uint32_t* begins, const uint32_t* ends, int bins, int words, int n,
                                            int most, float* scale, float* off)
{
    const int lane = threadIdx.x & 31;
    int held = 0;  // ends in the window that begins in bin `lane`, at first that bin alone
    if (lane < bins) {
        int at = lane % words;  // lanes a bank apart
#pragma unroll 1
        for (int w = 0; w < words; ++w) {
            held += __popc(begins[lane * words + at]) + __popc(ends[lane * words + at]);
            at = at + 1 < words ? at + 1 : 0;
        }
    }
    const uint32_t used = __ballot_sync(0xffffffffu, held > 0);
    if (__popc(used) > most + bins / 4) return false;
#pragma unroll 1
    for (int width = 1; width <= most; width *= 2) {
        const uint32_t window = ((1u << width) - 1u) << lane, beside = used & ~window;
        const uint32_t fits = __ballot_sync(0xffffffffu, lane + width <= bins && 4 * held >= 5 * n &&
                                                             !(beside & (window << 1 | window >> 1)) &&
                                                             4 * __popc(beside) <= bins);
        if (fits) {
            const float zoom = (float)(bins / width), s = *scale * zoom, o = *off - (float)(__ffs((int)fits) - 1);
            if (!(*scale > 0.0f && s < 1e30f)) return false;
            __syncwarp();
            if (lane == 0) {
                *off = o * zoom;
                *scale = s;
            }
            return true;
        }
        held += __shfl_down_sync(0xffffffffu, held, width);
    }
    return false;
}
constexpr int kMaxNarrow = 12;  // steps, of 2 to 32 times each
// Up to so many boxes keep the whole extent: testing all of them costs less than the look at the bins
// in a small launch (64x64 points, 8 boxes: 33.6 us a pass with it, 32.9 without; 1080p, 14 boxes and the
// slab: sampling 320 and 330 us, energy sampler 95 and 106, by loops over all boxes 400 and 146; 16 boxes
// and 6 distant walls are narrowed: 321 and 95, not narrowed 345 and 122).
constexpr int kFewToNarrow = 16;

// Builds the table of n (1 .. kMaxBoxes) boxes [n][6] into out, by a whole block of 96 to 256
// threads; s_mask: its masks in shared memory, or a scratch copy of them there (box_mask_bytes).
__device__ __forceinline__ void build_box_table(const float* __restrict__ boxes, int n, char* out, uint32_t* s_mask)
{
    __shared__ float s_lim[8][6];
    __shared__ float s_scale[3], s_off[3];
    const int bins = box_bins(n), words = 2 * box_words(n), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto clear = [&]() {
        for (int i = threadIdx.x; i < 6 * bins * words; i += blockDim.x) s_mask[i] = 0u;
    };
    clear();
    // the extent of the finite ends (infinite and as good as infinite ones are clamped)
    float lim[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
    float4* box = reinterpret_cast<float4*>(out + 32 + box_mask_bytes(n));
    bool swapped = false;
    for (int b = threadIdx.x; b < n; b += blockDim.x) {
        const float* v = boxes + 6 * b;
        for (int k = 0; k < 3; ++k) {
            const float lo = box_lower(v, k), hi = box_upper(v, k);
            if (fabsf(lo) < 1e18f) lim[k] = fminf(lim[k], lo), lim[3 + k] = fmaxf(lim[3 + k], lo);
            if (fabsf(hi) < 1e18f) lim[k] = fminf(lim[k], hi), lim[3 + k] = fmaxf(lim[3 + k], hi);
        }
        swapped = swapped || v[3] < v[0] || v[4] < v[1] || v[5] < v[2];
        box[2 * b] = make_float4(v[0], v[1], v[2], 0.0f);
        box[2 * b + 1] = make_float4(v[3], v[4], v[5], 0.0f);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float y = __shfl_xor_sync(0xffffffffu, lim[k], o);
            lim[k] = k < 3 ? fminf(lim[k], y) : fmaxf(lim[k], y);
        }
        if (lane == 0) s_lim[warp][k] = lim[k];
    }
    swapped = __syncthreads_or(swapped);
    if (threadIdx.x < 3) {
        const int k = threadIdx.x;
        float lo = s_lim[0][k], hi = s_lim[0][3 + k];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
            lo = fminf(lo, s_lim[w][k]);
            hi = fmaxf(hi, s_lim[w][3 + k]);
        }
        float scale = (float)bins / (hi - lo);
        if (!(hi > lo && scale < 1e30f)) scale = 0.0f;  // no extent: one bin
        s_scale[k] = scale;
        s_off[k] = -lo * scale;  // NaN without a finite end: every box is kept
    }
    __syncthreads();
    const float scale0 = warp < 3 ? s_scale[warp] : 0.0f, off0 = warp < 3 ? s_off[warp] : 0.0f;
    bool wide = warp >= 3;  // this warp's axis keeps its bins
    for (int step = 0;; ++step) {
        for (int i = threadIdx.x; i < 3 * n; i += blockDim.x) {
            const int b = i / 3, k = i % 3;
            const float* v = boxes + 6 * b;
            const int j0 = box_bin_lo(__fmaf_rn(box_lower(v, k), s_scale[k], s_off[k]), bins);
            const int j1 = box_bin_hi(__fmaf_rn(box_upper(v, k), s_scale[k], s_off[k]), bins);
            atomicOr(&s_mask[(2 * k * bins + j0) * words + (b >> 5)], 1u << (b & 31));
            atomicOr(&s_mask[((2 * k + 1) * bins + j1) * words + (b >> 5)], 1u << (b & 31));
        }
        __syncthreads();
        if (n <= kFewToNarrow) break;
        bool again = false;
        if (!wide) {
            const uint32_t* begins = s_mask + 2 * warp * bins * words;
            // the first step from a quarter of the bins, which evenly spread boxes do not meet
            again = narrow_bins(begins, begins + bins * words, bins, words, n, step ? bins / 2 : bins / 4,
                                &s_scale[warp], &s_off[warp]);
            wide = !again;
            if (again && step == kMaxNarrow) {  // ends that no bins tell apart: as it was
                __syncwarp();
                s_scale[warp] = scale0;
                s_off[warp] = off0;
                wide = true;
            }
        }
        if (!__syncthreads_or(again)) break;
        clear();
        __syncthreads();
    }
    if (threadIdx.x < 2) {
        const float* v = threadIdx.x ? s_off : s_scale;
        const float w = threadIdx.x == 0 && swapped ? 1.0f : 0.0f;
        reinterpret_cast<float4*>(out)[threadIdx.x] = make_float4(v[0], v[1], v[2], w);
    }
    // begins: up the bins, ends: down; up to eight words by warps, a lane a bin (in turn, by a thread a
    // word, it took as long as all the rest), more by threads
    if (words <= 8) {
        for (int k = warp; k < 6; k += (int)(blockDim.x >> 5)) {
            uint32_t* row = s_mask + (k * bins + lane) * words;
#pragma unroll 2
            for (int w = 0; w < words; ++w) {
                uint32_t v = row[w];
#pragma unroll
                for (int o = 1; o < 32; o <<= 1)
                    v |= __shfl_sync(0xffffffffu, v, k & 1 ? min(lane + o, 31) : max(lane - o, 0));
                row[w] = v;
            }
        }
    } else {
        for (int i = threadIdx.x; i < 6 * words; i += blockDim.x) {
            const int k = i / words, w = i % words;
            uint32_t run = 0;
            for (int s = 0; s < bins; ++s) {
                const int j = k & 1 ? bins - 1 - s : s;
                run |= s_mask[(k * bins + j) * words + w];
                s_mask[(k * bins + j) * words + w] = run;
            }
        }
    }
    __syncthreads();
    uint32_t* mask = reinterpret_cast<uint32_t*>(out + 32);
    if (mask != s_mask)
        for (int i = threadIdx.x; i < 6 * bins * words; i += blockDim.x) mask[i] = s_mask[i];
}

// The same out of line, for the sampling kernels: in line it cost those that do not run it 1 % (1080p
// passes 382.5 -> 386.7 us), while a call in the energy sampler costs that one 4 % (spills).
__device__ __noinline__ void build_box_table_call(const float* __restrict__ boxes, int n, char* out, uint32_t* s_mask)
{
    build_box_table(boxes, n, out, s_mask);
}

// The same by a block that writes the table to global memory.
__device__ __forceinline__ void build_box_table_global(const float* __restrict__ boxes, int n, char* out)
{
    __shared__ uint32_t s_mask[box_mask_bytes(kMaxBoxes) / 4];
    static_assert(box_mask_bytes(kMaxBoxes) >= box_mask_bytes(256), "largest table");
    build_box_table(boxes, n, out, s_mask);
}

// The table copied to shared memory by all threads of the block (the caller synchronises).
// SELF: without a table (nullptr) the block builds its own from the boxes.
// CALL: that out of line.
template <bool SELF = false, bool CALL = false>
__device__ __forceinline__ BoxTable stage_box_table(void* s_table, const void* table, int n,
                                                    const float* boxes = nullptr)
{
    if (SELF && !table && n > 0) {
        char* out = static_cast<char*>(s_table);
        uint32_t* masks = reinterpret_cast<uint32_t*>(out + 32);
        if (CALL) build_box_table_call(boxes, n, out, masks);
        else build_box_table(boxes, n, out, masks);
        return BoxTable{static_cast<const char*>(s_table), n};
    }
    const float4* src = static_cast<const float4*>(table);
    float4* dst = static_cast<float4*>(s_table);
    if (n > 0)
        for (int i = threadIdx.x; i < (int)(box_table_bytes(n) / 16); i += blockDim.x) dst[i] = src[i];
    return BoxTable{static_cast<const char*>(s_table), n};
}

}  // namespace
}  // namespace rll
