// Render-time sampling (Section 3, "Main contribution"; Section 3.1: "sampling
// the cdf is performed by a standard binary search").
//
// One thread per shading point, its samples in turn, or a lane per sample
// (Split, below); occluder boxes staged in shared memory once per block. Per
// sample:
//   hash lookup / lazy insert of the (jittered) 5-d cell   (64-bit CAS)
//   binary search of the cell's C for the cluster s        (log2 m loads of one row)
//   in-cluster choice: bound-driven descent (a 64 + 16-byte record of both
//   children per level, both bounds in packed f32x2 arithmetic) or a uniform
//   pick over the cluster's lights
//   uniform point on the light triangle, contribution, shadow segment vs the
//   boxes that can meet it (box_bins.cuh)
//   estimate accumulation and one learning record (key, |c|).
// The decisions (cell, branch, visibility) are exact binary32 formulas; the
// cdf and descent comparisons u * total < c are made exactly with one fma.

#include <cuda_runtime.h>

#include "rll_device.cuh"
#include "rll_internal.h"
#include "sample_core.cuh"

namespace rll {
namespace {

// of the energy sampler: 72 registers a thread at four blocks an SM (256 threads with 64 registers spill:
// 64K lights, 64 boxes, 4 samples a point at 1080p 298 us, now 294)
constexpr int kThreads = 224;

// THREADS x MINB: block size and the resident blocks per SM the registers are
// held to (128 x 8: 64 registers, 32 warps per SM; 128 x 6: 80 registers).
// Blocks of 128 rather than 256 threads at the same occupancy: a block's
// slowest descent holds fewer lanes back (measured 1 % faster; 64-thread
// blocks lose it again to staging the boxes twice as often).
// How a launch splits its samples. ONE: one sample a point, a thread a point (without sample_point's
// loop: 1080p sampling 359 -> 343 us). LOOP: a thread a point, its samples in turn. LANES: a lane a
// sample (sample_points).
enum Split { ONE, LOOP, LANES };

template <int P, int MODE, bool DBG, int SPLIT, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_sample(SampleArgs a)
{
    pdl_begin();
    extern __shared__ float4 s_boxes[];
    const BoxTable bt = stage_box_table<SPLIT != LOOP, true>(s_boxes, a.box_table, a.n_boxes, a.boxes);
    if constexpr (SPLIT == LANES) {
        __shared__ float s_est[THREADS / 32][kWarpEst];
        __syncthreads();
        const uint32_t warp = threadIdx.x >> 5;
        const int64_t p0 = a.p_begin + ((int64_t)blockIdx.x * (THREADS / 32) + warp) * a.warp_points;
        if (p0 < a.p_end)
            sample_points<P, MODE, DBG>(a, p0, (uint32_t)min((int64_t)a.warp_points, a.p_end - p0), bt, s_est[warp]);
    } else {
        __syncthreads();
        const int64_t p = a.p_begin + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (p >= a.p_end) return;
        if constexpr (SPLIT == ONE) {
            float est[3];
            sample_one<P, MODE, DBG>(a, load_point(a, p), (uint32_t)p, bt, est);
#pragma unroll
            for (int k = 0; k < 3; ++k) a.rgb[k * a.n_points + p] = est[k];
        } else {
            sample_point<P, MODE, DBG>(a, p, bt);
        }
    }
}

// Energy-based baseline (Section 4): inversion of the cdf of leaf power, by the binary search over all
// lights whose first kPowerLevels probes, the same for every sample up to their outcomes, each block
// keeps in shared memory as a heap (node h's children 2h, where the probe is above the draw, and 2h +
// 1): probes of so long an array are gathers of one sector each (64K lights, 4 samples a point,
// 1080p: 392 us -> 318). The blocks are those that fit the device and stride over the points, so that
// each builds heap and box table once and the launch needs no table of the context's (311 -> 292 us).
constexpr int kPowerLevels = 9;  // 2 KB beside the box table of up to 45 KB

__global__ void __launch_bounds__(kThreads, 4) k_sample_power(SampleArgs a, int32_t* light_out)
{
    pdl_begin();
    extern __shared__ float4 s_boxes[];
    __shared__ float s_probe[1 << kPowerLevels];
    const BoxTable bt = stage_box_table<true>(s_boxes, nullptr, a.n_boxes, a.boxes);
    const uint32_t last = (uint32_t)a.n_lights - 1u;
    for (uint32_t h = 1 + threadIdx.x; h < (1u << kPowerLevels); h += blockDim.x) {
        uint32_t lo = 0, hi = last;
        for (int b = 30 - __clz((int)h); b >= 0 && lo < hi; --b) {  // the way to h from the root
            const uint32_t mid = (lo + hi) >> 1;
            if (h >> b & 1u) lo = mid + 1;
            else hi = mid;
        }
        s_probe[h] = a.light_cdf[(lo + hi) >> 1];  // unused where the search has ended
    }
    __syncthreads();
    const int64_t np = a.n_points;
    const float total = a.light_cdf[last];
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < np; p += (int64_t)gridDim.x * blockDim.x) {
        const float x0 = a.pos[p], x1 = a.pos[np + p], x2 = a.pos[2 * np + p];
        const float n0 = a.nrm[p], n1 = a.nrm[np + p], n2 = a.nrm[2 * np + p];
        const float alb = a.albedo[p];
        float acc0 = 0.0f, acc1 = 0.0f, acc2 = 0.0f;
        for (int j = 0; j < a.spp; ++j) {
            const uint32_t sid = (uint32_t)(p * a.spp + j);
            SampleStream rs;
            rs.init(a.seed, sid, a.frame);
            const float u = rs.draw(kDrawCut);
            uint32_t lo = 0, hi = last, h = 1;
            for (int l = 0; l < kPowerLevels && lo < hi; ++l) {
                const uint32_t mid = (lo + hi) >> 1;
                const bool above = __fmaf_rn(-u, total, s_probe[h]) > 0.0f;
                h = 2 * h + !above;
                if (above) hi = mid;
                else lo = mid + 1;
            }
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                if (__fmaf_rn(-u, total, a.light_cdf[mid]) > 0.0f) hi = mid;
                else lo = mid + 1;
            }
            const float pl = a.nodes[last + lo].phi / total;
            const LightRec Lr = load_light(a.lights + lo);
            const ShadeOut o = shade(Lr, x0, x1, x2, n0, n1, n2, alb, pl, 1.0f, rs.draw(kDrawTriA), rs.draw(kDrawTriB),
                                     bt, 0);
            acc0 += o.est[0];
            acc1 += o.est[1];
            acc2 += o.est[2];
            if (light_out) light_out[sid] = (int32_t)lo;
        }
        const float inv_spp = 1.0f / (float)a.spp;
        a.rgb[p] = acc0 * inv_spp;
        a.rgb[np + p] = acc1 * inv_spp;
        a.rgb[2 * np + p] = acc2 * inv_spp;
    }
}

// The table of the occluder boxes (box_bins.cuh), one block.
__global__ void __launch_bounds__(256) k_box_table(const float* __restrict__ boxes, int n, char* __restrict__ out)
{
    pdl_begin();
    build_box_table_global(boxes, n, out);
}

template <int P, int MODE, bool DBG, int SPLIT, int THREADS, int MINB>
cudaError_t launch(const SampleArgs& a, cudaStream_t s)
{
    const int64_t per_block = SPLIT == LANES ? (int64_t)(THREADS / 32) * a.warp_points : THREADS;
    const unsigned blocks = (unsigned)((a.p_end - a.p_begin + per_block - 1) / per_block);
    const size_t smem = a.n_boxes ? box_table_bytes(a.n_boxes) : 0;
    return launch_pdl(k_sample<P, MODE, DBG, SPLIT, THREADS, MINB>, dim3(blocks), dim3(THREADS), smem, s, a);
}

template <int P, int MODE>
cudaError_t launch_m(const SampleArgs& a, bool dbg, int minb, cudaStream_t s)
{
    if (dbg) return launch<P, MODE, true, LOOP, 256, 3>(a, s);
    if (a.warp_points)
        return minb == 4 ? launch<P, MODE, false, LANES, 128, 8>(a, s) : launch<P, MODE, false, LANES, 128, 6>(a, s);
    if (a.spp == 1)
        return minb == 4 ? launch<P, MODE, false, ONE, 128, 8>(a, s) : launch<P, MODE, false, ONE, 128, 6>(a, s);
    return minb == 4 ? launch<P, MODE, false, LOOP, 128, 8>(a, s) : launch<P, MODE, false, LOOP, 128, 6>(a, s);
}

template <int P>
cudaError_t launch_p(const SampleArgs& a, int mode, bool dbg, int minb, cudaStream_t s)
{
    if (mode == RLL_MODE_UNIFORM) return launch_m<P, RLL_MODE_UNIFORM>(a, dbg, minb, s);
    if (mode == RLL_MODE_DESCENT2) return launch_m<P, RLL_MODE_DESCENT2>(a, dbg, minb, s);
    return launch_m<P, RLL_MODE_DESCENT>(a, dbg, minb, s);
}

}  // namespace

int sample_and_shade(rll_ctx* ctx, rll_grid* g, const rll_tree* t, const float* pos, const float* nrm,
                     const float* albedo, const float* footprint, int64_t n_points, const float* boxes, int n_boxes,
                     uint64_t seed,
                     uint32_t frame, int spp, float* rgb, uint32_t* rec_key, float* rec_val,
                     const rll_sample_debug* dbg)
{
    // Up to 64 boxes and one wave of blocks: each block builds the boxes' table for itself, about as
    // long as a block alone takes, but without a launch (64x64 points: 42 -> 39 us a pass). Sampling of
    // 4 096 points at 1, 64, 65, 256 and 512 boxes with the launch 14.1, 17.0, 17.1, 29.4, 50.6 us,
    // without 12.9, 16.0, 16.1, 27.1, 47.6; of 150 000 points, about a wave, two runs of one side differ
    // by more than the sides do. The line lies at the boxes of one mask word, on the safe side of where
    // every block's own build would cost a full wave more. In larger launches the copies do.
    const uint32_t warp_points = lane_split(n_points, spp, 32 * (int64_t)device_sm_count(ctx->device));
    const int64_t warps = warp_points ? (n_points + warp_points - 1) / warp_points : (n_points + 31) / 32;
    const bool loop = (spp > 1 && !warp_points) || (dbg && (dbg->light || dbg->p_cut || dbg->p_in));
    const bool self = !loop && n_boxes <= 64 && warps <= 32 * (int64_t)device_sm_count(ctx->device);
    const void* table = nullptr;
    const int rc = self ? RLL_OK : box_table(ctx, boxes, n_boxes, ctx->stream, &table);
    if (rc != RLL_OK) return rc;
    return sample_and_shade_range(ctx, g, t, pos, nrm, albedo, footprint, n_points, 0, n_points, boxes, n_boxes, seed,
                                  frame, spp, rgb, rec_key, rec_val, dbg, ctx->stream, table);
}

int box_table(rll_ctx* ctx, const float* boxes, int n_boxes, cudaStream_t stream, const void** out)
{
    *out = nullptr;
    if (n_boxes <= 0) return RLL_OK;
    const int rc = check_cuda(ctx,
                              launch_pdl(k_box_table, dim3(1), dim3(256), 0, stream, boxes, n_boxes,
                                         static_cast<char*>(ctx->box_table)),
                              "box table");
    if (rc == RLL_OK) *out = ctx->box_table;
    return rc;
}

int sample_and_shade_range(rll_ctx* ctx, rll_grid* g, const rll_tree* t, const float* pos, const float* nrm,
                           const float* albedo, const float* footprint, int64_t n_points, int64_t p_begin,
                           int64_t p_end, const float* boxes, int n_boxes, uint64_t seed, uint32_t frame, int spp,
                           float* rgb, uint32_t* rec_key, float* rec_val, const rll_sample_debug* dbg,
                           cudaStream_t stream, const void* table)
{
    if (p_end <= p_begin) return RLL_OK;
    SampleArgs a{};
    a.box_table = table;
    a.pos = pos;
    a.nrm = nrm;
    a.albedo = albedo;
    a.n_points = n_points;
    a.p_begin = p_begin;
    a.p_end = p_end;
    a.boxes = boxes;
    a.n_boxes = n_boxes;
    a.keys = g->keys;
    a.cut = g->cut;
    a.C = g->C;
    a.Hl = g->Hl;
    a.levels = g->levels;
    a.footprint = footprint;
    a.M = g->M;
    a.m = g->m;
    a.def_cut = g->def_cut;
    a.def_C = g->def_C;
    for (int k = 0; k < 3; ++k) a.origin[k] = g->p.origin[k];
    a.h = g->p.cell_size;
    a.nb = g->p.normal_bins;
    a.jitter = g->p.jitter;
    a.reward_mode = g->p.reward_mode;
    a.pairs = t->pairs;
    a.tail_tex = t->tail_tex;
    a.quads = t->quads;
    a.quad_tex = t->quad_tex;
    a.nodes = t->nodes;
    a.lights = t->lights;
    a.light_cdf = t->light_cdf;
    a.n_lights = t->n;
    a.seed = seed;
    a.frame = frame;
    a.spp = spp;
    a.warp_points = lane_split(p_end - p_begin, spp, 32 * (int64_t)device_sm_count(ctx->device));
    a.rgb = rgb;
    a.rec_key = rec_key;
    a.rec_val = rec_val;
    a.status = ctx->d_status;
    const bool use_dbg = dbg && (dbg->light || dbg->p_cut || dbg->p_in);
    if (use_dbg) {
        a.dbg_light = dbg->light;
        a.dbg_pcut = dbg->p_cut;
        a.dbg_pin = dbg->p_in;
    }
    cudaError_t e;
    const int minb = ctx->sample_min_blocks;
    const int mode = g->p.in_cluster_mode;
    switch (g->p.precision) {
    case RLL_PREC_FP16: e = launch_p<RLL_PREC_FP16>(a, mode, use_dbg, minb, stream); break;
    case RLL_PREC_BF16: e = launch_p<RLL_PREC_BF16>(a, mode, use_dbg, minb, stream); break;
    default: e = launch_p<RLL_PREC_FP32>(a, mode, use_dbg, minb, stream);
    }
    return check_cuda(ctx, e, "sample_and_shade");
}

int sample_power(rll_ctx* ctx, const rll_tree* t, const float* pos, const float* nrm, const float* albedo,
                 int64_t n_points, const float* boxes, int n_boxes, uint64_t seed, uint32_t frame, int spp,
                 float* rgb, int32_t* light_out)
{
    if (n_points == 0) return RLL_OK;
    SampleArgs a{};
    a.pos = pos;
    a.nrm = nrm;
    a.albedo = albedo;
    a.n_points = n_points;
    a.boxes = boxes;
    a.n_boxes = n_boxes;
    a.nodes = t->nodes;
    a.lights = t->lights;
    a.light_cdf = t->light_cdf;
    a.n_lights = t->n;
    a.seed = seed;
    a.frame = frame;
    a.spp = spp;
    a.rgb = rgb;
    const size_t smem = n_boxes ? box_table_bytes(n_boxes) : 0;
    const unsigned blocks = resident_blocks(ctx, k_sample_power, n_points, kThreads, smem);
    return check_cuda(ctx, launch_pdl(k_sample_power, dim3(blocks), dim3(kThreads), smem, ctx->stream, a, light_out),
                      "sample_power");
}

}  // namespace rll
