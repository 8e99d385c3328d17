// Per-point light sampling shared by the single-grid kernel (sample.cu) and
// the persistent batched kernel (batched.cu): hash lookup / lazy insert, cdf
// binary search, in-cluster choice, light point, shadow test, estimate and
// learning record. See sample.cu for the method notes.
#pragma once

#include <cuda_runtime.h>

#include "box_bins.cuh"
#include "rll_device.cuh"

namespace rll {

// cluster bits of a batched record key (cut sizes up to 64)
constexpr uint32_t kBatchClusterBits = 6;

struct SampleArgs {
    const float* pos;
    const float* nrm;
    const float* albedo;
    int64_t n_points;         // plane stride of pos / nrm / rgb
    int64_t p_begin, p_end;   // points this launch shades (k_sample)
    const float* boxes;
    int n_boxes;
    const void* box_table;    // of those boxes (box_bins.cuh; n_boxes > 0)
    unsigned long long* keys;
    const uint32_t* cut;
    const void* C;
    uint32_t Hl, M, m;        // slots per resolution level, cut size, cut length
    uint32_t levels;          // resolution levels (cell size * 2^l)
    const float* footprint;   // [P] or nullptr (every point at level 0)
    const uint32_t* def_cut;
    const void* def_C;
    float origin[3];
    float h;
    uint32_t nb;
    uint32_t jitter;
    uint32_t reward_mode;
    const PairRec* pairs;
    cudaTextureObject_t tail_tex;  // the pairs' powers and ids
    const QuadRec* quads;     // two-level descent records
    cudaTextureObject_t quad_tex;  // the quads' powers and ids
    const NodeRec* nodes;
    const LightRec* lights;
    const float* light_cdf;
    int64_t n_lights;
    unsigned long long seed;
    uint32_t frame;
    int spp;
    uint32_t warp_points;     // points a warp takes at a time, a lane a sample; 0: a thread a point
    float* rgb;
    uint32_t* rec_key;
    float* rec_val;
    int32_t* dbg_light;
    float* dbg_pcut;
    float* dbg_pin;
    uint32_t* status;
    // record key encoding: 0 -> slot * M + cluster (one grid); 1 -> ((cell_base
    // + slot) << kBatchClusterBits) | cluster (many grids sorted together)
    uint32_t key_cells;
    uint32_t cell_base;
};

// Level of a point with footprint f: the smallest l with h * 2^l >= f, i.e.
// ceil(log2(f / h)) from the binary32 quotient (exponent and mantissa bits),
// clamped to [0, levels - 1]; f <= h and NaN give 0.
__device__ __forceinline__ uint32_t footprint_level(float f, float h, uint32_t levels)
{
    const float r = fdiv(f, h);
    if (!(r > 1.0f)) return 0u;
    const uint32_t b = __float_as_uint(r);
    const uint32_t l = ((b >> 23) & 0xFFu) - 127u + ((b & 0x7FFFFFu) != 0u);
    return min(l, levels - 1u);
}

// Lookup with lazy creation in the slot range of one level: linear probing
// from level * Hl + (fmix64(key) mod Hl) for at most kMaxProbes slots.
__device__ __forceinline__ int64_t lookup_insert(unsigned long long* keys, uint32_t Hl, uint32_t level,
                                                 unsigned long long key)
{
    const unsigned long long h = fmix64(key);
    for (int i = 0; i < kMaxProbes; ++i) {
        const uint32_t slot = level * Hl + (uint32_t)((h + (unsigned long long)i) & (unsigned long long)(Hl - 1));
        const unsigned long long k = __ldcg(keys + slot);
        if (k == key) return slot;
        if (k == kEmptyKey) {
            const unsigned long long old = atomicCAS(keys + slot, kEmptyKey, key);
            if (old == kEmptyKey || old == key) return slot;
        }
    }
    return -1;
}

// the geometry of two nodes
__device__ __forceinline__ NodePair load_pair(const PairRec* p)
{
    const Words8 u = ldg_words8(p), v = ldg_words8(reinterpret_cast<const char*>(p) + 32);
    auto pair = [](const Words8& w, int k) {
        return make_float2(__uint_as_float(w.w[2 * k]), __uint_as_float(w.w[2 * k + 1]));
    };
    return NodePair{pair(u, 0), pair(u, 1), pair(u, 2), pair(u, 3), pair(v, 0), pair(v, 1), pair(v, 2), v.w[6], v.w[7]};
}

__device__ __forceinline__ LightRec load_light(const LightRec* p)
{
    LightRec r;
    Words8* d = reinterpret_cast<Words8*>(&r);
    d[0] = ldg_words8(p);
    d[1] = ldg_words8(reinterpret_cast<const char*>(p) + 32);
    return r;
}

// A shadow segment's direction component: one with |d| < 2^-100 (the segment
// does not move along that axis; 1/d would be infinite and the slab planes
// undefined) is taken as 2^-100 with the sign of d. o * 2^100 is then exact,
// the planes lie at t = (b - o) 2^100 rounded, and the segment is inside that
// slab exactly when b_min < o < b_max -- the decision for a parallel segment.
__device__ __forceinline__ float seg_dir(float d)
{
    return fabsf(d) >= 0x1p-100f ? d : copysignf(0x1p-100f, d);
}

// Above the rounding error of the shadow test's slab planes (a few ulps of |o| + |y|).
__device__ __forceinline__ float shadow_margin(float o, float y) { return 1e-5f * (1.0f + fabsf(o) + fabsf(y)); }

// Whether the segment o + t d, t in (0, kShadowTmax), crosses a box (i = 1 / d, q = -o i).
__device__ __forceinline__ bool slabs_cross(const float4& bmin, const float4& bmax, float i0, float i1, float i2,
                                            float q0, float q1, float q2)
{
    const float ta0 = __fmaf_rn(bmin.x, i0, q0), tb0 = __fmaf_rn(bmax.x, i0, q0);
    const float ta1 = __fmaf_rn(bmin.y, i1, q1), tb1 = __fmaf_rn(bmax.y, i1, q1);
    const float ta2 = __fmaf_rn(bmin.z, i2, q2), tb2 = __fmaf_rn(bmax.z, i2, q2);
    float tn = fmaxf(0.0f, fminf(ta0, tb0));
    float tf = fminf(kShadowTmax, fmaxf(ta0, tb0));
    tn = fmaxf(tn, fminf(ta1, tb1));
    tf = fminf(tf, fmaxf(ta1, tb1));
    tn = fmaxf(tn, fminf(ta2, tb2));
    tf = fminf(tf, fmaxf(ta2, tb2));
    return tn < tf;
}

namespace {
// The shadow test of box sets in which a box has a minimum above its maximum: such a box counts only
// where the segment's bounding box spans it (the ends compared as they are given). The table takes it
// for the box between its ends, which is where it can meet a segment. Out of line and of no use to
// other sets: 1080p sampling 320 us with and without it, energy sampler 87 (a mark at every box, tested
// where a box blocks, cost the energy sampler 12 %; a call behind the test 2 to 5 % of the sampling).
__device__ __noinline__ bool spanned_box_blocks(BoxTable bt, float o0, float o1, float o2, float y0, float y1,
                                                float y2)
{
    const float i0 = fdiv(1.0f, seg_dir(fsub(y0, o0))), i1 = fdiv(1.0f, seg_dir(fsub(y1, o1))),
                i2 = fdiv(1.0f, seg_dir(fsub(y2, o2)));
    const float q0 = -fmul(o0, i0), q1 = -fmul(o1, i1), q2 = -fmul(o2, i2);
    const float e0 = shadow_margin(o0, y0), e1 = shadow_margin(o1, y1), e2 = shadow_margin(o2, y2);
    const float l0 = fminf(o0, y0) - e0, l1 = fminf(o1, y1) - e1, l2 = fminf(o2, y2) - e2;
    const float h0 = fmaxf(o0, y0) + e0, h1 = fmaxf(o1, y1) + e1, h2 = fmaxf(o2, y2) + e2;
    const float4* s_box = bt.boxes();
    return bt.any(l0, l1, l2, h0, h1, h2, [&](int b) {
        const float4 bmin = s_box[2 * b], bmax = s_box[2 * b + 1];
        if (bmin.x > h0 || bmax.x < l0 || bmin.y > h1 || bmax.y < l1 || bmin.z > h2 || bmax.z < l2) return false;
        return slabs_cross(bmin, bmax, i0, i1, i2, q0, q1, q2);
    });
}
}  // namespace

struct ShadeOut {
    float est[3];
    float reward;
};

// light point, shadow test, contribution (x, n: shading point and normal)
__device__ __forceinline__ ShadeOut shade(const LightRec& L, float x0, float x1, float x2, float n0, float n1,
                                          float n2, float albedo, float p_cut, float p_in, float ua, float ub,
                                          const BoxTable& bt, uint32_t reward_mode)
{
    const float su = fsqrt(ua);
    const float b0 = fsub(1.0f, su), b1 = fmul(ub, su), b2 = fsub(su, b1);
    const float y0 = fadd(fadd(fmul(b0, L.v0[0]), fmul(b1, L.v1[0])), fmul(b2, L.v2[0]));
    const float y1 = fadd(fadd(fmul(b0, L.v0[1]), fmul(b1, L.v1[1])), fmul(b2, L.v2[1]));
    const float y2 = fadd(fadd(fmul(b0, L.v0[2]), fmul(b1, L.v1[2])), fmul(b2, L.v2[2]));
    const float o0 = fadd(x0, fmul(kShadowOffset, n0));
    const float o1 = fadd(x1, fmul(kShadowOffset, n1));
    const float o2 = fadd(x2, fmul(kShadowOffset, n2));
    const float i0 = fdiv(1.0f, seg_dir(fsub(y0, o0))), i1 = fdiv(1.0f, seg_dir(fsub(y1, o1))),
                i2 = fdiv(1.0f, seg_dir(fsub(y2, o2)));
    const float q0 = -fmul(o0, i0), q1 = -fmul(o1, i1), q2 = -fmul(o2, i2);
    // Conservative prefilter: a box can only block the segment if it meets the
    // segment's bounding box widened by shadow_margin, so no box the exact
    // slab test would report is skipped and the decision is unchanged.
    const float e0 = shadow_margin(o0, y0), e1 = shadow_margin(o1, y1), e2 = shadow_margin(o2, y2);
    const float4* s_box = bt.boxes();
    auto blocks = [&](int b) { return slabs_cross(s_box[2 * b], s_box[2 * b + 1], i0, i1, i2, q0, q1, q2); };
    const bool occluded =
        bt.swapped() ? spanned_box_blocks(bt, o0, o1, o2, y0, y1, y2)
                     : bt.any(fminf(o0, y0) - e0, fminf(o1, y1) - e1, fminf(o2, y2) - e2, fmaxf(o0, y0) + e0,
                              fmaxf(o1, y1) + e1, fmaxf(o2, y2) + e2, blocks);
    ShadeOut o;
    const float wx = y0 - x0, wy = y1 - x1, wz = y2 - x2;
    const float d2 = wx * wx + wy * wy + wz * wz;
    const float inv_d = rsqrtf(d2);
    const float cx = fmaxf(0.0f, (n0 * wx + n1 * wy + n2 * wz) * inv_d);
    const float cl = fmaxf(0.0f, -(L.n[0] * wx + L.n[1] * wy + L.n[2] * wz) * inv_d);
    const float geo = (occluded || !(d2 > 0.0f)) ? 0.0f : __fdividef(cx * cl, d2);
    const float f = albedo * 0.31830988618379067f;
    const float c0 = f * L.le[0] * geo, c1 = f * L.le[1] * geo, c2 = f * L.le[2] * geo;
    // a zero contribution is zero whatever its pdf (a long-unrewarded
    // cluster's probability may underflow binary32)
    const float w = geo > 0.0f ? __fdividef(__fdividef(L.area, p_cut), p_in) : 0.0f;
    o.est[0] = c0 * w;
    o.est[1] = c1 * w;
    o.est[2] = c2 * w;
    const float lum = 0.2126f * c0 + 0.7152f * c1 + 0.0722f * c2;
    o.reward = !(lum > 0.0f) ? 0.0f : (reward_mode == RLL_REWARD_CLUSTER ? __fdividef(lum * L.area, p_in) : lum * L.area);
    return o;
}

// Cell, cluster and triangle draws of one sample (draws 0-2 and 4-8).
struct Setup {
    uint4 w2;        // Philox block 2: the last jitter draw, then the first three of the descent
    uint32_t node;   // cut node of the chosen cluster
    float p_cut;     // its probability under the cell's cdf
    float ua, ub;    // triangle point draws
    uint32_t rec;    // learning record key (kInvalidRecord if the table is full)
    int64_t slot;
    uint32_t s;
};

template <int P>
__device__ __forceinline__ Setup setup_sample(const SampleArgs& a, SampleStream& rs, float x0, float x1, float x2,
                                              float n0, float n1, float n2, uint32_t level)
{
    using T = typename Store<P>::T;
    const T* Ctab = static_cast<const T*>(a.C);
    const T* Cdef = static_cast<const T*>(a.def_C);
    const uint32_t m = a.m;
    Setup o;
    o.w2 = rs.block_words(2);
    float jit[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (a.jitter) {
        const uint4 w = rs.block_words(1);
        jit[0] = u24(w.x);
        jit[1] = u24(w.y);
        jit[2] = u24(w.z);
        jit[3] = u24(w.w);
        jit[4] = u24(o.w2.x);
    }
    const float h_cell = fmul(a.h, (float)(1u << level));  // exact: a power of two
    const unsigned long long key = cell_key(x0, x1, x2, n0, n1, n2, a.origin, h_cell, a.nb, a.jitter != 0, jit);
    const int64_t slot = lookup_insert(a.keys, a.Hl, level, key);
    const T* crow;
    const uint32_t* cutrow;
    if (slot >= 0) {
        crow = Ctab + slot * a.M;
        cutrow = a.cut + slot * a.M;
    } else {
        crow = Cdef;
        cutrow = a.def_cut;
        atomicOr(a.status, (uint32_t)RLL_E_TABLE_FULL);
    }
    // cluster: first s with C(s) > u * C(m-1)
    const float u = rs.draw(kDrawCut);
    const float total = Store<P>::load(crow[m - 1]);
    uint32_t lo = 0, hi = m - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__fmaf_rn(-u, total, Store<P>::load(crow[mid])) > 0.0f) hi = mid;
        else lo = mid + 1;
    }
    o.s = lo;
    o.slot = slot;
    const float cprev = lo > 0 ? Store<P>::load(crow[lo - 1]) : 0.0f;
    o.p_cut = (Store<P>::load(crow[lo]) - cprev) / total;
    o.node = cutrow[lo];
    if ((int64_t)o.node >= 2 * a.n_lights - 1) {  // corrupt cut row: flag, sample from the root
        atomicOr(a.status, (uint32_t)RLL_E_DEVICE);
        o.node = 0;
    }
    o.ua = rs.draw(kDrawTriA);
    o.ub = rs.draw(kDrawTriB);
    o.rec = slot < 0 ? kInvalidRecord
                     : (a.key_cells ? ((a.cell_base + (uint32_t)slot) << kBatchClusterBits) | lo
                                    : (uint32_t)slot * a.M + lo);
    return o;
}

// One level of the bound-driven descent below internal node `node` (ud: the
// level's draw; nx*: the shading point negated, n*: its normal, broadcast to
// both components). Both children's bounds in one packed evaluation; they are
// compared without a division: w_L = num_L den_R, w_R = num_R den_L; their
// powers if both vanish.
__device__ __forceinline__ void descent_step(const SampleArgs& a, uint32_t& node, float& p_in, float ud,
                                             float2 nx0, float2 nx1, float2 nx2, float2 n0, float2 n1, float2 n2)
{
    const float4 t = tex1Dfetch<float4>(a.tail_tex, (int)node);  // powers, then ids
    const Bound2 b = importance2(load_pair(a.pairs + node), make_float2(t.x, t.y), nx0, nx1, nx2, n0, n1, n2);
    float wl = fmul(b.num.x, b.den.y), wr = fmul(b.num.y, b.den.x);
    float ssum = fadd(wl, wr);
    if (!(ssum > 0.0f)) {
        wl = t.x;
        wr = t.y;
        ssum = fadd(wl, wr);
    }
    bool left;
    float ratio;
    if (ssum > 0.0f) {
        left = __fmaf_rn(ud, ssum, -wl) < 0.0f;
        ratio = __fdividef(left ? wl : wr, wl + wr);  // continuous: pdf only
    } else {
        left = ud < 0.5f;
        ratio = 0.5f;
    }
    p_in *= ratio;
    node = __float_as_uint(left ? t.z : t.w);
}

// One step of the two-level descent below internal node `node` (ud: the
// step's draw): its candidates (2 to 4 valid, in light order, the valid ones
// first), weights num / max(den, 1e-30), binary32 prefix sums in order; the first
// prefix above u * S is chosen (exact, one fma), probability (P_i -
// P_{i-1}) / S; powers, then uniform over the valid candidates, when all
// weights vanish. Two candidates a bound, from four 32-byte loads and two
// texels (one candidate a bound from twelve 16-byte loads of 48-byte records:
// 1 601 x 901 points, binary16 tables: 369 us a pass, now 312).
__device__ __forceinline__ void descent2_step(const SampleArgs& a, uint32_t& node, float& p_in, float ud, float2 nx0,
                                              float2 nx1, float2 nx2, float2 n0, float2 n1, float2 n2)
{
    const float4 phi = tex1Dfetch<float4>(a.quad_tex, (int)(2 * node));
    const float4 idf = tex1Dfetch<float4>(a.quad_tex, (int)(2 * node + 1));
    const uint32_t id[4] = {__float_as_uint(idf.x), __float_as_uint(idf.y), __float_as_uint(idf.z),
                            __float_as_uint(idf.w)};
    const QuadRec* q = a.quads + node;
    const Bound2 b0 = importance2(load_pair(&q->pair[0]), make_float2(phi.x, phi.y), nx0, nx1, nx2, n0, n1, n2);
    const Bound2 b1 = importance2(load_pair(&q->pair[1]), make_float2(phi.z, phi.w), nx0, nx1, nx2, n0, n1, n2);
    const int k = 2 + (id[2] != 0xFFFFFFFFu) + (id[3] != 0xFFFFFFFFu);
    const float w[4] = {fdiv(b0.num.x, fmaxf(b0.den.x, 1e-30f)), fdiv(b0.num.y, fmaxf(b0.den.y, 1e-30f)),
                        fdiv(b1.num.x, fmaxf(b1.den.x, 1e-30f)), fdiv(b1.num.y, fmaxf(b1.den.y, 1e-30f))};
    float pre[4], S = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        S = fadd(S, i < k ? w[i] : 0.0f);
        pre[i] = S;
    }
    if (!(S > 0.0f)) {  // rare: the candidates' powers
        const float power[4] = {phi.x, phi.y, phi.z, phi.w};
        S = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            S = fadd(S, i < k ? power[i] : 0.0f);
            pre[i] = S;
        }
    }
    int pick;
    if (S > 0.0f) {
        pick = k - 1;
#pragma unroll
        for (int i = 3; i >= 0; --i)
            if (i < k && __fmaf_rn(ud, S, -pre[i]) < 0.0f) pick = i;
    } else {
        const uint32_t u24v = (uint32_t)(ud * 16777216.0f);
        pick = (int)(((unsigned long long)u24v * (unsigned long long)k) >> 24);
    }
    // the chosen candidate's interval and id by selects (no indexed arrays)
    float lo = 0.0f, hi = pre[0];
    node = id[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) {
        if (pick == i) {
            lo = pre[i - 1];
            hi = pre[i];
            node = id[i];
        }
    }
    p_in *= S > 0.0f ? (hi - lo) / S : 1.0f / (float)k;  // continuous: pdf only
}

// Light index of the node a descent ended on. A descent that ran into the
// depth bound (only on a corrupt tree: no builder comes near it) is flagged
// and takes the first light of the node it reached.
__device__ __forceinline__ int64_t leaf_or_flag(const SampleArgs& a, uint32_t node, int64_t nl1)
{
    if ((int64_t)node >= nl1) return (int64_t)node - nl1;
    atomicOr(a.status, (uint32_t)RLL_E_DEVICE);
    return (int64_t)a.nodes[node].begin;
}

// One shading point of the G-buffer and the grid level of its footprint.
struct Point {
    float x0, x1, x2, n0, n1, n2, alb;
    uint32_t level;
};
__device__ __forceinline__ Point load_point(const SampleArgs& a, int64_t p)
{
    const int64_t np = a.n_points;
    return Point{a.pos[p], a.pos[np + p], a.pos[2 * np + p], a.nrm[p], a.nrm[np + p], a.nrm[2 * np + p], a.albedo[p],
                 a.footprint ? footprint_level(__ldg(a.footprint + p), a.h, a.levels) : 0u};
}

// Sample `sid` of a shading point, one thread: its estimate in est, its learning record and
// diagnostics to their arrays.
template <int P, int MODE, bool DBG>
__device__ __forceinline__ void sample_one(const SampleArgs& a, const Point& pt, uint32_t sid, const BoxTable& bt,
                                           float est[3])
{
    const float x0 = pt.x0, x1 = pt.x1, x2 = pt.x2, n0 = pt.n0, n1 = pt.n1, n2 = pt.n2, alb = pt.alb;
    const uint32_t level = pt.level;
    const int64_t nl1 = a.n_lights - 1;
    const uint32_t nl1u = (uint32_t)nl1;  // internal node ids are below it (at most 2^24 lights)
    SampleStream rs;
    rs.init(a.seed, sid, a.frame);
    const Setup su = setup_sample<P>(a, rs, x0, x1, x2, n0, n1, n2, level);
    uint32_t node = su.node;
    float p_in = 1.0f;
    int64_t light;
    const float2 vn0 = make_float2(n0, n0), vn1 = make_float2(n1, n1), vn2 = make_float2(n2, n2);
    const float2 vx0 = make_float2(-x0, -x0), vx1 = make_float2(-x1, -x1), vx2 = make_float2(-x2, -x2);
    if (MODE == RLL_MODE_UNIFORM) {
        const NodeRec& r = a.nodes[node];
        const uint32_t w = r.end - r.begin;
        const uint32_t u24v = (uint32_t)(rs.draw(kDrawUniform) * 16777216.0f);
        light = (int64_t)r.begin + (int64_t)(((unsigned long long)u24v * w) >> 24);
        p_in = 1.0f / (float)w;
    } else if (MODE == RLL_MODE_DESCENT2) {
        // step l takes draw kDrawDescent + l, one copy of the step, the words rotated
        uint4 w = su.w2;
#pragma unroll 1
        for (uint32_t l = 0; node < nl1u && l < (uint32_t)kMaxTreeDepth; ++l) {
            const uint32_t k = (kDrawDescent + l) & 3u;
            if (k == 0) w = rs.block_words((kDrawDescent + l) >> 2);
            const float ud = u24(k == 0 ? w.x : w.y);
            if (k != 0) w = make_uint4(0u, w.z, w.w, 0u);
            descent2_step(a, node, p_in, ud, vx0, vx1, vx2, vn0, vn1, vn2);
        }
        light = leaf_or_flag(a, node, nl1);
    } else {
        // Level l takes draw kDrawDescent + l: words 1..3 of Philox block 2, then four levels per block.
        // Five copies of the step in all: the first three levels share one, the rest are unrolled so
        // that every word index is a constant. The kernel's length counts: with seven copies, each
        // with the library's square roots in line, a warp's instruction fetches missed the SM's cache
        // (1080p, 4K and sky-dome sampling 331, 1 596 and 492 us; now 314, 1 537 and 431; four copies:
        // 322, 1 574, 443; one: 330, 1 608, 443).
        static_assert(kDrawDescent == 9, "descent draws start at word 1 of block 2");
        uint4 w = su.w2;
#pragma unroll 1
        for (int k = 0; k < 3 && node < nl1u; ++k) {
            descent_step(a, node, p_in, u24(w.y), vx0, vx1, vx2, vn0, vn1, vn2);
            w = make_uint4(0u, w.z, w.w, 0u);
        }
        for (uint32_t b = 3; node < nl1u && b < (uint32_t)(kMaxTreeDepth / 4); ++b) {
            w = rs.block_words(b);
            descent_step(a, node, p_in, u24(w.x), vx0, vx1, vx2, vn0, vn1, vn2);
            if (node < nl1u) descent_step(a, node, p_in, u24(w.y), vx0, vx1, vx2, vn0, vn1, vn2);
            if (node < nl1u) descent_step(a, node, p_in, u24(w.z), vx0, vx1, vx2, vn0, vn1, vn2);
            if (node < nl1u) descent_step(a, node, p_in, u24(w.w), vx0, vx1, vx2, vn0, vn1, vn2);
        }
        light = leaf_or_flag(a, node, nl1);
    }
    const LightRec Lr = load_light(a.lights + light);
    const ShadeOut o = shade(Lr, x0, x1, x2, n0, n1, n2, alb, su.p_cut, p_in, su.ua, su.ub, bt, a.reward_mode);
    est[0] = o.est[0];
    est[1] = o.est[1];
    est[2] = o.est[2];
    if (a.rec_key) {
        a.rec_key[sid] = su.rec;
        a.rec_val[sid] = o.reward;
    }
    if (DBG) {
        if (a.dbg_light) a.dbg_light[sid] = (int32_t)light;
        if (a.dbg_pcut) a.dbg_pcut[sid] = su.p_cut;
        if (a.dbg_pin) a.dbg_pin[sid] = p_in;
    }
}

// All samples of shading point p, one thread.
template <int P, int MODE, bool DBG>
__device__ __forceinline__ void sample_point(const SampleArgs& a, int64_t p, const BoxTable& bt)
{
    const int64_t np = a.n_points;
    const Point pt = load_point(a, p);
    float acc[3] = {0.0f, 0.0f, 0.0f};
    for (int j = 0; j < a.spp; ++j) {
        float est[3];
        sample_one<P, MODE, DBG>(a, pt, (uint32_t)(p * a.spp + j), bt, est);
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[k] += est[k];
    }
    const float inv_spp = 1.0f / (float)a.spp;
#pragma unroll
    for (int k = 0; k < 3; ++k) a.rgb[k * np + p] = acc[k] * inv_spp;
}

// Floats of shared memory that a warp of sample_points needs: a round's estimates, and the sums of
// the point that a round ends in, in one place for even rounds and one for odd ones (a round reads
// the one before's while other lanes write its own).
constexpr int kWarpEst = 3 * 32 + 2 * 3;

// How a launch of n_points points of spp samples on a device that holds `warps` warps splits them:
// the points a warp of sample_points takes at a time, or 0 for a thread a point. The cost of a split
// is a warp's rounds (of 32 lanes, spp samples one after another with a thread a point) times the
// waves of warps, and half a wave for the last one; a round of sample_points costs about 5 % more
// than a sample of each of 32 points (its sums, and samples of one point in a warp share no more
// cache lines than neighbouring points do). Sampling in us, sample_points / a thread a point, 64K
// lights: 2 samples of 20K, 160K, 1.28M points 26 / 35, 74 / 83, 476 / 465; 7 of 20K 45 / 108; 16 of
// 20K, 80K, 320K 72 / 230, 225 / 313, 860 / 1003.
inline uint32_t lane_split(int64_t n_points, int spp, int64_t warps)
{
    if (spp == 1) return 0u;
    auto cost = [&](uint32_t points, double rounds) {
        const double waves = (double)((n_points + points - 1) / points) / (double)warps;
        return rounds * ((waves > 0.5 ? waves : 0.5) + 0.5);
    };
    uint32_t best = 0;
    double least = cost(32, spp);
    for (uint32_t k = 1; k <= 32; k *= 2) {
        const double c = 1.05 * cost(k, (double)(((int64_t)k * spp + 31) / 32));
        if (c < least) {
            least = c;
            best = k;
        }
    }
    return best;
}

// All samples of `count` consecutive shading points from p0 (count <= warp_points), by one warp: a
// lane a sample, 32 consecutive samples a round, so that few points of many samples still
// fill the device, a round's lanes share their points' cells and the records are written side by
// side. A point's estimates are summed in sample order, by a lane a point and channel, through s_est
// (kWarpEst floats of this warp's) across rounds: the same sums as one thread a point makes.
// (Whole passes: 200 x 120 points at 64 samples, 256-leaf cuts, 1 010 -> 458 us: a thread a point put
// 1.2 blocks on an SM; 64 x 64 points at 4 samples 59 -> 48 us.)
template <int P, int MODE, bool DBG>
__device__ __forceinline__ void sample_points(const SampleArgs& a, int64_t p0, uint32_t count, const BoxTable& bt,
                                              float* s_est)
{
    const int64_t np = a.n_points;
    const uint32_t lane = threadIdx.x & 31u, spp = (uint32_t)a.spp, total = count * spp;
    const float inv_spp = 1.0f / (float)a.spp;
#pragma unroll 1
    for (uint32_t base = 0; base < total; base += 32) {
        const uint32_t i = base + lane;
        float est[3] = {0.0f, 0.0f, 0.0f};
        if (i < total) sample_one<P, MODE, DBG>(a, load_point(a, p0 + i / spp), (uint32_t)(p0 * a.spp) + i, bt, est);
#pragma unroll
        for (int k = 0; k < 3; ++k) s_est[32 * k + lane] = est[k];
        __syncwarp();
        const uint32_t end = min(base + 32, total), q0 = base / spp, q1 = (end - 1) / spp;
        const uint32_t carry = 96 + 3 * ((base >> 5) & 1u), before = 96 + 99 - carry;
        for (uint32_t t = lane; t < 3 * (q1 - q0 + 1); t += 32) {
            const uint32_t q = q0 + t / 3, ch = t % 3;
            const uint32_t from = max(q * spp, base), to = min((q + 1) * spp, end);
            float acc = from == q * spp ? 0.0f : s_est[before + ch];
            for (uint32_t j = from; j < to; ++j) acc += s_est[32 * ch + (j - base)];
            if (to == (q + 1) * spp) a.rgb[ch * np + p0 + q] = acc * inv_spp;
            else s_est[carry + ch] = acc;
        }
        __syncwarp();
    }
}

}  // namespace rll
