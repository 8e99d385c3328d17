// Device-side building blocks of the GB300 Reinforcement Lightcuts Learning
// library: record layouts, Philox4x32-10, the binary32 decision arithmetic,
// table storage formats.
//
// Decision arithmetic. Every floating-point value that decides an integer
// (hash cell, Morton code, descent branch, shadow test, split choice) is
// evaluated with explicitly rounded binary32 intrinsics (__fadd_rn, __fmul_rn,
// ...), so that no multiply-add is contracted and the result is the IEEE
// value of the stated formula. Continuous quantities (contribution, pdf,
// reward) use ordinary fp32 arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "../../include/rll.h"

namespace rll {

constexpr unsigned long long kEmptyKey = 0xFFFFFFFFFFFFFFFFull;
constexpr uint32_t kInvalidRecord = 0xFFFFFFFFu;
constexpr int kMaxProbes = 64;
constexpr int kMaxCut = 256;
// Bound of every walk over the light tree: far above any builder's depth (radix tree of 64-bit
// keys: <= 64 levels; SAOH: < 250 levels at 2^24 lights; median: ceil(log2 n)).
constexpr int kMaxTreeDepth = 4096;
constexpr int kMaxBoxes = 1024;
constexpr uint32_t kMaxSplitIterations = 256;
constexpr float kShadowOffset = 1e-4f;
constexpr float kShadowTmax = 0.9999f;

// Node bounds record, 64 bytes (every node: export, uniform in-cluster
// choice, split-collapse).
struct __align__(16) NodeRec {
    float bmin[3];
    float bmax[3];
    float phi;       // power bound: sum over lights of lum(Le) * area
    float axis[3];   // orientation cone axis
    float cos_t;     // orientation cone: cos of the half angle
    uint32_t id;     // node id (leaf of sorted light l: n - 1 + l)
    uint32_t begin;  // first sorted light
    uint32_t end;    // one past the last sorted light
};
static_assert(sizeof(NodeRec) == 64, "NodeRec must be 64 bytes");

// Descent constants of a node: the importance bound's, precomputed (binary32,
// same operations as on the fly).
struct DescRec {
    float c[3];      // AABB centre
    float r2;        // squared half diagonal
    float r;         // half diagonal
    float phi;       // power bound
    float axis[3];   // cone axis
    float cos_t;     // cone cos(theta)
    float sin_t;     // cone sin(theta)
    uint32_t id;     // node id
};

// The DescRec fields of both children of one internal node, interleaved
// (x: left child, y: right child) so that a load yields packed operands of
// the paired bound below: 64 bytes of geometry, two 256-bit loads, and 16
// bytes of powers and ids in an array of their own. r2 is r r, formed at use;
// cs holds (1 - cos theta, sin theta) of each child as two binary16 values
// (exactly the DescRec values; cos theta = 1 - v is exact).
// The sampling kernel was bound by the L1's gather rate: a divergent load
// costs about a cycle per distinct 32-byte sector and instruction (measured
// with 32 random records a warp: 123 cycles as five 16-byte loads of one
// 80-byte record, 107 as 64 + 16 bytes with 256-bit loads), and its load pipe
// was 89 % busy. The powers and ids go through the texture path, whose data
// stage works beside the load pipe (85 -> 75 % busy). 1080p sampling 395 us
// (80-byte records) -> 382 (wide loads) -> 359 (and the texture path); 4K
// bfloat16 1 850 -> 1 764 -> 1 667 us.
struct __align__(32) PairRec {
    float2 c0, c1, c2, r;
    float2 a0, a1, a2;
    uint2 cs;
};
static_assert(sizeof(PairRec) == 64, "PairRec must be 64 bytes");
struct __align__(16) PairTail {
    float phi[2];
    uint32_t id[2];
};
static_assert(sizeof(PairTail) == 16, "PairTail must be 16 bytes");

// The two-level descent's candidates below one internal node, two and two as
// above, and their powers and ids (two texels).
struct __align__(32) QuadRec {
    PairRec pair[2];
};
struct __align__(16) QuadTail {
    float phi[4];
    uint32_t id[4];
};
static_assert(sizeof(QuadRec) == 128 && sizeof(QuadTail) == 32, "two-level record sizes");

// Sorted light, 64 bytes (two 256-bit loads).
struct __align__(32) LightRec {
    float v0[3];
    float v1[3];
    float v2[3];
    float le[3];     // current RGB radiance
    float n[3];      // unit winding normal
    float area;
};
static_assert(sizeof(LightRec) == 64, "LightRec must be 64 bytes");

// ---------------------------------------------------------------- exact ops
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fsqrt(float a) { return __fsqrt_rn(a); }

// 32 bytes by one load instruction (p 32-byte aligned, not written while the kernel runs)
struct __align__(32) Words8 {
    uint32_t w[8];
};
__device__ __forceinline__ Words8 ldg_words8(const void* p)
{
    Words8 v;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]),
          "=r"(v.w[7])
        : "l"(p));
    return v;
}

// ---------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon et al., SC'11): 10 rounds, multipliers 0xD2511F53 and
// 0xCD9E8D57, key bumped by 0x9E3779B9 / 0xBB67AE85 between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x);
        const uint32_t lo1 = 0xCD9E8D57u * c.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

// uniform in [0, 1): top 24 bits times 2^-24 (exact in binary32)
__device__ __forceinline__ float u24(uint32_t x) { return __uint2float_rn(x >> 8) * 0x1p-24f; }

// Draw layout of one light sample: draw i is word (i mod 4) of
// Philox(counter = (sample id, frame, i / 4, 0), key = (seed lo, seed hi)).
//   0 cut search, 1-2 triangle point, 3 uniform in-cluster choice,
//   4-7 jitter x, y, z, normal u, 8 jitter normal v, 9 + k descent level k.
enum : uint32_t {
    kDrawCut = 0, kDrawTriA = 1, kDrawTriB = 2, kDrawUniform = 3, kDrawJit = 4, kDrawDescent = 9
};

struct SampleStream {
    uint2 key;
    uint32_t sample_id, frame;
    uint32_t block;
    uint4 words;

    __device__ __forceinline__ void init(unsigned long long seed, uint32_t sid, uint32_t fr)
    {
        key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
        sample_id = sid;
        frame = fr;
        block = 0xFFFFFFFFu;
    }
    // the four words of Philox block b (draws 4b .. 4b + 3)
    __device__ __forceinline__ uint4 block_words(uint32_t b)
    {
        if (b != block) {
            words = philox4x32_10(make_uint4(sample_id, frame, b, 0u), key);
            block = b;
        }
        return words;
    }
    __device__ __forceinline__ float draw(uint32_t i)
    {
        const uint32_t b = i >> 2;
        if (b != block) {
            words = philox4x32_10(make_uint4(sample_id, frame, b, 0u), key);
            block = b;
        }
        const uint32_t k = i & 3u;
        const uint32_t w = k == 0 ? words.x : (k == 1 ? words.y : (k == 2 ? words.z : words.w));
        return u24(w);
    }
};

// ---------------------------------------------------------------- hashing
// MurmurHash3 64-bit finaliser (Appleby).
__device__ __forceinline__ unsigned long long fmix64(unsigned long long k)
{
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k;
}

__device__ __forceinline__ uint32_t quant_pos(float p, float o, float h, bool jit, float u)
{
    float t = fdiv(fsub(p, o), h);
    if (jit) t = fadd(t, fsub(u, 0.5f));
    float f = floorf(t);
    f = fminf(fmaxf(f, -32767.0f), 32766.0f);
    return (uint32_t)((int)f + 32768);
}

__device__ __forceinline__ uint32_t quant_nrm(float a, uint32_t nb, bool jit, float u)
{
    float q = fmul(fmul(fadd(a, 1.0f), 0.5f), (float)nb);
    if (jit) q = fadd(q, fsub(u, 0.5f));
    float f = floorf(q);
    f = fminf(fmaxf(f, 0.0f), (float)(nb - 1));
    return (uint32_t)f;
}

// 5-d cell key: 16-bit biased x, y, z cells, 8-bit octahedral normal bins
// (y up). Never equals kEmptyKey (the top byte is at most 254).
__device__ __forceinline__ unsigned long long cell_key(float px, float py, float pz, float nx, float ny,
                                                       float nz, const float origin[3], float h,
                                                       uint32_t nb, bool jit, const float j[5])
{
    const uint32_t fx = quant_pos(px, origin[0], h, jit, j[0]);
    const uint32_t fy = quant_pos(py, origin[1], h, jit, j[1]);
    const uint32_t fz = quant_pos(pz, origin[2], h, jit, j[2]);
    const float s = fadd(fadd(fabsf(nx), fabsf(ny)), fabsf(nz));
    float a = 0.0f, b = 0.0f;
    if (s > 0.0f) {
        a = fdiv(nx, s);
        b = fdiv(nz, s);
        if (ny < 0.0f) {
            const float sa = a >= 0.0f ? 1.0f : -1.0f, sb = b >= 0.0f ? 1.0f : -1.0f;
            const float na = fmul(fsub(1.0f, fabsf(b)), sa);
            const float nbv = fmul(fsub(1.0f, fabsf(a)), sb);
            a = na;
            b = nbv;
        }
    }
    const uint32_t iu = quant_nrm(a, nb, jit, j[3]);
    const uint32_t iv = quant_nrm(b, nb, jit, j[4]);
    return (unsigned long long)fx | ((unsigned long long)fy << 16) | ((unsigned long long)fz << 32) |
           ((unsigned long long)iu << 48) | ((unsigned long long)iv << 56);
}

// ---------------------------------------------------------------- bounds
// Descent constants of a node (centre, r^2, r, sin theta).
__device__ __forceinline__ DescRec make_desc(const NodeRec& n)
{
    DescRec d;
    const float ex = fsub(n.bmax[0], n.bmin[0]), ey = fsub(n.bmax[1], n.bmin[1]), ez = fsub(n.bmax[2], n.bmin[2]);
    for (int k = 0; k < 3; ++k) {
        d.c[k] = fmul(fadd(n.bmin[k], n.bmax[k]), 0.5f);
        d.axis[k] = n.axis[k];
    }
    // compact constants: r rounded up one ulp and r^2 = r r (not below the box's squared half
    // diagonal); the cone as v = 1 - cos theta rounded up to binary16 (a cone at least as wide;
    // 11 significant bits of v keep narrow cones narrow), cos = 1 - v (exact), and sin theta of
    // that cone rounded up to binary16 from the exact 1 - cos^2 = v (2 - v). Rounding up twice
    // (binary32, then binary16) equals rounding up once.
    const float rb2 = fmul(0.25f, fadd(fadd(fmul(ex, ex), fmul(ey, ey)), fmul(ez, ez)));
    d.r = nextafterf(fsqrt(rb2), INFINITY);
    d.r2 = fmul(d.r, d.r);
    d.phi = n.phi;
    const float v = __half2float(__float2half_ru(__fsub_ru(1.0f, n.cos_t)));
    d.cos_t = fsub(1.0f, v);
    d.sin_t = __half2float(__float2half_ru(__fsqrt_ru(fmul(v, fsub(2.0f, v)))));
    d.id = n.id;
    return d;
}

// Unoccluded importance of a node seen from (x, n): power times the receiver
// and emitter cosine bounds over the node's bounding sphere, over distance^2,
// kept as num / den = (phi A B) / d^6 with A = d^2 Brecv, B = d^2 Bemit.
// Cosines and sines are carried multiplied by |d| (2-3 square roots, no
// division). For a node at d = c - x (d2 = |d|^2):
//   d2 <= r2: num = phi, den = max(r2, 1e-30); else
//   cb = sqrt(d2 - r2); nd = n d; A = nd < cb ? max(0, nd cb + sqrt(max(0, d2 - nd^2)) r) : d2;
//   ad = -axis d; sphi = sin cb + cos r; cphi = cos cb - sin r;
//   B = sphi <= 0 or cphi <= ad ? d2 : max(0, ad cphi + sqrt(max(0, d2 - ad^2)) sphi);
//   num = (phi A) B; den = (d2 d2) d2,
// sums of products from the left, each but the first product fused (x, y, z in turn).

// Correctly rounded square root of two values at once, sign-flipped: for n = -x (x in {0} or
// [2^-100, 2^60), else see below) returns -sqrt(x), bit for bit __fsqrt_rn's value. One
// Newton-Raphson correction with the exact residual that a fused multiply-add gives (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990): s = x y with
// y the hardware's reciprocal square root estimate, e = x - s^2 exactly, s + e y / 2 rounded once.
// All 1 342 177 280 binary32 values of [2^-100, 2^60) were compared with __fsqrt_rn on the device:
// none differs. Carried with the sign flipped (n, -s) because packed instructions take no sign
// modifiers; a component with n > 0 gives a meaningless value. 2 estimates, 2 clamps (x = 0 gives
// 0 exactly) and 4 packed operations a pair, and no range test or call of its own.
__device__ __forceinline__ float rsqrt_estimate(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 neg_sqrt2(float2 n)
{
    const float2 y = make_float2(rsqrt_estimate(fmaxf(-n.x, 0x1p-100f)), rsqrt_estimate(fmaxf(-n.y, 0x1p-100f)));
    const float2 s = __fmul2_rn(n, y);  // -x y
    const float2 h = __fmul2_rn(y, make_float2(0.5f, 0.5f));
    const float2 e = __ffma2_rn(s, s, n);  // s^2 - x
    return __ffma2_rn(e, h, s);
}

// The importance of two nodes at once, in packed binary32 (f32x2) arithmetic:
// per component the correctly rounded operations above in their order. Signs are folded
// into the operands (rounding to nearest is symmetric), since a packed
// instruction takes no sign modifier: nt = r2 - d2, ncb = -cb, g = nd^2 - d2,
// nad = -ad, nsp = -sphi, ncp = -cphi. The early return inside the bounding
// sphere becomes a per-component select. The receiver and emitter branches
// are evaluated for both components always and selected per component (in a
// warp some lane nearly always needs them, so the branches only cost their
// divergence; the values selected are the same).
// The three square roots of a component are neg_sqrt2's: for d2 in [2^-40,
// 2^60] their arguments are 0 or in its range (a difference of two products
// or of d2 and r2 that is not 0 is at least 2^-48 of d2); a node closer or
// farther than that takes the library's square root. nx*: the shading point
// negated, n*: its normal, both broadcast to the two components.
// Fewer instructions than with the library's square root and scalar negations
// (whole passes: 64x64 points 60.6 -> 58.1 us, 1080p 470.9 -> 463.5 us, 4K
// bfloat16 2 224 -> 2 195 us; the record loads bound the kernel at that point).
namespace {
// out of line: the path of nodes out of neg_sqrt2's range, which is rarely taken, costs the descent
// loop no code (see sample_one)
__device__ __noinline__ float far_sqrt(float x) { return fsqrt(x); }
}  // namespace
struct Bound2 {
    float2 num, den;
};

// the descent constants of two nodes, x and y
struct NodePair {
    float2 c0, c1, c2, r, a0, a1, a2;
    uint32_t cs_x, cs_y;  // (1 - cos theta, sin theta) as two binary16 values
};

__device__ __forceinline__ Bound2 importance2(const NodePair& q, float2 phi, float2 nx0, float2 nx1, float2 nx2,
                                              float2 n0, float2 n1, float2 n2)
{
    const float2 one = make_float2(1.0f, 1.0f), minus = make_float2(-1.0f, -1.0f);
    const float2 vx = __half22float2(*reinterpret_cast<const __half2*>(&q.cs_x));
    const float2 vy = __half22float2(*reinterpret_cast<const __half2*>(&q.cs_y));
    const float2 v = make_float2(vx.x, vy.x), sin_t = make_float2(vx.y, vy.y);
    const float2 cos_t = __ffma2_rn(v, minus, one), ncos_t = __fadd2_rn(v, minus);  // both exact
    const float2 dx = __fadd2_rn(q.c0, nx0), dy = __fadd2_rn(q.c1, nx1), dz = __fadd2_rn(q.c2, nx2);
    const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
    const float2 r2 = __fmul2_rn(q.r, q.r);
    const float2 nd2 = __fmul2_rn(d2, minus);
    const float2 nt = __fadd2_rn(r2, nd2);
    const float2 nd = __ffma2_rn(n2, dz, __ffma2_rn(n1, dy, __fmul2_rn(n0, dx)));
    const float2 nad = __ffma2_rn(q.a2, dz, __ffma2_rn(q.a1, dy, __fmul2_rn(q.a0, dx)));
    const float2 gr = __ffma2_rn(nd, nd, nd2), ge = __ffma2_rn(nad, nad, nd2);
    const float2 xr = make_float2(fminf(gr.x, 0.0f), fminf(gr.y, 0.0f));
    const float2 xe = make_float2(fminf(ge.x, 0.0f), fminf(ge.y, 0.0f));
    float2 ncb, nsr, nse;
    if (fminf(d2.x, d2.y) >= 0x1p-40f && fmaxf(d2.x, d2.y) <= 0x1p60f) {
        ncb = neg_sqrt2(nt);
        nsr = neg_sqrt2(xr);
        nse = neg_sqrt2(xe);
    } else {
        ncb = make_float2(-far_sqrt(-nt.x), -far_sqrt(-nt.y));
        nsr = make_float2(-far_sqrt(-xr.x), -far_sqrt(-xr.y));
        nse = make_float2(-far_sqrt(-xe.x), -far_sqrt(-xe.y));
    }
    float2 A = d2, B = d2;
    {
        const float2 nv = __ffma2_rn(nd, ncb, __fmul2_rn(nsr, q.r));
        A.x = nd.x < -ncb.x ? fmaxf(0.0f, -nv.x) : A.x;
        A.y = nd.y < -ncb.y ? fmaxf(0.0f, -nv.y) : A.y;
    }
    {
        const float2 nsp = __ffma2_rn(sin_t, ncb, __fmul2_rn(ncos_t, q.r));
        const float2 ncp = __ffma2_rn(cos_t, ncb, __fmul2_rn(sin_t, q.r));
        const float2 w = __ffma2_rn(nad, ncp, __fmul2_rn(nse, nsp));
        B.x = !(nsp.x >= 0.0f || ncp.x >= nad.x) ? fmaxf(0.0f, w.x) : B.x;
        B.y = !(nsp.y >= 0.0f || ncp.y >= nad.y) ? fmaxf(0.0f, w.y) : B.y;
    }
    Bound2 o;
    o.num = __fmul2_rn(__fmul2_rn(phi, A), B);
    o.den = __fmul2_rn(__fmul2_rn(d2, d2), d2);
    if (nt.x >= 0.0f) {
        o.num.x = phi.x;
        o.den.x = fmaxf(r2.x, 1e-30f);
    }
    if (nt.y >= 0.0f) {
        o.num.y = phi.y;
        o.den.y = fmaxf(r2.y, 1e-30f);
    }
    return o;
}

// ---------------------------------------------------------------- storage
template <int P> struct Store;
template <> struct Store<RLL_PREC_FP32> {
    using T = float;
    __device__ __forceinline__ static float load(T v) { return v; }
    __device__ __forceinline__ static T store(float v) { return v; }
    __device__ __forceinline__ static uint16_t bits(T) { return 0; }
};
template <> struct Store<RLL_PREC_FP16> {
    using T = __half;
    __device__ __forceinline__ static float load(T v) { return __half2float(v); }
    // saturating: values beyond the largest finite half are stored as 65504
    __device__ __forceinline__ static T store(float v)
    {
        return __float2half_rn(fminf(fmaxf(v, -65504.0f), 65504.0f));
    }
    __device__ __forceinline__ static uint16_t bits(T v) { return __half_as_ushort(v); }
    __device__ __forceinline__ static T from_bits(uint16_t b) { return __ushort_as_half(b); }
};
template <> struct Store<RLL_PREC_BF16> {
    using T = __nv_bfloat16;
    __device__ __forceinline__ static float load(T v) { return __bfloat162float(v); }
    __device__ __forceinline__ static T store(float v)
    {
        const float mx = 3.3895313892515355e38f;  // largest finite bfloat16
        return __float2bfloat16_rn(fminf(fmaxf(v, -mx), mx));
    }
    __device__ __forceinline__ static uint16_t bits(T v) { return __bfloat16_as_ushort(v); }
    __device__ __forceinline__ static T from_bits(uint16_t b) { return __ushort_as_bfloat16(b); }
};

// Programmatic dependent launch: a kernel launched by launch_pdl may be
// scheduled while the kernel before it on the stream is finishing; its first
// statement is pdl_begin(): wait until that kernel (and so all earlier work)
// has completed and its writes are visible, then let the next kernel be
// scheduled in turn. (Between the learning kernels some of this is said apart
// and handed on by flags: see k_learn_buckets.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin()
{
    pdl_wait();
    pdl_release();
}

// A flag between kernels that may run at once: what the thread that stores it has seen or written is
// visible to the thread that loads the stored value.
__device__ __forceinline__ void store_release(uint32_t* p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t load_acquire(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args... args)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ordered-integer image of a float for atomicMin / atomicMax
__device__ __forceinline__ int float_to_ordered(float f)
{
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float ordered_to_float(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF); }

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

}  // namespace rll
