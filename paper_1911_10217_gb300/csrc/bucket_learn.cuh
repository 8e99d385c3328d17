// Learning step on records bucketed by cell (Section 3, Eq. 1 and Eq. 2),
// shared by the single-grid entry point (learn.cu) and the batched form
// (batched.cu). A key decoder (valid / cell / cluster of a record key) and a
// row map (Q and C rows, cut size and length, alpha and eps of a cell) adapt
// it to either record layout. See learn.cu for the method notes.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

#include "learn_core.cuh"
#include "rll_device.cuh"
#include "rll_internal.h"

namespace rll {
namespace {  // every translation unit that includes this header gets its own copies

// one cell's rows and learning parameters
template <int P>
struct RowRef {
    typename Store<P>::T* Q;
    typename Store<P>::T* C;
    uint32_t M, m;
    float alpha, eps;
};

// ---------------------------------------------------------------- bucketed learning
// counters ctr[kLearnCounters]: [0] touched cells, [1] bucket space claimed, [2] cells for
// the sorting block path, [3] cells for the two-warp path, [4] [5] [7] work
// counters of the block, warp and two-warp phases, [6] cells for the grouping
// block path, [8] [9] flags: claim complete, scatter complete (kClaimed,
// kScattered: see k_learn_buckets); lists[2 * cells]: the grouping list (two-warp cells from the
// front, block cells from the back), then the sorting list
constexpr int kClaimed = 8, kScattered = 9;
constexpr int kBucketThreads = 256;
constexpr int kTilesPerWarp = 4;         // 32-record tiles one warp counts / scatters
constexpr uint32_t kWarpBucket = 240;    // records of a cell one warp orders in shared memory
constexpr uint32_t kPairBucket = 512;    // records of a cell two warps order together
constexpr uint32_t kBlockGroup = 1024;   // records of a cell one block orders by grouping and ranking
constexpr int kBigThreads = 1024;
constexpr uint32_t kBlockSort = 8 * kBigThreads;  // records of a cell one block sorts in shared memory, one tile
constexpr uint32_t kDigits = 256;
// two arrays of a tile's records, and the warps' digit counters (radix_pass)
constexpr size_t kBigSmem =
    2 * kBlockSort * sizeof(unsigned long long) + (kBigThreads / 32 + 1) * kDigits * sizeof(uint32_t);

// 1. record counts per cell and each record's rank among its cell's records
// (the cell's count before its warp's group, plus the lanes of the group
// below it); the first adder of a cell appends it to the touched list, one
// append per block. Each warp takes kTilesPerWarp tiles of 32 consecutive
// records. The ranks follow arrival order; the per-cell ordering restores
// sample order.
template <class Dec>
__global__ void __launch_bounds__(kBucketThreads)
k_bucket_count(const uint32_t* __restrict__ rec_key, int64_t n, Dec dec, uint32_t* __restrict__ cursor,
               uint32_t* __restrict__ touched, uint32_t* __restrict__ ctr, uint32_t* __restrict__ rank)
{
    pdl_begin();
    __shared__ uint32_t s_warp[kBucketThreads / 32];
    __shared__ uint32_t s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t tile0 = ((int64_t)blockIdx.x * (kBucketThreads / 32) + warp) * kTilesPerWarp;
    uint32_t slot[kTilesPerWarp], peers[kTilesPerWarp], old[kTilesPerWarp];
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
        const int64_t i = (tile0 + u) * 32 + lane;
        const uint32_t key = i < n ? __ldg(rec_key + i) : 0xFFFFFFFFu;
        slot[u] = dec.valid(key) ? dec.cell(key) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) peers[u] = __match_any_sync(0xffffffffu, slot[u]);
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
        old[u] = 1u;
        if (slot[u] != 0xFFFFFFFFu && lane == __ffs(peers[u]) - 1)
            old[u] = atomicAdd(cursor + slot[u], (uint32_t)__popc(peers[u]));
    }
    uint32_t fresh = 0;
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
        const uint32_t b = __shfl_sync(0xffffffffu, old[u], __ffs(peers[u]) - 1);
        if (slot[u] != 0xFFFFFFFFu) rank[(tile0 + u) * 32 + lane] = b + __popc(peers[u] & lanemask_lt());
        fresh += old[u] == 0u;
    }
    // cells this block saw first: one append for all of them
    uint32_t x = fresh;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t tot = 0;
        for (int w = 0; w < kBucketThreads / 32; ++w) {
            const uint32_t v = s_warp[w];
            s_warp[w] = tot;
            tot += v;
        }
        s_base = tot ? atomicAdd(ctr, tot) : 0u;
    }
    __syncthreads();
    if (!fresh) return;
    uint32_t base = s_base + s_warp[warp] + x - fresh;
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u)
        if (old[u] == 0u) touched[base++] = slot[u];
}

// 2. one contiguous bucket per touched cell (one atomic per warp), by `warps` warps of which this is
// number `first`
__device__ __forceinline__ void claim_cells(uint32_t first, uint32_t warps, uint32_t total, const uint32_t* touched,
                                            uint32_t* ctr, uint32_t* cursor, uint32_t* start, uint32_t* len,
                                            uint32_t* group_list, uint32_t* sort_list, uint32_t cells)
{
    const int lane = threadIdx.x & 31;
    for (uint32_t w = first; w * 32 < total; w += warps) {
        const uint32_t c = w * 32 + lane;
        const uint32_t slot = c < total ? __ldcg(touched + c) : 0u;
        const uint32_t cnt = c < total ? __ldcg(cursor + slot) : 0u;
        uint32_t x = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        uint32_t base = 0;
        if (lane == 31) base = atomicAdd(ctr + 1, x);
        base = __shfl_sync(0xffffffffu, base, 31);
        if (c < total) {
            start[c] = base + x - cnt;
            len[c] = cnt;
            cursor[slot] = base + x - cnt;
        }
        // cells above one warp's capacity: to the two-warp list (front of the grouping list),
        // the block list (its back) or the sorting list
        const bool to_pair = c < total && cnt > kWarpBucket && cnt <= kPairBucket;
        const bool to_group = c < total && cnt > kPairBucket && cnt <= kBlockGroup;
        const bool to_sort = c < total && cnt > kBlockGroup;
        const uint32_t pm = __ballot_sync(0xffffffffu, to_pair);
        const uint32_t gm = __ballot_sync(0xffffffffu, to_group), sm = __ballot_sync(0xffffffffu, to_sort);
        uint32_t pb = 0, gb = 0, sb = 0;
        if (lane == 0 && pm) pb = atomicAdd(ctr + 3, (uint32_t)__popc(pm));
        if (lane == 0 && gm) gb = atomicAdd(ctr + 6, (uint32_t)__popc(gm));
        if (lane == 0 && sm) sb = atomicAdd(ctr + 2, (uint32_t)__popc(sm));
        pb = __shfl_sync(0xffffffffu, pb, 0);
        gb = __shfl_sync(0xffffffffu, gb, 0);
        sb = __shfl_sync(0xffffffffu, sb, 0);
        const uint32_t below = (1u << lane) - 1u;
        if (to_pair) group_list[pb + __popc(pm & below)] = c;
        if (to_group) group_list[cells - 1u - (gb + __popc(gm & below))] = c;
        if (to_sort) sort_list[sb + __popc(sm & below)] = c;
    }
}

__global__ void __launch_bounds__(kBucketThreads)
k_bucket_claim(const uint32_t* __restrict__ touched, uint32_t* __restrict__ ctr, uint32_t* __restrict__ cursor,
               uint32_t* __restrict__ start, uint32_t* __restrict__ len, uint32_t* __restrict__ group_list,
               uint32_t* __restrict__ sort_list, uint32_t cells)
{
    pdl_begin();
    claim_cells(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), gridDim.x * (blockDim.x >> 5),
                *(volatile uint32_t*)ctr, touched, ctr, cursor, start, len, group_list, sort_list, cells);
}

// 3. every record to its cell's bucket, at the bucket start (the claim left it
// in the cell's cursor) plus the record's rank: sample id, cluster and reward;
// no atomics
// Bucket entry of a record: sample id, cluster, reward bits in one 8-byte
// word. Up to 2^24 records: cluster << 56 | sample id << 32 | reward bits (one
// store per record); above: sample id << 32 | reward bits, the cluster in a
// byte array beside it.
struct Bucket {
    unsigned long long* word;
    uint8_t* s;  // nullptr: the cluster is in the word
    __device__ __forceinline__ void put(uint32_t d, uint32_t id, uint32_t cls, uint32_t bits) const
    {
        if (!s) {
            word[d] = ((unsigned long long)(cls << 24 | id) << 32) | bits;
        } else {
            word[d] = ((unsigned long long)id << 32) | bits;
            s[d] = (uint8_t)cls;
        }
    }
    __device__ __forceinline__ void get(uint32_t d, uint32_t& id, uint32_t& cls, uint32_t& bits) const
    {
        const unsigned long long e = word[d];
        bits = (uint32_t)e;
        if (!s) {
            id = (uint32_t)(e >> 32) & 0xFFFFFFu;
            cls = (uint32_t)(e >> 56);
        } else {
            id = (uint32_t)(e >> 32);
            cls = s[d];
        }
    }
};

template <class Dec>
__global__ void __launch_bounds__(kBucketThreads)
k_bucket_scatter(const uint32_t* __restrict__ rec_key, const float* __restrict__ rec_val, int64_t n, Dec dec,
                 const uint32_t* __restrict__ cursor, const uint32_t* __restrict__ rank, Bucket bucket,
                 uint32_t* __restrict__ ctr)
{
    pdl_wait();
    if (threadIdx.x == 0) {  // the flag before the block's release: see k_learn_buckets
        if (blockIdx.x == 0) store_release(ctr + kClaimed, 1u);
        pdl_release();
    }
    const int64_t i0 = (int64_t)blockIdx.x * kBucketThreads * kTilesPerWarp + threadIdx.x;
    uint32_t key[kTilesPerWarp], val[kTilesPerWarp], rk[kTilesPerWarp], at[kTilesPerWarp];
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
        const int64_t i = i0 + (int64_t)u * kBucketThreads;
        key[u] = i < n ? __ldg(rec_key + i) : 0xFFFFFFFFu;
        val[u] = i < n ? __float_as_uint(__ldg(rec_val + i)) : 0u;
        rk[u] = i < n ? __ldg(rank + i) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) at[u] = dec.valid(key[u]) ? __ldg(cursor + dec.cell(key[u])) : 0u;
#pragma unroll
    for (int u = 0; u < kTilesPerWarp; ++u) {
        if (!dec.valid(key[u])) continue;
        bucket.put(at[u] + rk[u], (uint32_t)(i0 + (int64_t)u * kBucketThreads), dec.cluster(key[u]), val[u]);
    }
}

// 1. to 3. for few records in one launch: one cluster of blocks, its barrier between the steps, the
// counters cleared and the ranks kept in registers. The three launches, a clearing and the gaps
// between them took longer than the work (16 384 records, 64x64 points: 44.5 -> 42 us a pass; 12 288,
// 48.3 -> 46.5; with four times as many records a thread, 30 000 records: 52.9 -> 55.7); above
// kSmallRecords more SMs than a cluster's are worth more than the launches.
constexpr int kSmallBlocks = 8, kSmallThreads = 1024, kSmallItems = 2;
constexpr int64_t kSmallRecords = (int64_t)kSmallBlocks * kSmallThreads * kSmallItems;

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <class Dec>
__global__ void __cluster_dims__(kSmallBlocks, 1, 1) __launch_bounds__(kSmallThreads)
k_bucket_small(const uint32_t* __restrict__ rec_key, const float* __restrict__ rec_val, uint32_t n, Dec dec,
               uint32_t* cursor, uint32_t* touched, uint32_t* ctr, uint32_t* start, uint32_t* len,
               uint32_t* group_list, uint32_t* sort_list, uint32_t cells, Bucket bucket)
{
    pdl_wait();
    const uint32_t lane = threadIdx.x & 31u, g = blockIdx.x * kSmallThreads + threadIdx.x;
    if (g < (uint32_t)kLearnCounters) ctr[g] = 0u;
    __threadfence();
    cluster_sync();
    uint32_t key[kSmallItems], rank[kSmallItems];
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u) {
        const uint32_t i = (uint32_t)u * (kSmallBlocks * kSmallThreads) + g;
        key[u] = i < n ? __ldg(rec_key + i) : 0xFFFFFFFFu;
    }
    uint32_t peers[kSmallItems];
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u)
        peers[u] = __match_any_sync(0xffffffffu, dec.valid(key[u]) ? dec.cell(key[u]) : 0xFFFFFFFFu);
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u) {
        rank[u] = 1u;
        if (dec.valid(key[u]) && lane == (uint32_t)(__ffs(peers[u]) - 1))
            rank[u] = atomicAdd(cursor + dec.cell(key[u]), (uint32_t)__popc(peers[u]));
    }
    uint32_t fresh = 0;
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u) fresh |= (rank[u] == 0u) << u;
    uint32_t x = __popc(fresh);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    uint32_t at = 0;
    if (lane == 31 && x) at = atomicAdd(ctr, x);
    at = __shfl_sync(0xffffffffu, at, 31) + x - __popc(fresh);
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u) {
        if (fresh >> u & 1u) touched[at++] = dec.cell(key[u]);
        rank[u] = __shfl_sync(0xffffffffu, rank[u], __ffs(peers[u]) - 1) + __popc(peers[u] & lanemask_lt());
    }
    __threadfence();
    cluster_sync();
    claim_cells(g >> 5, kSmallBlocks * kSmallThreads / 32, *(volatile uint32_t*)ctr, touched, ctr, cursor, start, len,
                group_list, sort_list, cells);
    __threadfence();
    cluster_sync();
    if (threadIdx.x == 0) {  // the flag before the block's release: see k_learn_buckets
        if (blockIdx.x == 0) store_release(ctr + kClaimed, 1u);
        pdl_release();
    }
#pragma unroll
    for (int u = 0; u < kSmallItems; ++u) {
        const uint32_t i = (uint32_t)u * (kSmallBlocks * kSmallThreads) + g;
        if (!dec.valid(key[u])) continue;
        bucket.put(__ldcg(cursor + dec.cell(key[u])) + rank[u], i, dec.cluster(key[u]), __float_as_uint(__ldg(rec_val + i)));
    }
}

// Shared arrays of one team (a warp, a pair of warps or a block) ordering one cell's records (at most
// `cap` records, cut sizes up to CLUS), in the team's shared memory: A = bucket order, then (cluster,
// sample) order; B = grouped by cluster.
template <uint32_t CLUS>
struct CellOrder {
    uint32_t *a_sid, *a_val, *b_sid, *b_val;
    uint32_t *start;  // [CLUS] first position of each cluster in B
    uint32_t *cur;    // [CLUS] scatter cursors, then one past the last position
    float* q;         // [CLUS]
    uint8_t *a_s, *b_s;
    // Once Eq. 1 is composed, the record arrays (the first 16 cap bytes) are dead: they give the float
    // and 16-bit scratch rows (CLUS entries each) of Eq. 2 and split-collapse.
    float* scratch_c;
    uint16_t* scratch_bits;

    static constexpr size_t bytes(uint32_t cap) { return 18u * (size_t)cap + 12u * CLUS; }
    __device__ __forceinline__ CellOrder(void* p, uint32_t cap)
    {
        a_sid = static_cast<uint32_t*>(p);
        a_val = a_sid + cap;
        b_sid = a_val + cap;
        b_val = b_sid + cap;
        start = b_val + cap;
        cur = start + CLUS;
        q = reinterpret_cast<float*>(cur + CLUS);
        a_s = reinterpret_cast<uint8_t*>(q + CLUS);
        b_s = a_s + cap;
        scratch_c = static_cast<float*>(p);
        scratch_bits = reinterpret_cast<uint16_t*>(scratch_c + CLUS);
    }
};

// Split-collapse policy of the learning kernels: NoSplit leaves it to a
// separate call; a policy with kOn = true runs it on each cell right after the
// cell's Eq. 1, before the one Eq. 2 rebuild. row(cell) gives the cell's cut
// row, its light tree, threshold T and step limit.
struct SplitRow {
    uint32_t* cut;
    const NodeRec* nodes;
    const int32_t *parent, *left, *right;
    float T;
    uint32_t max_iter;
    int64_t n_nodes;
};
struct NoSplit {
    static constexpr bool kOn = false;
    __device__ __forceinline__ SplitRow row(uint32_t) const { return SplitRow{}; }
};
// one grid: cut rows of M entries at cut + slot M
struct WithSplit {
    static constexpr bool kOn = true;
    uint32_t* cut;
    uint32_t M;
    const NodeRec* nodes;
    const int32_t *parent, *left, *right;
    float T;
    uint32_t max_iter;
    int64_t n_nodes;
    __device__ __forceinline__ SplitRow row(uint32_t slot) const
    {
        return SplitRow{cut + (int64_t)slot * M, nodes, parent, left, right, T, max_iter, n_nodes};
    }
};


// The threads that order one cell together; its first warp also scans and finishes. One kind of object
// for all three sizes, so that the learning kernel holds its per-cell code once (a copy for each size
// was 3 % slower at 64x64 points and 1 % at 128 leaves, equal elsewhere; see warp_rebuild_cdf).
struct Team {
    uint32_t tid, size;  // 32, 64 or the block
    __device__ __forceinline__ bool lead() const { return tid < 32; }
    __device__ __forceinline__ void sync() const
    {
        if (size == 32) {
            __syncwarp();
        } else if (size == 64) {  // warps 2p and 2p + 1: named barrier 1 + p (0 is __syncthreads)
            // immediate barrier ids (a register id would reserve all 16 barriers of the block)
            switch (threadIdx.x >> 6) {
            case 0: asm volatile("bar.sync 1, 64;" ::: "memory"); break;
            case 1: asm volatile("bar.sync 2, 64;" ::: "memory"); break;
            default: asm volatile("bar.sync 3, 64;" ::: "memory"); break;
            }
        } else {
            __syncthreads();
        }
    }
};
template <int P, int U = 4>
__device__ __forceinline__ void load_q_row(const typename Store<P>::T* qrow, uint32_t m, float* q)
{
#pragma unroll U
    for (uint32_t s = threadIdx.x & 31; s < m; s += 32) q[s] = Store<P>::load(qrow[s]);
}

template <int P, int U = 4>
__device__ __forceinline__ void store_q_row(typename Store<P>::T* qrow, uint32_t m, float* q)
{
#pragma unroll U
    for (uint32_t s = threadIdx.x & 31; s < m; s += 32) {
        const typename Store<P>::T st = Store<P>::store(q[s]);
        qrow[s] = st;
        q[s] = Store<P>::load(st);
    }
}

// Last step of one cell, by one warp: Q (q, m entries) stored to the table
// precision (q then holds the stored values); with a split policy,
// split-collapse on those values and the rows it changed stored; then Eq. 2
// from the final Q. Scratch rows of kMaxCut entries: cs, nc, c, bits.
template <int P, int U = 4, class Split>
__device__ void finish_cell(const Split& sp, uint32_t slot, float* q, uint32_t m, float eps,
                            typename Store<P>::T* qrow, typename Store<P>::T* crow, uint32_t* cs, uint32_t* nc,
                            float* c, uint16_t* bits, uint32_t* status)
{
    store_q_row<P, U>(qrow, m, q);
    __syncwarp();
    if constexpr (Split::kOn) {
        const int lane = threadIdx.x & 31;
        const SplitRow r = sp.row(slot);
        if (load_cut_row<U>(r.cut, cs, m, r.n_nodes, status)) {
            const uint32_t steps = split_collapse_steps<P, U>(cs, q, c, nc, m, r.nodes, r.parent, r.left, r.right,
                                                              r.T, r.max_iter, r.n_nodes);
            if (steps) {
#pragma unroll U
                for (uint32_t s = lane; s < m; s += 32) {
                    r.cut[s] = cs[s];
                    qrow[s] = Store<P>::store(q[s]);  // exact: q holds table values
                }
                __syncwarp();
            }
        }
    }
    warp_rebuild_cdf<P, U>(q, (int)m, eps, crow, c, bits);
}

// Eq. 1 + Eq. 2 of one cell from its bucket of nr <= cap records: grouped
// by cluster (counting sort, any order inside a group), then each record's
// rank by sample id inside its group is counted, which puts them in
// (cluster, sample) order; warp 0 of the team composes, stores Q and
// rebuilds C. Called by every thread of the team.
template <int P, uint32_t CLUS, class Split>
__device__ __forceinline__ void learn_cell_grouped(const Team& team, const CellOrder<CLUS>& o, const Bucket& bucket,
                                                   uint32_t b0, uint32_t nr, uint32_t M, uint32_t m, float alpha,
                                                   float eps, typename Store<P>::T* qrow, typename Store<P>::T* crow,
                                                   const Split& sp, uint32_t slot, uint32_t* status)
{
    constexpr int U = CLUS <= 64 ? 1 : 4;  // see warp_rebuild_cdf
    const uint32_t t = team.tid, T = team.size;
    const int lane = threadIdx.x & 31;
    const bool w0 = team.lead();
#pragma unroll U
    for (uint32_t s = t; s < M; s += T) o.start[s] = 0u;
    if (w0) load_q_row<P, U>(qrow, m, o.q);
    team.sync();
    // the bucket, four records a thread in flight at once
    for (uint32_t k0 = t; k0 < nr; k0 += 4 * T) {
        uint32_t rs[4], rsid[4], rval[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t k = k0 + u * T;
            rs[u] = rsid[u] = rval[u] = 0u;
            if (k < nr) bucket.get(b0 + k, rsid[u], rs[u], rval[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t k = k0 + u * T;
            if (k < nr) {
                o.a_sid[k] = rsid[u];
                o.a_val[k] = rval[u];
                o.a_s[k] = (uint8_t)rs[u];
                atomicAdd(&o.start[rs[u]], 1u);
            }
        }
    }
    team.sync();
    if (w0) {  // cluster starts: exclusive scan over M bins, ipl consecutive bins a lane
        const uint32_t ipl = (M + 31) >> 5, lo = lane * ipl, hi = min(M, lo + ipl);
        uint32_t sum = 0;
#pragma unroll U
        for (uint32_t s = lo; s < hi; ++s) sum += o.start[s];
        uint32_t y = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, y, d);
            if (lane >= d) y += v;
        }
        uint32_t run = y - sum;
#pragma unroll U
        for (uint32_t s = lo; s < hi; ++s) {
            const uint32_t c = o.start[s];
            o.start[s] = run;
            o.cur[s] = run;
            run += c;
        }
    }
    team.sync();
    for (uint32_t k = t; k < nr; k += T) {
        const uint32_t s = o.a_s[k];
        const uint32_t d = atomicAdd(&o.cur[s], 1u);
        if (d >= nr) {  // impossible unless the counts are corrupt: flag, skip the write
            atomicOr(status, (uint32_t)RLL_E_DEVICE);
            continue;
        }
        o.b_sid[d] = o.a_sid[k];
        o.b_val[d] = o.a_val[k];
        o.b_s[d] = (uint8_t)s;
    }
    team.sync();
    for (uint32_t k = t; k < nr; k += T) {
        const uint32_t s = o.b_s[k], sid = o.b_sid[k];
        const uint32_t lo = o.start[s], hi = o.cur[s];
        const uint32_t end = min(hi, nr);
        uint32_t rank = 0, j = lo;
        for (; j + 4 <= end; j += 4) {
            const uint32_t x0 = o.b_sid[j], x1 = o.b_sid[j + 1], x2 = o.b_sid[j + 2], x3 = o.b_sid[j + 3];
            rank += (x0 < sid) + (x1 < sid) + (x2 < sid) + (x3 < sid);
        }
        for (; j < end; ++j) rank += o.b_sid[j] < sid;
        if (lo + rank >= nr) {
            atomicOr(status, (uint32_t)RLL_E_DEVICE);
            continue;
        }
        o.a_s[lo + rank] = (uint8_t)s;
        o.a_val[lo + rank] = o.b_val[k];
    }
    team.sync();
    if (T == 32) {
        learn_records<P>([&](uint32_t j) { return make_uint2(o.a_s[j], o.a_val[j]); }, nr, m, alpha, o.q);
    } else {  // a block or a pair: warp w of the team composes the groups of clusters w, w + warps, ...
        const uint32_t warps = T >> 5;
        const GroupScan scan(alpha);
#pragma unroll U
        for (uint32_t s = t >> 5; s < M; s += warps) {
            const uint32_t lo = o.start[s], hi = o.cur[s];
            if (hi <= lo || s >= m) continue;
            const float q = scan.run([&](uint32_t j) { return o.a_val[lo + j]; }, hi - lo, o.q[s]);
            if (lane == 0) o.q[s] = q;
        }
        team.sync();
    }
    if (w0)  // cluster starts and cursors are dead too: the cut scratch rows
        finish_cell<P, U>(sp, slot, o.q, m, eps, qrow, crow, o.start, o.cur, o.scratch_c, o.scratch_bits, status);
}

// Eq. 1 of one cell whose records are sorted by (cluster, sample id), by a
// whole block: cluster s occupies positions gs[s] .. ge[s]; cls(j) is the
// cluster and val(j) the reward bits of record j. Warp w composes clusters
// w, w + warps, ... (disjoint Q entries). All threads of the block call it.
template <int P, class Cls, class Val>
__device__ void compose_sorted_block(Cls cls, Val val, uint32_t nr, uint32_t M, uint32_t m, float alpha, float* q,
                                     uint32_t* gs, uint32_t* ge)
{
    for (uint32_t s = threadIdx.x; s < M; s += blockDim.x) gs[s] = ge[s] = 0u;
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < nr; j += blockDim.x) {
        const uint32_t s = cls(j);
        if (s >= M) continue;
        if (j == 0 || cls(j - 1) != s) gs[s] = j;
        if (j + 1 == nr || cls(j + 1) != s) ge[s] = j + 1;
    }
    __syncthreads();
    const uint32_t warps = blockDim.x >> 5;
    const GroupScan scan(alpha);
    for (uint32_t s = threadIdx.x >> 5; s < M; s += warps) {
        const uint32_t lo = gs[s], hi = ge[s];
        if (hi <= lo || s >= m) continue;
        const float qs = scan.run([&](uint32_t j) { return val(lo + j); }, hi - lo, q[s]);
        if ((threadIdx.x & 31) == 0) q[s] = qs;
    }
    __syncthreads();
}

// 4. Eq. 1 + Eq. 2 of every touched cell of at most kBlockGroup records in
// one persistent launch. Phase 0: blocks take the cells of the block list
// (more than kPairBucket records; the ordering of the warp path done by the
// whole block, warps composing different clusters in parallel). Phase 1: the
// block's warp pairs take the cells of the two-warp list (kWarpBucket ..
// kPairBucket records), three cells per block at a time; where there are no
// more such cells than blocks, blocks take them in phase 0 (64-sample tile:
// 305 us a pass, now 295). Phase 2: warps take
// the touched cells one by one and order those of at most kWarpBucket records
// themselves. Every phase draws from a work counter (ctr[4], ctr[7],
// ctr[5]), so the long cells start first and the teams that drew one join the
// next phase late instead of leaving a tail; a warp fetches its next cell
// index while it works on the current one. Shared memory: one slab per warp;
// a pair's arrays lie in its two warps' slabs, the block's across all.
template <uint32_t CLUS>
struct LearnSmem {
    using O = CellOrder<CLUS>;
    static constexpr size_t kPairHalf = (O::bytes(kPairBucket) + 1) / 2;
    static constexpr size_t kSlab = ((O::bytes(kWarpBucket) > kPairHalf ? O::bytes(kWarpBucket) : kPairHalf) + 15) &
                                    ~(size_t)15;
    static_assert(16u * kWarpBucket >= 6u * CLUS, "record arrays too small for the scratch rows");
};

template <int P, int WARPS, int MINB, uint32_t CLUS, class Rows, class Split>
__global__ void __launch_bounds__(WARPS * 32, MINB)
k_learn_buckets(const Bucket bucket, uint32_t* ctr, const uint32_t* group_list, const uint32_t* touched,
                const uint32_t* start, const uint32_t* len, uint32_t* __restrict__ cursor, Rows rows, Split sp,
                uint32_t* __restrict__ status, uint32_t cells)
{
    // Launched after k_learn_big, whose cells are others. Where it has cells, this kernel runs beside
    // it: it starts when every block of k_learn_big has released it, each after its wait for the
    // scatter, and ends only when k_learn_big has, so that whatever follows this kernel follows both.
    // Where it has none, k_learn_big releases this kernel at once and ends with the scatter, for which
    // this kernel's blocks wait in their places.
    // A release lets the next kernel start and makes nothing visible to it; that is done by two flags,
    // cleared with the counters. kClaimed: block 0 of the scatter stores it behind its wait for the
    // claim (k_bucket_small: behind the claim), before it releases; k_learn_big loads it and then reads
    // its cells' count. kScattered: block 0 of k_learn_big, which has cells, stores it behind its wait
    // for the scatter, before it releases; this kernel loads it, and so knows that it runs beside, and
    // that counts, lists and buckets can be read (by ordinary loads: the lists' pointers are not
    // restrict). A thread that does not see its flag waits for the kernel before its own.
    const bool beside = load_acquire(ctr + kScattered) != 0u;
    if (!beside) pdl_wait();
    pdl_release();
    static_assert(WARPS == 6, "three warp pairs, named barriers 1 .. 3");
    using L = LearnSmem<CLUS>;
    static_assert(CellOrder<CLUS>::bytes(kBlockGroup) <= WARPS * L::kSlab, "block arrays exceed the slabs");
    __shared__ __align__(16) unsigned char smem[WARPS * L::kSlab];
    __shared__ uint32_t s_next, s_pair[WARPS / 2];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t n_block_list = *(volatile const uint32_t*)(ctr + 6);
    uint32_t n_pair = *(volatile const uint32_t*)(ctr + 3);
    uint32_t n_group = n_block_list;
    if (n_group + n_pair <= gridDim.x) {  // a block for each of them: the pairs' cells too
        n_group += n_pair;
        n_pair = 0;
    }
    const uint32_t total = *(volatile const uint32_t*)ctr;
    uint32_t phase = n_group ? 0u : (n_pair ? 1u : 2u);
    // A team's first cell is its own number; only then does it draw from the phase's counter, whose
    // values follow the teams' numbers. Warps draw several cells at a time, an eighth of their share of
    // those left but at most 8: all the warps' draws of single cells from one address, one after another in the
    // L2, held a warp back for 5 000 cycles of the 17 000 that it spent on a cell (1080p; 12 000 of
    // 21 000 with two cells a warp). Passes: 64x64 points 40.5 -> 33.7 us, preview 80 -> 76, 1080p
    // 384 -> 378, 4K 1 843 -> 1 835 (with a quarter of the share at once 1 865: a tail).
    const uint32_t teams = gridDim.x * WARPS;
    auto share = [&](uint32_t left) { return min(max(left / (8 * teams), 1u), 8u); };
    const uint32_t chunk0 = share(total);
    bool first = true;              // of the phase
    uint32_t next = 0, end = 0;     // phase 2: the warp's cells
    uint32_t ahead = 0, len_ahead = 0;  // its next draw, `ahead` on lane 0
    for (;;) {
        uint32_t w;  // index of the next cell in the touched list
        Team team;
        if (phase == 0) {
            uint32_t bi = blockIdx.x;
            if (!first && n_group > gridDim.x) {
                if (threadIdx.x == 0) s_next = gridDim.x + atomicAdd(ctr + 4, 1u);
                __syncthreads();
                bi = s_next;
                __syncthreads();
            }
            if (bi >= n_group || (!first && n_group <= gridDim.x)) {  // uniform across the block: it leaves phase 0
                phase = 1;
                first = true;
                continue;
            }
            first = false;
            w = group_list[bi < n_block_list ? cells - 1u - bi : bi - n_block_list];
            team = Team{threadIdx.x, (uint32_t)(WARPS * 32)};
        } else if (phase == 1) {
            const uint32_t pairs = gridDim.x * (WARPS / 2);
            team = Team{threadIdx.x & 63u, 64u};
            uint32_t pi = blockIdx.x * (WARPS / 2) + (warp >> 1);
            if (!first && n_pair > pairs) {
                if (team.tid == 0) s_pair[warp >> 1] = pairs + atomicAdd(ctr + 7, 1u);
                team.sync();
                pi = s_pair[warp >> 1];
                team.sync();
            }
            if (pi >= n_pair || (!first && n_pair <= pairs)) {  // uniform across the pair: it leaves phase 1
                phase = 2;
                first = true;
                continue;
            }
            first = false;
            w = group_list[pi];
        } else {
            team = Team{lane, 32u};
            if (first || next == end) {
                const uint32_t count = first ? chunk0 : len_ahead;
                if (first) next = (blockIdx.x * WARPS + warp) * chunk0;
                else next = teams * chunk0 + __shfl_sync(0xffffffffu, ahead, 0);
                first = false;
                if (next >= total) break;
                end = min(next + count, total);
                len_ahead = share(total - next);
                ahead = total;
                if (lane == 0 && teams * chunk0 < total) ahead = atomicAdd(ctr + 5, len_ahead);
            }
            w = next++;
        }
        const uint32_t slot = touched[w], nr = len[w], b0 = start[w];
        if (phase == 2 && nr > kWarpBucket) continue;
        const RowRef<P> r = rows.row(slot);
        const uint32_t slab = phase == 0 ? 0u : (phase == 1 ? warp & ~1u : warp);
        const uint32_t cap = phase == 0 ? kBlockGroup : (phase == 1 ? kPairBucket : kWarpBucket);
        learn_cell_grouped<P>(team, CellOrder<CLUS>(smem + slab * L::kSlab, cap), bucket, b0, nr, r.M, r.m, r.alpha,
                              r.eps, r.Q, r.C, sp, slot, status);
        if (team.tid == 0) cursor[slot] = 0u;
        if (phase != 2) team.sync();
    }
    if (beside) pdl_wait();
}

// One stable pass of a radix sort over n records by a whole block (kBigThreads): records move from
// src to dst in increasing order of the 8 bits at `shift`, equal ones in their order. Tiles of
// kBlockSort records are placed one after another: a warp ranks up to 256 consecutive records of the
// tile, 32 a round (__match_any groups equal digits, the group's first lane advances the warp's
// counter of that digit), then one scan over the counters by (digit, warp), eight a thread, gives
// every record's place in the tile's order. s_wc [kDigits][kWcStride]: a digit's counters of the
// warps lie 33 apart, so that neither the ranking nor the scan meets bank conflicts. s_base
// [kDigits], s_sum [32]: shared memory.
constexpr uint32_t kWcStride = kBigThreads / 32 + 1;

__device__ __forceinline__ void radix_pass(const unsigned long long* src, unsigned long long* dst, uint32_t n,
                                           int shift, uint32_t* s_wc, uint32_t* s_base, uint32_t* s_sum)
{
    constexpr uint32_t kRounds = kBlockSort / kBigThreads, kWarps = kBigThreads / 32;
    static_assert(kWarps == 32 && kDigits * kWarps == 8 * kBigThreads, "eight counters a thread");
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    const uint32_t rounds = min(kRounds, (n + kBigThreads - 1) / kBigThreads);  // of a warp in a tile
    auto digit = [&](unsigned long long e) { return (uint32_t)(e >> shift) & (kDigits - 1); };
    // exclusive prefix over the block's threads (two barriers)
    auto block_scan = [&](uint32_t v) {
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_sum[warp] = x;
        __syncthreads();
        uint32_t w = s_sum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const uint32_t before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
        return (warp ? before : 0u) + x - v;
    };
    const bool one = n <= kBlockSort;
    if (!one) {  // where each digit's records begin, over all tiles
        if (t < kDigits) s_base[t] = 0u;
        __syncthreads();
        for (uint32_t k0 = 0; k0 < n; k0 += kBigThreads) {
            const uint32_t k = k0 + t, d = k < n ? digit(src[k]) : kDigits;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            if (d < kDigits && lane == (uint32_t)(__ffs(peers) - 1)) atomicAdd(&s_base[d], (uint32_t)__popc(peers));
        }
        __syncthreads();
        const uint32_t first = block_scan(t < kDigits ? s_base[t] : 0u);
        __syncthreads();
        if (t < kDigits) s_base[t] = first;
    }
    for (uint32_t tile = 0; tile < n; tile += kBlockSort) {
        for (uint32_t k = t; k < kDigits * kWcStride; k += kBigThreads) s_wc[k] = 0u;
        __syncthreads();
        unsigned long long rec[kRounds];
        uint32_t at[kRounds];  // digit << 16 | rank among the warp's records of that digit
#pragma unroll
        for (uint32_t r = 0; r < kRounds; ++r) {
            rec[r] = 0ull;
            at[r] = kDigits << 16;
            if (r >= rounds) continue;
            const uint32_t k = tile + (warp * rounds + r) * 32 + lane;
            if (k < n) rec[r] = src[k];
            const uint32_t d = k < n ? digit(rec[r]) : kDigits;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const int leader = __ffs(peers) - 1;
            uint32_t old = 0;
            if (d < kDigits && lane == (uint32_t)leader) {
                old = s_wc[d * kWcStride + warp];
                s_wc[d * kWcStride + warp] = old + (uint32_t)__popc(peers);
            }
            old = __shfl_sync(0xffffffffu, old, leader);
            at[r] = d << 16 | (old + (uint32_t)__popc(peers & lanemask_lt()));
            __syncwarp();
        }
        __syncthreads();
        uint32_t* mine = s_wc + (t >> 2) * kWcStride + 8 * (t & 3u);  // digit t / 4, eight warps
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = mine[k];
            sum += c[k];
        }
        uint32_t run = block_scan(sum);
        if (!one) {  // after the digit's records of the tiles before: its place less its place in the tile
            const uint32_t tile_first = __shfl_sync(0xffffffffu, run, lane & ~3u);
            const uint32_t tile_end = __shfl_sync(0xffffffffu, run + sum, lane | 3u);
            const uint32_t base = s_base[t >> 2];
            __syncwarp();
            if ((t & 3u) == 0) s_base[t >> 2] = base + tile_end - tile_first;
            run += base - tile_first;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            mine[k] = run;
            run += c[k];
        }
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kRounds; ++r) {
            const uint32_t d = at[r] >> 16;
            if (d < kDigits) dst[s_wc[d * kWcStride + warp] + (at[r] & 0xFFFFu)] = rec[r];
        }
        __syncthreads();
    }
}

// 5b. one block per cell of the sorting list (more than kBlockGroup records), which it puts in
// (cluster, sample id) order by radix passes over the ids' bits (of n_ids ids; less the cell's smallest
// one, where they have more than 24) and the clusters. Up to kBlockSort records whose ids span 24 bits, in shared memory: words (cluster << 24 |
// id) << 32 | reward. Others in global scratch, the cell's part of the bucket and of `wide` in turn:
// words cluster << 32 | id, rewards read by sample id at the end. Then Eq. 1 (warps composing
// different clusters) and Eq. 2. A cell of 8 192 records takes four passes of one tile; the bitonic
// network that this replaces took 91 steps with a barrier each, and its global form 105 and more
// 200 x 120 points at 64 samples, 483 such cells: 186 us -> 103).
template <int P, class Rows, class Split>
__global__ void __launch_bounds__(kBigThreads)
k_learn_big(const Bucket bucket, unsigned long long* __restrict__ wide, const float* __restrict__ rec_val,
            uint32_t* ctr, const uint32_t* touched, const uint32_t* start, const uint32_t* len, const uint32_t* big,
            uint32_t* __restrict__ cursor, Rows rows, Split sp, uint32_t* __restrict__ status, uint32_t n_ids)
{
    if (load_acquire(ctr + kClaimed) == 0u) pdl_wait();  // see k_learn_buckets
    const uint32_t n_big = *(volatile const uint32_t*)(ctr + 2);
    if (n_big == 0) {
        pdl_release();
        pdl_wait();
        return;
    }
    pdl_wait();
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) store_release(ctr + kScattered, 1u);
        pdl_release();
    }
    extern __shared__ unsigned long long s_rec[];      // two tiles, then the warps' digit counters
    uint32_t* s_wc = reinterpret_cast<uint32_t*>(s_rec + 2 * kBlockSort);
    __shared__ float s_q[kMaxCut], s_c[kMaxCut];
    __shared__ uint16_t s_b[kMaxCut];
    __shared__ uint32_t s_gs[kMaxCut], s_ge[kMaxCut], s_lim[2], s_base[kDigits], s_sum[32];
    for (uint32_t bi = blockIdx.x; bi < n_big; bi += gridDim.x) {
        const uint32_t w = big[bi];
        const uint32_t slot = touched[w], b0 = start[w], nr = len[w];
        const RowRef<P> r = rows.row(slot);
        const uint32_t M = r.M, m = r.m;
        const float alpha = r.alpha;
        if (threadIdx.x < 32) load_q_row<P>(r.Q, m, s_q);
        uint32_t lo = 0, hi = n_ids - 1u;
        if (bucket.s) {  // ids of more than 24 bits: the cell's smallest and largest
            if (threadIdx.x < 2) s_lim[threadIdx.x] = threadIdx.x ? 0u : 0xFFFFFFFFu;
            __syncthreads();
            lo = 0xFFFFFFFFu;
            hi = 0u;
            for (uint32_t k = threadIdx.x; k < nr; k += blockDim.x) {
                uint32_t id, cls, bits;
                bucket.get(b0 + k, id, cls, bits);
                lo = min(lo, id);
                hi = max(hi, id);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(&s_lim[0], lo);
                atomicMax(&s_lim[1], hi);
            }
            __syncthreads();
            lo = s_lim[0];
            hi = s_lim[1];
        }
        const int id_bits = 32 - __clz((int)(hi - lo));
        const bool small = nr <= kBlockSort && id_bits <= 24;
        unsigned long long* src = small ? s_rec : wide + b0;
        unsigned long long* dst = small ? s_rec + kBlockSort : bucket.word + b0;
        for (uint32_t k = threadIdx.x; k < nr; k += blockDim.x) {
            uint32_t id, cls, bits;
            bucket.get(b0 + k, id, cls, bits);
            id -= lo;
            src[k] = small ? ((unsigned long long)(cls << 24 | id) << 32) | bits : ((unsigned long long)cls << 32) | id;
        }
        __syncthreads();
        for (int shift = 0; shift < id_bits + 8; shift += 8) {  // the ids' digits, then the clusters
            const int at = shift < id_bits ? shift : (small ? 24 : 32);
            radix_pass(src, dst, nr, small ? 32 + at : at, s_wc, s_base, s_sum);
            unsigned long long* other = src;
            src = dst;
            dst = other;
            if (shift >= id_bits) break;
        }
        if (!small) {
            for (uint32_t k = threadIdx.x; k < nr; k += blockDim.x) {
                const unsigned long long e = src[k];
                src[k] = (e & 0xFFFFFFFF00000000ull) | __float_as_uint(__ldg(rec_val + lo + (uint32_t)e));
            }
            __syncthreads();
        }
        const int cls_at = small ? 56 : 32;
        compose_sorted_block<P>([&](uint32_t j) { return (uint32_t)(src[j] >> cls_at); },
                                [&](uint32_t j) { return (uint32_t)src[j]; }, nr, M, m, alpha, s_q, s_gs, s_ge);
        if (threadIdx.x < 32) {  // the cluster bounds are dead: the cut scratch rows
            finish_cell<P>(sp, slot, s_q, m, r.eps, r.Q, r.C, s_gs, s_ge, s_c, s_b, status);
            if (threadIdx.x == 0) cursor[slot] = 0u;
        }
        __syncthreads();
    }
}

// k_learn_big's shared-memory opt-in (above the 48 KB default), once per
// device and precision
template <int P, class Rows, class Split>
cudaError_t big_smem_attribute(int device)
{
    static std::mutex mu;
    static bool done[64] = {};
    std::lock_guard<std::mutex> lock(mu);
    if (device >= 0 && device < 64 && done[device]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(k_learn_big<P, Rows, Split>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kBigSmem);
    if (e == cudaSuccess && device >= 0 && device < 64) done[device] = true;
    return e;
}

// scratch of launch_bucketed_learn for n records: 8-byte bucket entries,
// cluster bytes (above 2^24 records), and the record ranks and in-place sort
// buffer (8 B: the ranks until the scatter, then the sort keys of cells above
// kBlockSort records)
inline size_t bucketed_scratch_bytes(int64_t n)
{
    const size_t n4 = ((size_t)n * 4 + 255) & ~(size_t)255, n1 = ((size_t)n + 255) & ~(size_t)255;
    return 2 * n4 + n1 + 8 * (size_t)n;
}

// Enqueues the whole learning step for n >= 1 records (cut sizes up to
// max_cut), every kernel with the programmatic launch dependency (those up to
// the scatter wait for their predecessors first, the last two as k_learn_buckets
// says). Clears ctr first; the caller holds
// `cursor` [cells] at zero (left at zero again); touched, start,
// len [cells] and lists [2 * cells] are outputs and scratch. Counters: ctr[0]
// touched cells, [1] claimed records, [2] sorting list, [3] two-warp list,
// [6] block list, [4] [5] [7] work counters of k_learn_buckets, [8] [9] flags.
template <int P, class Dec, class Rows, class Split = NoSplit>
cudaError_t launch_bucketed_learn(cudaStream_t s, int device, int sms, const uint32_t* rec_key,
                                  const float* rec_val, int64_t n, Dec dec, Rows rows, uint32_t cells,
                                  uint32_t* cursor, uint32_t* touched, uint32_t* start, uint32_t* len,
                                  uint32_t* ctr, uint32_t* lists, void* scratch, uint32_t* status,
                                  uint32_t max_cut, Split sp = Split{})
{
    const size_t n4 = ((size_t)n * 4 + 255) & ~(size_t)255, n1 = ((size_t)n + 255) & ~(size_t)255;
    char* ws = static_cast<char*>(scratch);
    // 8-byte entries in the first 2 n4 bytes; the cluster bytes after them once sample ids need
    // more than 24 bits
    Bucket bucket{reinterpret_cast<unsigned long long*>(ws),
                  n <= (int64_t)1 << 24 ? nullptr : reinterpret_cast<uint8_t*>(ws + 2 * n4)};
    auto* wide = reinterpret_cast<unsigned long long*>(ws + 2 * n4 + n1);
    const int64_t per_block = (int64_t)kBucketThreads * kTilesPerWarp;
    const unsigned rblocks = (unsigned)((n + per_block - 1) / per_block);
    uint32_t* group_list = lists;
    uint32_t* sort_list = lists + cells;
    // record ranks: the first 4 n bytes of the in-place sort buffer (dead until k_learn_big)
    uint32_t* rank = reinterpret_cast<uint32_t*>(wide);
    cudaError_t e0;
    if (n <= kSmallRecords) {
        e0 = launch_pdl(k_bucket_small<Dec>, dim3(kSmallBlocks), dim3(kSmallThreads), 0, s, rec_key, rec_val, (uint32_t)n,
                        dec, cursor, touched, ctr, start, len, group_list, sort_list, cells, bucket);
    } else {
        e0 = cudaMemsetAsync(ctr, 0, kLearnCounters * sizeof(uint32_t), s);
        if (e0 == cudaSuccess)
            e0 = launch_pdl(k_bucket_count<Dec>, dim3(rblocks), dim3(kBucketThreads), 0, s, rec_key, n, dec, cursor,
                            touched, ctr, rank);
        if (e0 == cudaSuccess)
            e0 = launch_pdl(k_bucket_claim, dim3(sms * 2), dim3(kBucketThreads), 0, s, touched, ctr, cursor, start,
                            len, group_list, sort_list, cells);
        if (e0 == cudaSuccess)
            e0 = launch_pdl(k_bucket_scatter<Dec>, dim3(rblocks), dim3(kBucketThreads), 0, s, rec_key, rec_val, n, dec,
                            cursor, rank, bucket, ctr);
    }
    if (e0 != cudaSuccess) return e0;
    // k_learn_big first, k_learn_buckets beside it: its blocks, few and long, take the place they need,
    // and without cells for them they cost nothing (whole passes: 64-sample tile 346 -> 307 us, path
    // vertices 479 -> 467, others equal)
    e0 = big_smem_attribute<P, Rows, Split>(device);
    if (e0 == cudaSuccess)
        e0 = launch_pdl(k_learn_big<P, Rows, Split>, dim3(sms), dim3(kBigThreads), kBigSmem, s, bucket, wide, rec_val,
                        ctr, touched, start, len, sort_list, cursor, rows, sp, status, (uint32_t)n);
    if (e0 != cudaSuccess) return e0;
    // cuts of at most 64 leaves: per-cluster arrays of 64 entries (30.5 KB of shared memory per
    // block), 56 registers, 6 blocks per SM; larger cuts: 256 entries (44.4 KB), 5 blocks per SM
    if (max_cut <= 64)
        return launch_pdl(k_learn_buckets<P, 6, 6, 64, Rows, Split>, dim3(sms * 6), dim3(6 * 32), 0, s, bucket, ctr,
                          group_list, touched, start, len, cursor, rows, sp, status, cells);
    return launch_pdl(k_learn_buckets<P, 6, 5, kMaxCut, Rows, Split>, dim3(sms * 5), dim3(6 * 32), 0, s, bucket, ctr,
                      group_list, touched, start, len, cursor, rows, sp, status, cells);
}

}  // namespace
}  // namespace rll
