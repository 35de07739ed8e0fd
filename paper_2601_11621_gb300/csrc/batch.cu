// batch.cu -- many exact quantities computed together (uneven n, mixed kinds).
//
// Phase 1 (Sec. 3.1) once for the whole batch: one sieve up to the largest
// limit, then one thread per (request, prime) marks the primes with e_p >= 1
// (Sec. 2) and the primes of request r are written out e_p times each, request
// after request.
// Phase 2 (Sec. 3.2) as one segmented, level-synchronous product tree: every
// level of every request's tree is multiplied by the same batched launches
// (schoolbook, one-block transform or multi-pass transform, by slot size).
// A segment with an odd node count at some level gets a node of value 1
// appended, so adjacent pairs never straddle two requests.  The product over
// a request's primes, each repeated e_p times, is prod_e Q_e^e: the powers
// P_e = Q_e^e of Algorithm 2 are formed inside the tree rather than by
// separate square-and-multiply chains, which keeps the whole batch in a
// handful of launches per level.
#include "cat_internal.cuh"
#include "legendre.cuh"

#include <string.h>

#include <algorithm>
#include <vector>

namespace cat {

DevBuf<uint32_t> sieve_primes(Ctx &c, uint64_t limit, uint64_t *count, cudaStream_t s);
void exclusive_scan_u32(Ctx &c, uint32_t *data, size_t n, cudaStream_t s, uint32_t *sum = nullptr);

namespace {

constexpr int kBatchLeafSlot = 8;

// index r with pre[r] <= t < pre[r+1] (pre ascending, pre[0] = 0)
__device__ __forceinline__ int find_segment(const uint64_t *pre, int count, uint64_t t)
{
    int lo = 0, hi = count;  // pre[lo] <= t < pre[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// first[k] = the segment of flat index k tile (of the last one past the end).
// The blocks that work on tiles of consecutive indices each look it up here:
// with a search of 12 to 17 dependent loads at the head of every block
// or thread instead, the index of 4,096 requests' products took 65 us (now 35)
// and their leaf nodes 196 us (now 136, with the leaves' loads ahead of the
// multiplications).
__global__ void tile_segments(const uint64_t *pre, int count, int tile, unsigned ntiles, int *first)
{
    chain_wait();
    const unsigned k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < ntiles) first[k] = find_segment(pre, count, (uint64_t)k * tile);
}

// The segment of flat index t (< pre[count]), walking on from r; a thread more
// than a few segments further searches for itself.
__device__ __forceinline__ int walk_segment(const uint64_t *pre, int count, int r, uint64_t t)
{
    for (int k = 0; k < 8 && pre[r + 1] <= t; k++) r++;
    return pre[r + 1] <= t ? find_segment(pre, count, t) : r;
}

constexpr int kNodeTile = 256;  // nodes and products per block

// pi(limit_r) for each request: binary search in the ascending prime list
__global__ void count_primes_le(const uint32_t *primes, uint64_t np, const uint64_t *limits,
                                int count, uint64_t *out)
{
    chain_wait();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= count) return;
    uint64_t lo = 0, hi = np;  // first index with primes[i] > limit
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if ((uint64_t)primes[mid] <= limits[r]) lo = mid + 1; else hi = mid;
    }
    out[r] = lo;
}

struct ReqDev {
    uint32_t n;
    int kind;
};

// floor(2^32 / p) of every prime (2^31 - 1 for p = 2)
__global__ void prime_inverses(const uint32_t *primes, uint64_t np, uint32_t *inv)
{
    chain_wait();
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < np) inv[i] = 0xffffffffu / primes[i];
}

// Flat indices: (request r, prime index t - pre[r]), pre the prefix sums of the
// requests' prime counts.  A tile is 2,048 of them, one block's; a block of
// threads walks on from the tile's first request.
constexpr int kFlatTile = 2048;
constexpr int kFlatThreads = 256;
constexpr int kFlatWords = kFlatTile / kFlatThreads;  // 32 indices each, per warp

// Whether request q's exponent of p needs Legendre's formula (else it is 0 or
// 1: a prime above sqrt(2n) of a binomial kind).
__device__ __forceinline__ bool full_exponent(uint32_t p, const ReqDev &q)
{
    return q.kind == CAT_FACTORIAL || (uint64_t)p * p <= 2 * (uint64_t)q.n;
}

// unit_exponent with n mod p from the reciprocal (a quotient estimate short by
// at most one)
__device__ __forceinline__ uint32_t unit_exponent_inv(uint32_t p, uint32_t pinv, const ReqDev &q)
{
    uint32_t m = q.n - __umulhi(q.n, pinv) * p;
    m = min(m, m - p);
    return 2 * m >= p && !(q.kind == CAT_CATALAN && m == p - 1) ? 1u : 0u;
}

// A warp's kFlatWords x 32 indices from `base` on, when they all belong to one
// request and none of its primes there needs the full exponent (all but a few
// per cent of them in requests of thousands of primes): the request's data are
// then the warp's, and the loads of its indices don't wait for one another.
struct UnitRun {
    ReqDev q;
    uint64_t i;  // of the first index's prime
    __device__ __forceinline__ bool find(const uint32_t *primes, const uint64_t *pre, int count,
                                         const ReqDev *reqs, int &r, uint64_t base, uint64_t total)
    {
        if (base + 32 * kFlatWords > total) return false;
        r = walk_segment(pre, count, r, base);
        if (base + 32 * kFlatWords > pre[r + 1]) return false;
        q = reqs[r];
        i = base - pre[r];
        return !full_exponent(primes[i], q);
    }
};

// Which flat indices have e_p >= 1, a bit each, their count per tile, and per
// request the further leaves of its primes with e_p >= 2.  n mod p comes from
// the prime's reciprocal (a high product and one correction).
//
// A bit per index is all that the leaves' places need (batch_leaves), where
// storing, scanning and reading back a 4-byte exponent per index moved 20 bytes
// each: this, the scans and batch_leaves take 0.39 ms instead of 1.54 ms for the
// 86 M indices of 4,096 requests.
__global__ void __launch_bounds__(kFlatThreads) batch_flags(const uint32_t *primes,
                                                           const uint32_t *inv,
                                                           const uint64_t *pre, int count,
                                                           const int *first,
                                                           const ReqDev *reqs, uint32_t *flags,
                                                           uint32_t *tiles, uint32_t *extra,
                                                           unsigned int *negative)
{
    chain_wait();
    __shared__ uint32_t sums[kFlatThreads / 32];
    const uint64_t total = pre[count], t0 = (uint64_t)blockIdx.x * kFlatTile;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t base = t0 + (uint64_t)wid * (kFlatTile / 8);
    uint32_t cnt = 0;
    int r = first[blockIdx.x];
    UnitRun u;
    if (u.find(primes, pre, count, reqs, r, base, total)) {
        const uint32_t *pp = primes + u.i + lane, *pv = inv + u.i + lane;
        uint32_t mask[kFlatWords];
#pragma unroll
        for (int it = 0; it < kFlatWords; it++) {
            const uint32_t p = pp[32 * it];
            mask[it] = __ballot_sync(0xffffffffu, unit_exponent_inv(p, pv[32 * it], u.q));
        }
#pragma unroll
        for (int it = 0; it < kFlatWords; it++) {
            if (lane == it) flags[(base >> 5) + it] = mask[it];
            cnt += __popc(mask[it]);
        }
    } else for (int it = 0; it < kFlatWords; it++) {
        const uint64_t t = base + 32 * it + lane;
        uint32_t e = 0;
        if (t < total) {
            r = walk_segment(pre, count, r, t);
            const uint64_t i = t - pre[r];
            const uint32_t p = primes[i];
            const ReqDev q = reqs[r];
            if (full_exponent(p, q)) {
                const int64_t v = exponent_of(p, q.n, q.kind);
                if (v < 0) atomicOr(negative, 1u);
                e = v < 0 ? 0u : (uint32_t)v;
                if (e > 1) atomicAdd(&extra[r], e - 1);
            } else {
                e = unit_exponent_inv(p, inv[i], q);
            }
        }
        const uint32_t mask = __ballot_sync(0xffffffffu, e > 0);
        if (lane == 0) flags[(base >> 5) + it] = mask;
        cnt += __popc(mask);
    }
    if (lane == 0) sums[wid] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < kFlatThreads / 32; w++) s += sums[w];
        tiles[blockIdx.x] = s;
    }
}

// rank[r]: the number of set flags before request r's first index (r = count:
// all of them), from the scanned tile counts.
__global__ void batch_ranks(const uint64_t *pre, int count, const uint32_t *flags,
                            const uint32_t *tiles, uint32_t *rank)
{
    chain_wait();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r > count) return;
    const uint64_t t = pre[r];
    uint32_t c = tiles[t / kFlatTile];
    for (uint64_t w = t / kFlatTile * (kFlatTile / 32); w < t >> 5; w++) c += __popc(flags[w]);
    if (t & 31) c += __popc(flags[t >> 5] & ((1u << (t & 31)) - 1));
    rank[r] = c;
}

// The leaves: a request's primes with e_p >= 1 in order, then the further
// copies of those with e_p >= 2 (in any order: cursor counts them).  With xs
// the exclusive scan of `extra`, request r's leaves start at rank[r] + xs[r].
__global__ void __launch_bounds__(kFlatThreads) batch_leaves(
    const uint32_t *primes, const uint64_t *pre, int count, const int *first, const ReqDev *reqs,
    const uint32_t *flags, const uint32_t *tiles, const uint32_t *rank, const uint32_t *xs,
    uint32_t *cursor, uint32_t *leaves)
{
    chain_wait();
    __shared__ uint32_t sums[kFlatThreads / 32];
    const uint64_t total = pre[count], t0 = (uint64_t)blockIdx.x * kFlatTile;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t base = t0 + (uint64_t)wid * (kFlatTile / 8);
    uint32_t mask[kFlatWords], cnt = 0;
#pragma unroll
    for (int it = 0; it < kFlatWords; it++) {
        mask[it] = flags[(base >> 5) + it];
        cnt += __popc(mask[it]);
    }
    if (lane == 0) sums[wid] = cnt;
    __syncthreads();
    uint32_t at = tiles[blockIdx.x];
    for (int w = 0; w < wid; w++) at += sums[w];
    int r = first[blockIdx.x];
    UnitRun u;
    if (u.find(primes, pre, count, reqs, r, base, total)) {
        const uint32_t *pp = primes + u.i + lane;
        uint32_t *to = leaves + at + xs[r];
#pragma unroll
        for (int it = 0; it < kFlatWords; it++) {
            if (mask[it] >> lane & 1) to[__popc(mask[it] & ((1u << lane) - 1))] = pp[32 * it];
            to += __popc(mask[it]);
        }
        return;
    }
#pragma unroll 1
    for (int it = 0; it < kFlatWords; it++) {
        const uint64_t t = base + 32 * it + lane;
        if (t < total && (mask[it] >> lane & 1)) {
            r = walk_segment(pre, count, r, t);
            const uint32_t p = primes[t - pre[r]];
            leaves[at + __popc(mask[it] & ((1u << lane) - 1)) + xs[r]] = p;
            const ReqDev q = reqs[r];
            if (full_exponent(p, q)) {
                const uint32_t e = (uint32_t)exponent_of(p, q.n, q.kind);
                if (e > 1) {
                    const uint32_t k = rank[r + 1] + xs[r] + atomicAdd(&cursor[r], e - 1);
                    for (uint32_t j = 0; j + 1 < e; j++) leaves[k + j] = p;
                }
            }
        }
        at += __popc(mask[it]);
    }
}

// node j of segment r = product of its leaves [lpn j, lpn j + lpn) (missing
// ones = 1; the caller picks lpn so that the product fits eight limbs),
// written to node dpos[r] + j of out
__global__ void batch_leaf_nodes(const uint32_t *leaves, const uint64_t *seg,
                                 const uint64_t *node_pre, const uint64_t *dpos, int count,
                                 const int *first_seg, int lpn, uint32_t *out)
{
    chain_wait();
    const uint64_t total = node_pre[count];
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int r = first_seg ? walk_segment(node_pre, count, first_seg[blockIdx.x], t)
                            : find_segment(node_pre, count, t);
    const uint64_t first = seg[r] + (t - node_pre[r]) * (uint64_t)lpn, end = seg[r + 1];
    uint32_t acc[kBatchLeafSlot];
#pragma unroll
    for (int j = 0; j < kBatchLeafSlot; j++) acc[j] = j == 0;
    for (int k0 = 0; k0 < lpn; k0 += 4) {
        uint32_t x[4];  // loaded together, ahead of the multiplications
#pragma unroll
        for (int k = 0; k < 4; k++)
            x[k] = k0 + k < lpn && first + k0 + k < end ? leaves[first + k0 + k] : 1u;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            uint32_t carry = 0;
#pragma unroll
            for (int j = 0; j < kBatchLeafSlot; j++) {
                const uint64_t v = (uint64_t)acc[j] * x[k] + carry;
                acc[j] = (uint32_t)v;
                carry = (uint32_t)(v >> 32);
            }
        }
    }
    const uint64_t node = dpos[r] + (t - node_pre[r]);
    uint4 *o = reinterpret_cast<uint4 *>(out + node * kBatchLeafSlot);
    o[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
    o[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
}

__global__ void batch_copy(const CopyJob *jobs, int njobs)
{
    for (int j = blockIdx.y; j < njobs; j += gridDim.y) {
        const CopyJob J = jobs[j];
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < J.cap;
             i += (uint64_t)gridDim.x * blockDim.x) {
            uint32_t v;
            if (!J.src)
                v = i == 0;
            else
                v = i < J.len ? J.src[i] : 0u;
            J.dst[i] = v;
        }
    }
}

// normalised length of each output region (one block per request, scanning
// down from the top)
__global__ void batch_lengths(const uint32_t *out, const uint64_t *off, const uint64_t *cap,
                              uint64_t *len)
{
    chain_wait();
    __shared__ unsigned long long best;
    const int r = blockIdx.x;
    const uint64_t n = block_top(out + off[r], 0, cap[r], &best);
    if (threadIdx.x == 0) len[r] = n;
}

template <typename T>
DevBuf<T> upload(Ctx &c, const std::vector<T> &h, cudaStream_t s)
{
    DevBuf<T> d(c, h.size() ? h.size() : 1, s);
    if (!h.empty())
        CAT_CUDA(cudaMemcpyAsync(d.get(), h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice,
                                 s));
    return d;
}

}  // namespace

void run_copy_jobs(Ctx &c, const std::vector<CopyJob> &jobs, cudaStream_t s)
{
    if (jobs.empty()) return;
    DevBuf<CopyJob> d_jobs = upload(c, jobs, s);
    const int nj = (int)jobs.size();
    batch_copy<<<dim3(64, std::min(nj, 4096)), 256, 0, s>>>(d_jobs.get(), nj);
    CAT_LAUNCH("batch_copy");
    CAT_CUDA(cudaStreamSynchronize(s));
}

namespace {

// A copy job of the segmented tree, planned before the level buffers exist:
// offsets into the launch's source and destination levels (src == kOne
// writes the value 1; dst_abs, when set, replaces the destination level).
struct LevelJob {
    uint64_t src, dst;
    uint32_t *dst_abs;
    uint64_t len, cap;
};
constexpr uint64_t kOne = ~(uint64_t)0;

__global__ void batch_copy_level(const LevelJob *jobs, int njobs, const uint32_t *src_base,
                                 uint32_t *dst_base)
{
    chain_wait();
    for (int j = blockIdx.y; j < njobs; j += gridDim.y) {
        const LevelJob J = jobs[j];
        uint32_t *dst = J.dst_abs ? J.dst_abs : dst_base + J.dst;
        const uint32_t *src = J.src == kOne ? nullptr : src_base + J.src;
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < J.cap;
             i += (uint64_t)gridDim.x * blockDim.x)
            dst[i] = src ? (i < J.len ? src[i] : 0u) : (uint32_t)(i == 0);
    }
}

// Output nodes of all the tree's products, every level's products numbered
// one after another: run i covers products [rs[i], rs[i+1]) and sends them
// to nodes dst[i], dst[i] + 1, ... of their level's output.
__global__ void batch_level_index(const uint64_t *rs, const uint64_t *dst, int runs,
                                  const int *first, uint32_t *index)
{
    chain_wait();
    const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= rs[runs]) return;
    const int i = first ? walk_segment(rs, runs, first[blockIdx.x], k) : find_segment(rs, runs, k);
    index[k] = (uint32_t)(dst[i] + (k - rs[i]));
}

}  // namespace

// The segmented level-synchronous product tree (see segmented_tree in
// cat_internal.cuh).  Level 0 multiplies eight leaves per node; every later
// level multiplies adjacent pairs of the whole level in one batched call.
//
// Every level's node counts follow from the segment lengths alone, so the
// whole schedule is planned on the host first and uploaded once; the levels
// then run back to back without waiting for the device.  A level's buffer
// holds the segments still multiplying, each padded to an even node count
// by a node of value 1, then the segments that are down to one node (their
// roots, copied out).  Each product is written straight to its node of the
// next level's buffer through an index table, so that no level is gathered
// or re-packed between products.
void segmented_tree(Ctx &c, const uint32_t *leaves, const std::vector<uint64_t> &seg,
                    std::vector<TreeRoot> &roots, cudaStream_t s, int leaf_bits)
{
    const size_t count = seg.size() - 1;
    const int nr = (int)count;
    // leaves per first-level node: their product stays below 2^(32 * 8)
    const int lpn = leaves_per_node(leaf_bits);
    struct Level {
        size_t slot;
        uint64_t padded, nodes;  // padded multiplying nodes; all nodes of the buffer
        size_t job0, njobs;      // pads and root copies of this level's buffer
        uint64_t maxcap;         // the longest of them (limbs), which sizes the launch
        uint64_t prod0;          // first product (all levels numbered in turn)
        size_t run0, nruns;      // runs of this level's products
    };
    std::vector<LevelJob> jobs;
    std::vector<Level> levels;
    std::vector<uint64_t> rs{0}, rdst;  // runs of products
    auto root_dst = [&](size_t r, uint64_t len, uint64_t &cap) -> uint32_t * {
        TreeRoot &t = roots[r];
        if (t.dst) {
            cap = t.cap;
            return t.dst;
        }
        const uint64_t n = std::max<uint64_t>(len, 1);
        t.big.buf = DevBuf<uint32_t>(c, n, s);
        t.big.n = n;
        cap = n;
        return t.big.buf.get();
    };
    // positions of a level's nodes: multiplying segments first, each padded
    // to an even count, then the one-node segments
    auto layout = [&](const std::vector<uint64_t> &cnt, std::vector<uint64_t> &pos,
                      uint64_t &padded, uint64_t &nodes) {
        uint64_t at = 0;
        for (size_t r = 0; r < count; r++)
            if (cnt[r] >= 2) {
                pos[r] = at;
                at += cnt[r] + (cnt[r] & 1);
            }
        padded = at;
        for (size_t r = 0; r < count; r++)
            if (cnt[r] == 1) pos[r] = at++;
        nodes = at;
    };
    std::vector<uint64_t> cnt(count), node_pre(count + 1, 0), pos(count, 0), nxt_cnt(count),
        nxt_pos(count, 0);
    for (size_t r = 0; r < count; r++) {
        cnt[r] = (seg[r + 1] - seg[r] + lpn - 1) / lpn;
        node_pre[r + 1] = node_pre[r] + cnt[r];
    }
    uint64_t padded = 0, nodes = 0, prod = 0;
    layout(cnt, pos, padded, nodes);
    const std::vector<uint64_t> pos0 = pos;
    const uint64_t nodes0 = nodes;
    for (size_t r = 0; r < count; r++)  // empty segments: the value 1
        if (seg[r + 1] == seg[r]) {
            uint64_t cap = 0;
            uint32_t *d = root_dst(r, 1, cap);
            jobs.push_back(LevelJob{kOne, 0, d, 1, cap});
        }
    for (size_t slot = kBatchLeafSlot;; slot *= 2) {
        Level lv{slot, padded, nodes, 0, 0, 0, prod, rs.size() - 1, 0};
        lv.job0 = levels.empty() ? 0 : jobs.size();
        for (size_t r = 0; r < count; r++) {
            if (cnt[r] >= 2 && (cnt[r] & 1))
                jobs.push_back(LevelJob{kOne, (pos[r] + cnt[r]) * slot, nullptr, 1, slot});
            if (cnt[r] == 1) {
                const uint64_t len = std::min<uint64_t>(slot, seg[r + 1] - seg[r]);
                uint64_t cap = 0;
                uint32_t *d = root_dst(r, len, cap);
                jobs.push_back(LevelJob{pos[r] * slot, 0, d, std::min(len, cap), cap});
            }
        }
        lv.njobs = jobs.size() - lv.job0;
        for (size_t j = lv.job0; j < jobs.size(); j++) lv.maxcap = std::max(lv.maxcap, jobs[j].cap);
        if (padded == 0) {
            levels.push_back(lv);
            break;
        }
        for (size_t r = 0; r < count; r++) nxt_cnt[r] = cnt[r] >= 2 ? (cnt[r] + 1) / 2 : 0;
        uint64_t npadded = 0, nnodes = 0;
        layout(nxt_cnt, nxt_pos, npadded, nnodes);
        for (size_t r = 0; r < count; r++)
            if (cnt[r] >= 2) {
                rs.push_back(rs.back() + nxt_cnt[r]);
                rdst.push_back(nxt_pos[r]);
            }
        lv.nruns = rs.size() - 1 - lv.run0;
        prod += padded / 2;
        levels.push_back(lv);
        cnt.swap(nxt_cnt);
        pos.swap(nxt_pos);
        padded = npadded;
        nodes = nnodes;
    }
    const uint64_t total_prod = prod;
    const int runs = (int)rdst.size();
    // one upload: segment starts, level-0 node offsets and positions, runs,
    // jobs
    std::vector<uint64_t> blob;
    auto put = [&](const std::vector<uint64_t> &v) {
        const size_t at = blob.size();
        blob.insert(blob.end(), v.begin(), v.end());
        return at;
    };
    const size_t at_seg = put(seg), at_np = put(node_pre), at_pos = put(pos0), at_rs = put(rs),
                 at_rd = put(rdst), at_jobs = blob.size();
    static_assert(sizeof(LevelJob) % sizeof(uint64_t) == 0, "LevelJob packs into words");
    blob.resize(at_jobs + jobs.size() * (sizeof(LevelJob) / sizeof(uint64_t)));
    if (!jobs.empty()) memcpy(blob.data() + at_jobs, jobs.data(), jobs.size() * sizeof(LevelJob));
    DevBuf<uint64_t> d_blob = upload(c, blob, s);
    const uint64_t *d = d_blob.get();
    const LevelJob *d_jobs = reinterpret_cast<const LevelJob *>(d + at_jobs);
    DevBuf<uint32_t> index(c, std::max<uint64_t>(total_prod, 1), s);
    const uint64_t tn = node_pre[count];
    const unsigned iblocks = (unsigned)((total_prod + kNodeTile - 1) / kNodeTile);
    const unsigned nblocks = (unsigned)((tn + kNodeTile - 1) / kNodeTile);
    // the tiles' first segments, where the blocks come in several waves (with
    // fewer a launch costs more than the searches, which then overlap; us per
    // batch, searches : table, at 331 blocks 544 : 548, 921 871 : 882, 1,267
    // 1,036 : 1,040, 2,712 1,712 : 1,710, 21,639 10,772 : 10,725)
    const bool table = std::max(iblocks, nblocks) > 8 * (unsigned)c.num_sms;
    DevBuf<int> first(c, table ? (size_t)iblocks + nblocks + 1 : 1, s);
    const int *ifirst = table ? first.get() : nullptr, *nfirst = table ? ifirst + iblocks : nullptr;
    if (table && iblocks) {
        launch_chained(tile_segments, (iblocks + 255) / 256, 256, 0, s, d + at_rs, runs, kNodeTile,
                       iblocks, first.get());
        CAT_LAUNCH("tile_segments");
    }
    if (table && nblocks) {
        launch_chained(tile_segments, (nblocks + 255) / 256, 256, 0, s, d + at_np, nr, kNodeTile,
                       nblocks, first.get() + iblocks);
        CAT_LAUNCH("tile_segments");
    }
    if (total_prod) {
        launch_chained(batch_level_index, iblocks, kNodeTile, 0, s, d + at_rs, d + at_rd, runs,
                       ifirst, index.get());
        CAT_LAUNCH("batch_level_index");
    }
    DevBuf<uint32_t> cur(c, std::max<uint64_t>(nodes0, 1) * kBatchLeafSlot, s);
    {
        const int tok = prof_begin(c, "batch_leaf_nodes", s);
        if (tn)
            launch_chained(batch_leaf_nodes, nblocks, kNodeTile, 0, s, leaves, d + at_seg,
                           d + at_np, d + at_pos, nr, nfirst, lpn, cur.get());
        CAT_LAUNCH("batch_leaf_nodes");
        prof_end(c, tok, s, 4.0 * (double)(seg[count] - seg[0]) + 32.0 * (double)tn);
    }
    for (size_t li = 0; li < levels.size(); li++) {
        const Level &lv = levels[li];
        if (lv.njobs) {
            // blocks per job by the longest job (2,048 limbs a block), jobs
            // spread over the grid's second dimension
            const unsigned gx = (unsigned)std::min<uint64_t>(64, (lv.maxcap + 2047) / 2048);
            launch_chained(batch_copy_level,
                           dim3(std::max(1u, gx), (unsigned)std::min<size_t>(lv.njobs, 65535)), 256,
                           0, s, d_jobs + lv.job0, (int)lv.njobs, cur.get(), cur.get());
            CAT_LAUNCH("batch_copy_level");
        }
        if (lv.padded == 0) break;
        const size_t slot = lv.slot, nprod = lv.padded / 2, ns = 2 * slot;
        DevBuf<uint32_t> nxt(c, levels[li + 1].nodes * ns, s);
        const uint32_t *ix = index.get() + lv.prod0;
        if (slot > c.comba_max_slot || !comba_level(c, cur.get(), slot, nprod, nxt.get(), s, ix)) {
            std::vector<uint32_t> host_ix;
            if (ns > ((size_t)1 << c.max_log)) {  // products by pieces, placed from the host
                host_ix.resize(nprod);
                for (size_t i = lv.run0; i < lv.run0 + lv.nruns; i++)
                    for (uint64_t k = rs[i]; k < rs[i + 1]; k++)
                        host_ix[k - lv.prod0] = (uint32_t)(rdst[i] + (k - rs[i]));
            }
            ntt_level(c, cur.get(), slot, nprod, nxt.get(), s, ix,
                      host_ix.empty() ? nullptr : host_ix.data());
        }
        cur = std::move(nxt);
    }
}

// Batched Phase 1 + Phase 2 for requests whose exponents are small (every
// prime written e_p times); request r's result goes to out + offsets[r]
// (room for bound_limbs limbs), its normalised length to lengths[r].
static void batch_core(Ctx &c, const cat_request *reqs, size_t count, uint32_t *out,
                       const uint64_t *offsets, uint64_t *lengths, cudaStream_t s)
{
    if (count == 0) return;
    std::vector<uint64_t> limits(count), caps(count);
    std::vector<ReqDev> rd(count);
    uint64_t M = 0;
    for (size_t r = 0; r < count; r++) {
        rd[r] = ReqDev{(uint32_t)reqs[r].n, reqs[r].kind};
        limits[r] = reqs[r].kind == CAT_FACTORIAL ? reqs[r].n : 2 * reqs[r].n;
        M = std::max(M, limits[r]);
        caps[r] = bound_limbs(reqs[r].n, reqs[r].kind);
    }
    const int nr = (int)count;
    // ---- Phase 1: shared sieve, exponents, leaves
    uint64_t np = 0;
    DevBuf<uint32_t> primes = sieve_primes(c, std::max<uint64_t>(M, 2), &np, s);
    DevBuf<uint64_t> d_limits = upload(c, limits, s);
    DevBuf<uint64_t> d_pi(c, count, s);
    launch_chained(count_primes_le, (nr + 255) / 256, 256, 0, s, primes.get(), np, d_limits.get(),
                   nr, d_pi.get());
    CAT_LAUNCH("count_primes_le");
    std::vector<uint64_t> pi(count), pre(count + 1, 0);
    CAT_CUDA(cudaMemcpyAsync(pi.data(), d_pi.get(), 8 * count, cudaMemcpyDeviceToHost, s));
    CAT_CUDA(cudaStreamSynchronize(s));
    for (size_t r = 0; r < count; r++) pre[r + 1] = pre[r] + pi[r];
    const uint64_t F = pre[count];
    if (F >= (1ull << 32)) fail(CAT_EINVAL, "batch too large");
    DevBuf<uint64_t> d_pre = upload(c, pre, s);
    DevBuf<ReqDev> d_req = upload(c, rd, s);
    const size_t ntiles = (size_t)((F + kFlatTile - 1) / kFlatTile);
    DevBuf<int> first(c, ntiles + 1, s);
    DevBuf<uint32_t> flags(c, ntiles * (kFlatTile / 32) + 1, s), tiles(c, ntiles + 1, s);
    // per request: ranks and the extra leaves' starts (count + 1 each), the
    // sign flag, then the cursors
    DevBuf<uint32_t> words(c, 3 * count + 3, s);
    uint32_t *rank = words.get(), *xs = rank + count + 1, *neg = xs + count + 1, *cursor = neg + 1;
    CAT_CUDA(cudaMemsetAsync(words.get(), 0, 4 * (3 * count + 3), s));
    CAT_CUDA(cudaMemsetAsync(tiles.get() + ntiles, 0, 4, s));
    if (F) {
        DevBuf<uint32_t> inv(c, np, s);
        launch_chained(prime_inverses, (unsigned)((np + 255) / 256), 256, 0, s, primes.get(), np,
                       inv.get());
        CAT_LAUNCH("prime_inverses");
        launch_chained(tile_segments, (unsigned)((ntiles + 255) / 256), 256, 0, s, d_pre.get(), nr,
                       kFlatTile, (unsigned)ntiles, first.get());
        CAT_LAUNCH("tile_segments");
        const int tok = prof_begin(c, "batch_flags", s);
        launch_chained(batch_flags, (unsigned)ntiles, kFlatThreads, 0, s, primes.get(), inv.get(),
                       d_pre.get(), nr, first.get(), d_req.get(), flags.get(), tiles.get(), xs,
                       neg);
        CAT_LAUNCH("batch_flags");
        prof_end(c, tok, s, 4.0 * (double)F);
    }
    exclusive_scan_u32(c, tiles.get(), ntiles + 1, s);
    exclusive_scan_u32(c, xs, count + 1, s);
    launch_chained(batch_ranks, (nr + 256) / 256, 256, 0, s, d_pre.get(), nr, flags.get(),
                   tiles.get(), rank);
    CAT_LAUNCH("batch_ranks");
    std::vector<uint32_t> hw(2 * count + 3);
    CAT_CUDA(cudaMemcpyAsync(hw.data(), words.get(), 4 * hw.size(), cudaMemcpyDeviceToHost, s));
    CAT_CUDA(cudaStreamSynchronize(s));
    if (hw[2 * count + 2]) fail(CAT_ENOTINTEGRAL, "a prime exponent is negative");
    std::vector<uint64_t> seg(count + 1);
    for (size_t r = 0; r <= count; r++) seg[r] = (uint64_t)hw[r] + hw[count + 1 + r];
    const uint32_t total_leaves = (uint32_t)seg[count];
    DevBuf<uint32_t> leaves(c, total_leaves ? total_leaves : 1, s);
    if (F) {
        const int tok = prof_begin(c, "batch_leaves", s);
        launch_chained(batch_leaves, (unsigned)ntiles, kFlatThreads, 0, s, primes.get(),
                       d_pre.get(), nr, first.get(), d_req.get(), flags.get(), tiles.get(), rank,
                       xs, cursor, leaves.get());
        CAT_LAUNCH("batch_leaves");
        prof_end(c, tok, s, 4.0 * (double)F + 4.0 * total_leaves);
    }
    primes.reset();
    flags.reset();
    tiles.reset();
    first.reset();

    // ---- Phase 2: one segmented tree over all requests
    std::vector<TreeRoot> roots(count);
    for (size_t r = 0; r < count; r++) {
        roots[r].dst = out + offsets[r];
        roots[r].cap = caps[r];
    }
    segmented_tree(c, leaves.get(), seg, roots, s, bits_below(M));  // leaves: primes <= M
    leaves.reset();
    // ---- lengths
    DevBuf<uint64_t> d_off = upload(c, std::vector<uint64_t>(offsets, offsets + count), s);
    DevBuf<uint64_t> d_cap = upload(c, caps, s);
    DevBuf<uint64_t> d_len(c, count, s);
    launch_chained(batch_lengths, nr, 256, 0, s, out, d_off.get(), d_cap.get(), d_len.get());
    CAT_LAUNCH("batch_lengths");
    CAT_CUDA(cudaMemcpyAsync(lengths, d_len.get(), 8 * count, cudaMemcpyDeviceToHost, s));
    CAT_CUDA(cudaStreamSynchronize(s));
}

// Factorials beyond this n have exponents far above 1 (v_2(n!) ~ n), so
// writing every prime e_p times would blow up the tree; they are computed one
// by one through the grouped path instead.
constexpr uint64_t kBatchFactorialMax = 64;

// out: the results back to back, request r at offsets[r] with room for
// bound_limbs(n_r, kind_r) limbs; lengths[r] = normalised length.
void exact_batch(Ctx &c, const cat_request *reqs, size_t count, uint32_t *out, size_t cap,
                 uint64_t *offsets, uint64_t *lengths, cudaStream_t s)
{
    NvtxRange range("batch");
    if (count == 0) return;
    uint64_t total_cap = 0;
    for (size_t r = 0; r < count; r++) {
        if (reqs[r].n >= (1ull << 31)) fail(CAT_EINVAL, "n must be below 2^31");
        if (reqs[r].kind < CAT_CATALAN || reqs[r].kind > CAT_FACTORIAL)
            fail(CAT_EINVAL, "unknown kind");
        offsets[r] = total_cap;
        total_cap += bound_limbs(reqs[r].n, reqs[r].kind);
    }
    if (total_cap > cap) {
        lengths[0] = total_cap;
        fail(CAT_ERANGE, "output capacity too small for the batch");
    }
    std::vector<cat_request> small;
    std::vector<uint64_t> small_off, small_len;
    std::vector<size_t> small_idx, single_idx;
    for (size_t r = 0; r < count; r++) {
        if (reqs[r].kind == CAT_FACTORIAL && reqs[r].n >= kBatchFactorialMax) {
            single_idx.push_back(r);
        } else {
            small_idx.push_back(r);
            small.push_back(reqs[r]);
            small_off.push_back(offsets[r]);
        }
    }
    small_len.resize(small.size());
    batch_core(c, small.data(), small.size(), out, small_off.data(), small_len.data(), s);
    for (size_t i = 0; i < small_idx.size(); i++) lengths[small_idx[i]] = small_len[i];
    for (size_t r : single_idx) {
        cat_factorization f{};
        factor(c, reqs[r].n, reqs[r].kind, &f, s);
        Big v;
        try {
            v = reconstruct(c, &f, s, bits_below(reqs[r].n));  // primes <= n
        } catch (...) {
            factor_free(c, &f, s);
            throw;
        }
        factor_free(c, &f, s);
        const uint64_t capr = bound_limbs(reqs[r].n, reqs[r].kind);
        if (v.n > capr) fail(CAT_ERANGE, "result longer than its bound");
        run_copy_jobs(c, {CopyJob{v.buf.get(), out + offsets[r], v.n, capr}}, s);
        lengths[r] = v.n;
    }
}

size_t batch_bound(const cat_request *reqs, size_t count)
{
    size_t t = 0;
    for (size_t r = 0; r < count; r++) t += bound_limbs(reqs[r].n, reqs[r].kind);
    return t;
}

}  // namespace cat
