// phase1.cu -- Phase 1 of the method on the device (Sec. 3.1, Algorithm 1):
// the primes up to the sieve limit by a segmented Sieve of Eratosthenes, the
// exponent of each prime by Legendre's formula (Sec. 2), and the grouping of
// the primes with e > 0 by exponent into CSR form.
//
// Sieve.  The seed primes up to sqrt(limit) < 2^16 are a prefix of the
// context's table.  The odd numbers up to the limit are cut into segments of
// 2^13 .. 2^18 (one bit each, at most 32 KiB of shared memory per block).
// Primes 3..31 are struck word by word from bit patterns; primes 37..511 are
// struck by whole warps (one multiple per lane); larger seed primes by one
// thread each.  The bitmap and a prime count per unit of 2^13 odd numbers go
// to global memory; an exclusive scan of the counts gives every unit its first
// output position.
//
// Exponents.  2n < 2^32, so every term floor(m / p^k) is a 32-bit division;
// primes above sqrt(m) take one division per factorial.  c_p = v_p(n+1) is
// the valuation of n+1 at p, which equals the exponent of p in the
// trial-division factorisation of n+1 of Algorithm 1 step 2.
//
// Grouping.  (e, p) pairs are sorted stably by e (least-significant-digit
// radix sort, pairs with e = 0 dropped in the first pass), so primes stay
// ascending within each group; group starts are then collected.
//
// Binomial kinds.  For C(n) and C(2n, n) every prime above sqrt(2n) has
// exponent 0 or 1 (one base-p carry), found with one division inside the
// sieve; the sieve keeps only the primes with exponent 1 and they are written
// in order straight into the e = 1 group.  Only the seed primes (below
// sqrt(2n) <= 65536) go through Legendre's formula, and one block sorts them
// by exponent.  Such a Phase 1 is four launches and one read-back (what the
// CSR's size depends on).
#include "cat_internal.cuh"
#include "legendre.cuh"

#include <algorithm>
#include <math.h>
#include <string.h>

namespace cat {

void exclusive_scan_u32(Ctx &c, uint32_t *data, size_t n, cudaStream_t s, uint32_t *sum = nullptr);

constexpr int kUnitLog = 13;                     // odd numbers per counting unit (log2)
constexpr int kUnitWords = (1 << kUnitLog) / 32;  // 256 words
constexpr int kMaxSegLog = 18;                   // odd numbers per segment, at most (log2)
constexpr int kMaxSegUnits = 1 << (kMaxSegLog - kUnitLog);
constexpr int kSieveThreads = 512;
constexpr uint32_t kMediumPrime = 37;       // first prime struck by atomics
constexpr uint32_t kLargePrime = 512;       // thread-per-prime from here (measured best)

// ------------------------------------------------------------ segments

struct SieveArgs {
    const uint32_t *seeds;  // ascending odd primes <= sqrt(limit)
    uint32_t i_med, i_large, nseeds;  // index ranges: [0,i_med) small (3..31 are
                                       // patterned), [i_med,i_large) medium, rest large
    uint32_t imax;          // largest odd index i with 2i+1 <= limit
    int seg_log;            // log2 odd numbers per segment
    uint32_t *bits;         // out: bit set = prime
    uint32_t *counts;       // out: primes per unit
    // unit_kind >= 0: keep only the primes p > root (p^2 > 2 unit_n) whose
    // exponent in the quantity of that kind is 1 (all others are 0 there);
    // counts then count the kept primes, and *total gets every odd prime.
    int unit_kind;
    uint32_t unit_n, root;
    unsigned int *total;
};

__constant__ uint32_t c_small_primes[10] = {3, 5, 7, 11, 13, 17, 19, 23, 29, 31};

__global__ void __launch_bounds__(kSieveThreads) sieve_segments(SieveArgs a)
{
    chain_wait();
    extern __shared__ uint32_t bm[];
    __shared__ uint32_t unit_count[kMaxSegUnits], all_count;
    const uint32_t seg = blockIdx.x;
    const int seg_words = 1 << (a.seg_log - 5);
    const uint32_t ibase = seg << a.seg_log;  // odd index of bit 0
    if (threadIdx.x < kMaxSegUnits) unit_count[threadIdx.x] = 0;
    if (threadIdx.x == 0) all_count = 0;
    // words of this segment at or below the last odd index (the last segment,
    // or the only one of a small limit, is sieved only that far)
    const uint32_t used = (uint32_t)std::min<uint64_t>(seg_words, (a.imax - ibase) / 32 + 1);
    const uint64_t used_bits = 32ull * used;
    // primes 3..31: bit b of word w is odd number x = 2(ibase + 32 w + b) + 1;
    // p | x  <=>  ibase + 32 w + b = (p - 1)/2 (mod p)
    // (the primes are compile-time constants, so i0 mod p is a multiply and a
    // shift; the word's bits b0, b0 + p, ... are one shift of the pattern
    // of p's multiples below 64)
    constexpr uint32_t kSmall[10] = {3, 5, 7, 11, 13, 17, 19, 23, 29, 31};
    for (int w = threadIdx.x; w < (int)used; w += blockDim.x) {
        const uint32_t i0 = ibase + 32u * w;
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < 10; k++) {
            const uint32_t p = kSmall[k];
            uint64_t multiples = 0;
            for (uint32_t b = 0; b < 64; b += p) multiples |= 1ull << b;
            const uint32_t r = i0 % p;
            uint32_t b0 = (p - 1) / 2 + p - r;  // in (0, 2p)
            if (b0 >= p) b0 -= p;
            m |= (uint32_t)(multiples << b0);
        }
        bm[w] = m;
    }
    __syncthreads();
    // smallest odd number here (below the limit, so below 2^32)
    const uint32_t lo_num = 2u * ibase + 1u;
    const uint32_t ubits = (uint32_t)used_bits;
    // bit index of the first odd multiple of p at or above max(lo_num, p^2),
    // or ubits when there is none in this segment (32-bit remainder: lo_num
    // and p < 2^16 fit 32 bits; the sums in 64 bits)
    auto first_bit = [&](uint32_t p) -> uint32_t {
        const uint32_t r = lo_num % p;
        uint64_t x0 = (uint64_t)lo_num + (r ? p - r : 0u);
        if (x0 < (uint64_t)p * p) x0 = (uint64_t)p * p;
        if (!(x0 & 1)) x0 += p;
        const uint64_t f = (x0 - 1) / 2 - ibase;
        return f < ubits ? (uint32_t)f : ubits;
    };
    // medium primes: one warp per prime, one multiple per lane
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (uint32_t j = a.i_med + wid; j < a.i_large; j += nw) {
        const uint32_t p = a.seeds[j];
        for (uint32_t i = first_bit(p) + (uint32_t)lane * p; i < ubits; i += 32 * p)
            atomicOr(&bm[i >> 5], 1u << (i & 31));
    }
    // large primes: one thread per prime
    for (uint32_t j = a.i_large + threadIdx.x; j < a.nseeds; j += blockDim.x) {
        const uint32_t p = a.seeds[j];
        for (uint32_t i = first_bit(p); i < ubits; i += p)
            atomicOr(&bm[i >> 5], 1u << (i & 31));
    }
    __syncthreads();
    if (seg == 0 && threadIdx.x == 0) {
        uint32_t w0 = bm[0];
        w0 |= 1u;  // 1 is not prime
        for (int k = 0; k < 10; k++) {  // the pattern struck p itself
            const uint32_t i = (c_small_primes[k] - 1) / 2;
            w0 &= ~(1u << i);
        }
        bm[0] = w0;
    }
    __syncthreads();
    uint32_t all = 0;
    uint32_t *out = a.bits + (size_t)seg * seg_words;
    // (a warp's 32 words lie in one unit: units and segments are multiples of
    // 256 words, the block's threads a multiple of 32)
    for (int w = threadIdx.x; w < seg_words; w += blockDim.x) {
        const uint64_t i0 = (uint64_t)ibase + 32u * w;
        uint32_t v = w < (int)used ? ~bm[w] : 0u;
        if (i0 > a.imax) v = 0;
        else if (i0 + 31 > a.imax) v &= (uint32_t)((2ull << (a.imax - i0)) - 1);
        if (a.unit_kind >= 0) {
            all += __popc(v);
            if (2 * i0 + 1 > a.unit_n) {
                // every number of the word is above n (so above root): a prime
                // p in (n, 2n] has e_p = 1 (floor(2n/p) = 1, floor(n/p) = 0),
                // except p = n + 1 for C(n), which divides n + 1
                if (a.unit_kind == CAT_CATALAN && ((a.unit_n + 1) & 1)) {
                    const uint64_t j = (uint64_t)a.unit_n / 2;  // odd index of n + 1
                    if (j >= i0 && j < i0 + 32) v &= ~(1u << (j - i0));
                }
            } else {
                uint32_t keep = 0;
                for (uint32_t m = v; m; m &= m - 1) {
                    const int b = __ffs(m) - 1;
                    const uint32_t p = (uint32_t)(2 * (i0 + b) + 1);
                    if (p > a.root && unit_exponent(p, a.unit_n, a.unit_kind)) keep |= 1u << b;
                }
                v = keep;
            }
        }
        out[w] = v;
        const uint32_t cnt = __reduce_add_sync(0xffffffffu, __popc(v));
        if (lane == 0 && cnt) atomicAdd(&unit_count[w / kUnitWords], cnt);
    }
    all = __reduce_add_sync(0xffffffffu, all);
    if (lane == 0 && all) atomicAdd(&all_count, all);
    __syncthreads();
    const int units = seg_words / kUnitWords;
    if ((int)threadIdx.x < units) a.counts[seg * units + threadIdx.x] = unit_count[threadIdx.x];
    if (threadIdx.x == 0 && a.unit_kind >= 0) atomicAdd(a.total, all_count);
}

// ----------------------------------------------------------- exponents

// The primes of a unit, in order, by one warp: 32 words at a time (one per
// lane), a warp scan of the bit counts placing each lane's primes in the
// warp's shared stage (32 x 32 words); f(tot) then takes the stage's tot
// primes.  f must not change the stage's order; the warp is converged.
template <class F>
__device__ __forceinline__ void unit_primes(const uint32_t *bits, uint32_t unit, uint32_t *st,
                                            F &&f)
{
    const int lane = threadIdx.x & 31;
    const uint32_t *b = bits + (size_t)unit * kUnitWords;
    uint32_t w[kUnitWords / 32];
#pragma unroll
    for (int it = 0; it < kUnitWords / 32; it++) w[it] = b[it * 32 + lane];
#pragma unroll
    for (int it = 0; it < kUnitWords / 32; it++) {
        const uint32_t c = __popc(w[it]);
        uint32_t incl = c;
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t at = incl - c;
        const uint32_t ibase = (unit << kUnitLog) + 32u * (it * 32 + lane);
        for (uint32_t m = w[it]; m; m &= m - 1) st[at++] = 2 * (ibase + __ffs(m) - 1) + 1;
        __syncwarp();
        f(tot);
        __syncwarp();
    }
}

constexpr int kExpandThreads = 256;
constexpr int kExpandWarps = kExpandThreads / 32;

struct ExpandArgs {
    const uint32_t *bits;
    const uint32_t *unit_offsets;  // exclusive scan of the per-unit counts
    uint32_t units;
    Ratio r;                       // the quantity (a kind of n, or a factorial ratio)
    uint64_t *items;               // out: (e << 32) | p, all primes ascending (item 0: 2)
    unsigned int *max_e;
    unsigned int *negative;
};

// One warp per unit: its primes in order with their exponents, one prime per
// lane at a time (a lane per word, with as many primes as the word holds, left
// most lanes waiting: 163 -> 43 us at the limit 10^7 with three terms).
__global__ void __launch_bounds__(kExpandThreads) expand_exponents(ExpandArgs a)
{
    chain_wait();
    __shared__ uint32_t stage[kExpandWarps][32 * 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t unit = blockIdx.x * kExpandWarps + wid;
    uint32_t emax = 0, neg = 0;
    auto put = [&](size_t at, uint32_t p) {
        const int64_t e = exponent_of(p, a.r);
        if (e < 0) neg = 1;
        const uint32_t eu = e < 0 ? 0u : (uint32_t)e;
        emax = max(emax, eu);
        a.items[at] = ((uint64_t)eu << 32) | p;
    };
    if (unit < a.units) {
        size_t pos = (size_t)a.unit_offsets[unit] + 1;
        uint32_t *st = stage[wid];
        unit_primes(a.bits, unit, st, [&](uint32_t tot) {
            for (uint32_t k = lane; k < tot; k += 32) put(pos + k, st[k]);
            pos += tot;
        });
        if (unit == 0 && lane == 0) put(0, 2u);
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    neg = __reduce_or_sync(0xffffffffu, neg);
    if (lane == 0) {
        if (emax) atomicMax(a.max_e, emax);
        if (neg) atomicOr(a.negative, 1u);
    }
}

// ------------------------------------------------------- radix grouping

constexpr int kRsThreads = 256;
constexpr int kRsItems = 16;                     // per thread
constexpr int kRsTile = kRsThreads * kRsItems;   // 4096
constexpr int kRsWarps = kRsThreads / 32;

// item (warp w, iteration it, lane) of a tile is element
// tile*4096 + w*512 + it*32 + lane: warp-major, so warp order = element order.
__device__ __forceinline__ size_t rs_index(size_t tile, int w, int it, int lane)
{
    return tile * kRsTile + (size_t)w * (32 * kRsItems) + it * 32 + lane;
}

struct RsArgs {
    const uint64_t *in;
    uint64_t *out;
    size_t count;
    int shift, bits;    // digit = (e >> shift) & (2^bits - 1), e = item >> 32
    int drop_zero;      // first pass: items with e == 0 are dropped
    uint32_t *counts;   // [digit][tile]
    size_t tiles;
};

__global__ void __launch_bounds__(kRsThreads) rs_histogram(RsArgs a)
{
    chain_wait();
    __shared__ uint32_t h[256];
    const int nb = 1 << a.bits;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const size_t tile = blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int it = 0; it < kRsItems; it++) {
        const size_t i = rs_index(tile, w, it, lane);
        if (i < a.count) {
            const uint32_t e = (uint32_t)(a.in[i] >> 32);
            if (!(a.drop_zero && e == 0)) atomicAdd(&h[(e >> a.shift) & (nb - 1)], 1u);
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nb; d += blockDim.x) a.counts[(size_t)d * a.tiles + tile] = h[d];
}

__global__ void __launch_bounds__(kRsThreads) rs_scatter(RsArgs a)
{
    chain_wait();
    __shared__ uint32_t wh[kRsWarps][256];
    const int nb = 1 << a.bits;
    for (int i = threadIdx.x; i < kRsWarps * 256; i += blockDim.x) (&wh[0][0])[i] = 0;
    __syncthreads();
    const size_t tile = blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t item[kRsItems];
    uint32_t rank[kRsItems];
    int digit[kRsItems];
    for (int it = 0; it < kRsItems; it++) {
        const size_t i = rs_index(tile, w, it, lane);
        int d = -1;
        uint64_t v = 0;
        if (i < a.count) {
            v = a.in[i];
            const uint32_t e = (uint32_t)(v >> 32);
            if (!(a.drop_zero && e == 0)) d = (int)((e >> a.shift) & (nb - 1));
        }
        item[it] = v;
        digit[it] = d;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (d >= 0 && lane == leader) {
            base = wh[w][d];
            wh[w][d] = base + __popc(peers);
        }
        base = __shfl_sync(0xffffffffu, base, leader);
        rank[it] = base + __popc(peers & ((1u << lane) - 1));
        __syncwarp();
    }
    __syncthreads();
    // exclusive scan over warps per digit, plus the global digit offset
    for (int d = threadIdx.x; d < nb; d += blockDim.x) {
        uint32_t run = a.counts[(size_t)d * a.tiles + tile];
        for (int k = 0; k < kRsWarps; k++) {
            const uint32_t c = wh[k][d];
            wh[k][d] = run;
            run += c;
        }
    }
    __syncthreads();
    for (int it = 0; it < kRsItems; it++)
        if (digit[it] >= 0) a.out[wh[w][digit[it]] + rank[it]] = item[it];
}

// group starts: positions i with e_i != e_{i-1}, appended as (e, i)
__global__ void group_starts(const uint64_t *items, size_t count, uint64_t *starts,
                             unsigned int *nstarts, uint32_t *primes)
{
    chain_wait();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const uint64_t v = items[i];
    primes[i] = (uint32_t)v;
    const uint32_t e = (uint32_t)(v >> 32);
    if (i == 0 || (uint32_t)(items[i - 1] >> 32) != e) {
        const unsigned k = atomicAdd(nstarts, 1u);
        starts[2 * k] = e;
        starts[2 * k + 1] = i;
    }
}

// The primes of the bitmap in ascending order, written to primes[first + ...]
// (with_two: 2 at primes[0]); one warp per unit.
__global__ void __launch_bounds__(kExpandThreads) expand_primes(const uint32_t *bits,
                                                               const uint32_t *unit_offsets,
                                                               uint32_t units, uint32_t *primes,
                                                               uint32_t first, int with_two)
{
    chain_wait();
    __shared__ uint32_t stage[kExpandWarps][32 * 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t unit = blockIdx.x * kExpandWarps + wid;
    if (with_two && blockIdx.x == 0 && threadIdx.x == 0) primes[0] = 2;
    if (unit >= units) return;
    size_t pos = (size_t)unit_offsets[unit] + first;
    uint32_t *st = stage[wid];
    unit_primes(bits, unit, st, [&](uint32_t tot) {
        for (uint32_t k = lane; k < tot; k += 32) primes[pos + k] = st[k];
        pos += tot;
    });
}

// The seed primes of a binomial kind grouped by exponent, by one block: the
// exponents (one prime per thread at a time), then a stable counting sort
// (every thread counts a stretch of consecutive seeds per exponent, one warp
// per exponent scans its counts over the threads), primes with e = 0 dropped.
// Exponents are at most 31 (p^e <= 2n).  sorted takes the grouped primes, info
// the groups beside the sieve's counts.
constexpr int kSeedThreads = 512;
constexpr int kMaxSeeds = 6542;  // primes below 2^16
constexpr int kSeedsPerThread = (kMaxSeeds + kSeedThreads - 1) / kSeedThreads;
constexpr size_t kSeedSmem = (size_t)kMaxSeedGroups * kSeedThreads * 2;

__global__ void __launch_bounds__(kSeedThreads) group_seeds(const uint32_t *seeds, uint32_t ns,
                                                           Ratio r, const uint32_t *kept,
                                                           const uint32_t *total, uint32_t *sorted,
                                                           Phase1Info *info)
{
    chain_wait();
    extern __shared__ uint16_t cnt[];  // [exponent][thread]
    __shared__ uint8_t ex[kMaxSeeds];
    __shared__ uint32_t bin_total[kMaxSeedGroups], bin_base[kMaxSeedGroups], negative;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < kMaxSeedGroups * kSeedThreads; i += kSeedThreads) cnt[i] = 0;
    if (tid == 0) negative = 0;
    __syncthreads();
    for (uint32_t i = tid; i < ns; i += kSeedThreads) {
        const int64_t e = exponent_of(seeds[i], r);
        if (e < 0) atomicOr(&negative, 1u);
        ex[i] = e < 0 ? 0 : (uint8_t)e;
    }
    __syncthreads();
    const uint32_t i0 = tid * kSeedsPerThread, i1 = min(ns, i0 + kSeedsPerThread);
    for (uint32_t i = i0; i < i1; i++) cnt[ex[i] * kSeedThreads + tid]++;
    __syncthreads();
    for (int e = wid; e < kMaxSeedGroups; e += kSeedThreads / 32) {
        uint32_t run = 0;
        for (int t = lane; t < kSeedThreads; t += 32) {
            const uint32_t c = cnt[e * kSeedThreads + t];
            uint32_t incl = c;
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            cnt[e * kSeedThreads + t] = (uint16_t)(run + incl - c);
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) bin_total[e] = run;
    }
    __syncthreads();
    if (tid == 0) {
        uint32_t at = 0, ng = 0;
        for (int e = 1; e < kMaxSeedGroups; e++) {
            bin_base[e] = at;
            if (bin_total[e]) {
                info->exp[ng] = e;
                info->off[ng] = at;
                ng++;
            }
            at += bin_total[e];
        }
        info->off[ng] = at;
        info->ngroups = ng;
        info->negative = negative;
        info->kept = *kept;
        info->total = *total;
    }
    __syncthreads();
    for (uint32_t i = i0; i < i1; i++) {
        const uint32_t e = ex[i];
        if (e) sorted[bin_base[e] + cnt[e * kSeedThreads + tid]++] = seeds[i];
    }
}

// The CSR of a binomial kind: blocks [0, expand_blocks) write the large primes
// behind the n1 seeds with e = 1; the last block writes the grouped seeds
// around them and the group table.
struct CsrArgs {
    const uint32_t *bits, *unit_offsets;
    uint32_t units, expand_blocks;
    const uint32_t *sorted;   // grouped seeds
    uint32_t nsorted, n1, nl; // all of them, those with e = 1, the large primes
    uint32_t *primes;
    uint32_t ng;
    uint64_t *exps, *offs;
    uint64_t h_exps[kMaxSeedGroups + 1], h_offs[kMaxSeedGroups + 2];
};

__global__ void __launch_bounds__(kExpandThreads) write_csr(CsrArgs a)
{
    chain_wait();
    __shared__ uint32_t stage[kExpandWarps][32 * 32];
    if (blockIdx.x == a.expand_blocks) {
        for (uint32_t i = threadIdx.x; i < a.nsorted; i += kExpandThreads)
            a.primes[i < a.n1 ? i : i + a.nl] = a.sorted[i];
        for (uint32_t i = threadIdx.x; i <= a.ng; i += kExpandThreads) {
            a.exps[i] = a.h_exps[i];
            a.offs[i] = a.h_offs[i];
        }
        return;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t unit = blockIdx.x * kExpandWarps + wid;
    if (unit >= a.units) return;
    size_t pos = (size_t)a.unit_offsets[unit] + a.n1;
    uint32_t *st = stage[wid];
    unit_primes(a.bits, unit, st, [&](uint32_t tot) {
        for (uint32_t k = lane; k < tot; k += 32) a.primes[pos + k] = st[k];
        pos += tot;
    });
}

// ------------------------------------------------------------ host side

static uint64_t isqrt64(uint64_t x)
{
    uint64_t r = (uint64_t)sqrtl((long double)x);
    while (r > 0 && r * r > x) r--;
    while ((r + 1) * (r + 1) <= x) r++;
    return r;
}

// log2 odd numbers per segment: 2^18 (32 KiB of bitmap) when that still gives
// every SM several rounds of its four resident blocks, down to 2^13 for short
// sieves, so that their few numbers spread over the SMs (limits 2 10^5: 26 ->
// 17 us, 10^7: 37 -> 18, 10^8: 73 -> 61, 2 10^8: 97 either way).
static int segment_log(uint32_t odds, int num_sms)
{
    int lg = kMaxSegLog;
    while (lg > kUnitLog && (odds >> lg) < 8u * (uint32_t)num_sms) lg--;
    return lg;
}

// The segmented sieve up to `limit` (>= 2): the bitmap of the odd primes and
// the exclusive scan of the units' counts, whose sum goes to words[0]; nothing
// is read back.  With unit_kind >= 0 (a binomial kind of n, limit = 2n) the
// bitmap keeps only the primes above sqrt(2n) with exponent 1, words[1] gets
// the number of all odd primes, and the seeds are exactly the primes up to
// sqrt(2n).
struct SieveOut {
    DevBuf<uint32_t> bits, offsets, words;
    uint32_t units = 0, nseeds = 0;
};

static SieveOut run_sieve(Ctx &c, uint64_t limit, cudaStream_t s, int unit_kind = -1,
                          uint32_t unit_n = 0)
{
    SieveOut o;
    const uint64_t root = isqrt64(limit);
    auto below = [&](uint64_t x) {  // seeds <= x
        return (uint32_t)(std::upper_bound(c.host_seeds.begin(), c.host_seeds.end(), x) -
                          c.host_seeds.begin());
    };
    o.nseeds = below(root);
    // odd seeds only for the segment sieve
    const uint32_t nodd = o.nseeds ? o.nseeds - 1 : 0;
    const uint32_t i_med = std::min(nodd, below(kMediumPrime - 1) - 1);
    const uint32_t i_large = std::min(nodd, below(kLargePrime - 1) - 1);
    // odd indices 0..imax (odd number 2i+1 <= limit)
    const uint32_t imax = (uint32_t)((limit - 1) / 2);
    const int lg = segment_log(imax, c.num_sms);
    const uint32_t nsegs = (imax >> lg) + 1;
    o.units = nsegs << (lg - kUnitLog);
    o.bits = DevBuf<uint32_t>(c, (size_t)o.units * kUnitWords, s);
    o.offsets = DevBuf<uint32_t>(c, o.units, s);
    o.words = DevBuf<uint32_t>(c, 2, s);
    CAT_CUDA(cudaMemsetAsync(o.words.get(), 0, 8, s));
    SieveArgs sa{c.seeds + 1, i_med, i_large, nodd, imax, lg, o.bits.get(), o.offsets.get(),
                 unit_kind, unit_n, (uint32_t)root, o.words.get() + 1};
    const int tok = prof_begin(c, "sieve_segments", s);
    launch_chained(sieve_segments, nsegs, std::min(kSieveThreads, 1 << (lg - 5)),
                   (size_t)4 << (lg - 5), s, sa);
    CAT_LAUNCH("sieve_segments");
    prof_end(c, tok, s, 4.0 * (double)o.units * kUnitWords);
    exclusive_scan_u32(c, o.offsets.get(), o.units, s, o.words.get());
    return o;
}

void factor(Ctx &c, uint64_t n, int kind, cat_factorization *out, cudaStream_t s)
{
    if (n >= (1ull << 31)) fail(CAT_EINVAL, "n must be below 2^31");
    if (kind < CAT_CATALAN || kind > CAT_FACTORIAL) fail(CAT_EINVAL, "unknown kind");
    Ratio r{};
    r.kind = kind;
    r.n = (uint32_t)n;
    factor_ratio(c, r, out, s);
}

// (e, p) items with e = 0 dropped, grouped by e: primes ascending within each
// group, groups by ascending e, offs[k] = start of group k (offs has one more
// entry than exps, ending in count).
struct Grouped {
    DevBuf<uint32_t> primes;
    std::vector<uint64_t> exps, offs{0};
    uint64_t count = 0;
};

static Grouped group_items(Ctx &c, DevBuf<uint64_t> &items, size_t count, uint32_t max_e,
                           cudaStream_t s)
{
    Grouped g;
    // stable radix sort by e, dropping e = 0
    int ebits = 0;
    while (ebits < 32 && (max_e >> ebits)) ebits++;
    DevBuf<uint64_t> alt(c, std::max<size_t>(count, 1), s);
    DevBuf<uint32_t> kept(c, 1, s);
    uint64_t *src = items.get(), *dst = alt.get();
    int tok;
    for (int shift = 0, pass = 0; pass == 0 || shift < ebits; pass++) {
        const int bitsd = std::max(1, std::min(8, ebits - shift));
        const size_t tiles = (count + kRsTile - 1) / kRsTile;
        if (tiles == 0) break;
        const size_t nbins = (size_t)1 << bitsd;
        DevBuf<uint32_t> cnt(c, nbins * tiles, s);
        RsArgs ra{src, dst, count, shift, bitsd, pass == 0 ? 1 : 0, cnt.get(), tiles};
        tok = prof_begin(c, "rs_histogram", s);
        launch_chained(rs_histogram, (unsigned)tiles, kRsThreads, 0, s, ra);
        CAT_LAUNCH("rs_histogram");
        prof_end(c, tok, s, 8.0 * (double)count);
        exclusive_scan_u32(c, cnt.get(), nbins * tiles, s, kept.get());
        tok = prof_begin(c, "rs_scatter", s);
        launch_chained(rs_scatter, (unsigned)tiles, kRsThreads, 0, s, ra);
        CAT_LAUNCH("rs_scatter");
        prof_end(c, tok, s, 16.0 * (double)count);
        // only the first pass drops items
        if (pass == 0) count = *read_back(c, kept.get(), 1, s);
        std::swap(src, dst);
        shift += bitsd;
        if (ebits == 0) break;
    }
    g.count = count;
    if (count == 0) return g;
    g.primes = DevBuf<uint32_t>(c, count, s);
    DevBuf<uint64_t> starts(c, 2 * count, s);
    DevBuf<unsigned int> nst(c, 1, s);
    CAT_CUDA(cudaMemsetAsync(nst.get(), 0, 4, s));
    launch_chained(group_starts, (unsigned)((count + 255) / 256), 256, 0, s, src, count,
                   starts.get(), nst.get(), g.primes.get());
    CAT_LAUNCH("group_starts");
    const unsigned int ng = *read_back(c, nst.get(), 1, s);
    std::vector<uint64_t> hst(2 * (size_t)ng);
    CAT_CUDA(cudaMemcpyAsync(hst.data(), starts.get(), 16 * (size_t)ng, cudaMemcpyDeviceToHost,
                             s));
    CAT_CUDA(cudaStreamSynchronize(s));
    std::vector<std::pair<uint64_t, uint64_t>> gs(ng);
    for (size_t k = 0; k < ng; k++) gs[k] = {hst[2 * k], hst[2 * k + 1]};
    std::sort(gs.begin(), gs.end());
    g.offs.clear();
    for (auto &x : gs) {
        g.exps.push_back(x.first);
        g.offs.push_back(x.second);
    }
    g.offs.push_back(count);
    return g;
}

// Catalan or central binomial kinds with n >= 2.  Every prime above sqrt(2n)
// has exponent 0 or 1; the sieve keeps those with 1 and they are written in
// order straight into the e = 1 group, after the seed primes with e = 1.  The
// seed primes (<= sqrt(2n), at most 6542) are grouped by one block; their
// groups with e >= 2 follow.
static void factor_unit(Ctx &c, const Ratio &r, uint64_t limit, cat_factorization *out,
                        cudaStream_t s)
{
    SieveOut sv = run_sieve(c, limit, s, r.kind, r.n);
    const uint32_t ns = sv.nseeds;
    DevBuf<uint32_t> sorted(c, std::max<uint32_t>(ns, 1), s);
    DevBuf<Phase1Info> d_info(c, 1, s);
    int tok = prof_begin(c, "group_seeds", s);
    launch_chained(group_seeds, 1, kSeedThreads, kSeedSmem, s, c.seeds, ns, r, sv.words.get(),
                   sv.words.get() + 1, sorted.get(), d_info.get());
    CAT_LAUNCH("group_seeds");
    prof_end(c, tok, s, 8.0 * (double)ns);
    Phase1Info h;
    memcpy(&h, read_back(c, d_info.get(), sizeof(h) / 4, s), sizeof(h));
    if (h.negative) fail(CAT_ENOTINTEGRAL, "a prime exponent is negative");
    CsrArgs a{};
    a.nl = h.kept;
    a.n1 = h.ngroups && h.exp[0] == 1 ? h.off[1] : 0;
    a.nsorted = h.off[h.ngroups];
    const uint64_t npos = (uint64_t)a.nsorted + a.nl;
    if (a.n1 + a.nl) a.h_exps[a.ng++] = 1;
    for (uint32_t k = a.n1 ? 1 : 0; k < h.ngroups; k++) {
        a.h_offs[a.ng] = (uint64_t)h.off[k] + a.nl;
        a.h_exps[a.ng++] = h.exp[k];
    }
    a.h_offs[a.ng] = npos;
    DevBuf<uint32_t> primes(c, std::max<uint64_t>(npos, 1), s);
    DevBuf<uint64_t> d_exps(c, a.ng + 1, s), d_offs(c, a.ng + 1, s);
    a.bits = sv.bits.get();
    a.unit_offsets = sv.offsets.get();
    a.units = sv.units;
    a.expand_blocks = a.nl ? (sv.units + kExpandWarps - 1) / kExpandWarps : 0;
    a.sorted = sorted.get();
    a.primes = primes.get();
    a.exps = d_exps.get();
    a.offs = d_offs.get();
    tok = prof_begin(c, "write_csr", s);
    launch_chained(write_csr, a.expand_blocks + 1, kExpandThreads, 0, s, a);
    CAT_LAUNCH("write_csr");
    prof_end(c, tok, s, 4.0 * (double)sv.units * kUnitWords + 4.0 * (double)npos);
    out->host_exps = new uint64_t[a.ng + 1];
    out->host_offsets = new uint64_t[a.ng + 1];
    std::copy(a.h_exps, a.h_exps + a.ng + 1, out->host_exps);
    std::copy(a.h_offs, a.h_offs + a.ng + 1, out->host_offsets);
    out->num_groups = a.ng;
    out->num_primes = npos;
    out->primes_sieved = (uint64_t)h.total + 1;  // plus the prime 2
    out->exps = d_exps.release();
    out->offsets = d_offs.release();
    out->primes = primes.release();
}

// Phase 1 for any Ratio: primes up to the largest factorial argument (2n for
// the binomial kinds, n for n!, the largest term of a ratio).
void factor_ratio(Ctx &c, const Ratio &r, cat_factorization *out, cudaStream_t s)
{
    NvtxRange range("phase1: sieve, exponents, grouping");
    *out = cat_factorization{};
    const int kind = r.kind;
    const uint64_t n = r.n;
    uint64_t limit = kind == CAT_FACTORIAL ? n : 2 * n;
    if (kind == kRatioKind) {
        limit = 0;
        for (int i = 0; i < r.ka; i++) limit = std::max<uint64_t>(limit, r.a[i]);
        for (int j = 0; j < r.kb; j++) limit = std::max<uint64_t>(limit, r.b[j]);
    }
    if ((kind == CAT_CATALAN || kind == CAT_CENTRAL_BINOMIAL) && n >= 2) {
        factor_unit(c, r, limit, out, s);
        return;
    }
    std::vector<uint64_t> h_exps, h_offs{0};
    DevBuf<uint32_t> primes_out;
    uint64_t sieved = 0, npos = 0;
    if (limit >= 2) {
        SieveOut sv = run_sieve(c, limit, s);
        sieved = (uint64_t)*read_back(c, sv.words.get(), 1, s) + 1;  // plus the prime 2
        // exponents
        DevBuf<uint64_t> items(c, sieved, s);
        DevBuf<unsigned int> flags(c, 2, s);
        CAT_CUDA(cudaMemsetAsync(flags.get(), 0, 8, s));
        ExpandArgs ea{sv.bits.get(), sv.offsets.get(), sv.units, r, items.get(), flags.get(),
                      flags.get() + 1};
        const int tok = prof_begin(c, "expand_exponents", s);
        launch_chained(expand_exponents, (sv.units + kExpandWarps - 1) / kExpandWarps,
                       kExpandThreads, 0, s, ea);
        CAT_LAUNCH("expand_exponents");
        prof_end(c, tok, s, 4.0 * (double)sv.units * kUnitWords + 8.0 * (double)sieved);
        sv = SieveOut{};
        const uint32_t *hf = read_back(c, flags.get(), 2, s);
        if (hf[1]) fail(CAT_ENOTINTEGRAL, "a prime exponent is negative");
        Grouped g = group_items(c, items, sieved, hf[0], s);
        npos = g.count;
        primes_out = std::move(g.primes);
        h_exps = std::move(g.exps);
        h_offs = std::move(g.offs);
    }
    const size_t ng = h_exps.size();
    DevBuf<uint64_t> d_exps(c, ng + 1, s), d_offs(c, ng + 1, s);
    if (!primes_out.get()) primes_out = DevBuf<uint32_t>(c, 1, s);
    out->host_exps = new uint64_t[ng + 1];
    out->host_offsets = new uint64_t[ng + 1];
    for (size_t k = 0; k < ng; k++) out->host_exps[k] = h_exps[k];
    out->host_exps[ng] = 0;
    for (size_t k = 0; k <= ng; k++) out->host_offsets[k] = h_offs[k];
    CAT_CUDA(cudaMemcpyAsync(d_exps.get(), out->host_exps, 8 * (ng + 1),
                             cudaMemcpyHostToDevice, s));
    CAT_CUDA(cudaMemcpyAsync(d_offs.get(), out->host_offsets, 8 * (ng + 1),
                             cudaMemcpyHostToDevice, s));
    CAT_CUDA(cudaStreamSynchronize(s));
    out->num_groups = ng;
    out->num_primes = npos;
    out->primes_sieved = sieved;
    out->exps = d_exps.release();
    out->offsets = d_offs.release();
    out->primes = primes_out.release();
}

DevBuf<uint32_t> sieve_primes(Ctx &c, uint64_t limit, uint64_t *count, cudaStream_t s)
{
    *count = 0;
    if (limit < 2) return DevBuf<uint32_t>(c, 1, s);
    SieveOut sv = run_sieve(c, limit, s);
    const uint64_t sieved = (uint64_t)*read_back(c, sv.words.get(), 1, s) + 1;
    DevBuf<uint32_t> primes(c, sieved, s);
    const int tok = prof_begin(c, "expand_primes", s);
    launch_chained(expand_primes, (sv.units + kExpandWarps - 1) / kExpandWarps, kExpandThreads, 0,
                   s, sv.bits.get(), sv.offsets.get(), sv.units, primes.get(), 1, 1);
    CAT_LAUNCH("expand_primes");
    prof_end(c, tok, s, 4.0 * (double)sv.units * kUnitWords + 4.0 * (double)sieved);
    *count = sieved;
    return primes;
}

void factor_free(Ctx &c, cat_factorization *f, cudaStream_t s)
{
    if (!f) return;
    dev_free(c, f->exps, 8 * (f->num_groups + 1), s);
    dev_free(c, f->offsets, 8 * (f->num_groups + 1), s);
    dev_free(c, f->primes, 4 * (f->num_primes ? f->num_primes : 1), s);
    delete[] f->host_exps;
    delete[] f->host_offsets;
    *f = cat_factorization{};
}

}  // namespace cat
