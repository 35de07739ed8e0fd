// tree.cu -- Phase 2 of the method (Sec. 3.2, Algorithm 2): the balanced
// product tree, binary powering and the final product, as level-synchronous
// batched multiplications on the device.
//
// Product tree.  The leaves (32-bit primes) are combined eight at a time into
// 8-limb nodes; every further level multiplies adjacent nodes (2i, 2i+1) of a
// fixed slot size S into slots of 2S limbs (a product of 2^k values below 2^32
// always fits 2^k limbs), with an odd last node carried up unchanged.  All
// products of one level are one batched launch: schoolbook (Comba) kernels
// for small slots, a one-block transform for products up to 2^12 limbs, and
// the multi-pass transform above.  Nodes of a level hold equally many primes,
// which is what keeps the tree balanced.
#include "cat_internal.cuh"
#include "length_bits.h"

#include <math.h>

#include <algorithm>
#include <vector>

namespace cat {

// comba.cu
void leaf_level(Ctx &c, const uint32_t *values, size_t count, const Repeats &rep, uint32_t *out,
                size_t nodes, int lpn, cudaStream_t s);
// ntt.cu
void ntt_mul(Ctx &c, const uint32_t *a, size_t na, const uint32_t *b, size_t nb,
             uint32_t *out, cudaStream_t s);

constexpr size_t kLeafSlot = 8;

static Big make_one(Ctx &c, cudaStream_t s)
{
    Big r;
    r.buf = DevBuf<uint32_t>(c, 1, s);
    static const uint32_t one = 1;
    CAT_CUDA(cudaMemcpyAsync(r.buf.get(), &one, 4, cudaMemcpyHostToDevice, s));
    CAT_CUDA(cudaStreamSynchronize(s));
    r.n = 1;
    return r;
}

// Length of x[0..n) after dropping zero top limbs, reading only the top few
// limbs when they decide it.
size_t trim(Ctx &c, const uint32_t *x, size_t n, cudaStream_t s)
{
    if (n == 0) return 0;
    const size_t k = std::min<size_t>(n, 4);
    const uint32_t *h = read_back(c, x + n - k, (int)k, s);
    for (size_t i = k; i-- > 0;)
        if (h[i]) return n - k + i + 1;
    return normalized_length(c, x, n - k, s);
}

// Relative cost of a butterfly in the prime set of a product of 2^n limbs
// (measured: set 1 ~1.1x and set 2 ~1.5x the lazy set 0).
static double set_cost(int n)
{
    const int ps = set_for(n - 1);
    return ps == 0 ? 1.0 : (ps == 1 ? 1.1 : 1.5);
}

static int clog2(size_t x)
{
    int n = 0;
    while (((size_t)1 << n) < x) n++;
    return n;
}

// For a long x and a short y: the chunk transform size 2^k whose estimated
// cost (transform points x log2 points x set cost, and 4 per limb of the result)
// beats one product of nx + ny limbs, or 0 if none does.  2 chunks + 1
// transforms are what a product in transforms of 2^13 points or more takes (y's
// is shared); shorter chunks take y's again each and an overlap pass besides.
// Measured (us, one product : chunks), where chunks are taken: 2 10^7 x 6.7 10^6
// limbs 1,426 : 1,236, 5 10^6 x 1.7 10^6 382 : 317, 10^6 x 10^5 112 : 95; but
// 4 10^5 x 1.95 10^5 78 : 83 and 50,000 x 1,667 48 : 67: below about 5 10^5
// limbs the estimate sees no fixed costs and one product would do as well or
// better.  Where they are not taken: 5 10^6 x 2.4 10^6 383 : 387, 4 10^5 x 10^5
// 68 : 69, 10^5 x 1.7 10^4 48 : 48.
static int chunk_log(const Ctx &c, size_t nx, size_t ny)
{
    if (nx < 2 * ny || nx + ny <= 4096) return 0;
    const int nf = clog2(nx + ny);
    double best = nf <= c.max_log ? 3.0 * ldexp(1.0, nf) * nf * set_cost(nf) : 1e300;
    int bk = 0;
    for (int k = std::max(1, clog2(2 * ny)); k <= std::min(c.max_log, nf); k++) {
        const double L = ldexp(1.0, k), M = L - (double)ny;
        const double chunks = ceil((double)nx / M);
        const double cost = (2.0 * chunks + 1.0) * L * k * set_cost(k) + 4.0 * (double)(nx + ny);
        if (cost < best) {
            best = cost;
            bk = k;
        }
    }
    return bk;
}

void mul_into(Ctx &c, const uint32_t *a, size_t na, const uint32_t *b, size_t nb,
              uint32_t *out, cudaStream_t s)
{
    if (na == 0 || nb == 0) {
        if (na + nb) CAT_CUDA(cudaMemsetAsync(out, 0, 4 * (na + nb), s));
        return;
    }
    // unbalanced: chunks of the long operand against the short one
    {
        const bool swap = na < nb;
        const uint32_t *x = swap ? b : a, *y = swap ? a : b;
        const size_t nx = swap ? nb : na, ny = swap ? na : nb;
        if (const int k = chunk_log(c, nx, ny)) {
            mul_chunked(c, x, nx, y, ny, k, out, s);
            return;
        }
    }
    if (na + nb <= ((size_t)1 << c.max_log)) {
        ntt_mul(c, a, na, b, nb, out, s);
        return;
    }
    // longer than one transform: pieces of at most 2^26 limbs, accumulated
    CAT_CUDA(cudaMemsetAsync(out, 0, 4 * (na + nb), s));
    mul_acc(c, a, na, b, nb, out, na + nb, false, s);
}

static Big copy_big(Ctx &c, const uint32_t *a, size_t n, cudaStream_t s);
static Big mul_big(Ctx &c, const Big &x, const Big &y, cudaStream_t s, bool exact = true);

// Levels above the leaves of a tree over `count` values, lpn to a node.
static int tree_depth(size_t count, int lpn)
{
    size_t nodes = (count + lpn - 1) / lpn;
    int d = 0;
    for (; nodes > 1; d++) nodes = (nodes + 1) / 2;
    return d;
}

// The product of values[0 .. count) (times *extra when given).  extra joins
// the tree as one node: the count is padded with values 1 up to a multiple of
// a slot size S >= extra's length, plus S more, so that at slot S the last
// node is exactly 1 and extra takes its place.  Every node still fits its
// slot, so the levels above are unchanged; only when the padding would add a
// level is extra multiplied in at the end instead.  exact = false returns the
// top slot (zero-padded) as the length instead of reading the true length
// back: no host synchronisation.  With `direct` the last product goes straight
// to the caller's buffer when one transform forms it.
Big tree_product(Ctx &c, const uint32_t *values, size_t count, cudaStream_t s, const Big *extra,
                 bool exact, int leaf_bits, const Repeats *rep, Direct *direct)
{
    NvtxRange range("product tree");
    static const Repeats none{};
    if (!rep) rep = &none;
    const size_t own = count;
    count += rep->groups ? rep->start[rep->groups] - rep->start[0] : 0;
    if (count == 0) return extra ? copy_big(c, extra->buf.get(), extra->n, s) : make_one(c, s);
    const int lpn = leaves_per_node(leaf_bits);
    size_t total = count, inj_slot = 0;
    if (extra) {
        size_t S = 2 * kLeafSlot;
        while (S < extra->n) S <<= 1;
        const size_t per = S / kLeafSlot * (size_t)lpn;  // leaves under one node of slot S
        const size_t padded = (count + per - 1) / per * per + per;
        if (tree_depth(padded, lpn) == tree_depth(count, lpn)) {
            total = padded;
            inj_slot = S;
        }
    }
    size_t slot = kLeafSlot;
    size_t nodes = (total + lpn - 1) / lpn;
    DevBuf<uint32_t> cur(c, nodes * slot, s);
    leaf_level(c, values, own, *rep, cur.get(), nodes, lpn, s);
    while (nodes > 1) {
        NvtxRange level("tree level");
        if (direct && direct->out && nodes == 2 && !extra && slot > c.comba_max_slot &&
            ntt_level_whole(c, slot)) {
            const size_t len = std::min(2 * slot, direct->len);
            ntt_pair(c, cur.get(), slot, direct->out, len, s);
            direct->used = true;
            Big r;
            r.n = trim(c, direct->out, len, s);
            return r;
        }
        const size_t nprod = nodes / 2, odd = nodes & 1, nn = nprod + odd, ns = 2 * slot;
        DevBuf<uint32_t> nxt(c, nn * ns, s);
        if (slot > c.comba_max_slot || !comba_level(c, cur.get(), slot, nprod, nxt.get(), s))
            ntt_level(c, cur.get(), slot, nprod, nxt.get(), s);
        if (odd) {
            CAT_CUDA(cudaMemcpyAsync(nxt.get() + nprod * ns, cur.get() + (nodes - 1) * slot,
                                     4 * slot, cudaMemcpyDeviceToDevice, s));
            CAT_CUDA(cudaMemsetAsync(nxt.get() + nprod * ns + slot, 0, 4 * slot, s));
        }
        if (ns == inj_slot) {  // the last node covers only padding: replace its 1 by extra
            uint32_t *last = nxt.get() + (nn - 1) * ns;
            CAT_CUDA(cudaMemcpyAsync(last, extra->buf.get(), 4 * extra->n,
                                     cudaMemcpyDeviceToDevice, s));
            if (extra->n < ns)
                CAT_CUDA(cudaMemsetAsync(last + extra->n, 0, 4 * (ns - extra->n), s));
            inj_slot = 0;
            extra = nullptr;
        }
        cur = std::move(nxt);
        nodes = nn;
        slot = ns;
    }
    Big r;
    r.n = exact ? normalized_length(c, cur.get(), slot, s) : slot;
    r.buf = std::move(cur);
    if (extra) return mul_big(c, r, *extra, s, exact);
    return r;
}

static Big copy_big(Ctx &c, const uint32_t *a, size_t n, cudaStream_t s)
{
    Big r;
    r.buf = DevBuf<uint32_t>(c, n ? n : 1, s);
    if (n) CAT_CUDA(cudaMemcpyAsync(r.buf.get(), a, 4 * n, cudaMemcpyDeviceToDevice, s));
    r.n = n;
    return r;
}

// x y; exact = false keeps the bound x.n + y.n as the length (zero top limbs)
// instead of reading the true length back.
static Big mul_big(Ctx &c, const Big &x, const Big &y, cudaStream_t s, bool exact)
{
    Big r;
    const size_t n = x.n + y.n;
    r.buf = DevBuf<uint32_t>(c, n ? n : 1, s);
    mul_into(c, x.buf.get(), x.n, y.buf.get(), y.n, r.buf.get(), s);
    r.n = exact ? trim(c, r.buf.get(), n, s) : n;
    return r;
}

// x y for numbers whose bits are tracked: the product's length bound comes from
// its bits (length_bits.h: never below the true length, and at most one limb
// above it), so that a chain of products needs no read-back between its steps.
static Big mul_bits(Ctx &c, const Big &x, const Big &y, cudaStream_t s)
{
    Big r = mul_big(c, x, y, s, false);
    r.bits = product_bits(x.bits, y.bits);
    r.n = std::min<size_t>(r.n, bits_limbs(r.bits));
    return r;
}

// a^e, left-to-right binary (the powering step of Algorithm 2).  Squarings reuse
// one forward transform.  exact = false takes a (nonzero) as given, with zero
// top limbs allowed, and returns a bound as the length: no host
// synchronisation; exact = true reads a's length and top limbs first and the
// result's length last, and nothing between.
Big power(Ctx &c, const uint32_t *a, size_t na, uint64_t e, cudaStream_t s, bool exact)
{
    NvtxRange range("power");
    Big base = copy_big(c, a, na, s);
    if (exact) {
        // a caller's buffer may be zero far above the value (four stretches of
        // the one block, then the whole chip: 1,000 limbs below 4 million zeros,
        // to the third power, 90 us; 1,776 us by the block alone, 62 without zeros)
        Big *p = &base;
        normalize_all(c, &p, 1, s, 4096);
    }
    if (e == 0) return make_one(c, s);
    if (base.n == 0) return base;
    Big r = copy_big(c, base.buf.get(), base.n, s);
    r.bits = base.bits;
    int top = 63;
    while (!((e >> top) & 1)) top--;
    for (int bit = top - 1; bit >= 0; bit--) {
        r = exact ? mul_bits(c, r, r, s) : mul_big(c, r, r, s, false);
        if ((e >> bit) & 1) r = exact ? mul_bits(c, r, base, s) : mul_big(c, r, base, s, false);
    }
    if (exact) r.n = trim(c, r.buf.get(), r.n, s);
    return r;
}

// Factorisations with more exponent groups than this (n! has about 2 sqrt(n))
// take the bit-decomposed form below; Catalan numbers and central binomials
// (at most 33 groups) always take Algorithm 2 as written.
constexpr uint64_t kManyGroups = kMaxRepeats;

// Leaves of the bit segments: segment b holds the primes of the groups whose
// exponent has bit b set, group after group.
constexpr int kExpBits = 64;
struct BitSegments {
    uint64_t start[kExpBits + 1];
};

// at[b ng + g]: the first leaf of group g in segment b; block b scans the
// groups, 1,024 at a time.
__global__ void __launch_bounds__(1024) bit_offsets(const uint64_t *exps, const uint64_t *offs,
                                                    uint32_t ng,
                                                    const __grid_constant__ BitSegments seg,
                                                    uint64_t *at)
{
    chain_wait();
    __shared__ uint64_t wsum[32];
    const int b = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t run = seg.start[b];
    for (uint32_t g0 = 0; g0 < ng; g0 += 1024) {
        const uint32_t g = g0 + threadIdx.x;
        const uint64_t c = g < ng && (exps[g] >> b & 1) ? offs[g + 1] - offs[g] : 0;
        uint64_t incl = c;
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        uint64_t before = 0, total = 0;
        for (int w = 0; w < 32; w++) {
            before += w < wid ? wsum[w] : 0;
            total += wsum[w];
        }
        if (g < ng) at[(size_t)b * ng + g] = run + before + incl - c;
        run += total;
        __syncthreads();
    }
}

// One thread per prime of the groups: its group by bisection, then one leaf per
// bit of the exponent.
__global__ void bit_leaves(const uint32_t *primes, const uint64_t *exps, const uint64_t *offs,
                           uint32_t ng, const uint64_t *at, uint32_t *leaves)
{
    chain_wait();
    const uint64_t i = offs[0] + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= offs[ng]) return;
    uint32_t lo = 0, hi = ng;  // offs[lo] <= i < offs[hi]
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (offs[mid] <= i) lo = mid;
        else hi = mid;
    }
    const uint32_t p = primes[i];
    const uint64_t k = i - offs[lo];
    uint64_t e = exps[lo];
    while (e) {
        const int b = __ffsll((long long)e) - 1;
        e &= e - 1;
        leaves[at[(size_t)b * ng + lo] + k] = p;
    }
}

// prod_e Q_e^e = prod_b R_b^(2^b), R_b = prod of Q_e over the groups whose
// exponent has bit b set.  All R_b come from one segmented tree over the
// primes (segment b = the primes of those groups), then
// X = R_top; X = X^2 R_b for b below the top bit.  Same integer as
// Algorithm 2 with about 2 log2(max e) large multiplications instead of one
// powering chain per group.
static Big reconstruct_bits(Ctx &c, const cat_factorization *f, cudaStream_t s, int leaf_bits)
{
    uint64_t emax = 0;
    for (uint64_t g = 0; g < f->num_groups; g++) emax = std::max(emax, f->host_exps[g]);
    int B = 0;
    while (B < kExpBits && (emax >> B)) B++;
    std::vector<uint64_t> seg(B + 1, 0);
    for (uint64_t g = 0; g < f->num_groups; g++)
        for (int b = 0; b < B; b++)
            if ((f->host_exps[g] >> b) & 1)
                seg[b + 1] += f->host_offsets[g + 1] - f->host_offsets[g];
    for (int b = 0; b < B; b++) seg[b + 1] += seg[b];
    if (seg[B] == 0) return make_one(c, s);
    DevBuf<uint32_t> leaves(c, seg[B], s);
    const uint32_t ng = (uint32_t)f->num_groups;
    std::vector<uint64_t> groups;
    {
        const uint64_t *exps = f->exps, *offs = f->offsets;
        DevBuf<uint64_t> d_groups;
        if (!exps) {  // a caller's factorisation
            groups.assign(f->host_exps, f->host_exps + ng);
            groups.insert(groups.end(), f->host_offsets, f->host_offsets + ng + 1);
            d_groups = DevBuf<uint64_t>(c, groups.size(), s);
            CAT_CUDA(cudaMemcpyAsync(d_groups.get(), groups.data(), 8 * groups.size(),
                                     cudaMemcpyHostToDevice, s));
            exps = d_groups.get();
            offs = exps + ng;
        }
        const uint64_t np = f->host_offsets[ng] - f->host_offsets[0];
        DevBuf<uint64_t> at(c, (size_t)B * ng, s);
        BitSegments sb{};
        std::copy(seg.begin(), seg.end(), sb.start);
        launch_chained(bit_offsets, B, 1024, 0, s, exps, offs, ng, sb, at.get());
        CAT_LAUNCH("bit_offsets");
        const int tok = prof_begin(c, "bit_leaves", s);
        launch_chained(bit_leaves, (unsigned)((np + 255) / 256), 256, 0, s, f->primes, exps, offs,
                       ng, at.get(), leaves.get());
        CAT_LAUNCH("bit_leaves");
        prof_end(c, tok, s, 4.0 * (double)(np + seg[B]));
    }
    std::vector<TreeRoot> R(B);
    segmented_tree(c, leaves.get(), seg, R, s, leaf_bits);
    leaves.reset();
    std::vector<Big *> roots;
    for (int b = 0; b < B; b++) {
        // a root's slot has a limb per leaf; its value ends with the leaves' bits
        Big &r = R[b].big;
        r.n = std::min<size_t>(r.n, (seg[b + 1] - seg[b]) * (uint64_t)leaf_bits / 32 + 1);
        roots.push_back(&r);
    }
    // (the bounds exceed the lengths by a few per cent, which the roots' blocks
    // scan side by side)
    normalize_all(c, roots.data(), B, s);
    Big X = std::move(R[B - 1].big);
    for (int b = B - 2; b >= 0; b--) {
        X = mul_bits(c, X, X, s);
        if (seg[b + 1] > seg[b]) X = mul_bits(c, X, R[b].big, s);
    }
    X.n = trim(c, X.buf.get(), X.n, s);
    return X;
}

// The groups with e >= 2 as leaves of Q_1's own tree, every prime e times (the
// same integer, re-associated), when that adds at most a quarter to the tree
// or 4,096 leaves; false otherwise.  For C(n) and C(2n, n) those primes are at
// most sqrt(2n), so they are a handful of leaves, where forming every Q_e, its
// power and their product took about 25 short launches one after the other at
// n = 10^5 and 40 at the paper's n (with the last product straight into the
// caller's buffer: C(10^5) 0.43 -> 0.22 ms, C(5 10^7) 2.27 -> 1.92,
// C(2,050,572,903) 81.2 -> 80.6).  The line bounds the leaves, one per unit of
// an exponent, to the tree's own size; the powers do not win above it.  Measured
// (us, powers : leaves) on (3n)! / n!^3, whose groups with e = 2 hold 0.9 times
// Q_1's primes: n = 20,000 (3,168 more leaves, leaves taken) 484 : 278, 50,000
// (7,211, powers taken) 681 : 313, 10^6 (110,545, powers taken) 887 : 453.
static bool repeat_leaves(const cat_factorization *f, Repeats &rep, uint64_t &off1, uint64_t &cnt1)
{
    uint64_t more = 0;
    off1 = cnt1 = 0;
    rep.base = f->primes;
    for (uint64_t g = 0; g < f->num_groups; g++) {
        const uint64_t off = f->host_offsets[g], cnt = f->host_offsets[g + 1] - off;
        const uint64_t e = f->host_exps[g];
        if (e == 1) {
            off1 = off;
            cnt1 = cnt;
            continue;
        }
        if (e > 0xffffffffull || cnt > (1ull << 40) / e) return false;
        rep.off[rep.groups] = off;
        rep.times[rep.groups] = (uint32_t)e;
        rep.start[rep.groups] = more;
        more += e * cnt;
        rep.start[++rep.groups] = more;
    }
    for (int g = 0; g <= rep.groups; g++) rep.start[g] += cnt1;  // behind Q_1's leaves
    return more <= std::max<uint64_t>(cnt1 / 4, 4096);
}

// Algorithm 2: Q_e by the tree, P_e = Q_e^e, then the P_e combined by
// repeatedly multiplying the two shortest (equal-length operands meet
// first, so intermediates stay as short as possible).
Big reconstruct(Ctx &c, const cat_factorization *f, cudaStream_t s, int leaf_bits, Direct *direct)
{
    NvtxRange range("phase2: reconstruction");
    if (f->num_groups > kManyGroups) return reconstruct_bits(c, f, s, leaf_bits);
    {
        Repeats rep;
        uint64_t off1 = 0, cnt1 = 0;
        if (repeat_leaves(f, rep, off1, cnt1))
            return tree_product(c, f->primes + off1, cnt1, s, nullptr, true, leaf_bits, &rep,
                                direct);
    }
    // P_e = Q_e^e for e >= 2 first, combined into R; then Q_1's tree takes R
    // in as one of its nodes, so that the long P_1 needs no final product
    // (the same integer: the final product of the P_e, re-associated).  The
    // small P_e and R carry length bounds (zero top limbs), so that none of
    // their many short steps waits for a read-back; only the end result is
    // normalised.
    std::vector<Big> P;
    int64_t g1 = -1;
    for (uint64_t g = 0; g < f->num_groups; g++) {
        if (f->host_exps[g] == 1) {
            g1 = (int64_t)g;
            continue;
        }
        const uint64_t off = f->host_offsets[g], cnt = f->host_offsets[g + 1] - off;
        Big Q = tree_product(c, f->primes + off, cnt, s, nullptr, false, leaf_bits);
        P.push_back(power(c, Q.buf.get(), Q.n, f->host_exps[g], s, false));
    }
    while (P.size() > 1) {
        std::sort(P.begin(), P.end(), [](const Big &x, const Big &y) { return x.n > y.n; });
        Big x = std::move(P.back());
        P.pop_back();
        Big y = std::move(P.back());
        P.pop_back();
        P.push_back(mul_big(c, x, y, s, false));
    }
    if (g1 < 0) {
        if (P.empty()) return make_one(c, s);
        P[0].n = normalized_length(c, P[0].buf.get(), P[0].n, s);
        return std::move(P[0]);
    }
    const uint64_t off = f->host_offsets[g1], cnt = f->host_offsets[g1 + 1] - off;
    return tree_product(c, f->primes + off, cnt, s, P.empty() ? nullptr : &P[0], true, leaf_bits);
}

}  // namespace cat
