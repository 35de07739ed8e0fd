// comba.cu -- the lower levels of the balanced product tree (Sec. 3.2):
// many independent small products by schoolbook multiplication: column-wise
// ("Comba") with 96-bit column accumulators, by a thread (8 limbs) or a warp
// per product, or row-wise by one or two threads per product where there are
// enough products (comba_rows).
//
// Layout: a tree level is an array of nodes in fixed slots of S limbs (node i
// at [i S, (i+1) S)), zero-padded.  A product of 2^k values below 2^32 always
// fits in 2^k limbs, so the product of adjacent nodes (2i, 2i+1) fits the
// next level's slot of 2S limbs exactly.
#include "cat_internal.cuh"
#include "length_bits.h"

#include <string.h>

namespace cat {

// c2:c1:c0 += a * b  (96-bit accumulator)
__device__ __forceinline__ void mac96(uint32_t a, uint32_t b, uint32_t &c0, uint32_t &c1,
                                      uint32_t &c2)
{
    asm("mad.lo.cc.u32 %0, %3, %4, %0;\n\t"
        "madc.hi.cc.u32 %1, %3, %4, %1;\n\t"
        "addc.u32 %2, %2, 0;\n\t"
        : "+r"(c0), "+r"(c1), "+r"(c2)
        : "r"(a), "r"(b));
}

// --------------------------------------------------------------- leaves

constexpr int kLeafSlot = 8;

// Leaf idx of a tree over values[0 .. count) followed by the repeated groups
// (1 past the end).
__device__ __forceinline__ uint32_t leaf_value(const uint32_t *v, size_t count, const Repeats &rep,
                                               size_t idx)
{
    if (idx < count) return v[idx];
    int g = 0;
    while (g < rep.groups && idx >= rep.start[g + 1]) g++;
    return g < rep.groups ? rep.base[rep.off[g] + (idx - rep.start[g]) / rep.times[g]] : 1u;
}

// Node i (eight limbs) = product of the leaves [lpn i, lpn i + lpn) (those
// past the end count as 1; the caller picks lpn so that the product fits),
// accumulated by single-limb multiplications.
__global__ void leaf_products(const uint32_t *v, size_t count, const __grid_constant__ Repeats rep,
                              uint32_t *out, size_t nodes, int lpn)
{
    chain_wait();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nodes) return;
    uint32_t acc[kLeafSlot];
#pragma unroll
    for (int j = 0; j < kLeafSlot; j++) acc[j] = 0;
    acc[0] = 1;
    for (int k = 0; k < lpn; k++) {
        const uint32_t x = leaf_value(v, count, rep, i * (size_t)lpn + k);
        uint32_t carry = 0;
#pragma unroll
        for (int j = 0; j < kLeafSlot; j++) {
            const uint64_t t = (uint64_t)acc[j] * x + carry;
            acc[j] = (uint32_t)t;
            carry = (uint32_t)(t >> 32);
        }
    }
    uint4 *o = reinterpret_cast<uint4 *>(out + i * kLeafSlot);
    o[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
    o[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
}

// ---------------------------------------------- one product per thread

template <int S>
__global__ void comba_thread(const uint32_t *in, size_t nprod, uint32_t *out,
                             const uint32_t *out_index)
{
    chain_wait();
    const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nprod) return;
    const uint4 *a4 = reinterpret_cast<const uint4 *>(in + 2 * k * S);
    uint32_t A[S], B[S], O[2 * S];
#pragma unroll
    for (int i = 0; i < S / 4; i++) {
        const uint4 x = a4[i], y = a4[S / 4 + i];
        A[4 * i] = x.x; A[4 * i + 1] = x.y; A[4 * i + 2] = x.z; A[4 * i + 3] = x.w;
        B[4 * i] = y.x; B[4 * i + 1] = y.y; B[4 * i + 2] = y.z; B[4 * i + 3] = y.w;
    }
    uint32_t c0 = 0, c1 = 0, c2 = 0;
#pragma unroll
    for (int col = 0; col < 2 * S - 1; col++) {
#pragma unroll
        for (int i = 0; i < S; i++) {
            const int j = col - i;
            if (j >= 0 && j < S) mac96(A[i], B[j], c0, c1, c2);
        }
        O[col] = c0;
        c0 = c1;
        c1 = c2;
        c2 = 0;
    }
    O[2 * S - 1] = c0;
    const size_t node = out_index ? (size_t)out_index[k] : k;
    uint4 *o4 = reinterpret_cast<uint4 *>(out + 2 * node * S);
#pragma unroll
    for (int i = 0; i < S / 2; i++)
        o4[i] = make_uint4(O[4 * i], O[4 * i + 1], O[4 * i + 2], O[4 * i + 3]);
}

// ------------------------------------------------ one product per warp

constexpr int kWarpsPerBlock = 8;

// Lane l owns output columns [l W, l W + W), W = 2S/32 >= 2, and the lanes
// step through i = 0 .. S-1 together: column col gains A[i] B[col - i], B read
// as zero outside [0, S).  At step i lane l needs B[l W - i + w], w < W: a
// window that slides down by one word per step, so a step is one broadcast
// read of A[i], one new word of B and W multiply-adds.  The zero-padded copy
// of B (word j at j' = j + S, j' < 3S) is stored skewed, j' at j' + j' / W, so
// that the lanes' reads, W words apart, fall in distinct banks (W + 1 is odd).
//
// The column sums form a number N_l = low_l + high_l 2^(32W) per lane with
// high_l < 2^41; the product is sum_l (low_l + high_{l-1}) 2^(32 W l).  Each
// lane's addition low_l + high_{l-1} carries at most one bit out, and the
// one-bit carries are resolved by a generate/propagate scan across the warp.
template <int S>
__global__ void __launch_bounds__(32 * kWarpsPerBlock) comba_warp(const uint32_t *in,
                                                                  size_t nprod, uint32_t *out,
                                                                  const uint32_t *out_index)
{
    chain_wait();
    constexpr int W = 2 * S / 32;
    static_assert(W >= 2, "warp Comba needs at least two columns per lane");
    constexpr int PADN = 3 * S;              // padded indices j' in [0, 3S)
    constexpr int BWORDS = PADN + PADN / W;  // skewed layout
    __shared__ uint32_t smA[kWarpsPerBlock][S];
    __shared__ uint32_t smB[kWarpsPerBlock][BWORDS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const size_t k = (size_t)blockIdx.x * kWarpsPerBlock + wid;
    if (k >= nprod) return;
    const uint32_t *src = in + 2 * k * S;
    uint32_t *A = smA[wid], *Bs = smB[wid];
    for (int i = lane; i < S; i += 32) A[i] = src[i];
    for (int jp = lane; jp < PADN; jp += 32) {
        const int j = jp - S;
        Bs[jp + jp / W] = (j >= 0 && j < S) ? src[S + j] : 0u;
    }
    __syncwarp();
    uint32_t c0[W], c1[W], c2[W], b[W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        c0[w] = c1[w] = c2[w] = 0;
        const int jp = lane * W + w + S;
        b[w] = Bs[jp + jp / W];
    }
#pragma unroll
    for (int i = 0; i < S; i++) {
        const uint32_t a = A[i];
#pragma unroll
        for (int w = 0; w < W; w++) mac96(a, b[w], c0[w], c1[w], c2[w]);
        if (i + 1 < S) {
#pragma unroll
            for (int w = W - 1; w > 0; w--) b[w] = b[w - 1];
            // j' = l W + (S - i - 1) with S - i - 1 >= 0: j' / W = l + (S - i - 1) / W
            b[0] = Bs[lane * (W + 1) + (S - i - 1) + (S - i - 1) / W];
        }
    }
    uint32_t limb[W];
    // carry the running 96-bit sum through the lane's columns
    uint32_t r0 = 0, r1 = 0, r2 = 0;
#pragma unroll
    for (int w = 0; w < W; w++) {
        asm("add.cc.u32 %0, %0, %3;\n\t"
            "addc.cc.u32 %1, %1, %4;\n\t"
            "addc.u32 %2, %2, %5;\n\t"
            : "+r"(r0), "+r"(r1), "+r"(r2)
            : "r"(c0[w]), "r"(c1[w]), "r"(c2[w]));
        limb[w] = r0;
        r0 = r1;
        r1 = r2;
        r2 = 0;
    }
    const uint64_t high = ((uint64_t)r1 << 32) | r0;
    uint64_t hprev = __shfl_up_sync(0xffffffffu, high, 1);
    if (lane == 0) hprev = 0;
    // low + hprev
    uint64_t t = (uint64_t)limb[0] + (uint32_t)hprev;
    limb[0] = (uint32_t)t;
    t = (t >> 32) + limb[1] + (uint32_t)(hprev >> 32);
    limb[1] = (uint32_t)t;
    uint32_t cy = (uint32_t)(t >> 32);
#pragma unroll
    for (int w = 2; w < W; w++) {
        t = (uint64_t)limb[w] + cy;
        limb[w] = (uint32_t)t;
        cy = (uint32_t)(t >> 32);
    }
    bool ones = true;
#pragma unroll
    for (int w = 0; w < W; w++) ones = ones && limb[w] == 0xffffffffu;
    // generate/propagate scan: (g, p) o (g', p') = (g | (p & g'), p & p')
    uint32_t g = cy, p = ones ? 1u : 0u;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t go = __shfl_up_sync(0xffffffffu, g, off);
        const uint32_t po = __shfl_up_sync(0xffffffffu, p, off);
        if (lane >= off) {
            g = g | (p & go);
            p = p & po;
        }
    }
    uint32_t cin = __shfl_up_sync(0xffffffffu, g, 1);
    if (lane == 0) cin = 0;
#pragma unroll
    for (int w = 0; w < W; w++) {
        t = (uint64_t)limb[w] + cin;
        limb[w] = (uint32_t)t;
        cin = (uint32_t)(t >> 32);
    }
    const size_t node = out_index ? (size_t)out_index[k] : k;
    uint32_t *o = out + 2 * node * S + lane * W;
#pragma unroll
    for (int w = 0; w < W; w++) o[w] = limb[w];
}

// ------------------------------------- one product per thread, row by row

// The lowest P + 1 words of a running sum V as two rows of aligned 64-bit
// pieces, V = sum_j e[j] 2^(32 j) + sum_j o[j] 2^(32 (j + 1)).  row() returns
// V's lowest word after V <- floor(V / 2^32) + a B, the caller passing the old
// o as e and the old e as o: the pieces of a row's products with B's even
// words fall on e, those with its odd words on o one place further down, so
// that the shift is the choice of the destination.  Each piece is one wide
// multiply-add with carry in and out; V < 2^(32 (P + 1)) always, so the
// carries end in o's top word.
template <int P>
__device__ __forceinline__ uint32_t comba_row(uint32_t (&e)[P], uint32_t (&o)[P], uint32_t a,
                                              const uint32_t (&b)[P])
{
    asm volatile("add.cc.u32 %0, %0, %1;" : "+r"(e[0]) : "r"(o[1]));
#pragma unroll
    for (int k = 0; k + 2 < P; k += 2)
        asm volatile("madc.lo.cc.u32 %0, %2, %3, %4;\n\t"
                     "madc.hi.cc.u32 %1, %2, %3, %5;"
                     : "=r"(o[k]), "=r"(o[k + 1])
                     : "r"(a), "r"(b[k + 1]), "r"(o[k + 2]), "r"(o[k + 3]));
    asm volatile("madc.lo.cc.u32 %0, %2, %3, 0;\n\t"
                 "madc.hi.u32 %1, %2, %3, 0;"
                 : "=r"(o[P - 2]), "=r"(o[P - 1]) : "r"(a), "r"(b[P - 1]));
    asm volatile("mad.lo.cc.u32 %0, %2, %3, %0;\n\t"
                 "madc.hi.cc.u32 %1, %2, %3, %1;"
                 : "+r"(e[0]), "+r"(e[1]) : "r"(a), "r"(b[0]));
#pragma unroll
    for (int k = 2; k < P; k += 2)
        asm volatile("madc.lo.cc.u32 %0, %2, %3, %0;\n\t"
                     "madc.hi.cc.u32 %1, %2, %3, %1;"
                     : "+r"(e[k]), "+r"(e[k + 1]) : "r"(a), "r"(b[k]));
    asm volatile("addc.u32 %0, %0, 0;" : "+r"(o[P - 1]));
    return e[0];
}

// A product's operands a, b (S words each) in shared memory, a at 0 and b at
// kB; products are kStride (odd) words apart, so that a warp's accesses to the
// same word of each fall in distinct banks (with two threads per product the
// gap puts the second thread's words half the banks away).
template <int S, int T>
struct CombaRows {
    static constexpr int kPer = 32 / T;  // products per warp
    static constexpr int kB = S + (T == 2 ? 16 : 0);
    static constexpr int kStride = kB + S + 1;
    static constexpr size_t kBytes = 4 * (size_t)kPer * kStride;
};

// T threads per product, thread t with words [t P, t P + P) of b (P = S / T)
// in registers, all of a's words in turn from shared memory.  Each row emits
// one word; the words of thread 0 take the place of a's, those of thread 1 of
// b's, and the two threads' numbers are added at the end.
//
// Bound by the multiply pipe, whose heavy half (the wide products) is 90 % busy
// at S = 64, 80 % at 32 and 72 % at 16 (counted), where a warp per product
// spends half of its multiply-adds on B's zero padding and four instructions
// on each.  A level of 2^25 limbs, before -> after: slots of 16 69 -> 54 us
// (a thread per product reading its 128 bytes alone), 32 220 -> 81 us, 64
// 292 -> 186 us.
template <int S, int T>
__global__ void __launch_bounds__(32) comba_rows(const uint32_t *in, size_t nprod, uint32_t *out,
                                                 const uint32_t *out_index)
{
    chain_wait();
    using R = CombaRows<S, T>;
    constexpr int P = S / T;
    static_assert((T == 1 || T == 2) && P % 4 == 0 && S % 8 == 0, "shape");
    extern __shared__ uint32_t comba_smem[];
    const int lane = threadIdx.x;
    const size_t k0 = (size_t)blockIdx.x * R::kPer;
    const int np = nprod - k0 < (size_t)R::kPer ? (int)(nprod - k0) : R::kPer;
    {
        const uint32_t *src = in + 2 * k0 * S;
        const int words = 2 * S * np;
        for (int w = lane; w < words; w += 32) {
            const int q = w / (2 * S), i = w % (2 * S);
            const uint32_t to = (uint32_t)__cvta_generic_to_shared(
                comba_smem + q * R::kStride + i + (i >= S ? R::kB - S : 0));
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(src + w));
        }
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    // products past the last one work on whatever is in their words
    const int t = T == 1 ? 0 : lane / R::kPer;
    uint32_t *A = comba_smem + (lane % R::kPer) * R::kStride, *B = A + R::kB;
    uint32_t *em = t ? B : A;
    uint32_t b[P], e[P], o[P];
#pragma unroll
    for (int j = 0; j < P; j++) {
        b[j] = B[t * P + j];
        e[j] = o[j] = 0;
    }
    if (T > 1) __syncwarp();
    uint32_t a0 = A[0], a1 = A[1];
#pragma unroll 1
    for (int i = 0; i < S; i += 2) {
        // the next two words of a (those past the last are b's or the gap's, unused)
        const uint32_t n0 = A[i + 2], n1 = A[i + 3];
        if (T > 1) __syncwarp();
        em[i] = comba_row<P>(e, o, a0, b);
        em[i + 1] = comba_row<P>(o, e, a1, b);
        a0 = n0;
        a1 = n1;
    }
    // V / 2^32 = words e[1 .. P) and o[0 .. P), the roles as after an even row:
    // o is the row that held the last emitted word
    uint32_t top[P];
    {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < P; j++) {
            const uint64_t v = (uint64_t)(j + 1 < P ? o[j + 1] : 0u) + e[j] + c;
            top[j] = (uint32_t)v;
            c = (uint32_t)(v >> 32);
        }
    }
    if (T == 1) {
#pragma unroll
        for (int j = 0; j < P; j++) B[j] = top[j];
    } else {
        __syncwarp();
        uint32_t c = 0;
        if (t == 0) {
            // words [P, S) += the other thread's first, then its next P meet top
#pragma unroll 4
            for (int j = 0; j < P; j++) {
                const uint64_t v = (uint64_t)A[P + j] + B[j] + c;
                A[P + j] = (uint32_t)v;
                c = (uint32_t)(v >> 32);
            }
#pragma unroll
            for (int j = 0; j < P; j++) {
                const uint64_t v = (uint64_t)top[j] + B[P + j] + c;
                B[j] = (uint32_t)v;
                c = (uint32_t)(v >> 32);
            }
        }
        c = __shfl_sync(0xffffffffu, c, lane % R::kPer);
        if (t == 1) {
#pragma unroll
            for (int j = 0; j < P; j++) {
                const uint64_t v = (uint64_t)top[j] + c;
                B[P + j] = (uint32_t)v;
                c = (uint32_t)(v >> 32);
            }
        }
    }
    __syncwarp();
    for (int q = 0; q < np; q++) {
        const size_t node = out_index ? (size_t)out_index[k0 + q] : k0 + q;
        uint32_t *dst = out + 2 * node * S;
        const uint32_t *from = comba_smem + q * R::kStride;
#pragma unroll
        for (int i = lane; i < 2 * S; i += 32) dst[i] = from[i + (i >= S ? R::kB - S : 0)];
    }
}

template <int S, int T>
void launch_rows(const uint32_t *in, size_t nprod, uint32_t *out, cudaStream_t s,
                 const uint32_t *out_index)
{
    using R = CombaRows<S, T>;
    static_assert(R::kBytes <= 48 * 1024, "no opt-in needed");
    launch_chained(comba_rows<S, T>, (unsigned)((nprod + R::kPer - 1) / R::kPer), 32, R::kBytes, s,
                   in, nprod, out, out_index);
}

// ------------------------------------------------------------ utilities

// Largest i + 1 with x[i] != 0, reduced into *top (0 if all zero).
__global__ void find_top(const uint32_t *x, size_t n, unsigned long long *top)
{
    chain_wait();
    unsigned long long best = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        if (x[i]) best = i + 1;
    for (int off = 16; off; off >>= 1) {
        const unsigned long long o = __shfl_down_sync(0xffffffffu, best, off);
        best = o > best ? o : best;
    }
    if ((threadIdx.x & 31) == 0 && best) atomicMax(top, best);
}

struct TopsArgs {
    const uint32_t *x[kMaxTops];
    uint64_t n[kMaxTops];
    uint64_t scan;
    uint64_t *out;  // per number: normalised length, top two limbs
};

// One block per number, scanning down from the top for the highest nonzero
// limb, `scan` limbs of it at most.  A number whose scanned limbs are all zero
// is left at the length below them, its top limbs 0.
__global__ void __launch_bounds__(1024) number_tops(const __grid_constant__ TopsArgs a)
{
    chain_wait();
    __shared__ unsigned long long best;
    const uint32_t *x = a.x[blockIdx.x];
    const uint64_t len = a.n[blockIdx.x], low = len > a.scan ? len - a.scan : 0;
    const uint64_t n = block_top(x, low, len, &best);
    if (threadIdx.x == 0) {
        a.out[2 * blockIdx.x] = n;
        a.out[2 * blockIdx.x + 1] =
            n > low ? (uint64_t)x[n - 1] << 32 | (n > 1 ? x[n - 2] : 0u) : 0u;
    }
}

// ----------------------------------------------------------- host side

void leaf_level(Ctx &c, const uint32_t *values, size_t count, const Repeats &rep, uint32_t *out,
                size_t nodes, int lpn, cudaStream_t s)
{
    const int tok = prof_begin(c, "leaf_products", s);
    launch_chained(leaf_products, (unsigned)((nodes + 255) / 256), 256, 0, s, values, count, rep,
                   out, nodes, lpn);
    CAT_LAUNCH("leaf_products");
    prof_end(c, tok, s, 4.0 * (double)count + 32.0 * (double)nodes,
             4.0 * (double)count + 32.0 * (double)nodes);
}

// Products of adjacent slot-limb nodes into 2*slot-limb slots, for slots
// handled by schoolbook multiplication.  Returns false if slot is too large.
bool comba_level(Ctx &c, const uint32_t *in, size_t slot, size_t nprod, uint32_t *out,
                 cudaStream_t s, const uint32_t *out_index)
{
    if (nprod == 0) return true;
    if (slot > 256) return false;
    // Rows from two products per lane and SM on: below that a warp per product
    // spreads the few products over more of the chip (8,189 products of 32 and
    // 64 limbs: 5.2 and 11.3 us by warps, 6.0 and 11.8 us by rows; 16,381: 8.2
    // and 20.7 us, 6.2 and 16.6 us).  A row's latency keeps one thread per
    // product ahead at 32 limbs (2^19 products: 81 us, two threads 104 us) and
    // two at 64, whose registers else leave nine warps per SM (2^18: 207 and
    // 186 us).  Products of 16 limbs go by rows at any count.
    const bool rows = slot == 16 || (slot <= 64 && nprod >= 64 * (size_t)c.num_sms);
    const char *name = slot == 8 ? "comba_thread" : rows ? "comba_rows" : "comba_warp";
    const int tok = prof_begin(c, name, s);
    const unsigned tb = 256;
    const unsigned gt = (unsigned)((nprod + tb - 1) / tb);
    const unsigned gw = (unsigned)((nprod + kWarpsPerBlock - 1) / kWarpsPerBlock);
    switch (slot) {
    case 8: launch_chained(comba_thread<8>, gt, tb, 0, s, in, nprod, out, out_index); break;
    case 16: launch_rows<16, 1>(in, nprod, out, s, out_index); break;
    case 32:
        if (rows) launch_rows<32, 1>(in, nprod, out, s, out_index);
        else launch_chained(comba_warp<32>, gw, 32 * kWarpsPerBlock, 0, s, in, nprod, out,
                            out_index);
        break;
    case 64:
        if (rows) launch_rows<64, 2>(in, nprod, out, s, out_index);
        else launch_chained(comba_warp<64>, gw, 32 * kWarpsPerBlock, 0, s, in, nprod, out,
                            out_index);
        break;
    case 128: launch_chained(comba_warp<128>, gw, 32 * kWarpsPerBlock, 0, s, in, nprod, out,
                             out_index); break;
    case 256: launch_chained(comba_warp<256>, gw, 32 * kWarpsPerBlock, 0, s, in, nprod, out,
                             out_index); break;
    default: return false;
    }
    CAT_LAUNCH("comba_level");
    prof_end(c, tok, s, 16.0 * (double)slot * (double)nprod, 16.0 * (double)slot * (double)nprod);
    return true;
}

void normalize_all(Ctx &c, Big *const *x, int count, cudaStream_t s, uint64_t scan)
{
    if (count > kMaxTops) fail(CAT_EINVAL, "too many numbers");
    if (count == 0) return;
    DevBuf<uint64_t> d(c, 2 * (size_t)count, s);
    TopsArgs a{};
    for (int i = 0; i < count; i++) {
        a.x[i] = x[i]->buf.get();
        a.n[i] = x[i]->n;
    }
    a.scan = scan;
    a.out = d.get();
    launch_chained(number_tops, count, 1024, 0, s, a);
    CAT_LAUNCH("number_tops");
    uint32_t h[4 * kMaxTops];
    memcpy(h, read_back(c, d.get(), 4 * count, s), 16 * (size_t)count);
    for (int i = 0; i < count; i++) {
        uint64_t n = (uint64_t)h[4 * i + 1] << 32 | h[4 * i];
        uint64_t top = (uint64_t)h[4 * i + 3] << 32 | h[4 * i + 2];
        if (n && !top) {  // zeros as far as the block scanned
            n = normalized_length(c, a.x[i], n, s);
            if (n) {
                const int k = n > 1 ? 2 : 1;
                const uint32_t *t = read_back(c, a.x[i] + n - k, k, s);
                top = (uint64_t)t[k - 1] << 32 | (k > 1 ? t[0] : 0u);
            }
        }
        x[i]->n = n;
        x[i]->bits = top_bits(n, top);
    }
}

size_t normalized_length(Ctx &c, const uint32_t *x, size_t n, cudaStream_t s)
{
    if (n == 0) return 0;
    DevBuf<unsigned long long> scratch;
    unsigned long long *top = c.dev_word;
    if (!top) {
        scratch = DevBuf<unsigned long long>(c, 1, s);
        top = scratch.get();
    }
    CAT_CUDA(cudaMemsetAsync(top, 0, sizeof(unsigned long long), s));
    const size_t threads = 256;
    size_t blocks = (n + threads - 1) / threads;
    const size_t cap = (size_t)c.num_sms * 8;
    if (blocks > cap) blocks = cap;
    launch_chained(find_top, (unsigned)blocks, threads, 0, s, x, n, top);
    CAT_LAUNCH("find_top");
    const uint32_t *h = read_back(c, top, 2, s);
    return (size_t)((uint64_t)h[1] << 32 | h[0]);
}

}  // namespace cat
