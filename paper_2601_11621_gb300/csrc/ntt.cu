// ntt.cu -- exact big-integer multiplication by a five-prime number-theoretic
// transform (NTT), Chinese remaindering and carry propagation.
//
// This is the multiplication the reconstruction phase spends its time in
// (Sec. 3.2; Sec. 6 reports that the big products dominate the run time, and
// Sec. 6.3 assumes an FFT-based multiplication for large operands).  The
// method is the classical one: pairs of limbs of a and b are the 64-bit
// coefficients of two polynomials; their cyclic convolution of length
// 2^np >= (na + nb) / 2 is computed modulo five primes q_i (forward
// transforms, pointwise product, inverse transform), the exact coefficients
// are recovered by Chinese remaindering, and their 160-bit values are summed
// into 32-bit limbs with carry propagation.  A product of 2^n limbs takes
// transforms of 2^np points, np = n - 1.
//
// Transform layout.  The forward transform is an in-place decimation-in-
// frequency transform (natural order in, bit-reversed order out); the inverse
// is the matching decimation-in-time transform (bit-reversed in, natural out),
// so no permutation pass is needed.  A length-2^np transform is split into
// passes that each run 2^r-point sub-transforms in shared memory (the
// "four-step" factorisation L = L1 * L2 applied recursively): column passes
// over strided sub-arrays, each followed by the twiddle w_M^(col * k1), and a
// final row pass over contiguous runs of 2^r points.  The last forward row
// pass, the pointwise product and the first inverse row pass are fused.
// Transforms of up to 2^11 points run entirely inside one thread block,
// including the remaindering and carries; transforms of 2^12 points run in a
// row pass alone, straight from the operands' limbs.
#include "cat_internal.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

namespace cat {

// --------------------------------------------------------------- constants

#define CAT_SET_ROW(f, s) \
    {f(ntt_prime(s, 0)), f(ntt_prime(s, 1)), f(ntt_prime(s, 2)), f(ntt_prime(s, 3)), \
     f(ntt_prime(s, 4))}
#define CAT_SET_CONST(f) {CAT_SET_ROW(f, 0), CAT_SET_ROW(f, 1), CAT_SET_ROW(f, 2)}
#define CAT_Q(q) (q)
__constant__ uint32_t c_q[kNumSets][kNumPrimes] = CAT_SET_CONST(CAT_Q);
__constant__ uint32_t c_qinv[kNumSets][kNumPrimes] = CAT_SET_CONST(inv32);

#undef CAT_SET_ROW
#undef CAT_SET_CONST
#undef CAT_Q

// Entries [0, 16) of every stage table (the twiddles of stage bits below 4,
// [set][prime][direction][index] in the stage table's own layout and
// multiplier form), for the register rounds with B = 0, whose twiddle indices
// are compile-time constants: served from constant memory they are uniform
// operands instead of registers held across the round.
__constant__ uint2 c_tw_low[kNumSets][kNumPrimes][2][16];

void upload_low_twiddles(const uint2 *tables)
{
    uint2 h[kNumSets][kNumPrimes][2][16];
    for (int set = 0; set < kNumSets; set++)
        for (int p = 0; p < kNumPrimes; p++)
            for (int d = 0; d < 2; d++)
                for (int j = 0; j < 16; j++)
                    h[set][p][d][j] =
                        tables[(((size_t)set * kNumPrimes + p) * 2 + d) * kTwPerDir + j];
    CAT_CUDA(cudaMemcpyToSymbol(c_tw_low, h, sizeof(h)));
}

// Chinese remaindering constants of a set.  With M the product of its primes
// and y_i = c (M/q_i)^-1 mod q_i, the coefficient is c = sum_i y_i (M/q_i) -
// k M with k = floor(sum_i y_i / q_i).  The factor (M/q_i)^-1 rides on the
// pointwise product's scale, so the inverse transform delivers y_i itself.
struct Words {
    uint32_t w[6];
};

// M, or M / q_skip, in base 2^32 (dec: base 10^9), least significant first
constexpr Words crt_product(int set, int skip, bool dec)
{
    Words r{};
    r.w[0] = 1;
    const uint64_t base = dec ? (uint64_t)kDecBase : (1ull << 32);
    for (int i = 0; i < kNumPrimes; i++) {
        if (i == skip) continue;
        uint64_t carry = 0;
        for (int j = 0; j < 6; j++) {
            const uint64_t v = (uint64_t)r.w[j] * ntt_prime(set, i) + carry;
            r.w[j] = (uint32_t)(v % base);
            carry = v / base;
        }
    }
    return r;
}

// word j of 2^160 - M
constexpr uint32_t crt_neg_m(int set, int j)
{
    const Words m = crt_product(set, -1, false);
    uint32_t borrow = 0, r = 0;
    for (int i = 0; i <= j; i++) {
        const uint64_t v = (uint64_t)m.w[i] + borrow;
        r = (uint32_t)(0u - (uint32_t)v);
        borrow = v != 0 ? 1u : 0u;
    }
    return r;
}

// (M/q_i)^-1 mod q_i
constexpr uint32_t crt_inverse(int set, int i)
{
    const uint32_t q = ntt_prime(set, i);
    uint64_t x = 1;
    for (int j = 0; j < kNumPrimes; j++)
        if (j != i) x = x * (ntt_prime(set, j) % q) % q;
    return powmod_u32(x, q - 2, q);
}

// Pointwise scale S = 2^-np (M/q_i)^-1 mod q_i, folded into the product's
// second factor: 2^32 S in Shoup's form for sets 0 and 1, 2^64 S (Montgomery)
// for set 2, so that pmul(x, y) = x y S.
struct Scale {
    uint2 c[kNumPrimes];
};

static uint32_t scale_value(int set, int i, int np)
{
    const uint32_t q = ntt_prime(set, i);
    const uint32_t inv2n = powmod_u32((q + 1) / 2, (uint64_t)np, q);  // 2^-np
    return to_mont_c(mulmod_u64(inv2n, crt_inverse(set, i), q), q);    // 2^32 S
}

static Scale make_scale(int set, int np)
{
    Scale s;
    for (int i = 0; i < kNumPrimes; i++) {
        const uint32_t q = ntt_prime(set, i);
        const uint32_t r = scale_value(set, i, np);
        s.c[i] = set_shoup(set) ? make_uint2(r, shoup_c(r, q)) : make_uint2(to_mont_c(r, q), 0u);
    }
    return s;
}

// The operands' input multipliers (coef_in): 1 and the word base (2^32, or
// 10^9 for decimal digits), both times the pointwise scale 2^32 S of 2^np
// points for the operand that takes it in advance (np >= 0).
struct CoefMuls {
    CoefMul c[kNumPrimes];
};

static CoefMuls make_coef(int set, bool dec, int np = -1)
{
    auto form = [&](uint32_t w, uint32_t q) {
        if (set_shoup(set)) return make_uint2(w, shoup_c(w, q));
        const uint32_t m = to_mont_c(w, q);
        return make_uint2(m, m * inv32(q));
    };
    CoefMuls m;
    for (int i = 0; i < kNumPrimes; i++) {
        const uint32_t q = ntt_prime(set, i);
        const uint32_t b = (uint32_t)((dec ? (uint64_t)kDecBase : (1ull << 32)) % q);
        const uint32_t r = np < 0 ? 1u : scale_value(set, i, np);
        m.c[i].w0 = form(r, q);
        m.c[i].w1 = form(mulmod_u64(r, b, q), q);
    }
    return m;
}

// -------------------------------------------------------------- twiddles

__device__ __forceinline__ const uint2 *tw_table(const uint2 *tw, int set, int p, int dir)
{
    return tw + (((size_t)set * kNumPrimes + p) * 2 + dir) * kTwPerDir;
}

// w^E 2^32 mod q (the Montgomery form of w^E, below q) from the three small
// tables.  In Shoup-form sets the third table holds w^(2^18 j) 2^32, so two
// Shoup products give the Montgomery form directly; in set 2 all entries are
// Montgomery forms and Montgomery products keep that form.
template <int PS>
__device__ __forceinline__ uint32_t tw_pow_mont(const uint2 *T, uint32_t E, uint32_t q,
                                                uint32_t qinv)
{
    const uint2 a = __ldg(&T[kTwStage + (E & (kTwSmall - 1))]);
    const uint2 b = __ldg(&T[kTwStage + kTwSmall + ((E >> 9) & (kTwSmall - 1))]);
    const uint2 c = __ldg(&T[kTwStage + 2 * kTwSmall + (E >> 18)]);
    if constexpr (PS == 2) {
        return mont_mul_pre(mont_mul_pre(a.x, b.x, b.y, q), c.x, c.y, q);
    } else {
        return csub(shoup(shoup(a.x, b.x, b.y, q), c.x, c.y, q), q);
    }
}

// x v for any 32-bit x and a Montgomery-form multiplier vm = v 2^32 mod q,
// into the set's forward range (x vm < 2^32 q).
template <int PS>
__device__ __forceinline__ uint32_t mul_mont(uint32_t x, uint32_t vm, uint32_t q, uint32_t qinv)
{
    if constexpr (PS == 0) {
        return mont2(x, vm, q, qinv);
    } else if constexpr (PS == 1) {
        return csub(mont2(x, vm, q, qinv), q);
    } else {
        return mont_mul(x, vm, q, qinv);
    }
}

// Product of two Montgomery-form multipliers, reduced below q, with the
// second one's companion up = um q^-1 mod 2^32 precomputed (three multiplies:
// the low word of vm um times q^-1 is vm up).
template <int PS>
__device__ __forceinline__ uint32_t mont_step(uint32_t vm, uint32_t um, uint32_t up, uint32_t q)
{
    if constexpr (PS == 2) return mont_mul_pre(vm, um, up, q);
    const uint32_t hi = __umulhi(vm, um);
    const uint32_t m = vm * up;
    return csub(hi - __umulhi(m, q) + q, q);
}

// ----------------------------------------------- remaindering and carries

// acc += r (M/q_I) over five words, as two chains of 64-bit products: e at
// words 0, 2 and 4, o at words 1 and 3, so that no product waits for the
// carry of its neighbour word.
struct Acc160 {
    uint32_t e0, e1, e2, e3, e4, o0, o1, o2, o3;
};

template <int PS, int I>
__device__ __forceinline__ void crt_acc(uint32_t r, Acc160 &a)
{
    constexpr Words m = crt_product(PS, I, false);
    constexpr uint32_t m0 = m.w[0], m1 = m.w[1], m2 = m.w[2], m3 = m.w[3];
    static_assert(m.w[4] == 0, "M/q_i fits four words");
    asm("mad.lo.cc.u32 %0, %5, %6, %0;\n\t"
        "madc.hi.cc.u32 %1, %5, %6, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %7, %2;\n\t"
        "madc.hi.cc.u32 %3, %5, %7, %3;\n\t"
        "addc.u32 %4, %4, 0;\n\t"
        : "+r"(a.e0), "+r"(a.e1), "+r"(a.e2), "+r"(a.e3), "+r"(a.e4)
        : "r"(r), "r"(m0), "r"(m2));
    asm("mad.lo.cc.u32 %0, %4, %5, %0;\n\t"
        "madc.hi.cc.u32 %1, %4, %5, %1;\n\t"
        "madc.lo.cc.u32 %2, %4, %6, %2;\n\t"
        "madc.hi.u32 %3, %4, %6, %3;\n\t"
        : "+r"(a.o0), "+r"(a.o1), "+r"(a.o2), "+r"(a.o3)
        : "r"(r), "r"(m1), "r"(m3));
}

// The coefficient's five words from its residues y_i = r[i] mod q_i (any
// 32-bit representatives): c = sum_i r_i (M/q_i) - k M.  k = floor(sum_i
// r_i/q_i) comes from a fixed-point sum of r_i floor(2^57/q_i) / 2^32 in units
// of 2^-25, short of the true sum by at most 10 units (1 per floor of the
// quotient and of the product); c/M < 0.895 in every set, so the fraction
// never reaches the next integer with 16 units added.  The sum stays below
// 20 M < 2^160.  Against Garner's mixed radix this takes no modular products
// at all (20 + 5 word products instead of 10 Shoup products and 10).
template <int PS>
__device__ __forceinline__ void crt5(const uint32_t (&r)[kNumPrimes], uint32_t (&w)[5])
{
    constexpr uint32_t f0 = (uint32_t)((1ull << 57) / ntt_prime(PS, 0)),
                       f1 = (uint32_t)((1ull << 57) / ntt_prime(PS, 1)),
                       f2 = (uint32_t)((1ull << 57) / ntt_prime(PS, 2)),
                       f3 = (uint32_t)((1ull << 57) / ntt_prime(PS, 3)),
                       f4 = (uint32_t)((1ull << 57) / ntt_prime(PS, 4));
    const uint32_t k = (__umulhi(r[0], f0) + __umulhi(r[1], f1) + __umulhi(r[2], f2) +
                        __umulhi(r[3], f3) + __umulhi(r[4], f4) + 16u) >>
                       25;
    Acc160 a{0, 0, 0, 0, 0, 0, 0, 0, 0};
    crt_acc<PS, 0>(r[0], a);
    crt_acc<PS, 1>(r[1], a);
    crt_acc<PS, 2>(r[2], a);
    crt_acc<PS, 3>(r[3], a);
    crt_acc<PS, 4>(r[4], a);
    // - k M modulo 2^160
    constexpr uint32_t n0 = crt_neg_m(PS, 0), n1 = crt_neg_m(PS, 1), n2 = crt_neg_m(PS, 2),
                       n3 = crt_neg_m(PS, 3), n4 = crt_neg_m(PS, 4);
    asm("mad.lo.cc.u32 %0, %5, %6, %0;\n\t"
        "madc.hi.cc.u32 %1, %5, %6, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %7, %2;\n\t"
        "madc.hi.cc.u32 %3, %5, %7, %3;\n\t"
        "madc.lo.u32 %4, %5, %8, %4;\n\t"
        : "+r"(a.e0), "+r"(a.e1), "+r"(a.e2), "+r"(a.e3), "+r"(a.e4)
        : "r"(k), "r"(n0), "r"(n2), "r"(n4));
    asm("mad.lo.cc.u32 %0, %4, %5, %0;\n\t"
        "madc.hi.cc.u32 %1, %4, %5, %1;\n\t"
        "madc.lo.cc.u32 %2, %4, %6, %2;\n\t"
        "madc.hi.u32 %3, %4, %6, %3;\n\t"
        : "+r"(a.o0), "+r"(a.o1), "+r"(a.o2), "+r"(a.o3)
        : "r"(k), "r"(n1), "r"(n3));
    w[0] = a.e0;
    asm("add.cc.u32 %0, %4, %8;\n\t"
        "addc.cc.u32 %1, %5, %9;\n\t"
        "addc.cc.u32 %2, %6, %10;\n\t"
        "addc.u32 %3, %7, %11;\n\t"
        : "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4])
        : "r"(a.e1), "r"(a.e2), "r"(a.e3), "r"(a.e4), "r"(a.o0), "r"(a.o1), "r"(a.o2),
          "r"(a.o3));
}

// digit D of M/q_i summed over the primes: sum_i r_i (digit D of M/q_i)
template <int PS, int D>
__device__ __forceinline__ uint64_t crt_dec_column(const uint32_t (&r)[kNumPrimes])
{
    constexpr uint32_t d0 = crt_product(PS, 0, true).w[D], d1 = crt_product(PS, 1, true).w[D],
                       d2 = crt_product(PS, 2, true).w[D], d3 = crt_product(PS, 3, true).w[D],
                       d4 = crt_product(PS, 4, true).w[D];
    return (uint64_t)r[0] * d0 + (uint64_t)r[1] * d1 + (uint64_t)r[2] * d2 + (uint64_t)r[3] * d3 +
           (uint64_t)r[4] * d4;
}

// The coefficient's five base-10^9 digits (digit operands: c < 2^25 10^36 <
// 10^44), the same sum with M/q_i and M written in base 10^9, modulo 10^45.
// A column stays below 10^9 sum_i r_i < 2^64: residues below 2q in set 0
// (10^9 sum 2q = 9.6 10^18), below q otherwise (at most 1.15 10^19).
template <int PS>
__device__ __forceinline__ void crt5_dec(const uint32_t (&r_in)[kNumPrimes], uint32_t (&w)[5])
{
    uint32_t r[kNumPrimes];
#pragma unroll
    for (int i = 0; i < kNumPrimes; i++)
        r[i] = PS == 0 ? csub(r_in[i], 2 * ntt_prime(0, i)) : r_in[i];
    constexpr uint32_t f0 = (uint32_t)((1ull << 57) / ntt_prime(PS, 0)),
                       f1 = (uint32_t)((1ull << 57) / ntt_prime(PS, 1)),
                       f2 = (uint32_t)((1ull << 57) / ntt_prime(PS, 2)),
                       f3 = (uint32_t)((1ull << 57) / ntt_prime(PS, 3)),
                       f4 = (uint32_t)((1ull << 57) / ntt_prime(PS, 4));
    const uint64_t k = (__umulhi(r[0], f0) + __umulhi(r[1], f1) + __umulhi(r[2], f2) +
                        __umulhi(r[3], f3) + __umulhi(r[4], f4) + 16u) >>
                       25;  // at most 9
    constexpr uint32_t m0 = crt_product(PS, -1, true).w[0], m1 = crt_product(PS, -1, true).w[1],
                       m2 = crt_product(PS, -1, true).w[2], m3 = crt_product(PS, -1, true).w[3],
                       m4 = crt_product(PS, -1, true).w[4];
    // each column plus 16 10^9 (more than k times a digit of M and 16), whose
    // 16 the next column gives back
    constexpr uint64_t kBias = 16ull * kDecBase;
    uint64_t v = crt_dec_column<PS, 0>(r) + kBias - k * m0, q = v / kDecBase;
    w[0] = (uint32_t)(v - q * kDecBase);
    v = crt_dec_column<PS, 1>(r) + kBias - k * m1 + q - 16u;
    q = v / kDecBase;
    w[1] = (uint32_t)(v - q * kDecBase);
    v = crt_dec_column<PS, 2>(r) + kBias - k * m2 + q - 16u;
    q = v / kDecBase;
    w[2] = (uint32_t)(v - q * kDecBase);
    v = crt_dec_column<PS, 3>(r) + kBias - k * m3 + q - 16u;
    q = v / kDecBase;
    w[3] = (uint32_t)(v - q * kDecBase);
    v = crt_dec_column<PS, 4>(r) + kBias - k * m4 + q - 16u;
    w[4] = (uint32_t)(v % kDecBase);
}

// The carry map of a run in compact form.  A run takes its carry-in c in
// {0,1,2,3} into its lowest limb, and one more carry leaves it only if that
// limb overflows and every other limb is the largest digit; so its map is
// c -> b + [c >= t] with b the carry-out for c = 0 and t in {1,2,3} (or 4,
// never).  Compositions keep the form, (f o g)(c) = b_f + [b_g + [c >= t_g]
// >= t_f], with t = 0 for "always".  Packed as b << 4 | t; kUnitId (t = 15)
// is the identity, for threads without limbs.
constexpr uint32_t kUnitId = 15u;

__device__ __forceinline__ uint32_t unit_eval(uint32_t m, uint32_t c)
{
    return m == kUnitId ? c : (m >> 4) + (c >= (m & 15u) ? 1u : 0u);
}

// f o g
__device__ __forceinline__ uint32_t unit_compose(uint32_t f, uint32_t g)
{
    const uint32_t tf = f & 15u, bg = g >> 4, tg = g & 15u;
    const uint32_t t = bg >= tf ? 0u : (bg + 1u == tf ? tg : 4u);
    uint32_t r = (f & ~15u) | t;
    r = g == kUnitId ? f : r;
    return f == kUnitId ? g : r;
}

// Scan of compact run maps over the threads of the block, in thread order:
// returns the carry into thread t's run for a carry-in of 0 ahead of thread 0,
// and the composition of all the block's maps through *total.  wsm holds 32
// words.  Synchronises internally.
__device__ uint32_t block_carry_scan(uint32_t f, uint32_t *wsm, uint32_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    uint32_t inc = f;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc = unit_compose(inc, o);
    }
    __syncthreads();
    if (lane == 31) wsm[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = lane < nw ? wsm[lane] : kUnitId;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w = unit_compose(w, o);
        }
        wsm[lane] = w;
    }
    __syncthreads();
    const uint32_t cin_warp = wid > 0 ? unit_eval(wsm[wid - 1], 0u) : 0u;
    const uint32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
    *total = wsm[nw - 1];
    return lane > 0 ? unit_eval(ex, cin_warp) : cin_warp;
}

// The same for the runs of one tile, in a block of up to 16 warps that uses wsm
// for nothing else before: one barrier, every warp folding the maps of the
// warps before it; only thread 0 folds them all, when total is wanted.
__device__ __forceinline__ uint32_t tile_carry_scan(uint32_t f, uint32_t *wsm, uint32_t *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    uint32_t inc = f;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc = unit_compose(inc, o);
    }
    uint32_t c = 0;
    if (nw > 1) {
        if (lane == 31) wsm[wid] = inc;
        __syncthreads();
        for (int i = 0; i < wid; i++) c = unit_eval(wsm[i], c);
        if (total && threadIdx.x == 0) {
            uint32_t t = wsm[0];
            for (int i = 1; i < nw; i++) t = unit_compose(wsm[i], t);
            *total = t;
        }
    } else if (total) {
        *total = __shfl_sync(0xffffffffu, inc, 31);
    }
    const uint32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
    return lane > 0 ? unit_eval(ex, c) : c;
}

constexpr int kLimbsPerThread = 8;

constexpr int kCoefsPerThread = kLimbsPerThread / 2;

// The limbs of a thread's run of four consecutive coefficients j0 + i, words
// w[i][0..4] each.  Limb 2j sums words 0 of coefficient j, 2 of j - 1 and 4
// of j - 2, limb 2j + 1 words 1 of j and 3 of j - 1, so the run also needs
// words 2, 3 and 4 of coefficient j0 - 1 (h2, h3, h4b) and word 4 of j0 - 2
// (h4a).
struct CoefRun {
    uint32_t w[kCoefsPerThread][5];
    uint32_t h2, h3, h4a, h4b;
    __device__ __forceinline__ uint64_t operator()(int i) const
    {
        const int j = i >> 1;
        if (i & 1) return (uint64_t)w[j][1] + (j >= 1 ? w[j - 1][3] : h3);
        return (uint64_t)w[j][0] + (j >= 1 ? w[j - 1][2] : h2) +
               (j >= 2 ? w[j - 2][4] : (j == 0 ? h4a : h4b));
    }
};

// The halo words from the preceding thread: by shuffle inside a warp, through
// hsm (4 x 32 words) across warps; thread 0 keeps what its run holds (the
// block's predecessor).  Every thread of the block calls this.
__device__ __forceinline__ void run_halo(CoefRun &r, uint32_t *hsm)
{
    constexpr int C = kCoefsPerThread;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t a = __shfl_up_sync(0xffffffffu, r.w[C - 1][2], 1);
    const uint32_t b = __shfl_up_sync(0xffffffffu, r.w[C - 1][3], 1);
    const uint32_t c = __shfl_up_sync(0xffffffffu, r.w[C - 2][4], 1);
    const uint32_t d = __shfl_up_sync(0xffffffffu, r.w[C - 1][4], 1);
    if (lane == 31) {
        hsm[wid] = r.w[C - 1][2];
        hsm[32 + wid] = r.w[C - 1][3];
        hsm[64 + wid] = r.w[C - 2][4];
        hsm[96 + wid] = r.w[C - 1][4];
    }
    __syncthreads();
    if (lane) {
        r.h2 = a;
        r.h3 = b;
        r.h4a = c;
        r.h4b = d;
    } else if (wid) {
        r.h2 = hsm[wid - 1];
        r.h3 = hsm[32 + wid - 1];
        r.h4a = hsm[64 + wid - 1];
        r.h4b = hsm[96 + wid - 1];
    }
}

// Limb sums and carries for one tile of runs, one run of LPT limbs per thread
// (limb j0 + i, j0 = LPT * threadIdx.x, sums
// sum(i); limbs at or past tile_len are none), in base 2^32 or (DEC) 10^9,
// plus (ADD) the addend limbs add[j] for j < add_count.  In both bases a limb
// sums at most two full words, a coefficient's top word or digit (below 2^26
// or 10^8: coefficients stay below 2^153, or 10^44 for digit operands), the
// addend and a carry <= 3, so carries stay in {0, 1, 2, 3}.  Writes limbs j <
// min(tile_len, out_count) to out and returns the tile's carry map in compact
// form in thread 0's *tile_map (it fits a byte; null: not wanted).  The tile's
// own carry-in is assumed 0.  DEC / ADD: 1 or 0 when known at compile time, -1
// when the runtime flag (dec, add != null) decides.  LPT: limbs per run.
template <int DEC, int ADD, int LPT = kLimbsPerThread, class SUM>
__device__ __forceinline__ void tile_carry(SUM &&sum, int tile_len, uint32_t *out,
                                           long out_count, bool dec_rt, const uint32_t *add,
                                           long add_count, uint32_t *wsm, uint32_t *tile_map)
{
    static_assert(LPT % 4 == 0, "limbs are stored 16 bytes at a time");
    const bool dec = DEC < 0 ? dec_rt : DEC == 1;
    if (ADD == 0) add = nullptr;
    const int j0 = threadIdx.x * LPT;
    const uint32_t top = dec ? kDecBase - 1 : 0xffffffffu;  // largest limb
    uint32_t limb[LPT];
    uint32_t carry = 0;
    uint32_t f = kUnitId;
    if (j0 < tile_len) {
#pragma unroll
        for (int i = 0; i < LPT; i++) {
            const uint32_t ad = (add && j0 + i < add_count) ? add[j0 + i] : 0u;
            const uint64_t v = sum(i) + ad + carry;
            if (dec) {
                const uint32_t v32 = (uint32_t)v;  // < 3.1 10^9 + 3 < 2^32
                carry = (v32 >= kDecBase) + (v32 >= 2 * kDecBase) + (v32 >= 3 * kDecBase);
                limb[i] = v32 - carry * kDecBase;
            } else {
                limb[i] = (uint32_t)v;
                carry = (uint32_t)(v >> 32);
            }
        }
        bool ones = true;
#pragma unroll
        for (int i = 1; i < LPT; i++) ones = ones && limb[i] == top;
        // a carry-in c leaves the run iff ones and limb[0] + c > top
        const uint32_t t = (ones && limb[0] >= top - 2u) ? top + 1u - limb[0] : 4u;
        f = (carry << 4) | t;
    }
    const uint32_t cin = tile_carry_scan(f, wsm, tile_map);
    if (j0 < tile_len) {
        uint32_t c = cin;
#pragma unroll
        for (int i = 0; i < LPT; i++) {
            const uint64_t v = (uint64_t)limb[i] + c;
            c = dec ? (uint32_t)(v >= kDecBase) : (uint32_t)(v >> 32);
            limb[i] = dec ? (uint32_t)(v - (uint64_t)c * kDecBase) : (uint32_t)v;
        }
        if (j0 + LPT <= tile_len && j0 + LPT <= out_count &&
            (reinterpret_cast<uintptr_t>(out + j0) & 15) == 0) {
            uint4 *o4 = reinterpret_cast<uint4 *>(out + j0);
#pragma unroll
            for (int i = 0; i < LPT / 4; i++)
                o4[i] = make_uint4(limb[4 * i], limb[4 * i + 1], limb[4 * i + 2], limb[4 * i + 3]);
        } else {
#pragma unroll
            for (int i = 0; i < LPT; i++)
                if (j0 + i < tile_len && j0 + i < out_count) out[j0 + i] = limb[i];
        }
    }
}

constexpr int kTileThreads = 256;
constexpr int kTile = kTileThreads * kLimbsPerThread;  // 2048 limbs

constexpr int kTileCoefs = kTile / 2;

struct CrtArgs {
    const uint32_t *G;  // inverse-transformed residues [prime][product][2^np]
    size_t gpstride;
    int np;             // log2 points
    Sink sink;          // product k's limbs (out_len <= 2^(np+1))
    uint8_t *tile_maps; // [product][tiles], compact carry maps
    // when set, the products are summed, product k at coefficient k step
    // (a multiple of 4), and a product reaches into the next one's stretch only
    uint32_t step, nprod;
};

// The residues of N consecutive coefficients from j on (runs of 4 start at
// multiples of 4) of the sum of the products step coefficients apart: product
// k = j / step from its own coefficient r on, and the tail of product k - 1.
template <int PS, int N>
__device__ __forceinline__ void summed_residues(const CrtArgs &a, uint32_t j,
                                                uint32_t (&x)[N][kNumPrimes])
{
    const uint32_t k = j / a.step, r = j - k * a.step;
    const bool own = k < a.nprod, tail = k >= 1 && k <= a.nprod && a.step + r < (1u << a.np);
    const uint32_t *go = a.G + ((size_t)k << a.np) + r;
    const uint32_t *gt = a.G + ((size_t)(k - 1) << a.np) + a.step + r;
#pragma unroll
    for (int p = 0; p < kNumPrimes; p++) {
        uint32_t u[N] = {}, v[N] = {};
        if constexpr (N == 4) {
            if (own) {
                const uint4 w = *reinterpret_cast<const uint4 *>(go + p * a.gpstride);
                u[0] = w.x; u[1] = w.y; u[2] = w.z; u[3] = w.w;
            }
            if (tail) {
                const uint4 w = *reinterpret_cast<const uint4 *>(gt + p * a.gpstride);
                v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
            }
        } else {
            if (own) u[0] = go[p * a.gpstride];
            if (tail) v[0] = gt[p * a.gpstride];
        }
        const uint32_t q = c_q[PS][p];
#pragma unroll
        for (int i = 0; i < N; i++) {
            // below 2^32: set 0's residues lie in [0, 4q), the others' in
            // [0, q), q < 2^30, 2^31 and 2^32
            if constexpr (PS == 0) {
                x[i][p] = min(u[i], u[i] - 2 * q) + min(v[i], v[i] - 2 * q);
            } else if constexpr (PS == 1) {
                x[i][p] = u[i] + v[i];
            } else {
                const uint32_t t = q - v[i];
                x[i][p] = u[i] >= t ? u[i] - t : u[i] + v[i];
            }
        }
    }
}

template <int PS, bool DEC>
__device__ __forceinline__ void coef_words(const uint32_t (&r)[kNumPrimes], uint32_t (&w)[5])
{
    if constexpr (DEC) crt5_dec<PS>(r, w);
    else crt5<PS>(r, w);
}

// Five blocks per SM (48 registers): the kernel waits on its loads and
// barriers, not on a pipe (6.21 -> 5.95 ms per C(2,050,572,903) with the one
// barrier fewer of tile_carry_scan; 6.53 at four blocks).
// One tile of 1,024 coefficients (2,048 limbs) per block: each thread
// remainders its run of four (one 16-byte load per prime: tiles, runs and the
// prime arrays are multiples of 4 words apart) and sums them into limbs.
//
// SUM: one product from the products of a long operand's chunks.  The chunks'
// coefficients meet as residues, so that every coefficient is remaindered and
// carried once; before, the chunk products were written out as limbs and
// added by a pass of their own (a 2^23 x 2^21 limb product: 556 -> 505 us;
// 52,063 x 23,097 limbs, whose last chunk was a product by itself: 85 -> 56 us).
template <int PS, bool DEC, bool ADD, bool SUM>
__global__ void __launch_bounds__(kTileThreads, SUM ? 4 : 5) crt_carry_tiles(CrtArgs a)
{
    chain_wait();
    __shared__ uint32_t wsm[32];
    __shared__ uint32_t hsm[128];
    const size_t tiles = SUM ? (size_t)gridDim.x : ((size_t)1 << a.np) / kTileCoefs;
    const size_t k = blockIdx.x / tiles;
    const size_t t = blockIdx.x % tiles;
    const size_t jt = t * kTileCoefs;
    const size_t node = sink_node(a.sink, k);
    const uint32_t *g0 = a.G + (k << a.np) + jt;
    const int j0 = threadIdx.x * kCoefsPerThread;
    uint32_t r[kCoefsPerThread][kNumPrimes];
    if constexpr (SUM) {
        summed_residues<PS>(a, (uint32_t)jt + j0, r);
    } else {
#pragma unroll
        for (int p = 0; p < kNumPrimes; p++) {
            const uint4 x = *reinterpret_cast<const uint4 *>(g0 + p * a.gpstride + j0);
            r[0][p] = x.x; r[1][p] = x.y; r[2][p] = x.z; r[3][p] = x.w;
        }
    }
    // the tile's predecessor: coefficients jt - 2 and jt - 1 (none for tile 0),
    // by the first two threads side by side, loaded beside their runs so that
    // the latencies overlap
    const bool pred = threadIdx.x < 2 && t > 0;
    uint32_t pr[kNumPrimes] = {};
    if (pred) {
        if constexpr (SUM) {
            uint32_t x[1][kNumPrimes];
            summed_residues<PS>(a, (uint32_t)jt + threadIdx.x - 2, x);
#pragma unroll
            for (int p = 0; p < kNumPrimes; p++) pr[p] = x[0][p];
        } else {
#pragma unroll
            for (int p = 0; p < kNumPrimes; p++)
                pr[p] = g0[(long)(p * a.gpstride) + (int)threadIdx.x - 2];
        }
    }
    CoefRun run;
#pragma unroll
    for (int i = 0; i < kCoefsPerThread; i++) coef_words<PS, DEC>(r[i], run.w[i]);
    run.h2 = run.h3 = run.h4a = run.h4b = 0;
    if (threadIdx.x < 32 && t > 0) {
        uint32_t d[5] = {};
        if (pred) coef_words<PS, DEC>(pr, d);
        run.h4a = __shfl_sync(0xffffffffu, d[4], 0);
        run.h2 = __shfl_sync(0xffffffffu, d[2], 1);
        run.h3 = __shfl_sync(0xffffffffu, d[3], 1);
        run.h4b = __shfl_sync(0xffffffffu, d[4], 1);
    }
    run_halo(run, hsm);
    const Sink &o = a.sink;
    const size_t lt = t * kTile;  // first limb
    const long remaining = (long)o.out_len - (long)lt;
    const uint32_t *add = ADD ? o.add + k * o.add_tstride + lt : nullptr;
    uint32_t map;
    tile_carry<DEC ? 1 : 0, ADD ? 1 : 0>(run, kTile, o.out + node * o.out_tstride + lt, remaining,
                                         DEC, add, (long)o.add_len - (long)lt, wsm, &map);
    if (threadIdx.x == 0) a.tile_maps[blockIdx.x] = (uint8_t)map;
}

// The carries between the tiles of each product, from the tiles' compact
// maps: block b of a product folds the maps of the tiles before its own
// blockDim.x (each thread a stretch of b consecutive ones, then a block scan),
// scans its own tiles' maps from there, and every thread adds its tile's
// carry-in to the tile's first limbs (rarely more than one), in base 2^32 or
// (dec) 10^9.  One launch for any length: the refolded maps are at most 64 KB
// per block (64 blocks at 2^27 limbs) and stay in L2.  Before, one block per
// product scanned all its tiles and a second launch fixed them: 31 + 6 us at
// 2^26 limbs and 6 + 6 us for short products.
__global__ void __launch_bounds__(1024) carry_resolve(const uint8_t *maps, size_t tiles, int nb,
                                                      uint32_t *out, size_t out_tstride,
                                                      size_t out_len, bool dec,
                                                      const uint32_t *out_index)
{
    chain_wait();
    __shared__ uint32_t wsm[32];
    const size_t k = blockIdx.x / nb, b = blockIdx.x % nb;
    const uint8_t *m = maps + k * tiles;
    uint32_t c0 = 0, total;
    if (b) {
        const uint8_t *st = m + (size_t)threadIdx.x * b;
        uint32_t f = kUnitId;
        for (size_t i = 0; i < b; i++) f = unit_compose(st[i], f);
        block_carry_scan(f, wsm, &total);
        c0 = unit_eval(total, 0u);
        __syncthreads();
    }
    const size_t t = b * blockDim.x + threadIdx.x;
    uint32_t f = t < tiles ? m[t] : kUnitId;
    // the block's first tile takes c0: its map becomes the constant f(c0)
    if (threadIdx.x == 0) f = (unit_eval(f, c0) << 4) | 4u;
    uint32_t c = block_carry_scan(f, wsm, &total);
    if (threadIdx.x == 0) c = c0;
    if (!c || t >= tiles) return;
    uint32_t *o = out + (out_index ? (size_t)out_index[k] : k) * out_tstride;
    size_t j = t * kTile;
    const size_t end = std::min(j + kTile, out_len);
    for (; c && j < end; j++) {
        const uint64_t v = (uint64_t)o[j] + c;
        if (dec) {
            c = v >= kDecBase ? 1u : 0u;
            o[j] = (uint32_t)(v - (uint64_t)c * kDecBase);
        } else {
            o[j] = (uint32_t)v;
            c = (uint32_t)(v >> 32);
        }
    }
}

#include "ntt_kernels.cuh"

// ------------------------------------------ whole product in one block

struct FusedArgs {
    const uint32_t *A;
    size_t a_tstride;
    uint32_t a_len;
    const uint32_t *B;  // b_tstride 0: the same B for every product
    size_t b_tstride;
    uint32_t b_len;
    int a_al, b_al;     // every operand starts on an 8-byte boundary
    size_t nprod;
    Sink sink;
    const uint2 *tw;
    CoefMuls ca, cb;    // cb carries the pointwise scale
};

constexpr int kFusedMaxLog = 11;  // 2^11 points: products of 2^12 limbs

// Points of all products of a one-block multiply of 2^lr points (several
// short products share a block, at most one per thread) and its threads, one
// group of 16 points of both operands each.
__host__ __device__ constexpr int fused_points(int lr)
{
    return lr >= 9 ? 1 << lr : (lr >= 4 ? 512 : 32 << lr);
}
__host__ __device__ constexpr int fused_threads(int lr)
{
    return fused_points(lr) >= 512 ? fused_points(lr) / 16 : 32;
}

// The first forward round's input of product c of a block: both operands
// (NA = 2), or, with the operands as columns, operand a (c = 0) or b (c = 1)
// of one product.
template <bool ZT>
struct RawIn {
    static constexpr bool kZeroTop = ZT;
    const uint32_t *a, *b;
    size_t sa, sb;  // limbs between consecutive products' operands
    uint32_t la, lb;
    bool al_a, al_b;
    uint32_t q;
    CoefMul ca, cb;
    template <int E, int B, int NA>
    __device__ __forceinline__ void load(uint32_t (&x)[NA][1 << E], int base, int c) const
    {
        if constexpr (NA == 2) {
            load_coefs<E, B, ZT>(x[0], a + c * sa, base, la, al_a, ca, q);
            load_coefs<E, B, ZT>(x[1], b + c * sb, base, lb, al_b, cb, q);
        } else {
            CoefMul m;
            m.w0.x = c ? cb.w0.x : ca.w0.x;
            m.w0.y = c ? cb.w0.y : ca.w0.y;
            m.w1.x = c ? cb.w1.x : ca.w1.x;
            m.w1.y = c ? cb.w1.y : ca.w1.y;
            load_coefs<E, B, ZT>(x[0], c ? b : a, base, c ? lb : la, c ? al_b : al_a, m, q);
        }
    }
};

// The first product's operands k0, and prime p's input.
template <bool ZT>
__device__ __forceinline__ RawIn<ZT> raw_in(const FusedArgs &a, size_t k0, int p, uint32_t q)
{
    return RawIn<ZT>{a.A + k0 * a.a_tstride,
                     a.B + k0 * a.b_tstride,
                     a.a_tstride,
                     a.b_tstride,
                     a.a_len,
                     a.b_len,
                     a.a_al != 0,
                     a.b_al != 0,
                     q,
                     a.ca.c[p],
                     a.cb.c[p]};
}

// Forward rounds rd .. NR - 2 in shared memory, C columns and NA arrays.
template <int LR, int C, int NR, int NA, int T, int RD, class IO>
__device__ __forceinline__ void forward_rounds(const IO &io, const TwRef &T0, uint32_t q, int cols)
{
    if constexpr (RD < NR - 1) {
        round_io<LR, C, dif_base(LR, RD, NR), round_size(LR, RD, NR), true, NA, false, 0, T>(
            io, io, T0, q, cols);
        __syncthreads();
        forward_rounds<LR, C, NR, NA, T, RD + 1>(io, T0, q, cols);
    }
}

// Inverse rounds rd .. NR - 1.
template <int LR, int C, int NR, int T, int RD, class IO>
__device__ __forceinline__ void inverse_rounds(const IO &io, const TwRef &Ti, uint32_t q, int cols)
{
    if constexpr (RD < NR) {
        round_io<LR, C, dit_base(LR, RD, NR), dit_size(LR, RD, NR), false, 1, false, 0, T>(
            io, io, Ti, q, cols);
        __syncthreads();
        inverse_rounds<LR, C, NR, T, RD + 1>(io, Ti, q, cols);
    }
}

// The last forward round of both operands (arrays io and io + C 2^LR), the
// pointwise product and the first inverse round share one register round
// (their stage bits coincide), as in the row pass; the product replaces
// operand a.
template <int LR, int C, int NR, int T, class IO>
__device__ __forceinline__ void middle_round(const IO &io, const TwRef &T0, const TwRef &Ti,
                                             uint32_t q, uint32_t qinv, int cols)
{
    constexpr int EL = round_size(LR, NR - 1, NR);
    static_assert(EL == dit_size(LR, 0, NR), "mirrored rounds");
    constexpr int NGC = (1 << LR) >> EL;
#pragma unroll 1
    for (int g = threadIdx.x; g < cols * NGC; g += T) {
        const int c = g / NGC, base = (g & (NGC - 1)) << EL;
        uint32_t x[2][1 << EL];
        io.template load<EL, 0, 2>(x, base, c);
        dif_stages<EL, 0, 2, 0>(x, 0, T0, q);
        uint32_t z[1][1 << EL];
#pragma unroll
        for (int j = 0; j < (1 << EL); j++) z[0][j] = mul_mont<0>(x[0][j], x[1][j], q, qinv);
        dit_stages<EL, 0, 1, 0>(z, 0, Ti, q);
        io.template store<EL, 0, 1>(z, base, c);
    }
    __syncthreads();
}

// The limbs of a block's products from their coefficients' words in shared
// memory: word p of coefficient j at s[p PN + swz(j)], products of N = 2^LR
// coefficients back to back, a run of limbs per thread from the first
// coefficient j0 (a multiple of 4).  The limbs are asked for in order; every
// fourth coefficient reads the next four coefficients' words, 16 bytes each.
template <int N, int PN>
struct SmemRun {
    const uint32_t *s;
    int j0;
    uint32_t w[5][4];
    uint32_t h2, h3, h4a, h4b;  // the words that the run before hands over (CoefRun)
    __device__ __forceinline__ SmemRun(const uint32_t *words, int first) : s(words), j0(first) {}
    __device__ __forceinline__ uint64_t operator()(int i)
    {
        const int j = (i >> 1) & 3;
        if ((i & 7) == 0) {
            if (i) {
                h2 = w[2][3];
                h3 = w[3][3];
                h4a = w[4][2];
                h4b = w[4][3];
            } else {
                // coefficients j0 - 1 and j0 - 2 of the same product, if any
                // (read here, not at construction: a thread without limbs may
                // have a j0 past the arrays)
                const bool one = (j0 & (N - 1)) >= 1, two = (j0 & (N - 1)) >= 2;
                h2 = one ? s[2 * PN + swz(j0 - 1)] : 0u;
                h3 = one ? s[3 * PN + swz(j0 - 1)] : 0u;
                h4b = one ? s[4 * PN + swz(j0 - 1)] : 0u;
                h4a = two ? s[4 * PN + swz(j0 - 2)] : 0u;
            }
#pragma unroll
            for (int p = 0; p < 5; p++) {
                if (N >= 4) {
                    const uint4 v =
                        *reinterpret_cast<const uint4 *>(s + p * PN + swz(j0 + (i >> 1)));
                    w[p][0] = v.x; w[p][1] = v.y; w[p][2] = v.z; w[p][3] = v.w;
                } else {
#pragma unroll
                    for (int t = 0; t < 4; t++)
                        w[p][t] = t < N ? s[p * PN + swz(j0 + t)] : 0u;
                }
            }
        }
        if (i & 1) return (uint64_t)w[1][j] + (j >= 1 ? w[3][j - 1] : h3);
        return (uint64_t)w[0][j] + (j >= 1 ? w[2][j - 1] : h2) +
               (j >= 2 ? w[4][j - 2] : (j == 0 ? h4a : h4b));
    }
};

// The carries and the output of a block's products k0 .. k0 + cols - 1.
template <int LPT, int N, int PN>
__device__ __forceinline__ void block_limbs(const FusedArgs &a, size_t k0, int cols,
                                            const uint32_t *words, uint32_t *wsm)
{
    const Sink &o = a.sink;
    const int j0 = threadIdx.x * LPT;     // first limb of the run
    const int c = j0 / (2 * N);           // its product
    const size_t k = k0 + c;
    static_assert(2 * N % LPT == 0, "a run lies within one product");
    const bool live = c < cols;
    // the product's limbs start at limb `base` of the tile
    const long base = (long)c * 2 * N;
    uint32_t *out = live ? o.out + sink_node(o, k) * o.out_tstride - base : nullptr;
    const uint32_t *add = live && o.add ? o.add + k * o.add_tstride - base : nullptr;
    tile_carry<-1, -1, LPT>(SmemRun<N, PN>{words, j0 / 2}, cols * 2 * N, out,
                            base + (long)o.out_len, o.dec, add, base + (long)o.add_len, wsm,
                            nullptr);
}

// Whole products in one block: the five primes in turn (per prime both
// forward transforms, the pointwise product and the inverse transform in
// shared memory), then remaindering and carries.
// A block holds one product of 2^10 or 2^11 points or as many shorter ones as
// fill 2^9, one group of 16 points of both operands per thread: every thread
// has a group in every round of four stages, both operands share the stage
// twiddles, and up to 2^9 points the block is a single warp, whose barriers
// cost next to nothing.  Sixteen warps per SM at up to 128 registers do
// better here than 32 warps with half of them idle between the barriers of
// the middle and inverse rounds: the levels of 2^8 .. 2^11 points of
// C(2,050,572,903) 11.4 -> 10.5 ms (2^24 limbs of products take 260 us at 2^7
// points, 285, 335, 354 and 365 at 2^11).
// Layout (words): six arrays of PN; prime p's transforms use arrays p
// (operands a, then the products, whose residues stay there) and p + 1
// (operands b; the next prime overwrites them): 24 PN bytes, four blocks of
// 2^11 points per SM.  The coefficients' words then replace the residues in
// place.  The products' limbs form one tile: no carry leaves a product, so the
// scan needs no boundaries between them.
template <int LR, bool ZT>
__global__ void __launch_bounds__(fused_threads(LR), 512 / fused_threads(LR))
    ntt_mul_fused(FusedArgs a)
{
    chain_wait();
    extern __shared__ uint32_t sm[];
    __shared__ uint32_t wsm[32];
    constexpr int N = 1 << LR, PN = fused_points(LR), P = PN / N;
    constexpr int T = fused_threads(LR), NR = rounds_of(LR);
    const size_t k0 = (size_t)blockIdx.x * P;
    const int cols = (int)(a.nprod - k0 < (size_t)P ? a.nprod - k0 : (size_t)P);
#pragma unroll 1
    for (int p = 0; p < kNumPrimes; p++) {
        const uint32_t q = c_q[0][p], qinv = c_qinv[0][p];
        const TwRef T0{tw_table(a.tw, 0, p, 0), p};
        const TwRef Ti{tw_table(a.tw, 0, p, 1), p};
        const SmemIO<LR, P, false, true> io{sm + p * PN};
        round_io<LR, P, dif_base(LR, 0, NR), round_size(LR, 0, NR), true, 2, false, 0, T>(
            raw_in<ZT>(a, k0, p, q), io, T0, q, cols);
        __syncthreads();
        if constexpr (NR == 1) {
            // up to 16 points: elementwise in the swizzled space, then back
            for (int i = threadIdx.x; i < PN; i += T)
                io.s[i] = mul_mont<0>(io.s[i], io.s[PN + i], q, qinv);
            __syncthreads();
            inverse_rounds<LR, P, NR, T, 0>(io, Ti, q, cols);
        } else {
            forward_rounds<LR, P, NR, 2, T, 1>(io, T0, q, cols);
            middle_round<LR, P, NR, T>(io, T0, Ti, q, qinv, cols);
            inverse_rounds<LR, P, NR, T, 1>(io, Ti, q, cols);
        }
    }
    // the coefficients' words in place of their residues
    for (int j = threadIdx.x; j < cols * N; j += T) {
        uint32_t *x = sm + swz(j);
        uint32_t r[kNumPrimes], w[5];
#pragma unroll
        for (int p = 0; p < kNumPrimes; p++) r[p] = x[p * PN];
        if (a.sink.dec) crt5_dec<0>(r, w);
        else crt5<0>(r, w);
#pragma unroll
        for (int p = 0; p < 5; p++) x[p * PN] = w[p];
    }
    __syncthreads();
    constexpr int LPT = 2 * PN / T;  // 32 limbs
    block_limbs<LPT, N, PN>(a, k0, cols, sm, wsm);
}

// The same for few products at a time: a cluster of five blocks per product,
// one prime each, so that a product's primes run side by side instead of in
// turn, the operands as two columns, in blocks of N / 4 threads with rounds of
// at most three stages (a shorter serial chain per thread).  Every block then
// remainders a fifth of the coefficients from all five blocks' residues
// (distributed shared memory) into the first block's shared memory, which
// carries and writes out.  The cluster barriers are the hardware's; the blocks
// of a cluster always run together.
constexpr int kClusterMinLog = 5;  // shorter products: the schoolbook sizes
__host__ __device__ constexpr int cluster_threads(int lr)
{
    const int t = (1 << lr) / 4;
    return t < 32 ? 32 : t;
}

template <int LR, bool ZT>
__global__ void __cluster_dims__(kNumPrimes, 1, 1) __launch_bounds__(cluster_threads(LR))
    ntt_mul_cluster(FusedArgs a)
{
    chain_wait();
    namespace cg = cooperative_groups;
    extern __shared__ uint32_t sm[];
    __shared__ uint32_t wsm[32];
    constexpr int N = 1 << LR;
    constexpr int T = cluster_threads(LR), NR = (LR + 2) / 3;
    cg::cluster_group cluster = cg::this_cluster();
    const int p = blockIdx.x % kNumPrimes;  // the block's rank in its cluster
    const size_t k = blockIdx.x / kNumPrimes;
    const uint32_t q = c_q[0][p], qinv = c_qinv[0][p];
    const TwRef T0{tw_table(a.tw, 0, p, 0), p};
    const TwRef Ti{tw_table(a.tw, 0, p, 1), p};
    const SmemIO<LR, 2, false> xy{sm};  // columns: operands a and b
    const SmemIO<LR, 1, false> io{sm};  // arrays: b follows a
    round_io<LR, 2, dif_base(LR, 0, NR), round_size(LR, 0, NR), true, 1, false, 0, T>(
        raw_in<ZT>(a, k, p, q), xy, T0, q);
    __syncthreads();
    forward_rounds<LR, 2, NR, 1, T, 1>(xy, T0, q, 2);
    middle_round<LR, 1, NR, T>(io, T0, Ti, q, qinv, 1);
    inverse_rounds<LR, 1, NR, T, 1>(io, Ti, q, 1);
    cluster.sync();
    uint32_t *words = sm + 2 * N;
    uint32_t *out = cluster.map_shared_rank(words, 0);
    for (int j = p * T + (int)threadIdx.x; j < N; j += kNumPrimes * T) {
        uint32_t r[kNumPrimes], w[5];
#pragma unroll
        for (int i = 0; i < kNumPrimes; i++) r[i] = cluster.map_shared_rank(sm, i)[swz(j)];
        if (a.sink.dec) crt5_dec<0>(r, w);
        else crt5<0>(r, w);
#pragma unroll
        for (int i = 0; i < 5; i++) out[i * N + swz(j)] = w[i];
    }
    cluster.sync();  // no block reads another's shared memory after this
    constexpr int LPT = 2 * N / T > kLimbsPerThread ? 2 * N / T : kLimbsPerThread;
    if (p == 0) block_limbs<LPT, N, N>(a, k, 1, words, wsm);
}

// ------------------------------------------------------------ host side

struct NttPlan {
    int np = 0;
    int ncol = 0;
    int rcol[3] = {0, 0, 0};
    int rrow = 0;
};

// The default row-pass size of a transform of 2^np points: as long as the
// columns fit one pass, rows of 2^12 points (at least 2^4 column rows), but
// 2^10 where that leaves 2^5 or 2^6 column rows; above 2^22 points, where the
// columns take two passes whatever the rows, rows of 2^9.  Measured (ms per
// level of 2^27 limbs, rows of 2^9 : 2^10 : 2^11 : 2^12): np = 17 3.74 : 3.74 :
// 3.81 : 3.92, 18 4.00 : 3.87 : 3.93 : 3.95, 20 5.10 : 4.42 : 4.29 : 4.16, 22
// 5.17 : 5.19 : 5.42 : 4.76, 23 5.14 : 5.21 : 5.33 : 5.46, 25 5.27 : 5.26 : 5.48 :
// 5.53.
int default_row(int np)
{
    if (np > 22) return 9;
    if (np == 17 || np == 18) return 10;
    return std::min(12, np - kColMinLog);
}

// The plan of a product of 2^n limbs (2^np points, np = n - 1 >= 12): a row
// pass of up to 2^12 points and column passes of at most 2^10 rows, split as
// evenly as possible.  2^12 points take the row pass alone.  A row-pass size
// tuned for this device (Ctx::row_log: rows of 2^9 .. 2^12 points) replaces
// the default.  plan_row_ok: the row sizes a tuning table may name for a
// product of 2^n limbs (at most two column passes of at least 2 rows, at
// least 2^4 in prime sets 1 and 2, whose column passes are built for 2^4 ..
// 2^10 rows; the bounds are those of tables written for 2^n points, one stage
// more than the transform has, and every size they allow has a plan).
bool plan_row_ok(int n, int rrow)
{
    if (n > kLogMaxNtt || rrow < 9 || rrow > kRowMaxLog) return false;
    const int rem = n - rrow;
    const int ncol = (rem + kColMaxLog - 1) / kColMaxLog;
    if (rem < 2 || ncol > 2) return false;
    return rem / ncol >= (set_for(n - 1) == 0 ? 2 : kColMinLog);
}

static NttPlan make_plan(const Ctx &c, int np)
{
    NttPlan P;
    P.np = np;
    const int n = np + 1;
    if (np <= kRowMaxLog) {  // the row pass alone
        P.rrow = np;
        return P;
    }
    P.rrow = default_row(np);
    if (n <= kLogMaxNtt && c.row_log[n] && plan_row_ok(n, c.row_log[n])) P.rrow = c.row_log[n];
    int rem = np - P.rrow;
    P.ncol = (rem + kColMaxLog - 1) / kColMaxLog;
    for (int i = 0; i < P.ncol; i++) {
        P.rcol[i] = rem / (P.ncol - i);
        rem -= P.rcol[i];
    }
    std::sort(P.rcol, P.rcol + P.ncol, [](int x, int y) { return x > y; });
    return P;
}

// Raise the kernel's dynamic shared-memory limit when dynamic plus static
// shared memory (a few hundred bytes here) could pass the default 48 KiB.
template <typename K>
static void set_smem(K kernel, size_t bytes)
{
    if (bytes > 40 * 1024)
        CAT_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)bytes));
}

template <int LR, int PS>
static void launch_col(bool fwd, dim3 grid, cudaStream_t s, const ColArgs &a)
{
    const size_t smem = ((size_t)1 << (LR + col_log_c(LR))) * sizeof(uint32_t);
    // the first pass of operands of at most half the transform (every tree
    // level; lengths count limbs, two per point) knows its upper half is zero
    const bool zt = fwd && a.src && std::max(a.src_len, a.src_y_len) <= ((size_t)1 << a.m);
    if (zt) {
        set_smem(ntt_col_fwd<LR, PS, kColV, 2>, smem);
        launch_chained(ntt_col_fwd<LR, PS, kColV, 2>, grid, kColFwdThreads, smem, s, a);
    } else if (fwd && a.src) {
        set_smem(ntt_col_fwd<LR, PS, kColV, 1>, smem);
        launch_chained(ntt_col_fwd<LR, PS, kColV, 1>, grid, kColFwdThreads, smem, s, a);
    } else if (fwd) {
        set_smem(ntt_col_fwd<LR, PS, kColV, 0>, smem);
        launch_chained(ntt_col_fwd<LR, PS, kColV, 0>, grid, kColFwdThreads, smem, s, a);
    } else {
        set_smem(ntt_col_inv<LR, PS, kColV>, smem);
        launch_chained(ntt_col_inv<LR, PS, kColV>, grid, kColInvThreads, smem, s, a);
    }
}

// ps: the prime set of the transform (set_for)
// The twiddles of a column pass of 2^r rows over blocks of 2^m points (set
// ps, direction dir): entry row 2^(m-r) + col = w^((col bitrev_r(row)) << shift)
// in Montgomery form, the value the pass would otherwise compute for that
// point (tw_pow_mont, exactly as the stepping reaches it).
template <int PS>
__global__ void col_twiddle_table(const uint2 *tw, int m, int r, int dir, uint32_t *tab)
{
    const int p = blockIdx.y;
    const uint32_t q = c_q[PS][p], qinv = c_qinv[PS][p];
    const uint2 *T = tw_table(tw, PS, p, dir);
    const int shift = set_log_root(PS) - m;
    const uint32_t cols = 1u << (m - r);
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << m);
         i += gridDim.x * blockDim.x) {
        const uint32_t row = i >> (m - r), col = i & (cols - 1);
        tab[((size_t)p << m) + i] =
            tw_pow_mont<PS>(T, (col * bitrev(row, r)) << shift, q, qinv);
    }
}

// A column pass's twiddle table, built on first use; null when the context
// computes its twiddles (a budgeted context, or no room for the table).
static const uint32_t *col_twiddles(Ctx &c, int ps, int m, int r, int dir, cudaStream_t s)
{
    if (!c.col_tw_tables || c.budget || c.shared_budget) return nullptr;
    for (const Ctx::ColTwTable &t : c.col_tw)
        if (t.ps == ps && t.m == m && t.lr == r && t.dir == dir) return t.p;
    uint32_t *p = nullptr;
    if (cudaMalloc(&p, ((size_t)kNumPrimes << m) * sizeof(uint32_t)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    const unsigned blocks = (unsigned)std::min<size_t>(((size_t)1 << m) / 256 + 1, 4096);
    const dim3 grid(blocks, kNumPrimes);
    if (ps == 0) col_twiddle_table<0><<<grid, 256, 0, s>>>(c.twiddles, m, r, dir, p);
    else if (ps == 1) col_twiddle_table<1><<<grid, 256, 0, s>>>(c.twiddles, m, r, dir, p);
    else col_twiddle_table<2><<<grid, 256, 0, s>>>(c.twiddles, m, r, dir, p);
    CAT_LAUNCH("col_twiddle_table");
    c.col_tw.push_back(Ctx::ColTwTable{ps, m, r, dir, p});
    return p;
}

void drop_col_twiddles(Ctx &c)
{
    if (c.col_tw.empty()) return;
    cudaDeviceSynchronize();  // no pass still reads them
    for (const Ctx::ColTwTable &t : c.col_tw) cudaFree(t.p);
    c.col_tw.clear();
}

// One operand source of a batched product.
struct Operand {
    const uint32_t *p;
    size_t tstride;  // limbs between consecutive transforms (for batches)
    size_t len;      // valid limbs per transform
    // the transform with fewer limbs than the others, if any
    unsigned ragged = ~0u;
    size_t ragged_len = 0;
};
constexpr Operand kNoSource{nullptr, 0, 0};

// One column pass over `total` points (blocks of 2^m points, 2^r rows).
//
// scaled (first forward passes): 1 = the call's last transform (or its only
// one) is an operand b, 2 = the odd ones are (adjacent pairs); their input
// multipliers then carry the pointwise scale.
//
// x: the sources of a first forward pass (p null otherwise); y, when given,
// the source of the call's last transform (the second operand of a product or
// the common one of broadcast products), so that both operands of a single
// product share one launch.
static void col_pass(Ctx &c, int ps, bool fwd, uint32_t *data, size_t pstride, size_t total,
                     int m, int r, const Operand &x, const Operand *y, bool dec, cudaStream_t s,
                     int scaled = 0)
{
    const uint32_t *src = x.p;
    auto aligned16 = [](const Operand &o) {
        return (reinterpret_cast<uintptr_t>(o.p) & 15) == 0 && (o.tstride & 3) == 0;
    };
    ColArgs a;
    a.coef = make_coef(ps, dec);
    a.coef_b = scaled ? make_coef(ps, dec, m) : a.coef;
    a.odd_b = scaled == 2;
    a.src_al = aligned16(x);
    a.last = y || scaled == 1 ? (unsigned)(total >> m) - 1u : ~0u;
    a.src_y = y ? y->p : x.p;
    a.src_y_len = y ? y->len : x.len;
    a.src_y_al = aligned16(y ? *y : x);
    // (measured per C(2,050,572,903): tables in every pass beat computed
    // twiddles at every block size, the first forward passes' large tables
    // included, once the table loads go through the read-only path)
    const int tmax = src ? c.col_tw_first_max_log : c.col_tw_max_log;
    a.twtab = m <= tmax ? col_twiddles(c, ps, m, r, fwd ? 0 : 1, s) : nullptr;
    a.data = data;
    a.pstride = pstride;
    a.m = m;
    a.src = src;
    a.src_tstride = x.tstride;
    a.src_len = x.len;
    a.ragged = x.ragged;
    a.ragged_len = x.ragged_len;
    a.tw = c.twiddles;
    const size_t ctas = total >> (r + col_log_c(r));
    a.nblk = (unsigned)(total >> m);
    dim3 grid((unsigned)ctas, kNumPrimes);
    // algorithmic bytes: every point of the five prime arrays read and
    // written once (the first forward pass reads limbs instead)
    double bytes = 8.0 * kNumPrimes * (double)total;
    if (src)
        bytes = 4.0 * kNumPrimes * (double)total +
                4.0 * (double)x.len * (double)((total >> m) - (y ? 1 : 0)) +
                (y ? 4.0 * (double)y->len : 0.0);
    const char *name = !fwd ? "ntt_col_inv" : src ? "ntt_col_fwd_first" : "ntt_col_fwd";
    const int tok = prof_begin(c, name, s);
    if (ps == 0) {
        switch (r) {
        case 1: launch_col<1, 0>(fwd, grid, s, a); break;
        case 2: launch_col<2, 0>(fwd, grid, s, a); break;
        case 3: launch_col<3, 0>(fwd, grid, s, a); break;
        case 4: launch_col<4, 0>(fwd, grid, s, a); break;
        case 5: launch_col<5, 0>(fwd, grid, s, a); break;
        case 6: launch_col<6, 0>(fwd, grid, s, a); break;
        case 7: launch_col<7, 0>(fwd, grid, s, a); break;
        case 8: launch_col<8, 0>(fwd, grid, s, a); break;
        case 9: launch_col<9, 0>(fwd, grid, s, a); break;
        case 10: launch_col<10, 0>(fwd, grid, s, a); break;
        default: fail(CAT_EINVAL, "column pass size out of range");
        }
    } else if (ps == 1) {
        // 2^23 .. 2^25 points: column passes of 2^5 .. 2^8 rows
        switch (r) {
        case 4: launch_col<4, 1>(fwd, grid, s, a); break;
        case 5: launch_col<5, 1>(fwd, grid, s, a); break;
        case 6: launch_col<6, 1>(fwd, grid, s, a); break;
        case 7: launch_col<7, 1>(fwd, grid, s, a); break;
        case 8: launch_col<8, 1>(fwd, grid, s, a); break;
        case 9: launch_col<9, 1>(fwd, grid, s, a); break;
        case 10: launch_col<10, 1>(fwd, grid, s, a); break;
        default: fail(CAT_EINVAL, "column pass size out of range");
        }
    } else {
        // 2^26 points: column passes of 2^7 .. 2^9 rows
        switch (r) {
        case 4: launch_col<4, 2>(fwd, grid, s, a); break;
        case 5: launch_col<5, 2>(fwd, grid, s, a); break;
        case 6: launch_col<6, 2>(fwd, grid, s, a); break;
        case 7: launch_col<7, 2>(fwd, grid, s, a); break;
        case 8: launch_col<8, 2>(fwd, grid, s, a); break;
        case 9: launch_col<9, 2>(fwd, grid, s, a); break;
        case 10: launch_col<10, 2>(fwd, grid, s, a); break;
        default: fail(CAT_EINVAL, "column pass size out of range");
        }
    }
    CAT_LAUNCH(fwd ? "ntt_col_fwd" : "ntt_col_inv");
    prof_end(c, tok, s, bytes);
}

template <int LR, int PS>
static void launch_row_t(dim3 grid, cudaStream_t s, const RowArgs &a, bool pre)
{
    if (pre) {  // broadcast products, the common transform complete
        const size_t smem = ((size_t)1 << kRowMaxLog) * sizeof(uint32_t);
        set_smem(ntt_row_mul_bcast<LR, PS>, smem);
        launch_chained(ntt_row_mul_bcast<LR, PS>, grid, kRowThreads, smem, s, a);
    } else if (a.mode == PAIR_SQUARE) {
        const size_t smem = ((size_t)1 << kRowMaxLog) * sizeof(uint32_t);
        set_smem(ntt_row_mul<LR, true, PS>, smem);
        launch_chained(ntt_row_mul<LR, true, PS>, grid, kRowThreads, smem, s, a);
    } else {
        const size_t smem = ((size_t)2 << kRowMaxLog) * sizeof(uint32_t);
        set_smem(ntt_row_mul<LR, false, PS>, smem);
        launch_chained(ntt_row_mul<LR, false, PS>, grid, kRowThreads, smem, s, a);
    }
}

// The fused row pass of nprod products of 2^np points with prime set ps
// (pre: broadcast products whose common transform ntt_row_fwd completed).
static void launch_row(int ps, int lr, size_t nprod, int np, cudaStream_t s, const RowArgs &a,
                       bool pre = false)
{
    dim3 grid((unsigned)(nprod << (np - kRowMaxLog)), kNumPrimes);
    if (ps == 0) {
        switch (lr) {
        case 9: launch_row_t<9, 0>(grid, s, a, pre); break;
        case 10: launch_row_t<10, 0>(grid, s, a, pre); break;
        case 11: launch_row_t<11, 0>(grid, s, a, pre); break;
        case 12: launch_row_t<12, 0>(grid, s, a, pre); break;
        default: fail(CAT_EINVAL, "row pass size out of range");
        }
    } else if (ps == 1) {
        switch (lr) {
        case 9: launch_row_t<9, 1>(grid, s, a, pre); break;
        case 10: launch_row_t<10, 1>(grid, s, a, pre); break;
        case 11: launch_row_t<11, 1>(grid, s, a, pre); break;
        case 12: launch_row_t<12, 1>(grid, s, a, pre); break;
        default: fail(CAT_EINVAL, "row pass size out of range");
        }
    } else {
        switch (lr) {
        case 9: launch_row_t<9, 2>(grid, s, a, pre); break;
        case 10: launch_row_t<10, 2>(grid, s, a, pre); break;
        case 11: launch_row_t<11, 2>(grid, s, a, pre); break;
        case 12: launch_row_t<12, 2>(grid, s, a, pre); break;
        default: fail(CAT_EINVAL, "row pass size out of range");
        }
    }
    CAT_LAUNCH("ntt_row_mul");
}

template <int LR, int PS>
static void launch_row_fwd_t(dim3 grid, cudaStream_t s, const RowArgs &a)
{
    const size_t smem = ((size_t)1 << kRowMaxLog) * sizeof(uint32_t);
    set_smem(ntt_row_fwd<LR, PS>, smem);
    launch_chained(ntt_row_fwd<LR, PS>, grid, kRowThreads, smem, s, a);
}

// The row pass's forward rounds of one transform of 2^np points in place (the
// common operand of broadcast products; a.F at its slot).
static void launch_row_fwd(int ps, int lr, int np, cudaStream_t s, const RowArgs &a)
{
    dim3 grid((unsigned)((size_t)1 << (np - kRowMaxLog)), kNumPrimes);
    switch (ps * 16 + lr) {
    case 9: launch_row_fwd_t<9, 0>(grid, s, a); break;
    case 10: launch_row_fwd_t<10, 0>(grid, s, a); break;
    case 11: launch_row_fwd_t<11, 0>(grid, s, a); break;
    case 12: launch_row_fwd_t<12, 0>(grid, s, a); break;
    case 16 + 9: launch_row_fwd_t<9, 1>(grid, s, a); break;
    case 16 + 10: launch_row_fwd_t<10, 1>(grid, s, a); break;
    case 16 + 11: launch_row_fwd_t<11, 1>(grid, s, a); break;
    case 16 + 12: launch_row_fwd_t<12, 1>(grid, s, a); break;
    case 32 + 9: launch_row_fwd_t<9, 2>(grid, s, a); break;
    case 32 + 10: launch_row_fwd_t<10, 2>(grid, s, a); break;
    case 32 + 11: launch_row_fwd_t<11, 2>(grid, s, a); break;
    case 32 + 12: launch_row_fwd_t<12, 2>(grid, s, a); break;
    default: fail(CAT_EINVAL, "row pass size out of range");
    }
    CAT_LAUNCH("ntt_row_fwd");
}

// Remaindering of a batch, specialised by prime set and by the sink's mode
// (base 10^9 or 2^32, with or without an addend).
template <int PS>
static void launch_crt_ps(unsigned grid, cudaStream_t s, const CrtArgs &a)
{
    const bool dec = a.sink.dec, add = a.sink.add != nullptr;
    if (a.step)  // binary, without an addend (mul_chunked)
        launch_chained(crt_carry_tiles<PS, false, false, true>, grid, kTileThreads, 0, s, a);
    else if (dec && add)
        launch_chained(crt_carry_tiles<PS, true, true, false>, grid, kTileThreads, 0, s, a);
    else if (dec)
        launch_chained(crt_carry_tiles<PS, true, false, false>, grid, kTileThreads, 0, s, a);
    else if (add)
        launch_chained(crt_carry_tiles<PS, false, true, false>, grid, kTileThreads, 0, s, a);
    else
        launch_chained(crt_carry_tiles<PS, false, false, false>, grid, kTileThreads, 0, s, a);
}

static void launch_crt(int ps, unsigned grid, cudaStream_t s, const CrtArgs &a)
{
    if (ps == 0)
        launch_crt_ps<0>(grid, s, a);
    else if (ps == 1)
        launch_crt_ps<1>(grid, s, a);
    else
        launch_crt_ps<2>(grid, s, a);
}

// Whether every operand of a batch (tstride limbs apart) starts on an 8-byte
// boundary, so that a coefficient is one 8-byte load.
static int aligned8(const uint32_t *p, size_t tstride)
{
    return (reinterpret_cast<uintptr_t>(p) & 7) == 0 && (tstride & 1) == 0;
}

template <bool SQ, bool ZT>
static void launch_row_limbs_t(size_t nprod, cudaStream_t s, const RowLimbArgs &a)
{
    const size_t smem = ((size_t)(SQ ? 1 : 2) << kRowMaxLog) * sizeof(uint32_t);
    set_smem(ntt_row_limbs<SQ, ZT>, smem);
    launch_chained(ntt_row_limbs<SQ, ZT>, dim3((unsigned)nprod, kNumPrimes), kRowThreads, smem, s,
                   a);
}

// The whole transforms of nprod products of 2^12 points, from limbs.
static void launch_row_limbs(size_t nprod, bool square, cudaStream_t s, const RowLimbArgs &a)
{
    const bool zt = std::max(a.a_len, a.b_len) <= (1u << kRowMaxLog);
    if (square) {
        if (zt) launch_row_limbs_t<true, true>(nprod, s, a);
        else launch_row_limbs_t<true, false>(nprod, s, a);
    } else {
        if (zt) launch_row_limbs_t<false, true>(nprod, s, a);
        else launch_row_limbs_t<false, false>(nprod, s, a);
    }
    CAT_LAUNCH("ntt_row_limbs");
}

// Scratch of one batch of multi-pass products: what is null is taken from the
// context's pool when it is needed; the no-allocation multiply brings its fixed
// arrays, a caller that has another way to go its own allocations.
struct MulScratch {
    DevBuf<uint32_t> Fb, Gb;
    DevBuf<uint8_t> mb;
    uint32_t *F = nullptr, *G = nullptr;
    uint8_t *maps = nullptr;
};

// The carries of nprod products of `tiles` tiles each, whose compact tile
// maps are in maps.
static void carry_finish(Ctx &c, const uint8_t *maps, size_t nprod, size_t tiles, const Sink &sink,
                         cudaStream_t s)
{
    const int tok = prof_begin(c, "carry_resolve", s);
    const size_t threads = std::min<size_t>(1024, (tiles + 31) / 32 * 32);
    const size_t nb = (tiles + threads - 1) / threads;
    launch_chained(carry_resolve, (unsigned)(nprod * nb), (unsigned)threads, 0, s, maps, tiles,
                   (int)nb, sink.out, sink.out_tstride, sink.out_len, sink.dec, sink.out_index);
    CAT_LAUNCH("carry_resolve");
    prof_end(c, tok, s, (double)(nprod * tiles));
}

// Batched products of transforms of 2^np >= 2^12 points.
//  mode PAIR_ADJACENT:  nprod products of transforms (2k, 2k+1) of `x`
//                       (2 nprod transforms, tstride apart);
//  mode PAIR_FIRST_TWO: one product of x and y;
//  mode PAIR_SQUARE:    nprod squares of x's transforms;
//  mode PAIR_BROADCAST: nprod products of x's transforms (tstride apart) with
//                       one y, whose transform is computed once.
// With step, the products (PAIR_BROADCAST, np >= 13) are summed into one, each
// step coefficients (a multiple of 4) after the one before, and none reaches
// past the next one's stretch of step.
static void ntt_mul_multipass(Ctx &c, int np, int mode, size_t nprod, Operand x, Operand y,
                              const Sink &sink, cudaStream_t s, MulScratch &&m = MulScratch{},
                              uint32_t step = 0)
{
    const NttPlan P = make_plan(c, np);
    const int PS = set_for(np);
    const bool dec = sink.dec;
    const size_t N = (size_t)1 << np;
    const size_t ntf = mode == PAIR_ADJACENT ? 2 * nprod
                       : mode == PAIR_SQUARE ? nprod
                       : mode == PAIR_BROADCAST ? nprod + 1
                                                : 2;
    const size_t fp = ntf * N, gp = nprod * N;
    // the products' own bytes: operands read and products written once
    const double unit = 4.0 * (double)nprod * (double)(x.len + sink.out_len) +
                        (mode == PAIR_SQUARE ? 0.0
                         : mode == PAIR_BROADCAST ? 4.0 * (double)y.len
                                                  : 4.0 * (double)nprod * (double)y.len);
    int tok;
    if (P.ncol == 0) {
        // the row pass alone, from the operands' limbs
        if (!m.G) {
            m.Gb = DevBuf<uint32_t>(c, gp * kNumPrimes, s);
            m.G = m.Gb.get();
        }
        RowLimbArgs ra;
        ra.A = x.p;
        ra.B = mode == PAIR_ADJACENT ? x.p + x.tstride : (mode == PAIR_SQUARE ? x.p : y.p);
        ra.a_tstride = mode == PAIR_ADJACENT ? 2 * x.tstride : x.tstride;
        ra.b_tstride = mode == PAIR_ADJACENT ? 2 * x.tstride
                       : mode == PAIR_SQUARE ? x.tstride
                                             : 0;
        ra.a_len = (uint32_t)x.len;
        ra.b_len = (uint32_t)(mode == PAIR_ADJACENT || mode == PAIR_SQUARE ? x.len : y.len);
        ra.a_al = aligned8(ra.A, ra.a_tstride);
        ra.b_al = aligned8(ra.B, ra.b_tstride);
        ra.G = m.G;
        ra.gpstride = gp;
        ra.tw = c.twiddles;
        ra.scale = make_scale(PS, np);
        ra.ca = make_coef(PS, dec);
        ra.cb = make_coef(PS, dec, np);
        tok = prof_begin(c, "ntt_row_limbs", s);
        launch_row_limbs(nprod, mode == PAIR_SQUARE, s, ra);
        prof_end(c, tok, s, 4.0 * kNumPrimes * (double)gp + unit, unit);
    } else {
        if (!m.F) {
            m.Fb = DevBuf<uint32_t>(c, fp * kNumPrimes, s);
            m.F = m.Fb.get();
        }
        uint32_t *F = m.F;
        // forward column passes (operand b's input multipliers take the
        // pointwise scale)
        const int r0 = P.rcol[0];
        // one launch for the operands of a single or a broadcast product,
        // unless only one of them fills its transform's upper half and the
        // transform is long: apart, the other's zero half is left out (us,
        // apart : together, one product whose operands fill 0.65 and 0.35 of it:
        // 2^13 points 48.7 : 46.2, 2^17 55.7 : 54.0, 2^18 67.9 : 67.5, 2^20 122.5 :
        // 120.0, 2^22 383.0 : 380.6, 2^23 732.5 : 732.3)
        const bool two = mode == PAIR_FIRST_TWO || mode == PAIR_BROADCAST;
        const bool together =
            two && (np <= 17 || (x.len <= N) == (y.len <= N));
        if (together) {
            col_pass(c, PS, true, F, fp, fp, np, r0, x, &y, dec, s, 1);
        } else if (two) {
            col_pass(c, PS, true, F, fp, fp - N, np, r0, x, nullptr, dec, s);
            col_pass(c, PS, true, F + fp - N, fp, N, np, r0, y, nullptr, dec, s, 1);
        } else {
            col_pass(c, PS, true, F, fp, fp, np, r0, x, nullptr, dec, s,
                     mode == PAIR_ADJACENT ? 2 : 0);
        }
        int mm = np - r0;
        for (int i = 1; i < P.ncol; i++) {
            col_pass(c, PS, true, F, fp, fp, mm, P.rcol[i], kNoSource, nullptr, false, s);
            mm -= P.rcol[i];
        }
        // fused row pass
        if (!m.G) {
            m.Gb = DevBuf<uint32_t>(c, gp * kNumPrimes, s);
            m.G = m.Gb.get();
        }
        RowArgs ra;
        ra.F = F;
        ra.fpstride = fp;
        ra.G = m.G;
        ra.gpstride = gp;
        ra.np = np;
        ra.mode = mode;
        ra.tw = c.twiddles;
        ra.scale = make_scale(PS, np);
        // broadcast products: y's transform completed once, in its slot, so that
        // the row pass transforms only the x's
        const bool pre = mode == PAIR_BROADCAST && nprod >= 2;
        if (pre) {
            RowArgs ya = ra;
            ya.F = F + nprod * N;
            tok = prof_begin(c, "ntt_row_fwd", s);
            launch_row_fwd(PS, P.rrow, np, s, ya);
            prof_end(c, tok, s, 8.0 * (double)N * kNumPrimes);
        }
        tok = prof_begin(c, "ntt_row_mul", s);
        launch_row(PS, P.rrow, nprod, np, s, ra, pre);
        prof_end(c, tok, s, (mode == PAIR_SQUARE ? 8.0 : 12.0) * kNumPrimes * (double)gp, unit);
        m.Fb.reset();
        // inverse column passes, reverse order
        for (int i = P.ncol - 1; i >= 0; i--) {
            int mi = np;
            for (int j = 0; j < i; j++) mi -= P.rcol[j];
            col_pass(c, PS, false, m.G, gp, gp, mi, P.rcol[i], kNoSource, nullptr, false, s);
        }
    }
    // remaindering and carries
    const size_t sums = step ? 1 : nprod;
    const size_t tiles = step ? (sink.out_len + kTile - 1) / kTile : N / kTileCoefs;
    if (!m.maps) {
        m.mb = DevBuf<uint8_t>(c, sums * tiles, s);
        m.maps = m.mb.get();
    }
    CrtArgs ca;
    ca.G = m.G;
    ca.gpstride = gp;
    ca.np = np;
    ca.sink = sink;
    ca.tile_maps = m.maps;
    ca.step = step;
    ca.nprod = (uint32_t)nprod;
    tok = prof_begin(c, "crt_carry_tiles", s);
    launch_crt(PS, (unsigned)(sums * tiles), s, ca);
    CAT_LAUNCH("crt_carry_tiles");
    prof_end(c, tok, s, 4.0 * kNumPrimes * (double)gp + 4.0 * (double)sums * (double)sink.out_len);
    carry_finish(c, m.maps, sums, tiles, sink, s);
}

template <int LR, bool ZT>
static void launch_fused_t(size_t nprod, bool spread, cudaStream_t s, const FusedArgs &a)
{
    if constexpr (LR >= kClusterMinLog) {
        if (spread) {
            const size_t smem = 7 * ((size_t)1 << LR) * sizeof(uint32_t);
            set_smem(ntt_mul_cluster<LR, ZT>, smem);
            launch_chained(ntt_mul_cluster<LR, ZT>, (unsigned)(nprod * kNumPrimes),
                           cluster_threads(LR), smem, s, a);
            return;
        }
    }
    constexpr size_t PN = fused_points(LR), P = PN >> LR;
    const size_t smem = 6 * PN * sizeof(uint32_t);
    set_smem(ntt_mul_fused<LR, ZT>, smem);
    launch_chained(ntt_mul_fused<LR, ZT>, (unsigned)((nprod + P - 1) / P), fused_threads(LR), smem,
                   s, a);
}

// Whether a batch of one-block products takes a cluster of five blocks per
// product: while the clusters' threads fit the chip's 2,048 per SM about once,
// at most 512 products.  Measured (us per launch, one block : cluster): one
// product of 2^10 points 26.9 : 8.6, of 2^8 20.9 : 8.1, of 2^5 12.8 : 6.6; 256
// products of 2^10 points 28.9 : 22.8, 512 34.8 : 37.3; of 2^11 points 128
// products 32.5 : 26.0, 256 36.9 : 42.6; of 2^9 points 512 products 27.0 : 20.8,
// 1,024 33.1 : 34.0; of 2^5 points 512 products 18.8 : 10.8, 2,048 20.7 : 29.1.
static bool spread_primes(size_t nprod, int lr, int num_sms)
{
    if (nprod == 1) return true;
    return nprod <= 512 && nprod * kNumPrimes * (size_t)cluster_threads(lr) * 8 <=
                               (size_t)num_sms * 2048 * 9;
}

template <int LR>
static void launch_fused(size_t nprod, bool spread, cudaStream_t s, const FusedArgs &a)
{
    // operands of at most half the transform (every tree level)
    if (std::max(a.a_len, a.b_len) <= (1u << LR))
        launch_fused_t<LR, true>(nprod, spread, s, a);
    else
        launch_fused_t<LR, false>(nprod, spread, s, a);
}

static void ntt_mul_small(Ctx &c, int np, size_t nprod, Operand x, Operand y, bool square,
                          const Sink &sink, cudaStream_t s)
{
    FusedArgs a;
    a.A = x.p;
    a.a_tstride = x.tstride;
    a.a_len = (uint32_t)x.len;
    a.B = y.p;  // squares are short and alone here: x twice
    a.b_tstride = y.tstride;
    a.b_len = (uint32_t)y.len;
    a.a_al = aligned8(x.p, x.tstride);
    a.b_al = aligned8(y.p, y.tstride);
    a.nprod = nprod;
    a.sink = sink;
    a.tw = c.twiddles;
    a.ca = make_coef(0, sink.dec);
    a.cb = make_coef(0, sink.dec, np);
    const bool spread = np >= kClusterMinLog && spread_primes(nprod, np, c.num_sms);
    const int tok = prof_begin(c, spread ? "ntt_mul_cluster" : "ntt_mul_fused", s);
    switch (np) {
    case 1: launch_fused<1>(nprod, spread, s, a); break;
    case 2: launch_fused<2>(nprod, spread, s, a); break;
    case 3: launch_fused<3>(nprod, spread, s, a); break;
    case 4: launch_fused<4>(nprod, spread, s, a); break;
    case 5: launch_fused<5>(nprod, spread, s, a); break;
    case 6: launch_fused<6>(nprod, spread, s, a); break;
    case 7: launch_fused<7>(nprod, spread, s, a); break;
    case 8: launch_fused<8>(nprod, spread, s, a); break;
    case 9: launch_fused<9>(nprod, spread, s, a); break;
    case 10: launch_fused<10>(nprod, spread, s, a); break;
    case 11: launch_fused<11>(nprod, spread, s, a); break;
    default: fail(CAT_EINVAL, "one-block transform size out of range");
    }
    CAT_LAUNCH(spread ? "ntt_mul_cluster" : "ntt_mul_fused");
    const double unit =
        4.0 * (double)nprod * (double)(x.len + (square ? 0 : y.len) + sink.out_len);
    prof_end(c, tok, s, unit, unit);
}

static int ceil_log2(size_t x)
{
    int n = 0;
    while (((size_t)1 << n) < x) n++;
    return n;
}

// log2 of the points of a product of `limbs` limbs: coefficients of two limbs,
// ceil(na / 2) + ceil(nb / 2) - 1 <= (na + nb) / 2 of them
static int points_log(size_t limbs) { return std::max(1, ceil_log2(limbs) - 1); }

// Level products of the fixed-slot product tree: nprod products of adjacent
// slot-limb nodes of `level`, each written into a 2*slot-limb slot of out.
void ntt_level(Ctx &c, const uint32_t *level, size_t slot, size_t nprod, uint32_t *out,
               cudaStream_t s, const uint32_t *out_index, const uint32_t *out_index_host)
{
    const int np = points_log(2 * slot);
    Operand x{level, slot, slot};
    if (np + 1 > c.max_log) {  // longer than one transform: each pair by pieces
        if (out_index && !out_index_host) fail(CAT_EINVAL, "indexed level needs its host table");
        for (size_t k = 0; k < nprod; k++) {
            uint32_t *o = out + 2 * (out_index ? (size_t)out_index_host[k] : k) * slot;
            CAT_CUDA(cudaMemsetAsync(o, 0, 8 * slot, s));
            mul_acc(c, level + 2 * k * slot, slot, level + (2 * k + 1) * slot, slot, o, 2 * slot,
                    false, s);
        }
        return;
    }
    Sink sink = plain_sink(out, 2 * slot, 2 * slot);
    sink.out_index = out_index;
    if (np <= kFusedMaxLog) {
        Operand a{level, 2 * slot, slot}, b{level + slot, 2 * slot, slot};
        ntt_mul_small(c, np, nprod, a, b, false, sink, s);
    } else {
        ntt_mul_multipass(c, np, PAIR_ADJACENT, nprod, x, x, sink, s);
    }
}

bool ntt_level_whole(const Ctx &c, size_t slot) { return points_log(2 * slot) + 1 <= c.max_log; }

void ntt_pair(Ctx &c, const uint32_t *pair, size_t slot, uint32_t *out, size_t len, cudaStream_t s)
{
    const int np = points_log(2 * slot);
    const Operand a{pair, 2 * slot, slot}, b{pair + slot, 2 * slot, slot};
    if (np <= kFusedMaxLog)
        ntt_mul_small(c, np, 1, a, b, false, plain_sink(out, 0, len), s);
    else
        ntt_mul_multipass(c, np, PAIR_FIRST_TWO, 1, a, b, plain_sink(out, 0, len), s);
}

// out[0 .. na+nb) = a * b by the transform (na + nb <= 2^27).
void ntt_mul(Ctx &c, const uint32_t *a, size_t na, const uint32_t *b, size_t nb,
             uint32_t *out, cudaStream_t s)
{
    const size_t len = na + nb;
    const int np = points_log(len);
    if (np > kLogMaxPts) fail(CAT_EINVAL, "operands too long for one transform");
    const bool square = (a == b && na == nb);
    Operand x{a, 0, na}, y{b, 0, nb};
    if (np <= kFusedMaxLog) {
        ntt_mul_small(c, np, 1, x, square ? x : y, square, plain_sink(out, 0, len), s);
    } else if (square) {
        ntt_mul_multipass(c, np, PAIR_SQUARE, 1, x, x, plain_sink(out, 0, len), s);
    } else {
        ntt_mul_multipass(c, np, PAIR_FIRST_TWO, 1, x, y, plain_sink(out, 0, len), s);
    }
}

// nprod products x_k y, x_k at x + k xstride (xlen limbs each), one y (ylen
// limbs), into `sink`; xlen + ylen <= 2^27.  y is transformed once.
void mul_broadcast(Ctx &c, const uint32_t *x, size_t xstride, size_t xlen, size_t nprod,
                   const uint32_t *y, size_t ylen, const Sink &sink, cudaStream_t s)
{
    if (nprod == 0) return;
    const int np = points_log(xlen + ylen);
    if (np > kLogMaxPts) fail(CAT_EINVAL, "operands too long for one transform");
    Operand ox{x, xstride, xlen}, oy{y, 0, ylen};
    if (nprod == 1 && x == y && xlen == ylen) {  // a square: one forward transform
        if (np <= kFusedMaxLog)
            ntt_mul_small(c, np, 1, ox, ox, true, sink, s);
        else
            ntt_mul_multipass(c, np, PAIR_SQUARE, 1, ox, ox, sink, s);
        return;
    }
    if (np <= kFusedMaxLog)
        ntt_mul_small(c, np, nprod, ox, oy, false, sink, s);
    else
        ntt_mul_multipass(c, np, PAIR_BROADCAST, nprod, ox, oy, sink, s);
}

// ------------------------------------------------ long products by pieces

// acc[j] += t[j] (t zero past tn) over one tile of 2048 limbs, carries within
// the tile; the tile's carry map goes to tile_maps.
__global__ void __launch_bounds__(kTileThreads) add_tiles(uint32_t *acc, size_t R,
                                                          const uint32_t *t, size_t tn, bool dec,
                                                          uint8_t *tile_maps)
{
    chain_wait();
    __shared__ uint32_t wsm[32];
    const size_t jt = (size_t)blockIdx.x * kTile;
    const int j0 = threadIdx.x * kLimbsPerThread;
    auto limb = [&](int i) -> uint64_t {
        const size_t j = jt + j0 + i;
        return j < tn ? t[j] : 0u;
    };
    const int tile_len = (int)(R - jt < (size_t)kTile ? R - jt : (size_t)kTile);
    uint32_t map;
    tile_carry<-1, 1>(limb, tile_len, acc + jt, tile_len, dec, acc + jt, tile_len, wsm, &map);
    if (threadIdx.x == 0) tile_maps[blockIdx.x] = (uint8_t)map;
}

// acc[0 .. R) += t[0 .. tn) in base 2^32 or (dec) 10^9, the carries carried
// through all of acc (the sum must fit R limbs; limbs of t past R are zero).
void add_into(Ctx &c, uint32_t *acc, size_t R, const uint32_t *t, size_t tn, bool dec,
              cudaStream_t s)
{
    if (R == 0 || tn == 0) return;
    const size_t tiles = (R + kTile - 1) / kTile;
    if (tiles > 0x7fffffffu) fail(CAT_EINVAL, "addition too long");
    DevBuf<uint8_t> maps(c, tiles, s);
    const int tok = prof_begin(c, "add_tiles", s);
    launch_chained(add_tiles, (unsigned)tiles, kTileThreads, 0, s, acc, R, t, tn, dec, maps.get());
    CAT_LAUNCH("add_tiles");
    prof_end(c, tok, s, 8.0 * (double)R + 4.0 * (double)tn);
    carry_finish(c, maps.get(), 1, tiles, Sink{acc, 0, R, dec, nullptr, 0, 0}, s);
}

// acc[0 .. R) += x y for operands of any length: pieces of Mx and My limbs
// with Mx + My <= 2^max_log, so that every piece product fits one transform,
// each added in at its offset (the sum must fit R limbs).  Both pieces are
// 2^(max_log - 1) limbs, or an operand shorter than that is one piece and the
// other takes the rest of the transform.
void mul_acc(Ctx &c, const uint32_t *x, size_t xlen, const uint32_t *y, size_t ylen,
             uint32_t *acc, size_t R, bool dec, cudaStream_t s)
{
    if (xlen == 0 || ylen == 0) return;
    const size_t L = (size_t)1 << c.max_log, M = L / 2;
    size_t Mx = M, My = M;
    if (xlen < M) {
        Mx = xlen;
        My = L - xlen;
    } else if (ylen < M) {
        My = ylen;
        Mx = L - ylen;
    }
    for (size_t i = 0; i < xlen; i += Mx)
        for (size_t j = 0; j < ylen; j += My) {
            if (i + j >= R) continue;
            const size_t lx = std::min(Mx, xlen - i), ly = std::min(My, ylen - j);
            DevBuf<uint32_t> t(c, lx + ly, s);
            mul_broadcast(c, x + i, 0, lx, 1, y + j, ly,
                          Sink{t.get(), 0, lx + ly, dec, nullptr, 0, 0}, s);
            add_into(c, acc + i + j, R - (i + j), t.get(), lx + ly, dec, s);
        }
}

// ------------------------------------------- unbalanced products by chunks

// The product of a long x (nx limbs) and a short y (ny limbs) from chunk
// products: chunk i = x[iM, iM + M) times y lies in slot i of T (M + ny
// words), and belongs at offset iM, so it overlaps the next chunk's product by
// ny limbs.  Limb j of the result sums t1 = slot k's word j - kM (k = j / M,
// the last slot also covers its tail) and t2 = slot k-1's word M + (j - kM)
// when j - kM < ny.
__device__ __forceinline__ uint64_t overlap_sum(const uint32_t *T, size_t M, size_t ny,
                                                size_t chunks, size_t j)
{
    size_t k = j / M;
    const bool past = k >= chunks;
    if (past) k = chunks - 1;
    const size_t r = j - k * M;
    const uint32_t t1 = r < M + ny ? T[k * (M + ny) + r] : 0u;
    const uint32_t t2 = (!past && k >= 1 && r < ny) ? T[(k - 1) * (M + ny) + M + r] : 0u;
    return (uint64_t)t1 + t2;
}

__global__ void __launch_bounds__(kTileThreads) overlap_tiles(const uint32_t *T, size_t M,
                                                              size_t ny, size_t chunks,
                                                              uint32_t *out, size_t R,
                                                              uint8_t *tile_maps)
{
    chain_wait();
    __shared__ uint32_t wsm[32];
    const size_t jt = (size_t)blockIdx.x * kTile;
    const size_t j0 = jt + threadIdx.x * kLimbsPerThread;
    auto limb = [&](int i) -> uint64_t {
        return j0 + i < R ? overlap_sum(T, M, ny, chunks, j0 + i) : 0u;
    };
    const int tile_len = (int)(R - jt < (size_t)kTile ? R - jt : (size_t)kTile);
    uint32_t map;
    tile_carry<0, 0>(limb, tile_len, out + jt, tile_len, false, nullptr, 0, wsm, &map);
    if (threadIdx.x == 0) tile_maps[blockIdx.x] = (uint8_t)map;
}

// The scratch of n broadcast products of 2^np points and `tiles` tile maps, as
// one block: false, with nothing taken, where a budget or the device has no
// room for it.
static bool take_scratch(Ctx &c, int np, size_t n, size_t tiles, MulScratch &m, cudaStream_t s)
{
    const size_t points = (size_t)kNumPrimes << np;
    try {
        m.Gb = DevBuf<uint32_t>(c, (2 * n + 1) * points + (tiles + 3) / 4, s);
    } catch (const Error &e) {
        if (e.code != CAT_ENOMEM) throw;
        return false;
    }
    m.F = m.Gb.get();
    m.G = m.F + (n + 1) * points;
    m.maps = reinterpret_cast<uint8_t *>(m.G + n * points);
    return true;
}

// out[0 .. nx + ny) = x y by chunks of M = 2^k - ny >= ny limbs of x, each
// multiplied by y in one batch (y transformed once).
//
// Transforms of 2^13 points or more sum the chunk products as residues (M
// rounded down to whole runs of four coefficients; at least ny still, 2^(k-1)
// being a multiple of 8 limbs and not below ny); the last chunk is shorter.
// The one-block and one-row products write limbs, which overlap_tiles adds; so
// do longer ones where there is no room for all chunks' residues at once (10
// bytes per limb of 2 n + 1 transforms: up to four chunks of which the last is
// short take less one after the other).  The room is taken, not asked for: a
// budget may be shared with other threads.
void mul_chunked(Ctx &c, const uint32_t *x, size_t nx, const uint32_t *y, size_t ny, int k,
                 uint32_t *out, cudaStream_t s)
{
    const size_t L = (size_t)1 << k, M = L - ny, slot = L;
    if (ny == 0 || M < ny) fail(CAT_EINVAL, "chunk size below the short operand");
    const size_t m = M & ~(size_t)7, n = (nx + m - 1) / m;
    MulScratch scratch;
    if (k - 1 > kRowMaxLog && take_scratch(c, k - 1, n, (nx + ny + kTile - 1) / kTile, scratch, s)) {
        Operand ox{x, m, m}, oy{y, 0, ny};
        ox.ragged = (unsigned)(n - 1);
        ox.ragged_len = nx - (n - 1) * m;
        ntt_mul_multipass(c, k - 1, PAIR_BROADCAST, n, ox, oy, plain_sink(out, 0, nx + ny), s,
                          std::move(scratch), (uint32_t)(m / 2));
        return;
    }
    const size_t full = nx / M, rem = nx - full * M, chunks = full + (rem ? 1 : 0);
    DevBuf<uint32_t> T(c, chunks * slot, s);
    if (full) mul_broadcast(c, x, M, M, full, y, ny, plain_sink(T.get(), slot, slot), s);
    if (rem) {
        uint32_t *last = T.get() + full * slot;
        CAT_CUDA(cudaMemsetAsync(last, 0, 4 * slot, s));
        mul_broadcast(c, x + full * M, 0, rem, 1, y, ny, plain_sink(last, 0, rem + ny), s);
    }
    const size_t R = nx + ny, tiles = (R + kTile - 1) / kTile;
    DevBuf<uint8_t> maps(c, tiles, s);
    const int tok = prof_begin(c, "overlap_tiles", s);
    launch_chained(overlap_tiles, (unsigned)tiles, kTileThreads, 0, s, T.get(), M, ny, chunks, out,
                   R, maps.get());
    CAT_LAUNCH("overlap_tiles");
    prof_end(c, tok, s, 4.0 * (double)(chunks * slot) + 4.0 * (double)R);
    carry_finish(c, maps.get(), 1, tiles, plain_sink(out, 0, R), s);
}

// --------------------------------------- multiplication without allocation
//
// For callers that must not allocate device memory: code running where
// cudaMalloc is not allowed or not wanted (inside a host callback, a caller
// that owns all device memory through its own arena, or a process whose
// allocator is already saturated).  The transform scratch and the twiddle
// tables of this variant live in file-scope __device__ arrays of fixed size,
// reserved when the library is loaded, on every device that loads it, until
// the process exits.  Products of up to kNoAllocMaxLimbs limbs fit.

constexpr int kNoAllocLog = 16;
constexpr size_t kNoAllocMaxLimbs = (size_t)1 << kNoAllocLog;   // na + nb limit
constexpr size_t kNoAllocN = kNoAllocMaxLimbs / 2;  // points
// words: F (5 primes x 2 transforms x N), G (5 x N), tile maps, top index
constexpr size_t kNoAllocF = 2 * kNumPrimes * kNoAllocN;
constexpr size_t kNoAllocG = kNumPrimes * kNoAllocN;
constexpr size_t kNoAllocMapWords = 64;
constexpr size_t kNoAllocWords = kNoAllocF + kNoAllocG + kNoAllocMapWords + 2;

static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocWords];
static __device__ __align__(256) uint2 g_noalloc_twiddles[kTwTotal];

// Largest i + 1 with x[i] != 0 into *top (which the caller clears).
__global__ void noalloc_top(const uint32_t *x, size_t n, unsigned long long *top)
{
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

struct NoAllocDevice {
    bool ready = false;
    uint32_t *scratch = nullptr;  // device address of g_noalloc_scratch
    uint2 *twiddles = nullptr;    // device address of g_noalloc_twiddles
};
static NoAllocDevice g_noalloc_dev[64];
static uint2 g_noalloc_tw_host[kTwTotal];

// Once per device, with that device current: resolve the device addresses of
// the two arrays and fill the twiddle table (same layout as the context's).
static std::mutex g_noalloc_mutex;

static int noalloc_setup(int dev)
{
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoAllocDevice &d = g_noalloc_dev[dev];
    if (d.ready) return CAT_OK;
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return CAT_ECUDA;
    d.scratch = (uint32_t *)p;
    if (cudaGetSymbolAddress(&p, g_noalloc_twiddles) != cudaSuccess) return CAT_ECUDA;
    d.twiddles = (uint2 *)p;
    try {
        twiddle_tables_host(g_noalloc_tw_host);
    } catch (...) {
        return CAT_ECUDA;
    }
    if (cudaMemcpyToSymbol(g_noalloc_twiddles, g_noalloc_tw_host, sizeof(g_noalloc_tw_host)) !=
        cudaSuccess)
        return CAT_ECUDA;
    try {
        upload_low_twiddles(g_noalloc_tw_host);
    } catch (...) {
        return CAT_ECUDA;
    }
    d.ready = true;
    return CAT_OK;
}

// The product through the same kernels as ntt_mul, with all scratch taken
// from the static array.
static void noalloc_mul(const NoAllocDevice &d, const uint32_t *a, size_t na, const uint32_t *b,
                        size_t nb, uint32_t *out, cudaStream_t s)
{
    Ctx local;  // no device resources: only the twiddle pointer is used
    local.twiddles = d.twiddles;
    local.col_tw_tables = false;  // the passes compute their twiddles: nothing allocated
    const size_t len = na + nb;
    const int np = points_log(len);
    Operand x{a, 0, na}, y{b, 0, nb};
    if (np <= kFusedMaxLog) {
        ntt_mul_small(local, np, 1, x, y, false, plain_sink(out, 0, len), s);
        return;
    }
    MulScratch m;
    m.F = d.scratch;
    m.G = d.scratch + kNoAllocF;
    m.maps = (uint8_t *)(d.scratch + kNoAllocF + kNoAllocG);
    ntt_mul_multipass(local, np, PAIR_FIRST_TWO, 1, x, y, plain_sink(out, 0, len), s, std::move(m));
}

}  // namespace cat

extern "C" int bigint_mul_noalloc(const uint32_t *a, size_t na, const uint32_t *b, size_t nb,
                                  uint32_t *out, size_t cap, size_t *out_len, void *stream)
{
    using namespace cat;
    if (!out_len || (na && !a) || (nb && !b) || (cap && !out)) return CAT_EINVAL;
    // beyond the static scratch (written so that na + nb cannot wrap around)
    if (na > kNoAllocMaxLimbs || nb > kNoAllocMaxLimbs - na) return CAT_ENOMEM;
    if (cap < na + nb) return CAT_ERANGE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return CAT_ECUDA;
    const int rc = noalloc_setup(dev);
    if (rc != CAT_OK) return rc;
    const NoAllocDevice &d = g_noalloc_dev[dev];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    try {
        if (na == 0 || nb == 0) {
            if (na + nb) CAT_CUDA(cudaMemsetAsync(out, 0, 4 * (na + nb), s));
            CAT_CUDA(cudaStreamSynchronize(s));
            *out_len = 0;
            return CAT_OK;
        }
        noalloc_mul(d, a, na, b, nb, out, s);
        unsigned long long *top = (unsigned long long *)(d.scratch + kNoAllocF + kNoAllocG +
                                                         kNoAllocMapWords);
        CAT_CUDA(cudaMemsetAsync(top, 0, sizeof(*top), s));
        noalloc_top<<<64, 256, 0, s>>>(out, na + nb, top);
        CAT_LAUNCH("noalloc_top");
        unsigned long long h = 0;
        CAT_CUDA(cudaMemcpyAsync(&h, top, sizeof(h), cudaMemcpyDeviceToHost, s));
        CAT_CUDA(cudaStreamSynchronize(s));
        *out_len = (size_t)h;
        return CAT_OK;
    } catch (const Error &e) {
        return e.code;
    } catch (...) {
        return CAT_ECUDA;
    }
}
