// length_bits.h -- length bounds of products from the operands' bits (host
// arithmetic only): a number is tracked by `bits` with value <= 2^bits, so that
// a chain of products needs no read-back of the lengths between.
#pragma once

#include <math.h>
#include <stddef.h>
#include <stdint.h>

namespace cat {

// More than x by 2^-40 of it: above every rounding (2^-53 each) of the
// operations below, so that a bound stays one for any length; the 128 steps of
// a power with a 64-bit exponent widen it by 2^-33 in all, less than a limb up
// to 2^38 bits.
inline double widened(double x) { return x * (1.0 + 0x1p-40); }

// Bits of a number of n limbs whose highest limb and the one below it (0 for
// n = 1) are the high and the low word of top.  0 for the value 1, whose powers
// then keep their one limb.
inline double top_bits(uint64_t n, uint64_t top)
{
    if (n == 0 || (n == 1 && top == (uint64_t)1 << 32)) return 0;
    if (n == 1) return widened(log2((double)(top >> 32)));
    // the value is below 2^(32 (n - 2)) (top + 1), and top + 1 adds less than
    // 1e-9 bits to top's 33 or more
    return widened(32.0 * (double)(n - 2) + log2((double)top) + 1e-9);
}

// Bits of a product.
inline double product_bits(double x, double y) { return widened(x + y); }

// Limbs that hold every number of at most 2^bits.
inline size_t bits_limbs(double bits) { return (size_t)(bits / 32.0) + 1; }

}  // namespace cat
