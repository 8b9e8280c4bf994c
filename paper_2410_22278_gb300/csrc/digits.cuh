// Balanced 8-bit digits of the split-precision operands (ozaki.cu): an integer
// V, |V| < 2^62, as sum_{s < S} d_s 2^{55 - 8s} plus a rest of at most half of
// the last place, d_s in [-128, 128].  Two forms of the same sum:
//   * for operands read through all S digits (the structure factors and the
//     products with the density, cut for every G): with
//     W = V + digit_offset(S) the digits are plain bits of W,
//     d_0 = W >> 55 and d_s = byte s of W - 128;
//   * for operands cut once and read through fewer digits too (the density and
//     its factor): every prefix is V rounded to nearest, d_s = P_s - 256
//     P_{s-1} with P_s = round(V / 2^{55 - 8s}).
// An offset that always held the half places of seven digits left up to 0.502
// of the last place after fewer, and 0.002 of it on average: a bias in every
// element.
#pragma once

namespace jk {

__host__ __device__ constexpr long long digit_offset(int S)
{
    long long b = 1LL << (62 - 8 * S);  // half of the last place
    for (int s = 1; s < S; ++s) b += 128LL << (55 - 8 * s);
    return b;
}
__host__ __device__ inline int digit_top(long long W) { return (int)(W >> 55); }
__host__ __device__ inline unsigned digit_byte(long long W, int s) { return (unsigned)(W >> (55 - 8 * s)) & 255u; }
// the low 32 bits of P_s
__host__ __device__ inline unsigned digit_prefix(long long V, int s) { return (unsigned)((V + (1LL << (54 - 8 * s))) >> (55 - 8 * s)); }

}  // namespace jk
