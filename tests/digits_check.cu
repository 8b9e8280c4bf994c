// Host-side check of the balanced digits of the split-precision operands
// (digits.cuh): the same __host__ __device__ functions the slicing kernels run,
// over random V of every magnitude and every S.  Prints the values whose S
// digits do not sum to V rounded to the nearest multiple of the last place
// (ties upwards), for the form read through all S digits and for every prefix
// of the form read through fewer, and the number of digits out of range.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../paper_2410_22278_gb300/csrc/digits.cuh"

using namespace jk;

int main()
{
    std::mt19937_64 rng(2410);
    long long wrong = 0, wrong_prefix = 0, range = 0;
    for (int S = 1; S <= 7; ++S) {
        const int shift = 55 - 8 * (S - 1);
        for (int i = 0; i < 1000000; ++i) {
            const int drop = 2 + (int)(rng() % 20);
            long long V = i < 2 ? (1LL << 62) - 1 : (long long)(rng() >> drop);
            if (rng() & 1) V = -V;
            const long long W = V + digit_offset(S), want = ((V + (1LL << (shift - 1))) >> shift) * (1LL << shift);
            long long sum = 0, sum_prefix = 0;
            unsigned p = 0;
            for (int s = 0; s < S; ++s) {
                const int d = s == 0 ? digit_top(W) : (int)digit_byte(W, s) - 128;
                const unsigned q = digit_prefix(V, s);
                const int e = (int)(q - 256u * p);
                p = q;
                range += std::abs(d) > 128 || std::abs(e) > 128;
                sum += (long long)d * (1LL << (55 - 8 * s));
                sum_prefix += (long long)e * (1LL << (55 - 8 * s));
            }
            wrong += sum != want;
            wrong_prefix += sum_prefix != want;
        }
    }
    std::printf("%lld %lld %lld\n", wrong, wrong_prefix, range);
}
