// mean_of_sum<2> (csrc/element_mean.h) against the division by three, bit for bit: the given number of random
// bit patterns (every exponent, subnormal, infinite and NaN ones among them), every exponent's values around its
// power of two and around one and a half times it, and the largest values. Prints the number of differences.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <random>

#include "element_mean.h"

static long bad = 0;
static void check(double s) {
    for (double v : {s, -s}) {
        const volatile double three = 3.0;
        const double a = knp::mean_of_sum<2>(v), b = v / three;
        if (b != b ? a == a : std::memcmp(&a, &b, sizeof a) != 0) {
            if (bad++ < 5) std::printf("%a: %a, not %a\n", v, a, b);
        }
    }
}

int main(int, char** argv) {
    std::mt19937_64 rng(std::strtoull(argv[2], nullptr, 10));
    for (long n = std::atol(argv[1]); n > 0; --n) {
        const uint64_t bits = rng();
        double s;
        std::memcpy(&s, &bits, sizeof s);
        check(s);
    }
    for (uint64_t e = 0; e <= 0x7ff; ++e)
        for (uint64_t m : {uint64_t(0), uint64_t(1) << 51})
            for (int64_t d = -64; d <= 64; ++d) {
                const uint64_t bits = ((e << 52) | m) + (uint64_t)d;
                double s;
                std::memcpy(&s, &bits, sizeof s);
                check(s);
            }
    check(0.0);
    check(std::numeric_limits<double>::infinity());
    check(std::numeric_limits<double>::max());
    std::printf("%ld\n", bad);
}
