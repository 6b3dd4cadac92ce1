// Host check of div_int (fp64_math.cuh) against the division operator, over
// significands that reach its digit bounds: random, short, all ones, near
// ties and exact quotients, operands next to one another, and the special
// values. argv[1]: pairs. SVM_DIV_SEED_ULP moves the reciprocal's FP32 seed by
// so many units of its last place (the device's seed is approximate).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "fp64_math.cuh"

using namespace svmgb;

int main(int argc, char **argv)
{
    const long n = argc > 1 ? atol(argv[1]) : 1000000;
    std::mt19937_64 g(5);
    long bad = 0;
    auto check = [&](double a, double b) {
        const double want = a / b, got = div_int(a, b);
        if (double_to_bits(want) == double_to_bits(got) || (std::isnan(want) && std::isnan(got))) return;
        if (++bad < 5) printf("%a / %a = %a, got %a\n", a, b, want, got);
    };
    auto make = [&](uint64_t m, int e) { return bits_to_double(((uint64_t)e << 52) | (m & 0xfffffffffffffull)); };
    for (long i = 0; i < n; ++i) {
        uint64_t a = g(), b = g();
        switch (i % 8) {
        case 1: b &= 0xffffffff00000ull; break;
        case 2: b &= 0xff; break;
        case 3: a &= 0xfffff; break;
        case 4: b |= 0xfffffffffff00ull; break;
        case 5: a |= 0xffffffffff000ull; break;
        case 6: b = a + g() % 16 - 8; break;
        case 7: {   // a rounded product over one factor: exact quotients and near ties
            const double q = make(g(), 1023), d = make(g() & (i & 8 ? ~0ull : 0xfffffff000000ull), 1023);
            check(q * d, d);
            continue;
        }
        default: break;
        }
        check(make(a, 1000 + (int)(a >> 58)), make(b, 1000 + (int)(b >> 58)));
        check(bits_to_double(g()), bits_to_double(g()));
    }
    const double sp[] = {0.0, -0.0, 1.0, 2.0, 1e-12, 1.5, 3.0, 5e-324, 1e-308, 2.2250738585072014e-308,
                         1.7976931348623157e308, INFINITY, NAN, -1.0, -7e-300, 9e299};
    for (double a : sp)
        for (double b : sp) check(a, b);
    printf("bad %ld\n", bad);
    return bad != 0;
}
