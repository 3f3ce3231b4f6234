// df64_convert_check.cu -- df64_split (df64.cuh) on the CPU against the
// conversion by FP64 arithmetic, over random values, powers of two, ties,
// the edges of the integer form's range, zeros, denormals, infinities and NaN.
// Built and run by tests/test_df64_convert_host.py.  Prints the number of
// values and of mismatches.
#include <stdio.h>

#include "df64.cuh"

using namespace isofft;

static uint64_t s_state = 88172645463325252ull;
static uint64_t rnd()
{
    s_state ^= s_state << 13;
    s_state ^= s_state >> 7;
    s_state ^= s_state << 17;
    return s_state;
}
static long n_values = 0, n_bad = 0;
static bool same(double a, double b) { return f64_bits(a) == f64_bits(b) || (a != a && b != b); }

static void one(double d)
{
    ++n_values;
    const df64 want(d), got = df64_split(d);
    const bool tie = ((uint32_t)f64_bits(d) & 0x1fffffffu) == 0x10000000u;
    bool ok = tie && fabs(d) < 1e38 && fabs(d) > 1e-25 ? (double)got.hi + (double)got.lo == d
                  : same(want.hi, got.hi) && (same(want.lo, got.lo) || (want.lo == 0 && got.lo == 0));
    if (!ok && ++n_bad <= 5) fprintf(stderr, "%a: (%a, %a) want (%a, %a)\n", d, got.hi, got.lo, want.hi, want.lo);
}

int main()
{
    for (long i = 0; i < 4000000; ++i) {
        const uint64_t b = rnd();
        one(f64_of(b));                                                          // any bit pattern
        one(f64_of((b & 0x800fffffffffffffull) | (uint64_t)(900 + b % 300) << 52));  // around the range
        if (i % 64 == 0) {
            const uint64_t e = (uint64_t)(940 + (b >> 40) % 220) << 52, sg = b & 0x8000000000000000ull;
            one(f64_of(sg | e));                            // powers of two and their neighbours
            one(f64_of((sg | e) - 1));
            one(f64_of((sg | e) + 1));
            one(f64_of(sg | e | (b & 0xfffffe0000000ull) | 0x10000000ull));  // ties
            one(f64_of(sg | e | 0xfffffffffffffull));       // rounds up into the next binade
            one(f64_of(sg | e | 0xffffff0000000ull));
        }
    }
    const double special[] = {0.0, -0.0, 1.0 / 0.0, -1.0 / 0.0, 0.0 / 0.0, 4.9e-324, 1e-310, 3.4e38, 1.7e308, 1e-38, -1e-45};
    for (double d : special) one(d);
    printf("%ld %ld\n", n_values, n_bad);
    return 0;
}
