// df64_rounding_check.cu -- the float-pair radix 3 and the product with the
// spectrum (fft_engine.cuh) on the CPU: the radix 3 against its definition in
// normalised float-pair arithmetic (operators of df64.cuh), on normalised and
// lazily summed inputs of random magnitudes; the product for results that are
// normalised (adding the parts again changes neither).
// Built and run by tests/test_df64_rounding_host.py.  Prints, for each, the
// number of values and of those that fail.
#include <math.h>
#include <stdio.h>

#include "fft_engine.cuh"

using namespace isofft;

static uint64_t s_state = 88172645463325252ull;
static double rnd()  // uniform in [-1, 1), times a power of two of 2^-20 to 2^20
{
    s_state ^= s_state << 13;
    s_state ^= s_state >> 7;
    s_state ^= s_state << 17;
    return ldexp((double)(int64_t)s_state, -63 + (int)(s_state % 41) - 20);
}
static df64 value(bool lazy) { return lazy ? df64_add_lazy(df64_add_lazy(df64(rnd()), df64(rnd())), df64(rnd())) : df64(rnd()); }
static Cx<df64> norm(Cx<df64> v) { return {df64_renorm(v.x), df64_renorm(v.y)}; }

int main()
{
    const df64 s3(0.8660254037844387), half(0.5);
    long n = 0, bad = 0;
    for (long i = 0; i < 1000000; ++i) {
        Cx<df64> a[3], b[3];
        for (int j = 0; j < 3; ++j) a[j] = {value(i & 1), value(i & 1)};
        const Cx<df64> sum = norm(cadd(a[1], a[2])), dif = norm(csub(a[1], a[2]));
        const Cx<df64> t = {a[0].x - half * sum.x, a[0].y - half * sum.y}, u = {dif.y * s3, -(dif.x * s3)};
        b[0] = cadd(a[0], sum);
        b[1] = cadd(t, u);
        b[2] = csub(t, u);
        Dft<df64, 3>::run(a);
        for (int j = 0; j < 3; ++j) {
            const df64 got[2] = {a[j].x, a[j].y}, want[2] = {b[j].x, b[j].y};
            for (int c = 0; c < 2; ++c, ++n) bad += got[c].hi != want[c].hi || got[c].lo != want[c].lo;
        }
    }
    printf("radix3 %ld %ld\n", n, bad);
    n = bad = 0;
    for (long i = 0; i < 1000000; ++i) {
        const Cx<df64> v = cscale(Cx<df64>{df64(rnd()), df64(rnd())}, df64(rnd()));
        const Cx<df64> w = norm(v);
        n += 2;
        bad += v.x.hi != w.x.hi || v.x.lo != w.x.lo;
        bad += v.y.hi != w.y.hi || v.y.lo != w.y.lo;
    }
    printf("product %ld %ld\n", n, bad);
    return 0;
}
