// inv_sqrt_check.cu -- inv_sqrt (inv_sqrt.cuh) on the device against 1 / sqrt in
// long double: random mantissas over every exponent of the float range and past
// it, powers of two, squares, and both sides of the range's ends.  Built and run
// by tests/test_gpu_inv_sqrt.py.  Prints the number of values and the largest
// error in units of the last place, inside the float range and outside.
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "inv_sqrt.cuh"

static __global__ void k_check(const double *x, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = isofft::inv_sqrt(x[i]);
}

int main()
{
    std::vector<double> x;
    uint64_t s = 88172645463325252ull;
    auto mant = [&]() {
        s ^= s << 13;
        s ^= s >> 7;
        s ^= s << 17;
        return 1.0 + ldexp((double)(s >> 12), -52);
    };
    for (int e = -300; e <= 300; ++e) {
        for (int i = 0; i < 3000; ++i) x.push_back(ldexp(mant(), e));
        const double p = ldexp(1.0, e);
        x.insert(x.end(), {p, nextafter(p, 0.0), nextafter(p, 2 * p)});
    }
    for (int i = 1; i < 3000; ++i) x.push_back((double)i * i);
    for (double end : {1e-37, 1e37}) {
        double lo = end, hi = end;
        for (int i = 0; i < 64; ++i) {
            x.insert(x.end(), {lo, hi});
            lo = nextafter(lo, 0.0);
            hi = nextafter(hi, 2 * end);
        }
    }
    const int n = (int)x.size();
    std::vector<double> y(n);
    double *dx = nullptr, *dy = nullptr;
    if (cudaMalloc(&dx, n * sizeof(double)) || cudaMalloc(&dy, n * sizeof(double))) return 1;
    cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    k_check<<<(n + 255) / 256, 256>>>(dx, dy, n);
    if (cudaMemcpy(y.data(), dy, n * sizeof(double), cudaMemcpyDeviceToHost)) return 1;
    long double worst[2] = {0, 0};
    for (int i = 0; i < n; ++i) {
        const long double want = 1.0L / sqrtl((long double)x[i]);
        int e;
        frexpl(want, &e);
        const long double ulps = fabsl((long double)y[i] - want) / ldexpl(1.0L, e - 53);
        const int out = !(x[i] < 1e37 && x[i] > 1e-37);
        if (!(ulps <= worst[out])) worst[out] = ulps;
    }
    printf("%d %.4Lf %.4Lf\n", n, worst[0], worst[1]);
    return 0;
}
