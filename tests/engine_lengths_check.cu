// engine_lengths_check.cu -- the line shapes of the lengths between powers of
// two and 3/2 of them (launch.h), through the driver of engine_host_check.cu.
//
// Built and run by tests/test_engine_lengths_host.py (host code only; no GPU).
// Prints one line per case: "<name> <max error / max |X|>".
#define main engine_host_check_main
#include "engine_host_check.cu"
#undef main

template <typename T>
static void check_more(const char *tag)
{
#define Y(L) check<T, YShape<T, L>, L>(tag, "y", L);
#define Z(L) check<T, ZShape<T, L>, L>(tag, "z", L + 1);
#define X(L)                                   \
    check<T, XShape<T, L>, L>(tag, "x", L + 2); \
    check<T, XShapeF<T, L>, L>(tag, "xf", L + 3);
    Y(144) Y(288) Y(576) Y(1152) Y(2048)
    Z(288) Z(576) Z(1152) Z(1536) Z(2048)
    X(144) X(288) X(576) X(1024)
    if (sizeof(T) == 4) {  // FP32 only
        Y(324) Y(432) Y(648) Y(1296)
        Z(324) Z(1296)
        X(162) X(324) X(648)
    } else {
        Z(144) X(72)
    }
}

int main()
{
    check_more<float>("f32");
    check_more<double>("f64");
    check_more<df64>("df64");
    // the FP64 lines of the spectrum build
    check<double, Shape<double, 324>, 324>("f64", "col", 1);
    check<double, Shape<double, 432>, 432>("f64", "col", 2);
    check<double, Shape<double, 648>, 648>("f64", "col", 3);
    check<double, Shape<double, 1296>, 1296>("f64", "col", 4);
    return 0;
}
