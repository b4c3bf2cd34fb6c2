// log_tab (csrc/log_tab.cuh) on the host, against the long double logarithm:
// prints the largest error in units of the last place over each range, then
// the results for the arguments that it hands to log().  Test infrastructure;
// built by tests/test_log_tab.py.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>

#define __device__
#define __forceinline__ inline
#define __ldg(p) (*(p))
static int64_t bits(double x) {
    int64_t b;
    std::memcpy(&b, &x, 8);
    return b;
}
static int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static int __double2loint(double x) { return (int)bits(x); }
static double __hiloint2double(int hi, int lo) {
    const int64_t b = (int64_t)((uint64_t)(uint32_t)hi << 32 | (uint32_t)lo);
    double x;
    std::memcpy(&x, &b, 8);
    return x;
}
using std::fma;
using std::log;
#include "../paper_1307_2666_gb300/csrc/log_tab.cuh"

static double ulps(double x) {
    const long double e = std::log((long double)x);
    const double y = hif::log_tab(x), s = std::fabs((double)e);
    if (e == 0.0L) return y == 0.0 ? 0.0 : 1e30;
    return (double)(std::fabs((long double)y - e) / (long double)(std::nextafter(s, 1e300) - s));
}

int main() {
    std::mt19937_64 gen(5);
    const double lo[] = {0.98, 0.996, 0.5, 1e-12, 1e-300, 1.0 - 1e-6}, hi[] = {1.02, 1.008, 2.0, 1e12, 1e300, 1.0 + 1e-6};
    for (int q = 0; q < 6; ++q) {
        std::uniform_real_distribution<double> u(std::log(lo[q]), std::log(hi[q]));
        double worst = ulps(0.99803960884952103);
        for (int i = 0; i < 400000; ++i) worst = std::fmax(worst, ulps(std::exp(u(gen))));
        std::printf("%.4f ", worst);
    }
    double worst = 0.0;                               // both sides of every switch of the table's rows
    for (int i = 0; i <= 1024; ++i)
        for (double x = 1.0 + i / 1024.0, k = -8; k <= 8; ++k)
            for (int e = -2; e <= 1; ++e) worst = std::fmax(worst, ulps(std::ldexp(x + k * 0x1p-52, e)));
    std::printf("%.4f\n", worst);
    const double inf = std::numeric_limits<double>::infinity(), sub = 4.9e-324;
    std::printf("%d %d %d %d %d\n", hif::log_tab(0.0) == -inf, hif::log_tab(inf) == inf, std::isnan(hif::log_tab(-1.0)),
                std::isnan(hif::log_tab(std::nan(""))), hif::log_tab(sub) == std::log(sub));
    return 0;
}
