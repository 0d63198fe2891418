// Host check of the FP64 gate table (csrc/mm_gate_table64.h): builds it for the
// given dt and, for every line "V m h n" on stdin, prints the three gates
// stepped with the table, and in long double, and with the rates evaluated
// directly in double.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "mm_gate_table64.h"

template <class T>
static T ratio(T x) { return x == 0 ? T(1) : x / std::expm1(x); }

template <class T>
static void direct(T V, T dt, const T x[3], T out[3])
{
    const T a[3] = {ratio<T>(-(V + 40) / 10), T(0.07L) * std::exp(-(V + 65) / 20), T(0.1L) * ratio<T>(-(V + 55) / 10)};
    const T b[3] = {4 * std::exp(-(V + 65) / 18), 1 / (1 + std::exp(-(V + 35) / 10)),
                    T(0.125L) * std::exp(-(V + 65) / 80)};
    for (int g = 0; g < 3; ++g) {
        const T s = a[g] + b[g], X = a[g] / s;
        out[g] = X + (x[g] - X) * std::exp(-dt * s);
    }
}

int main(int argc, char **argv)
{
    if (argc != 2) return 2;
    const double dt = std::atof(argv[1]);
    constexpr int I = mmg::kTab64Intervals;
    std::vector<mmg::Quad64> tab((size_t)mmg::kTab64Quads * I);
    mmg::build_table64(dt, tab.data());
    double V, x[3];
    while (std::scanf("%lf %lf %lf %lf", &V, &x[0], &x[1], &x[2]) == 4) {
        if (!mmg::in_table(V)) return 3;
        const mmg::Index64 t = mmg::index64(V);
        if (t.i < 0 || t.i >= I || !(std::fabs(t.u) <= 0.5)) return 4;
        for (int g = 0; g < 3; ++g) {
            double XD[2];
            for (int k = 0; k < 2; ++k) {
                const mmg::Quad64 *f = tab.data() + (size_t)(3 * (2 * g + k)) * I + t.i;
                mmg::Quad32 s;
                std::memcpy(&s, f + 2 * I, 16);
                XD[k] = k == 0 ? mmg::eval64_rest(f[0], f[I], s, t) : mmg::eval64(f[0], f[I], s, t);
            }
            std::printf("%.17g ", mmg::step64(x[g], XD[0], XD[1]));
        }
        long double xl[3] = {x[0], x[1], x[2]}, ol[3];
        double od[3];
        direct<long double>(V, dt, xl, ol);
        direct<double>(V, dt, x, od);
        for (int g = 0; g < 3; ++g) std::printf("%.21Lg ", ol[g]);
        for (int g = 0; g < 3; ++g) std::printf("%.17g ", od[g]);
        std::printf("\n");
    }
    return 0;
}
