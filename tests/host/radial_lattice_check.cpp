// Host check of the closed forms on the grid's lattice (radial.h, Lattice) against the same forms in long
// double: prints, per lambda and N, the largest error of I(p, q) and J(n) in units of
// 2^-53 times the size of the terms the form subtracts, and how often I(0, q) is not J(q) to the bit.
#include <cmath>
#include <cstdio>

#include "../../paper_1211_0540_gb300/csrc/radial.h"

using LD = long double;
static const LD kPiL = 3.14159265358979323846264338327950288L;

int main() {
    using namespace bte::radial;
    const double L = 6.0, u = std::ldexp(1.0, -53);
    const LD z = kPiL / (2 * (LD)L);
    for (double lam : {0.0, 1.0})
        for (int N : {8, 16, 32, 48}) {
            const Lattice R{L, lam, 0.5 * (kPi / L)};
            auto C = [&](LD t, LD *size) {
                if (t == 0) return *size = lam == 0 ? (LD)L : (LD)L * L / 2;
                const LD k = z * t, s = std::sin(kPiL / 2 * t) / k, h = std::sin(kPiL / 4 * t);
                *size = lam == 0 ? 1 / std::fabs(k) : L / std::fabs(k) + 2 / (k * k);
                return lam == 0 ? s : L * s - 2 * h * h / (k * k);
            };
            double eI = 0, eJ = 0;
            int differ = 0;
            const int h = N / 2;
            for (int p = 0; p <= 3 * h * h; p += 1 + N / 16)
                for (int q = p & 1; q <= 3 * (N - 1) * (N - 1); q += 2 * (1 + N / 8)) {
                    if (p == 0 || q == 0) {
                        differ += R.I(p, q) != R.J(p + q);
                        continue;
                    }
                    const LD a = std::sqrt((LD)p), b = std::sqrt((LD)q), den = 2 * z * z * a * b;
                    LD s0, s1;
                    const LD I = (C((LD)(p - q) / (a + b), &s0) - C(a + b, &s1)) / den;  // a - b without cancellation
                    eI = std::fmax(eI, (double)(std::fabs(R.I(p, q) - I) / (u * (std::fabs(s0) + s1) / den)));
                }
            for (int n = 1; n <= 12 * h * h; n += 3) {
                const LD c = z * std::sqrt((LD)n), x = c * L, s = std::sin(x), co = std::cos(x);
                const LD J = lam == 0 ? (s - x * co) / (c * c * c) : (2 * x * s - (x * x - 2) * co - 2) / (c * c * c * c);
                const LD size = lam == 0 ? (1 + x) / (c * c * c) : (2 * x + x * x + 4) / (c * c * c * c);
                eJ = std::fmax(eJ, (double)(std::fabs(R.J(n) - J) / (u * size)));
            }
            std::printf("%g %d %.3f %.3f %d\n", lam, N, eI, eJ, differ);
        }
    return 0;
}
