// Host check of the half-spectrum convolution's index rules (bte_internal.h):
// for a random real f and weights of the lattice invariants, the sums over the
// stored pencils' blocks, in the order of pair_visit, against the plain sum over
// every mode with zero extension, after the real part of the inverse transform.
// Prints one line per N: N max|difference| / max|Q|, N <= 12. For every N, counts
// the pairs that the visits miss, repeat, or give two different invariants
// (0 expected), and the m3 of a k3 that are not one run mod N.
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <set>
#include <vector>

#include "../../paper_1211_0540_gb300/csrc/bte_internal.h"

using namespace bte;
using cd = std::complex<double>;

struct Inv {
    int p = 0, q = 0, s = 0;
    void add(int k, int m, int N) {  // one dimension's part for the index pair (k, m) on the mesh
        const int a = k - N / 2, b = m - N / 2;
        p += a * a;
        q += (2 * b - a) * (2 * b - a);
        s += b * b;
    }
};
static double weight(const Inv &v) { return std::cos(0.31 * v.p) + std::sin(0.17 * v.q + 0.05) - 0.4 * std::cos(0.23 * v.s); }

static bool on3(const int k[3], const int m[3], int N) {
    return pair_on_grid(k[0], m[0], N) && pair_on_grid(k[1], m[1], N) && pair_on_grid(k[2], m[2], N);
}
static double half(const int k[3], const int m[3], int N) {
    int ks[3], ms[3];
    Inv a, b;
    for (int d = 0; d < 3; ++d) {
        ks[d] = mode_mirror(k[d], N);
        ms[d] = mode_mirror(m[d], N);
        a.add(k[d], m[d], N);
        b.add(ks[d], ms[d], N);
    }
    return ((on3(k, m, N) ? weight(a) : 0.0) + (on3(ks, ms, N) ? weight(b) : 0.0)) *
           (pencil_self_mirrored(k[0], k[1], N) ? 0.5 : 1.0);
}

static std::vector<double> inverse(const std::vector<cd> &Q, int N) {
    const double w = 2 * 3.14159265358979323846 / N;
    const int h = N / 2, M = N * N * N;
    std::vector<cd> a = Q, b(M);
    int st[3] = {1, N, N * N};
    for (int d = 0; d < 3; ++d) {
        for (int i = 0; i < M; ++i) {
            const int j = (i / st[d]) % N, base = i - j * st[d];
            cd s = 0;
            for (int k = 0; k < N; ++k) s += a[base + k * st[d]] * std::polar(1.0, w * (k - h) * (j - h));
            b[i] = s;
        }
        a.swap(b);
    }
    std::vector<double> r(M);
    for (int i = 0; i < M; ++i) r[i] = a[i].real();
    return r;
}

static void sums(int N) {
    const int h = N / 2, M = N * N * N, T = N;
    std::mt19937 g(N);
    std::uniform_real_distribution<double> u(0, 1);
    std::vector<cd> x(M), fh(M), Q1(M), Q2(M);
    for (auto &v : x) v = u(g);
    std::vector<cd> a = x, b(M);
    int st[3] = {1, N, N * N};
    for (int d = 0; d < 3; ++d) {
        for (int i = 0; i < M; ++i) {
            const int k = (i / st[d]) % N, base = i - k * st[d];
            cd s = 0;
            for (int j = 0; j < N; ++j)
                s += a[base + j * st[d]] * std::polar(1.0, -2 * 3.14159265358979323846 / N * (k - h) * (j - h));
            b[i] = s;
        }
        a.swap(b);
    }
    fh = a;
    for (int k = 0; k < M; ++k) {  // the plain sum
        const int kk[3] = {k / (N * N), (k / N) % N, k % N};
        for (int m = 0; m < M; ++m) {
            const int mm[3] = {m / (N * N), (m / N) % N, m % N};
            if (!on3(kk, mm, N)) continue;
            Inv v;
            for (int d = 0; d < 3; ++d) v.add(kk[d], mm[d], N);
            Q1[k] += weight(v) * fh[m] * fh[((kk[0] - mm[0] + h) * N + kk[1] - mm[1] + h) * N + kk[2] - mm[2] + h];
        }
    }
    for (int k1 = 0; k1 < N; ++k1)
        for (int k2 = 0; k2 < N; ++k2) {
            if (!pencil_stored(k1, k2, N)) continue;
            for (int m1 = 0; m1 < N; ++m1)
                for (int m2 = 0; m2 < N; ++m2) {
                    const int n1 = pair_partner(k1, m1, N), n2 = pair_partner(k2, m2, N);
                    if (m1 > n1 || (m1 == n1 && m2 > n2)) continue;
                    for (int i = 0; i < pair_visits(N, T); ++i)
                        for (int k3 = 0; k3 < N; ++k3) {
                            const int m3 = i % N, n3 = pair_partner(k3, m3, N);
                            if (!pair_visit(k3, i, N, T)) continue;
                            const int k[3] = {k1, k2, k3}, m[3] = {m1, m2, m3}, n[3] = {n1, n2, n3};
                            double w = half(k, m, N);
                            if (m1 != n1 || m2 != n2) w += half(k, n, N);
                            Q2[(k1 * N + k2) * N + k3] += w * fh[(m1 * N + m2) * N + m3] * fh[(n1 * N + n2) * N + n3];
                        }
                }
        }
    const auto r1 = inverse(Q1, N), r2 = inverse(Q2, N);
    double e = 0, mag = 0;
    for (int i = 0; i < M; ++i) {
        e = std::fmax(e, std::fabs(r1[i] - r2[i]));
        mag = std::fmax(mag, std::fabs(r1[i]));
    }
    std::printf("sum %d %.3e\n", N, e / mag);
}

static void rules(int N, int T) {
    int bad = 0;
    for (int k = 0; k < N; ++k) {
        std::multiset<int> seen;
        for (int i = 0; i < pair_visits(N, T); ++i)
            if (pair_visit(k, i, N, T)) seen.insert(i % N);
        int runs = 0, kept = 0;
        for (int m = 0; m < N; ++m) {
            const int n = pair_partner(k, m, N);
            kept += pair_kept(k, m, N);
            bad += (int)seen.count(m) != (pair_kept(k, m, N) ? 1 : 0);
            bad += pair_kept(k, m, N) != pair_kept(k, n, N) || pair_partner(k, n, N) != m;
            runs += pair_kept(k, m, N) && !pair_kept(k, (m + N - 1) % N, N);
            if (pair_on_grid(k, m, N) && pair_on_grid_mirrored(k, m, N)) {
                Inv a, b;
                a.add(k, m, N);
                b.add(mode_mirror(k, N), mode_mirror(m, N), N);
                bad += a.p != b.p || a.q != b.q || a.s != b.s;
            }
        }
        bad += runs != (kept == N ? 0 : 1);
        for (int k1 = 0; k1 < N; ++k1)  // one pencil of each mirror pair, self-mirrored ones once
            bad += pencil_stored(k, k1, N) + pencil_stored(mode_mirror(k, N), mode_mirror(k1, N), N) !=
                   (pencil_self_mirrored(k, k1, N) ? 2 : 1);
    }
    std::printf("rules %d %d\n", N, bad);
}

int main() {
    sums(8);
    sums(12);
    rules(8, 8);
    rules(12, 12);
    rules(16, 16);
    rules(24, 12);
    rules(32, 16);
    rules(48, 16);
    return 0;
}
