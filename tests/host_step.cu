// Host check (no GPU) of the packed header functions the step's kernels call.
//  1. to_modes, moments and from_modes on pairs, the two components different:
//     unit populations of every direction give the columns of the transform,
//     exactly, unit modes w_i times its rows; random populations return.
//  2. load_force: 36 w_i c_i for a unit density at neighbour i, exactly.
//  3. noise_unit(k)^2 bnorm(k) = 1.
//  4. one_to_two: the angle's fraction (w >> 9) 2^-23, exactly.
//  5. DensitySink: the pair's put leaves what the single values' do.
//  6. SphereTest decides as node_inside does, for nodes at distance
//     R (1 + e), e from 1e-16 to 1, on axes of 8 to 2^20 nodes, across
//     periodic wraps and beside walls, with most nodes decided in float.
//  7. pop_sums: populations of sizes 2^-30 to 1, either sign, to 19 roundings of
//     FP64 of their magnitudes.
//  8. from_modes of random densities: the mean relative error of f_0 vanishes
//     (its roundings average out to 3e-10 over the 20000: 2e-9 allowed), those of
//     the others are within 2^-26.
// Prints one line and returns 0 when all hold.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "flbm_fused.cuh"
#include "flbm_host.cuh"

using namespace flbm;

struct UnitPsi {
    int at;
    float a, b;
    __host__ __device__ Pair psi(int i) const { return i == at ? Pair{b, a} : splat(0.0f); }
};

static double w_of(int i) { return i == 0 ? 1.0 / 3 : (i < 7 ? 1.0 / 18 : 1.0 / 36); }

int main()
{
    int failed = 0;
    std::mt19937_64 g(0x5eedu);
    std::uniform_real_distribution<float> U(0.0f, 0.2f);

    // 1. E[k][i] from the FP64 transform of the observables.
    double E[19][19];
    for (int i = 0; i < 19; ++i) {
        double f[19] = {0}, m[19];
        f[i] = 1.0;
        to_modes(f, m);
        for (int k = 0; k < 19; ++k) E[k][i] = m[k];
    }
    for (int i = 0; i < 19; ++i) {
        const int q = (i + 7) % 19;  // the other component's direction
        Pair f[19], m[19], rho, j[3];
        for (int d = 0; d < 19; ++d) f[d] = Pair{d == i ? 1.0f : 0.0f, d == q ? 3.0f : 0.0f};
        to_modes(f, m);
        for (int k = 0; k < 19; ++k) failed += (double)m[k].x != E[k][i] || (double)m[k].y != 3.0 * E[k][q];
        moments(f, rho, j);
        failed += rho.x != 1.0f || rho.y != 3.0f;
        for (int a = 0; a < 3; ++a) failed += (double)j[a].x != E[1 + a][i] || (double)j[a].y != 3.0 * E[1 + a][q];
        Pair n[19], o[19];
        for (int k = 0; k < 19; ++k) n[k] = Pair{k == i ? 1.0f : 0.0f, k == q ? 1.0f : 0.0f};
        from_modes(n, o);
        for (int d = 0; d < 19; ++d) {
            failed += std::fabs(o[d].x - w_of(d) * E[i][d]) > 1e-7 * std::fabs(w_of(d) * E[i][d]) + 1e-9;
            failed += std::fabs(o[d].y - w_of(d) * E[q][d]) > 1e-7 * std::fabs(w_of(d) * E[q][d]) + 1e-9;
        }
    }
    for (int t = 0; t < 5000; ++t) {
        Pair f[19], m[19], o[19];
        for (int i = 0; i < 19; ++i) f[i] = Pair{U(g), U(g)};
        to_modes(f, m);
        for (int k = 0; k < 19; ++k) m[k] = Pair{m[k].x / bnorm(k), m[k].y / bnorm(k)};
        from_modes(m, o);
        for (int i = 0; i < 19; ++i) failed += std::fabs(o[i].x - f[i].x) > 2e-6f || std::fabs(o[i].y - f[i].y) > 2e-6f;
    }

    // 2.
    for (int i = 1; i < 19; ++i) {
        NodeState<true> s;
        load_force(UnitPsi{i, 5.0f, 1.0f}, s);
        const int c[3] = {cxv(i), cyv(i), czv(i)};
        for (int a = 0; a < 3; ++a) {
            const float want = (i < 7 ? 2.0f : 1.0f) * (float)c[a];
            failed += s.g[a].x != want || s.g[a].y != 5.0f * want;
        }
    }

    // 3.
    for (int k = 4; k < 19; ++k) failed += std::fabs((double)noise_unit(k) * noise_unit(k) * bnorm(k) - 1.0) > 3e-7;

    // 4.
    for (int t = 0; t < 20000; ++t) {
        const uint32_t w = t < 4 ? (uint32_t)t * 0x55555555u : (uint32_t)g();
        failed += (double)(one_to_two(w) - 1.0f) != (double)(w >> 9) / 8388608.0;
    }

    // 5.
    for (int t = 0; t < 2000; ++t) {
        const int size = 4 + (int)(g() % 300), pos = (int)(g() % (unsigned)size);
        std::vector<float2> a((size_t)kXchDirs * size, make_float2(0.f, 0.f)), b = a;
        DensitySink sa(reinterpret_cast<float*>(a.data()), pos, size), sb(reinterpret_cast<float*>(b.data()), pos, size);
        for (int i = 0; i < 19; ++i) {
            const Pair v{U(g), U(g)};
            const bool bounced = g() % 4 == 0;
            sa.put(i, v, bounced);
            sb.put(0, i, v.x, bounced);
            sb.put(1, i, v.y, bounced);
        }
        for (size_t q = 0; q < a.size(); ++q) failed += a[q].x != b[q].x || a[q].y != b[q].y;
        for (int l = 0; l < 2; ++l)
            for (int q = 0; q < 3; ++q) failed += sa.own[l][q] != sb.own[l][q];
    }

    // 6.
    std::uniform_real_distribution<double> unit(0.0, 1.0);
    std::normal_distribution<double> normal;
    long long nodes = 0, in_float = 0, inside = 0;
    for (int t = 0; t < 400000; ++t) {
        KParams P{};
        int* const L[3] = {&P.lx, &P.ly, &P.lz};
        for (int a = 0; a < 3; ++a) {
            *L[a] = (int)std::exp2(3.0 + (a == (int)(t % 3) ? 17.0 : 5.0) * unit(g));
            P.wall[a] = (int)(g() % 2);
        }
        const int least = std::min({P.lx, P.ly, P.lz});
        P.R = 0.5 + unit(g) * std::max(0.5, 0.5 * least - 2.5);
        // a node, and a centre at distance R (1 + e) from it along a random direction
        int c[3];
        double d[3], n2 = 0.0, X[3];
        for (int a = 0; a < 3; ++a) {
            c[a] = (int)(g() % (unsigned)*L[a]);
            d[a] = normal(g);
            n2 += d[a] * d[a];
        }
        const double e = (g() % 2 ? 1.0 : -1.0) * std::pow(10.0, -16.0 * unit(g));
        bool ok = true;
        for (int a = 0; a < 3; ++a) {
            X[a] = c[a] - P.R * (1.0 + e) * d[a] / std::sqrt(n2);
            if (P.wall[a]) ok = ok && X[a] >= 0.0 && X[a] <= *L[a] - 1.0;
            else if (X[a] < 0.0) X[a] += *L[a];
            else if (X[a] >= *L[a]) X[a] -= *L[a];
        }
        if (!ok) continue;
        const SphereTest s(X, P);
        const bool want = node_inside(c, X, P);
        failed += s.inside(c, X, P) != want;
        ++nodes;
        inside += want;
        in_float += std::fabs(e) * 2.0 * P.R * P.R > 2.0 * s.margin;
    }
    // 7.
    for (int t = 0; t < 20000; ++t) {
        const long long N = 1 + (long long)(g() % 5), m = (long long)(g() % (unsigned long long)N);
        std::vector<float> f((size_t)(38 * N));
        for (float& v : f) v = (float)((g() % 2 ? 1.0 : -1.0) * std::exp2(-30.0 * unit(g)));
        double got[2];
        pop_sums(f.data(), m, N, got);
        for (int l = 0; l < 2; ++l) {
            long double sum = 0.0L, size = 0.0L;
            for (int i = 0; i < 19; ++i) {
                sum += f[(19 * l + i) * N + m];
                size += std::fabs(f[(19 * l + i) * N + m]);
            }
            failed += std::fabs((double)(got[l] - sum)) > (double)(19.0L * size) * 0x1p-53;
        }
    }
    // 8.
    {
        const int count = 20000;
        double bias[19] = {0};
        for (int t = 0; t < count; ++t) {
            float n[19] = {0}, f[19];
            n[0] = (float)(0.03 + 3.0 * unit(g));
            from_modes(n, f);
            for (int i = 0; i < 19; ++i) bias[i] += (f[i] / (w_of(i) * n[0]) - 1.0) / count;
        }
        for (int i = 0; i < 19; ++i) failed += std::fabs(bias[i]) > (i == 0 ? 2e-9 : 0x1p-26);
    }
    failed += !(nodes > 100000 && inside > nodes / 4 && in_float > nodes / 20);
    std::printf("nodes %lld inside %lld clear %lld failed %d\n", nodes, inside, in_float, failed);
    return failed == 0 ? 0 : 1;
}
