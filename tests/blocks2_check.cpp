// Test program (built and run by tests/test_blocks2.py, host only): the 2D
// boundary blocks as per-thread records (build_blocks2), phase by phase as the
// kernel runs them, against a relaxation's sweeps over the whole grid: the
// interior red and black half-sweep, the ghost sweep, lambda x (red band, black
// band, ghosts).  Prints "name failures count" lines; arguments: n, coarsest n,
// lambda, band width, block.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "gcmg_internal.h"

using namespace gcmg;

int main(int argc, char **argv) {
    const int n = std::atoi(argv[1]), nc = std::atoi(argv[2]), lambda = std::atoi(argv[3]);
    const double delta = std::atof(argv[4]);
    std::vector<double> phi((size_t)n * n);
    const double h = 2.0 / (n - 1);
    for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++) {
            const double x = -1 + i * h, y = -1 + j * h;
            phi[(size_t)i * n + j] = std::sqrt(x * x + y * y) - 0.5 - 0.15 * std::sin(5 * std::atan2(y, x));
        }
    std::vector<HostLevel> H;
    build_hierarchy(2, n, nc, phi.data(), delta, H);
    long fails = 0, race = 0, bounds = 0;
    auto report = [&](const char *name, long f, long cnt) {
        std::printf("%s %ld %ld\n", name, f, cnt);
        fails += f;
    };
    unsigned rng = 777;
    auto uni = [&]() { rng = rng * 1664525u + 1013904223u; return (double)(rng >> 8) / (1 << 24) - 0.5; };
    for (HostLevel &L : H) {
        build_boundary_blocks(L, lambda, 32);
        const Block2Host B = build_blocks2(L);
        const Block2Dev &d = B.d;
        std::printf("records %d %d %d\n", L.n, d.m, d.nt);
        if (d.m == 0) continue;
        std::vector<double> u(L.nn, 0.0), f(L.nn, 0.0), g(L.ng());
        for (int64_t p = 0; p < L.nn; p++)
            if ((L.type[p] & NODE_KIND) != NODE_OUT) u[p] = uni(), f[p] = uni();
        for (auto &x : g) x = uni();
        const double h2 = L.h * L.h;
        // the sweeps on the whole grid
        std::vector<double> w(u);
        auto sweep = [&](bool band, int colour) {
            for (int64_t p = 0; p < L.nn; p++) {
                const uint8_t t = L.type[p];
                if ((t & NODE_KIND) != NODE_IN || (band && !(t & NODE_BAND)) || ((p / L.n + p % L.n) & 1) != colour) continue;
                double s = h2 * f[p];
                s += w[p - L.n];
                s += w[p + L.n];
                s += w[p - 1];
                s += w[p + 1];
                w[p] = s * 0.25;
            }
        };
        auto ghosts = [&]() {
            std::vector<double> t(L.ng());
            for (int64_t q = 0; q < L.ng(); q++) {
                double s = 0;
                for (int k = 0; k < 9; k++) s += L.wD[q * KMAX + k] * w[L.stn[q * KMAX + k]];
                t[q] = w[L.ghost_node[q]] + 0.9 * (g[q] - s);
            }
            for (int64_t q = 0; q < L.ng(); q++) w[L.ghost_node[q]] = t[q];
        };
        sweep(false, 0);
        sweep(false, 1);
        ghosts();
        for (int k = 0; k < lambda; k++) { sweep(true, 0); sweep(true, 1); ghosts(); }
        std::vector<double> out(u);
        std::vector<int> hit(L.nn, 0);
        for (int c = 0; c < d.ncomp; c++) {
            std::vector<double> val(d.nodes + 2 * d.gh, NAN);
            std::vector<uint8_t> wrote(val.size(), 0);
            int pn = 0;
            std::vector<std::pair<size_t, double>> put;
            std::vector<size_t> rd;
            auto barrier = [&]() {
                for (auto &x : put) { if (wrote[x.first]++) race++; }
                for (size_t a : rd) if (wrote[a]) race++;
                for (auto &x : put) { val[x.first] = x.second; wrote[x.first] = 0; }
                put.clear();
                rd.clear();
            };
            auto at = [&](unsigned s) {
                const size_t a = (s & 0x7fffu) + ((s >> 15) ? pn : 0);
                if (a >= val.size()) { bounds++; return 0.0; }
                rd.push_back(a);
                return val[a];
            };
            for (int i = 0; i < d.nodes; i++)
                if (B.node[(size_t)c * d.nodes + i] >= 0) val[i] = u[B.node[(size_t)c * d.nodes + i]];
            auto rec = [&](const std::vector<uint32_t> &v, int per, int k) { return &v[((size_t)c * per + k) * 4]; };
            for (int j = 0; j < d.gh; j++)
                if ((int)rec(B.g1, d.gh, j)[3] >= 0) val[d.nodes + j] = u[rec(B.g1, d.gh, j)[2]];
            auto inside = [&](const std::vector<uint32_t> &v, int per) {
                for (int k = 0; k < per; k++) {
                    const uint32_t *r = rec(v, per, k);
                    if ((int)r[3] < 0) continue;
                    double s = h2 * f[r[3]];
                    s += at(r[0] >> 16);
                    s += at(r[1] & 0xffff);
                    s += at(r[1] >> 16);
                    s += at(r[2]);
                    put.push_back({r[0] & 0xffff, s * 0.25});
                }
                barrier();
            };
            auto gsweep = [&]() {
                for (int j = 0; j < d.gh; j++) {
                    const uint32_t *a = rec(B.g0, d.gh, j), *b = rec(B.g1, d.gh, j);
                    if ((int)b[3] < 0) continue;
                    const int64_t q = (int)b[3];
                    double s = 0;
                    for (int k = 0; k < 8; k++) s += L.wD[q * KMAX + k] * at((k & 1) ? a[k / 2] >> 16 : a[k / 2] & 0xffff);
                    s += L.wD[q * KMAX + 8] * at(b[0]);
                    rd.push_back(d.nodes + j + pn);
                    put.push_back({(size_t)d.nodes + j + (d.gh - pn), val[d.nodes + j + pn] + 0.9 * (g[q] - s)});
                }
                barrier();
                pn = d.gh - pn;
            };
            inside(B.p_red, d.pred);
            inside(B.p_black, d.pblack);
            gsweep();
            for (int k = 0; k < lambda; k++) { inside(B.e_red, d.red); inside(B.e_black, d.black); gsweep(); }
            for (int i = 0; i < d.wb; i++) {
                const int32_t p = B.w[((size_t)c * d.wb + i) * 2];
                if (p < 0) continue;
                out[p] = at((unsigned)B.w[((size_t)c * d.wb + i) * 2 + 1]);
                hit[p]++;
            }
        }
        long bad = 0, cnt = 0;
        for (int64_t p = 0; p < L.nn; p++) {
            const uint8_t t = L.type[p];
            const bool own = (t & NODE_KIND) == NODE_GHOST || ((t & NODE_KIND) == NODE_IN && (t & NODE_BAND));
            if (hit[p] != (own ? 1 : 0) || (own && std::memcmp(&out[p], &w[p], sizeof(double)))) bad++;
            cnt += own;
        }
        report("blocks", bad, cnt);
    }
    report("race", race, 1);
    report("bounds", bounds, 1);
    return fails ? 1 : 0;
}
