// Test program (built and run by tests/test_sweep3.py, host only): the band
// sweeps of a torus' levels block by block as the kernel runs them -- a whole
// sweep a launch, own values through compact arrays -- against the same sweeps
// over the level's lists.  Prints one line "name failures count" per check:
// values (bitwise), coverage (every updated node own to one block), races
// (an entry reads what its own phase writes), bounds.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "cluster3d.h"

using namespace gcmg;

int main(int argc, char **argv) {
    const int n = argc > 1 ? std::atoi(argv[1]) : 65, nc = argc > 2 ? std::atoi(argv[2]) : 9;
    const int blocks = argc > 3 ? std::atoi(argv[3]) : 7;
    std::vector<double> phi((size_t)n * n * n);
    const double h = 2.0 / (n - 1);
    for (int i = 0; i < n; i++)
        for (int j = 0; j < n; j++)
            for (int k = 0; k < n; k++) {
                const double x = -1 + i * h, y = -1 + j * h, z = -1 + k * h;
                phi[((size_t)i * n + j) * n + k] = std::sqrt(std::pow(std::sqrt(x * x + y * y) - 0.5, 2) + z * z) - 0.25;
            }
    std::vector<HostLevel> H;
    build_hierarchy(3, n, nc, phi.data(), 3.0, H);
    long fails = 0;
    auto report = [&](const char *name, long f, long cnt) {
        std::printf("%s %ld %ld\n", name, f, cnt);
        fails += f;
    };
    unsigned rng = 777;
    auto uni = [&]() { rng = rng * 1664525u + 1013904223u; return (double)(rng >> 8) / (1 << 24) - 0.5; };
    for (HostLevel &L : H) {
        const Sweep3Program P = build_sweep3(L, blocks);
        if (P.records.empty()) {
            report("no_program", 1, 1);
            continue;
        }
        const Sweep3Layout &y = P.lay;
        std::vector<double> u(L.nn, 0.0), f(L.nn, 0.0), g(L.ng());
        for (int64_t p = 0; p < L.nn; p++)
            if ((L.type[p] & NODE_KIND) != NODE_OUT) u[p] = uni(), f[p] = uni();
        for (auto &x : g) x = uni();
        std::vector<double> w(u), gt(L.ng()), cx[2], cg[2];
        for (int64_t q = 0; q < L.ng(); q++) gt[q] = u[L.ghost_node[q]];
        for (auto &x : cx) x.assign(y.inside, NAN);
        for (auto &x : cg) x.assign(L.ng(), NAN);
        cg[0] = gt;
        long bounds = 0, race = 0, cover = 0, entries = 0;
        const int lambda = 4;
        std::vector<double> out(u);
        for (int k = 0; k < lambda; k++) {
            const bool last = k + 1 == lambda;
            std::vector<int> own(L.nn, 0), own_c(y.inside, 0);
            for (int r = 0; r < y.blocks; r++) {
                const uint8_t *rec = P.records.data() + (size_t)r * y.stride;
                const int32_t *hd = (const int32_t *)rec, *node = (const int32_t *)(rec + y.node);
                const int32_t *cid = (const int32_t *)(rec + y.cid), *gs = (const int32_t *)(rec + y.gslot);
                const uint16_t *ent = (const uint16_t *)(rec + y.ent), *gst = (const uint16_t *)(rec + y.gst);
                if (hd[S3_NIN] > y.max_in || hd[S3_NGS] > y.max_gs || hd[S3_NE] > y.max_e || hd[S3_OWN_G] > y.max_g ||
                    hd[S3_OWN_IN] > hd[S3_NIN] || hd[S3_OWN_G] > hd[S3_NGS] || hd[S3_RED] > hd[S3_NE] ||
                    hd[S3_BASE] + hd[S3_OWN_IN] > y.inside || y.gst + 64 * y.max_g != y.stride || y.stride % 16 ||
                    y.gst % 16 || y.ent % 16) {
                    bounds++;
                    continue;
                }
                std::vector<double> val(y.max_in + y.max_gs, NAN);
                for (int i = 0; i < hd[S3_NIN]; i++) {
                    if (cid[i] >= y.inside || node[i] < 0 || node[i] >= L.nn) { bounds++; continue; }
                    val[i] = k && cid[i] >= 0 ? cx[(k - 1) & 1][cid[i]] : u[node[i]];
                }
                for (int i = 0; i < hd[S3_NGS]; i++) {
                    if (gs[i] < 0 || gs[i] >= L.ng()) { bounds++; continue; }
                    val[y.max_in + i] = cg[k & 1][gs[i]];
                }
                auto get = [&](int s) {
                    if (s >= (int)val.size() || (s < y.max_in ? s >= hd[S3_NIN] : s - y.max_in >= hd[S3_NGS])) {
                        bounds++;
                        return 0.0;
                    }
                    return val[s];
                };
                auto inside = [&](int e0, int e1) {
                    std::vector<uint8_t> wrote(val.size(), 0);
                    for (int e = e0; e < e1; e++) {
                        if (ent[8 * e] >= hd[S3_NIN] || wrote[ent[8 * e]]++) { bounds++; return; }
                    }
                    for (int e = e0; e < e1; e++) {
                        const uint16_t *q = ent + 8 * e;
                        for (int a = 1; a < 7; a++) race += wrote[q[a]];
                        double nb = get(q[1]) + get(q[2]) + get(q[3]) + get(q[4]);
                        nb += get(q[5]) + get(q[6]);
                        val[q[0]] = (L.h * L.h * f[node[q[0]]] + nb) * (1.0 / 6.0);
                    }
                };
                inside(0, hd[S3_RED]);
                inside(hd[S3_RED], hd[S3_NE]);
                entries += hd[S3_NE];
                for (int i = 0; i < hd[S3_OWN_IN]; i++) {
                    own[node[i]]++;
                    own_c[hd[S3_BASE] + i]++;
                    if (cid[i] != hd[S3_BASE] + i) bounds++;
                    (last ? out[node[i]] : cx[k & 1][hd[S3_BASE] + i]) = val[i];
                }
                for (int e = 0; e < hd[S3_OWN_G]; e++) {
                    const int64_t q = gs[e];
                    double s = 0;
                    for (int a = 0; a < 27; a++) s += L.wD[q * KMAX + a] * get(gst[((size_t)(a / 8) * y.max_g + e) * 8 + a % 8]);
                    own[L.ghost_node[q]]++;
                    (last ? out[L.ghost_node[q]] : cg[(k + 1) & 1][q]) = val[y.max_in + e] + 0.9 * (g[q] - s);
                }
            }
            long n_upd = 0;
            for (int64_t p = 0; p < L.nn; p++) n_upd += own[p], cover += own[p] > 1;
            for (int x : own_c) cover += x != 1;
            cover += n_upd != (long)(L.band_red.size() + L.band_black.size() + L.ghost_node.size());
            // the same sweep over the lists
            auto sweep = [&](const std::vector<int32_t> &list) {
                for (int32_t p : list) {
                    double nb = w[p - L.stride[2]] + w[p + L.stride[2]] + w[p - L.stride[0]] + w[p + L.stride[0]];
                    nb += w[p - L.stride[1]] + w[p + L.stride[1]];
                    w[p] = (L.h * L.h * f[p] + nb) * (1.0 / 6.0);
                }
            };
            sweep(L.band_red);
            sweep(L.band_black);
            for (int64_t q = 0; q < L.ng(); q++) {
                double s = 0;
                for (int a = 0; a < 27; a++) s += L.wD[q * KMAX + a] * w[L.stn[q * KMAX + a]];
                gt[q] = w[L.ghost_node[q]] + 0.9 * (g[q] - s);
            }
            for (int64_t q = 0; q < L.ng(); q++) w[L.ghost_node[q]] = gt[q];
        }
        long bad = 0;
        for (int64_t p = 0; p < L.nn; p++) bad += !(out[p] == w[p]);
        report("values", bad, (long)L.ng());
        report("coverage", cover, y.inside);
        report("race", race, entries);
        report("bounds", bounds, y.blocks);
        std::fprintf(stderr, "n %d ng %ld inside %d blocks %d max_in %d max_gs %d max_e %d max_g %d stride %d entries/own %.2f\n", L.n,
                     (long)L.ng(), y.inside, y.blocks, y.max_in, y.max_gs, y.max_e, y.max_g, y.stride,
                     (double)entries / lambda / y.inside);
    }
    return fails ? 1 : 0;
}
