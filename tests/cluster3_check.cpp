// Test program (built and run by tests/test_cluster3.py, host only): the 3D
// cluster programs of a torus, phase by phase as the kernel runs them, against
// the same sweeps over the level's lists on the global grid.  Prints one line
// "name failures count" per check: values (bitwise), copies that nobody sent,
// reads of something written in the same phase (a race between two block
// barriers), bounds.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "cluster3d.h"

using namespace gcmg;

struct Rank {
    const int32_t *h, *lnode, *gq;
    const uint16_t *ent, *gst;
    const uint32_t *copies;
    std::vector<double> val, inbox[2];
};

static long race = 0, bounds = 0, stale = 0;

struct Program {
    const HostLevel &L;
    const Cluster3Program &P;
    const std::vector<double> &f, &g;
    std::vector<Rank> R;
    int par = 0, in = 0;
    Program(const HostLevel &l, const Cluster3Program &p, const std::vector<double> &u, const std::vector<double> &f_,
            const std::vector<double> &g_)
        : L(l), P(p), f(f_), g(g_), R(C3_RANKS) {
        const Cluster3Layout &y = P.lay;
        for (int r = 0; r < C3_RANKS; r++) {
            const uint8_t *rec = P.records.data() + (size_t)r * y.stride;
            Rank &K = R[r];
            K.h = (const int32_t *)rec;
            K.lnode = (const int32_t *)(rec + y.lnode);
            K.ent = (const uint16_t *)(rec + y.ent);
            K.gq = (const int32_t *)(rec + y.gq);
            K.gst = (const uint16_t *)(rec + y.gst);
            K.copies = (const uint32_t *)(rec + y.copies);
            K.val.assign(y.max_in + 2 * y.max_gs, NAN);
            for (auto &b : K.inbox) b.assign(y.max_in + y.max_gs, NAN);
            if (K.h[C3_NIN] > y.max_in || K.h[C3_NGS] > y.max_gs || K.h[C3_NE] > y.max_e || K.h[C3_OWN_G] > y.max_g ||
                K.h[C3_HI3] > K.h[C3_NIN] || K.h[C3_HG2] > K.h[C3_NGS] || K.h[C3_OWN_IN] > K.h[C3_HI0])
                bounds++;
            for (int i = 0; i < K.h[C3_NIN]; i++) K.val[i] = u[K.lnode[i]];
            for (int i = 0; i < K.h[C3_NGS]; i++)
                K.val[y.max_in + i] = K.val[y.max_in + y.max_gs + i] = u[K.lnode[y.max_in + i]];
        }
    }
    // one rank's phase between two block barriers: what it reads must not be what it writes
    std::vector<size_t> reads;
    std::vector<std::pair<size_t, double>> writes;
    double get(Rank &K, unsigned s) {
        const size_t a = (s & 0x7fffu) + ((s >> 15) ? (size_t)par * P.lay.max_gs : 0);
        if (a >= K.val.size()) { bounds++; return NAN; }
        reads.push_back(a);
        return K.val[a];
    }
    void put(Rank &K, size_t a, double x) {
        if (a >= K.val.size()) { bounds++; return; }
        writes.push_back({a, x});
    }
    void block_barrier(Rank &K) {
        std::vector<uint8_t> wrote(K.val.size(), 0);
        for (auto &w : writes) { if (wrote[w.first]++) race++; K.val[w.first] = w.second; }
        for (size_t a : reads) if (wrote[a]) race++;
        reads.clear();
        writes.clear();
    }
    void send(Rank &K, unsigned first, double x) {
        if (first == 0xffff) return;
        for (unsigned c = first;; c++) {
            if ((uint8_t *)(K.copies + c + 1) > (uint8_t *)K.h + P.lay.stride) { bounds++; return; }
            const uint32_t w = K.copies[c];
            const int r = (int)((w >> 16) & 0x7fff);
            if (r >= C3_RANKS || (w & 0xffff) >= R[r].inbox[0].size()) { bounds++; return; }
            R[r].inbox[in][w & 0xffff] = x;
            if (w >> 31) break;
        }
    }
    void inside(Rank &K, int lo, int hi) {
        for (int e = K.h[lo]; e < K.h[hi]; e++) {
            const uint16_t *q = K.ent + 8 * e;
            double nb = get(K, q[1]) + get(K, q[2]) + get(K, q[3]) + get(K, q[4]);
            nb += get(K, q[5]) + get(K, q[6]);
            const double x = (L.h * L.h * f[K.lnode[q[0]]] + nb) * (1.0 / 6.0);
            put(K, q[0], x);
            send(K, q[7], x);
        }
        block_barrier(K);
    }
    void ghosts(Rank &K, bool zone) {
        const Cluster3Layout &y = P.lay;
        const size_t po = (size_t)(1 - par) * y.max_gs;
        for (int e = zone ? K.h[C3_GZ] : 0; e < K.h[C3_OWN_G]; e++) {
            auto src = [&](int k) { return K.gst[((size_t)(k / 8) * y.max_g + e) * 8 + k % 8]; };
            const int64_t q = K.gq[e];
            double s = 0;
            for (int k = 0; k < 27; k++) s += L.wD[q * KMAX + k] * get(K, src(k));
            const double x = get(K, 0x8000u | (unsigned)(y.max_in + e)) + 0.9 * (g[q] - s);
            put(K, y.max_in + po + e, x);
            send(K, src(27), x);
        }
        block_barrier(K);
    }
    void refresh(int i0, int i1, int g0, int g1) {   // header fields; -1: nothing
        const Cluster3Layout &y = P.lay;
        par ^= 1;
        for (Rank &K : R) {
            for (int i = i0 < 0 ? 0 : K.h[i0]; i < (i0 < 0 ? 0 : K.h[i1]); i++) {
                if (K.inbox[in][i] != K.inbox[in][i]) stale++;   // nobody sent it in this sweep
                K.val[i] = K.inbox[in][i];
            }
            for (int i = K.h[g0]; i < K.h[g1]; i++) {
                if (K.inbox[in][y.max_in + i] != K.inbox[in][y.max_in + i]) stale++;
                K.val[y.max_in + par * y.max_gs + i] = K.inbox[in][y.max_in + i];
            }
            K.inbox[in].assign(y.max_in + y.max_gs, NAN);
        }
        in ^= 1;
    }
    void run(bool lead, int lambda, int mu) {
        const Cluster3Layout &y = P.lay;
        if (lead) {
            for (Rank &K : R) ghosts(K, false);
            refresh(-1, -1, C3_HG0, C3_HG2);
        }
        for (int k = 0; k < lambda; k++) {
            for (Rank &K : R) {
                inside(K, C3_RB0, C3_RB1);
                inside(K, C3_BB0, C3_BB1);
                ghosts(K, false);
            }
            refresh(C3_HI0, C3_HI2, C3_HG0, C3_HG2);
        }
        for (int k = 0; k < mu; k++) {
            for (Rank &K : R) {
                if (k == 0 && P.band)
                    for (int i = 0; i < K.h[C3_NGS]; i++)
                        put(K, y.max_in + (par ^ 1) * y.max_gs + i, K.val[y.max_in + par * y.max_gs + i]);
                inside(K, C3_RZ0, C3_RZ1);
                inside(K, C3_BZ0, C3_BZ1);
                ghosts(K, P.band);
            }
            refresh(C3_HI1, C3_HI3, C3_HG1, C3_HG2);
        }
    }
};

int main(int argc, char **argv) {
    const int n = argc > 1 ? std::atoi(argv[1]) : 65, nc = argc > 2 ? std::atoi(argv[2]) : 9;
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
    unsigned rng = 12345;
    auto uni = [&]() { rng = rng * 1664525u + 1013904223u; return (double)(rng >> 8) / (1 << 24) - 0.5; };
    for (HostLevel &L : H) {
        for (int split = 0; split < 2; split++) {   // all Dirichlet (no junction), then Neumann where B_z < 0
            for (int64_t q = 0; q < L.ng(); q++) L.bc[q] = split && L.B[q * 3 + 2] < 0;
            build_junction(L, split ? 2.0 : 0.0, 0);
            if (!split) L.junction.zred.clear(), L.junction.zblack.clear(), L.junction.zghost.clear();
            std::vector<double> u(L.nn, 0.0), f(L.nn, 0.0), g(L.ng());
            for (int64_t p = 0; p < L.nn; p++)
                if ((L.type[p] & NODE_KIND) != NODE_OUT) u[p] = uni(), f[p] = uni();
            for (auto &x : g) x = uni();
            for (int band = 0; band < 2; band++) {
                const Cluster3Program P = build_cluster3(L, band != 0);
                if (P.records.empty()) {
                    report("no_program", band || split ? 1 : 0, 1);
                    continue;
                }
                const int lambda = band ? 2 : 0, mu = split ? 3 : 0;
                Program C(L, P, u, f, g);
                C.run(band != 0, lambda, mu);
                // the same sweeps over the lists
                std::vector<double> w(u), t(L.ng());
                auto sweep = [&](const std::vector<int32_t> &list) {
                    for (int32_t p : list) {
                        double nb = w[p - 1] + w[p + 1] + w[p - L.stride[0]] + w[p + L.stride[0]];
                        nb += w[p - L.stride[1]] + w[p + L.stride[1]];
                        w[p] = (L.h * L.h * f[p] + nb) * (1.0 / 6.0);
                    }
                };
                std::vector<int32_t> all(L.ng());
                for (int64_t q = 0; q < L.ng(); q++) all[q] = (int32_t)q;
                auto jacobi = [&](const std::vector<int32_t> &list) {
                    for (int32_t q : list) {
                        double s = 0;
                        for (int k = 0; k < 27; k++) s += L.wD[(int64_t)q * KMAX + k] * w[L.stn[(int64_t)q * KMAX + k]];
                        t[q] = w[L.ghost_node[q]] + 0.9 * (g[q] - s);
                    }
                    for (int32_t q : list) w[L.ghost_node[q]] = t[q];
                };
                if (band) jacobi(all);
                for (int k = 0; k < lambda; k++) { sweep(L.band_red); sweep(L.band_black); jacobi(all); }
                for (int k = 0; k < mu; k++) {
                    sweep(L.junction.zred);
                    sweep(L.junction.zblack);
                    jacobi(L.junction.zghost);
                }
                std::vector<double> out(u);
                std::vector<int> hit(L.nn, 0);
                for (Rank &K : C.R) {
                    for (int i = 0; i < K.h[C3_OWN_IN]; i++) out[K.lnode[i]] = K.val[i], hit[K.lnode[i]]++;
                    for (int i = 0; i < K.h[C3_OWN_G]; i++) {
                        const int32_t p = K.lnode[P.lay.max_in + i];
                        out[p] = K.val[P.lay.max_in + C.par * P.lay.max_gs + i];
                        hit[p]++;
                    }
                }
                long bad = 0, cnt = 0;
                for (int64_t p = 0; p < L.nn; p++) {
                    if (std::memcmp(&out[p], &w[p], sizeof(double))) bad++;
                    if (hit[p] > 1) bad++;
                    cnt += hit[p];
                }
                report(band ? "band_and_zone" : "zone", bad, cnt);
            }
        }
    }
    report("stale", stale, 1);
    report("race", race, 1);
    report("bounds", bounds, 1);
    return fails ? 1 : 0;
}
