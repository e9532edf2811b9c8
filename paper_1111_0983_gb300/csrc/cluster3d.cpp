// Host side of the 3D cluster program: splits the updated nodes of a level
// over the ranks of a thread-block cluster and numbers what each rank keeps.
#include "cluster3d.h"

#include <algorithm>
#include <cstring>

namespace gcmg {

namespace {

// node -> int32 (open addressing; the nodes touched are few against the grid)
struct NodeMap {
    std::vector<int64_t> key;
    std::vector<int32_t> val;
    size_t mask = 0, used = 0;
    explicit NodeMap(size_t expect) {
        size_t n = 64;
        while (n < 2 * expect) n *= 2;
        key.assign(n, -1);
        val.assign(n, 0);
        mask = n - 1;
    }
    size_t slot(int64_t k) const {
        size_t h = (size_t)(((uint64_t)k * 0x9E3779B97F4A7C15ull) >> 20) & mask;
        while (key[h] >= 0 && key[h] != k) h = (h + 1) & mask;
        return h;
    }
    int32_t get(int64_t k, int32_t none) const {
        const size_t h = slot(k);
        return key[h] == k ? val[h] : none;
    }
    void set(int64_t k, int32_t v) {
        size_t h = slot(k);
        if (key[h] != k) {
            if (2 * ++used > mask) {
                NodeMap wider(2 * used);
                for (size_t i = 0; i <= mask; i++)
                    if (key[i] >= 0) wider.set(key[i], val[i]);
                *this = std::move(wider);
                h = slot(k);
            }
            key[h] = k;
        }
        val[h] = v;
    }
};

struct Node {
    int32_t p, q;      // node; ghost number, or -1
    int c[3];
    uint8_t black, inband, inzone;
};

// splits nodes [b, e) into `parts` ranges of about equal weight by cutting the
// longest axis of their box at the weighted median, again and again
void bisect(std::vector<Node> &N, size_t b, size_t e, int parts, int first, std::vector<size_t> &start) {
    if (parts == 1) {
        start[first] = b;
        return;
    }
    int lo[3] = {1 << 30, 1 << 30, 1 << 30}, hi[3] = {-1, -1, -1};
    for (size_t i = b; i < e; i++)
        for (int a = 0; a < 3; a++) {
            lo[a] = std::min(lo[a], N[i].c[a]);
            hi[a] = std::max(hi[a], N[i].c[a]);
        }
    int ax = 0;
    for (int a = 1; a < 3; a++)
        if (hi[a] - lo[a] > hi[ax] - lo[ax]) ax = a;
    // a ghost's update reads 27 values, an inside node's 7
    auto weight = [](const Node &x) { return x.q >= 0 ? 4 : 1; };
    std::sort(N.begin() + b, N.begin() + e, [ax](const Node &x, const Node &y) {
        return x.c[ax] != y.c[ax] ? x.c[ax] < y.c[ax] : x.p < y.p;
    });
    int64_t total = 0, run = 0;
    for (size_t i = b; i < e; i++) total += weight(N[i]);
    size_t m = b;
    while (m < e && 2 * run < total) run += weight(N[m++]);
    bisect(N, b, m, parts / 2, first, start);
    bisect(N, m, e, parts - parts / 2, first + parts / 2, start);
}

int align16(int x) { return (x + 15) & ~15; }

}  // namespace

Cluster3Program build_cluster3(const HostLevel &L, bool band) {
    Cluster3Program out;
    out.band = band;
    if (L.dim != 3) return out;
    const LocalProgram &Z = L.junction;
    // the updated nodes
    std::vector<Node> N;
    NodeMap at(band ? L.band_red.size() + L.band_black.size() + L.ghost_node.size() : Z.zred.size() * 4 + 16);
    auto add = [&](int64_t p, int32_t q, bool inband, bool inzone) {
        const int32_t i = at.get(p, -1);
        if (i >= 0) {
            N[i].inband |= inband;
            N[i].inzone |= inzone;
            return;
        }
        Node x;
        x.p = (int32_t)p;
        x.q = q;
        x.c[0] = (int)(p / L.stride[0]);
        x.c[1] = (int)(p % L.stride[0] / L.stride[1]);
        x.c[2] = (int)(p % L.stride[1]);
        x.black = (x.c[0] + x.c[1] + x.c[2]) & 1;
        x.inband = inband;
        x.inzone = inzone;
        at.set(p, (int32_t)N.size());
        N.push_back(x);
    };
    if (band) {
        for (int32_t p : L.band_red) add(p, -1, true, false);
        for (int32_t p : L.band_black) add(p, -1, true, false);
        for (int64_t q = 0; q < L.ng(); q++) add(L.ghost_node[q], (int32_t)q, true, false);
    }
    for (int32_t p : Z.zred) add(p, -1, false, true);
    for (int32_t p : Z.zblack) add(p, -1, false, true);
    for (int32_t q : Z.zghost) add(L.ghost_node[q], q, false, true);
    if (N.empty()) return out;
    std::vector<size_t> start(C3_RANKS + 1, N.size());
    bisect(N, 0, N.size(), C3_RANKS, 0, start);
    auto reads = [&](const Node &x, int64_t *rd) {
        if (x.q < 0) {   // the order of the sweeps' sum: axis 2, axis 0, axis 1
            const int64_t s[3] = {L.stride[2], L.stride[0], L.stride[1]};
            for (int a = 0; a < 3; a++) {
                rd[2 * a] = x.p - s[a];
                rd[2 * a + 1] = x.p + s[a];
            }
            return 6;
        }
        for (int k = 0; k < 27; k++) rd[k] = L.stn[(int64_t)x.q * KMAX + k];
        return 27;
    };
    auto is_ghost = [&](int64_t p) { return (L.type[p] & NODE_KIND) == NODE_GHOST; };
    // order within a rank: inside (red, black; band only, both, zone only), then ghosts (zone ones last)
    auto klass = [](const Node &x) {
        if (x.q >= 0) return x.inzone ? 9 : 8;
        return (x.black ? 3 : 0) + (x.inband ? (x.inzone ? 1 : 0) : 2);
    };
    for (int r = 0; r < C3_RANKS; r++)
        std::sort(N.begin() + start[r], N.begin() + start[r + 1], [&](const Node &x, const Node &y) {
            const int a = klass(x), b = klass(y);
            return a != b ? a < b : x.p < y.p;
        });
    struct Rank {
        std::vector<int32_t> in, gs;   // slots -> node
        int own_in = 0, own_g = 0;
        int bound[11] = {};
    };
    std::vector<Rank> R(C3_RANKS);
    std::vector<NodeMap> slot;         // per rank: node -> slot (inside or ghost)
    // (slot, rank) pairs of the copies of an updated node, by its index in N
    std::vector<std::vector<uint32_t>> cps(N.size());
    Cluster3Layout &y = out.lay;
    for (size_t i = 0; i < N.size(); i++) at.set(N[i].p, (int32_t)i);
    for (int r = 0; r < C3_RANKS; r++) {
        Rank &K = R[r];
        slot.emplace_back(4 * (start[r + 1] - start[r]) + 16);
        NodeMap &S = slot.back();
        for (size_t i = start[r]; i < start[r + 1]; i++) {
            std::vector<int32_t> &l = N[i].q >= 0 ? K.gs : K.in;
            S.set(N[i].p, (int32_t)l.size());
            l.push_back(N[i].p);
            for (int k = klass(N[i]) + 1; k < 11; k++) K.bound[k]++;
        }
        K.own_in = (int)K.in.size();
        K.own_g = (int)K.gs.size();
        int64_t rd[27];
        for (size_t i = start[r]; i < start[r + 1]; i++) {
            const int m = reads(N[i], rd);
            for (int k = 0; k < m; k++) {
                if (S.get(rd[k], -1) >= 0) continue;
                std::vector<int32_t> &l = is_ghost(rd[k]) ? K.gs : K.in;
                S.set(rd[k], (int32_t)l.size());
                l.push_back((int32_t)rd[k]);
                const int32_t o = at.get(rd[k], -1);   // updated by another rank: a copy there
                if (o >= 0) cps[o].push_back((uint32_t)r << 16 | (uint32_t)(l.size() - 1));
            }
        }
        y.max_in = std::max(y.max_in, (int)K.in.size());
        y.max_gs = std::max(y.max_gs, (int)K.gs.size());
        y.max_e = std::max(y.max_e, K.own_in);
        y.max_g = std::max(y.max_g, K.own_g);
    }
    y.max_in = (y.max_in + 3) & ~3;
    y.max_gs = (y.max_gs + 3) & ~3;
    if (y.max_in + y.max_gs >= 0x8000) return out;
    int max_c = 0;
    for (int r = 0; r < C3_RANKS; r++) {
        int nc = 0;
        for (size_t i = start[r]; i < start[r + 1]; i++) nc += (int)cps[i].size();
        max_c = std::max(max_c, nc);
    }
    if (max_c >= 0xffff) return out;
    y.lnode = C3_HDR * 4;
    y.ent = align16(y.lnode + 4 * (y.max_in + y.max_gs));
    y.gq = y.ent + 16 * y.max_e;
    y.gst = align16(y.gq + 4 * y.max_g);
    y.copies = y.gst + 64 * y.max_g;
    y.stride = align16(y.copies + 4 * max_c);
    out.records.assign((size_t)C3_RANKS * y.stride, 0);
    for (int r = 0; r < C3_RANKS; r++) {
        const Rank &K = R[r];
        uint8_t *rec = out.records.data() + (size_t)r * y.stride;
        int32_t *h = reinterpret_cast<int32_t *>(rec);
        h[C3_NIN] = (int)K.in.size();
        h[C3_NGS] = (int)K.gs.size();
        h[C3_OWN_IN] = K.own_in;
        h[C3_OWN_G] = K.own_g;
        h[C3_RB0] = K.bound[0];
        h[C3_RB1] = K.bound[2];
        h[C3_RZ0] = K.bound[1];
        h[C3_RZ1] = K.bound[3];
        h[C3_BB0] = K.bound[3];
        h[C3_BB1] = K.bound[5];
        h[C3_BZ0] = K.bound[4];
        h[C3_BZ1] = K.bound[6];
        h[C3_GZ] = K.bound[9] - K.bound[8];
        int32_t *ln = reinterpret_cast<int32_t *>(rec + y.lnode);
        std::copy(K.in.begin(), K.in.end(), ln);
        std::copy(K.gs.begin(), K.gs.end(), ln + y.max_in);
        uint16_t *ent = reinterpret_cast<uint16_t *>(rec + y.ent);
        int32_t *gq = reinterpret_cast<int32_t *>(rec + y.gq);
        uint16_t *gst = reinterpret_cast<uint16_t *>(rec + y.gst);
        uint32_t *cp = reinterpret_cast<uint32_t *>(rec + y.copies);
        int nc = 0, ie = 0, ig = 0;
        int64_t rd[27];
        for (size_t i = start[r]; i < start[r + 1]; i++) {
            uint16_t first = 0xffff;
            if (!cps[i].empty()) {
                first = (uint16_t)nc;
                for (uint32_t c : cps[i]) cp[nc++] = c;
                cp[nc - 1] |= 0x80000000u;
            }
            const int m = reads(N[i], rd);
            uint16_t src[27];
            for (int k = 0; k < m; k++) {
                const int s = slot[r].get(rd[k], -1);
                src[k] = (uint16_t)(is_ghost(rd[k]) ? 0x8000 | (y.max_in + s) : s);
            }
            if (N[i].q < 0) {
                uint16_t *e = ent + 8 * ie;
                e[0] = (uint16_t)ie;   // an own inside entry's slot is its number
                for (int k = 0; k < 6; k++) e[1 + k] = src[k];
                e[7] = first;
                ie++;
            } else {
                gq[ig] = N[i].q;
                for (int k = 0; k < 28; k++)
                    gst[((size_t)(k / 8) * y.max_g + ig) * 8 + k % 8] = k < 27 ? src[k] : first;
                ig++;
            }
        }
    }
    return out;
}

}  // namespace gcmg
