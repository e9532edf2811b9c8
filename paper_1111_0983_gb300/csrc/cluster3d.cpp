// Host side of the 3D cluster program: splits the updated nodes of a level
// over the ranks of a thread-block cluster and numbers what each rank keeps.
#include "cluster3d.h"

#include <algorithm>
#include <cstring>
#include <exception>
#include <thread>

#include "host_threads.h"

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

// f and g, at the same time if `apart` (and a thread can be had); an exception of
// either reaches the caller after both have ended
template <typename F, typename G>
void both(bool apart, F &&f, G &&g) {
    std::exception_ptr error;
    std::thread t;
    if (apart) try {
            t = std::thread([&]() {
                try {
                    f();
                } catch (...) {
                    error = std::current_exception();
                }
            });
        } catch (...) {   // here then
            apart = false;
        }
    try {
        if (!apart) f();
        g();
    } catch (...) {
        if (t.joinable()) t.join();
        throw;
    }
    if (t.joinable()) t.join();
    if (error) std::rethrow_exception(error);
}

// splits nodes [b, e) into `parts` ranges of about equal weight by cutting the
// longest axis of their box at the weighted share, again and again
void bisect(std::vector<Node> &N, std::vector<Node> &tmp, size_t b, size_t e, int parts, int first,
            std::vector<size_t> &start) {
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
    int64_t total = 0, run = 0;
    std::vector<size_t> at(e > b ? hi[ax] - lo[ax] + 2 : 1, 0);   // counting sort along the axis
    for (size_t i = b; i < e; i++) {
        at[N[i].c[ax] - lo[ax] + 1]++;
        total += weight(N[i]);
    }
    for (size_t k = 1; k < at.size(); k++) at[k] += at[k - 1];
    for (size_t i = b; i < e; i++) tmp[b + at[N[i].c[ax] - lo[ax]]++] = N[i];
    std::copy(tmp.begin() + b, tmp.begin() + e, N.begin() + b);
    size_t m = b;
    while (m < e && parts * run < total * (parts / 2)) run += weight(N[m++]);
    both(e - b > 4096, [&]() { bisect(N, tmp, b, m, parts / 2, first, start); },
         [&]() { bisect(N, tmp, m, e, parts - parts / 2, first + parts / 2, start); });
}

int align16(int x) { return (x + 15) & ~15; }

}  // namespace

std::atomic<long long> g_program_builds{0};

Cluster3Program build_cluster3(const HostLevel &L, bool band) {
    g_program_builds++;
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
    std::vector<Node> tmp(N.size());
    bisect(N, tmp, 0, N.size(), C3_RANKS, 0, start);
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
    // order of a rank's own nodes: inside, then ghosts (zone ones last)
    auto klass = [](const Node &x) { return x.q < 0 ? 0 : x.inzone ? 2 : 1; };
    for_each_index(C3_RANKS, N.size() / 4096, [&](int r) {
        std::sort(N.begin() + start[r], N.begin() + start[r + 1], [&](const Node &x, const Node &y) {
            const int a = klass(x), b = klass(y);
            return a != b ? a < b : x.p < y.p;
        });
    });
    struct Entry {
        int32_t i;       // index in N
        uint8_t band, zone;
    };
    struct Rank {
        std::vector<int32_t> in, gs;   // slots -> node
        std::vector<Entry> ent;        // own and halo entries, in sweep order
        int own_in = 0, own_g = 0, zone_g = 0;
        int hi[4] = {}, hg[3] = {};
        int bound[7] = {};             // entries before (colour, class) 3 * colour + class
    };
    std::vector<Rank> R(C3_RANKS);
    std::vector<NodeMap> slot;         // per rank: node -> slot (inside or ghost)
    // (rank, slot) pairs of the copies of an updated node, by its index in N
    std::vector<std::vector<uint32_t>> cps(N.size());
    Cluster3Layout &y = out.lay;
    for (size_t i = 0; i < N.size(); i++) at.set(N[i].p, (int32_t)i);
    for (int r = 0; r < C3_RANKS; r++) slot.emplace_back(4 * (start[r + 1] - start[r]) + 16);
    for_each_index(C3_RANKS, N.size() / 256, [&](int r) {
        Rank &K = R[r];
        const int32_t b0 = (int32_t)start[r], e0 = (int32_t)start[r + 1];
        NodeMap &S = slot[r];
        for (int32_t i = b0; i < e0; i++) {
            std::vector<int32_t> &l = N[i].q >= 0 ? K.gs : K.in;
            S.set(N[i].p, (int32_t)l.size());
            l.push_back(N[i].p);
            K.zone_g += N[i].q >= 0 && N[i].inzone;
        }
        K.own_in = (int)K.in.size();
        K.own_g = (int)K.gs.size();
        // the entries: a sweep's own nodes, the blacks its own ghosts read, the
        // reds those blacks and ghosts read
        NodeMap ent_of(2 * (size_t)(e0 - b0) + 16);   // node -> entry
        auto entry = [&](int32_t i, bool zone) {
            const int32_t k = ent_of.get(N[i].p, -1);
            if (k >= 0) {
                (zone ? K.ent[k].zone : K.ent[k].band) = 1;
                return;
            }
            ent_of.set(N[i].p, (int32_t)K.ent.size());
            K.ent.push_back({i, (uint8_t)!zone, (uint8_t)zone});
        };
        int64_t rd[27];
        for (int zone = band ? 0 : 1; zone < 2; zone++) {
            auto in_sweep = [&](const Node &x) { return zone ? x.inzone != 0 : x.inband != 0; };
            // inside nodes of one colour that the updates of `list` read
            auto cone = [&](const std::vector<int32_t> &list, int black) {
                for (int32_t i : list) {
                    const int m = reads(N[i], rd);
                    for (int k = 0; k < m; k++) {
                        const int32_t o = at.get(rd[k], -1);
                        if (o >= 0 && N[o].q < 0 && N[o].black == black && in_sweep(N[o])) entry(o, zone != 0);
                    }
                }
            };
            std::vector<int32_t> g, bl;
            for (int32_t i = b0; i < e0; i++) {
                if (!in_sweep(N[i])) continue;
                if (N[i].q >= 0) g.push_back(i);
                else entry(i, zone != 0);
            }
            cone(g, 1);
            for (const Entry &x : K.ent)
                if (N[x.i].black && (zone ? x.zone : x.band)) bl.push_back(x.i);
            cone(bl, 0);
            cone(g, 0);
        }
        auto cls = [&](const Entry &x) { return 3 * (int)N[x.i].black + (x.band ? (x.zone ? 1 : 0) : 2); };
        std::sort(K.ent.begin(), K.ent.end(), [&](const Entry &x, const Entry &z) {
            return cls(x) != cls(z) ? cls(x) < cls(z) : N[x.i].p < N[z.i].p;
        });
        for (const Entry &x : K.ent)
            for (int k = cls(x) + 1; k < 7; k++) K.bound[k]++;
        // every other node the updates touch: halo (updated by another rank) or read only
        std::vector<int32_t> halo_in, halo_g, fixed_in, fixed_g;
        auto touch = [&](int64_t p) {
            if (S.get(p, -1) >= 0) return;
            S.set(p, 0);   // seen; numbered below
            const bool upd = at.get(p, -1) >= 0;
            if (is_ghost(p)) (upd ? halo_g : fixed_g).push_back((int32_t)p);
            else (upd ? halo_in : fixed_in).push_back((int32_t)p);
        };
        for (const Entry &x : K.ent) {
            touch(N[x.i].p);
            const int m = reads(N[x.i], rd);
            for (int k = 0; k < m; k++) touch(rd[k]);
        }
        for (int32_t i = b0; i < e0; i++)
            if (N[i].q >= 0) {
                const int m = reads(N[i], rd);
                for (int k = 0; k < m; k++) touch(rd[k]);
            }
        auto group = [&](int32_t p) {   // band only, both, zone only
            const Node &x = N[at.get(p, -1)];
            return x.inband ? (x.inzone ? 1 : 0) : 2;
        };
        auto by_group = [&](int32_t a, int32_t c) { return group(a) != group(c) ? group(a) < group(c) : a < c; };
        std::sort(halo_in.begin(), halo_in.end(), by_group);
        std::sort(halo_g.begin(), halo_g.end(), by_group);
        K.hi[0] = K.hi[1] = K.hi[2] = K.hi[3] = K.own_in;
        for (int32_t p : halo_in)
            for (int k = group(p) + 1; k < 4; k++) K.hi[k]++;
        K.hg[0] = K.hg[1] = K.own_g;
        K.hg[2] = K.own_g + (int)halo_g.size();
        for (int32_t p : halo_g) K.hg[1] += group(p) == 0;
        for (const auto *l : {&halo_in, &fixed_in})
            for (int32_t p : *l) {
                S.set(p, (int32_t)K.in.size());
                K.in.push_back(p);
            }
        for (const auto *l : {&halo_g, &fixed_g})
            for (int32_t p : *l) {
                S.set(p, (int32_t)K.gs.size());
                K.gs.push_back(p);
            }
    });
    for (const Rank &K : R) {
        y.max_in = std::max(y.max_in, (int)K.in.size());
        y.max_gs = std::max(y.max_gs, (int)K.gs.size());
        y.max_e = std::max(y.max_e, (int)K.ent.size());
        y.max_g = std::max(y.max_g, K.own_g);
    }
    y.max_in = (y.max_in + 3) & ~3;
    y.max_gs = (y.max_gs + 3) & ~3;
    if (y.max_in + y.max_gs >= 0x8000) return out;
    for (int r = 0; r < C3_RANKS; r++) {   // the halo slots are copies of other ranks' nodes
        const Rank &K = R[r];
        for (int i = K.own_in; i < K.hi[3]; i++) cps[at.get(K.in[i], -1)].push_back((uint32_t)r << 16 | (uint32_t)i);
        for (int i = K.own_g; i < K.hg[2]; i++)
            cps[at.get(K.gs[i], -1)].push_back((uint32_t)r << 16 | (uint32_t)(y.max_in + i));
    }
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
    for_each_index(C3_RANKS, N.size() / 256, [&](int r) {
        const Rank &K = R[r];
        uint8_t *rec = out.records.data() + (size_t)r * y.stride;
        int32_t *h = reinterpret_cast<int32_t *>(rec);
        h[C3_NIN] = (int)K.in.size();
        h[C3_NGS] = (int)K.gs.size();
        h[C3_OWN_IN] = K.own_in;
        h[C3_OWN_G] = K.own_g;
        h[C3_NE] = (int)K.ent.size();
        h[C3_RB0] = K.bound[0];
        h[C3_RB1] = K.bound[2];
        h[C3_RZ0] = K.bound[1];
        h[C3_RZ1] = K.bound[3];
        h[C3_BB0] = K.bound[3];
        h[C3_BB1] = K.bound[5];
        h[C3_BZ0] = K.bound[4];
        h[C3_BZ1] = K.bound[6];
        h[C3_GZ] = K.own_g - K.zone_g;
        for (int k = 0; k < 4; k++) h[C3_HI0 + k] = K.hi[k];
        for (int k = 0; k < 3; k++) h[C3_HG0 + k] = K.hg[k];
        int32_t *ln = reinterpret_cast<int32_t *>(rec + y.lnode);
        std::copy(K.in.begin(), K.in.end(), ln);
        std::copy(K.gs.begin(), K.gs.end(), ln + y.max_in);
        uint16_t *ent = reinterpret_cast<uint16_t *>(rec + y.ent);
        int32_t *gq = reinterpret_cast<int32_t *>(rec + y.gq);
        uint16_t *gst = reinterpret_cast<uint16_t *>(rec + y.gst);
        uint32_t *cp = reinterpret_cast<uint32_t *>(rec + y.copies);
        int nc = 0;
        int64_t rd[27];
        auto copies_of = [&](int32_t i) {   // only this rank's own nodes are sent
            uint16_t first = 0xffff;
            if (i >= (int32_t)start[r] && i < (int32_t)start[r + 1] && !cps[i].empty()) {
                first = (uint16_t)nc;
                for (uint32_t c : cps[i]) cp[nc++] = c;
                cp[nc - 1] |= 0x80000000u;
            }
            return first;
        };
        auto source = [&](int64_t p) {
            const int s = slot[r].get(p, -1);
            return (uint16_t)(is_ghost(p) ? 0x8000 | (y.max_in + s) : s);
        };
        for (size_t k = 0; k < K.ent.size(); k++) {
            const Node &x = N[K.ent[k].i];
            uint16_t *e = ent + 8 * k;
            e[0] = source(x.p);
            reads(x, rd);
            for (int a = 0; a < 6; a++) e[1 + a] = source(rd[a]);
            e[7] = copies_of(K.ent[k].i);
        }
        int ig = 0;
        for (int32_t i = (int32_t)start[r]; i < (int32_t)start[r + 1]; i++) {
            if (N[i].q < 0) continue;
            gq[ig] = N[i].q;
            reads(N[i], rd);
            for (int k = 0; k < 28; k++)
                gst[((size_t)(k / 8) * y.max_g + ig) * 8 + k % 8] = k < 27 ? source(rd[k]) : copies_of(i);
            ig++;
        }
    });
    return out;
}

Sweep3Program build_sweep3(const HostLevel &L, int blocks) {
    g_program_builds++;
    Sweep3Program out;
    if (L.dim != 3 || blocks < 1) return out;
    std::vector<Node> N;
    N.reserve(L.band_red.size() + L.band_black.size() + L.ghost_node.size());
    auto add = [&](int64_t p, int32_t q) {
        Node x;
        x.p = (int32_t)p;
        x.q = q;
        x.c[0] = (int)(p / L.stride[0]);
        x.c[1] = (int)(p % L.stride[0] / L.stride[1]);
        x.c[2] = (int)(p % L.stride[1]);
        x.black = (x.c[0] + x.c[1] + x.c[2]) & 1;
        x.inband = 1;
        x.inzone = 0;
        N.push_back(x);
    };
    for (int32_t p : L.band_red) add(p, -1);
    for (int32_t p : L.band_black) add(p, -1);
    for (int64_t q = 0; q < L.ng(); q++) add(L.ghost_node[q], (int32_t)q);
    if (N.empty()) return out;
    std::vector<size_t> start(blocks + 1, N.size());
    std::vector<Node> tmp(N.size());
    bisect(N, tmp, 0, N.size(), blocks, 0, start);
    NodeMap at(N.size());   // updated node -> index in N
    std::vector<int32_t> base(blocks + 1, 0);
    for_each_index(blocks, N.size() / 4096, [&](int r) {
        std::sort(N.begin() + start[r], N.begin() + start[r + 1], [](const Node &x, const Node &y) {
            const int a = x.q < 0 ? x.black : 2, b = y.q < 0 ? y.black : 2;
            return a != b ? a < b : x.p < y.p;
        });
        for (size_t i = start[r]; i < start[r + 1]; i++) base[r + 1] += N[i].q < 0;
    });
    for (int r = 0; r < blocks; r++) base[r + 1] += base[r];
    std::vector<int32_t> cid(N.size(), -1);   // place of an inside node in the compact array
    for (int r = 0; r < blocks; r++)
        for (size_t i = start[r]; i < start[r + 1]; i++) {
            at.set(N[i].p, (int32_t)i);
            if (N[i].q < 0) cid[i] = base[r] + (int32_t)(i - start[r]);   // inside nodes come first
        }
    struct Block {
        std::vector<int32_t> in, gs, red, black;   // slots -> node; entries (index in N)
        std::vector<uint16_t> ent, gst;
        std::vector<int32_t> in_cid, gs_q;
        int own_in = 0, own_g = 0;
    };
    std::vector<Block> B(blocks);
    auto work = [&](int r) {
        int64_t rd[27];
        Block &K = B[r];
        const int32_t b0 = (int32_t)start[r], e0 = (int32_t)start[r + 1];
        NodeMap S(6 * (size_t)(e0 - b0) + 64), in_ent(4 * (size_t)(e0 - b0) + 64);
        auto reads = [&](const Node &x) {
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
        auto touch = [&](int64_t p) {
            if (S.get(p, -1) >= 0) return;
            const int32_t o = at.get(p, -1);
            if ((L.type[p] & NODE_KIND) == NODE_GHOST) {
                S.set(p, (int32_t)K.gs.size());
                K.gs.push_back((int32_t)p);
                K.gs_q.push_back(N[o].q);   // every ghost is updated
            } else {
                S.set(p, (int32_t)K.in.size());
                K.in.push_back((int32_t)p);
                K.in_cid.push_back(o < 0 ? -1 : cid[o]);
            }
        };
        for (int32_t i = b0; i < e0; i++) {
            touch(N[i].p);
            if (N[i].q < 0) {
                in_ent.set(N[i].p, 1);
                (N[i].black ? K.black : K.red).push_back(i);
                K.own_in++;
            } else {
                K.own_g++;
            }
        }
        // the blacks the own ghosts read, the reds those blacks and ghosts read
        auto cone = [&](int32_t i, int black) {
            const int m = reads(N[i]);
            for (int k = 0; k < m; k++) {
                const int32_t o = at.get(rd[k], -1);
                if (o < 0 || N[o].q >= 0 || N[o].black != black || in_ent.get(N[o].p, 0)) continue;
                in_ent.set(N[o].p, 1);
                (black ? K.black : K.red).push_back(o);
            }
        };
        for (int32_t i = b0; i < e0; i++)
            if (N[i].q >= 0) cone(i, 1);
        for (size_t k = 0; k < K.black.size(); k++) cone(K.black[k], 0);
        for (int32_t i = b0; i < e0; i++)
            if (N[i].q >= 0) cone(i, 0);
        for (const auto *l : {&K.red, &K.black})
            for (int32_t i : *l) {
                touch(N[i].p);
                const int m = reads(N[i]);
                for (int k = 0; k < m; k++) touch(rd[k]);
            }
        for (int32_t i = b0; i < e0; i++)
            if (N[i].q >= 0) {
                const int m = reads(N[i]);
                for (int k = 0; k < m; k++) touch(rd[k]);
            }
    };
    for_each_index(blocks, N.size() / 256, work);
    Sweep3Layout &y = out.lay;
    y.blocks = blocks;
    y.inside = base[blocks];
    for (const Block &K : B) {
        y.max_in = std::max(y.max_in, (int)K.in.size());
        y.max_gs = std::max(y.max_gs, (int)K.gs.size());
        y.max_e = std::max(y.max_e, (int)(K.red.size() + K.black.size()));
        y.max_g = std::max(y.max_g, K.own_g);
    }
    y.max_in = (y.max_in + 3) & ~3;
    if (y.max_in + y.max_gs >= 0x10000) return out;
    y.node = S3_HDR * 4;
    y.cid = y.node + 4 * y.max_in;
    y.gslot = y.cid + 4 * y.max_in;
    y.ent = align16(y.gslot + 4 * y.max_gs);
    y.gst = y.ent + 16 * y.max_e;
    y.stride = y.gst + 64 * y.max_g;
    out.records.assign((size_t)blocks * y.stride, 0);
    auto write = [&](int r) {
        const Block &K = B[r];
        NodeMap S(2 * (K.in.size() + K.gs.size()) + 64);
        for (size_t i = 0; i < K.in.size(); i++) S.set(K.in[i], (int32_t)i);
        for (size_t i = 0; i < K.gs.size(); i++) S.set(K.gs[i], y.max_in + (int32_t)i);
        uint8_t *rec = out.records.data() + (size_t)r * y.stride;
        int32_t *h = reinterpret_cast<int32_t *>(rec);
        h[S3_NIN] = (int)K.in.size();
        h[S3_NGS] = (int)K.gs.size();
        h[S3_OWN_IN] = K.own_in;
        h[S3_OWN_G] = K.own_g;
        h[S3_RED] = (int)K.red.size();
        h[S3_NE] = (int)(K.red.size() + K.black.size());
        h[S3_BASE] = base[r];
        std::copy(K.in.begin(), K.in.end(), reinterpret_cast<int32_t *>(rec + y.node));
        std::copy(K.in_cid.begin(), K.in_cid.end(), reinterpret_cast<int32_t *>(rec + y.cid));
        std::copy(K.gs_q.begin(), K.gs_q.end(), reinterpret_cast<int32_t *>(rec + y.gslot));
        uint16_t *e = reinterpret_cast<uint16_t *>(rec + y.ent), *g = reinterpret_cast<uint16_t *>(rec + y.gst);
        const int64_t s[3] = {L.stride[2], L.stride[0], L.stride[1]};
        for (const auto *l : {&K.red, &K.black})
            for (int32_t i : *l) {
                const int64_t p = N[i].p;
                e[0] = (uint16_t)S.get(p, 0);
                for (int a = 0; a < 3; a++) {
                    e[1 + 2 * a] = (uint16_t)S.get(p - s[a], 0);
                    e[2 + 2 * a] = (uint16_t)S.get(p + s[a], 0);
                }
                e += 8;
            }
        for (int k = 0; k < K.own_g; k++)
            for (int a = 0; a < 27; a++)
                g[((size_t)(a / 8) * y.max_g + k) * 8 + a % 8] =
                    (uint16_t)S.get(L.stn[(int64_t)K.gs_q[k] * KMAX + a], 0);
    };
    for_each_index(blocks, N.size() / 1024, write);
    return out;
}

std::vector<Cluster3Program> build_cluster3_levels(const std::vector<HostLevel> &H, const std::vector<Cluster3Want> &want) {
    std::vector<Cluster3Program> out(want.size());
    for_each_index((int)want.size(), want.size(), [&](int i) { out[i] = build_cluster3(H[want[i].level], want[i].band); });
    return out;
}

}  // namespace gcmg
