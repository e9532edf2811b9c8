// 3D boundary phases as one thread-block cluster over distributed shared
// memory: the host-built program (cluster3d.cpp) and its kernel (cluster3d.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "gcmg_internal.h"

namespace gcmg {

constexpr int C3_RANKS = 16;      // CTAs of the cluster
constexpr int C3_THREADS = 512;   // of a CTA, at most

// Header of a rank's record: counts and list bounds (ints).  A sweep (red,
// black, ghosts) runs in a rank without waiting for the others: besides its own
// nodes it updates the inside nodes of other ranks that its own updates of the
// same sweep read (halo entries).  Entries are ordered by colour, within a colour
// band sweep only | both | zone sweep only, so that a sweep takes one range.
enum {
    C3_NIN,                   // inside slots: own, halo, read only
    C3_NGS,                   // ghost slots: own, halo, read only
    C3_OWN_IN, C3_OWN_G,      // own nodes, written back
    C3_NE,                    // inside entries
    C3_RB0, C3_RB1,           // red entries of a band sweep
    C3_RZ0, C3_RZ1,           // red entries of a zone sweep
    C3_BB0, C3_BB1, C3_BZ0, C3_BZ1,   // black
    C3_GZ,                    // first zone ghost among the own ghosts
    // halo slots, refreshed after a sweep: inside band only from HI0 on, both
    // from HI1, zone only from HI2, end HI3; ghosts off the zone from HG0, in the
    // zone from HG1, end HG2
    C3_HI0, C3_HI1, C3_HI2, C3_HI3, C3_HG0, C3_HG1, C3_HG2,
    C3_HDR = 24
};

// The partition of the updated nodes over the cluster's ranks.  Every rank
// has a record of `stride` bytes with the same section offsets:
//   ints    header
//   lnode   int32 per slot: global node (inside slots, then ghost slots)
//   ent     8 x uint16 per inside entry: its slot, 6 sources in the order of
//           the sweeps' sum, first copy (0xffff: none)
//   gq      int32 per own ghost: ghost number
//   gst     4 x max_g x 8 uint16: the 27 stencil sources, first copy
//   copies  uint32: rank << 16 | slot (ghosts: max_in + ghost slot), bit 31 =
//           last; the halo slots of other ranks that hold the entry's value
// A source is an inside slot, or 0x8000 | (max_in + ghost slot).
struct Cluster3Layout {
    int stride = 0, lnode = 0, ent = 0, gq = 0, gst = 0, copies = 0;   // bytes
    int max_in = 0, max_gs = 0, max_e = 0, max_g = 0;                  // most per rank
};

struct Cluster3Program {
    bool band = false;               // holds the band sweeps too (else the zone sweeps alone)
    Cluster3Layout lay;
    std::vector<uint8_t> records;    // C3_RANKS * stride; empty: no program
};

// Program of level L's junction zone (L.junction's lists) and, with `band`,
// of its ghost and band sweeps.  Empty if there is nothing to do or a rank's
// slots do not fit 15 bits.
Cluster3Program build_cluster3(const HostLevel &L, bool band);

// Programs of several levels, built side by side on the host's threads.
struct Cluster3Want {
    int level;
    bool band;
};
std::vector<Cluster3Program> build_cluster3_levels(const std::vector<HostLevel> &H, const std::vector<Cluster3Want> &want);

// programs of either kind built on the host so far, by all contexts
extern std::atomic<long long> g_program_builds;

// Device copy of a program.
struct Cluster3Dev {
    Cluster3Layout lay;
    uint8_t *records = nullptr;
    bool band = false;
    bool fits32 = false, fits64 = false;   // per precision: shared memory, and the cluster can be resident
    bool stale = true;                     // out of date with the boundary types
};

template <typename T>
size_t cluster3_smem(const Cluster3Layout &l);
// whether a cluster of this program's size can be resident on the device
template <typename T>
bool cluster3_fits(const Cluster3Layout &l, int device);
// lead: the relaxation's ghost sweep first; then lambda band sweeps, mu zone sweeps
template <typename T>
void launch_cluster3(const LevelView<T> &v, const Cluster3Dev &P, bool lead, int lambda, int mu, cudaStream_t s);

// ---- band sweeps of larger levels, one launch a sweep
// The updated nodes are split into blocks; a block runs a whole band sweep
// (red, black, ghosts) on its own nodes and the inside nodes of other blocks
// that its updates read.  Between launches the own values of all blocks lie in
// compact arrays (block after block), the ghosts' in arrays over the ghosts.
// Every block has a record of `stride` bytes with the same section offsets:
//   ints   header (S3_*)
//   node   int32 per inside slot: grid node (own, halo, read only)
//   cid    int32 per inside slot: place in the compact array, -1: read only
//   gslot  int32 per ghost slot (own first): ghost number
//   ent    8 x uint16 per entry, red then black: its slot, 6 sources in the
//          order of the sweeps' sum
//   gst    4 x max_g x 8 uint16: the 27 stencil sources of an own ghost
// A source is an inside slot or max_in + ghost slot.
enum { S3_NIN, S3_NGS, S3_OWN_IN, S3_OWN_G, S3_RED, S3_NE, S3_BASE, S3_HDR = 8 };
struct Sweep3Layout {
    int blocks = 0, stride = 0, node = 0, cid = 0, gslot = 0, ent = 0, gst = 0;
    int max_in = 0, max_gs = 0, max_e = 0, max_g = 0;
    int inside = 0;   // entries of the compact array
};
struct Sweep3Program {
    Sweep3Layout lay;
    std::vector<uint8_t> records;   // blocks * stride; empty: no program
};
Sweep3Program build_sweep3(const HostLevel &L, int blocks);

struct Sweep3Dev {
    Sweep3Layout lay;
    uint8_t *records = nullptr;
    void *x[2] = {nullptr, nullptr};   // compact values of the inside nodes (the cycle precision)
    void *g = nullptr;                 // ghost values beside LevelView::gtmp
};
template <typename T>
size_t sweep3_smem(const Sweep3Layout &l);
template <typename T>
bool sweep3_fits(const Sweep3Layout &l, int device);
// lambda >= 2 band sweeps after the ghosts' new values have been put into
// v.gtmp; leaves u with every new value
template <typename T>
void launch_sweep3(const LevelView<T> &v, const Sweep3Dev &P, int lambda, cudaStream_t s);

}  // namespace gcmg
