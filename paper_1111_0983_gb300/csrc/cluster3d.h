// 3D boundary phases as one thread-block cluster over distributed shared
// memory: the host-built program (cluster3d.cpp) and its kernel (cluster3d.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

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

// Device copy of a program.
struct Cluster3Dev {
    Cluster3Layout lay;
    uint8_t *records = nullptr;
    bool band = false;
    bool fits32 = false, fits64 = false;   // per precision: shared memory, and the cluster can be resident
};

template <typename T>
size_t cluster3_smem(const Cluster3Layout &l);
// whether a cluster of this program's size can be resident on the device
template <typename T>
bool cluster3_fits(const Cluster3Layout &l, int device);
// lead: the relaxation's ghost sweep first; then lambda band sweeps, mu zone sweeps
template <typename T>
void launch_cluster3(const LevelView<T> &v, const Cluster3Dev &P, bool lead, int lambda, int mu, cudaStream_t s);

}  // namespace gcmg
