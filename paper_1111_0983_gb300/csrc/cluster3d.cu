// The ghost, band and junction-zone phases of one 3D boundary relaxation as
// one launch: a thread-block cluster whose CTAs keep a part of the updated
// nodes each, with the values, stencils and weights in shared memory.  A CTA
// runs a whole sweep (red, black, ghosts) on its own: it also updates the few
// inside nodes of its neighbours that its own updates of the sweep read.  It
// sends its own new values straight into an inbox in the CTAs that hold copies
// of them (distributed shared memory); after the sweep's one cluster barrier
// each CTA refreshes its copies from the inbox.
//
// What bounds a small level's boundary phases is not their work but that they
// are dozens of dependent steps: a launch a phase costs 1.5 us (the launch, and
// a round trip to L2 for the values the previous one wrote).  Here a phase is
// a few shared-memory reads and a block barrier, and a sweep a cluster barrier,
// which takes 1,000 cycles with 16 CTAs whatever they do.  Measured, ten zone
// sweeps at 33^3: 43 us with a launch a phase, 18 us with a cluster barrier a
// phase, 12-13 us so.  Clusters of 8 CTAs: 5 % slower from 65^3 on.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "cluster3d.h"
#include "ctx.h"
#include "gcmg_internal.h"
#include "kernels.h"
#include "kernels_dev.cuh"

namespace gcmg {

namespace {

using namespace dev;

__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address in the cluster of what lies at `local` in CTA `rank`
__device__ __forceinline__ unsigned remote(unsigned local, unsigned rank) {
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}
__device__ __forceinline__ void store_remote(unsigned a, float x) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}
__device__ __forceinline__ void store_remote(unsigned a, double x) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(x) : "memory");
}

// where an entry's value goes besides its slot: the first copy's address (inbox
// 0), the index of the next one in the copy list (0xffff: no more)
struct Dest {
    unsigned addr, next;
    bool any;
};
// an inside entry, and an own ghost, held in registers: sources as slots with a
// bit each for those that are ghosts (two values)
template <typename T>
struct InsideRec {
    T h2f;
    int me, o[6];
    unsigned two;
    Dest d;
    bool on;
};
template <typename T>
struct GhostRec {
    static constexpr int NW = sizeof(T) == 4 ? 27 : 1;   // FP64 weights stay in shared memory
    T w[NW], gc, gg;
    int o[27];
    unsigned two;
    Dest d;
    bool on;
};

// Ghosts have two values each (Jacobi: a sweep reads the old ones of the
// others): ghost slot g at max_in + g (parity 0) and max_in + max_gs + g.  Two
// inboxes of max_in + max_gs values, used in turn: a CTA sends into one again
// after a barrier at which the receiver had emptied it.
template <typename T>
__global__ void __launch_bounds__(C3_THREADS, 1) k_cluster3d(LevelView<T> v, Cluster3Layout L,
                                                             const uint8_t *__restrict__ records, int lead, int lambda,
                                                             int mu, int band) {
    extern __shared__ __align__(16) unsigned char smem_c3[];
    pdl_trigger();
    const int tid = threadIdx.x, nt = blockDim.x;
    unsigned char *rec = smem_c3;
    T *val = reinterpret_cast<T *>(rec + L.stride);   // max_in + 2 max_gs
    T *inbox = val + L.max_in + 2 * L.max_gs;             // 2 x (max_in + max_gs)
    T *sf = inbox + 2 * (L.max_in + L.max_gs);            // h^2 f of the inside entries
    T *gg = sf + L.max_e;                                 // own ghosts: g, mu dt, 27 weights (slot major)
    T *gc = gg + L.max_g;
    T *gw = gc + L.max_g;
    // the record, then through it the weights: fixed while a solve runs, read
    // before the wait for the previous launch
    const uint8_t *src = records + (size_t)blockIdx.x * L.stride;
    for (int i = tid * 16; i < L.stride; i += nt * 16) cp_async16(rec + i, src + i);
    cp_async_wait_all();
    __syncthreads();
    const int *h = reinterpret_cast<const int *>(rec);
    const int32_t *lnode = reinterpret_cast<const int32_t *>(rec + L.lnode);
    const uint4 *ent = reinterpret_cast<const uint4 *>(rec + L.ent);
    const int32_t *gq = reinterpret_cast<const int32_t *>(rec + L.gq);
    const uint4 *gst = reinterpret_cast<const uint4 *>(rec + L.gst);
    const uint32_t *copies = reinterpret_cast<const uint32_t *>(rec + L.copies);
    const int nin = h[C3_NIN], ngs = h[C3_NGS], own_in = h[C3_OWN_IN], own_g = h[C3_OWN_G], ne = h[C3_NE];
    for (int e = tid; e < own_g; e += nt) {
        const int q = gq[e];
        cp_async(&gc[e], &v.gc[q]);
#pragma unroll
        for (int k = 0; k < 27; k++) cp_async(&gw[k * L.max_g + e], &v.gw[(int64_t)k * v.ng + q]);
    }
    pdl_wait();
    for (int i = tid; i < nin; i += nt) cp_async(&val[i], &v.u[lnode[i]]);
    for (int i = tid; i < ngs; i += nt) {
        const T *u = &v.u[lnode[L.max_in + i]];
        cp_async(&val[L.max_in + i], u);
        cp_async(&val[L.max_in + L.max_gs + i], u);
    }
    for (int e = tid; e < ne; e += nt) cp_async(&sf[e], &v.f[lnode[ent[e].x & 0xffffu]]);
    for (int e = tid; e < own_g; e += nt) cp_async(&gg[e], &v.gg[gq[e]]);
    cp_async_wait_all();
    for (int e = tid; e < ne; e += nt) sf[e] = mul_rn(v.h2, sf[e]);   // its own copies: no barrier needed
    cluster_barrier();   // every CTA runs: its inbox may be written

    const int box = L.max_in + L.max_gs;
    const unsigned inbox0 = (unsigned)__cvta_generic_to_shared(inbox), box_bytes = box * (unsigned)sizeof(T);
    int par = 0, in = 0;   // the ghosts' current values, the inbox in use
    auto dest = [&](unsigned first) {
        Dest d{0, 0xffffu, first != 0xffffu};
        if (d.any) {
            const uint32_t w = copies[first];
            d.addr = remote(inbox0 + (w & 0xffffu) * (unsigned)sizeof(T), (w >> 16) & 0x7fffu);
            if (!(w >> 31)) d.next = first + 1;
        }
        return d;
    };
    auto send = [&](const Dest &d, T x) {
        if (!d.any) return;
        store_remote(d.addr + in * box_bytes, x);
        for (unsigned c = d.next; c != 0xffffu;) {
            const uint32_t w = copies[c];
            store_remote(remote(inbox0 + in * box_bytes + (w & 0xffffu) * (unsigned)sizeof(T), (w >> 16) & 0x7fffu), x);
            c = w >> 31 ? 0xffffu : c + 1;
        }
    };
    // after a sweep: the copies of inside slots [i0, i1) and ghost slots [g0, g1)
    auto refresh = [&](int i0, int i1, int g0, int g1) {
        cluster_barrier();
        const T *b = inbox + in * box;
        for (int i = i0 + tid; i < i1; i += nt) val[i] = b[i];
        for (int i = g0 + tid; i < g1; i += nt) val[L.max_in + par * L.max_gs + i] = b[L.max_in + i];
        in ^= 1;
        __syncthreads();
    };
    // Gauss-Seidel form of Eq. (jac2d), 7 points: the sums of k_rb_list in the
    // same order.  A thread's first entry of a sweep's range is in registers.
    auto load_inside = [&](int e, int e1) {
        InsideRec<T> r;
        r.on = e < e1;
        r.two = 0;
        if (r.on) {
            const uint4 q = ent[e];
            const unsigned s[6] = {q.x >> 16, q.y & 0xffffu, q.y >> 16, q.z & 0xffffu, q.z >> 16, q.w & 0xffffu};
            r.me = q.x & 0xffffu;
            r.h2f = sf[e];
#pragma unroll
            for (int k = 0; k < 6; k++) {
                r.o[k] = s[k] & 0x7fffu;
                r.two |= (s[k] >> 15) << k;
            }
            r.d = dest(q.w >> 16);
        }
        return r;
    };
    auto do_inside = [&](const InsideRec<T> &r) {
        if (!r.on) return;
        const int pn = par * L.max_gs;
        T x[6];
#pragma unroll
        for (int k = 0; k < 6; k++) x[k] = val[r.o[k] + ((r.two >> k & 1u) ? pn : 0)];
        T nb = x[0] + x[1] + x[2] + x[3];
        nb += x[4] + x[5];
        const T y = (r.h2f + nb) * (T)(1.0 / 6.0);
        val[r.me] = y;
        send(r.d, y);
    };
    auto inside = [&](const InsideRec<T> &first, int e0, int e1) {
        do_inside(first);
        for (int e = e0 + tid + nt; e < e1; e += nt) do_inside(load_inside(e, e1));
    };
    // Eqs. (dir2d)/(neu2d) at the own ghosts from g0 on
    auto load_ghost = [&](int e) {
        GhostRec<T> r;
        r.on = e < own_g;
        r.two = 0;
        if (r.on) {
            unsigned first = 0xffffu;
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const uint4 q = gst[c * L.max_g + e];
                const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const unsigned s = (k & 1) ? w[k / 2] >> 16 : w[k / 2] & 0xffffu;
                    if (8 * c + k < 27) {
                        r.o[8 * c + k] = s & 0x7fffu;
                        r.two |= (s >> 15) << (8 * c + k);
                    } else if (8 * c + k == 27) {
                        first = s;
                    }
                }
            }
            if (GhostRec<T>::NW == 27)
#pragma unroll
                for (int k = 0; k < GhostRec<T>::NW; k++) r.w[k] = gw[k * L.max_g + e];
            r.gc = gc[e];
            r.gg = gg[e];
            r.d = dest(first);
        }
        return r;
    };
    auto do_ghost = [&](const GhostRec<T> &r, int e) {
        if (!r.on) return;
        const int pn = par * L.max_gs, po = L.max_gs - pn;
        T s = 0;
#pragma unroll
        for (int k = 0; k < 27; k++)
            s += (GhostRec<T>::NW == 27 ? r.w[k % GhostRec<T>::NW] : gw[k * L.max_g + e]) *
                 val[r.o[k] + ((r.two >> k & 1u) ? pn : 0)];
        const T x = val[L.max_in + pn + e] + r.gc * (r.gg - s);
        val[L.max_in + po + e] = x;
        send(r.d, x);
    };
    auto ghosts = [&](const GhostRec<T> &first, int g0) {
        do_ghost(first, g0 + tid);
        for (int e = g0 + tid + nt; e < own_g; e += nt) do_ghost(load_ghost(e), e);
    };
    if (lead || lambda > 0) {
        const GhostRec<T> g = load_ghost(tid);
        const InsideRec<T> r = load_inside(h[C3_RB0] + tid, h[C3_RB1]), b = load_inside(h[C3_BB0] + tid, h[C3_BB1]);
        if (lead) {
            ghosts(g, 0);
            par ^= 1;
            refresh(0, 0, h[C3_HG0], h[C3_HG2]);
        }
        for (int k = 0; k < lambda; k++) {
            inside(r, h[C3_RB0], h[C3_RB1]);
            __syncthreads();
            inside(b, h[C3_BB0], h[C3_BB1]);
            __syncthreads();
            ghosts(g, 0);
            par ^= 1;
            refresh(h[C3_HI0], h[C3_HI2], h[C3_HG0], h[C3_HG2]);
        }
    }
    if (mu > 0) {
        const int gz = band ? h[C3_GZ] : 0;
        const GhostRec<T> g = load_ghost(gz + tid);
        const InsideRec<T> r = load_inside(h[C3_RZ0] + tid, h[C3_RZ1]), b = load_inside(h[C3_BZ0] + tid, h[C3_BZ1]);
        // the ghosts off the zone keep their value from here on: both parities
        // (the other one is not read before the ghost sweep)
        if (band)
            for (int i = tid; i < ngs; i += nt)
                val[L.max_in + (par ^ 1) * L.max_gs + i] = val[L.max_in + par * L.max_gs + i];
        for (int k = 0; k < mu; k++) {
            inside(r, h[C3_RZ0], h[C3_RZ1]);
            __syncthreads();
            inside(b, h[C3_BZ0], h[C3_BZ1]);
            __syncthreads();
            ghosts(g, gz);
            par ^= 1;
            refresh(h[C3_HI1], h[C3_HI3], h[C3_HG1], h[C3_HG2]);
        }
    }
    for (int i = tid; i < own_in; i += nt) v.u[lnode[i]] = val[i];
    for (int i = tid; i < own_g; i += nt) v.u[lnode[L.max_in + i]] = val[L.max_in + par * L.max_gs + i];
}

// threads of a CTA: one a ghost and an entry of a colour where 512 allow it; no
// more warps than that, since each of them takes part in the cluster barrier
// (the zone sweeps of the torus at 33^3: 14.8 us with 512 threads, 11.8 with 256)
unsigned cluster3_threads(const Cluster3Layout &l) {
    unsigned t = 128;
    while (t < C3_THREADS && (int)t < std::max(l.max_g, (l.max_e + 1) / 2)) t *= 2;
    return t;
}

// launch configuration of a program (attributes in `at`)
template <typename T>
cudaLaunchConfig_t cluster3_config(const Cluster3Layout &l, cudaStream_t s, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C3_RANKS);
    cfg.blockDim = dim3(cluster3_threads(l));
    cfg.dynamicSmemBytes = cluster3_smem<T>(l);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C3_RANKS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cfg;
}

}  // namespace

template <typename T>
size_t cluster3_smem(const Cluster3Layout &l) {
    return (size_t)l.stride +
           sizeof(T) * (3 * (size_t)l.max_in + 4 * (size_t)l.max_gs + l.max_e + 29 * (size_t)l.max_g);
}

template <typename T>
bool cluster3_fits(const Cluster3Layout &l, int device) {
    int most = 0;
    if (cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        cluster3_smem<T>(l) > (size_t)most)
        return false;
    // per kernel, not per launch: allow the device's maximum, and 16 CTAs (the portable size is 8)
    if (cudaFuncSetAttribute(k_cluster3d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess ||
        cudaFuncSetAttribute(k_cluster3d<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = cluster3_config<T>(l, nullptr, at);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_cluster3d<T>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

template <typename T>
void launch_cluster3(const LevelView<T> &v, const Cluster3Dev &P, bool lead, int lambda, int mu, cudaStream_t s) {
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t cfg = cluster3_config<T>(P.lay, s, at);
    g_launches++;
    ck(cudaLaunchKernelEx(&cfg, k_cluster3d<T>, v, P.lay, (const uint8_t *)P.records, (int)lead, lambda, mu,
                          (int)P.band),
       "cluster launch");
}

template size_t cluster3_smem<float>(const Cluster3Layout &);
template size_t cluster3_smem<double>(const Cluster3Layout &);
template bool cluster3_fits<float>(const Cluster3Layout &, int);
template bool cluster3_fits<double>(const Cluster3Layout &, int);
template void launch_cluster3<float>(const LevelView<float> &, const Cluster3Dev &, bool, int, int, cudaStream_t);
template void launch_cluster3<double>(const LevelView<double> &, const Cluster3Dev &, bool, int, int, cudaStream_t);

}  // namespace gcmg
