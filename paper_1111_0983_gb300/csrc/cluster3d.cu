// The ghost, band and junction-zone phases of one 3D boundary relaxation as
// one launch: a thread-block cluster whose CTAs keep a part of the updated
// nodes each, with the values, stencils and weights in shared memory, and send
// a value that another CTA reads straight into that CTA's copy of it
// (distributed shared memory).  Between two phases a cluster barrier (an
// arrival on each neighbour's mbarrier instead measured 10 % slower: either way
// the sent values have to be acknowledged before the arrival).
//
// What bounds a small level's boundary phases is not their work but that they
// are dozens of dependent steps: a launch a phase costs 1.5 us (the launch, and
// a round trip to L2 for the values the previous one wrote).  Here a phase is
// a few shared-memory reads and a barrier.
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

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// store into the shared memory of the cluster's CTA `rank` at the address that
// `local` has in this CTA
__device__ __forceinline__ void send(unsigned local, unsigned rank, float x) {
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}
__device__ __forceinline__ void send(unsigned local, unsigned rank, double x) {
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(x) : "memory");
}

// Ghosts have two values each (Jacobi: a sweep reads the old ones of the
// others): ghost slot g at max_in + g (parity 0) and max_in + max_gs + g.
template <typename T>
__global__ void __launch_bounds__(C3_THREADS, 1) k_cluster3d(LevelView<T> v, Cluster3Layout L,
                                                             const uint8_t *__restrict__ records, int lead, int lambda,
                                                             int mu, int band) {
    extern __shared__ __align__(16) unsigned char smem_c3[];
    pdl_trigger();
    const int tid = threadIdx.x, nt = C3_THREADS;
    unsigned char *rec = smem_c3;
    T *val = reinterpret_cast<T *>(rec + L.stride);   // max_in + 2 max_gs
    T *sf = val + L.max_in + 2 * L.max_gs;                // h^2 f of the own inside entries
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
    const int nin = h[C3_NIN], ngs = h[C3_NGS], own_in = h[C3_OWN_IN], own_g = h[C3_OWN_G];
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
    for (int e = tid; e < own_in; e += nt) cp_async(&sf[e], &v.f[lnode[e]]);
    for (int e = tid; e < own_g; e += nt) cp_async(&gg[e], &v.gg[gq[e]]);
    cp_async_wait_all();
    for (int e = tid; e < own_in; e += nt) sf[e] = mul_rn(v.h2, sf[e]);   // its own copies: no barrier needed
    cluster_barrier();

    const unsigned vbase = (unsigned)__cvta_generic_to_shared(val);
    int par = 0;   // the ghosts' current values
    auto at = [&](unsigned s, int pn) -> T { return val[(s & 0x7fffu) + ((s >> 15) ? pn : 0)]; };
    // the value also goes to every rank that keeps a copy (slot offset `add`)
    auto send_copies = [&](unsigned first, int add, T x) {
        if (first == 0xffffu) return;
        for (unsigned c = first;; c++) {
            const uint32_t w = copies[c];
            send(vbase + ((w & 0xffffu) + add) * (unsigned)sizeof(T), (w >> 16) & 0x7fffu, x);
            if (w >> 31) break;
        }
    };
    // Gauss-Seidel form of Eq. (jac2d), 7 points, entries [e0, e1): the sums of
    // k_rb_list in the same order
    auto inside = [&](int e0, int e1) {
        const int pn = par * L.max_gs;
        for (int e = e0 + tid; e < e1; e += nt) {
            const uint4 r = ent[e];
            T nb = at(r.x >> 16, pn) + at(r.y & 0xffffu, pn) + at(r.y >> 16, pn) + at(r.z & 0xffffu, pn);
            nb += at(r.z >> 16, pn) + at(r.w & 0xffffu, pn);
            const T x = (sf[e] + nb) * (T)(1.0 / 6.0);
            val[e] = x;
            send_copies(r.w >> 16, 0, x);
        }
    };
    // Eqs. (dir2d)/(neu2d) at the own ghosts from g0 on
    auto ghosts = [&](int g0) {
        const int pn = par * L.max_gs, po = L.max_gs - pn;
        for (int e = g0 + tid; e < own_g; e += nt) {
            T s = 0;
            unsigned first = 0xffffu;
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const uint4 r = gst[c * L.max_g + e];
                const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int k = 0; k < 8; k++) {
                    const unsigned idx = (k & 1) ? w[k / 2] >> 16 : w[k / 2] & 0xffffu;
                    if (8 * c + k < 27) s += gw[(8 * c + k) * L.max_g + e] * at(idx, pn);
                    else if (8 * c + k == 27) first = idx;
                }
            }
            const T x = val[L.max_in + pn + e] + gc[e] * (gg[e] - s);
            val[L.max_in + po + e] = x;
            send_copies(first, L.max_in + po, x);
        }
    };
    if (lead) {
        ghosts(0);
        par ^= 1;
        cluster_barrier();
    }
    for (int k = 0; k < lambda; k++) {
        inside(h[C3_RB0], h[C3_RB1]);
        cluster_barrier();
        inside(h[C3_BB0], h[C3_BB1]);
        cluster_barrier();
        ghosts(0);
        par ^= 1;
        cluster_barrier();
    }
    for (int k = 0; k < mu; k++) {
        // the ghosts off the zone keep their value from here on: both parities
        // (the other one is not read before the next ghost sweep's barrier)
        if (k == 0 && band)
            for (int i = tid; i < ngs; i += nt)
                val[L.max_in + (par ^ 1) * L.max_gs + i] = val[L.max_in + par * L.max_gs + i];
        inside(h[C3_RZ0], h[C3_RZ1]);
        cluster_barrier();
        inside(h[C3_BZ0], h[C3_BZ1]);
        cluster_barrier();
        ghosts(band ? h[C3_GZ] : 0);
        par ^= 1;
        cluster_barrier();
    }
    for (int i = tid; i < own_in; i += nt) v.u[lnode[i]] = val[i];
    for (int i = tid; i < own_g; i += nt) v.u[lnode[L.max_in + i]] = val[L.max_in + par * L.max_gs + i];
}

// launch configuration of a program (attributes in `at`)
template <typename T>
cudaLaunchConfig_t cluster3_config(const Cluster3Layout &l, cudaStream_t s, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C3_RANKS);
    cfg.blockDim = dim3(C3_THREADS);
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
    return (size_t)l.stride + sizeof(T) * ((size_t)l.max_in + 2 * (size_t)l.max_gs + l.max_e + 29 * (size_t)l.max_g);
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
