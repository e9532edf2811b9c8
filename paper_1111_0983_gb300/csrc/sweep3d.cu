// Band sweeps of the larger 3D levels, one launch a sweep.  A launch a phase
// (red, black, ghosts) costs three launches and three round trips to L2 a sweep;
// here a block runs the whole sweep in shared memory, updating besides its own
// nodes the inside nodes of other blocks that its updates read (about as many
// again; no ghost twice, whose 27-point update is the dear one), and the launch
// boundary exchanges the values through compact arrays.  What bounds it: latency of
// the phases, and L2, which a launch reads its whole program from (257^3: 116 MB
// through L2 a launch, records with their padding, weights and values, 24 % of its
// rate over the 15 us of a cold launch, up to 60 % over the 6 us of one in a solve).
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

constexpr int S3_THREADS = 256;

// xin: compact values of the updated inside nodes (null: from u), gin: the
// ghosts' values; xout, gout: where the own new values go (null: into u, which
// the launch then reads at nodes that no block updates only)
template <typename T>
__global__ void __launch_bounds__(S3_THREADS) k_sweep3(LevelView<T> v, Sweep3Layout L,
                                                       const uint8_t *__restrict__ records,
                                                       const T *__restrict__ xin, const T *__restrict__ gin,
                                                       T *__restrict__ xout, T *__restrict__ gout) {
    extern __shared__ __align__(16) unsigned char smem_s3[];
    if (sizeof(T) == 4) pdl_trigger();
    const int tid = threadIdx.x, nt = S3_THREADS;
    unsigned char *rec = smem_s3;
    T *val = reinterpret_cast<T *>(rec + L.stride);   // max_in, max_gs
    T *sf = val + L.max_in + L.max_gs;                // f of the entries
    // the block's record, then through it the weights: fixed, read before the wait
    const uint8_t *src = records + (size_t)blockIdx.x * L.stride;
    for (int i = tid * 16; i < L.stride; i += nt * 16) cp_async16(rec + i, src + i);
    cp_async_wait_all();
    __syncthreads();
    const int *h = reinterpret_cast<const int *>(rec);
    const int32_t *node = reinterpret_cast<const int32_t *>(rec + L.node);
    const int32_t *cid = reinterpret_cast<const int32_t *>(rec + L.cid);
    const int32_t *gslot = reinterpret_cast<const int32_t *>(rec + L.gslot);
    const uint4 *ent = reinterpret_cast<const uint4 *>(rec + L.ent);
    const uint4 *gst = reinterpret_cast<const uint4 *>(rec + L.gst);
    const int nin = h[S3_NIN], ngs = h[S3_NGS], own_in = h[S3_OWN_IN], own_g = h[S3_OWN_G];
    const int red = h[S3_RED], ne = h[S3_NE];
    T w[27], gc = 0, gg = 0;
    int q = -1;
    if (tid < own_g) {   // the thread's first ghost
        q = gslot[tid];
        gc = v.gc[q];
#pragma unroll
        for (int k = 0; k < 27; k++) w[k] = v.gw[(int64_t)k * v.ng + q];
    }
    pdl_wait();
    for (int i = tid; i < nin; i += nt) {
        const int c = xin ? cid[i] : -1;
        cp_async(&val[i], c >= 0 ? &xin[c] : &v.u[node[i]]);
    }
    for (int i = tid; i < ngs; i += nt) cp_async(&val[L.max_in + i], &gin[gslot[i]]);
    for (int e = tid; e < ne; e += nt) cp_async(&sf[e], &v.f[node[ent[e].x & 0xffffu]]);
    if (q >= 0) gg = v.gg[q];
    cp_async_wait_all();
    __syncthreads();
    // Gauss-Seidel form of Eq. (jac2d), 7 points: the sums of k_rb_list in the same order
    auto inside = [&](int e0, int e1) {
        for (int e = e0 + tid; e < e1; e += nt) {
            const uint4 r = ent[e];
            T nb = val[r.x >> 16] + val[r.y & 0xffffu] + val[r.y >> 16] + val[r.z & 0xffffu];
            nb += val[r.z >> 16] + val[r.w & 0xffffu];
            val[r.x & 0xffffu] = (mul_rn(v.h2, sf[e]) + nb) * (T)(1.0 / 6.0);
        }
    };
    inside(0, red);
    __syncthreads();
    inside(red, ne);
    __syncthreads();
    const int base = h[S3_BASE];
    for (int i = tid; i < own_in; i += nt) {
        if (xout) xout[base + i] = val[i];
        else v.u[node[i]] = val[i];
    }
    // Eqs. (dir2d)/(neu2d) at the own ghosts: all of them read the old ghost values
    auto ghost = [&](int e, int qe, const T *we, int64_t stride, T gce, T gge) {
        T s = 0;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const uint4 r = gst[c * L.max_g + e];
            const unsigned x[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int k = 0; k < 8; k++)
                if (8 * c + k < 27)
                    s += we[(8 * c + k) * stride] * val[(k & 1) ? x[k / 2] >> 16 : x[k / 2] & 0xffffu];
        }
        const T y = val[L.max_in + e] + gce * (gge - s);
        if (gout) gout[qe] = y;
        else v.u[v.gnode[qe]] = y;
    };
    if (q >= 0) ghost(tid, q, w, 1, gc, gg);
    for (int e = tid + nt; e < own_g; e += nt) {
        const int qe = gslot[e];
        ghost(e, qe, &v.gw[qe], v.ng, v.gc[qe], v.gg[qe]);
    }
}

}  // namespace

template <typename T>
size_t sweep3_smem(const Sweep3Layout &l) {
    return (size_t)l.stride + sizeof(T) * ((size_t)l.max_in + (((size_t)l.max_gs + 1) & ~(size_t)1) + l.max_e);
}

template <typename T>
bool sweep3_fits(const Sweep3Layout &l, int device) {
    int most = 0;
    if (cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        sweep3_smem<T>(l) > (size_t)most)
        return false;
    if (cudaFuncSetAttribute(k_sweep3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

template <typename T>
void launch_sweep3(const LevelView<T> &v, const Sweep3Dev &P, int lambda, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P.lay.blocks);
    cfg.blockDim = dim3(S3_THREADS);
    cfg.dynamicSmemBytes = sweep3_smem<T>(P.lay);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    T *x[2] = {(T *)P.x[0], (T *)P.x[1]}, *g[2] = {v.gtmp, (T *)P.g};
    for (int k = 0; k < lambda; k++) {
        const bool last = k + 1 == lambda;
        g_launches++;
        ck(cudaLaunchKernelEx(&cfg, k_sweep3<T>, v, P.lay, (const uint8_t *)P.records,
                              (const T *)(k == 0 ? nullptr : x[(k - 1) & 1]), (const T *)g[k & 1],
                              last ? (T *)nullptr : x[k & 1], last ? (T *)nullptr : g[(k + 1) & 1]),
           "sweep launch");
    }
}

template size_t sweep3_smem<float>(const Sweep3Layout &);
template size_t sweep3_smem<double>(const Sweep3Layout &);
template bool sweep3_fits<float>(const Sweep3Layout &, int);
template bool sweep3_fits<double>(const Sweep3Layout &, int);
template void launch_sweep3<float>(const LevelView<float> &, const Sweep3Dev &, int, cudaStream_t);
template void launch_sweep3<double>(const LevelView<double> &, const Sweep3Dev &, int, cudaStream_t);

}  // namespace gcmg
