// Learned initial guess (no counterpart in the paper): six dilated 3x3
// convolutions, 4 -> 32 -> 32 -> 32 -> 32 -> 32 -> 2 channels, ReLU after the
// first five, BF16 operands with FP32 accumulation on the tcgen05 tensor cores.
//
// Layout.  Images are zero-padded by P (the largest dilation) on every side
// and flattened: pixel q = (b * Hp + i) * Wp + j, Hp = H + 2P, Wp = W + 2P.
// A tensor of C channels is stored channel-group-major, [C/8][npix][8] BF16,
// so each group is an array of 16-byte pixel rows.  That is exactly the
// layout of one column of 8x16-byte core matrices of a K-major (pixels x
// channels) operand, and a tap of the stencil -- a shift of the pixel index
// by di*d*Wp + dj*d -- is a shift of the operand's start address by a whole
// number of 16-byte rows: the implicit GEMM needs no im2col copy.
//
// Tiles and chains.  A tile is 128 consecutive pixels of one image row (M =
// 128 of the MMAs).  With dilation d the tiles of rows i, i + d, i + 2d, ... in
// one column of tiles share their input rows: row i is tap row +1, 0 and -1 of
// three successive tiles.  A CTA therefore walks down such a chain with a ring
// of row segments of 128 + 2d pixels in shared memory (four to eight in the
// convolution, as shared memory allows; four of 128 in the weight gradients):
// each tile brings in one new segment (18.6 KB at d = 81) instead of three.
// Images much narrower than 128 pixels take tiles over their flattened rows, each
// with three segments of its own (cnn_tiles.h).
//
// Convolution (forward, and backward to the input): N = output channels, K =
// input channels in slices of 16, summed over the 9 taps.  Warp roles: a
// producer (bulk copies), an MMA issuer, four epilogue warps; four TMEM
// accumulators, so that loads, MMAs and epilogues of different tiles overlap.
// Weight gradients: D[slot, ci][tap column, co] = sum_q x[q][ci] dz[q - s][co]
// with the pixels as K, both operands MN-major; the 16 channel groups of the
// whole ring (4 slots x 4 groups) are the M = 128 rows of one MMA and three
// shifted copies of dz its N = 96 columns, so one MMA serves all nine taps.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "cnn_tiles.h"
#include "gcmg_cnn.h"

namespace {

using namespace gcmg_cnn_tiles;

constexpr int kLayers = 6;
constexpr int kCin[kLayers] = {4, 32, 32, 32, 32, 32};
constexpr int kCout[kLayers] = {32, 32, 32, 32, 32, 2};
constexpr int kMaxDil = 96;
constexpr int kRing = 4;              // row segments in shared memory (convolution: at least,
constexpr int kMaxRing = 8;           // and at most, see ConvArgs::ring)
constexpr int kAcc = 4;               // TMEM accumulators of the convolution
constexpr int kDzStages = 4;          // staged gradient tiles of the weight gradients
// a CTA's share of the bias gradients (an atomic to each of the same 32 words, 26
// ns) in tiles of the convolution (0.6 us)
constexpr double kDbCta = 1.0 / 20;
constexpr int kConvThreads = 192;     // producer, MMA issuer, four epilogue warps
constexpr long kWaitLimit = 1L << 22; // bounded mbarrier polls

// ------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor, no swizzle: start, leading-dimension and
// stride-dimension byte offsets (all >> 4), descriptor version 1
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// instruction descriptor of kind::f16: BF16 A and B, FP32 D, M x N, major-ness
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n, int a_mn, int b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// polls the barrier's phase with a bound; false if it never completed
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase) {
    for (long it = 0; it < kWaitLimit; it++) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

template <int NCOLS>
__device__ __forceinline__ void tmem_alloc(uint32_t slot) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(NCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int NCOLS>
__device__ __forceinline__ void tmem_free(uint32_t taddr) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(NCOLS) : "memory");
}

// 32 lanes x 16 / 32 consecutive FP32 columns of the accumulator
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat16 x = __float2bfloat16_rn(a), y = __float2bfloat16_rn(b);
    return (uint32_t)__bfloat16_as_ushort(x) | ((uint32_t)__bfloat16_as_ushort(y) << 16);
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// ------------------------------------------------------------ convolution
// MODE 0: y = bf16(relu(acc + bias)); 1: out[b][c][i][j] = acc + bias (c < 2);
// 2: y = bf16(acc * (gate > 0)) (backward to the input of the layer below) and
// db[c] += the sum of the stored values over the pixels
struct ConvArgs {
    const uint4 *x;       // [GIN][npix] pixel rows
    const uint4 *w;       // [9][GIN][NOUT] rows of 8 input channels
    const float *bias;    // NOUT
    uint4 *y;             // [NOUT / 8][npix]
    float *out;           // MODE 1: [B][2][H][W]
    const uint4 *gate;    // MODE 2: [NOUT / 8][npix]
    float *db;            // MODE 2: NOUT
    Geo geo;
    Tiles ch;
    int dil;
    int ring;             // segments in shared memory
    int *err;
};

// bulk copy of `bytes` (a multiple of 16) from global to shared memory,
// completing as transaction bytes on `mbar`
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(mbar)
        : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

// Positions number the segments a CTA loads, over all of its items; position p
// lies in ring slot p % ring.  Tile k of an item whose first segment has
// position p0 reads positions p0 + k, + 1, + 2 (tap rows -1, 0, +1).
// Every wait is bounded; after one that ran out (ok = false) a role waits no
// more, and the kernel reports it through a.err.
// Several CTAs an SM (TMEM columns, shared memory), each with ring - 3 segments
// in flight: three of six slots at small dilations, two of five at 81.
// Measured, 8 images of 513^2, 32 -> 32 channels, forward: 366 us a layer with
// three segments a tile, one accumulator and the border's tiles computed too;
// 76-94 us so (2.9-3.6 TB/s of activations read and written once).  Backward to
// the input 721 -> 101-123 us (reads the gate too).  Counters of a forward layer
// (4 images): shared memory 64 % (the operands, read again for each tap), tensor
// pipe 21 %, DRAM 31 %, L2 20 %.
template <int GIN, int NOUT, int MODE>
__global__ void __launch_bounds__(kConvThreads) k_conv(ConvArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int seg = kTile + 2 * a.dil;                            // pixels of a segment
    uint4 *sx = reinterpret_cast<uint4 *>(smem);                  // [ring][GIN][seg]
    uint4 *sw = sx + a.ring * GIN * seg;                           // 9 * GIN * NOUT rows
    uint64_t *bars = reinterpret_cast<uint64_t *>(sw + 9 * GIN * NOUT);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * kMaxRing + 2 * kAcc + 1);
    float *part = reinterpret_cast<float *>(tslot + 2);            // MODE 2: a warp's sums, NOUT each
    const uint32_t full = smem_u32(bars), empty = full + 8 * kMaxRing, afull = empty + 8 * kMaxRing,
                   afree = afull + 8 * kAcc, wbar = afree + 8 * kAcc;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 1) tmem_alloc<kAcc * NOUT>(smem_u32(tslot));
    if (threadIdx.x == 0) {
        for (int i = 0; i < a.ring; i++) {
            mbar_init(full + 8 * i, 1);
            mbar_init(empty + 8 * i, 1);
        }
        for (int i = 0; i < kAcc; i++) {
            mbar_init(afull + 8 * i, 1);
            mbar_init(afree + 8 * i, 4);   // one arrival an epilogue warp
        }
        mbar_init(wbar, 1);
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tslot;
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (ok) ok = mbar_wait(bar, parity & 1u);
    };
    TileItem it;

    if (warp == 0) {
        if (lane == 0) {   // producer
            mbar_expect(wbar, 9 * GIN * NOUT * 16);
            bulk_g2s(smem_u32(sw), a.w, 9 * GIN * NOUT * 16, wbar);
            int s = 0, round = 0, sent = 0;   // slot of the next position and how often the ring was filled
            for (int t = blockIdx.x; t < a.ch.items; t += gridDim.x) {
                if (!a.ch.item(a.geo, t, &it)) continue;
                // pixel of the first segment: dil rows and dil columns before the tile
                long q = it.q - (long)a.dil * a.geo.Wp - a.dil;
                for (int p = 0; p < it.cnt + 2; p++, q += (long)a.dil * a.geo.Wp) {
                    wait(empty + 8 * s, (uint32_t)round + 1u);
                    if (!ok) break;
                    mbar_expect(full + 8 * s, (uint32_t)(GIN * seg * 16));
                    for (int g = 0; g < GIN; g++)
                        bulk_g2s(smem_u32(sx + (s * GIN + g) * seg), a.x + (long)g * a.geo.gs + q, (uint32_t)(seg * 16),
                                 full + 8 * s);
                    sent = min(sent + 1, a.ring);
                    if (++s == a.ring) s = 0, round++;
                }
                if (!ok) break;
            }
            // every copy has landed before the CTA ends (in a complete run the
            // MMAs have waited for them already)
            for (; sent > 0; sent--) {
                if (--s < 0) s = a.ring - 1, round--;
                mbar_wait(full + 8 * s, (uint32_t)round & 1u);
            }
            mbar_wait(wbar, 0);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            constexpr uint32_t idesc = idesc_bf16(kTile, NOUT, 0, 0);
            const uint32_t xa = smem_u32(sx), wa = smem_u32(sw);
            int tile = 0;
            int s0 = 0, sn = 0, round = 0;   // slot of the tile's first position; of the next one to arrive
            auto after = [&](int i, int d) { return i + d < a.ring ? i + d : i + d - a.ring; };
            wait(wbar, 0);
            for (int t = blockIdx.x; t < a.ch.items && ok; t += gridDim.x) {
                if (!a.ch.item(a.geo, t, &it)) continue;
                for (int k = 0; k < it.cnt; k++, tile++) {
                    for (int p = k ? 2 : 0; p < 3; p++) {
                        wait(full + 8 * sn, (uint32_t)round);
                        if (++sn == a.ring) sn = 0, round++;
                    }
                    const int ac = tile % kAcc;
                    wait(afree + 8 * ac, (uint32_t)(tile / kAcc) + 1u);
                    if (!ok) break;
                    tc_after();
                    const uint32_t d = tmem + (uint32_t)(ac * NOUT);
                    uint32_t acc = 0;
#pragma unroll 1
                    for (int tr = 0; tr < 3; tr++) {
                        const uint32_t xs = xa + (uint32_t)(after(s0, tr) * GIN * seg) * 16;
#pragma unroll
                        for (int tc = 0; tc < 3; tc++)
#pragma unroll
                            for (int gp = 0; gp < GIN / 2; gp++) {
                                const uint64_t ad = sdesc(xs + (uint32_t)(2 * gp * seg + tc * a.dil) * 16, seg * 16, 128);
                                const uint64_t bd =
                                    sdesc(wa + (((tr * 3 + tc) * GIN + 2 * gp) * NOUT) * 16, NOUT * 16, 128);
                                mma_bf16(d, ad, bd, idesc, acc);
                                acc = 1;
                            }
                    }
                    mma_commit(afull + 8 * ac);
                    mma_commit(empty + 8 * s0);
                    if (k + 1 == it.cnt) {   // the item's last two segments serve no other tile
                        mma_commit(empty + 8 * after(s0, 1));
                        mma_commit(empty + 8 * after(s0, 2));
                        s0 = after(s0, 2);
                    }
                    s0 = after(s0, 1);
                }
            }
        }
        __syncwarp();
    } else {   // epilogue: warp w reads the TMEM lanes 32 (w % 4)
        const int ew = warp & 3;
        const uint32_t lane_addr = tmem + ((uint32_t)(ew * 32) << 16);
        float dbs[MODE == 2 ? NOUT : 1];
#pragma unroll
        for (int e = 0; e < (MODE == 2 ? NOUT : 1); e++) dbs[e] = 0.0f;
        float bias[MODE == 0 ? NOUT : 1];
        if (MODE == 0) {
#pragma unroll
            for (int e = 0; e < NOUT; e++) bias[MODE == 0 ? e : 0] = a.bias[e];
        }
        int tile = 0;
        for (int t = blockIdx.x; t < a.ch.items && ok; t += gridDim.x) {
            if (!a.ch.item(a.geo, t, &it)) continue;
            for (int k = 0; k < it.cnt && ok; k++, tile++) {
                int i, j;
                const bool in = a.ch.at(a.geo, it, k, ew * 32 + lane, &i, &j);
                const long q = it.q + (long)k * a.dil * a.geo.Wp + ew * 32 + lane;
                uint4 gt[MODE == 2 ? NOUT / 8 : 1];
                if (MODE == 2 && in) {
#pragma unroll
                    for (int g = 0; g < NOUT / 8; g++) gt[g] = a.gate[(long)g * a.geo.gs + q];
                }
                const int ac = tile % kAcc;
                wait(afull + 8 * ac, (uint32_t)(tile / kAcc));
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_after();
                float v[NOUT];
                tmem_ld16(lane_addr + (uint32_t)(ac * NOUT), v);
                if (NOUT == 32) tmem_ld16(lane_addr + (uint32_t)(ac * NOUT) + 16, v + 16);
                tc_before();   // the accumulator is read: the issuer may overwrite it
                __syncwarp();
                if (lane == 0) mbar_arrive(afree + 8 * ac);
                if (!in) continue;
                if (MODE == 1) {
                    for (int ch = 0; ch < 2; ch++)
                        a.out[(((size_t)it.b * 2 + ch) * a.geo.H + i) * a.geo.W + j] = v[ch] + a.bias[ch];
                } else {
#pragma unroll
                    for (int g = 0; g < NOUT / 8; g++) {
                        float o[8];
                        if (MODE == 0) {
#pragma unroll
                            for (int e = 0; e < 8; e++) o[e] = fmaxf(v[8 * g + e] + bias[MODE == 0 ? 8 * g + e : 0], 0.0f);
                        } else {
                            const uint32_t gw[4] = {gt[g].x, gt[g].y, gt[g].z, gt[g].w};
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                o[2 * e] = bf16_lo(gw[e]) > 0.0f ? v[8 * g + 2 * e] : 0.0f;
                                o[2 * e + 1] = bf16_hi(gw[e]) > 0.0f ? v[8 * g + 2 * e + 1] : 0.0f;
                            }
                        }
                        const uint32_t w[4] = {pack_bf16(o[0], o[1]), pack_bf16(o[2], o[3]), pack_bf16(o[4], o[5]),
                                               pack_bf16(o[6], o[7])};
                        if (MODE == 2) {
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                dbs[8 * g + 2 * e] += bf16_lo(w[e]);
                                dbs[8 * g + 2 * e + 1] += bf16_hi(w[e]);
                            }
                        }
                        a.y[(long)g * a.geo.gs + q] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
        }
        // one sum a CTA: the atomics of all CTAs go to the same NOUT words, one after
        // the other (16 images of 128 x 16, 456 CTAs: 63-72 us a layer with a sum a warp, 18 so)
        if (MODE == 2) {
#pragma unroll
            for (int e = 0; e < NOUT; e++) {
                float s = dbs[e];
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) part[ew * NOUT + e] = s;
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");   // the epilogue warps
            const int e = ew * 32 + lane;
            if (e < NOUT) atomicAdd(&a.db[e], (part[e] + part[NOUT + e]) + (part[2 * NOUT + e] + part[3 * NOUT + e]));
        }
    }
    if (!ok) atomicExch(a.err, 1);
    tc_before();
    __syncthreads();
    if (warp == 1) {
        tc_after();
        tmem_free<kAcc * NOUT>(tmem);
    }
}

// --------------------------------------------------------- weight gradient
// dw[co][ci][t] += sum over the CTA's tiles of x[q][ci] dz[q - s_t][co], with
// the chains of k_conv.  A ring slot holds one row's 128 pixels of x; a
// gradient tile is staged three times, shifted by the tap columns, so that one
// MMA multiplies all 4 slots x GB groups (M rows) of x by the 3 x 8 GA columns
// of the gradient (K = 16 pixels): the MMA's time is that of reading its A
// operand, whatever N.  A slot holds tap row (slot - first position) mod 4 of
// the tile, so the accumulators are kept per class = first position mod 4; the
// class's fourth slot (being loaded, or of the next item) yields rows nobody
// reads.  Pixels past the image's last column are staged as zeros.
// Measured, 8 images of 513^2: 2469 us a layer with a tap and 16 pixels an MMA
// and nothing staged ahead, 253 us with the ring and one MMA a tap column, 192
// us with one MMA for the three.  Counters (4 images): no unit is busy -- tensor
// pipe 10 %, its operand reads 11 %, shared memory 14 %, L2 13 %, DRAM 20 % -- and
// the SMs' shares are uneven (608 MMAs on one, 446 on average): waits within the one
// chain a CTA walks.  Three chains a CTA, each with a ring, and five gradient
// stages measured 225 us all the same; why is open.
struct DwArgs {
    const uint4 *dz;      // [GA][npix]
    const uint4 *x;       // [GB][npix]
    float *dw;            // [co][ci][9] of this layer (FP32, accumulated)
    int cout, cin;        // real channel counts
    Geo geo;
    Tiles ch;
    int dil;
    int *err;
};

template <int GA, int GB>
__global__ void __launch_bounds__(128, 1) k_conv_dw(DwArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int N = 3 * 8 * GA;                                 // (tap column, output channel)
    uint4 *sx = reinterpret_cast<uint4 *>(smem);                  // [kRing][GB][kTile], 16 groups readable
    uint4 *sz = sx + 16 * kTile;                                  // [kDzStages][3][GA][kTile]
    float *red = reinterpret_cast<float *>(sz + kDzStages * 3 * GA * kTile);   // [9][32 ci][32 co]
    uint64_t *bars = reinterpret_cast<uint64_t *>(red + 9 * 32 * 32);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 2 * kRing + 2 * kDzStages + 1);
    const uint32_t full = smem_u32(bars), empty = full + 8 * kRing, zfull = empty + 8 * kRing,
                   zempty = zfull + 8 * kDzStages, done = zempty + 8 * kDzStages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (warp == 1) tmem_alloc<512>(smem_u32(tslot));
    if (threadIdx.x == 0) {
        for (int i = 0; i < kRing; i++) {
            mbar_init(full + 8 * i, 1);
            mbar_init(empty + 8 * i, 1);
        }
        for (int i = 0; i < kDzStages; i++) {
            mbar_init(zfull + 8 * i, 1);
            mbar_init(zempty + 8 * i, 1);
        }
        mbar_init(done, 1);
    }
    for (int e = threadIdx.x; e < 9 * 32 * 32; e += blockDim.x) red[e] = 0.0f;
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = *tslot;
    bool ok = true;
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (ok) ok = mbar_wait(bar, parity & 1u);
    };
    TileItem it;
    unsigned used = 0;   // classes with an accumulator (the same in every thread)
    {
        int pos = 0;
        for (int t = blockIdx.x; t < a.ch.items; t += gridDim.x) {
            if (!a.ch.item(a.geo, t, &it)) continue;
            for (int k = 0; k < min(it.cnt, kRing); k++) used |= 1u << ((pos + k) % kRing);
            pos += it.cnt + 2;
        }
    }

    if (warp == 0) {   // producer (the whole warp: it zeroes the tail of a gradient tile)
        int pos = 0, tile = 0;
        for (int t = blockIdx.x; t < a.ch.items && ok; t += gridDim.x) {
            if (!a.ch.item(a.geo, t, &it)) continue;
            const int width = it.width, padded = (width + 15) & ~15;
            for (int p = 0; p < it.cnt + 2 && ok; p++, pos++) {
                const long q = it.q + (long)(p - 1) * a.dil * a.geo.Wp;
                const int s = pos % kRing;
                wait(empty + 8 * s, (uint32_t)(pos / kRing) + 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (lane == 0) {
                    mbar_expect(full + 8 * s, (uint32_t)(GB * kTile * 16));
                    for (int g = 0; g < GB; g++)
                        bulk_g2s(smem_u32(sx + (s * GB + g) * kTile), a.x + (long)g * a.geo.gs + q, kTile * 16,
                                 full + 8 * s);
                }
                if (p < 1 || p > it.cnt) continue;   // the gradient tile of this row
                const int z = tile % kDzStages;
                wait(zempty + 8 * z, (uint32_t)(tile / kDzStages) + 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    pos++;   // this position's segment is on its way
                    break;
                }
                for (int e = lane; e < 3 * GA * (padded - width); e += 32) {
                    const int g = e / (padded - width), r = width + e % (padded - width);
                    sz[(z * 3 * GA + g) * kTile + r] = make_uint4(0, 0, 0, 0);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_expect(zfull + 8 * z, (uint32_t)(3 * GA * width * 16));
                    for (int tc = 0; tc < 3; tc++)
                        for (int g = 0; g < GA; g++)
                            bulk_g2s(smem_u32(sz + ((z * 3 + tc) * GA + g) * kTile),
                                     a.dz + (long)g * a.geo.gs + q + (1 - tc) * a.dil, (uint32_t)(width * 16),
                                     zfull + 8 * z);
                }
                tile++;
            }
        }
        if (lane == 0) {   // every copy has landed before the CTA ends
            for (int p = max(0, pos - kRing); p < pos; p++) mbar_wait(full + 8 * (p % kRing), (uint32_t)(p / kRing) & 1u);
            for (int p = max(0, tile - kDzStages); p < tile; p++)
                mbar_wait(zfull + 8 * (p % kDzStages), (uint32_t)(p / kDzStages) & 1u);
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {   // MMA issuer
            constexpr uint32_t idesc = idesc_bf16(kTile, N, 1, 1);
            const uint32_t xa = smem_u32(sx), za = smem_u32(sz);
            int pos = 0, tile = 0;
            unsigned begun = 0;
            for (int t = blockIdx.x; t < a.ch.items && ok; t += gridDim.x) {
                if (!a.ch.item(a.geo, t, &it)) continue;
                const int steps = (it.width + 15) / 16;
                for (int k = 0; k < it.cnt; k++, tile++) {
                    for (int p = k ? pos + k + 2 : pos; p <= pos + k + 2; p++)
                        wait(full + 8 * (p % kRing), (uint32_t)(p / kRing));
                    const int z = tile % kDzStages, cls = (pos + k) % kRing;
                    wait(zfull + 8 * z, (uint32_t)(tile / kDzStages));
                    if (!ok) break;
                    tc_after();
#pragma unroll 1
                    for (int ks = 0; ks < steps; ks++) {
                        const uint64_t ad = sdesc(xa + (uint32_t)(16 * ks) * 16, 128, kTile * 16);
                        const uint64_t bd = sdesc(za + (uint32_t)(z * 3 * GA * kTile + 16 * ks) * 16, 128, kTile * 16);
                        mma_bf16(tmem + (uint32_t)(cls * N), ad, bd, idesc, (begun >> cls & 1u) | (ks > 0 ? 1u : 0u));
                    }
                    begun |= 1u << cls;
                    mma_commit(zempty + 8 * z);
                    mma_commit(empty + 8 * cls);
                    if (k + 1 == it.cnt) {
                        mma_commit(empty + 8 * ((pos + k + 1) % kRing));
                        mma_commit(empty + 8 * ((pos + k + 2) % kRing));
                    }
                }
                pos += it.cnt + 2;
            }
            mma_commit(done);
            if (!mbar_wait(done, 0)) ok = false;
        }
        __syncwarp();
    }
    if (!ok) atomicExch(a.err, 2);
    tc_before();
    const bool good = __syncthreads_and(ok);
    tc_after();
    if (good) {
        // M row 32 warp + lane is (slot, ci); in step s warp w adds tap row
        // (w + s) mod 4 of its slot (GB = 4): no two warps touch the same sums
        const int row = 32 * warp + lane, slot = row / (8 * GB), ci = row % (8 * GB);
        for (int s = 0; s < kRing; s++) {
            const int di = (warp + s) & 3;
            // GB = 2: a warp holds two slots, whose lanes take the same tap row one after the other
            for (int h = 0; h < 4 / GB; h++) {
                const int sl = GB == 4 ? warp : 2 * warp + h;   // warp uniform
                const int cls = (sl - di) & 3;
                if (sl < kRing && di < 3 && (used >> cls & 1u)) {
                    for (int tc = 0; tc < 3; tc++)
#pragma unroll
                        for (int c0 = 0; c0 < 8 * GA; c0 += 16) {
                            float v[16];
                            tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(cls * N + tc * 8 * GA + c0), v);
                            if (slot == sl)
#pragma unroll
                                for (int k = 0; k < 16; k++) red[((di * 3 + tc) * 32 + ci) * 32 + ((c0 + k + ci) & 31)] += v[k];
                        }
                }
                __syncwarp();
            }
            __syncthreads();
        }
        for (int e = threadIdx.x; e < a.cout * a.cin * 9; e += blockDim.x) {
            const int t = e % 9, ci = (e / 9) % a.cin, co = e / (9 * a.cin);
            atomicAdd(&a.dw[e], red[(t * 32 + ci) * 32 + ((co + ci) & 31)]);
        }
    }
    tc_before();
    __syncthreads();
    if (warp == 1) {
        tc_after();
        tmem_free<512>(tmem);
    }
}

// ---------------------------------------------------------- small kernels
// input [B][4][H][W] FP32 -> [2][npix] rows at the image pixels (channels
// 4..15 zero; the border and the second group are zero from the start)
__global__ void k_pack_input(const float *__restrict__ in, uint4 *__restrict__ x, Geo geo, int B) {
    const int plane = geo.H * geo.W, e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= plane) return;
    const int i = e / geo.W, j = e - i * geo.W;
    for (int b = blockIdx.y; b < B; b += gridDim.y) {
        float c[4];
#pragma unroll
        for (int k = 0; k < 4; k++) c[k] = in[((size_t)b * 4 + k) * plane + e];
        x[((size_t)b * geo.Hp + geo.P + i) * geo.Wp + geo.P + j] =
            make_uint4(pack_bf16(c[0], c[1]), pack_bf16(c[2], c[3]), 0, 0);
    }
}

// dL/dout [B][2][H][W] FP32 -> [2][npix] rows at the image pixels (channels
// 2..15 zero), and the bias gradient of the last layer: db[c] += sum of the
// rounded values
__global__ void __launch_bounds__(256) k_pack_dout(const float *__restrict__ d, uint4 *__restrict__ x, Geo geo, int B, float *db) {
    const int plane = geo.H * geo.W;
    float s0 = 0.0f, s1 = 0.0f;
    for (int b = blockIdx.y; b < B; b += gridDim.y)
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < plane; e += gridDim.x * blockDim.x) {
            const int i = e / geo.W, j = e - i * geo.W;
            const uint32_t w = pack_bf16(d[(size_t)b * 2 * plane + e], d[((size_t)b * 2 + 1) * plane + e]);
            const size_t q = ((size_t)b * geo.Hp + geo.P + i) * geo.Wp + geo.P + j;
            x[q] = make_uint4(w, 0, 0, 0);
            x[(size_t)geo.gs + q] = make_uint4(0, 0, 0, 0);
            s0 += bf16_lo(w);
            s1 += bf16_hi(w);
        }
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    __shared__ float part[2][8];
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = s0;
        part[1][threadIdx.x >> 5] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float t = 0.0f;
        for (int w = 0; w < 8; w++) t += part[threadIdx.x][w];
        atomicAdd(&db[threadIdx.x], t);
    }
}

// masked squared error of channel 0 ([B][2][plane] arrays): dout_0 = 2 (out_0 -
// t_0) m_0 / count, dout_1 = 0, loss += sum (out_0 - t_0)^2 m_0 / count
__global__ void k_mse(const float *__restrict__ out, const float *__restrict__ t, const float *__restrict__ m,
                      float *__restrict__ dout, size_t n, size_t plane, float inv_count, double *loss) {
    double s = 0.0;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const bool ch0 = (e / plane) % 2 == 0;
        const float df = ch0 ? (out[e] - t[e]) * m[e] : 0.0f;
        dout[e] = 2.0f * df * inv_count;
        s += (double)df * df;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) tot += part[w];
        atomicAdd(loss, tot * inv_count);
    }
}

// Residual term of the loss, two passes over [B][H][W]: e = (out_0 - t_0) m_0,
// s = e_N + e_S + e_E + e_W - 4 e where m_1 = 1 (inside the image edge), else
// 0; loss += beta sum s^2 / count; then dout_0 += 2 beta / count *
// (-4 s + s_N + s_S + s_E + s_W) m_0.
__global__ void k_lap_s(const float *__restrict__ out, const float *__restrict__ t, const float *__restrict__ m,
                        float *__restrict__ s, int B, int H, int W, float scale, double *loss) {
    const size_t plane = (size_t)H * W;
    double acc = 0.0;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)B * plane;
         e += (size_t)gridDim.x * blockDim.x) {
        const size_t b = e / plane, p = e - b * plane;
        const int i = (int)(p / W), j = (int)(p - (size_t)i * W);
        const float *o0 = out + b * 2 * plane, *t0 = t + b * 2 * plane, *m0 = m + b * 2 * plane;
        float v = 0.0f;
        if (i > 0 && i < H - 1 && j > 0 && j < W - 1 && m0[plane + p] > 0.0f) {
            auto err = [&](size_t q) { return (o0[q] - t0[q]) * m0[q]; };
            v = err(p - W) + err(p + W) + err(p - 1) + err(p + 1) - 4.0f * err(p);
        }
        s[e] = v;
        acc += (double)v * v;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) tot += part[w];
        atomicAdd(loss, tot * scale);
    }
}

__global__ void k_lap_grad(const float *__restrict__ s, const float *__restrict__ m, float *__restrict__ dout, int B,
                           int H, int W, float scale2) {
    const size_t plane = (size_t)H * W;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)B * plane;
         e += (size_t)gridDim.x * blockDim.x) {
        const size_t b = e / plane, p = e - b * plane;
        const int i = (int)(p / W), j = (int)(p - (size_t)i * W);
        float g = -4.0f * s[e];
        if (i > 0) g += s[e - W];
        if (i < H - 1) g += s[e + W];
        if (j > 0) g += s[e - 1];
        if (j < W - 1) g += s[e + 1];
        dout[b * 2 * plane + p] += scale2 * g * m[b * 2 * plane + p];
    }
}

// BF16 operand copies of one layer's FP32 weights w[co][ci][9]:
// forward rows  wf[t][g][co][8] = w[co][8g + k][t]            (GIN groups, NOUT rows)
// backward rows wb[t][g][ci][8] = w[8g + k][ci][8 - t]         (GOUT groups, 32 rows)
__global__ void k_prep_weights(const float *__restrict__ w, int cout, int cin, int gin, int nout, int gout,
                               uint16_t *__restrict__ wf, uint16_t *__restrict__ wb) {
    const int nf = 9 * gin * nout * 8, nb = wb ? 9 * gout * 32 * 8 : 0;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < nf + nb; e += gridDim.x * blockDim.x) {
        float val = 0.0f;
        if (e < nf) {
            const int k = e % 8, co = (e / 8) % nout, g = (e / (8 * nout)) % gin, t = e / (8 * nout * gin);
            const int ci = 8 * g + k;
            if (co < cout && ci < cin) val = w[((size_t)co * cin + ci) * 9 + t];
            wf[e] = __bfloat16_as_ushort(__float2bfloat16_rn(val));
        } else {
            const int f = e - nf;
            const int k = f % 8, ci = (f / 8) % 32, g = (f / 256) % gout, t = f / (256 * gout);
            const int co = 8 * g + k;
            if (co < cout && ci < cin) val = w[((size_t)co * cin + ci) * 9 + (8 - t)];
            wb[f] = __bfloat16_as_ushort(__float2bfloat16_rn(val));
        }
    }
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const float gi = g[e];
    const float mi = b1 * m[e] + (1.0f - b1) * gi;
    const float vi = b2 * v[e] + (1.0f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    p[e] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

// ------------------------------------------------------------------ context
struct gcmg_cnn {
    int batch = 0, H = 0, W = 0, P = 0;
    int dil[kLayers] = {1, 3, 9, 27, 81, 1};
    Geo geo{};
    cudaStream_t stream = nullptr;
    int device = 0;
    int64_t nparams = 0;
    int64_t woff[kLayers] = {}, boff[kLayers] = {};
    float *p = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;   // FP32 master, gradient, Adam moments
    uint16_t *wf[kLayers] = {}, *wb[kLayers] = {};
    uint4 *act[kLayers] = {};    // act[0] = packed input, act[l] = output of layer l (l = 1..5)
    uint4 *dz[2] = {};           // ping-pong gradients
    float *out = nullptr, *dout = nullptr, *lap_s = nullptr;
    double *d_loss = nullptr;
    int *d_err = nullptr;
    int adam_t = 0;
    int sms = 148;
    size_t guard = 0;            // zero rows before and after each channel group
    size_t smem_sm = 0;          // shared memory of an SM
    size_t smem_cta = 0;         // of a CTA at most
    std::string err;
    std::vector<void *> allocs;
};

namespace {

struct Fail {
    gcmg_status s;
    std::string m;
};

void ck(cudaError_t e, const char *what) {
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw Fail{GCMG_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e)};
    }
}

template <typename T>
T *alloc(gcmg_cnn *c, size_t n) {
    void *p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        throw Fail{GCMG_E_OOM, "device allocation failed"};
    }
    c->allocs.push_back(p);
    return static_cast<T *>(p);
}

int groups_in(int l) { return l == 0 ? 2 : 4; }
int nout_of(int l) { return l == kLayers - 1 ? 16 : 32; }

// shared memory of the convolution: the ring, the weights, the barriers, the epilogue warps' sums
size_t conv_smem(int gin, int nout, int dil, int ring) {
    return (size_t)(ring * gin * (kTile + 2 * dil) + 9 * gin * nout) * 16 + (2 * kMaxRing + 2 * kAcc + 2) * 8 + 16 * nout;
}
// of the weight gradients: 16 channel groups of x (the MMA's M rows), the
// staged gradients, the reduction buffer, the barriers; the kernel holds 512
// TMEM columns, so it asks for enough to sit alone on an SM
size_t dw_smem(int ga) {
    const size_t need = (size_t)(16 * kTile + kDzStages * 3 * ga * kTile) * 16 + 9 * 32 * 32 * 4 + 24 * 16;
    return std::max(need, (size_t)120 * 1024);
}

#define CNN_GUARD(c, ...)                                             \
    try {                                                             \
        __VA_ARGS__                                                   \
    } catch (const Fail &f) {                                         \
        if (c) (c)->err = f.m;                                        \
        return f.s;                                                   \
    }

void check_err(gcmg_cnn *c) {
    int e = 0;
    ck(cudaMemcpyAsync(&e, c->d_err, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "err");
    ck(cudaStreamSynchronize(c->stream), "sync");
    if (e) throw Fail{GCMG_E_TIMEOUT, "a tensor-core wait ran out (code " + std::to_string(e) + ")"};
}

void prep_weights(gcmg_cnn *c) {
    for (int l = 0; l < kLayers; l++) {
        const int gout = l == kLayers - 1 ? 2 : 4;
        k_prep_weights<<<64, 256, 0, c->stream>>>(c->p + c->woff[l], kCout[l], kCin[l], groups_in(l), nout_of(l),
                                                  gout, c->wf[l], c->wb[l]);
    }
    ck(cudaGetLastError(), "prep weights");
}

template <int GIN, int NOUT, int MODE>
void launch_conv(gcmg_cnn *c, ConvArgs a) {
    // resident CTAs an SM: shared memory (1 KB each is the system's), TMEM columns
    auto resident = [&](int ring) {
        const size_t smem = conv_smem(GIN, NOUT, a.dil, ring);
        return smem > c->smem_cta ? 0 : std::min({(int)(c->smem_sm / (smem + 1024)), 512 / (kAcc * NOUT), 4});
    };
    // the ring with the most segments in flight an SM of those that leave three
    // CTAs there (or what the smallest ring leaves, if fewer): a forward pass of 8
    // images of 513^2 takes 550 us with rings of 4, 509 so, 567 with two CTAs
    a.ring = kRing;
    const int least = std::min(3, resident(kRing));
    for (int r = kRing + 1; r <= kMaxRing; r++)
        if (resident(r) >= least && resident(r) * (r - 3) > resident(a.ring) * (a.ring - 3)) a.ring = r;
    const size_t smem = conv_smem(GIN, NOUT, a.dil, a.ring);
    const int per_sm = std::max(1, resident(a.ring));
    a.ch = make_tiles(c->geo, c->batch, a.dil, c->sms, per_sm, MODE == 2 ? kDbCta : 0.0);
    k_conv<GIN, NOUT, MODE><<<(unsigned)a.ch.grid, kConvThreads, smem, c->stream>>>(a);
    ck(cudaGetLastError(), "conv launch");
}

template <int GA, int GB>
void launch_dw(gcmg_cnn *c, DwArgs d) {
    d.ch = make_tiles(c->geo, c->batch, d.dil, c->sms, 1, 0.0);
    k_conv_dw<GA, GB><<<(unsigned)d.ch.grid, 128, dw_smem(GA), c->stream>>>(d);
    ck(cudaGetLastError(), "dw launch");
}

void forward(gcmg_cnn *c, const float *in, float *out) {
    const Geo g = c->geo;
    const unsigned images = (unsigned)std::min(c->batch, 65535);
    k_pack_input<<<dim3((unsigned)((c->H * c->W + 255) / 256), images), 256, 0, c->stream>>>(in, c->act[0], g, c->batch);
    for (int l = 0; l < kLayers; l++) {
        ConvArgs a{};
        a.x = c->act[l];
        a.w = reinterpret_cast<const uint4 *>(c->wf[l]);
        a.bias = c->p + c->boff[l];
        a.geo = g;
        a.dil = c->dil[l];
        a.err = c->d_err;
        if (l == 0) {
            a.y = c->act[1];
            launch_conv<2, 32, 0>(c, a);
        } else if (l < kLayers - 1) {
            a.y = c->act[l + 1];
            launch_conv<4, 32, 0>(c, a);
        } else {
            a.out = out;
            launch_conv<4, 16, 1>(c, a);
        }
    }
}

// parameter gradients into c->grad for dL/dout = dout (c->dout layout [B][2][H][W])
void backward(gcmg_cnn *c, const float *dout) {
    const Geo g = c->geo;
    ck(cudaMemsetAsync(c->grad, 0, c->nparams * sizeof(float), c->stream), "memset");
    const int plane = c->H * c->W;
    k_pack_dout<<<dim3((unsigned)std::min((plane + 255) / 256, std::max(1, 8 * c->sms / c->batch)),
                       (unsigned)std::min(c->batch, 65535)),
                  256, 0, c->stream>>>(dout, c->dz[0], g, c->batch, c->grad + c->boff[kLayers - 1]);
    int cur = 0;
    for (int l = kLayers - 1; l >= 0; l--) {
        const int ga = l == kLayers - 1 ? 2 : 4;
        DwArgs d{};
        d.dz = c->dz[cur];
        d.x = c->act[l];
        d.dw = c->grad + c->woff[l];
        d.cout = kCout[l];
        d.cin = kCin[l];
        d.geo = g;
        d.dil = c->dil[l];
        d.err = c->d_err;
        if (ga == 2) launch_dw<2, 4>(c, d);
        else if (l == 0) launch_dw<4, 2>(c, d);
        else launch_dw<4, 4>(c, d);
        if (l == 0) break;
        ConvArgs a{};
        a.x = c->dz[cur];
        a.w = reinterpret_cast<const uint4 *>(c->wb[l]);
        a.y = c->dz[cur ^ 1];
        a.gate = c->act[l];
        a.db = c->grad + c->boff[l - 1];
        a.geo = g;
        a.dil = c->dil[l];
        a.err = c->d_err;
        if (ga == 2) launch_conv<2, 32, 2>(c, a);
        else launch_conv<4, 32, 2>(c, a);
        cur ^= 1;
    }
}

}  // namespace

extern "C" {

int64_t gcmg_cnn_num_params(void) {
    int64_t n = 0;
    for (int l = 0; l < kLayers; l++) n += (int64_t)kCout[l] * kCin[l] * 9 + kCout[l];
    return n;
}

gcmg_status gcmg_cnn_create(int batch, int H, int W, const int *dilations, void *stream, gcmg_cnn **out) {
    if (!out) return GCMG_E_ARG;
    *out = nullptr;
    if (batch < 1 || H < 1 || W < 1) return GCMG_E_ARG;
    gcmg_cnn *c = new (std::nothrow) gcmg_cnn;
    if (!c) return GCMG_E_OOM;
    *out = c;
    if (dilations)
        for (int l = 0; l < kLayers; l++) {
            if (dilations[l] < 1 || dilations[l] > kMaxDil) {
                c->err = "dilations must lie in [1, 96]";
                return GCMG_E_ARG;
            }
            c->dil[l] = dilations[l];
        }
    int P = 0;
    for (int l = 0; l < kLayers; l++) P = std::max(P, c->dil[l]);
    const double npix = (double)batch * (H + 2 * P) * (W + 2 * P);
    if (npix >= 2.0e9) {
        c->err = "too many pixels";
        return GCMG_E_ARG;
    }
    c->batch = batch;
    c->H = H;
    c->W = W;
    c->P = P;
    // guard rows: the furthest tap of the last pixel of a tile, on either side
    c->guard = (size_t)P * (W + 2 * P) + P + kTile;
    c->geo = Geo{(int)npix, H + 2 * P, W + 2 * P, H, W, P, (int)((size_t)npix + 2 * c->guard)};
    c->stream = (cudaStream_t)stream;
    CNN_GUARD(c, {
        ck(cudaGetDevice(&c->device), "cudaGetDevice");
        int64_t off = 0;
        for (int l = 0; l < kLayers; l++) {
            c->woff[l] = off;
            off += (int64_t)kCout[l] * kCin[l] * 9;
            c->boff[l] = off;
            off += kCout[l];
        }
        c->nparams = off;
        c->p = alloc<float>(c, off);
        c->grad = alloc<float>(c, off);
        c->m = alloc<float>(c, off);
        c->v = alloc<float>(c, off);
        ck(cudaMemset(c->p, 0, off * sizeof(float)), "memset");
        ck(cudaMemset(c->m, 0, off * sizeof(float)), "memset");
        ck(cudaMemset(c->v, 0, off * sizeof(float)), "memset");
        for (int l = 0; l < kLayers; l++) {
            c->wf[l] = alloc<uint16_t>(c, (size_t)9 * groups_in(l) * nout_of(l) * 8);
            if (l > 0) c->wb[l] = alloc<uint16_t>(c, (size_t)9 * (l == kLayers - 1 ? 2 : 4) * 32 * 8);
        }
        ck(cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device), "attr");
        const size_t gs = (size_t)c->geo.gs;
        // each buffer: G groups of gs rows; the pointer skips the first guard
        c->act[0] = alloc<uint4>(c, 2 * gs) + c->guard;
        for (int l = 1; l < kLayers; l++) c->act[l] = alloc<uint4>(c, 4 * gs) + c->guard;
        c->dz[0] = alloc<uint4>(c, 4 * gs) + c->guard;
        c->dz[1] = alloc<uint4>(c, 4 * gs) + c->guard;
        c->out = alloc<float>(c, (size_t)batch * 2 * H * W);
        c->dout = alloc<float>(c, (size_t)batch * 2 * H * W);
        c->lap_s = alloc<float>(c, (size_t)batch * H * W);
        c->d_loss = alloc<double>(c, 1);
        c->d_err = alloc<int>(c, 1);
        ck(cudaMemset(c->d_err, 0, sizeof(int)), "memset");
        int most = 0, per_sm = 0;
        ck(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device), "attr");
        ck(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, c->device), "attr");
        c->smem_sm = (size_t)per_sm;
        c->smem_cta = (size_t)most;
        const auto allow = [&](auto *kernel) {
            ck(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most), "attr");
        };
        allow(k_conv<2, 32, 0>);
        allow(k_conv<4, 32, 0>);
        allow(k_conv<4, 16, 1>);
        allow(k_conv<2, 32, 2>);
        allow(k_conv<4, 32, 2>);
        allow(k_conv_dw<2, 4>);
        allow(k_conv_dw<4, 4>);
        allow(k_conv_dw<4, 2>);
        // zero every activation once: borders and guards stay zero from then on
        for (int l = 0; l < kLayers; l++) ck(cudaMemset(c->act[l] - c->guard, 0, (l ? 4 : 2) * gs * 16), "memset");
        ck(cudaMemset(c->dz[0] - c->guard, 0, 4 * gs * 16), "memset");
        ck(cudaMemset(c->dz[1] - c->guard, 0, 4 * gs * 16), "memset");
        return GCMG_OK;
    })
}

void gcmg_cnn_destroy(gcmg_cnn *c) {
    if (!c) return;
    for (void *p : c->allocs) cudaFree(p);
    delete c;
}

const char *gcmg_cnn_last_error(const gcmg_cnn *c) { return c ? c->err.c_str() : "null network"; }

gcmg_status gcmg_cnn_set_params(gcmg_cnn *c, const float *p_host, int64_t count) {
    if (!c || !p_host || count != c->nparams) return GCMG_E_ARG;
    CNN_GUARD(c, {
        ck(cudaMemcpyAsync(c->p, p_host, count * sizeof(float), cudaMemcpyHostToDevice, c->stream), "params");
        ck(cudaMemsetAsync(c->m, 0, count * sizeof(float), c->stream), "memset");
        ck(cudaMemsetAsync(c->v, 0, count * sizeof(float), c->stream), "memset");
        c->adam_t = 0;
        prep_weights(c);
        ck(cudaStreamSynchronize(c->stream), "sync");
        return GCMG_OK;
    })
}

gcmg_status gcmg_cnn_get_params(gcmg_cnn *c, float *p_host, int64_t count) {
    if (!c || !p_host || count != c->nparams) return GCMG_E_ARG;
    CNN_GUARD(c, {
        ck(cudaMemcpyAsync(p_host, c->p, count * sizeof(float), cudaMemcpyDeviceToHost, c->stream), "params");
        ck(cudaStreamSynchronize(c->stream), "sync");
        return GCMG_OK;
    })
}

gcmg_status gcmg_cnn_forward(gcmg_cnn *c, const float *in_dev, float *out_dev) {
    if (!c || !in_dev || !out_dev) return GCMG_E_ARG;
    CNN_GUARD(c, {
        forward(c, in_dev, out_dev);
        check_err(c);
        return GCMG_OK;
    })
}

gcmg_status gcmg_cnn_activation(gcmg_cnn *c, int layer, float *dst_dev) {
    if (!c || !dst_dev || layer < 0 || layer >= kLayers) return GCMG_E_ARG;
    CNN_GUARD(c, {
        // unpack [G][npix][8] BF16 -> [B][C][H][W] FP32 on the host side of the stream
        const int G = layer == 0 ? 2 : 4, C = layer == 0 ? 4 : 32;
        const size_t np = (size_t)c->geo.npix;
        std::vector<uint16_t> h((size_t)G * np * 8);
        for (int g = 0; g < G; g++)
            ck(cudaMemcpyAsync(h.data() + (size_t)g * np * 8, c->act[layer] + (size_t)g * c->geo.gs, np * 16,
                               cudaMemcpyDeviceToHost, c->stream),
               "act");
        ck(cudaStreamSynchronize(c->stream), "sync");
        std::vector<float> o((size_t)c->batch * C * c->H * c->W);
        for (int b = 0; b < c->batch; b++)
            for (int ch = 0; ch < C; ch++)
                for (int i = 0; i < c->H; i++)
                    for (int j = 0; j < c->W; j++) {
                        const size_t q = ((size_t)b * c->geo.Hp + i + c->P) * c->geo.Wp + j + c->P;
                        const uint32_t bits = (uint32_t)h[((size_t)(ch / 8) * np + q) * 8 + ch % 8] << 16;
                        float f;
                        std::memcpy(&f, &bits, 4);
                        o[(((size_t)b * C + ch) * c->H + i) * c->W + j] = f;
                    }
        ck(cudaMemcpyAsync(dst_dev, o.data(), o.size() * 4, cudaMemcpyHostToDevice, c->stream), "act");
        ck(cudaStreamSynchronize(c->stream), "sync");
        return GCMG_OK;
    })
}

gcmg_status gcmg_cnn_backward(gcmg_cnn *c, const float *dout_dev, float *grad_dev) {
    if (!c || !dout_dev || !grad_dev) return GCMG_E_ARG;
    CNN_GUARD(c, {
        backward(c, dout_dev);
        ck(cudaMemcpyAsync(grad_dev, c->grad, c->nparams * sizeof(float), cudaMemcpyDeviceToDevice, c->stream),
           "grad");
        check_err(c);
        return GCMG_OK;
    })
}

gcmg_status gcmg_cnn_train_step(gcmg_cnn *c, const float *in_dev, const float *target_dev, const float *mask_dev,
                                float mask_count, float lap_weight, float lap_count, float lr, double *loss_host) {
    if (!c || !in_dev || !target_dev || !mask_dev || !(mask_count > 0.0f) || lap_weight < 0.0f ||
        (lap_weight > 0.0f && !(lap_count > 0.0f)))
        return GCMG_E_ARG;
    CNN_GUARD(c, {
        forward(c, in_dev, c->out);
        ck(cudaMemsetAsync(c->d_loss, 0, sizeof(double), c->stream), "memset");
        const size_t n = (size_t)c->batch * 2 * c->H * c->W;
        k_mse<<<256, 256, 0, c->stream>>>(c->out, target_dev, mask_dev, c->dout, n, (size_t)c->H * c->W,
                                          1.0f / mask_count, c->d_loss);
        if (lap_weight > 0.0f) {
            k_lap_s<<<256, 256, 0, c->stream>>>(c->out, target_dev, mask_dev, c->lap_s, c->batch, c->H, c->W,
                                                lap_weight / lap_count, c->d_loss);
            k_lap_grad<<<256, 256, 0, c->stream>>>(c->lap_s, mask_dev, c->dout, c->batch, c->H, c->W,
                                                   2.0f * lap_weight / lap_count);
        }
        backward(c, c->dout);
        c->adam_t++;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.0f - std::pow(b1, (float)c->adam_t), c2 = 1.0f - std::pow(b2, (float)c->adam_t);
        k_adam<<<(unsigned)((c->nparams + 255) / 256), 256, 0, c->stream>>>(c->p, c->grad, c->m, c->v,
                                                                           (int)c->nparams, lr, b1, b2, 1e-8f, c1, c2);
        prep_weights(c);
        double loss = 0.0;
        ck(cudaMemcpyAsync(&loss, c->d_loss, sizeof(double), cudaMemcpyDeviceToHost, c->stream), "loss");
        check_err(c);
        if (loss_host) *loss_host = loss;
        return GCMG_OK;
    })
}

}  // extern "C"
