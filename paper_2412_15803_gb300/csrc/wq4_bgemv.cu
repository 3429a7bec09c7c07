// wq4_bgemv.cu -- the fused dequantize x GEMV for several activation rows: one
// decode step of a serving batch through one projection (Section 3, Table 1).
// It takes batch 5-32, batch 2-4 but for few long rows (and batch 2 below 8 Mi
// weights), rows that bulk copies cannot take from the sizes on where its ring
// wins (cuda_cores and copy_ring, wq4_gemv.cu), and wq4_gemm's calls of up to 16
// tokens.
//
// y[b][n] = fp16( sum_k (q(n,k) - 7) * s[n][k/32] * x[b][k] )
//
// The contraction runs on mma.sync m16n8k16: per 32-code group two MMAs add the
// group's exact fp16 products (q - 7) x in fp32, and the group's scales multiply
// the fp32 result into the running sums, so no weight is ever rounded and every
// fp16 scale is valid.  (tcgen05 would need the scale inside the fp16 operand,
// or one accumulator per group.)  A CTA owns tiles of weight rows; its warps
// are row groups times slices of every K chunk, and the slices' sums are added
// in slice order in shared memory at the tile's end: the same inputs give the
// same bits.  The next tile's chunks are in flight while a tile is finished.
//
// Two kernels:
//  * bgemv_tma_kernel (K % 256 == 0, 16-byte aligned scales): the tile loop of
//    wq4_tiles.cuh, weights as the MMA's 16 rows, chunks by tensor copies.
//  * bgemv_kernel (other rows): activations as the 16 rows and eight weight rows
//    as the columns, 16 warps, chunks of KG groups through a four-stage cp.async
//    ring, rows padded so that ldmatrix of the codes and the 16-byte loads of
//    the activations are free of bank conflicts.
//
// Measured (us a launch in a graph over copies of 520 MB, before: CUDA-core
// kernels that read the activations through L1): 3072 x 8192 batch 8 76.5 ->
// 6.9, 16384 x 3072 batch 8 100 -> 8.8 and batch 32 387 -> 17.4, 128256 x 4096
// batch 8 927 -> 54.7 (5.4 TB/s) and batch 32 3739 -> 119; 1003 x 2080 (copy
// ring) batch 5 7.3 -> 4.5.  Up to batch 8 the wide shapes are bound by
// instruction issue and HBM together, at batch 32 by the MMAs (two per tile,
// group and eight activation rows) and their issue; the narrow ones by the
// launch and a chunk's latency.
#include "wq4.h"
#include "wq4_device.cuh"
#include "wq4_host.h"
#include "wq4_items.cuh"
#include "wq4_tc.cuh"
#include "wq4_tiles.cuh"

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

namespace wq4 {
namespace {

constexpr int kBWarps = 16;
constexpr int kBThreads = kBWarps * 32;
constexpr int kBStages = 4;
constexpr int kScaleRegs = 4;      // scales a thread carries per chunk (S2)

struct BGemvParams {
    const uint32_t* W;
    const uint16_t* s;
    const uint16_t* x;
    uint16_t* y;
    int N, K, batch;
    int lkg;               // log2 of the groups per chunk
    int ks, gpw;           // K slices, groups of a chunk per slice (even)
    int tiles, nch;        // row tiles, chunks along K
    uint32_t stage_bytes, scale_off, x_off, red_off;
    int y4;                // two outputs may be stored at once
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Copies `bytes` (0 or 16) bytes and fills the rest of the 16 with zeros.
__device__ __forceinline__ void cp_async16z(uint32_t dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// XT: tiles of eight activation rows (batch <= 8 XT); R: tiles of eight
// weight rows per warp; S2: scales at any 2-byte address (else copied in
// 4-byte aligned pairs).
template <int XT, int R, bool S2>
__global__ void __launch_bounds__(kBThreads, 1) bgemv_kernel(const BGemvParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int MT = (XT + 1) / 2;                  // MMA row blocks of 16 activation rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, c = lane & 3;
    const int KG = 1 << p.lkg, G = p.K >> 5;
    const int ks = p.ks, rgs = kBWarps / ks, TR = 8 * R * rgs;
    const int rg = warp / ks, sl = warp - rg * ks;    // row group and K slice of this warp
    const uint32_t cpitch = 16u * KG + 16u, spitch = 2u * KG + 16u, xpitch = 64u * KG + 64u;
    const uint32_t smem0 = smem_addr(smem);
    const int mytiles = (p.tiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
    const int total = mytiles * p.nch;

    // ---- chunk loads: this thread's place in each copy is fixed; the row
    // advances by a constant step
    int lc = 0, ln0 = static_cast<int>(blockIdx.x) * TR, lstage = 0;
    [[maybe_unused]] uint16_t sreg[S2 ? kScaleRegs : 1];
    [[maybe_unused]] uint32_t sdst = 0;                                // stage the carried scales belong to
    [[maybe_unused]] int sng = 0;
    const size_t wrow = static_cast<size_t>(G) * 16, srow = static_cast<size_t>(G) * 2;
    const int crow = tid >> p.lkg, ccol = tid & (KG - 1), cstep = kBThreads >> p.lkg;
    constexpr int kLsg = S2 ? 0 : 1;                  // log2 of the scales per copy
    const int lsu = p.lkg - kLsg;                     // log2 of the scale copies per row
    const int qrow = tid >> lsu, qcol = (tid & ((1 << lsu) - 1)) << kLsg, qstep = kBThreads >> lsu;
    const int xrow = tid >> (p.lkg + 2), xcol = tid & (4 * KG - 1), xstep = kBThreads >> (p.lkg + 2);
    auto issue_w = [&](int stage, int n0, int ch) {
        const uint32_t base = smem0 + stage * p.stage_bytes;
        const int g0 = ch << p.lkg, ng = min(KG, G - g0), last = p.N - 1 - n0;   // rows past N repeat the last
        if (ccol < ng) {
            const uint8_t* src = reinterpret_cast<const uint8_t*>(p.W) + static_cast<size_t>(n0) * wrow + 16 * (g0 + ccol);
            uint32_t dst = base + crow * cpitch + 16 * ccol;
            for (int row = crow; row < TR; row += cstep, dst += cstep * cpitch)
                cp_async16(dst, src + static_cast<size_t>(min(row, last)) * wrow);
        }
        const uint8_t* src = reinterpret_cast<const uint8_t*>(p.s) + static_cast<size_t>(n0) * srow + 2 * (g0 + qcol);
        if constexpr (!S2) {
            if (qcol < ng) {
                uint32_t dst = base + p.scale_off + qrow * spitch + 2 * qcol;
                for (int row = qrow; row < TR; row += qstep, dst += qstep * spitch)
                    cp_async4(dst, src + static_cast<size_t>(min(row, last)) * srow);
            }
        } else {
            // scales at any 2-byte address: through registers, stored one chunk later
#pragma unroll
            for (int q = 0; q < kScaleRegs; ++q) {
                const int row = qrow + q * qstep;
                if (row < TR && qcol < ng)
                    sreg[q] = __ldg(reinterpret_cast<const uint16_t*>(src + static_cast<size_t>(min(row, last)) * srow));
            }
            sdst = base + p.scale_off + qrow * spitch + 2 * qcol;
            sng = ng;
        }
    };
    auto flush_scales = [&]() {
        if constexpr (S2) {
#pragma unroll
            for (int q = 0; q < kScaleRegs; ++q) {
                // an odd last group is paired with one of scale 0
                if (qrow + q * qstep < TR && qcol < ((sng + 1) & ~1))
                    asm volatile("st.shared.b16 [%0], %1;" ::"r"(sdst + q * qstep * spitch),
                                 "h"(qcol < sng ? sreg[q] : static_cast<uint16_t>(0))
                                 : "memory");
            }
            sng = 0;
        }
    };
    auto issue_x = [&](int stage, int ch) {
        const int g0 = ch << p.lkg, ng = min(KG, G - g0), xg = xcol >> 2;
        if (xg >= ((ng + 1) & ~1)) return;
        const uint32_t bytes = xg < ng ? 16u : 0u;     // an odd last group is paired with one of zeros
        const uint8_t* src = reinterpret_cast<const uint8_t*>(p.x) + 64 * static_cast<size_t>(g0) + (xg < ng ? 16 * xcol : 0);
        uint32_t dst = smem0 + stage * p.stage_bytes + p.x_off + xrow * xpitch + 16 * xcol;
        for (int row = xrow; row < 8 * XT; row += xstep, dst += xstep * xpitch)   // rows past the batch repeat the last
            cp_async16z(dst, src + static_cast<size_t>(min(row, p.batch - 1)) * (2 * static_cast<size_t>(p.K)), bytes);
    };
    auto advance = [&]() {
        if (++lc == p.nch) {
            lc = 0;
            ln0 += static_cast<int>(gridDim.x) * TR;
        }
        lstage = (lstage + 1) & (kBStages - 1);
    };

    // weights of the first chunks may be fetched while the previous kernel of
    // the stream finishes; activations only after it (programmatic dependent
    // launch).  The next kernel may begin then, and not before: it may fetch
    // weights that a kernel before this one wrote.
    {
        int c1 = 0, n1 = ln0;
        for (int i = 0; i < kBStages - 1 && i < total; ++i) {
            issue_w(i, n1, c1);
            flush_scales();
            if (++c1 == p.nch) {
                c1 = 0;
                n1 += static_cast<int>(gridDim.x) * TR;
            }
        }
    }
    grid_dependency_wait();
    grid_dependents_launch();
    for (int i = 0; i < kBStages - 1; ++i) {
        if (i < total) {
            issue_x(lstage, lc);
            advance();
        }
        cp_commit();
    }

    // ---- this lane's shared-memory offsets within a stage
    const int m = lane >> 3, lr = lane & 7;           // ldmatrix: matrix and row of this lane's address
    uint32_t coff;
    if (R == 1) coff = (8 * rg + lr) * cpitch + 16 * (m & 1);                          // groups j, j + 1
    else if (R == 2) coff = (16 * rg + 8 * (m & 1) + lr) * cpitch + 16 * (m >> 1);     // 2 tiles x 2 groups
    else coff = (8 * R * rg + 8 * min(m, R - 1) + lr) * cpitch;                        // R tiles of one group
    const uint32_t soff = p.scale_off + (8 * R * rg + 2 * c) * spitch;
    const uint32_t xoff = p.x_off + g * xpitch + 16 * c;
    const int j0 = sl * p.gpw;

    float acc[R][XT][2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int t = 0; t < XT; ++t) acc[r][t][0] = acc[r][t][1] = 0.f;

    int ch = 0, stage = 0, n0 = static_cast<int>(blockIdx.x) * TR;
    for (int f = 0; f < total; ++f) {
        cp_wait<kBStages - 2>();
        __syncthreads();
        flush_scales();                                // of chunk f + 2: read three barriers after its load
        if (f + kBStages - 1 < total) {
            issue_w(lstage, ln0, lc);
            issue_x(lstage, lc);
            advance();
        }
        cp_commit();

        const uint32_t base = smem0 + stage * p.stage_bytes;
        const int ng = min(KG, G - (ch << p.lkg));
        const int jend = min(j0 + p.gpw, ng);           // whole pairs: an odd last group has a zero partner
        for (int j = j0; j < jend; j += 2) {
            uint32_t sc0[R], sc1[R];                   // scales of groups j, j + 1: rows 2c and 2c + 1
#pragma unroll
            for (int r = 0; r < R; ++r) {
                sc0[r] = lds_u32(base + soff + (8 * r) * spitch + 2 * j);
                sc1[r] = lds_u32(base + soff + (8 * r + 1) * spitch + 2 * j);
            }
            uint32_t w[2][R > 2 ? 4 : 2];
            if (R == 1) {
                ldsm_x2(base + coff + 16 * j, w[0][0], w[1][0]);
            } else if (R == 2) {
                uint32_t t[4];
                ldsm_x4(base + coff + 16 * j, t);
                w[0][0] = t[0];
                w[0][1] = t[1];
                w[1][0] = t[2];
                w[1][1] = t[3];
            } else {
                ldsm_x4(base + coff + 16 * j, w[0]);
                ldsm_x4(base + coff + 16 * j + 16, w[1]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint4 v[2 * MT];
#pragma unroll
                for (int t = 0; t < XT; ++t) v[t] = pair_permute(lds_v4(base + xoff + (8 * t) * xpitch + 64 * (j + h)));
                if (XT & 1) v[XT] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    uint32_t q[4];
                    unpack_word(w[h][r], q);
                    const float s0 = h ? hi_f(sc0[r]) : lo_f(sc0[r]), s1 = h ? hi_f(sc1[r]) : lo_f(sc1[r]);
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        float d[4] = {0.f, 0.f, 0.f, 0.f};
                        mma_acc(d, v[2 * mt].x, v[2 * mt + 1].x, v[2 * mt].y, v[2 * mt + 1].y, q[0], q[1]);
                        mma_acc(d, v[2 * mt].z, v[2 * mt + 1].z, v[2 * mt].w, v[2 * mt + 1].w, q[2], q[3]);
                        acc[r][2 * mt][0] = fmaf(s0, d[0], acc[r][2 * mt][0]);
                        acc[r][2 * mt][1] = fmaf(s1, d[1], acc[r][2 * mt][1]);
                        if (2 * mt + 1 < XT) {
                            acc[r][2 * mt + 1 < XT ? 2 * mt + 1 : 0][0] = fmaf(s0, d[2], acc[r][2 * mt + 1 < XT ? 2 * mt + 1 : 0][0]);
                            acc[r][2 * mt + 1 < XT ? 2 * mt + 1 : 0][1] = fmaf(s1, d[3], acc[r][2 * mt + 1 < XT ? 2 * mt + 1 : 0][1]);
                        }
                    }
                }
            }
        }
        stage = (stage + 1) & (kBStages - 1);
        if (++ch < p.nch) continue;

        // ---- the tile is complete: lane (g, c) holds rows 8 r + 2c, + 1 of
        // its row group for batch rows 8 t + g
        auto store = [&](int row, int b, float v0, float v1) {
            const int n = n0 + row;
            if (b >= p.batch || n >= p.N) return;
            uint16_t* out = p.y + static_cast<size_t>(b) * p.N + n;
            const uint16_t h0 = float_to_half_bits(v0), h1 = float_to_half_bits(v1);
            if (p.y4) {
                *reinterpret_cast<uint32_t*>(out) = pack2(h0, h1);   // N even, n even
            } else {
                out[0] = h0;
                if (n + 1 < p.N) out[1] = h1;
            }
        };
        if (ks == 1) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int t = 0; t < XT; ++t) store(8 * (R * rg + r) + 2 * c, 8 * t + g, acc[r][t][0], acc[r][t][1]);
        } else {
            float2* red = reinterpret_cast<float2*>(smem + p.red_off);   // [warp][r][t][lane]
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int t = 0; t < XT; ++t)
                    red[((warp * R + r) * XT + t) * 32 + lane] = make_float2(acc[r][t][0], acc[r][t][1]);
            __syncthreads();
            // slices added in order; the next tile's sums are stored only
            // after a later barrier
            for (int e = tid; e < rgs * R * XT * 32; e += kBThreads) {
                const int ln = e & 31, q = e >> 5;                       // q = (row group, r, t)
                const int t = q % XT, qr = q / XT;
                const int r = qr % R, grp = qr / R;
                const float2* src = red + ((grp * ks * R + r) * XT + t) * 32 + ln;
                float2 sum = src[0];
                for (int k = 1; k < ks; ++k) {
                    const float2 o = src[k * R * XT * 32];
                    sum.x += o.x;
                    sum.y += o.y;
                }
                store(8 * (R * grp + r) + 2 * (ln & 3), 8 * t + (ln >> 2), sum.x, sum.y);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int t = 0; t < XT; ++t) acc[r][t][0] = acc[r][t][1] = 0.f;
        ch = 0;
        n0 += static_cast<int>(gridDim.x) * TR;
    }
    cp_wait<0>();
}

// ------------------------------------------------- tensor-copy kernel --
//
// Rows that tensor copies can take: the tile loop of wq4_tiles.cuh.
struct TGemvParams {
    TileGeom g;
    uint16_t* y;
    int N, batch;
    int y4;                // two outputs may be stored at once
    int check;             // a call of wq4_gemm: flag scales beyond +-8188, copy weights after the previous kernel
    uint32_t* err;
};

// Stores one tile of `wrows` rows a warp from row n0 on.
template <int XT, int R>
__device__ __forceinline__ void store_tile(const TGemvParams& p, float* red, int ks, int wrows, int n0, int tid, int warp,
                                           int lane, const float (&acc)[R][XT][4])
{
    constexpr int NW = kTWarps<XT>, kConsumers = 32 * NW;
    if (ks == 1) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int t = 0; t < XT; ++t)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = 16 * r + (lane >> 2) + 8 * (i >> 1), n = n0 + warp * wrows + row;
                    const int b = 8 * t + x_row(2 * (lane & 3) + (i & 1));
                    if (row < wrows && n < p.N && b < p.batch)
                        p.y[static_cast<size_t>(b) * p.N + n] = float_to_half_bits(acc[r][t][i]);
                }
        return;
    }
    store_sums<XT, R>(red, warp, lane, acc);
    named_barrier_sync(1, kConsumers);
    const int rgs = NW / ks, hrows = wrows >> 1;                 // pairs of rows per row group
    for (int e = tid; e < rgs * hrows * 8 * XT; e += kConsumers) {
        const int pr = e % hrows, q = e / hrows;                 // row pair; column and row group
        const int col = q % (8 * XT), grp = q / (8 * XT);
        const float2 sum = load_sums<XT, R>(red, grp, ks, col, 2 * pr);
        const int n = n0 + grp * wrows + 2 * pr, b = (col & ~7) + x_row(col & 7);
        if (b < p.batch && n < p.N) {
            uint16_t* out = p.y + static_cast<size_t>(b) * p.N + n;
            const uint16_t h0 = float_to_half_bits(sum.x), h1 = float_to_half_bits(sum.y);
            if (p.y4) {
                *reinterpret_cast<uint32_t*>(out) = pack2(h0, h1);   // N even, n even
            } else {
                out[0] = h0;
                if (n + 1 < p.N) out[1] = h1;
            }
        }
    }
    named_barrier_sync(1, kConsumers);                           // the sums' buffer is free again
}

// The CTA's tail, from row `row0` of the tails on: the last round's rows in
// tiles of 16 a warp, when one round of those takes them (128256 x 4096 is 3.3
// rounds of 256 rows).  A function of its own, so that the whole tiles' loop
// keeps its registers.
template <int XT>
__device__ __noinline__ bool tail_tile(const TGemvParams& p, uint8_t* smem, int tid, int row0, int slot, int par, bool ok)
{
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    TileGeom g = p.g;
    g.wrows = 16;
    TileWarp<XT, 1, false> tl(g, smem, tid >> 5, tid & 31);
    tl.slot = slot;
    tl.par = par;
    tl.ok = ok;
    float acc[1][XT][4];
    tl.tile(g, full, full + kTMaxSlots, p.check != 0, p.err, acc);
    store_tile<XT, 1>(p, reinterpret_cast<float*>(smem + g.red_off), g.ks, 16,
                      row0 + static_cast<int>(blockIdx.x) * 16 * (kTWarps<XT> / g.ks), tid, tid >> 5, tid & 31, acc);
    return tl.bad;
}

// The call's tensor maps: weights, scales, activations, and the tails' weights and
// scales where there are any.
template <bool TAIL>
struct TMaps {
    CUtensorMap m[TAIL ? 5 : 3];
};

template <int XT, int R, bool TAIL>
__global__ void __launch_bounds__(32 * (kTWarps<XT> + 1), 1)
    bgemv_tma_kernel(const __grid_constant__ TMaps<TAIL> t, const __grid_constant__ TGemvParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int NW = kTWarps<XT>, kConsumers = 32 * NW;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + kTMaxSlots;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ks = p.g.ks, wrows = p.g.wrows, rgs = NW / ks, TR = wrows * rgs;

    if (tid == kConsumers) {
        for (int i = 0; i < p.g.nslots; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NW);
        }
        mbar_fence_init();
    }
    __syncthreads();
    if (warp == NW) {
        if (lane == 0)
            tile_producer<XT, false, TAIL>(&t.m[0], &t.m[1], &t.m[2], &t.m[TAIL ? 3 : 0], &t.m[TAIL ? 4 : 1], p.g, 0, smem, full, empty, p.err, XT <= 2 && p.check);
        return;
    }

    grid_dependency_wait();               // y is written after the previous kernel
    grid_dependents_launch();             // ... and the next one may fetch weights that a kernel before this one wrote
    TileWarp<XT, R, false> tw(p.g, smem, warp, lane);
    {
        float acc[R][XT][4];
        for (int tile = blockIdx.x; tile < p.g.tiles; tile += gridDim.x) {
            tw.tile(p.g, full, empty, p.check != 0, p.err, acc);
            // (the operands of the call decide the loop's registers: at 17-24 rows
            // the first form is 5 % faster, 128256 x 4096 at 24 104 -> 99 us, at 25-32
            // the second 4 %)
            float* red = reinterpret_cast<float*>(smem + p.g.red_off);
            if constexpr (XT == 3)
                store_tile<XT, R>(p, red, p.g.ks, p.g.wrows, tile * TR, tid, tid >> 5, tid & 31, acc);
            else
                store_tile<XT, R>(p, red, ks, wrows, tile * TR, tid, warp, lane, acc);
        }
    }
    if constexpr (TAIL) {
        if (static_cast<int>(blockIdx.x) < p.g.tails)
            tw.bad = tail_tile<XT>(p, smem, tid, p.g.tiles * TR, tw.slot, tw.par, tw.ok) || tw.bad;
    }
    // a warp that gave up has not seen every copy land, but the producer waits
    // for them before it leaves
    if (tw.bad) atomicOr(p.err, kErrScale);
}

// ----------------------------------------------------------------- host --

struct BPlan {
    int R = 0, ks = 0, lkg = 0, tiles = 0, nch = 0;
    uint32_t stage_bytes = 0, scale_off = 0, x_off = 0, red_off = 0;
    size_t smem = 0;
};

// Tiles per warp, K slices and chunk length: the least estimated SM cycles.
// Per chunk the larger of the instructions of a scheduler's four warps, the
// MMA time (one m16n8k16 per two cycles and SM) and the copies at 50 bytes
// per cycle, plus a barrier; per tile the slices' sum.
bool plan_bgemv(int sms, size_t smem_max, int N, int K, int XT, bool s2, BPlan* best)
{
    const int G = K / 32, MT = (XT + 1) / 2;
    double best_c = 0.0;
    for (int R = 1; R <= 4; ++R)
        for (int ks = 1; ks <= kBWarps; ks *= 2)
            for (int lkg = 3; lkg <= 5; ++lkg) {
                const int KG = 1 << lkg, gpw = KG / ks;
                if (gpw < 2) continue;
                const int rgs = kBWarps / ks, TR = 8 * R * rgs;
                if (s2 && (R > 2 || TR * KG > kScaleRegs * kBThreads)) continue;
                BPlan q;
                q.R = R;
                q.ks = ks;
                q.lkg = lkg;
                q.scale_off = static_cast<uint32_t>(TR * (16 * KG + 16));
                q.x_off = static_cast<uint32_t>(align_up(q.scale_off + TR * (2 * KG + 16), 16));
                q.stage_bytes = static_cast<uint32_t>(align_up(q.x_off + 8 * XT * (64 * KG + 64), 128));
                q.red_off = q.stage_bytes * kBStages;
                q.smem = q.red_off + (ks > 1 ? static_cast<size_t>(kBWarps) * R * XT * 256 : 0);
                if (q.smem > smem_max) continue;
                q.tiles = (N + TR - 1) / TR;
                q.nch = (G + KG - 1) / KG;
                const int rounds = (q.tiles + sms - 1) / sms;
                const double instr = gpw * (5.0 * XT + 4 + R * (13.0 + 2 * MT + 2 * XT)) + 20.0 +
                                     (TR * KG * 1.5 + 32.0 * XT * KG) / kBThreads * 8.0;
                const double mma = static_cast<double>(kBWarps) * gpw * R * 2 * MT * 2.0;
                const double copy = (TR * 18.0 * KG + 512.0 * XT * KG) / 50.0;
                const double chunk = std::max(std::max(4.6 * instr, mma), copy) + 150.0;
                const double cost = rounds * (q.nch * chunk + (ks > 1 ? 150.0 + 20.0 * R * XT : 30.0 * R)) + 1500.0;
                if (best->R == 0 || cost < best_c) {
                    best_c = cost;
                    *best = q;
                }
            }
    return best->R != 0;
}

template <int XT, int R, bool S2>
cudaError_t launch_one(const cudaLaunchConfig_t& cfg, const BGemvParams& p, const DeviceInfo* di)
{
    static std::atomic<bool> ready[kMaxDevices];       // setting the attribute twice is harmless
    if (!ready[di->dev].load()) {
        const cudaError_t e =
            cudaFuncSetAttribute(bgemv_kernel<XT, R, S2>, cudaFuncAttributeMaxDynamicSharedMemorySize, di->smem_optin);
        if (e != cudaSuccess) return e;
        ready[di->dev].store(true);
    }
    return cudaLaunchKernelEx(&cfg, bgemv_kernel<XT, R, S2>, p);
}

template <int XT>
cudaError_t launch_xt(int R, bool s2, const cudaLaunchConfig_t& cfg, const BGemvParams& p, const DeviceInfo* di)
{
    if (s2) return R == 1 ? launch_one<XT, 1, true>(cfg, p, di) : launch_one<XT, 2, true>(cfg, p, di);
    switch (R) {
        case 1: return launch_one<XT, 1, false>(cfg, p, di);
        case 2: return launch_one<XT, 2, false>(cfg, p, di);
        case 3: return launch_one<XT, 3, false>(cfg, p, di);
        default: return launch_one<XT, 4, false>(cfg, p, di);
    }
}

template <int XT, int R, bool TAIL>
cudaError_t launch_tma(const cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const TGemvParams& p, const DeviceInfo* di)
{
    static std::atomic<bool> ready[kMaxDevices];       // setting the attribute twice is harmless
    if (!ready[di->dev].load()) {
        const cudaError_t e =
            cudaFuncSetAttribute(bgemv_tma_kernel<XT, R, TAIL>, cudaFuncAttributeMaxDynamicSharedMemorySize, di->smem_optin);
        if (e != cudaSuccess) return e;
        ready[di->dev].store(true);
    }
    TMaps<TAIL> t;
    std::copy(tm, tm + (TAIL ? 5 : 3), t.m);
    return cudaLaunchKernelEx(&cfg, bgemv_tma_kernel<XT, R, TAIL>, t, p);
}

template <int XT>
cudaError_t launch_tma_xt(int R, const cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const TGemvParams& p, const DeviceInfo* di)
{
    if constexpr (XT == 4)
        if (p.g.tails != 0) return launch_tma<XT, 2, true>(cfg, tm, p, di);    // one slice: 32 rows a warp at most
    if (R == 1) return launch_tma<XT, 1, false>(cfg, tm, p, di);
    if constexpr (XT != 2)
        if (R == 3) return launch_tma<XT, 3, false>(cfg, tm, p, di);
    return launch_tma<XT, 2, false>(cfg, tm, p, di);
}

// The launch shape of a GEMV's sizes, kept by this thread for its next call of
// the same ones: the search takes 0.7 us.  (Host time of a small batch 3-4 call:
// 3.6 us on the CUDA-core kernel, 4.7 here with a search a call, 3.9 now; the
// rest is three tensor maps, which hold the call's pointers.)
const TilePlan* gemv_plan(const DeviceInfo* di, int N, int K, int XT)
{
    struct Kept {
        int N = 0, K = 0, XT = 0, sms = 0, smem = 0;
        TilePlan plan;
    };
    thread_local Kept kept[64];
    const uint32_t h = (static_cast<uint32_t>(N) * 2654435761u) ^ (static_cast<uint32_t>(K / 256 * 4 + XT) * 2246822519u);
    Kept& k = kept[h >> 26];
    if (k.N != N || k.K != K || k.XT != XT || k.sms != di->sm_count || k.smem != di->smem_optin) {
        k = Kept{};
        if (!tile_plan(di->sm_count, static_cast<size_t>(di->smem_optin), N, K, XT, false, 0, &k.plan)) return nullptr;
        k.N = N;
        k.K = K;
        k.XT = XT;
        k.sms = di->sm_count;
        k.smem = di->smem_optin;
    }
    return &k.plan;
}

int launch_bgemv_tma(const DeviceInfo* di, const uint32_t* W, const uint16_t* s, const uint16_t* x, uint16_t* y, int N,
                     int K, int batch, bool check_scales, cudaStream_t stream)
{
    const int XT = (batch + 7) / 8;
    const TilePlan* plan = gemv_plan(di, N, K, XT);
    CUtensorMap tm[5];
    if (!plan || !tile_maps(tm, W, s, x, N, K, batch, K, XT, *plan, false)) return WQ4_ERR_CUDA;
    const TilePlan& b = *plan;
    TGemvParams p;
    p.g = b.g;
    p.y = y;
    p.N = N;
    p.batch = batch;
    p.y4 = (N % 2) == 0 && aligned(y, 4);
    p.check = check_scales ? 1 : 0;
    p.err = di->status;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b.grid);
    cfg.blockDim = dim3(32 * ((XT <= 2 ? kTWarps<1> : kTWarps<4>) + 1));
    cfg.dynamicSmemBytes = b.smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    switch (XT) {
        case 1: e = launch_tma_xt<1>(b.R, cfg, tm, p, di); break;
        case 2: e = launch_tma_xt<2>(b.R, cfg, tm, p, di); break;
        case 3: e = launch_tma_xt<3>(b.R, cfg, tm, p, di); break;
        default: e = launch_tma_xt<4>(b.R, cfg, tm, p, di); break;
    }
    return e == cudaSuccess ? WQ4_OK : WQ4_ERR_CUDA;
}

}  // namespace

// Per chunk the largest of the instructions of a scheduler's warps, the copies
// and the time a copy takes to land over the ring's depth; per round the sums of
// the slices.  Fitted to every choice over eight shapes of the 3B and 8B
// projections at batch 8, 16, 24 and 32 (times within 20 %, the choice 0.4 %
// from the best on average, at most 5 %).
bool tile_plan(int sms, size_t smem_max, int N, int K, int XT, bool stage, size_t extra, TilePlan* out)
{
    const int G = K / 32, NW = XT <= 2 ? kTWarps<1> : kTWarps<4>;
    double best = 0.0;
    out->R = 0;
    // (three row tiles on 16 warps only for a GEMV of up to eight rows: 28672 x
    // 4096 16.6 -> 15.2 us, 5120 x 3072 4.96 -> 4.31 at batch 8; with 9-16 rows
    // they spill, 128256 x 4096 75 -> 90, and the stages gain nothing)
    const int max_rows = NW == 8 || (XT == 1 && !stage) ? 48 : 32;
    for (int wrows = stage ? 16 : 8; wrows <= max_rows; wrows += stage ? 16 : 8)
        for (int ks = stage ? 2 : 1; ks <= NW; ks *= 2)
            for (int lkg = 3; lkg <= 5; ++lkg) {
                const int KG = 1 << lkg, gpw = KG / ks, boxes = KG / 8, R = (wrows + 15) / 16;
                if (gpw < 2 || gpw > 8) continue;
                const int rgs = NW / ks, TR = wrows * rgs;
                if (TR > (stage ? 128 : 256)) continue;
                TileGeom g;
                g.K = K;
                g.wrows = wrows;
                g.ks = ks;
                g.gpw = gpw;
                g.lkg = lkg;
                g.scale_off = static_cast<uint32_t>(boxes * TR * 128);
                g.x_off = static_cast<uint32_t>(align_up(g.scale_off + boxes * TR * 16, 1024));
                g.slot_bytes = g.x_off + boxes * XT * 4096;
                const size_t red = (ks > 1 ? static_cast<size_t>(NW) * 8 * XT * (16 * R + 4) * 4 : 0) + extra;
                if (smem_max < kTHeader + red) continue;
                const int nslots = static_cast<int>((smem_max - kTHeader - red) / g.slot_bytes);
                if (nslots < 3) continue;
                g.nslots = std::min(nslots, kTMaxSlots);
                g.red_off = kTHeader + g.nslots * g.slot_bytes;
                g.tiles = (N + TR - 1) / TR;
                g.nch = (G + KG - 1) / KG;
                int rounds = (g.tiles + sms - 1) / sms;
                auto round_cost = [&](int r, int rows) {
                    const double instr = gpw * (9.0 * XT + 2 + r * (22.0 + 13 * XT)) + 60.0;
                    const double copy = (rows * 18.0 * KG + 512.0 * XT * KG) / (NW == 16 ? 48.0 : 96.0);
                    const double chunk = std::max(std::max((NW == 16 ? 4.4 : 3.0) * instr, copy), 2200.0 / g.nslots);
                    return g.nch * chunk + (ks > 1 ? 900.0 + 130.0 * r * XT : 80.0 * r);
                };
                double cost = 0.0;
                // whole rounds, then a round of 16 rows a warp if that takes the rest
                // (25-32 activation rows, one slice, three whole rounds: 128256 x 4096 at
                // batch 32 129 -> 118 us; with fewer rows, with slices or after one round,
                // 45000 x 4096, a partial round of whole tiles was up to 10 % faster)
                g.tails = 0;
                const int rest = N - (rounds - 1) * sms * TR, TR2 = 16 * rgs;
                if (!stage && XT == 4 && ks == 1 && R > 1 && rounds > 3 && rest <= sms * TR2) {
                    --rounds;
                    g.tiles = rounds * sms;
                    g.tails = (rest + TR2 - 1) / TR2;
                    cost += round_cost(1, TR2);
                }
                cost += rounds * round_cost(R, TR);
                if (XT == 3 && R == 3) cost *= 1.05;               // measured slower than the model's time
                if (out->R == 0 || cost < best) {
                    best = cost;
                    out->g = g;
                    out->R = R;
                    out->grid = std::min(g.tiles, sms);
                    out->smem = g.red_off + red;
                }
            }
    return out->R != 0;
}

bool tile_maps(CUtensorMap tm[5], const uint32_t* W, const uint16_t* s, const uint16_t* x, int N, int K, int rows,
               int64_t x_pitch, int XT, const TilePlan& p, bool gu)
{
    const int NW = XT <= 2 ? kTWarps<1> : kTWarps<4>;
    const uint32_t TR = p.g.wrows * (NW / p.g.ks), TB = gu ? TR / 2 : TR, boxes = 1u << (p.g.lkg - 3);
    const uint64_t Ku = static_cast<uint64_t>(K), Nu = static_cast<uint64_t>(N);
    tm[3] = tm[4] = CUtensorMap{};
    if (p.g.tails != 0) {
        const uint32_t T2 = 16 * (NW / p.g.ks);
        if (!encode_tensor_map_3d(&tm[3], CU_TENSOR_MAP_DATA_TYPE_UINT8, W, {128, Nu, Ku / 256}, {Ku / 2, 128},
                                  {128, T2, boxes}, CU_TENSOR_MAP_SWIZZLE_128B) ||
            !encode_tensor_map_3d(&tm[4], CU_TENSOR_MAP_DATA_TYPE_UINT16, s, {8, Nu, Ku / 256}, {Ku / 16, 16},
                                  {8, T2, boxes}, CU_TENSOR_MAP_SWIZZLE_NONE))
            return false;
    }
    return encode_tensor_map_3d(&tm[0], CU_TENSOR_MAP_DATA_TYPE_UINT8, W, {128, Nu, Ku / 256}, {Ku / 2, 128},
                                {128, TB, boxes}, CU_TENSOR_MAP_SWIZZLE_128B) &&
           encode_tensor_map_3d(&tm[1], CU_TENSOR_MAP_DATA_TYPE_UINT16, s, {8, Nu, Ku / 256}, {Ku / 16, 16},
                                {8, TB, boxes}, CU_TENSOR_MAP_SWIZZLE_NONE) &&
           encode_tensor_map_3d(&tm[2], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x, {64, static_cast<uint64_t>(rows), Ku / 64},
                                {static_cast<uint64_t>(x_pitch) * 2, 128}, {64, static_cast<uint32_t>(8 * XT), 4 * boxes},
                                CU_TENSOR_MAP_SWIZZLE_128B);
}

int launch_bgemv(const DeviceInfo* di, const uint32_t* W, const uint16_t* s, const uint16_t* x, uint16_t* y, int N,
                 int K, int batch, cudaStream_t stream, bool check_scales)
{
    if ((K % 256) == 0 && aligned(s, 16)) return launch_bgemv_tma(di, W, s, x, y, N, K, batch, check_scales, stream);
    const int XT = (batch + 7) / 8;
    BGemvParams p;
    const bool s2 = (K % 64) != 0 || !aligned(s, 4);
    BPlan b;
    if (!plan_bgemv(di->sm_count, static_cast<size_t>(di->smem_optin), N, K, XT, s2, &b)) return WQ4_ERR_CUDA;
    p.W = W;
    p.s = s;
    p.x = x;
    p.y = y;
    p.N = N;
    p.K = K;
    p.batch = batch;
    p.lkg = b.lkg;
    p.ks = b.ks;
    p.gpw = (1 << b.lkg) / b.ks;
    p.tiles = b.tiles;
    p.nch = b.nch;
    p.stage_bytes = b.stage_bytes;
    p.scale_off = b.scale_off;
    p.x_off = b.x_off;
    p.red_off = b.red_off;
    p.y4 = (N % 2) == 0 && aligned(y, 4);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(b.tiles, di->sm_count));
    cfg.blockDim = dim3(kBThreads);
    cfg.dynamicSmemBytes = b.smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    switch (XT) {
        case 1: e = launch_xt<1>(b.R, s2, cfg, p, di); break;
        case 2: e = launch_xt<2>(b.R, s2, cfg, p, di); break;
        case 3: e = launch_xt<3>(b.R, s2, cfg, p, di); break;
        default: e = launch_xt<4>(b.R, s2, cfg, p, di); break;
    }
    return e == cudaSuccess ? WQ4_OK : WQ4_ERR_CUDA;
}

}  // namespace wq4
