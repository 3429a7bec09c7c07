// wq4_tiles.cuh -- the weight-tile loop of the batched kernels (batch 2-32) on
// the legacy tensor path (mma.sync m16n8k16), shared by the batched GEMV
// (wq4_bgemv.cu) and the batched decode stages (wq4_stage.cu).
//
// K % 256 == 0 and 16-byte aligned scales.  Weights are the 16 rows of the
// MMA (exact fp16 q - 7), activations its columns: two MMAs per 32-code group,
// row tile and eight activation rows add the group's products in fp32, and
// the group's scales multiply the fp32 result into the running sums, so no
// weight is rounded and every fp16 scale is valid.  (Activations as the rows
// take ~20 % more instructions a weight while the batch leaves half of the 16
// rows empty.)
//
// A CTA owns tiles of TR weight rows; its NW consumer warps are NW / KS row
// groups times KS slices of every K chunk.  A producer lane brings each chunk
// with three tensor copies: TR rows of codes (boxes of 128 bytes = 8 groups,
// 128-byte swizzle), TR rows of scales (16 bytes a box) and the batch's
// activations (boxes of 64 = 2 groups, 128-byte swizzle; rows past the batch
// read as zeros), each matrix seen as (position in the box, row, box).  One
// copy a matrix and chunk matters: with one copy per box the producer's issue
// rate (~85 cycles a copy) bound the narrow shapes.  The consumer warps wait
// only for the chunk they are at and drift apart by up to the ring's depth.
//
// GU (a fused gate_up matrix of 2 F rows): a tile is TR / 2 gate rows and the
// TR / 2 up rows that go with them; an MMA's rows 0-7 are gate rows, 8-15 the
// same up rows, so that a lane holds both.
#pragma once

#include "wq4_device.cuh"
#include "wq4_host.h"
#include "wq4_items.cuh"
#include "wq4_tc.cuh"

namespace wq4 {

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t r[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// d += A B (m16n8k16, fp16 in, fp32 out); see mma_16816 for the fragments.
__device__ __forceinline__ void mma_acc(float d[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1)
{
    const float c[4] = {d[0], d[1], d[2], d[3]};
    mma_16816(d, a0, a1, a2, a3, b0, b1, c);
}

constexpr int kTMaxSlots = 8;
constexpr int kTHeader = 1024;                    // full[8], empty[8]; the stages keep their factors from byte 256

// Consumer warps: 16 (96 registers a thread beside the producer) up to batch
// 16, else 8 (168) with up to 48 weight rows each: at 96 registers the sums of
// 24-32 activation rows spilled (128256 x 4096, batch 32: 396 us, with 8 warps
// 130; 12 warps 137, and narrow matrices lose their 8 K slices).
template <int XT>
constexpr int kTWarps = XT <= 2 ? 16 : 8;

struct TileGeom {
    int K;
    int lkg;               // log2 of the groups per chunk (8, 16 or 32)
    int wrows;             // weight rows per warp: a multiple of 8 up to 32 (48 with 8 warps); GU: of 16
    int ks, gpw;           // K slices, groups of a chunk per slice (2, 4 or 8)
    int tiles, nch, nslots;
    int tails;             // tiles of 16 rows a warp after the `tiles` ones (whole rounds of the grid then), or 0
    uint32_t slot_bytes, scale_off, x_off, red_off;
};

// The launch shape of the tile loop (tile_plan, wq4_bgemv.cu): rows per warp,
// K slices, chunk length and ring depth of the least estimated time.  stage:
// the decode stages' constraints (sums always go through shared memory, at
// least 16 rows a warp, room for `extra` bytes of epilogue scratch).
struct TilePlan {
    TileGeom g;
    int R = 0;             // row tiles of 16 per warp
    int grid = 0;
    size_t smem = 0;
};
bool tile_plan(int sms, size_t smem_max, int N, int K, int XT, bool stage, size_t extra, TilePlan* out);

// Tensor maps of one call: weights (N rows), scales and `rows` activation rows
// of pitch x_pitch elements; then weights and scales of the tails, if any.
bool tile_maps(CUtensorMap tm[5], const uint32_t* W, const uint16_t* s, const uint16_t* x, int N, int K, int rows,
               int64_t x_pitch, int XT, const TilePlan& p, bool gu);

// Activation row (of a tile of eight) that lane group g holds: neighbouring
// groups take rows four apart, so that the eight lanes of a 16-byte load phase
// (two rows, four chunks) hit different halves of the swizzled 128-byte lines.
__device__ __forceinline__ int x_row(int g) { return ((g & 1) << 2) | (g >> 1); }

__device__ __forceinline__ float lo_scale(uint32_t v) { return __low2float(*reinterpret_cast<const __half2*>(&v)); }
__device__ __forceinline__ float hi_scale(uint32_t v) { return __high2float(*reinterpret_cast<const __half2*>(&v)); }

// One lane: streams the CTA's chunks (tile blockIdx.x, + gridDim.x, ..., then
// its tail) into the ring.  up: GU's first up row.  late: the previous kernel
// may write the weights (they are fetched into L2 before it has finished; no
// GU, no tail).
template <int XT, bool GU, bool TAIL = false>
__device__ __forceinline__ void tile_producer(const CUtensorMap* tm_w, const CUtensorMap* tm_s, const CUtensorMap* tm_x,
                                              const CUtensorMap* tm_w2, const CUtensorMap* tm_s2, const TileGeom& p, int up,
                                              uint8_t* smem, uint64_t* full, uint64_t* empty, uint32_t* err, bool late = false)
{
    tc::prefetch_map(tm_w);
    tc::prefetch_map(tm_s);
    tc::prefetch_map(tm_x);
    const int TR = p.wrows * (kTWarps<XT> / p.ks), TB = GU ? TR / 2 : TR;
    const int grid = static_cast<int>(gridDim.x), nch = p.nch, nslots = p.nslots;
    const int wholes = (p.tiles - static_cast<int>(blockIdx.x) + grid - 1) / grid;
    const bool tail = TAIL && static_cast<int>(blockIdx.x) < p.tails;
    const int TR2 = 16 * (kTWarps<XT> / p.ks);
    const int nt = p.tiles * TR + static_cast<int>(blockIdx.x) * TR2;          // the tail's first row
    const int boxes = 1 << (p.lkg - 3), whole = wholes * nch, total = whole + (tail ? nch : 0);
    const uint32_t bytes = boxes * (TR * 144 + XT * 4096);
    auto load_w = [&](int slot, int f, int n0, int ch) {
        uint8_t* base = smem + kTHeader + static_cast<size_t>(slot) * p.slot_bytes;
        if (TAIL && f >= whole) {
            mbar_arrive_expect_tx(&full[slot], boxes * (TR2 * 144 + XT * 4096));
            tc::tma_load_3d(base, tm_w2, 0, nt, ch * boxes, &full[slot]);
            tc::tma_load_3d(base + p.scale_off, tm_s2, 0, nt, ch * boxes, &full[slot]);
            return;
        }
        mbar_arrive_expect_tx(&full[slot], bytes);
        tc::tma_load_3d(base, tm_w, 0, n0, ch * boxes, &full[slot]);
        if (GU) tc::tma_load_3d(base + boxes * TB * 128, tm_w, 0, up + n0, ch * boxes, &full[slot]);
        tc::tma_load_3d(base + p.scale_off, tm_s, 0, n0, ch * boxes, &full[slot]);
        if (GU) tc::tma_load_3d(base + p.scale_off + boxes * TB * 16, tm_s, 0, up + n0, ch * boxes, &full[slot]);
    };
    auto load_x = [&](int slot, int ch) {
        uint8_t* base = smem + kTHeader + static_cast<size_t>(slot) * p.slot_bytes;
        tc::tma_load_3d(base + p.x_off, tm_x, 0, 0, 4 * ch * boxes, &full[slot]);
    };
    // weights may be fetched while the previous kernel of the stream
    // finishes, activations only after it (programmatic dependent launch)
    int n0 = static_cast<int>(blockIdx.x) * TB, ch = 0;
    const int early = min(nslots, total);
    if (late) {
        for (int f = 0, c = 0, r = n0; f < early; ++f) {
            tc::tma_prefetch_3d(tm_w, 0, r, c * boxes);
            tc::tma_prefetch_3d(tm_s, 0, r, c * boxes);
            if (++c == nch) {
                c = 0;
                r += grid * TB;
            }
        }
        grid_dependency_wait();
    }
    for (int f = 0; f < early; ++f) {
        load_w(f, f, n0, ch);
        if (++ch == nch) {
            ch = 0;
            n0 += grid * TB;
        }
    }
    grid_dependency_wait();
    for (int f = 0, c = 0; f < early; ++f) {
        load_x(f, c);
        if (++c == nch) c = 0;
    }
    int slot = 0, par = 0, f = early;
    for (; f < total; ++f) {
        if (!mbar_wait(&empty[slot], par, err)) break;
        load_w(slot, f, n0, ch);
        load_x(slot, ch);
        if (++ch == nch) {
            ch = 0;
            n0 += grid * TB;
        }
        if (++slot == nslots) {
            slot = 0;
            par ^= 1;
        }
    }
    // every copy issued has landed before the CTA's memory goes away
    for (int i = max(0, f - nslots); i < f; ++i) mbar_wait(&full[i % nslots], (i / nslots) & 1, err);
}

// A consumer warp: XT tiles of eight activation rows, R row tiles of 16 (plain:
// the last one may hold eight rows; its other eight read what follows and are
// dropped).
template <int XT, int R, bool GU>
struct TileWarp {
    uint32_t smem0, coff, soff, hoffs, xoff;
    int j0, madd, lr, lane;
    int slot = 0, par = 0;
    bool ok = true;        // after a wait gave up, none is waited for
    bool bad = false;      // a scale beyond +-8188 was met (when checked)

    __device__ __forceinline__ TileWarp(const TileGeom& p, uint8_t* smem, int warp, int ln)
    {
        lane = ln;
        const int g = lane >> 2, c = lane & 3, m = lane >> 3;      // m: ldmatrix matrix of this lane's address
        const int rgs = kTWarps<XT> / p.ks, rg = warp / p.ks, sl = warp - rg * p.ks;
        const int TR = p.wrows * rgs, TB = GU ? TR / 2 : TR, boxes = 1 << (p.lkg - 3);
        const int row0 = rg * (GU ? p.wrows / 2 : p.wrows);
        lr = lane & 7;
        madd = m >> 1;
        j0 = sl * p.gpw;                                            // first group of the slice (it lies in one box of 8)
        smem0 = smem_addr(smem) + kTHeader;
        // matrices of a tile: rows 0-7 and 8-15 of group j, then of group j + 1
        coff = ((j0 >> 3) * TB + row0 + lr) * 128 + (m & 1) * (GU ? boxes * TB * 128 : 1024);
        soff = p.scale_off + ((j0 >> 3) * TB + row0 + g) * 16;
        hoffs = GU ? boxes * TB * 16 : 128;
        xoff = p.x_off + (j0 >> 1) * (XT * 1024) + x_row(g) * 128 + ((c ^ x_row(g)) << 4);
    }

    // All chunks of the next tile into acc: rows 16 r + g (0, 1) and + 8 (2, 3)
    // of the warp's, activation rows 8 t + x_row(2c), x_row(2c + 1).
    __device__ __forceinline__ void tile(const TileGeom& p, uint64_t* full, uint64_t* empty, bool check, uint32_t* err,
                                         float (&acc)[R][XT][4])
    {
        constexpr int kCT = GU ? 1024 : 2048, kST = GU ? 128 : 256;   // a row tile's codes and scales
        const int G = p.K >> 5;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int t = 0; t < XT; ++t) acc[r][t][0] = acc[r][t][1] = acc[r][t][2] = acc[r][t][3] = 0.f;
        for (int ch = 0; ch < p.nch; ++ch) {
            if (ok) ok = mbar_wait(&full[slot], par, err);
            const uint32_t base = smem0 + slot * p.slot_bytes;
            const int npair = min(p.gpw, G - (ch << p.lkg) - j0) >> 1;   // G is a multiple of 8
            const uint32_t cb = base + coff;
            uint32_t sa = base + soff + 2 * (j0 & 7), xa = base + xoff;
            int j = (j0 & 7) + madd;
#pragma unroll 1
            for (int k = 0; k < npair; ++k, sa += 4, xa += XT * 1024, j += 2) {
                uint32_t w[R][4], sa0[R], sb0[R];
                const uint32_t ca = cb + ((j ^ lr) << 4);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    ldsm_x4(ca + kCT * r, w[r]);
                    sa0[r] = lds_u32(sa + kST * r);             // scales of groups j, j + 1: row g
                    sb0[r] = lds_u32(sa + kST * r + hoffs);     // ... and row g + 8
                }
                // (wq4_gemm comes with at most 16 activation rows; in the larger
                // kernels the branch alone cost 4 %)
                if (XT <= 2 && !GU && check) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        // (the last tile's second eight rows may be none of this warp's)
                        const uint32_t sb = 16 * r + 8 < p.wrows ? sb0[r] & 0x7FFF7FFFu : 0u;
                        const uint32_t hi = __vmaxu2(sa0[r] & 0x7FFF7FFFu, sb);
                        bad = bad || (hi & 0xFFFFu) > kMaxFp16ScaleBits || (hi >> 16) > kMaxFp16ScaleBits;
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t qa[R][4], qb[R][4];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        unpack_word(w[r][2 * h], qa[r]);
                        unpack_word(w[r][2 * h + 1], qb[r]);
                    }
#pragma unroll
                    for (int t = 0; t < XT; ++t) {
                        const uint4 v = pair_permute(lds_v4((xa ^ (64 * h)) + 1024 * t));
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const float s0 = h ? hi_scale(sa0[r]) : lo_scale(sa0[r]);
                            const float s1 = h ? hi_scale(sb0[r]) : lo_scale(sb0[r]);
                            float d[4] = {0.f, 0.f, 0.f, 0.f};
                            mma_acc(d, qa[r][0], qb[r][0], qa[r][1], qb[r][1], v.x, v.y);
                            mma_acc(d, qa[r][2], qb[r][2], qa[r][3], qb[r][3], v.z, v.w);
                            acc[r][t][0] = fmaf(s0, d[0], acc[r][t][0]);
                            acc[r][t][1] = fmaf(s0, d[1], acc[r][t][1]);
                            acc[r][t][2] = fmaf(s1, d[2], acc[r][t][2]);
                            acc[r][t][3] = fmaf(s1, d[3], acc[r][t][3]);
                        }
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot]);
            if (++slot == p.nslots) {
                slot = 0;
                par ^= 1;
            }
        }
    }
};

// The K slices' sums in shared memory: [warp][activation column][row], pitch
// kRedPitch<R> (it spreads a store over the banks); column 8 t + i is
// activation row 8 t + x_row(i).
template <int R>
constexpr int kRedPitch = 16 * R + 4;

template <int XT, int R>
__device__ __forceinline__ void store_sums(float* red, int warp, int lane, const float (&acc)[R][XT][4])
{
    constexpr int P = kRedPitch<R>;
    float* mine = red + warp * (8 * XT * P) + 2 * (lane & 3) * P + (lane >> 2);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int t = 0; t < XT; ++t) {
            float* q = mine + 8 * t * P + 16 * r;
            q[0] = acc[r][t][0];
            q[P] = acc[r][t][1];
            q[8] = acc[r][t][2];
            q[P + 8] = acc[r][t][3];
        }
}

// Rows i, i + 1 (even i) of row group grp and column col, the ks slices added
// in order.
template <int XT, int R>
__device__ __forceinline__ float2 load_sums(const float* red, int grp, int ks, int col, int i)
{
    constexpr int P = kRedPitch<R>;
    const float2* src = reinterpret_cast<const float2*>(red + (grp * ks * 8 * XT + col) * P + i);
    float2 sum = src[0];
    for (int k = 1; k < ks; ++k) {
        const float2 o = src[k * (8 * XT * P / 2)];
        sum.x += o.x;
        sum.y += o.y;
    }
    return sum;
}

}  // namespace wq4
