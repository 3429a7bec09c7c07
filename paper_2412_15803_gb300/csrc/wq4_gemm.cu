// wq4_gemm.cu -- the 4-bit dequantize-and-multiply for many activation rows
// (prefill-shaped M: a prompt's tokens through one projection), on the
// tcgen05 tensor cores of sm_103a.
//
// Y[m][n] = fp16( sum_k x[m][k] * fp16((q(n,k) - 7) * s(n, k/32)) ), fp32 sums.
//
// A persistent grid walks (128 weight rows x T tokens) tiles, T = 64, 128,
// 192 or 256 chosen per call (pick_gemm), row tile major so that the CTAs
// running at one time share a weight tile through L2; where the tiles leave
// SMs idle, the CTAs of a cluster share a tile's K instead and add their fp32
// sums in rank order through distributed shared memory.  A producer warp
// brings the tile's codes and scales in blocks of 256 K (2-D tensor copies), a
// second one the tokens' activations (boxes of 64 K, 128-byte swizzle); three
// sets of four dequant warps take items of 128 K in turn and write the weights,
// dequantized to fp16 in natural K order, into 64-column A buffers in tensor
// memory (lane = weight row); one warp issues eight tcgen05.mma an item
// (kind::f16, M = 128, N = T, K = 16) into a T-column fp32 accumulator; eight
// epilogue warps move a finished accumulator through shared-memory transpose
// blocks to 16-byte stores while the next tile's MMAs run.  Every weight is
// rounded to fp16 once (relative error <= 2^-11, accumulated in fp32): within
// the library's accuracy contract.
//
// What bounds it: over long prompts the power limit (28672 x 4096 over 2048
// tokens: 363 -> 311 us, 1.55 PFLOP/s; in a loop the SMs settle at 1.42 GHz,
// where 256-token tiles run at 87 % of the MMA rate), over short ones the MMA
// issuer's own latency (~340 cycles a 64-wide chunk), the launch and the first
// weights, which are copied after the previous kernel.  Before, each 64-wide
// chunk cost the issuer ~870 cycles whatever the tile: one lane's branch with
// two waits and two commits for four MMAs.  5120 x 3072 over 77 tokens 22.7 ->
// 9.9 us, 3072 x 8192 over 1000 tokens 57 -> 36.7, 512 x 14336 over 200 tokens
// 91 -> 12.2.
#include "wq4.h"
#include "wq4_device.cuh"
#include "wq4_host.h"
#include "wq4_tc.cuh"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

namespace wq4 {
namespace {

// Warps: 0-11 dequant (three sets of four, items in turn), 12 and 13 the
// weight and activation producers, 14 the MMA issuer, 15 lets the next kernel
// launch, 16-23 epilogue (two groups of four, token blocks in turn).
constexpr int kGThreads = 768;
constexpr int kGSets = 3;
constexpr int kGWProd = 12, kGXProd = 13, kGIssuer = 14, kGTrigger = 15, kGEpi = 16;
constexpr int kGCodes = 128 * 128;    // a K block: 128 rows x 256 codes (128-byte swizzle)
constexpr int kGScales = 128 * 16;    // ... and 8 fp16 scales a row
constexpr int kGBlk = 64;             // tokens of a transpose block
constexpr int kGHeader = 1024;
constexpr int kGTmemCols = 512;

// Tile of 128 weight rows and TOK tokens (MMA N = TOK).  K moves in items of
// 128: one A buffer (64 columns) and, in one slot (TOK <= 128) or two, the
// tokens' activations; the weights in blocks of two items.
template <int TOK>
struct GCfg {
    static constexpr int kABufs = (kGTmemCols - TOK) / 64 < 6 ? (kGTmemCols - TOK) / 64 : 6;
    static constexpr int kXSub = TOK <= 128 ? 1 : 2;              // activation slots of an item
    static constexpr int kX = TOK * 2 * (128 / kXSub);            // activation slot: boxes of TOK tokens x 64 K fp16
    static constexpr int kW = kGCodes + kGScales;
    static constexpr int kXSlots = TOK == 256 ? 4 : (TOK == 192 ? 5 : (TOK == 128 ? 4 : 6));
    static constexpr int kWSlots = 3;
    static constexpr int kT = kGHeader;                           // two transpose blocks: kGBlk tokens x 128 outputs fp16
    static constexpr int kXRing = kT + 2 * kGBlk * 128 * 2;
    static constexpr int kWRing = kXRing + kXSlots * kX;
    static constexpr int kSmem = kWRing + kWSlots * kW;
    static_assert(kSmem <= 227 * 1024, "shared memory");
    static_assert(kXSlots * kX >= TOK * 128 * 4, "a split tile's sums go over the activation ring");
    static_assert((2 * kXSlots + 2 * kWSlots + 2 * kABufs + 3) * 8 <= 1008, "barriers");
};

struct GemmArgs {
    uint16_t* y;
    int N, K, M, rtiles, ttiles;
    int split;               // CTAs of a cluster that share a tile's K (1: persistent grid)
    uint32_t* err;
    int stall;               // test hook: WQ4_STALL_GEMM_X or _W leaves those copies out
};

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Four floats at the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr, uint32_t rank)
{
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(ra)
                 : "memory");
    return v;
}

// A ring position: slot and parity of the n-th use of a ring of S slots.
template <int S>
struct RingPos {
    int slot = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void next()
    {
        if (++slot == S) {
            slot = 0;
            par ^= 1u;
        }
    }
};

template <int TOK>
__global__ void __launch_bounds__(kGThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tm_codes, const __grid_constant__ CUtensorMap tm_scales,
                const __grid_constant__ CUtensorMap tm_x, const GemmArgs a)
{
    using C = GCfg<TOK>;
    constexpr int XS = C::kXSlots, WS = C::kWSlots, NA = C::kABufs;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* xfull = reinterpret_cast<uint64_t*>(smem);     // activations landed
    uint64_t* xempty = xfull + XS;
    uint64_t* wfull = xempty + XS;                           // codes and scales landed
    uint64_t* wempty = wfull + WS;
    uint64_t* afull = wempty + WS;
    uint64_t* aempty = afull + NA;
    uint64_t* dfull = aempty + NA;
    uint64_t* dempty = dfull + 1;
    uint64_t* drain = dempty + 1;
    uint32_t* tbase_sh = reinterpret_cast<uint32_t*>(smem + 1008);
    uint16_t* tbuf = reinterpret_cast<uint16_t*>(smem + C::kT);
    uint8_t* xring = smem + C::kXRing;
    uint8_t* wring = smem + C::kWRing;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // this CTA's K blocks [k0, k1) of 256 (all of them unless the cluster splits K)
    const int split = a.split, rank = static_cast<int>(blockIdx.x) % split;
    const int nblk = a.K >> 8;
    const int k0 = rank * nblk / split, k1 = (rank + 1) * nblk / split;
    const int tiles = a.rtiles * a.ttiles;
    const int u0 = static_cast<int>(blockIdx.x) / split, ustep = static_cast<int>(gridDim.x) / split;
    uint32_t* err = a.err;

    // A wait that gives up (bounded, flagged) leaves invalid outputs, but the
    // kernel still runs to its end: the dequant, issuer and epilogue warps then
    // wait no more and go on through every tile with every arrival (a lane or
    // warp that left its loop alone would leave the others in a warp-wide
    // instruction, or at a named barrier, for ever), and the producers, who stop,
    // refill a slot only after its last copy has landed, whoever released it.
    if (threadIdx.x == 0) {
        for (int i = 0; i < XS; ++i) {
            mbar_init(&xfull[i], 1);
            mbar_init(&xempty[i], 1);
        }
        for (int i = 0; i < WS; ++i) {
            mbar_init(&wfull[i], 1);
            mbar_init(&wempty[i], 8);    // 4 warps x 2 items
        }
        for (int i = 0; i < NA; ++i) {
            mbar_init(&afull[i], 4);
            mbar_init(&aempty[i], 1);
        }
        mbar_init(dfull, 1);
        mbar_init(dempty, 8);
        mbar_init(drain, 1);
        mbar_fence_init();
    }
    if (warp == kGIssuer) tc::tmem_alloc(tbase_sh, kGTmemCols);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *tbase_sh;
    const uint32_t dcol = tbase + kGTmemCols - TOK;

    if (warp == kGTrigger) {
        // the next kernel may begin once the previous one is complete: it may
        // fetch weights that the previous one wrote
        grid_dependency_wait();
        grid_dependents_launch();
    } else if (warp == kGWProd) {
        // ------------------------------------------------ weight producer
        if (lane == 0) {
            tc::prefetch_map(&tm_codes);
            tc::prefetch_map(&tm_scales);
            // The previous kernel may write the weights too: they are fetched into
            // L2 while it finishes and copied after it.  (Copied before, they would be
            // dequantized by the time it ends: 1024 x 1024 over 64 tokens 5.4 -> 4.2 us
            // in a row of calls, 128 x 256 over 17 3.2 -> 2.6.)
            if (u0 < tiles)
                for (int k = k0; k < min(k1, k0 + WS); ++k) {
                    tc::tma_prefetch_2d(&tm_codes, k * 128, (u0 / a.ttiles) * 128);
                    tc::tma_prefetch_2d(&tm_scales, k * 8, (u0 / a.ttiles) * 128);
                }
            grid_dependency_wait();
            RingPos<WS> w;
            int n = 0;
            bool ok = true;
            for (int u = a.stall == WQ4_STALL_GEMM_W ? tiles : u0; u < tiles && ok; u += ustep) {
                const int n0 = (u / a.ttiles) * 128;
                for (int k = k0; k < k1; ++k, ++n, w.next()) {
                    if (n >= WS && (!mbar_wait(&wempty[w.slot], w.par ^ 1u, err) || !mbar_wait(&wfull[w.slot], w.par ^ 1u, err))) {
                        ok = false;
                        break;
                    }
                    uint8_t* base = wring + static_cast<size_t>(w.slot) * C::kW;
                    mbar_arrive_expect_tx(&wfull[w.slot], C::kW);
                    tc::tma_load_2d(base, &tm_codes, k * 128, n0, &wfull[w.slot]);
                    tc::tma_load_2d(base + kGCodes, &tm_scales, k * 8, n0, &wfull[w.slot]);
                }
            }
            // every copy issued has landed before the CTA's memory goes away
            for (int i = max(0, n - WS); i < n; ++i) mbar_wait(&wfull[i % WS], (i / WS) & 1, err);
        }
    } else if (warp == kGXProd) {
        // -------------------------------------------- activation producer
        if (lane == 0) {
            tc::prefetch_map(&tm_x);
            grid_dependency_wait();
            RingPos<XS> x;
            int n = 0;
            bool ok = true;
            constexpr int kZ = 2 / C::kXSub;         // boxes of 64 K in a slot
            for (int u = a.stall == WQ4_STALL_GEMM_X ? tiles : u0; u < tiles && ok; u += ustep) {
                const int m0 = (u % a.ttiles) * TOK;
                for (int z = 4 * k0; z < 4 * k1; z += kZ, ++n, x.next()) {
                    if (n >= XS && (!mbar_wait(&xempty[x.slot], x.par ^ 1u, err) || !mbar_wait(&xfull[x.slot], x.par ^ 1u, err))) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&xfull[x.slot], C::kX);
                    tc::tma_load_3d(xring + static_cast<size_t>(x.slot) * C::kX, &tm_x, 0, m0, z, &xfull[x.slot]);
                }
            }
            for (int i = max(0, n - XS); i < n; ++i) mbar_wait(&xfull[i % XS], (i / XS) & 1, err);
        }
    } else if (warp == kGIssuer) {
        // ---------------------------------------------------- MMA issuer
        // Its own latency bounds the kernel unless an item is long: a wait
        // costs ~80 cycles even when it is over, a fence, a commit and an MMA
        // ~30 each (~60 an MMA from a single lane's branch, where the operands
        // are not warp-uniform; so the whole warp runs the loop and one elected
        // lane issues).  Hence eight MMAs an item, two or three waits.
        constexpr uint32_t idesc = tc::idesc_f16_f32(128, TOK);
        const bool leader = tc::elect_one();
        RingPos<XS> x;
        RingPos<NA> ab;
        int dit = 0;
        bool ok = true;
        const uint64_t xdesc = tc::sw128_kmajor_desc(smem_addr(xring));
        for (int u = u0; u < tiles; u += ustep, ++dit) {
            if (dit >= 1 && ok) ok = mbar_wait(dempty, (dit - 1) & 1, err);
            for (int it = 2 * k0; it < 2 * k1; ++it) {
                if (ok) ok = mbar_wait(&afull[ab.slot], ab.par, err);
#pragma unroll
                for (int sub = 0; sub < 2; ++sub) {
                    if (sub < C::kXSub && ok) ok = mbar_wait(&xfull[x.slot], x.par, err);
                    if (sub == 0) tc::fence_after_sync();
                    const uint64_t xd = xdesc + static_cast<uint64_t>(x.slot) * (C::kX >> 4) +
                                        (C::kXSub == 1 ? sub * (TOK * 128 >> 4) : 0);
                    if (leader) {
#pragma unroll
                        for (int s = 0; s < 4; ++s)
                            tc::mma_f16_ts(dcol, tbase + 64 * ab.slot + 32 * sub + 8 * s, xd + 2 * s, idesc,
                                           (it > 2 * k0 || sub + s > 0) ? 1u : 0u);
                        if (sub == 1) tc::commit(&aempty[ab.slot]);
                        if (C::kXSub == 2 || sub == 1) tc::commit(&xempty[x.slot]);
                    }
                    if (C::kXSub == 2 || sub == 1) x.next();
                }
                ab.next();
            }
            if (leader) tc::commit(dfull);
        }
        // all MMAs issued have completed before tensor memory is released
        if (leader) tc::commit(drain);
        mbar_wait(drain, 0, err);
    } else if (warp < 4 * kGSets) {
        // ---------------------------------------------------- dequant
        // Item i goes to A buffer i % NA and warp set i % 3, so that several
        // items' waits, unpacking and stores are in flight.  Lane = weight row;
        // 128 codes in natural K order, 64 at a time.
        const int set = warp >> 2, row = 32 * (warp & 3) + lane;
        const uint32_t lane_base = tbase + (static_cast<uint32_t>(32 * (warp & 3)) << 16);
        RingPos<WS> w;
        RingPos<NA> ab;
        int i = 0;
        bool ok = true;
        for (int u = u0; u < tiles; u += ustep) {
            for (int it = 2 * k0; it < 2 * k1; ++it, ++i, ab.next()) {
                if (it > 2 * k0 && (it & 1) == 0) w.next();
                if (i % kGSets != set) continue;
                if (ok) ok = mbar_wait(&wfull[w.slot], w.par, err) && (i < NA || mbar_wait(&aempty[ab.slot], ab.par ^ 1u, err));
                __syncwarp();
                const uint8_t* base = wring + static_cast<size_t>(w.slot) * C::kW;
                const uint8_t* crow = base + row * 128;
                const uint2 sv2 = *reinterpret_cast<const uint2*>(base + kGCodes + row * 16 + 8 * (it & 1));
#pragma unroll
                for (int sub = 0; sub < 2; ++sub) {
                    // groups j, j + 1 of the block's 8: codes and scales
                    const int j = 4 * (it & 1) + 2 * sub;
                    const uint4 cw0 = *reinterpret_cast<const uint4*>(crow + ((j ^ (row & 7)) << 4));
                    const uint4 cw1 = *reinterpret_cast<const uint4*>(crow + (((j + 1) ^ (row & 7)) << 4));
                    const uint32_t sv = sub ? sv2.y : sv2.x;
                    // (q - 7) s is rounded to fp16 below: a larger scale would overflow
                    if ((sv & 0x7FFFu) > kMaxFp16ScaleBits || ((sv >> 16) & 0x7FFFu) > kMaxFp16ScaleBits)
                        atomicOr(err, ok ? kErrScale : 0u);
                    const uint32_t words[8] = {cw0.x, cw0.y, cw0.z, cw0.w, cw1.x, cw1.y, cw1.z, cw1.w};
                    const uint32_t s0 = prmt(sv, sv, 0x1010u), s1 = prmt(sv, sv, 0x3232u);
                    uint32_t q[32];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t s2 = k < 4 ? s0 : s1;
                        uint32_t p[4];   // (k, k+4) pairs of the word
                        unpack_word(words[k], p);
                        q[4 * k + 0] = tc::hmul2_u32(prmt(p[0], p[1], 0x5410u), s2);   // k0 k1
                        q[4 * k + 1] = tc::hmul2_u32(prmt(p[2], p[3], 0x5410u), s2);   // k2 k3
                        q[4 * k + 2] = tc::hmul2_u32(prmt(p[0], p[1], 0x7632u), s2);   // k4 k5
                        q[4 * k + 3] = tc::hmul2_u32(prmt(p[2], p[3], 0x7632u), s2);   // k6 k7
                    }
                    tc::st16(lane_base + 64 * ab.slot + 32 * sub, q);
                    tc::st16(lane_base + 64 * ab.slot + 32 * sub + 16, q + 16);
                }
                tc::st_wait();
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&afull[ab.slot]);
                    mbar_arrive(&wempty[w.slot]);
                }
            }
            w.next();
        }
    } else if (warp >= kGEpi) {
        // ---------------------------------------------------- epilogue warps
        // warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (weight rows)
        grid_dependency_wait();          // y is written after the previous kernel
        const int quad = warp & 3, grp = (warp - kGEpi) >> 2;
        uint16_t* const tb0 = tbuf + grp * kGBlk * 128;
        const int row = 32 * quad + lane;   // 0..127 over the four warps
        const uint32_t lane_base = dcol + (static_cast<uint32_t>(32 * quad) << 16);
        int dit = 0;
        bool ok = true;
        for (int u = u0; u < tiles; u += ustep, ++dit) {
            const int n0 = (u / a.ttiles) * 128, m0 = (u % a.ttiles) * TOK;
            if (ok) ok = mbar_wait(dfull, dit & 1, err);
            __syncwarp();
            tc::fence_after_sync();
            if (split > 1) {
                // fp32 sums of this CTA's K chunks, [token][row], over the idle activation ring
                float* ps = reinterpret_cast<float*>(xring);
#pragma unroll 2
                for (int t = grp * (TOK / 2); t < (grp + 1) * (TOK / 2); t += 16) {
                    uint32_t d[16];
                    tc::ld16(lane_base + t, d);
                    tc::ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) ps[(t + i) * 128 + row] = __uint_as_float(d[i]);
                }
                break;
            }
            // token blocks go to the two groups in turn
            constexpr int kBlocks = TOK / kGBlk;
            if (grp >= kBlocks && lane == 0) mbar_arrive(dempty);
            for (int blk = grp; blk < kBlocks; blk += 2) {
                const int tb = blk * kGBlk;
                // (row, token) -> transpose block [token][row], fp16
#pragma unroll
                for (int t = 0; t < kGBlk; t += 32) {
                    uint32_t d[32];
                    tc::ld16(lane_base + tb + t, d);
                    tc::ld16(lane_base + tb + t + 16, d + 16);
                    tc::ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) tb0[(t + i) * 128 + row] = float_to_half_bits(__uint_as_float(d[i]));
                }
                if (blk + 2 >= kBlocks) {
                    // this group is done with the accumulator
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(dempty);
                }
                named_barrier_sync(3 + grp, 128);
#pragma unroll
                for (int i = 0; i < kGBlk / 8; ++i) {
                    const int chunk = row + 128 * i;
                    const int tok = chunk >> 4, seg = chunk & 15;
                    const int mm = m0 + tb + tok, n = n0 + 8 * seg;
                    if (mm < a.M && n < a.N)
                        *reinterpret_cast<uint4*>(a.y + static_cast<size_t>(mm) * a.N + n) =
                            *reinterpret_cast<const uint4*>(tb0 + tok * 128 + 8 * seg);
                }
                named_barrier_sync(3 + grp, 128);   // the block is free again
            }
        }
    }

    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == kGIssuer) tc::tmem_dealloc(tbase, kGTmemCols);
    if (split > 1) {
        // the cluster's sums are in: this CTA adds its share of the tokens in
        // rank order and stores them
        grid_dependency_wait();
        cluster_sync_all();
        const int n0 = (u0 / a.ttiles) * 128, m0 = (u0 % a.ttiles) * TOK;
        const int t0 = rank * TOK / split, t1 = (rank + 1) * TOK / split;
        const uint32_t ps = smem_addr(xring);
        for (int e = t0 * 32 + static_cast<int>(threadIdx.x); e < t1 * 32; e += kGThreads) {
            const int mm = m0 + (e >> 5), n = n0 + 4 * (e & 31);
            if (mm >= a.M || n >= a.N) continue;
            float4 sum = ld_cluster_f4(ps + 16 * e, 0);
            for (int r = 1; r < split; ++r) {
                const float4 v = ld_cluster_f4(ps + 16 * e, r);
                sum.x += v.x;
                sum.y += v.y;
                sum.z += v.z;
                sum.w += v.w;
            }
            uint2 o;
            o.x = static_cast<uint32_t>(float_to_half_bits(sum.x)) | (static_cast<uint32_t>(float_to_half_bits(sum.y)) << 16);
            o.y = static_cast<uint32_t>(float_to_half_bits(sum.z)) | (static_cast<uint32_t>(float_to_half_bits(sum.w)) << 16);
            *reinterpret_cast<uint2*>(a.y + static_cast<size_t>(mm) * a.N + n) = o;   // N % 8 == 0
        }
        cluster_sync_all();   // no CTA's memory goes away while another reads it
    }
}

template <int TOK>
cudaError_t gemm_launch(cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const GemmArgs& a)
{
    static std::atomic<bool> ready[64];                // per device; setting the attribute twice is harmless
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !ready[dev].load()) {
        e = cudaFuncSetAttribute(gemm_kernel<TOK>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<TOK>::kSmem);
        if (e != cudaSuccess) return e;
        if (dev < 64) ready[dev].store(true);
    }
    cfg.dynamicSmemBytes = GCfg<TOK>::kSmem;
    return cudaLaunchKernelEx(&cfg, gemm_kernel<TOK>, tm[0], tm[1], tm[2], a);
}

// Clusters of `split` CTAs that fit the device at once (cached per device).
template <int TOK>
int cluster_capacity(int dev, int split)
{
    static std::atomic<int> cached[64][9];
    if (dev < 64 && cached[dev][split].load()) return cached[dev][split].load();
    if (cudaFuncSetAttribute(gemm_kernel<TOK>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<TOK>::kSmem) !=
        cudaSuccess)
        return 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = split;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(split);
    cfg.blockDim = dim3(kGThreads);
    cfg.dynamicSmemBytes = GCfg<TOK>::kSmem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_kernel<TOK>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    if (dev < 64 && n > 0) cached[dev][split].store(n);
    return n;
}

struct GemmPlan {
    int tok = 0, split = 1;
};

// Token tile and K split: the least estimated time.  Per 64-wide K chunk a
// tile takes (us, one CTA alone .. every SM busy) 0.188 .. 0.205 with 64
// tokens, 0.203 .. 0.235 with 128, 0.214 .. 0.304 with 192 and 0.287 .. 0.394
// with 256, beside a launch's fixed 2.3, 2.65, 3.3 and 4; a split (the
// cluster's CTAs take K blocks in order, one tile a cluster, all resident)
// adds 1.3, 1.5 or 1.7 and 0.016, 0.023 or 0.03 a CTA.  Fitted to every choice
// over 34 sizes, each over copies of 520 MB: the picks are 0.1 % from the best on
// average, 3 % at most.  Measured: 5120 x 3072 over 77 tokens 11.6 us whole, 9.9
// split in 3; 512 x 14336 over 200 tokens 42 whole, 12.2 split in 8; 1024 x 1024
// over 300 tokens 5.6 whole, 6.4 split in 2.
GemmPlan pick_gemm(int N, int K, int M, int sms, int dev)
{
    static constexpr int kTok[4] = {64, 128, 192, 256};
    static constexpr double kB0[4] = {0.188, 0.203, 0.214, 0.287}, kB1[4] = {0.205, 0.235, 0.304, 0.394};
    static constexpr double kFix[4] = {2.3, 2.65, 3.3, 4.0};
    static constexpr double kSplit[4] = {1.3, 1.5, 1.7, 1.7}, kCta[4] = {0.0155, 0.023, 0.03, 0.03};
    GemmPlan best;
    double best_t = 1e300;
    const int nblk = K >> 8;
    for (int i = 3; i >= 0; --i) {
        const int64_t tiles = static_cast<int64_t>((N + 127) / 128) * ((M + kTok[i] - 1) / kTok[i]);
        auto rate = [&](double ctas) { return kB0[i] + (kB1[i] - kB0[i]) * std::min(1.0, ctas / sms); };
        for (int s = 1; s <= 8 && s <= nblk; ++s) {
            const double nch = 4.0 * ((nblk + s - 1) / s);
            double t = kFix[i];
            if (s == 1) {
                const int64_t full = tiles / sms, rest = tiles % sms;
                t += nch * (full * kB1[i] + (rest ? rate(static_cast<double>(rest)) : 0.0)) + 0.6 * full;
            } else {
                if (tiles * s > sms) break;
                t += nch * rate(static_cast<double>(tiles * s)) + kSplit[i] + kCta[i] * (tiles * s);
            }
            if (t >= best_t - 1e-9) continue;
            if (s > 1) {
                const int cap = i == 0   ? cluster_capacity<64>(dev, s)
                                : i == 1 ? cluster_capacity<128>(dev, s)
                                : i == 2 ? cluster_capacity<192>(dev, s)
                                         : cluster_capacity<256>(dev, s);
                if (tiles > cap) continue;
            }
            best_t = t;
            best.tok = kTok[i];
            best.split = s;
        }
    }
    return best;
}

// Up to this many tokens the batched GEMV kernel takes the call (exact
// weights; 5120 x 3072 over 8 tokens 5.3 us against 9.4 here, 128256 x 4096
// over 16 tokens 82.8 against 85.2).
constexpr int kGemvTokens = 16;

}  // namespace
}  // namespace wq4

using namespace wq4;

extern "C" int wq4_gemm(const uint32_t* W_packed, const uint16_t* scales, const uint16_t* x, uint16_t* y, int N, int K,
                        int M, void* stream)
{
    if (!W_packed || !scales || !x || !y) return WQ4_ERR_INVALID;
    if (N < 1 || K < 32 || M < 1 || (K % 32) != 0) return WQ4_ERR_INVALID;
    if ((K % 256) != 0 || (N % 8) != 0) return WQ4_ERR_UNSUPPORTED;
    if (static_cast<int64_t>(N) * K / 8 > (static_cast<int64_t>(1) << 40)) return WQ4_ERR_INVALID;
    if (!aligned(W_packed, 16) || !aligned(scales, 16) || !aligned(x, 16) || !aligned(y, 16)) return WQ4_ERR_ALIGN;
    const size_t yb = static_cast<size_t>(M) * N * 2, xb = static_cast<size_t>(M) * K * 2;
    const size_t wb = static_cast<size_t>(N) * K / 2, sb = static_cast<size_t>(N) * K / 16;
    if (overlaps(y, yb, x, xb) || overlaps(y, yb, W_packed, wb) || overlaps(y, yb, scales, sb)) return WQ4_ERR_INVALID;
    int dev = 0;
    const DeviceInfo* di = current_device_info(&dev);
    if (!di) return WQ4_ERR_CUDA;
    if (M <= kGemvTokens)
        return launch_bgemv(di, W_packed, scales, x, y, N, K, M, static_cast<cudaStream_t>(stream), true);
    const GemmPlan pl = pick_gemm(N, K, M, di->sm_count, dev);
    CUtensorMap tm[3];
    if (!encode_tensor_map_2d(&tm[0], CU_TENSOR_MAP_DATA_TYPE_UINT8, W_packed, static_cast<uint64_t>(K) / 2,
                              static_cast<uint64_t>(N), static_cast<uint64_t>(K) / 2, 128, 128,
                              CU_TENSOR_MAP_SWIZZLE_128B) ||
        !encode_tensor_map_2d(&tm[1], CU_TENSOR_MAP_DATA_TYPE_UINT16, scales, static_cast<uint64_t>(K) / 32,
                              static_cast<uint64_t>(N), static_cast<uint64_t>(K) / 16, 8, 128,
                              CU_TENSOR_MAP_SWIZZLE_NONE) ||
        !encode_tensor_map_3d(&tm[2], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, x,
                              {64, static_cast<uint64_t>(M), static_cast<uint64_t>(K) / 64}, {static_cast<uint64_t>(K) * 2, 128},
                              {64, static_cast<uint32_t>(pl.tok), pl.tok <= 128 ? 2u : 1u}, CU_TENSOR_MAP_SWIZZLE_128B))
        return WQ4_ERR_CUDA;
    GemmArgs a;
    a.y = y;
    a.N = N;
    a.K = K;
    a.M = M;
    a.rtiles = (N + 127) / 128;
    a.ttiles = (M + pl.tok - 1) / pl.tok;
    a.split = pl.split;
    a.err = status_word();
    if (!a.err) return WQ4_ERR_CUDA;
    a.stall = test_copy_stall();
    const int64_t tiles = static_cast<int64_t>(a.rtiles) * a.ttiles;
    if (tiles > (static_cast<int64_t>(1) << 30)) return WQ4_ERR_UNSUPPORTED;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = pl.split;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.split > 1 ? static_cast<int>(tiles) * pl.split
                                    : static_cast<int>(tiles < di->sm_count ? tiles : di->sm_count));
    cfg.blockDim = dim3(kGThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cfg.attrs = attr;
    cfg.numAttrs = pl.split > 1 ? 2 : 1;
    cudaError_t e;
    switch (pl.tok) {
        case 256: e = gemm_launch<256>(cfg, tm, a); break;
        case 192: e = gemm_launch<192>(cfg, tm, a); break;
        case 128: e = gemm_launch<128>(cfg, tm, a); break;
        default: e = gemm_launch<64>(cfg, tm, a); break;
    }
    return e == cudaSuccess ? WQ4_OK : WQ4_ERR_CUDA;
}
