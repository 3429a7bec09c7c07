// wq4_stage.cu -- the projections of the batched decode chain (batch 3-32):
// one kernel per stage (QKV, O, gate_up, down, LM head), recorded into a CUDA
// graph with programmatic dependent launch.
//
// A stage is the weight-tile loop of wq4_tiles.cuh (exact fp16 q - 7 on the
// legacy tensor path, group scales in fp32: 1/2048 closer per weight than the
// fp16-rounded tcgen05 stages before it) with the chain's glue as the tile's
// epilogue: row factors, residual adds, SiLU(gate) * up, the plain copies of
// every stage output, and per tile the sums of squares from which the next
// stage's RMS factors follow.  A warp beside the producer computes this
// stage's factors while the tiles run.  Weights may be fetched before the
// previous stage has finished, its outputs are read after: on the SMs that it
// leaves free, that is, since two blocks of ~200 KB do not share one.
//
// Measured (us a token, 3B shape, batch 4 / 8 / 16 / 32): 783 / 822 / 1093 /
// 1866, against 1176 / 1228 / 1349 / 2171 with tcgen05 stages, whose
// MMA-issuing lanes and K parts' exchange through global memory took most of
// a narrow stage.  Bound by each stage's launch, first chunk and epilogue
// (~3 us of ~7 at batch 8), then as the tile loop.
#include "wq4_stage_host.h"
#include "wq4_device.cuh"
#include "wq4_host.h"
#include "wq4_items.cuh"
#include "wq4_tiles.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <mutex>

namespace wq4 {
namespace {

constexpr int kFactors = 256;          // shared-memory byte offset of r_in[32], r_u[32] (before the ring)
static_assert(kFactors >= 16 * kTMaxSlots && kFactors + 64 * 4 <= kTHeader, "header");

struct StageArgs {
    TileGeom g;
    int type, N, B, H, F;
    float eps;
    const float* sq_in;     // sums of squares of this stage's input, [B][sq_ld], sq_in_n of them; null: factor 1
    const float* sq_u;      // O: of the layer input u
    int sq_in_n, sq_u_n, sq_ld;
    const uint16_t* res;    // O: the layer input u; down: x1; LM head: x_L
    uint16_t* y;            // QKV: qkv, O: o, gate_up: gate|up, down: d, LM head: logits
    uint16_t* y2;           // QKV: the query block (O's input), O: x1, gate_up: m, down: x2
    uint16_t* y3;           // O: v = fp16(r(u) u); LM head: v of x_L
    float* sq_out;          // sums of squares of the next stage's input, one per tile of its rows
    uint32_t sqs_off;       // shared-memory offset of the tile's squares
    uint32_t* err;
};

// fp16(a + b) for fp16 operands: the fp32 sum rounded once to fp16.
__device__ __forceinline__ uint16_t add_h(float a, float b) { return float_to_half_bits(a + b); }

// r[b] = 1 / sqrt(mean + eps) of every batch row from the per-tile sums of
// squares, by one warp, lanes strided over the tiles: the same order in every
// CTA.  Four rows at a time, so that their loads are in flight together.
__device__ __forceinline__ void rms_factors(const float* sq, int n, int ld, int B, int H, float eps, float* r, int lane)
{
    for (int b0 = 0; b0 < B; b0 += 4) {
        float t[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k = lane; k < n; k += 32)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (b0 + i < B) t[i] += __ldcg(sq + static_cast<size_t>(b0 + i) * ld + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float s = warp_sum(t[i]);
            if (lane == 0 && b0 + i < B) r[b0 + i] = rsqrtf(s * (1.f / static_cast<float>(H)) + eps);
        }
    }
}

template <int XT, int R, bool GU>
__global__ void __launch_bounds__(32 * (kTWarps<XT> + 2), 1)
    stage_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_s,
                 const __grid_constant__ CUtensorMap tm_x, const StageArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int NW = kTWarps<XT>, kConsumers = 32 * NW;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + kTMaxSlots;
    float* r_in = reinterpret_cast<float*>(smem + kFactors);
    float* r_u = r_in + 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ks = a.g.ks, wrows = a.g.wrows, rgs = NW / ks, TR = wrows * rgs;
    const int B = a.B, H = a.H, F = a.F;

    if (tid == kConsumers) {
        for (int i = 0; i < a.g.nslots; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], NW);
        }
        mbar_fence_init();
    }
    __syncthreads();
    grid_dependents_launch();
    if (warp == NW) {
        if (lane == 0) tile_producer<XT, GU>(&tm_w, &tm_s, &tm_x, nullptr, nullptr, a.g, F, smem, full, empty, a.err);
        return;
    }
    grid_dependency_wait();               // the previous stage's outputs are complete from here on
    if (warp == NW + 1) {
        // this stage's row factors, while the tiles run
        if (a.sq_in) rms_factors(a.sq_in, a.sq_in_n, a.sq_ld, B, H, a.eps, r_in, lane);
        else r_in[lane] = 1.f;
        if (a.sq_u) rms_factors(a.sq_u, a.sq_u_n, a.sq_ld, B, H, a.eps, r_u, lane);
        __syncwarp();
        named_barrier_sync(2, kConsumers + 32);
        return;
    }

    TileWarp<XT, R, GU> tw(a.g, smem, warp, lane);
    float acc[R][XT][4];
    float* red = reinterpret_cast<float*>(smem + a.g.red_off);
    float* sqs = reinterpret_cast<float*>(smem + a.sqs_off);       // [column][row pair], padded
    bool first = true;
    for (int tile = blockIdx.x; tile < a.g.tiles; tile += gridDim.x) {
        tw.tile(a.g, full, empty, false, a.err, acc);
        store_sums<XT, R>(red, warp, lane, acc);
        if (first) named_barrier_sync(2, kConsumers + 32);         // sums and factors are in
        else named_barrier_sync(1, kConsumers);
        first = false;
        if constexpr (GU) {
            const int TB = TR / 2, hrows = wrows >> 2;              // pairs of gate rows per row group
            for (int e = tid; e < rgs * hrows * 8 * XT; e += kConsumers) {
                const int pr = e % hrows, q = e / hrows;
                const int col = q % (8 * XT), grp = q / (8 * XT);
                const int b = (col & ~7) + x_row(col & 7);
                const int jr = 2 * pr, j = tile * TB + grp * (wrows >> 1) + jr;
                if (b >= B || j >= F) continue;
                const int i = 16 * (jr >> 3) + (jr & 7);            // MMA rows i, i + 1: gate, + 8: up
                const float2 sg = load_sums<XT, R>(red, grp, ks, col, i);
                const float2 su = load_sums<XT, R>(red, grp, ks, col, i + 8);
                const float rf = r_in[b];
                const uint16_t g0 = float_to_half_bits(rf * sg.x), g1 = float_to_half_bits(rf * sg.y);
                const uint16_t u0 = float_to_half_bits(rf * su.x), u1 = float_to_half_bits(rf * su.y);
                const float f0 = half_bits_to_float(g0), f1 = half_bits_to_float(g1);
                const uint16_t m0 = float_to_half_bits(f0 / (1.f + expf(-f0)) * half_bits_to_float(u0));
                const uint16_t m1 = float_to_half_bits(f1 / (1.f + expf(-f1)) * half_bits_to_float(u1));
                uint16_t* gu = a.y + static_cast<size_t>(b) * 2 * F + j;
                *reinterpret_cast<uint32_t*>(gu) = pack2(g0, g1);
                *reinterpret_cast<uint32_t*>(gu + F) = pack2(u0, u1);
                *reinterpret_cast<uint32_t*>(a.y2 + static_cast<size_t>(b) * F + j) = pack2(m0, m1);
            }
        } else {
            const int hrows = wrows >> 1, pairs = rgs * hrows;      // pairs of rows per row group, per tile
            const bool squares = a.sq_out && tile * TR < H;
            for (int e = tid; e < pairs * 8 * XT; e += kConsumers) {
                const int pr = e % hrows, q = e / hrows;
                const int col = q % (8 * XT), grp = q / (8 * XT);
                const int b = (col & ~7) + x_row(col & 7);
                const int n = tile * TR + grp * wrows + 2 * pr;
                const bool live = b < B && n < a.N;
                uint32_t rw = 0;                                    // the residual words
                if (live && a.res && n < H) rw = __ldcg(reinterpret_cast<const uint32_t*>(a.res + static_cast<size_t>(b) * H + n));
                const float2 s = load_sums<XT, R>(red, grp, ks, col, 2 * pr);
                float x0 = 0.f, x1 = 0.f;                           // the next stage's input at these rows
                if (live) {
                    const float rf = r_in[b];
                    const size_t at = static_cast<size_t>(b) * H + n;
                    if (a.type == kStQKV) {
                        const uint32_t w = pack2(float_to_half_bits(rf * s.x), float_to_half_bits(rf * s.y));
                        *reinterpret_cast<uint32_t*>(a.y + static_cast<size_t>(b) * a.N + n) = w;   // N even
                        if (n < H) {
                            *reinterpret_cast<uint32_t*>(a.y2 + at) = w;
                            x0 = lo_f(w);
                            x1 = hi_f(w);
                        }
                    } else if (a.type == kStO) {
                        const uint16_t o0 = float_to_half_bits(rf * s.x), o1 = float_to_half_bits(rf * s.y);
                        const float ru = r_u[b];
                        const uint16_t v0 = float_to_half_bits(ru * lo_f(rw)), v1 = float_to_half_bits(ru * hi_f(rw));
                        const uint32_t w = pack2(add_h(half_bits_to_float(v0), half_bits_to_float(o0)),
                                                 add_h(half_bits_to_float(v1), half_bits_to_float(o1)));
                        *reinterpret_cast<uint32_t*>(a.y + at) = pack2(o0, o1);
                        *reinterpret_cast<uint32_t*>(a.y2 + at) = w;
                        *reinterpret_cast<uint32_t*>(a.y3 + at) = pack2(v0, v1);
                        x0 = lo_f(w);
                        x1 = hi_f(w);
                    } else if (a.type == kStDOWN) {
                        const uint16_t d0 = float_to_half_bits(s.x), d1 = float_to_half_bits(s.y);
                        const uint32_t w = pack2(add_h(lo_f(rw), half_bits_to_float(d0)), add_h(hi_f(rw), half_bits_to_float(d1)));
                        *reinterpret_cast<uint32_t*>(a.y + at) = pack2(d0, d1);
                        *reinterpret_cast<uint32_t*>(a.y2 + at) = w;
                        x0 = lo_f(w);
                        x1 = hi_f(w);
                    } else {   // LM head; its first H rows also keep v = fp16(r x_L)
                        uint16_t* out = a.y + static_cast<size_t>(b) * a.N + n;   // N may be odd
                        out[0] = float_to_half_bits(rf * s.x);
                        if (n + 1 < a.N) out[1] = float_to_half_bits(rf * s.y);
                        if (n < H)
                            *reinterpret_cast<uint32_t*>(a.y3 + at) =
                                pack2(float_to_half_bits(rf * lo_f(rw)), float_to_half_bits(rf * hi_f(rw)));
                    }
                }
                if (squares) sqs[col * (pairs + 1) + grp * hrows + pr] = fmaf(x0, x0, x1 * x1);
            }
            if (squares) {
                // a warp per column adds the tile's squares in a fixed order
                named_barrier_sync(1, kConsumers);
                for (int col = warp; col < 8 * XT; col += NW) {
                    float t = 0.f;
                    for (int k = lane; k < pairs; k += 32) t += sqs[col * (pairs + 1) + k];
                    t = warp_sum(t);
                    const int b = (col & ~7) + x_row(col & 7);
                    if (lane == 0 && b < B) a.sq_out[static_cast<size_t>(b) * a.sq_ld + tile] = t;
                }
            }
        }
        named_barrier_sync(1, kConsumers);                          // sums and squares may be written again
    }
}

// Sums of squares of the 128-element tiles of a [B][H] input, a warp each.
__global__ void __launch_bounds__(256) squares_kernel(const uint16_t* __restrict__ x, int H, int B, int ld,
                                                      float* __restrict__ sq_out)
{
    grid_dependents_launch();
    grid_dependency_wait();
    const int lane = threadIdx.x & 31, nt = H / 128;
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i >= nt * B) return;
    const int b = i / nt, t = i - b * nt;
    const uint2 v = __ldcg(reinterpret_cast<const uint2*>(x + static_cast<size_t>(b) * H + 128 * t) + lane);
    const float a0 = lo_f(v.x), a1 = hi_f(v.x), a2 = lo_f(v.y), a3 = hi_f(v.y);
    const float s = warp_sum(fmaf(a0, a0, a1 * a1) + fmaf(a2, a2, a3 * a3));
    if (lane == 0) sq_out[static_cast<size_t>(b) * ld + t] = s;
}

// ----------------------------------------------------------------- host --

template <int XT, int R, bool GU>
cudaError_t launch_one(const cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const StageArgs& a, int smem_max)
{
    static std::atomic<bool> ready[64];                // per device; setting the attribute twice is harmless
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !ready[dev].load()) {
        e = cudaFuncSetAttribute(stage_kernel<XT, R, GU>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
        if (e != cudaSuccess) return e;
        if (dev < 64) ready[dev].store(true);
    }
    return cudaLaunchKernelEx(&cfg, stage_kernel<XT, R, GU>, tm[0], tm[1], tm[2], a);
}

template <int XT, bool GU>
cudaError_t launch_r(int R, const cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const StageArgs& a, int smem_max)
{
    if (R == 1) return launch_one<XT, 1, GU>(cfg, tm, a, smem_max);
    if constexpr (kTWarps<XT> == 8)
        if (R == 3) return launch_one<XT, 3, GU>(cfg, tm, a, smem_max);
    return launch_one<XT, 2, GU>(cfg, tm, a, smem_max);
}

template <bool GU>
cudaError_t launch_xt(int XT, int R, const cudaLaunchConfig_t& cfg, const CUtensorMap* tm, const StageArgs& a, int smem_max)
{
    switch (XT) {
        case 1: return launch_r<1, GU>(R, cfg, tm, a, smem_max);
        case 2: return launch_r<2, GU>(R, cfg, tm, a, smem_max);
        case 3: return launch_r<3, GU>(R, cfg, tm, a, smem_max);
        default: return launch_r<4, GU>(R, cfg, tm, a, smem_max);
    }
}

}  // namespace

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

bool encode_tensor_map_2d(CUtensorMap* m, CUtensorMapDataType dt, const void* base, uint64_t inner, uint64_t outer,
               uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t es[2] = {1, 1};
    return enc(m, dt, 2, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_tensor_map_3d(CUtensorMap* m, CUtensorMapDataType dt, const void* base, const std::array<uint64_t, 3>& dims,
                          const std::array<uint64_t, 2>& strides, const std::array<uint32_t, 3>& box,
                          CUtensorMapSwizzle swz)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return false;
    cuuint64_t d[3] = {dims[0], dims[1], dims[2]}, st[2] = {strides[0], strides[1]};
    cuuint32_t bx[3] = {box[0], box[1], box[2]}, es[3] = {1, 1, 1};
    return enc(m, dt, 3, const_cast<void*>(base), d, st, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int stage_launch_squares(const uint16_t* x, int H, int B, float* sq, cudaStream_t cs)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((H / 128 * B + 7) / 8);
    cfg.blockDim = dim3(256);
    cfg.stream = cs;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, squares_kernel, x, H, B, stage_sq_ld(H), sq) == cudaSuccess ? WQ4_OK : WQ4_ERR_CUDA;
}

// Every launch may overlap its set-up and weight stream with the tail of the
// previous one (programmatic dependent launch); it reads the previous stage's
// outputs only after that grid has completed.
int stage_record_token(const StageModel& m, cudaStream_t cs, const StageAttnHook* att)
{
    const int B = m.B, H = m.H, F = m.F, L = m.table->num_layers, XT = (B + 7) / 8;
    const StageBuffers& u = m.buf;
    const size_t LH = static_cast<size_t>(B) * H;
    const int ld = stage_sq_ld(H);
    float* sq_u = u.sq;                                           // [B][ld] each
    float* sq_a = u.sq + static_cast<size_t>(B) * ld;
    float* sq_x1 = u.sq + 2 * static_cast<size_t>(B) * ld;
    const struct { int N, K; } shape[5] = {{m.Nqkv, H}, {H, H}, {2 * F, H}, {H, F}, {m.V, H}};
    TilePlan plan[5];
    int tr[5];
    uint32_t sqs_bytes[5];
    for (int t = 0; t < 5; ++t) {
        // room for a tile's squares: 8 XT columns of up to 64 row pairs and a pad
        const size_t extra = align_up(static_cast<size_t>(8 * XT) * 65 * 4, 16);
        if (!tile_plan(m.sms, m.smem_max, shape[t].N, shape[t].K, XT, true, extra, &plan[t])) return WQ4_ERR_UNSUPPORTED;
        tr[t] = plan[t].g.wrows * ((XT <= 2 ? kTWarps<1> : kTWarps<4>) / plan[t].g.ks);
        sqs_bytes[t] = static_cast<uint32_t>(extra);
    }
    auto tiles_of = [&](int t) { return (H + tr[t] - 1) / tr[t]; };   // tiles that hold a row below H
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    bool ok = stage_launch_squares(u.x_stage, H, B, sq_u, cs) == WQ4_OK;
    auto stage = [&](int type, const wq4_mat& w, const uint16_t* x, StageArgs a) {
        const TilePlan& p = plan[type];
        CUtensorMap tm[5];
        ok = ok && tile_maps(tm, w.W, w.s, x, shape[type].N, shape[type].K, B, shape[type].K, XT, p, type == kStGU);
        if (!ok) return;
        a.g = p.g;
        a.type = type;
        a.N = shape[type].N;
        a.B = B;
        a.H = H;
        a.F = F;
        a.eps = m.table->rms_eps;
        a.sq_ld = ld;
        a.sqs_off = static_cast<uint32_t>(p.smem - sqs_bytes[type]);
        a.err = m.err;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(p.grid);
        cfg.blockDim = dim3(32 * ((XT <= 2 ? kTWarps<1> : kTWarps<4>) + 2));
        cfg.dynamicSmemBytes = p.smem;
        cfg.stream = cs;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const int smax = static_cast<int>(m.smem_max);
        const cudaError_t e = type == kStGU ? launch_xt<true>(XT, p.R, cfg, tm, a, smax) : launch_xt<false>(XT, p.R, cfg, tm, a, smax);
        ok = ok && e == cudaSuccess;
    };
    int nu = H / 128;                                             // sums of squares of the layer input
    for (int l = 0; l < L; ++l) {
        const wq4_layer& ly = m.table->layers[l];
        const uint16_t* ul = (l == 0) ? u.x_stage : u.pX2 + static_cast<size_t>(l - 1) * LH;
        StageArgs a{};
        a.sq_in = sq_u;
        a.sq_in_n = nu;
        a.y = u.pQKV + static_cast<size_t>(l) * B * m.Nqkv;
        a.y2 = u.qA;
        a.sq_out = sq_a;
        stage(kStQKV, ly.qkv, ul, a);
        // decode step: the attention output replaces the query block as O's input
        const uint16_t* oin = u.qA;
        int na = tiles_of(kStQKV);
        if (att) {
            ok = ok && att->record(att->ctx, l, cs, &oin, sq_a) == WQ4_OK;
            na = H / 128;
        }
        a = StageArgs{};
        a.sq_in = sq_a;
        a.sq_in_n = na;
        a.sq_u = sq_u;
        a.sq_u_n = nu;
        a.res = ul;
        a.y = u.pO + static_cast<size_t>(l) * LH;
        a.y2 = u.pX1 + static_cast<size_t>(l) * LH;
        a.y3 = u.pV + static_cast<size_t>(l) * LH;
        a.sq_out = sq_x1;
        stage(kStO, ly.o, oin, a);

        a = StageArgs{};
        a.sq_in = sq_x1;
        a.sq_in_n = tiles_of(kStO);
        a.y = u.pGU + static_cast<size_t>(l) * B * 2 * F;
        a.y2 = u.pM + static_cast<size_t>(l) * B * F;
        stage(kStGU, ly.gate_up, u.pX1 + static_cast<size_t>(l) * LH, a);

        a = StageArgs{};
        a.res = u.pX1 + static_cast<size_t>(l) * LH;
        a.y = u.pD + static_cast<size_t>(l) * LH;
        a.y2 = u.pX2 + static_cast<size_t>(l) * LH;
        a.sq_out = sq_u;                      // the next layer's (or the LM head's) input
        stage(kStDOWN, ly.down, u.pM + static_cast<size_t>(l) * B * F, a);
        nu = tiles_of(kStDOWN);
    }
    StageArgs a{};
    a.sq_in = sq_u;
    a.sq_in_n = nu;
    a.res = u.pX2 + static_cast<size_t>(L - 1) * LH;
    a.y = u.logits;
    a.y3 = u.pV + static_cast<size_t>(L) * LH;
    stage(kStLM, m.table->lm_head, u.pX2 + static_cast<size_t>(L - 1) * LH, a);
    return ok ? WQ4_OK : WQ4_ERR_CUDA;
}

}  // namespace wq4
