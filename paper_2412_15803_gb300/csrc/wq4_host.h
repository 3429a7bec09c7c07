// wq4_host.h -- host-side helpers shared by the library's translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "wq4_attn.h"

#include <array>
#include <cstddef>
#include <cstdint>

namespace wq4 {

constexpr int kMaxDevices = 64;

struct DeviceInfo {
    int sm_count = 0;
    int smem_optin = 0;      // max dynamic shared memory per block (opt-in)
    int coop_launch = 0;     // cooperative launch supported
    int dev = 0;             // its number
    uint32_t* status = nullptr;   // device address of the library's status word there
};

// Properties of the current device, queried once per device.
const DeviceInfo* current_device_info(int* device_out);

// Device address of the library's status word on the current device.
uint32_t* status_word();

// The copies that wq4_test_copy_stall leaves out.
int test_copy_stall();

// wq4_paged_attention that also leaves the sums of squares of every (row,
// query head)'s outputs in sq [batch][sq_ld] (null: none).
int launch_paged_attention(const wq4_kv_cache* cache, const uint16_t* q, int q_stride, const int32_t* seq_lens,
                           uint16_t* out, int out_stride, int batch, int n_q_heads, float scale, void* workspace,
                           size_t workspace_bytes, float* sq, int sq_ld, cudaStream_t stream);

// 2-D tiled tensor map (driver entry point, no libcuda link): dims
// {inner, outer} elements, row pitch row_bytes, box {box_inner, box_outer}.
bool encode_tensor_map_2d(CUtensorMap* m, CUtensorMapDataType dt, const void* base, uint64_t inner,
                          uint64_t outer, uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer,
                          CUtensorMapSwizzle swz);

// 3-D tiled tensor map: extents innermost first, byte strides of the outer two
// dimensions, box extents.
bool encode_tensor_map_3d(CUtensorMap* m, CUtensorMapDataType dt, const void* base, const std::array<uint64_t, 3>& dims,
                          const std::array<uint64_t, 2>& strides, const std::array<uint32_t, 3>& box,
                          CUtensorMapSwizzle swz);

// The batched GEMV (wq4_bgemv.cu): any N, K % 32 == 0, batch 1-32, scales at any
// 2-byte address.  check_scales (a call of wq4_gemm; 16-byte aligned scales, K %
// 256 == 0, batch <= 16 only): flag scales beyond +-8188 in the status word and
// copy weights only after the previous kernel, as wq4_gemm promises.
int launch_bgemv(const DeviceInfo* di, const uint32_t* W, const uint16_t* s, const uint16_t* x, uint16_t* y, int N,
                 int K, int batch, cudaStream_t stream, bool check_scales = false);

inline bool aligned(const void* p, size_t a)
{
    return (reinterpret_cast<uintptr_t>(p) % a) == 0;
}

inline bool overlaps(const void* a, size_t na, const void* b, size_t nb)
{
    const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
    return pa < pb + nb && pb < pa + na;
}

inline size_t align_up(size_t v, size_t a)
{
    return (v + a - 1) / a * a;
}

}  // namespace wq4
