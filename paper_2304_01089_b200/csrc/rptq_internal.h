// Internal declarations shared by the translation units of librptq.so. Not part of the C boundary.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "rptq.h"

namespace rptq {

// One entry per group of 32 padded positions ("unit"). A unit belongs to one cluster.
struct UnitInfo {
    float inv_s;      // (float)(1.0 / (double)s_c)
    int32_t zc;       // z_c - 0x4B400000: added to the bit pattern of (t + 1.5*2^23)
    int32_t j0;       // reordered channel index of the unit's first position
    int32_t nvalid;   // real (non-pad) positions in the unit, 0..32; real ones come first
};
static_assert(sizeof(UnitInfo) == 16, "UnitInfo is loaded as one 16-byte vector");

// Flags of one contraction step (32 consecutive padded positions) along K.
// FIRST / LAST: first / last step of its cluster (a cluster's steps need not be adjacent); SKIP: no
// cluster; BUF: which of the two accumulators the cluster uses.
enum : uint8_t { STEP_FIRST = 1, STEP_LAST = 2, STEP_SKIP = 4, STEP_BUF = 8 };

constexpr int kMaxGemmSegments = 1024;

// Byte offset of the 64-byte piece (row n, K block kb) in the tile-major packed weight buffer.
__host__ __device__ inline int64_t weight_tile_offset(int64_t n, int kb, int n_kb) { return ((n >> 7) * n_kb + kb) * 8192 + (n & 127) * 64; }

}  // namespace rptq

struct rptq_layout {
    int C = 0, g = 0, bits = 0, K_pad = 0, device = -1;
    int64_t row_bytes = 0;
    int n_units = 0;   // K_pad / 32
    int n_seg = 0;     // clusters with n_c > 0
    std::vector<int32_t> perm, size, zero;
    int z_min = 0, z_max = 0;            // over the non-empty clusters
    std::vector<int32_t> pos;            // [C]       padded position of reordered channel j
    std::vector<int32_t> unit_cluster;   // [n_units] owning cluster, -1 past the last cluster
    std::vector<float> scale;
    bool in_cluster_order = false;       // the units' clusters never decrease along the row
    std::vector<int32_t> cl_unit0;       // [g + 1] with in_cluster_order: first unit of each cluster, then the number of used units
    std::vector<int32_t> cl_ch_lo, cl_ch_hi;   // [g] smallest and largest channel of each cluster (C, -1 when empty)
    // device tables
    uint16_t* d_src = nullptr;          // [K_pad] channel read for each padded position (at pads: some channel, the code is masked)
    int32_t* d_jidx = nullptr;          // [K_pad] reordered index at each padded position, -1 at pads
    rptq::UnitInfo* d_unit = nullptr;   // [n_units]
    uint8_t* d_step_flags = nullptr;    // [n_units]
    float* d_seg_scale = nullptr;       // [n_seg]  s_c of the non-empty clusters, in the order their last steps come
    uint8_t* d_seg_buf = nullptr;       // [n_seg]  the accumulator each of them uses, same order
    float* d_cl_sz = nullptr;           // [g]      s_c * z_c
    float* d_cl_n = nullptr;            // [g]      n_c
    int32_t* d_seg_cluster = nullptr;   // [n_seg]  the cluster of each entry of d_seg_scale
    float2* d_unit_sz = nullptr;        // [n_units] {s_c, (float) z_c} of the unit's cluster ({1, 0} where there is none)
    int32_t* d_unit_cluster = nullptr;  // [n_units]
    int32_t* d_cl_unit0 = nullptr;      // [g + 1] cl_unit0
};

namespace rptq {

// The cluster GEMM for at most 16 tokens (small_m_gemm.cu).
struct SmallMParams {
    const uint8_t* a; int64_t a_row_bytes; int M, K_pad, n_units, n_kb;
    const uint8_t* w; int n_wtiles;
    const uint8_t* step_flags; const float2* unit_sz; const float* cl_sz; int g;
    const float* corr; const float* s_w; const int32_t* wsum; int64_t ld_w; const float* bias;
    int N, act, y_dtype; void* y; int64_t ldy; int* status;
    int tiles_per_block;                     // weight tiles of 128 channels a block takes (set by the launch)
};
namespace smallm {
bool fits(int M, int bits, int K_pad);
int launch(const SmallMParams& p, int bits, int device, cudaStream_t st);
}

// Programmatic dependent launch: every kernel of the library is launched so that its blocks may become resident, and
// run their set-up, while the kernel before it in the stream drains. pdl_wait() returns when that kernel has
// completed and its writes are visible; nothing but the layout's own tables (uploaded before rptq_layout_create
// returned) is touched before it. The kernel before may still be writing while this one is resident, so what a kernel of the
// library writes (codes, outputs, code sums, the no-alloc correction) is read with ordinary loads: the read-only path (__ldg, const
// __restrict__ arguments) is for what nothing writes while the kernel lives, the layout's tables and the weights'. pdl_trigger() lets the next kernel's blocks come in. A LayerNorm + GEMM pair of one token:
// 10.9 -> 10.0 us on the device, a LayerNorm launch 3.8 -> 2.7 us.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline int launch_kernel(void (*fn)(P...), dim3 grid, unsigned threads, size_t smem, unsigned cluster, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, fn, args...) == cudaSuccess ? RPTQ_OK : RPTQ_ERR_CUDA;
}

constexpr int kMaxDevices = 64;
// Names the calling thread's current context; no other context of the process ever has the same number. 0 where there is none yet.
uint64_t context_id();

// The dynamic shared memory a kernel may ask for, raised once per kernel and context (it is an attribute of the kernel in the
// context: one made after a reset, or beside the first, starts without it) to the most that any launch of it asks for. The
// runtime call costs about a microsecond of host time. `done`: a static of the caller.
struct SmemAllowed { std::atomic<uint64_t> context[kMaxDevices]; };
inline int allow_smem(const void* fn, int device, int bytes, SmemAllowed& done)
{
    const uint64_t id = context_id();
    const bool known = id != 0 && device >= 0 && device < kMaxDevices;
    if (known && done.context[device].load(std::memory_order_acquire) == id) return RPTQ_OK;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return RPTQ_ERR_CUDA;
    if (known) done.context[device].store(id, std::memory_order_release);
    return RPTQ_OK;
}

int sm_count(int device);    // of the device, asked for once; 0 on failure

int* device_status_word();   // the current context's status word (allocated with its first layout), RPTQ_OK when clear; nullptr on failure

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace rptq
