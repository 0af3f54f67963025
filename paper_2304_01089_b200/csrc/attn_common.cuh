// Shared by the attention kernels: launch parameters, packed-row readers and conversions of codes, and the host-side checks of
// per-head layouts.
#pragma once
#include <cuda_fp16.h>

#include "rptq_internal.h"
#include "tc.cuh"
#include "unpack.cuh"

namespace rptq {
namespace attn {

using namespace tc;

constexpr int MAX_UNITS = 8;                 // units of 32 positions per head
constexpr float NEG_BIG = -1.0e30f;

// One attention call. KV-only calls (rptq_attention_kv) have q_f16 and no q codes.
struct AttnParams {
    const uint8_t *q, *k, *v;
    const __half* q_f16; int64_t ldq;
    int64_t q_row_bytes, k_row_bytes, v_row_bytes;
    int bits_q, bits_k, bits_v;
    int Tq, Tk, H, hd, gh_k, gh_v, causal;   // Tq queries and Tk keys per sequence; hd channels per head (KV-only)
    const int32_t *cl_unit0_k, *cl_unit0_v;  // first unit of every cluster, one past the last one's end
    const int32_t *unit_cluster_k;
    const float2 *unit_sz_q, *unit_sz_k, *unit_sz_v;
    const uint16_t *src_k, *src_v;           // channel at each padded position
    const int32_t *jidx_k, *jidx_v;          // -1 at pad positions
    float inv_sP, s_P, qk_scale_log2e;
    __half* out;
    int64_t ldo;
    uint8_t* p_dbg;
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t pack_half2(float a, float b)
{
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// The nibbles at bit B of the two halves of w as a pair of fp16 numbers n - 8 (B = 0, 4, 8, 12).
template <int B>
__device__ __forceinline__ uint32_t nib_half(uint32_t w)
{
    const uint32_t t = ((B <= 6 ? w << (6 - B) : w >> (B - 6)) & 0x03C003C0u) | 0x4C004C00u;      // 16 + n
    const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&t), __float2half2_rn(-24.0f));
    return *reinterpret_cast<const uint32_t*>(&r);
}
// The bytes at bit B of the two halves of w as a pair of fp16 numbers n - 128 (B = 0, 8).
template <int B>
__device__ __forceinline__ uint32_t byte_half(uint32_t w)
{
    const uint32_t t = ((w >> B) & 0x00FF00FFu) | 0x64006400u;                                    // 1024 + n
    const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&t), __float2half2_rn(-1152.0f));
    return *reinterpret_cast<const uint32_t*>(&r);
}

// Bytes per key row of a staged packed tile: the 16-byte chunks of a head's units (one more where the head's first unit need not start
// on a boundary), rounded up to an odd number of chunks so that the eight rows (or four pairs of rows) a warp reads at once
// lie in different banks.
__host__ __device__ inline int raw_pitch(int bits, int units)
{
    const int c = (4 * bits * units + 15) / 16 + (bits == 3 ? 1 : 0);
    return 16 * (c | 1);
}

// Unit `unit` of a packed row (`row` 4-byte aligned for 3-bit codes, 16-byte aligned otherwise) as 32 bytes.
__device__ __forceinline__ void load_unit(const uint8_t* row, int unit, int bits, uint32_t (&o)[8])
{
    if (bits == 4) {
        const uint4 t = *(reinterpret_cast<const uint4*>(row) + unit);
        const uint32_t p[4] = {t.x, t.y, t.z, t.w};
        unpack_act32<4>(p, o);
    } else if (bits == 3) {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(row) + unit * 3;
        const uint32_t p[3] = {w[0], w[1], w[2]};
        unpack_act32<3>(p, o);
    } else {
        const uint4* w = reinterpret_cast<const uint4*>(row) + unit * 2;
        const uint4 a = w[0], b = w[1];
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    }
}

// Largest number of units a head takes in the layout (whose g clusters are n_heads equal groups).
inline int max_units_per_head(const rptq_layout_t* L, int n_heads)
{
    const int gh = L->g / n_heads;
    int m = 0;
    for (int h = 0; h < n_heads; ++h) {
        const int n = L->cl_unit0[(size_t)((h + 1) * gh)] - L->cl_unit0[(size_t)(h * gh)];
        m = n > m ? n : m;
    }
    return m;
}

// Head h's clusters hold exactly the channels h * hd .. (h + 1) * hd - 1.
inline bool heads_own_their_channels(const rptq_layout_t* L, int n_heads)
{
    if (L->C % n_heads) return false;
    const int gh = L->g / n_heads, hd = L->C / n_heads;
    for (int c = 0; c < L->g; ++c) {
        const size_t i = (size_t)c;
        if (L->cl_ch_hi[i] >= 0 && (L->cl_ch_lo[i] / hd != c / gh || L->cl_ch_hi[i] / hd != c / gh)) return false;
    }
    return true;
}

}  // namespace attn

// The decode kernel (attention_decode.cu): few queries per sequence, the keys split over a cluster of blocks.
namespace attn_decode {
bool fits(const attn::AttnParams& p, bool kv, int units_k, int units_v);     // false: the prefill kernel takes the call
int launch(const attn::AttnParams& p, bool kv, int units_k, int units_v, int n_seq, int dev, int n_sm, cudaStream_t st);
}
// The kernel for more queries (attention_prefill.cu). zq_min, zq_max: the range of the query's zero points (integer calls);
// v_heads_local: head h of V owns the channels h * hd .. (h + 1) * hd - 1.
namespace attn_prefill {
int launch(const attn::AttnParams& p, bool kv, int zq_min, int zq_max, int units_k, int units_v, int n_seq, bool v_heads_local, int dev, int n_sm, cudaStream_t st);
}
}  // namespace rptq
