// rptq_cluster_gemm: cluster-segmented integer GEMM (Appendix, second computation method).
//
//   acc_c[m][n] = sum_{k in segment c} X_q[m][k] * W_q[n][k]        int32, tcgen05.mma kind::i8
//   y[m][n]     = s_w[n] * sum_c s_c * (acc_c[m][n] - z_c * Wsum_c[n])  (+ bias) (ReLU) (re-quantise)
//
// Two variants of one kernel template. NCTA = 1: one persistent CTA per SM works on 128 (tokens) x
// 256 (output channels) tiles. NCTA = 2: the two CTAs of a cluster (an SM pair) share a 256 x 256
// tile through tcgen05.mma.cta_group::2 -- each CTA stages and unpacks its own 128 token rows and
// its own 128 of the 256 weight rows, which halves the weight unpacking and the shared-memory
// traffic per MMA; the first CTA of the pair issues the MMAs for both and its commits arrive on
// both CTAs' barriers; every CTA drains its own 128 accumulator lanes. No load is multicast.
// Warp roles (per CTA):
//   warp 0      bulk-copy producer: one contiguous 8 KiB cp.async.bulk per 128 weight rows per K
//               block (the packed weights are stored tile-major for this) into a ring of stages
//   warps 4-7   (MODE_DEQ: 4-11, two groups) unpack: packed codes -> 8-bit operands, written in the K-major 128-byte-swizzled
//               layout that the tensor core reads (weights become 16 * w, see unpack.cuh). The
//               activation codes of a K block are 48/64/128 bytes per token row, too narrow for the
//               copy engine to move at speed (measured: ~10 clk per row), so each unpack thread
//               fetches the words of its own items with cp.async into a private ring of
//               shared-memory slots, one to three K blocks ahead. 8-bit codes need no unpacking: with
//               CTA pairs they are copied straight into the operand stage (template flag A8)
//   warp 1      MMA issuer (the whole warp in converged control flow, one elected lane issues):
//               four tcgen05.mma (K = 32 each) per K block; each cluster accumulates
//               into one of two 256-column TMEM buffers (the layout's step flags say which) and
//               is committed at its last step. A cluster's steps need not be adjacent: in the
//               interleaved unit order a small cluster's step sits between those of a large one,
//               which keeps its buffer, so the small cluster's drain runs under the large
//               cluster's remaining products
//   warps 2-3   column tables: zero-point correction, s_w and bias of the columns of the tile to come, and
//               with per-cluster weight parameters the coefficients of each cluster's drain (they are
//               the same for every token row: formed once per block instead of in every epilogue thread.
//               1024 x 4096 x 16384, 16 clusters, LayerNorm included: 428 -> 147 us, 113 with all that follows)
//   warps 8-15  (MODE_DEQ: 12-19) epilogue: drain a finished cluster's accumulator (tcgen05.ld), add s_c * acc into
//               fp32 running sums held in registers while the next cluster's MMAs run; after the
//               last cluster apply the zero-point correction, s_w, bias, activation, and store
// Every wait is bounded: a wait that runs out sets RPTQ_ERR_DEVICE_TIMEOUT in the status word, every later one returns at once, the
// producer and the MMA issuer drain and stop, and the other roles run their loops to the end (whole warps that would
// leave them lane by lane could part).
#include <cuda_fp16.h>

#include <mutex>
#include <type_traits>

#include "pack.cuh"
#include "rptq_internal.h"
#include "tc.cuh"
#include "unpack.cuh"

namespace rptq {
namespace gemm {

using namespace tc;

constexpr int TILE_M = 128, TILE_N = 256, KBLK = 128;   // TILE_M is per CTA
enum { MODE_INT = 0, MODE_ASYM = 1, MODE_DEQ = 2 };      // see cluster_gemm_kernel
// MODE_DEQ: two groups of unpack warps (its conversions take three times as long), and an epilogue without running sums
constexpr int threads_of(int mode) { return mode == MODE_DEQ ? 640 : 512; }
constexpr int TABLE_WARP0 = 2, N_TABLE_WARPS = 2;
constexpr int UNPACK_WARP0 = 4, GROUP_WARPS = 4;          // warps of an unpack group
constexpr int n_unpack_warps(int mode) { return mode == MODE_DEQ ? 2 * GROUP_WARPS : GROUP_WARPS; }
constexpr int N_EPI_WARPS = 8;
// registers per thread after the in-kernel re-partition (the block is launched with 128, MODE_DEQ 96 each): the
// producer / MMA-issuer group, the unpack groups, the two epilogue groups (128 running sums per thread, none in MODE_DEQ). With 40 for its
// first group MODE_DEQ spills there, in the loops that feed the tensor core (one block, 8 bits, 128 x 9216 x 9216: 76 us, with 48 67)
constexpr int regs_wg0(int mode) { return mode == MODE_DEQ ? 48 : 40; }
constexpr int regs_unpack(int mode) { return mode == MODE_DEQ ? 104 : 88; }
constexpr int regs_epi(int mode) { return mode == MODE_DEQ ? 112 : 192; }
constexpr int regs_all(int mode) { return 128 * regs_wg0(mode) + 32 * n_unpack_warps(mode) * regs_unpack(mode) + 256 * regs_epi(mode); }
static_assert(regs_all(MODE_INT) <= 128 * 512 && regs_all(MODE_DEQ) <= 96 * 640, "register pool");
constexpr int A8_BYTES = TILE_M * KBLK;                  // 16 KiB of 8-bit activation operands per stage
constexpr int WTILE_BYTES = 8192;                        // one packed weight tile: 128 rows x 64 bytes

__host__ __device__ constexpr int w_rows(int ncta) { return TILE_N / ncta; }           // weight rows staged per CTA
// packed weight stages; the single-CTA variant (at most 128 tokens) is a weight stream and takes what shared memory is left
__host__ __device__ constexpr int n_p_stages(int ncta, int bits, int mode) 
{
    if (ncta == 2) return 4;
    return mode == MODE_DEQ ? 3 : bits == 3 ? 5 : 4;
}
__host__ __device__ constexpr int n_u_stages(int ncta, bool a8) { return ncta == 2 ? (a8 ? 5 : 4) : 2; }   // operand stages
// ring of packed activation K blocks fetched ahead by the unpack threads: one slot per token row
// per K block; the pitch is an odd number of 16-byte units (4 bits: four, and the pieces of a slot exchanged) so that the threads'
// vector reads of their own slots do not collide in the banks
__host__ __device__ constexpr int a_slot_pitch(int bits, int mode) { return mode == MODE_DEQ ? (bits == 8 ? 80 : 48) : bits == 3 ? 48 : bits == 4 ? 64 : 16 * bits + 16; }
// (one block, 3 bits: two K blocks, since the output staging has the room of the others; as fast as four were, and three, all that fits, are 1 to
// 3 % slower: 17 x 2048 x 8192 with clustered weights 15.7 and 16.0 us)
__host__ __device__ constexpr int n_a_stages(int ncta, int bits, int mode) { return bits == 8 || (ncta == 1 && bits == 3 && mode != MODE_DEQ) ? 2 : mode == MODE_DEQ ? 3 : 4; }

struct SmemLayout {
    int u_stage, p_stage, a_stage, off_p, off_a, off_flags, off_seg_scale, off_seg_buf, off_tab, off_seg_tab, off_seg_cl, off_stage, off_bar, total;
};
constexpr int OUT_ROW = 64;                              // output staging buffer of an epilogue warp: 32 rows of so many bytes (128 would fit in
                                                         // MODE_DEQ's one-block instances only, and is no faster there)
// rows of the column tables: zero-point correction (none in MODE_DEQ), s_w (none in MODE_ASYM, which applies it per cluster), bias. Rows that hold
// one constant cost the 8-bit one-block instance of MODE_ASYM a weight stage (32 x 4096 x 12288: 25.7 us with four, 26.2 with three)
__host__ __device__ constexpr int n_tab_rows(int mode) { return mode == MODE_INT ? 3 : 2; }
constexpr int SEG_SLOTS = 2;                             // ASYM: clusters whose column tables are held at a time
__host__ __device__ constexpr SmemLayout smem_layout(int ncta, int bits, bool a8, int mode)
{
    const bool asym = mode == MODE_ASYM;
    SmemLayout s{};
    s.u_stage = A8_BYTES + w_rows(ncta) * KBLK;
    s.p_stage = w_rows(ncta) * KBLK / 2;
    s.a_stage = a8 ? 0 : n_unpack_warps(mode) / GROUP_WARPS * TILE_M * a_slot_pitch(bits, mode);      // 8-bit activations go straight to the operand stage
    s.off_p = n_u_stages(ncta, a8) * s.u_stage;
    s.off_a = s.off_p + n_p_stages(ncta, bits, mode) * s.p_stage;
    s.off_flags = s.off_a + n_a_stages(ncta, bits, mode) * s.a_stage;
    s.off_seg_scale = s.off_flags + 2048;
    s.off_seg_buf = s.off_seg_scale + (mode == MODE_INT ? kMaxGemmSegments * 4 : 0);
    s.off_tab = s.off_seg_buf + (mode == MODE_DEQ ? 0 : kMaxGemmSegments);          // (DEQ: one accumulator per tile, no clusters)
    s.off_seg_tab = s.off_tab + 2 * n_tab_rows(mode) * TILE_N * 4;
    s.off_seg_cl = s.off_seg_tab + (asym ? SEG_SLOTS * 2 * TILE_N * 4 : 0);
    s.off_stage = s.off_seg_cl + (asym ? kMaxGemmSegments * 2 : 0);
    s.off_bar = s.off_stage + N_EPI_WARPS * 32 * OUT_ROW;
    s.total = s.off_bar + 320;
    return s;
}

struct Params {
    int M, N, n_kb, n_seg, g;
    int tiles_m, n_items;        // work items: the first n_full are whole tiles, every further tile is cut into 1 << split strips of columns
    int n_full, split;
    const uint8_t* a_codes;      // [M][a_row_bytes]
    int64_t a_row_bytes;
    const uint8_t* w_codes;      // tile-major: n_wtiles * n_kb tiles of 8 KiB
    int n_wtiles;
    const uint8_t* step_flags;
    const float* seg_scale;      // [n_seg] in the order the clusters' last steps come
    const uint8_t* seg_buf;      // [n_seg] accumulator of each, same order
    const float* cl_sz;
    const float* corr;           // optional [N]: sum_c s_c z_c Wsum_c[n] computed beforehand, else NULL
    const float* s_w;
    const int32_t* wsum;
    int64_t ld_w;
    // per-cluster asymmetric weight parameters (template flag ASYM): [g][ld_w] tables of s^W_c[n] and
    // z^W_c[n], the cluster of every entry of seg_scale, n_c, and the activation code sums [M][g]
    const float* sw_c;
    const int32_t* zw_c;
    const int32_t* seg_cluster;
    const float* cl_n;
    const int32_t* xsum;
    // first computation method (template mode MODE_DEQ): per unit of 32 positions {s_c, (float) z_c}
    const float2* unit_sz;
    const float* bias;
    int act, y_dtype;
    void* y;
    int64_t ldy;
    const UnitInfo* out_unit;
    int out_bits;
    int64_t out_row_bytes;
    int* status;
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// One contiguous global -> shared copy by the copy engine; completion is counted on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// The two tensor-core instructions below are executed by the WHOLE issuing warp in converged
// control flow; elect.sync picks the one lane that issues. Measured on an operand-resident loop: a
// tcgen05.mma issued from a branch that a single lane took costs the issuing thread ~120 clocks,
// one issued this way ~85, against 134 clocks of tensor-pipe time per instruction.
template <int NCTA>
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if constexpr (NCTA == 1) {
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
            ::"r"(bar) : "memory");
    } else {
        // arrives on the barrier at this offset in both CTAs of the pair
        const uint16_t mask = 3;
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
            ::"r"(bar), "h"(mask) : "memory");
    }
}
template <int NCTA>
__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (NCTA == 1) {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "@q tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
    }
}
// The four products of a K block inside one cluster, and the commit that frees its operand stage, with one election: a0, b0 the low words of
// the first step's descriptors (the high words are the same for every tile; the start address counts 16-byte units, 32 bytes a step)
constexpr uint32_t DESC_HI = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);       // of smem_desc_sw128
template <int NCTA>
__device__ __forceinline__ void tc_block_i8(uint32_t d_tmem, uint32_t a0, uint32_t b0, uint32_t idesc, uint32_t bar)
{
#define RPTQ_BLOCK(GROUP, COMMIT)                                                                                    \
    "{\n\t.reg .pred q, t;\n\t.reg .b64 da, db;\n\t.reg .b32 a, b;\n\t"                                               \
    "elect.sync _|q, 0xffffffff;\n\tsetp.eq.u32 t, 0, 0;\n\t"                                                         \
    "mov.b64 da, {%1, %4};\n\tmov.b64 db, {%2, %4};\n\t"                                                              \
    "@q tcgen05.mma.cta_group::" GROUP ".kind::i8 [%0], da, db, %3, t;\n\t"                                           \
    "add.u32 a, %1, 2;\n\tadd.u32 b, %2, 2;\n\tmov.b64 da, {a, %4};\n\tmov.b64 db, {b, %4};\n\t"                      \
    "@q tcgen05.mma.cta_group::" GROUP ".kind::i8 [%0], da, db, %3, t;\n\t"                                           \
    "add.u32 a, %1, 4;\n\tadd.u32 b, %2, 4;\n\tmov.b64 da, {a, %4};\n\tmov.b64 db, {b, %4};\n\t"                      \
    "@q tcgen05.mma.cta_group::" GROUP ".kind::i8 [%0], da, db, %3, t;\n\t"                                           \
    "add.u32 a, %1, 6;\n\tadd.u32 b, %2, 6;\n\tmov.b64 da, {a, %4};\n\tmov.b64 db, {b, %4};\n\t"                      \
    "@q tcgen05.mma.cta_group::" GROUP ".kind::i8 [%0], da, db, %3, t;\n\t"                                           \
    "@q tcgen05.commit.cta_group::" GROUP ".mbarrier::arrive::one.shared::cluster" COMMIT "\n\t}"
    if constexpr (NCTA == 1)
        asm volatile(RPTQ_BLOCK("1", ".b64 [%5];") ::"r"(d_tmem), "r"(a0), "r"(b0), "r"(idesc), "r"(DESC_HI), "r"(bar) : "memory");
    else
        asm volatile(RPTQ_BLOCK("2", ".multicast::cluster.b64 [%5], %6;") ::"r"(d_tmem), "r"(a0), "r"(b0), "r"(idesc), "r"(DESC_HI), "r"(bar), "h"((uint16_t)3) : "memory");
#undef RPTQ_BLOCK
}
// bf16 x bf16 -> fp32, same operand layout and issue pattern as tc_mma_i8 (K = 16 elements = 32 bytes)
template <int NCTA>
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (NCTA == 1) {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "elect.sync _|q, 0xffffffff;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
    }
}
// 16 lanes x 32 columns: v[4 j + 2 r + c] is row lane / 4 + 8 r, column 8 j + 2 (lane % 4) + c
__device__ __forceinline__ void tc_ld16xn(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
// 16 lanes x 16 columns in the same manner
__device__ __forceinline__ void tc_ld16xn(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(taddr) : "memory");
}
// four (two) 8 x 8 matrices of 16-bit values, matrix j's rows at the addresses that lanes 8 j .. 8 j + 7 name
__device__ __forceinline__ void stmatrixn(uint32_t addr, const uint32_t (&f)[2])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x2.shared.b16 [%0], {%1, %2};" ::"r"(addr), "r"(f[0]), "r"(f[1]) : "memory");
}
__device__ __forceinline__ void stmatrixn(uint32_t addr, const uint32_t (&f)[4])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(f[0]), "r"(f[1]), "r"(f[2]), "r"(f[3]) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t addr, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
// kind::i8, D = s32, A = unsigned 8-bit (activation codes), B = signed 8-bit (weights), both
// K-major, M = 128 per CTA, N = 256.
__host__ __device__ constexpr uint32_t instr_desc(int ncta)
{
    return (2u << 4) | (0u << 7) | (1u << 10) | ((uint32_t)(TILE_N >> 3) << 17) | ((uint32_t)((TILE_M * ncta) >> 4) << 24);
}

// kind::f16 with bfloat16 operands: D = fp32, A and B bfloat16, both K-major
__host__ __device__ constexpr uint32_t instr_desc_bf16(int ncta)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TILE_N >> 3) << 17) | ((uint32_t)((TILE_M * ncta) >> 4) << 24);
}
// two fp32 values rounded to bfloat16 (nearest even): lo in bits 0-15, hi in bits 16-31
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
// Byte i of w as the float 2^23 + byte: the byte is dropped into the low mantissa bits of 0x4B000000.
template <int I>
__device__ __forceinline__ float byte_as_magic(uint32_t w)
{
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7650u | (uint32_t)I));
}
// Four 8-bit values of one word -> four bfloat16, bytes 0 and 2 in one word, 1 and 3 in the other: v = (byte - c1) * s with
// c1 = 2^23 + z. byte - c1 is exact, the product is rounded once to fp32 and once more to bfloat16.
__device__ __forceinline__ void bytes_to_bf16(uint32_t w, float2 neg_c1, float2 s2, uint32_t& out_02, uint32_t& out_13)
{
    const float2 a = mul2(add2(make_float2(byte_as_magic<0>(w), byte_as_magic<2>(w)), neg_c1), s2);
    const float2 b = mul2(add2(make_float2(byte_as_magic<1>(w), byte_as_magic<3>(w)), neg_c1), s2);
    out_02 = pack_bf16(a.x, a.y);
    out_13 = pack_bf16(b.x, b.y);
}
// The two's complement nibbles in bits 0-3 and 16-19 as bfloat16: n with its sign bit flipped, dropped into the mantissa of
// 128, is 136 + w.
__device__ __forceinline__ uint32_t nibbles_to_bf16(uint32_t w)
{
    uint32_t d;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"((w & 0x000F000Fu) ^ 0x43084308u), "r"(0x43084308u));
    return d;
}

// ASYM: the weights carry one scale and one zero point per (cluster, output channel) (Appendix,
// W~_q,i = Q_k(W~_i, s^W_i, z^W_i)). The stored nibble is the code minus 8, so the integer products
// are acc' = sum X_q (W_q - 8) and the second method's four terms become
//   Y_q,c = acc'_c - (z^W_c[n] - 8) * sum_k X_q[m][k] - z^X_c * Wsum_c[n] + n_c z^X_c z^W_c[n] :
// the first two are applied per element while a cluster's accumulator is drained, the last two are a
// constant of the output column.
// MODE_DEQ: the first computation method of the Appendix (de-quantise, then one floating-point product):
// the unpack warps write X^ = s_c (X_q - z_c) as bfloat16 and the weight codes as bfloat16 integers, the MMAs are kind::f16 into ONE fp32 accumulator per tile -- no per-cluster
// accumulators, no drains at cluster boundaries -- and s_w[n] multiplies the finished sum. A bfloat16
// operand row of 128 bytes holds 64 positions, so a K block of 128 positions is two operand stages.
// ROWS (MODE_INT, CTA pairs): the epilogue holds its sums a token row per thread (see there).
template <int BITS, int NCTA, bool A8, int MODE, bool ROWS>
__global__ void __launch_bounds__(threads_of(MODE), 1)
cluster_gemm_kernel(const Params p)
{
    constexpr bool ASYM = MODE == MODE_ASYM, DEQ = MODE == MODE_DEQ;
    static_assert(!(DEQ && A8), "the de-quantising variant unpacks every bit width");
    static_assert(!ROWS || (MODE == MODE_INT && NCTA == 2), "rows");
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    constexpr SmemLayout SL = smem_layout(NCTA, BITS, A8, MODE);
    constexpr int THREADS = threads_of(MODE), EPI_WARP0 = UNPACK_WARP0 + n_unpack_warps(MODE);
    constexpr int TAB_ROWS = n_tab_rows(MODE);
    constexpr int W_ROWS = w_rows(NCTA);                 // weight rows this CTA stages and unpacks
    constexpr int N_P = n_p_stages(NCTA, BITS, MODE), N_U = n_u_stages(NCTA, A8);
    constexpr uint32_t kInstrDesc = DEQ ? instr_desc_bf16(NCTA) : instr_desc(NCTA);      // (of a whole tile)
    // dynamic shared memory is only guaranteed 16-byte alignment: round up to the swizzle span
    // (the offset is the same in both CTAs of a pair, as cta_group::2 descriptors require)
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));

    uint8_t* s_flags = smem + SL.off_flags;
    float* s_seg_scale = reinterpret_cast<float*>(smem + SL.off_seg_scale);
    uint8_t* s_seg_buf = smem + SL.off_seg_buf;
    float* s_tab = reinterpret_cast<float*>(smem + SL.off_tab);           // [2][TAB_ROWS][TILE_N]
    float4* s_seg_tab = reinterpret_cast<float4*>(smem + SL.off_seg_tab); // ASYM: [SEG_SLOTS][TILE_N / 2]
    uint16_t* s_seg_cl = reinterpret_cast<uint16_t*>(smem + SL.off_seg_cl);   // ASYM: the cluster of each segment
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SL.off_bar);
    // barrier indices
    constexpr int B_PFULL = 0, B_PEMPTY = B_PFULL + N_P, B_UFULL = B_PEMPTY + N_P, B_UEMPTY = B_UFULL + N_U,
                  B_ACCFULL = B_UEMPTY + N_U, B_ACCEMPTY = B_ACCFULL + 2, B_TAB = B_ACCEMPTY + 2, B_TABEMPTY = B_TAB + 2,
                  B_SEGFULL = B_TABEMPTY + 2, B_SEGEMPTY = B_SEGFULL + SEG_SLOTS, B_DRAIN = B_SEGEMPTY + SEG_SLOTS, N_BARS = B_DRAIN + 1;
    static_assert(N_BARS * 8 + 16 <= 320, "barrier block too small");
    uint32_t* s_tmem_ptr = reinterpret_cast<uint32_t*>(bars + N_BARS);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem_ptr + 1);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n_steps = p.n_kb * 4;
    const uint32_t cta_rank = NCTA == 2 ? cluster_ctarank() : 0u;       // rank 0 issues the MMAs
    const int pair_id = (int)blockIdx.x / NCTA, n_pairs = (int)gridDim.x / NCTA;
    // Work item -> token tile, first column, and how many times its 256 columns are halved
    auto item_of = [&](int w, int& mt, int& n0) {
        const int sh = w < p.n_full ? 0 : p.split, x = w - p.n_full;
        const int t = sh ? p.n_full + (x >> sh) : w, nt = t / p.tiles_m;
        mt = t - nt * p.tiles_m;
        n0 = nt * TILE_N + (sh ? (x & ((1 << sh) - 1)) * (TILE_N >> sh) : 0);
        return sh;
    };
    // arrive on a barrier that lives in the issuing CTA of the pair
    auto arrive_leader = [&](uint32_t b) { if constexpr (NCTA == 1) mbar_arrive(b); else mbar_arrive_remote(b, 0); };

    if (tid == 0) {
        for (int i = 0; i < N_P; ++i) { mbar_init(bar(B_PFULL + i), 1); mbar_init(bar(B_PEMPTY + i), n_unpack_warps(MODE)); }
        for (int i = 0; i < N_U; ++i) { mbar_init(bar(B_UFULL + i), GROUP_WARPS * NCTA); mbar_init(bar(B_UEMPTY + i), 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(B_ACCFULL + i), 1); mbar_init(bar(B_ACCEMPTY + i), N_EPI_WARPS * NCTA); mbar_init(bar(B_TAB + i), N_TABLE_WARPS);
            mbar_init(bar(B_TABEMPTY + i), N_EPI_WARPS);
        }
        for (int i = 0; i < SEG_SLOTS; ++i) { mbar_init(bar(B_SEGFULL + i), N_TABLE_WARPS); mbar_init(bar(B_SEGEMPTY + i), N_EPI_WARPS); }
        mbar_init(bar(B_DRAIN), 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < n_steps; i += THREADS) s_flags[i] = p.step_flags[i];
    if constexpr (!DEQ) for (int i = tid; i < p.n_seg; i += THREADS) {
        if constexpr (!ASYM) s_seg_scale[i] = p.seg_scale[i] * 0.0625f;        // operands were 16 * w
        s_seg_buf[i] = p.seg_buf[i];
    }
    if constexpr (ASYM) for (int i = tid; i < p.n_seg; i += THREADS) s_seg_cl[i] = (uint16_t)p.seg_cluster[i];
    if (warp == 1) {
        if constexpr (NCTA == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(s_tmem_ptr)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(s_tmem_ptr)) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    pdl_trigger();
    pdl_wait();                                        // (only the layout's tables have been read so far)
    __syncthreads();
    if constexpr (NCTA == 2) cluster_sync_all();       // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem_base = *s_tmem_ptr;

    // The register file is re-partitioned by warpgroup (the epilogue holds 128 running sums per
    // thread); each setmaxnreg is executed by the four warps of its group at one place.
    if (warp < UNPACK_WARP0) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(regs_wg0(MODE)));
      if (warp == 0) {
        // ------------------------------------------------------------ bulk-copy producer
        if (lane == 0) {
            uint32_t n_issued = 0;
            bool ok = true;
            for (int t = pair_id; t < p.n_items && ok; t += n_pairs) {
                // weight rows this CTA stages: whole 128-row tiles, or part of one; tiles past the end of the buffer are
                // skipped (their columns are never stored)
                int mt, n0;
                const int sh = item_of(t, mt, n0), rows = W_ROWS >> sh, row0 = n0 + (int)cta_rank * rows;
                const uint32_t bytes = rows < 128 ? (uint32_t)rows * 64 : (uint32_t)WTILE_BYTES;
                int n_valid = p.n_wtiles - (row0 >> 7);
                const int n_copies = rows < 128 ? 1 : rows >> 7;
                n_valid = n_valid < 0 ? 0 : (n_valid > n_copies ? n_copies : n_valid);
                const uint8_t* src = p.w_codes + (int64_t)(row0 >> 7) * p.n_kb * WTILE_BYTES + (row0 & 127) * 64;
                for (int kb = 0; kb < p.n_kb; ++kb, ++n_issued) {
                    const int s = n_issued % N_P;
                    const uint32_t ph = (n_issued / N_P) & 1;
                    if (!mbar_wait(bar(B_PEMPTY + s), ph ^ 1, s_abort)) { ok = false; break; }
                    const uint32_t dst = smem_base + SL.off_p + s * SL.p_stage;
                    mbar_arrive_expect_tx(bar(B_PFULL + s), (uint32_t)n_valid * bytes);
                    for (int j = 0; j < n_valid; ++j)
                        bulk_load(dst + j * WTILE_BYTES, src + ((int64_t)j * p.n_kb + kb) * WTILE_BYTES, bytes, bar(B_PFULL + s));
                }
            }
            if (!ok) {
                // let copies that were already issued land before the CTA's shared memory goes away
                const uint32_t lo = n_issued > N_P ? n_issued - N_P : 0;
                for (uint32_t i = lo; i < n_issued; ++i) mbar_wait(bar(B_PFULL + i % N_P), (i / N_P) & 1, s_abort, false);
            }
        }
      } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (first CTA of a pair only)
        if (cta_rank == 0) {
            // The whole warp runs this loop in converged control flow (every value in it is the same
            // in all lanes); one elected lane issues. It is a single stream of dependent
            // instructions, so the loop is kept short:
            // stage descriptors are built once, a K block's four step flags come as one word, and a
            // block that lies inside one cluster issues its four MMAs without any test.
            // (the loop runs over all K blocks of all of this pair's tiles with one counter: the
            // lane has few registers)
            uint32_t par = 0;                // bit b: parity of how many clusters accumulator b has held
            bool ok = true;
            const uint64_t a_desc0 = smem_desc_sw128(smem_base);
            const uint32_t* flags4 = reinterpret_cast<const uint32_t*>(s_flags);
            uint32_t f4 = flags4[0];
            const uint32_t total_kb = (uint32_t)(((p.n_items - pair_id + n_pairs - 1) / n_pairs) * p.n_kb);
            // (a pair has at most one strip, its last item; n_full is a multiple of the pairs)
            const uint32_t full_kb = p.split ? (uint32_t)(p.n_full / n_pairs * p.n_kb) : total_kb;
            const uint32_t strip_desc = (kInstrDesc & ~(0x3Fu << 17)) | ((uint32_t)(TILE_N >> p.split >> 3) << 17);
            uint32_t idesc = kInstrDesc;
            int kb = 0;
            if constexpr (DEQ) {
                // One accumulator per tile, the two buffers alternate from tile to tile; every operand
                // stage is half a K block (64 positions, four MMAs of K = 16).
                const uint32_t steps_per_tile = 2u * (uint32_t)p.n_kb, total_steps = 2u * total_kb;
                uint32_t in_tile = 0, b = 0;
                for (uint32_t n = 0; n < total_steps; ++n) {
                    const int st = n % N_U;
                    if (n == 2u * full_kb) idesc = strip_desc;
                    if (in_tile == 0) {
                        if (!mbar_wait_warp(bar(B_ACCEMPTY + b), ((par >> b) & 1u) ^ 1u, s_abort)) { ok = false; break; }
                        tc_fence_after();
                    }
                    if (!mbar_wait_warp(bar(B_UFULL + st), (n / N_U) & 1, s_abort)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t ad = a_desc0 + (uint64_t)(st * (SL.u_stage >> 4)), wd = ad + (uint64_t)(A8_BYTES >> 4);
                    const uint32_t d_tmem = tmem_base + b * TILE_N;
                    tc_mma_bf16<NCTA>(d_tmem, ad, wd, idesc, in_tile);
                    tc_mma_bf16<NCTA>(d_tmem, ad + 2, wd + 2, idesc, 1u);
                    tc_mma_bf16<NCTA>(d_tmem, ad + 4, wd + 4, idesc, 1u);
                    tc_mma_bf16<NCTA>(d_tmem, ad + 6, wd + 6, idesc, 1u);
                    tc_commit<NCTA>(bar(B_UEMPTY + st));
                    if (++in_tile == steps_per_tile) {
                        tc_commit<NCTA>(bar(B_ACCFULL + b));
                        par ^= 1u << b;
                        b ^= 1u;
                        in_tile = 0;
                    }
                }
            } else
            for (uint32_t n_kb_done = 0; n_kb_done < total_kb; ++n_kb_done) {
                    const int s = n_kb_done % N_U;
                    if (n_kb_done == full_kb) idesc = strip_desc;
                    kb = kb + 1 == p.n_kb ? 0 : kb + 1;
                    const uint32_t f4_next = flags4[kb];                              // read while waiting
                    if (!mbar_wait_warp(bar(B_UFULL + s), (n_kb_done / N_U) & 1, s_abort)) { ok = false; break; }
                    tc_fence_after();
                    // the start-address field counts 16-byte units: one stage further, 32 bytes per step;
                    // the weight operand follows the activation operand in the stage
                    const uint64_t ad = a_desc0 + (uint64_t)(s * (SL.u_stage >> 4)), wd = ad + (uint64_t)(A8_BYTES >> 4);
                    if (f4 == 0u || f4 == 0x01010101u * STEP_BUF) {
                        // four steps inside one cluster
                        const uint32_t d_tmem = tmem_base + (f4 ? TILE_N : 0);
                        tc_block_i8<NCTA>(d_tmem, (uint32_t)ad, (uint32_t)wd, idesc, bar(B_UEMPTY + s));
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t f = (f4 >> (8 * j)) & 0xFFu;
                            const uint32_t b = (f / STEP_BUF) & 1u;
                            const uint32_t d_tmem = tmem_base + b * TILE_N;
                            if ((f & (STEP_FIRST | STEP_LAST | STEP_SKIP)) == 0) {       // inside a cluster
                                tc_mma_i8<NCTA>(d_tmem, ad + 2 * j, wd + 2 * j, idesc, 1u);
                                continue;
                            }
                            if (f & STEP_SKIP) continue;
                            if (f & STEP_FIRST) {
                                // the accumulator's previous cluster has been drained
                                if (!mbar_wait_warp(bar(B_ACCEMPTY + b), ((par >> b) & 1u) ^ 1u, s_abort)) { ok = false; break; }
                                tc_fence_after();
                            }
                            tc_mma_i8<NCTA>(d_tmem, ad + 2 * j, wd + 2 * j, idesc, (f & STEP_FIRST) ? 0u : 1u);
                            if (f & STEP_LAST) {
                                tc_commit<NCTA>(bar(B_ACCFULL + b));
                                par ^= 1u << b;
                            }
                        }
                        if (!ok) break;
                        tc_commit<NCTA>(bar(B_UEMPTY + s));  // the stage may be overwritten once these MMAs have read it
                    }
                    f4 = f4_next;
            }
            if (!ok) {
                tc_commit<NCTA>(bar(B_DRAIN));
                mbar_wait(bar(B_DRAIN), 0, s_abort, false);
            }
        }
      } else {
        // ------------------------------------------------------------ column tables
        // Thread tt prepares columns 4 tt .. 4 tt + 3 of the tile ahead of the epilogue: the zero-point
        // correction, s_w and the bias of every tile, and with ASYM for every cluster of the tile the two
        // coefficients its drain needs per column.
        const int tt = tid - TABLE_WARP0 * 32;
        uint32_t n_tile = 0, n_seg_done = 0;
        for (int t = pair_id; t < p.n_items; t += n_pairs, ++n_tile) {
            int mt, n0;
            item_of(t, mt, n0);
            const int n = n0 + 4 * tt;                     // (of a strip, the lanes past its columns work for nothing)
            const bool vec = (p.ld_w & 3) == 0 && n + 4 <= p.ld_w;
            float corr[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (ASYM) {
                // y += s^X_c s^W_c[n] / 16 * (acc' + Z xsum), Z = -16 (z^W_c[n] - 8); the tile constant is
                // sum_c s^X_c z^X_c s^W_c[n] (Wsum_c[n] - n_c z^W_c[n]), summed over the clusters in their own order, not in the order in which
                // they end (2 to 5 % further from 64 bits): step sgi prepares segment sgi and adds cluster sgi
                auto add = [&](int c) {
                    if (!vec) return;
                    const int64_t i = (int64_t)c * p.ld_w + n;
                    const float4 sw4 = __ldg(reinterpret_cast<const float4*>(p.sw_c + i));
                    const int4 zw4 = __ldg(reinterpret_cast<const int4*>(p.zw_c + i)), ws4 = __ldg(reinterpret_cast<const int4*>(p.wsum + i));
                    const float sz = __ldg(p.cl_sz + c), nc = __ldg(p.cl_n + c);
                    corr[0] = __fmaf_rn(sz * sw4.x, (float)ws4.x - nc * (float)zw4.x, corr[0]);
                    corr[1] = __fmaf_rn(sz * sw4.y, (float)ws4.y - nc * (float)zw4.y, corr[1]);
                    corr[2] = __fmaf_rn(sz * sw4.z, (float)ws4.z - nc * (float)zw4.z, corr[2]);
                    corr[3] = __fmaf_rn(sz * sw4.w, (float)ws4.w - nc * (float)zw4.w, corr[3]);
                };
                for (int sgi = 0; sgi < p.n_seg; ++sgi, ++n_seg_done) {
                    const int64_t i = (int64_t)s_seg_cl[sgi] * p.ld_w + n;
                    float4 sw4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    int4 zw4 = make_int4(8, 8, 8, 8);
                    if (vec) {
                        sw4 = __ldg(reinterpret_cast<const float4*>(p.sw_c + i));
                        zw4 = __ldg(reinterpret_cast<const int4*>(p.zw_c + i));
                    }
                    const float sc = __ldg(p.seg_scale + sgi) * 0.0625f;
                    const uint32_t sl = n_seg_done % SEG_SLOTS;
                    mbar_wait(bar(B_SEGEMPTY + sl), ((n_seg_done / SEG_SLOTS) & 1) ^ 1, s_abort);
                    float4* d = s_seg_tab + sl * (TILE_N / 2) + 2 * tt;
                    d[0] = make_float4(sc * sw4.x, sc * sw4.y, (float)(128 - 16 * zw4.x), (float)(128 - 16 * zw4.y));
                    d[1] = make_float4(sc * sw4.z, sc * sw4.w, (float)(128 - 16 * zw4.z), (float)(128 - 16 * zw4.w));
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_SEGFULL + sl));
                    add(sgi);
                }
                for (int c = p.n_seg; c < p.g; ++c) add(c);          // (where some clusters are empty)
            } else if constexpr (!DEQ) {
                if (p.corr) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) if (n + e < p.N) corr[e] = p.corr[n + e];
                } else if (vec) {
#pragma unroll 4
                    for (int c = 0; c < p.g; ++c) {
                        const int4 ws = __ldg(reinterpret_cast<const int4*>(p.wsum + (int64_t)c * p.ld_w + n));
                        const float sz = __ldg(p.cl_sz + c);
                        corr[0] = __fmaf_rn(sz, (float)ws.x, corr[0]); corr[1] = __fmaf_rn(sz, (float)ws.y, corr[1]);
                        corr[2] = __fmaf_rn(sz, (float)ws.z, corr[2]); corr[3] = __fmaf_rn(sz, (float)ws.w, corr[3]);
                    }
                } else {
                    for (int c = 0; c < p.g; ++c) {
                        const float sz = __ldg(p.cl_sz + c);
#pragma unroll
                        for (int e = 0; e < 4; ++e) if (n + e < p.N) corr[e] = __fmaf_rn(sz, (float)__ldg(p.wsum + (int64_t)c * p.ld_w + n + e), corr[e]);
                    }
                }
            }
            const uint32_t b = n_tile & 1;
            mbar_wait(bar(B_TABEMPTY + b), ((n_tile >> 1) & 1) ^ 1, s_abort);
            float* tab = s_tab + b * TAB_ROWS * TILE_N + 4 * tt;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool in = n + e < p.N;
                if constexpr (!DEQ) tab[e] = corr[e];
                if constexpr (!ASYM) tab[(TAB_ROWS - 2) * TILE_N + e] = in ? __ldg(p.s_w + n + e) : 0.f;
                tab[(TAB_ROWS - 1) * TILE_N + e] = in && p.bias ? __ldg(p.bias + n + e) : 0.f;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_TAB + b));
        }
      }
    } else if (warp < EPI_WARP0) {
        // ------------------------------------------------------------ unpack warps
        if constexpr (DEQ) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(regs_unpack(MODE)));
        else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(regs_unpack(MODE)));
        const int ut = (tid - UNPACK_WARP0 * 32) & 127;        // within my group
        uint32_t n_done = 0;
        const int total_kb = ((p.n_items - pair_id + n_pairs - 1) / n_pairs) * p.n_kb;
        const int full_kb = p.split ? p.n_full / n_pairs * p.n_kb : total_kb;      // K blocks of whole tiles; those of a strip follow
        // Weight item i of this thread is row (ut >> 2) + 32 i, unit ut & 3, so its two chunk positions in
        // the swizzled row (16-byte chunk j of row r lives at position j ^ (r & 7)) are the same for every i.
        const int row0 = ut >> 2, unit = ut & 3, sw = row0 & 7;
        const uint32_t off0 = row0 * 128 + (((2 * unit) ^ sw) << 4), off1 = row0 * 128 + (((2 * unit + 1) ^ sw) << 4);
        constexpr int W_ITEMS = W_ROWS * 4 / 128;    // weight items per thread
        const uint32_t a_off = ut * 128, a_sw = ut & 7;          // my operand row and its swizzle
        int t_f = pair_id, kb_f = 0, n_fetched = 0;             // next K block to fetch
        const uint8_t* a_src = p.a_codes;
        if constexpr (A8) {
            // The codes are bytes already: a K block of a token row is 128 contiguous bytes. Eight
            // lanes copy the eight 16-byte chunks of one row (one cache line per row, so a warp-wide
            // cp.async touches 4 lines, not 32) straight into that row's swizzled place in the
            // operand stage; a warp covers its 32 rows in eight such instructions, PF K blocks
            // ahead of the weights. The stage is waited for (its previous MMAs have read it) first.
            constexpr int PF = N_U - 2;
            const int wrow = (warp - UNPACK_WARP0) * 32 + (lane >> 3), ch = lane & 7;   // rows wrow + 4 i, chunk ch
            const uint32_t d_even = (uint32_t)wrow * 128 + ((ch ^ (lane >> 3)) << 4);
            const uint32_t d_odd = (uint32_t)wrow * 128 + ((ch ^ ((lane >> 3) + 4)) << 4);
            const int64_t step4 = 4 * p.a_row_bytes;
            int n_rows_ok = 0;                               // how many of my 8 rows exist
            auto a8_tile = [&]() {
                int mt, n0;
                item_of(t_f, mt, n0);
                const int row = mt * (TILE_M * NCTA) + (int)cta_rank * TILE_M + wrow;
                const int left = p.M - row;
                n_rows_ok = left <= 0 ? 0 : (left + 3) >> 2;
                a_src = p.a_codes + (int64_t)(left > 0 ? row : 0) * p.a_row_bytes + 16 * ch;
            };
            a8_tile();
            auto fetch_next = [&]() {
                if (n_fetched < total_kb) {
                    const int s2 = n_fetched % N_U;
                    mbar_wait(bar(B_UEMPTY + s2), ((n_fetched / N_U) & 1) ^ 1, s_abort);
                    tc_fence_after();
                    const uint32_t dst = smem_base + s2 * SL.u_stage;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const bool v = i < n_rows_ok;
                        cp_async16(dst + ((i & 1) ? d_odd : d_even) + i * 512, v ? a_src + i * step4 : p.a_codes, v);
                    }
                    a_src += KBLK;
                    if (++kb_f == p.n_kb) { kb_f = 0; t_f += n_pairs; a8_tile(); }
                }
                ++n_fetched;
                cp_async_commit();                           // one group per K block, empty past the end
            };
#pragma unroll 1
            for (int i = 0; i < PF; ++i) fetch_next();
            for (int it = 0; it < total_kb; ++it, ++n_done) {
                const int sp = n_done % N_P, su = n_done % N_U;
                fetch_next();
                mbar_wait(bar(B_PFULL + sp), (n_done / N_P) & 1, s_abort);
                const uint32_t pw = smem_base + SL.off_p + sp * SL.p_stage;
                const uint32_t w_tile = smem_base + su * SL.u_stage + A8_BYTES;
                uint32_t pw_w[W_ITEMS][4];
#pragma unroll
                for (int i = 0; i < W_ITEMS; ++i) {
                    if (i == W_ITEMS / 2 && it >= full_kb) break;
                    const uint4 v = lds128(pw + (ut + i * 128) * 16);
                    pw_w[i][0] = v.x; pw_w[i][1] = v.y; pw_w[i][2] = v.z; pw_w[i][3] = v.w;
                }
#pragma unroll
                for (int i = 0; i < W_ITEMS; ++i) {
                    if (i == W_ITEMS / 2 && it >= full_kb) break;
                    uint32_t o[8];
                    unpack_w32_x16(pw_w[i], o);
                    sts128(w_tile + off0 + i * 4096, o[0], o[1], o[2], o[3]);
                    sts128(w_tile + off1 + i * 4096, o[4], o[5], o[6], o[7]);
                }
                cp_async_wait<PF>();                         // my copies of K block `it` have landed
                fence_proxy_async();          // make the generic-proxy writes visible to the tensor core
                __syncwarp();                 // ... and every lane's copies and stores of this warp
                if (lane == 0) { arrive_leader(bar(B_UFULL + su)); mbar_arrive(bar(B_PEMPTY + sp)); }
            }
            cp_async_wait<0>();
        } else if constexpr (DEQ) {
            // Two operand stages per K block, 64 positions each; group `grp` fills every other stage. A thread de-quantises units
            // 2 grp and 2 grp + 1 of its token row with their (s_c, z_c), and converts unit 2 grp + (ut & 1) of weight rows
            // (ut >> 1) + 64 i. Positions of every eight are stored in the order 0 2, 1 3, 4 6, 5 7 in both operands: the order in
            // which nibbles come out of a word in pairs (weights: three instructions for two codes).
            // One group of four warps, fp32 arithmetic for the weights too: 2800 clocks per K block, of which the products need 1070
            // (2048 x 4096 x 16384, 4 bits, LayerNorm included: 380 us). Two groups 306; all loads of a block before its first
            // store 287. Half of what is left is still the conversion (tensor pipe 55 % busy, ALU pipe 50 %).
            const int grp = warp >= UNPACK_WARP0 + GROUP_WARPS ? 1 : 0;
            constexpr int CH = BITS == 8 ? 4 : 2;            // 16-byte pieces of a row's K block that hold the two units
            constexpr int N_A = n_a_stages(NCTA, BITS, MODE), PITCH = a_slot_pitch(BITS, MODE);
            static_assert(PITCH == 16 * CH + 16, "slot");
            const uint32_t a_ring0 = smem_base + SL.off_a + grp * TILE_M * PITCH, a_ring = a_ring0 + ut * PITCH;
            uint32_t d_off[CH], s_off[CH];
            int r_of[CH];
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                const int c = 32 * i + lane;
                r_of[i] = (ut & ~31) + c / CH;
                d_off[i] = (uint32_t)r_of[i] * PITCH + 16u * (uint32_t)(c % CH);
                s_off[i] = (uint32_t)r_of[i] * (uint32_t)p.a_row_bytes + (uint32_t)((8 * BITS * grp) & ~15) + 16u * (uint32_t)(c % CH);
            }
            int rows_left = 0;
            auto fetch_tile_row = [&]() {
                int mt, n0;
                item_of(t_f, mt, n0);
                const int row0 = mt * (TILE_M * NCTA) + (int)cta_rank * TILE_M;
                rows_left = p.M - row0;
                a_src = p.a_codes + (int64_t)(rows_left > 0 ? row0 : 0) * p.a_row_bytes;
            };
            fetch_tile_row();
            auto fetch_next = [&]() {
                if (n_fetched < total_kb) {
                    const uint32_t dst = a_ring0 + (n_fetched % N_A) * SL.a_stage;
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        const bool v = r_of[i] < rows_left;
                        cp_async16(dst + d_off[i], v ? a_src + s_off[i] : p.a_codes, v);
                    }
                    a_src += 16 * BITS;
                    if (++kb_f == p.n_kb) { kb_f = 0; t_f += n_pairs; fetch_tile_row(); }
                }
                ++n_fetched;
                cp_async_commit();
            };
#pragma unroll 1
            for (int i = 0; i < N_A - 1; ++i) fetch_next();
            int kb_next = 0;
            const float2* unit_sz = p.unit_sz + 2 * grp;
            float2 sz_next[2] = {__ldg(unit_sz), __ldg(unit_sz + 1)};
            for (int it = 0; it < total_kb; ++it, ++n_done) {
                const int sp = n_done % N_P;
                const float2 sz[2] = {sz_next[0], sz_next[1]};
                kb_next = kb_next + 1 == p.n_kb ? 0 : kb_next + 1;
                sz_next[0] = __ldg(unit_sz + 4 * kb_next); sz_next[1] = __ldg(unit_sz + 4 * kb_next + 1);
                fetch_next();
                cp_async_wait<N_A - 1>();
                __syncwarp();
                uint32_t pa_w[2][BITS];
                {
                    uint32_t raw[4 * CH];
                    const uint32_t slot = a_ring + (it % N_A) * SL.a_stage;
#pragma unroll
                    for (int j = 0; j < CH; ++j) {
                        const uint4 v = lds128(slot + 16 * j);
                        raw[4 * j] = v.x; raw[4 * j + 1] = v.y; raw[4 * j + 2] = v.z; raw[4 * j + 3] = v.w;
                    }
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int j = 0; j < BITS; ++j) pa_w[u][j] = BITS == 3 && grp ? raw[2 + 3 * u + j] : raw[BITS * u + j];
                }
                const uint32_t n_step = 2u * n_done + (uint32_t)grp;
                const int st = n_step % N_U;
                mbar_wait(bar(B_PFULL + sp), (n_done / N_P) & 1, s_abort);
                // (all loads before the first store: they are not reordered)
                const uint32_t pw = smem_base + SL.off_p + sp * SL.p_stage, a_tile = smem_base + st * SL.u_stage, w_tile = a_tile + A8_BYTES;
                uint32_t pk[W_ROWS / 64][4];
#pragma unroll
                for (int i = 0; i < W_ROWS / 64; ++i) {
                    const uint4 v = lds128(pw + ((ut >> 1) + 64 * i) * 64 + (2 * grp + (ut & 1)) * 16);
                    pk[i][0] = v.x; pk[i][1] = v.y; pk[i][2] = v.z; pk[i][3] = v.w;
                }
                mbar_wait(bar(B_UEMPTY + st), ((n_step / N_U) & 1) ^ 1, s_abort);
                tc_fence_after();
#pragma unroll
                for (int uu = 0; uu < 2; ++uu) {
                    const float c1 = -(8388608.0f + sz[uu].y);
                    const float2 neg_c1 = make_float2(c1, c1), s2 = make_float2(sz[uu].x, sz[uu].x);
                    uint32_t o[8];
                    unpack_act32<BITS>(pa_w[uu], o);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t b0, b1, b2, b3;
                        bytes_to_bf16(o[2 * c], neg_c1, s2, b0, b1);
                        bytes_to_bf16(o[2 * c + 1], neg_c1, s2, b2, b3);
                        sts128(a_tile + a_off + (((4 * uu + c) ^ a_sw) << 4), b0, b1, b2, b3);
                    }
                }
#pragma unroll
                for (int i = 0; i < W_ROWS / 64; ++i) {
                    const int r = (ut >> 1) + 64 * i;
                    if (it >= full_kb && r >= (W_ROWS >> p.split)) break;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        sts128(w_tile + r * 128 + (((4 * (ut & 1) + c) ^ (r & 7)) << 4), nibbles_to_bf16(pk[i][c]), nibbles_to_bf16(pk[i][c] >> 8),
                               nibbles_to_bf16(pk[i][c] >> 4), nibbles_to_bf16(pk[i][c] >> 12));
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) { arrive_leader(bar(B_UFULL + st)); mbar_arrive(bar(B_PEMPTY + sp)); }
            }
            cp_async_wait<0>();
        } else {
        // Activation codes: this thread owns token row `ut` of the tile and unpacks it. A K block of a
        // row is 16 BITS contiguous bytes; the rows' K blocks are fetched N_A - 1 K blocks ahead with
        // 16-byte cp.async into one shared-memory slot per row. The 32 BITS chunks of a warp's 32 rows
        // are spread over the lanes in memory order (lane l of copy i takes chunk 32 i + l: row
        // (32 i + l) / BITS of the warp, part (32 i + l) % BITS), so that one warp-wide copy touches
        // 32 / BITS rows, not 32: the load path looks up one cache line per row touched, and with one
        // row per lane those look-ups, not the bytes, set the pace. A row's chunks are copied by
        // lanes of the row owner's own warp, so a __syncwarp after the wait is all the hand-over needs.
        constexpr int N_A = n_a_stages(NCTA, BITS, MODE), PITCH = a_slot_pitch(BITS, MODE);
        const uint32_t a_ring0 = smem_base + SL.off_a;
        const uint32_t a_ring = a_ring0 + ut * PITCH;
        auto slot_sw = [](int r) { return BITS == 4 ? (r >> 1) & 3 : 0; };      // (four pieces a row: exchanged in place of a pad)
        uint32_t d_off[BITS], s_off[BITS];               // where my chunks go in a ring stage / come from in the tile's rows
        int r_of[BITS];                                  // their rows within the tile
#pragma unroll
        for (int i = 0; i < BITS; ++i) {
            const int c = 32 * i + lane;
            r_of[i] = (ut & ~31) + c / BITS;
            d_off[i] = (uint32_t)r_of[i] * PITCH + 16u * (uint32_t)((c % BITS) ^ slot_sw(r_of[i]));
            s_off[i] = (uint32_t)r_of[i] * (uint32_t)p.a_row_bytes + 16u * (uint32_t)(c % BITS);
        }
        int rows_left = 0;                               // rows of the tile being fetched that exist
        auto fetch_tile_row = [&]() {
            int mt, n0;
            item_of(t_f, mt, n0);
            const int row0 = mt * (TILE_M * NCTA) + (int)cta_rank * TILE_M;
            rows_left = p.M - row0;
            a_src = p.a_codes + (int64_t)(rows_left > 0 ? row0 : 0) * p.a_row_bytes;
        };
        fetch_tile_row();
        auto fetch_next = [&]() {
            if (n_fetched < total_kb) {
                const uint32_t dst = a_ring0 + (n_fetched % N_A) * SL.a_stage;
#pragma unroll
                for (int i = 0; i < BITS; ++i) {
                    const bool v = r_of[i] < rows_left;
                    cp_async16(dst + d_off[i], v ? a_src + s_off[i] : p.a_codes, v);
                }
                a_src += 16 * BITS;
                if (++kb_f == p.n_kb) { kb_f = 0; t_f += n_pairs; fetch_tile_row(); }
            }
            ++n_fetched;
            cp_async_commit();                           // one group per K block, empty past the end
        };
#pragma unroll 1
        for (int i = 0; i < N_A - 1; ++i) fetch_next();
        for (int it = 0; it < total_kb; ++it, ++n_done) {
            const int sp = n_done % N_P, su = n_done % N_U;
            fetch_next();
            cp_async_wait<N_A - 1>();                    // my copies of K block `it` have landed
            __syncwarp();                                // ... and those of the lanes that copied my row
            uint32_t pa_w[4][BITS];                      // [unit][word]: unit u of the row is words BITS u ..
            {
                const uint32_t slot = a_ring + (it % N_A) * SL.a_stage;
                uint32_t raw[4 * BITS];
#pragma unroll
                for (int j = 0; j < BITS; ++j) {
                    const uint4 v = lds128(slot + 16 * (j ^ slot_sw(ut)));
                    raw[4 * j] = v.x; raw[4 * j + 1] = v.y; raw[4 * j + 2] = v.z; raw[4 * j + 3] = v.w;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int j = 0; j < BITS; ++j) pa_w[u][j] = raw[BITS * u + j];
            }
            mbar_wait(bar(B_PFULL + sp), (n_done / N_P) & 1, s_abort);
            mbar_wait(bar(B_UEMPTY + su), ((n_done / N_U) & 1) ^ 1, s_abort);
            tc_fence_after();
            const uint32_t pw = smem_base + SL.off_p + sp * SL.p_stage;
            const uint32_t a_tile = smem_base + su * SL.u_stage, w_tile = a_tile + A8_BYTES;
            // n_w: my weight items. Of a strip half of them (its rows, or as many more that no product reads). In code of its own for
            // each: a test inside costs the whole tiles 2 to 5 %.
            auto convert = [&](auto n_w) {
                constexpr int NW = decltype(n_w)::value;
                // all packed weight words of my items first (independent loads), then unpack and store
                uint32_t pw_w[NW][4];
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    const uint4 v = lds128(pw + (ut + i * 128) * 16);
                    pw_w[i][0] = v.x; pw_w[i][1] = v.y; pw_w[i][2] = v.z; pw_w[i][3] = v.w;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    uint32_t o[8];
                    unpack_act32<BITS>(pa_w[u], o);
                    sts128(a_tile + a_off + (((2 * u) ^ a_sw) << 4), o[0], o[1], o[2], o[3]);
                    sts128(a_tile + a_off + (((2 * u + 1) ^ a_sw) << 4), o[4], o[5], o[6], o[7]);
                }
#pragma unroll
                for (int i = 0; i < NW; ++i) {
                    uint32_t o[8];
                    unpack_w32_x16(pw_w[i], o);
                    sts128(w_tile + off0 + i * 4096, o[0], o[1], o[2], o[3]);
                    sts128(w_tile + off1 + i * 4096, o[4], o[5], o[6], o[7]);
                }
            };
            if (it < full_kb) convert(std::integral_constant<int, W_ITEMS>()); else convert(std::integral_constant<int, W_ITEMS / 2>());
            fence_proxy_async();          // make the generic-proxy stores visible to the tensor core
            __syncwarp();
            if (lane == 0) { arrive_leader(bar(B_UFULL + su)); mbar_arrive(bar(B_PEMPTY + sp)); }
        }
        cp_async_wait<0>();
        }
    } else {
        // ------------------------------------------------------------ epilogue warps
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(regs_epi(MODE)));
        const int ew = warp - EPI_WARP0;
        const int q = ew & 3, h = ew >> 2;           // TMEM lane quarter (= warp % 4), column half
        uint32_t n_tile_done = 0;
        uint32_t par = 0;                    // bit b: parity of how many clusters of accumulator b I have drained
        uint32_t n_seg_done = 0;                     // ASYM: clusters drained so far, over all tiles
        // Running sums. ROWS: columns 2 i, 2 i + 1 of the thread's row in R[i]. Otherwise the layout of the 16-lane tensor-memory loads: my
        // rows of the warp's 32 are 16 h + lane / 4 + 8 r, my columns 8 i + 2 (lane % 4) + {0, 1}, R[(i / 4 * 2 + h) * 8 + i % 4 * 2 + r].
        // With a thread per row, what belongs to a column is read by every thread, and a warp-wide load of 16 bytes takes four clocks of
        // the SM's shared-memory port even where all lanes read the same: 64 a drain of clustered weights (2048 of its 2125 clocks), 96 a tile
        // for the tables of the outputs; in the other layout a load serves four rows. But its tensor-memory loads take longer (some 66 clocks a
        // drain more), and a word of codes lies in four lanes. Which of the two is the faster depends on the number of clusters: see launch_gemm.
        float2 R[64];
        for (int t = pair_id; t < p.n_items; t += n_pairs, ++n_tile_done) {
            int mt, n0;
            const int sh = item_of(t, mt, n0), half_cols = 128 >> sh;      // columns of my half
            const int m0 = mt * (TILE_M * NCTA) + (int)cta_rank * TILE_M;
            float* tab = s_tab + (n_tile_done & 1) * TAB_ROWS * TILE_N;
            // a warp whose 32 accumulator lanes all lie beyond the last token row keeps the barriers'
            // protocol but reads and accumulates nothing (few-token calls: most of the tile is empty)
            const bool live = m0 + 32 * q < p.M;
#pragma unroll
            for (int i = 0; i < 64; ++i) R[i] = make_float2(0.f, 0.f);
            // outputs as codes: lane l holds the output layout's unit l of my columns, asked for before the sums (700 x 768 x 3072, 8
            // clusters: 14.4 -> 13.6 us); LATE: after them, since four registers more cost the drains of float outputs 1 %
            uint4 unit4 = make_uint4(0u, 0u, 0u, 0u);
            auto ask_units = [&]() {
                const int unit = (n0 + h * half_cols) / 32 + (lane & 3);
                if (p.y_dtype == RPTQ_OUT_CODES && 32 * unit < p.N) unit4 = __ldg(reinterpret_cast<const uint4*>(p.out_unit + unit));
            };
            constexpr bool LATE = MODE == MODE_INT && NCTA == 2 && !ROWS;
            if constexpr (!DEQ && !LATE) ask_units();
            // ASYM: my tokens' code sums of the cluster to come (rows past the last token read the last one's)
            const int32_t* xs_row[4] = {nullptr, nullptr, nullptr, nullptr};
            int xs_next[4] = {0, 0, 0, 0};
            if constexpr (ASYM) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    xs_row[i] = p.xsum + (int64_t)min(m0 + 32 * q + (lane >> 2) + 8 * i, p.M - 1) * p.g;
                    xs_next[i] = xs_row[i][s_seg_cl[0]];
                }
            }
            for (int sgi = 0; sgi < (DEQ ? 1 : p.n_seg); ++sgi) {
                const uint32_t buf = DEQ ? (n_tile_done & 1u) : (uint32_t)s_seg_buf[sgi];
                mbar_wait(bar(B_ACCFULL + buf), (par >> buf) & 1u, s_abort);
                par ^= 1u << buf;
                tc_fence_after();
                const float sc = ASYM ? 0.f : s_seg_scale[sgi];
                const float2 sc2 = make_float2(sc, sc);
                const uint32_t seg_slot = n_seg_done % SEG_SLOTS;
                const float4* seg_tab = s_seg_tab + seg_slot * (TILE_N / 2) + (h * half_cols >> 1) + (lane & 3);
                float xs[4] = {0.f, 0.f, 0.f, 0.f};
                if constexpr (ASYM) {
                    mbar_wait(bar(B_SEGFULL + seg_slot), (n_seg_done / SEG_SLOTS) & 1, s_abort);
                    ++n_seg_done;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        xs[i] = (float)xs_next[i];
                        if (sgi + 1 < p.n_seg) xs_next[i] = xs_row[i][s_seg_cl[sgi + 1]];
                    }
                }
                const uint32_t taddr = tmem_base + ((uint32_t)(32 * q) << 16) + buf * TILE_N + h * half_cols;
                if (live && !DEQ) {
                // R += s_c * acc, two columns per packed fused multiply-add: 32 columns of 16 rows (half hh of the warp's; ROWS: 16 columns). Both halves are asked
                // for at once and, with clustered weights, their coefficients before the wait for them: a wait in the middle has the next
                // load's latency behind it (1024 x 4096 x 16384, 16 clusters: 125 -> 112 us).
                auto accumulate = [&](const uint32_t (&v)[16], const float4 (&k)[4], int jc, int hh) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float2* r = R + (jc * 2 + hh) * 8 + 2 * j;
                        const float2 a0 = make_float2((float)(int)v[4 * j], (float)(int)v[4 * j + 1]), a1 = make_float2((float)(int)v[4 * j + 2], (float)(int)v[4 * j + 3]);
                        if constexpr (ASYM) {
                            // R += s^X_c s^W_c[n] / 16 (acc' - 16 (z^W_c[n] - 8) xsum)
                            const float2 kz = make_float2(k[j].z, k[j].w), ks = make_float2(k[j].x, k[j].y);
                            r[0] = fma2(ks, fma2(kz, make_float2(xs[2 * hh], xs[2 * hh]), a0), r[0]);
                            r[1] = fma2(ks, fma2(kz, make_float2(xs[2 * hh + 1], xs[2 * hh + 1]), a1), r[1]);
                        } else {
                            r[0] = fma2(sc2, a0, r[0]);
                            r[1] = fma2(sc2, a1, r[1]);
                        }
                    }
                };
#pragma unroll
                for (int jc = 0; jc < 4; ++jc) {
                    uint32_t va[16], vb[16];
                    float4 k[4];
                    if constexpr (ROWS) {
                        tc_ld16(taddr + 32 * jc, va);
                        tc_ld16(taddr + 32 * jc + 16, vb);
                    } else {
                        tc_ld16xn(taddr + 32 * jc, va);
                        tc_ld16xn(taddr + (16u << 16) + 32 * jc, vb);
                    }
                    if constexpr (ASYM) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) k[j] = seg_tab[(jc * 4 + j) * 4];
                    }
                    tc_wait_ld();
                    const bool more = jc < 3 && 32 * (jc + 1) < half_cols;
                    if (!more) {
                        // all of it has been read: the accumulator goes back before the last sums are formed
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive_leader(bar(B_ACCEMPTY + buf));
                    }
                    accumulate(va, k, jc, 0);
                    accumulate(vb, k, jc, 1);
                    if (!more) break;
                }
                }
                if constexpr (DEQ) break;                    // (the sums are read as the outputs are formed)
                if (ASYM || !live) {
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (ASYM) mbar_arrive(bar(B_SEGEMPTY + seg_slot));
                        if (!live) arrive_leader(bar(B_ACCEMPTY + buf));
                    }
                }
            }
            if constexpr (LATE) ask_units();
            mbar_wait(bar(B_TAB + (n_tile_done & 1)), (n_tile_done >> 1) & 1, s_abort);
            // y = s_w * (R - corr) + bias, activation, store. Rows leave through a buffer of the warp, in pieces of 64 bytes a row: whole memory
            // sectors, and few hand-overs between lanes (1999 x 2048 x 6144, 8 bits, fp32 out, with the LayerNorm: stores of a lane's own 16 bytes
            // 70 us, pieces of 32 bytes 55; 50.5 with these and with sums that are not held by rows)
            if (live) {
                const int mw = m0 + 32 * q, nb = n0 + h * half_cols;           // my warp's first row, my first column
                const bool relu = p.act == RPTQ_ACT_RELU;
                // piece j (16 bytes) of row r lies at j ^ sw(r): neither what a warp puts nor what it reads in one instruction meets in a bank
                constexpr int PIECES = OUT_ROW / 16, ROWS_I = 32 / PIECES;     // ROWS_I: rows that a warp-wide access covers
                const uint32_t stage = smem_base + SL.off_stage + ew * 32 * OUT_ROW;
                auto sw_f16 = [](int r) { return (r >> 1) & 3; };              // 16 bytes of eight rows at a time
                auto sw_f32 = [](int r) { return r & 2; };                     // 32 bytes of four rows at a time
                auto store = [&](auto sw, uint8_t* dst, int64_t row_bytes, int n_bytes) {   // dst: the warp's first row; n_bytes valid of OUT_ROW
                    __syncwarp();
                    const int j = lane % PIECES, r0 = lane / PIECES, left = n_bytes - 16 * j, rows = p.M - mw;
                    uint8_t* d = dst + r0 * row_bytes + 16 * j;
                    uint4 v[PIECES];
#pragma unroll
                    for (int i = 0; i < PIECES; ++i) v[i] = lds128(stage + (r0 + ROWS_I * i) * OUT_ROW + ((j ^ sw(r0 + ROWS_I * i)) << 4));
#pragma unroll
                    for (int i = 0; i < PIECES; ++i, d += ROWS_I * row_bytes) {
                        if (r0 + ROWS_I * i >= rows || left <= 0) continue;
                        if (left >= 16) { *reinterpret_cast<uint4*>(d) = v[i]; continue; }
                        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};       // the end of a ragged row
#pragma unroll
                        for (int k = 0; k < 7; ++k) if (2 * k < left) *reinterpret_cast<uint16_t*>(d + 2 * k) = (uint16_t)(w[k >> 1] >> (16 * (k & 1)));
                    }
                    __syncwarp();
                };
                // re-quantised outputs: column n is padded position n of the output layout (N is a multiple of 128)
                const int n_units = min(half_cols, p.N - nb) >> 5;
                uint8_t* const unit0 = static_cast<uint8_t*>(p.y) + (int64_t)mw * p.out_row_bytes + (nb >> 5) * 4 * p.out_bits;
                if constexpr (ROWS) {
                    const float4* t_row = reinterpret_cast<const float4*>(tab + h * half_cols);
                    auto own = [&](int piece) { return stage + lane * OUT_ROW + ((piece ^ sw_f16(lane)) << 4); };
                    auto finish = [&](int i, float2& lo, float2& hi) {         // columns 4 i .. 4 i + 3
                        const float4 c = t_row[i], w = t_row[TILE_N / 4 + i], b = t_row[TILE_N / 2 + i];
                        lo = fma2(make_float2(w.x, w.y), add2(R[2 * i], make_float2(-c.x, -c.y)), make_float2(b.x, b.y));
                        hi = fma2(make_float2(w.z, w.w), add2(R[2 * i + 1], make_float2(-c.z, -c.w)), make_float2(b.z, b.w));
                        if (relu) { lo.x = fmaxf(lo.x, 0.f); lo.y = fmaxf(lo.y, 0.f); hi.x = fmaxf(hi.x, 0.f); hi.y = fmaxf(hi.y, 0.f); }
                    };
                    auto h2 = [](float2 v) { const __half2 x = __floats2half2_rn(v.x, v.y); return *reinterpret_cast<const uint32_t*>(&x); };
                    if (p.y_dtype == RPTQ_OUT_F16) {
                        uint8_t* dst = static_cast<uint8_t*>(p.y) + ((int64_t)mw * p.ldy + nb) * 2;
                        const int n_bytes = 2 * min(p.N - nb, half_cols);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {                          // 32 columns
                            if (32 * u >= half_cols) break;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float2 v[4];
                                finish(8 * u + 2 * j, v[0], v[1]);
                                finish(8 * u + 2 * j + 1, v[2], v[3]);
                                sts128(own(j), h2(v[0]), h2(v[1]), h2(v[2]), h2(v[3]));
                            }
                            store(sw_f16, dst + 64 * u, p.ldy * 2, n_bytes - 64 * u);
                        }
                    } else if (p.y_dtype == RPTQ_OUT_F32) {
                        uint8_t* dst = static_cast<uint8_t*>(p.y) + ((int64_t)mw * p.ldy + nb) * 4;
                        const int n_bytes = 4 * min(p.N - nb, half_cols);
#pragma unroll
                        for (int c = 0; c < 8; ++c) {                          // 16 columns
                            if (16 * c >= half_cols) break;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float2 lo, hi;
                                finish(4 * c + j, lo, hi);
                                sts128(own(j), __float_as_uint(lo.x), __float_as_uint(lo.y), __float_as_uint(hi.x), __float_as_uint(hi.y));
                            }
                            store(sw_f16, dst + 64 * c, p.ldy * 4, n_bytes - 64 * c);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (u >= n_units) break;
                            const float inv_s = __uint_as_float(__shfl_sync(0xffffffffu, unit4.x, u));
                            const int zc = (int)__shfl_sync(0xffffffffu, unit4.y, u), nvalid = (int)__shfl_sync(0xffffffffu, unit4.w, u);
                            const float2 s2 = make_float2(inv_s, inv_s), c2 = make_float2(12582912.0f, 12582912.0f);
                            int qv[32];                                        // not yet clamped, the pack saturates
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float2 lo, hi;
                                finish(8 * u + i, lo, hi);
                                lo = fma2(lo, s2, c2); hi = fma2(hi, s2, c2);
                                qv[4 * i] = quant_int(lo.x, zc); qv[4 * i + 1] = quant_int(lo.y, zc);
                                qv[4 * i + 2] = quant_int(hi.x, zc); qv[4 * i + 3] = quant_int(hi.y, zc);
                            }
                            if (nvalid < 32) {
#pragma unroll
                                for (int e = 0; e < 32; ++e) qv[e] = e < nvalid ? qv[e] : 0;
                            }
                            // rows leave in pieces of up to 64 bytes, 3 bits: 48, those of a strip (which may begin between 16-byte boundaries) unit by unit
                            if (p.out_bits == 4) {
                                uint32_t w[4]; pack32_sat<4>(qv, w);
                                sts128(own(u), w[0], w[1], w[2], w[3]);
                                if (u + 1 == n_units) store(sw_f16, unit0, p.out_row_bytes, 16 * n_units);
                            } else if (p.out_bits == 8) {
                                uint32_t w[8]; pack32_sat<8>(qv, w);
                                sts128(own(2 * (u & 1)), w[0], w[1], w[2], w[3]);
                                sts128(own(2 * (u & 1) + 1), w[4], w[5], w[6], w[7]);
                                if ((u & 1) || u + 1 == n_units) store(sw_f16, unit0 + 32 * (u & 2), p.out_row_bytes, 32 * ((u & 1) + 1));
                            } else {
                                uint32_t w[3]; pack32_sat<3>(qv, w);
                                if (half_cols == 128) {
#pragma unroll
                                    for (int j = 0; j < 3; ++j) sts32(own((3 * u + j) >> 2) + 4 * ((3 * u + j) & 3), w[j]);
                                    if (u == 3) store(sw_f16, unit0, p.out_row_bytes, 48);
                                } else if (mw + lane < p.M) {
#pragma unroll
                                    for (int j = 0; j < 3; ++j) reinterpret_cast<uint32_t*>(unit0 + lane * p.out_row_bytes + 12 * u)[j] = w[j];
                                }
                            }
                        }
                    }
                } else {
                    const float2* t_corr = reinterpret_cast<const float2*>(tab + h * half_cols) + (lane & 3);
                    const float2* t_sw = t_corr + (TAB_ROWS - 2) * (TILE_N / 2);
                    const float2* t_bs = t_corr + (TAB_ROWS - 1) * (TILE_N / 2);
                    // J times 8 columns at a time (DEQ: its sums are not in registers, of which it has few: a rolled loop, and with one block, whose output
                    // phase is short, half as many columns: 100 x 4096 x 12288, 3 and 4 bits, 41.5 and 42.5 us -> 40.4 and 41.4)
                    constexpr int J = DEQ && NCTA == 1 ? 2 : 4;
                    auto each_step = [&](auto body) {
                        if constexpr (DEQ) {
#pragma unroll 1
                            for (int st = 0; 8 * J * st < half_cols; ++st) body(st);
                        } else {
                            body(std::integral_constant<int, 0>());
                            if (half_cols > 32) body(std::integral_constant<int, 1>());
                            if (half_cols > 64) { body(std::integral_constant<int, 2>()); body(std::integral_constant<int, 3>()); }
                        }
                    };
                    // DEQ: the finished fp32 sums are in tensor memory
                    const uint32_t t_acc = tmem_base + ((uint32_t)(32 * q) << 16) + (n_tile_done & 1u) * TILE_N + h * half_cols;
                    // my values of columns 8 (J st + j) + {0, 1}, rows lane / 4 + 8 k
                    auto finish = [&](int st, auto use) {
                        float2 own[4 * J];
                        if constexpr (DEQ) {
                            uint32_t v[2][4 * J];
                            tc_ld16xn(t_acc + 8 * J * st, v[0]);
                            tc_ld16xn(t_acc + (16u << 16) + 8 * J * st, v[1]);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 4 * J; ++i) own[i] = make_float2(__uint_as_float(v[i / (2 * J)][2 * (i % (2 * J))]), __uint_as_float(v[i / (2 * J)][2 * (i % (2 * J)) + 1]));
                        }
#pragma unroll
                        for (int j = 0; j < J; ++j) {
                            const int at = (J * st + j) * 4;
                            float2 c, w;
                            if constexpr (!DEQ) c = t_corr[at];
                            if constexpr (!ASYM) w = t_sw[at];
                            const float2 b = t_bs[at];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                float2 v;
                                if constexpr (DEQ) v = own[(k >> 1) * 2 * J + 2 * j + (k & 1)]; else v = add2(R[(st * 2 + (k >> 1)) * 8 + 2 * j + (k & 1)], make_float2(-c.x, -c.y));
                                if constexpr (ASYM) v = add2(v, b); else v = fma2(w, v, b);
                                if (relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); }
                                use(j, k, v);
                            }
                        }
                    };
                    if (p.y_dtype == RPTQ_OUT_F16) {
                        uint8_t* dst = static_cast<uint8_t*>(p.y) + ((int64_t)mw * p.ldy + nb) * 2;
                        const int n_bytes = 2 * min(p.N - nb, half_cols);
                        // (my lane names row 8 k + lane % 8, piece lane / 8 of the step's columns, to stmatrix)
                        each_step([&](auto at_st) {
                            const int st = at_st, j0 = J * st % 4;
                            uint32_t f[4][J];                                      // [k][j]
                            finish(st, [&](int j, int k, float2 v) { const __half2 x = __floats2half2_rn(v.x, v.y); f[k][j] = *reinterpret_cast<const uint32_t*>(&x); });
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int r = 8 * k + (lane & 7);
                                stmatrixn(stage + r * OUT_ROW + (((j0 + (lane >> 3) % J) ^ sw_f16(r)) << 4), f[k]);
                            }
                            const int from = 16 * (J * st - j0);
                            if (j0 + J == 4) store(sw_f16, dst + from, p.ldy * 2, n_bytes - from);
                        });
                    } else if (p.y_dtype == RPTQ_OUT_F32) {
                        uint8_t* dst = static_cast<uint8_t*>(p.y) + ((int64_t)mw * p.ldy + nb) * 4;
                        const int n_bytes = 4 * min(p.N - nb, half_cols);
                        const uint32_t put = stage + (lane >> 2) * OUT_ROW + 8 * (lane & 1);
                        const int piece = (lane & 3) >> 1;
                        each_step([&](auto at_st) {
                            const int st = at_st;
                            finish(st, [&](int j, int k, float2 v) {
                                sts64(put + 8 * k * OUT_ROW + (((2 * (j & 1) + piece) ^ sw_f32(lane >> 2)) << 4), v);      // (8 k changes no swizzle)
                                if (k == 3 && (j & 1)) {
                                    const int from = 32 * (J * st + j - 1);
                                    store(sw_f32, dst + from, p.ldy * 4, n_bytes - from);
                                }
                            });
                        });
                    } else if constexpr (!DEQ) {
                        // A word of eight nibbles is eight columns of a row, which four lanes hold, two codes each. Codes of at most four bits: a byte for
                        // each of a unit's four words goes through the warp's buffer as the fragment of a 16-bit matrix, which gives every lane the
                        // 16 bytes of its own row.
                        const int l = lane & 3;
#pragma unroll
                        for (int jc = 0; jc < 4; ++jc) {
                            if (jc >= n_units) break;
                            const float inv_s = __uint_as_float(__shfl_sync(0xffffffffu, unit4.x, jc));
                            const int zc = (int)__shfl_sync(0xffffffffu, unit4.y, jc), nvalid = (int)__shfl_sync(0xffffffffu, unit4.w, jc);
                            const float2 s2 = make_float2(inv_s, inv_s), c2 = make_float2(12582912.0f, 12582912.0f);
                            int qv[4][4][2];                                       // [row k][word j]: not yet clamped, the pack saturates
                            finish(jc, [&](int j, int k, float2 v) {
                                v = fma2(v, s2, c2);
                                qv[k][j][0] = quant_int(v.x, zc); qv[k][j][1] = quant_int(v.y, zc);
                            });
                            if (nvalid < 32) {
#pragma unroll
                                for (int j = 0; j < 4; ++j)
#pragma unroll
                                    for (int e = 0; e < 2; ++e)
#pragma unroll
                                        for (int k = 0; k < 4; ++k) qv[k][j][e] = 8 * j + 2 * l + e < nvalid ? qv[k][j][e] : 0;
                            }
                            if (p.out_bits == 8) {
                                uint8_t* row = unit0 + (lane >> 2) * p.out_row_bytes + jc * 32 + 8 * l;
#pragma unroll
                                for (int k = 0; k < 4; ++k, row += 8 * p.out_row_bytes) {
                                    // two codes of each of the unit's four pairs of words: lane l ends with pair l. With lane ^ 2 pairs 0, 1 (of lanes 0, 1) for 2, 3
                                    // (of lanes 2, 3), then with lane ^ 1 the even pair for the odd one
                                    auto two = [&](int j) { return sat_pack_u8(qv[k][j][1], qv[k][j][0], 0u); };
                                    const uint32_t lo = two(0) | (two(1) << 16), hi = two(2) | (two(3) << 16);
                                    const uint32_t own = l & 2 ? hi : lo, o2 = __shfl_xor_sync(0xffffffffu, l & 2 ? lo : hi, 2);
                                    const uint32_t x = l & 2 ? o2 : own, y = l & 2 ? own : o2;           // of lanes l & 1 and (l & 1) + 2
                                    const uint32_t even = __byte_perm(x, y, 0x5410), odd = __byte_perm(x, y, 0x7632);
                                    const uint32_t o1 = __shfl_xor_sync(0xffffffffu, l & 1 ? even : odd, 1);
                                    const uint32_t a = l & 1 ? o1 : even, c = l & 1 ? odd : o1;          // of the lower, the higher lane
                                    if (mw + (lane >> 2) + 8 * k < p.M)
                                        *reinterpret_cast<uint2*>(row) = make_uint2(__byte_perm(a, c, 0x5410), __byte_perm(a, c, 0x7632));
                                }
                                continue;
                            }
                            uint32_t x[4] = {0u, 0u, 0u, 0u};                      // byte j: codes 2 l (low nibble) and 2 l + 1 of word j
#pragma unroll
                            for (int k = 0; k < 4; ++k)
#pragma unroll
                                for (int j = 3; j >= 0; --j) x[k] = sat_pack_u4(qv[k][j][1], qv[k][j][0], x[k]);
                            const uint32_t own_row = stage + lane * OUT_ROW + ((jc ^ sw_f16(lane)) << 4);
                            stmatrixn(own_row, x);
                            __syncwarp();
                            const uint4 t = lds128(own_row);                       // word l: byte j is codes 2 l, 2 l + 1 of word j
                            const uint32_t a01 = __byte_perm(t.x, t.y, 0x5140), a23 = __byte_perm(t.x, t.y, 0x7362);
                            const uint32_t b01 = __byte_perm(t.z, t.w, 0x5140), b23 = __byte_perm(t.z, t.w, 0x7362);
                            uint32_t w[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                // codes 0, 1, 2, 3 of word j (bytes 0, 0, 1, 1 of its two) and 4, 5, 6, 7: low nibbles, high nibbles
                                const uint32_t lo = __byte_perm(j < 2 ? a01 : a23, 0u, j & 1 ? 0x3322 : 0x1100), hi = __byte_perm(j < 2 ? b01 : b23, 0u, j & 1 ? 0x3322 : 0x1100);
                                w[j] = (lo & 0x000F000Fu) | ((lo >> 4) & 0x0F000F00u) | ((hi << 4) & 0x00F000F0u) | (hi & 0xF000F000u);
                            }
                            uint8_t* row = unit0 + lane * p.out_row_bytes + jc * 4 * p.out_bits;
                            if (p.out_bits == 4) {
                                // back to the same place, and out in pieces of up to 64 bytes a row
                                sts128(own_row, w[0], w[1], w[2], w[3]);
                                if (jc + 1 == n_units)
                                    store(sw_f16, unit0, p.out_row_bytes, 16 * n_units);
                            } else {
                                auto clamp7 = [](uint32_t v) { return (v | (((v >> 3) & 0x11111111u) * 7u)) & 0x77777777u; };        // nibbles above 7 become 7
                                const uint32_t tail = clamp7(w[3]);
                                if (mw + lane < p.M) {
#pragma unroll
                                    for (int j = 0; j < 3; ++j) reinterpret_cast<uint32_t*>(row)[j] = clamp7(w[j]) | (((tail >> j) & 0x11111111u) << 3);
                                }
                            }
                        }
                    }
                }
            }
            if constexpr (DEQ) tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(B_TABEMPTY + (n_tile_done & 1)));
                if constexpr (DEQ) arrive_leader(bar(B_ACCEMPTY + (n_tile_done & 1)));
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if constexpr (NCTA == 2) cluster_sync_all();       // the peer no longer arrives here nor reads this CTA's memory
    tc_fence_after();
    if (warp == 1) {
        if constexpr (NCTA == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    if (tid == 0 && *s_abort && p.status) atomicExch(p.status, RPTQ_ERR_DEVICE_TIMEOUT);
}

// ---------------------------------------------------------------- host side
template <int BITS, int NCTA, bool A8, int MODE, bool ROWS = false>
static int launch(const Params& p, int dev, int n_sm, cudaStream_t st)
{
    constexpr SmemLayout SL = smem_layout(NCTA, BITS, A8, MODE);
    constexpr int THREADS = threads_of(MODE);
    const int smem = SL.total + 1024;     // slack for the in-kernel 1024-byte alignment
    const void* fn = reinterpret_cast<const void*>(cluster_gemm_kernel<BITS, NCTA, A8, MODE, ROWS>);
    static_assert(SL.total + 1024 <= 227 * 1024, "shared memory");
    static SmemAllowed done;
    static std::atomic<uint64_t> pool_ok{0};
    if (!(pool_ok.load(std::memory_order_acquire) >> (dev & 63) & 1u)) {
        cudaFuncAttributes attr;
        if (cudaFuncGetAttributes(&attr, fn) != cudaSuccess) return RPTQ_ERR_CUDA;
        // the register re-partition inside the kernel (setmaxnreg) assumes this pool; refuse to launch otherwise
        if (attr.numRegs * THREADS < regs_all(MODE)) return RPTQ_ERR_UNSUPPORTED;
        if (dev >= 0 && dev < 64) pool_ok.fetch_or(uint64_t(1) << dev, std::memory_order_release);
    }
    if (allow_smem(fn, dev, smem, done) != RPTQ_OK) return RPTQ_ERR_CUDA;
    const int slots = n_sm / NCTA;
    const int groups = p.n_items < slots ? p.n_items : slots;
    return launch_kernel(cluster_gemm_kernel<BITS, NCTA, A8, MODE, ROWS>, dim3((unsigned)(groups * NCTA)), THREADS, (size_t)smem, NCTA, st, p);
}

}  // namespace gemm
}  // namespace rptq

using namespace rptq;

// Argument checks shared by the entry points. Returns RPTQ_OK when a launch should follow.
static int check_gemm_args(const rptq_layout_t* Lin, const void* a_codes, int M, const void* w_codes,
                           const float* s_w, const int32_t* wsum, int64_t ld_w, const void* bias, int N,
                           int act, const rptq_layout_t* Lout, void* y, int y_dtype, int64_t ldy, int* dev_out)
{
    if (!Lin || !a_codes || !w_codes || !s_w || !wsum || !y) return RPTQ_ERR_INVALID_ARG;
    if (M < 0 || N <= 0 || ld_w < N) return RPTQ_ERR_INVALID_ARG;
    if (act != RPTQ_ACT_NONE && act != RPTQ_ACT_RELU) return RPTQ_ERR_INVALID_ARG;
    if (!aligned16(a_codes) || !aligned16(w_codes) || !aligned16(y) || !aligned16(s_w) || !aligned16(wsum) || !aligned16(bias))
        return RPTQ_ERR_INVALID_ARG;
    if (y_dtype == RPTQ_OUT_F32) {
        if (Lout || ldy < N || (ldy * 4) % 16) return RPTQ_ERR_INVALID_ARG;
    } else if (y_dtype == RPTQ_OUT_F16) {
        if (Lout || ldy < N || (ldy * 2) % 16) return RPTQ_ERR_INVALID_ARG;
    } else if (y_dtype == RPTQ_OUT_CODES) {
        if (!Lout || Lout->K_pad != N) return RPTQ_ERR_INVALID_ARG;
    } else {
        return RPTQ_ERR_INVALID_ARG;
    }
    if (Lin->g > kMaxGemmSegments || Lin->n_units > 2048) return RPTQ_ERR_UNSUPPORTED;
    int dev = -1;
    if (Lin->device < 0 || cudaGetDevice(&dev) != cudaSuccess) return RPTQ_ERR_CUDA;
    if (dev != Lin->device || (Lout && Lout->device != dev)) return RPTQ_ERR_INVALID_ARG;
    *dev_out = dev;
    return RPTQ_OK;
}

// Fills the launch parameters and launches the variant that fits M. `status` and `corr` may be NULL.
static int launch_gemm(const rptq_layout_t* Lin, const void* a_codes, int M, const void* w_codes,
                       const float* s_w, const int32_t* wsum, int64_t ld_w, const void* bias, int N,
                       int act, const rptq_layout_t* Lout, void* y, int y_dtype, int64_t ldy, void* stream,
                       int dev, int* status, const float* corr,
                       const float* sw_c = nullptr, const int32_t* zw_c = nullptr, const int32_t* xsum = nullptr, bool deq = false)
{
    gemm::Params p{};
    p.M = M; p.N = N; p.n_kb = Lin->K_pad / gemm::KBLK; p.n_seg = Lin->n_seg; p.g = Lin->g;
    // CTA pairs share a 256-row tile; one token tile or less gains nothing from pairing
    const int ncta = M > gemm::TILE_M ? 2 : 1;
    p.tiles_m = (M + gemm::TILE_M * ncta - 1) / (gemm::TILE_M * ncta);
    const int n_tiles = p.tiles_m * ((N + gemm::TILE_N - 1) / gemm::TILE_N);
    p.a_codes = static_cast<const uint8_t*>(a_codes); p.a_row_bytes = Lin->row_bytes;
    p.w_codes = static_cast<const uint8_t*>(w_codes); p.n_wtiles = (int)((ld_w + 127) / 128);
    p.step_flags = Lin->d_step_flags; p.seg_scale = Lin->d_seg_scale; p.seg_buf = Lin->d_seg_buf; p.cl_sz = Lin->d_cl_sz;
    p.s_w = s_w; p.wsum = wsum; p.ld_w = ld_w; p.bias = static_cast<const float*>(bias);
    p.act = act; p.y_dtype = y_dtype; p.y = y; p.ldy = ldy;
    p.out_unit = Lout ? Lout->d_unit : nullptr;
    p.out_bits = Lout ? Lout->bits : 0;
    p.out_row_bytes = Lout ? Lout->row_bytes : 0;
    p.status = status;
    p.corr = corr;
    p.sw_c = sw_c; p.zw_c = zw_c; p.xsum = xsum; p.seg_cluster = Lin->d_seg_cluster; p.cl_n = Lin->d_cl_n;

    const int n_sm = sm_count(dev);
    if (n_sm == 0) return RPTQ_ERR_CUDA;
    // The tiles of the last round, when they are at most half (a quarter) as many as there are blocks (pairs) to work on them, are
    // cut into two (four) strips of columns: the round then takes the time of a strip, about two thirds (half) of a tile's (a
    // strip's token codes are unpacked all the same). 200 x 9216 x 27648: 90 -> 86 us; 1024 x 4096 x 16384 with clustered weights
    // 136 -> 130; calls with fewer tiles than blocks up to 1.4 times as fast. With more tiles left than half the blocks a cut
    // would only add a round. (Re-quantised outputs: quarters against halves, 40 x 768 x 3072 8.9 -> 7.8 us, 128 x 2048 x 8192 20.1 -> 17.5.)
    const int slots = n_sm / ncta, rest = n_tiles % slots;
    p.split = rest == 0 ? 0 : 4 * rest <= slots ? 2 : 2 * rest <= slots ? 1 : 0;
    p.n_full = p.split ? n_tiles - rest : n_tiles;
    p.n_items = p.n_full + ((n_tiles - p.n_full) << p.split);
    auto st = static_cast<cudaStream_t>(stream);
    // a few tokens (decoding): the kernel that streams the weights through mma.sync with the channels as its M dimension
    if (!deq && !sw_c && y_dtype != RPTQ_OUT_CODES && smallm::fits(M, Lin->bits, Lin->K_pad)) {
        SmallMParams q{};
        q.a = p.a_codes; q.a_row_bytes = p.a_row_bytes; q.M = M; q.K_pad = Lin->K_pad; q.n_units = Lin->n_units; q.n_kb = p.n_kb;
        q.w = p.w_codes; q.n_wtiles = p.n_wtiles;
        q.step_flags = Lin->d_step_flags; q.unit_sz = Lin->d_unit_sz; q.cl_sz = Lin->d_cl_sz; q.g = Lin->g;
        q.corr = corr; q.s_w = s_w; q.wsum = wsum; q.ld_w = ld_w; q.bias = p.bias;
        q.N = N; q.act = act; q.y_dtype = y_dtype; q.y = y; q.ldy = ldy; q.status = status;
        return smallm::launch(q, Lin->bits, dev, st);
    }
    if (deq) {
        p.unit_sz = Lin->d_unit_sz;
        if (ncta == 2) {
            if (Lin->bits == 3) return gemm::launch<3, 2, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
            if (Lin->bits == 4) return gemm::launch<4, 2, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
            return gemm::launch<8, 2, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
        }
        if (Lin->bits == 3) return gemm::launch<3, 1, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
        if (Lin->bits == 4) return gemm::launch<4, 1, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
        return gemm::launch<8, 1, false, gemm::MODE_DEQ>(p, dev, n_sm, st);
    }
    if (sw_c) {
        if (ncta == 2) {
            if (Lin->bits == 3) return gemm::launch<3, 2, false, gemm::MODE_ASYM>(p, dev, n_sm, st);
            if (Lin->bits == 4) return gemm::launch<4, 2, false, gemm::MODE_ASYM>(p, dev, n_sm, st);
            return gemm::launch<8, 2, true, gemm::MODE_ASYM>(p, dev, n_sm, st);
        }
        if (Lin->bits == 3) return gemm::launch<3, 1, false, gemm::MODE_ASYM>(p, dev, n_sm, st);
        if (Lin->bits == 4) return gemm::launch<4, 1, false, gemm::MODE_ASYM>(p, dev, n_sm, st);
        return gemm::launch<8, 1, false, gemm::MODE_ASYM>(p, dev, n_sm, st);
    }
    // Sums by rows (see the epilogue) for CTA pairs with many clusters, whose drains set the pace: 4 bits, 16-lane layout -> rows, us: 2000 x 1024 x 4096
    // to fp16, 64 clusters 87.4 -> 81.5, 32 50.5 -> 47.9; 2048 x 4096 x 16384, 32: 188 -> 184; codes of 4096 x 2048 x 8192, 32: 190 -> 179. With few
    // the outputs' tables count for more: 2000 x 1024 x 4096 to fp32, 8 clusters: 25.5 and 26.0, 1999 x 2048 x 6144, 8 bits: 50.6 and 52.4
    // (with the LayerNorm); 16 clusters are even. Long clusters, whose drains pass under the products, would still be up to 1.7 % faster the other way
    // (1024 x 9216 x 9216, 32: 79.8 and 81.3), and so would be the rows for codes of few clusters (4096 x 768 x 3072, 8: 30.6 and 29.1), but
    // both linears of an MLP should run the same instance: one whose code the call before did not run costs 2 to 5 us more
    // (400 x 1328 x 3984 x 1328, 16 clusters: 37.6 with one, 41.2 with both).
    const bool by_rows = Lin->n_seg >= 20;
    if (ncta == 2) {
        if (Lin->bits == 3) return by_rows ? gemm::launch<3, 2, false, gemm::MODE_INT, true>(p, dev, n_sm, st) : gemm::launch<3, 2, false, gemm::MODE_INT>(p, dev, n_sm, st);
        if (Lin->bits == 4) return by_rows ? gemm::launch<4, 2, false, gemm::MODE_INT, true>(p, dev, n_sm, st) : gemm::launch<4, 2, false, gemm::MODE_INT>(p, dev, n_sm, st);
        // 8-bit codes need no unpacking
        return by_rows ? gemm::launch<8, 2, true, gemm::MODE_INT, true>(p, dev, n_sm, st) : gemm::launch<8, 2, true, gemm::MODE_INT>(p, dev, n_sm, st);
    }
    if (Lin->bits == 3) return gemm::launch<3, 1, false, gemm::MODE_INT>(p, dev, n_sm, st);
    if (Lin->bits == 4) return gemm::launch<4, 1, false, gemm::MODE_INT>(p, dev, n_sm, st);
    return gemm::launch<8, 1, false, gemm::MODE_INT>(p, dev, n_sm, st);
}

extern "C" int rptq_cluster_gemm_clustered(const rptq_layout_t* Lin, const void* a_codes, int M, const int32_t* xsum,
                                           const void* w_codes, const float* s_w, const int32_t* z_w, const int32_t* wsum,
                                           int64_t ld_w, const void* bias, int N, int act, const rptq_layout_t* Lout,
                                           void* y, int y_dtype, int64_t ldy, void* stream)
{
    int dev = -1;
    const int rc = check_gemm_args(Lin, a_codes, M, w_codes, s_w, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, &dev);
    if (rc != RPTQ_OK) return rc;
    if (!z_w || !xsum || !aligned16(z_w) || !aligned16(xsum)) return RPTQ_ERR_INVALID_ARG;
    if (ld_w % 4 != 0) return RPTQ_ERR_UNSUPPORTED;       // the tables are read four columns at a time
    if (M == 0) return RPTQ_OK;
    int* status = device_status_word();
    if (!status) return RPTQ_ERR_ALLOC;
    return launch_gemm(Lin, a_codes, M, w_codes, nullptr, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, stream, dev, status,
                       nullptr, s_w, z_w, xsum);
}

extern "C" int rptq_cluster_gemm(const rptq_layout_t* Lin, const void* a_codes, int M, const void* w_codes,
                                 const float* s_w, const int32_t* wsum, int64_t ld_w, const void* bias, int N,
                                 int act, const rptq_layout_t* Lout, void* y, int y_dtype, int64_t ldy, void* stream)
{
    int dev = -1;
    const int rc = check_gemm_args(Lin, a_codes, M, w_codes, s_w, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, &dev);
    if (rc != RPTQ_OK) return rc;
    if (M == 0) return RPTQ_OK;
    int* status = device_status_word();
    if (!status) return RPTQ_ERR_ALLOC;
    return launch_gemm(Lin, a_codes, M, w_codes, s_w, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, stream, dev, status, nullptr);
}

extern "C" int rptq_dequant_gemm(const rptq_layout_t* Lin, const void* a_codes, int M, const void* w_codes,
                                 const float* s_w, int64_t ld_w, const void* bias, int N, int act,
                                 void* y, int y_dtype, int64_t ldy, void* stream)
{
    int dev = -1;
    if (y_dtype != RPTQ_OUT_F32 && y_dtype != RPTQ_OUT_F16) return RPTQ_ERR_INVALID_ARG;
    // (the integer tables of the second method are not needed: any aligned non-null pointer passes the shared checks)
    const int rc = check_gemm_args(Lin, a_codes, M, w_codes, s_w, reinterpret_cast<const int32_t*>(s_w), ld_w, bias, N, act,
                                   nullptr, y, y_dtype, ldy, &dev);
    if (rc != RPTQ_OK) return rc;
    if (M == 0) return RPTQ_OK;
    int* status = device_status_word();
    if (!status) return RPTQ_ERR_ALLOC;
    return launch_gemm(Lin, a_codes, M, w_codes, s_w, nullptr, ld_w, bias, N, act, nullptr, y, y_dtype, ldy, stream, dev, status,
                       nullptr, nullptr, nullptr, nullptr, true);
}

// ---------------------------------------------------------------- entry point that allocates nothing
namespace rptq {
namespace gemm {

// Scratch of rptq_cluster_gemm_noalloc: one zero-point correction per output column, resident in
// every device that loads the library (256 KiB) until the process exits.
static __device__ __align__(256) float g_noalloc_corr[RPTQ_NOALLOC_MAX_N];

// corr[n] = sum_c s_c z_c Wsum_c[n], the same fused multiply-adds, in the same order, as the GEMM
// epilogue performs when it is given no table.
__global__ void noalloc_corr_kernel(const float* __restrict__ cl_sz, const int32_t* __restrict__ wsum, int64_t ld_w,
                                    int g, int N, float* __restrict__ corr)
{
    pdl_trigger();
    pdl_wait();
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float acc = 0.f;
    for (int c = 0; c < g; ++c) acc = __fmaf_rn(__ldg(cl_sz + c), (float)__ldg(wsum + (int64_t)c * ld_w + n), acc);
    corr[n] = acc;
}

// Device address of the scratch array, looked up once per context (each loads the library's code and arrays anew). In host code
// the array's name is only a handle for the runtime; the address a kernel can use comes from cudaGetSymbolAddress with that
// device current. One entry per device: the context that called last.
static int noalloc_scratch(int dev, float** out)
{
    struct Address { uint64_t context; float* p; };
    static std::mutex mu;
    static Address known[kMaxDevices] = {};
    if (dev < 0 || dev >= kMaxDevices) return RPTQ_ERR_UNSUPPORTED;
    const uint64_t id = context_id();
    std::lock_guard<std::mutex> lock(mu);
    if (id == 0 || known[dev].context != id) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_corr) != cudaSuccess || !p) return RPTQ_ERR_CUDA;
        known[dev] = {id, static_cast<float*>(p)};
    }
    *out = known[dev].p;
    return RPTQ_OK;
}

}  // namespace gemm
}  // namespace rptq

extern "C" int rptq_cluster_gemm_noalloc(const rptq_layout_t* Lin, const void* a_codes, int M, const void* w_codes,
                                         const float* s_w, const int32_t* wsum, int64_t ld_w, const void* bias, int N,
                                         int act, const rptq_layout_t* Lout, void* y, int y_dtype, int64_t ldy, void* stream)
{
    int dev = -1;
    int rc = check_gemm_args(Lin, a_codes, M, w_codes, s_w, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, &dev);
    if (rc != RPTQ_OK) return rc;
    if (N > RPTQ_NOALLOC_MAX_N) return RPTQ_ERR_UNSUPPORTED;    // more output columns than the resident table holds
    if (M == 0) return RPTQ_OK;
    float* corr = nullptr;
    rc = gemm::noalloc_scratch(dev, &corr);
    if (rc != RPTQ_OK) return rc;
    auto st = static_cast<cudaStream_t>(stream);
    // Every column the GEMM will read is rewritten here first, so nothing of the previous call's
    // contents survives where it matters and nothing needs to start at zero.
    rc = launch_kernel(gemm::noalloc_corr_kernel, dim3((unsigned)((N + 255) / 256)), 256, 0, 0, st, (const float*)Lin->d_cl_sz, wsum, ld_w, Lin->g, N, corr);
    if (rc != RPTQ_OK) return rc;
    return launch_gemm(Lin, a_codes, M, w_codes, s_w, wsum, ld_w, bias, N, act, Lout, y, y_dtype, ldy, stream, dev, nullptr, corr);
}
