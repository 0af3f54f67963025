// The cluster GEMM for at most 16 tokens (decoding): Appendix, second computation method, with the
// same arithmetic as the tcgen05 kernel of cluster_gemm.cu -- exact integer sums per cluster, the
// same fp32 fused multiply-adds in the same order afterwards -- so a token's result does not depend
// on which of the two kernels computed it.
//
// With so few tokens the product is bound by reading the packed weights once (N * K_pad / 2 bytes);
// the 128 x 256 tensor-memory tile of the large kernel would be almost empty and its unpacking of
// the weights to bytes in shared memory costs more than the reading. Here:
//   - a block owns 256 output channels (two 128-row weight tiles), 128 where there are no more tiles than SMs. A producer
//     warp streams their 8 KiB tiles, K block after K block, into an eight-stage shared-memory ring by tensor-map copies of
//     64-byte rows (ordinary loads keep too few bytes in flight per SM to fill the memory pipe with a read-only
//     stream);
//   - the tokens' codes sit in shared memory as 4-bit nibbles in the packed format of the 4-bit
//     codes (16 x K_pad / 2 bytes), written once per block;
//   - each of the 16 consumer warps owns 16 channels (weight rows) for the whole contraction and
//     multiplies with mma.sync m16n8k32: the weight rows are the instruction's M dimension (signed
//     8-bit operands = 16 w, as in the large kernel, three logic instructions per operand pair), the
//     tokens its N dimension (unsigned 8-bit), so the per-channel constants of the epilogue are
//     per-thread scalars. An instruction multiplies one unit of 32 positions: ldmatrix hands lane (g, t)
//     word t of every unit of rows g and g + 8 (a matrix = eight rows' 16 bytes of one unit), and the tokens' words are stored
//     so that one 16-byte load has the lane's word of all four units of a K block. So a unit's products go to its own
//     cluster's accumulator, and a cluster is drained where its last unit was multiplied.
//     (An instruction over one word of all four units needs no ldmatrix, but a K block
//     whose units belong to several clusters is then multiplied once per cluster with the others' lanes zeroed: twice the
//     instructions. 16 x 9216 x 36864, 3 bits, with the LayerNorm: 58.1 -> 51.4 us; the copies' 64-byte swizzle, which keeps
//     ldmatrix free of bank conflicts, 49.6.)
//   - the zero-point corrections (a sum over the clusters per channel) are formed by two warps of their own while the weights
//     stream, not at the end, and a consumer warp unpacks whole token rows, four units' loads at a time: 46.0 us (one token
//     44.7 -> 39.1; with the consumers' arithmetic left out 38.7: the weight stream bounds that, at 4.9 TB/s).
#include <cuda.h>
#include <cuda_fp16.h>

#include "rptq_internal.h"
#include "tc.cuh"
#include "unpack.cuh"

namespace rptq {
namespace smallm {

constexpr int CONSUMER_WARPS = 16;
constexpr int TABLE_WARPS = 2;
constexpr int THREADS = 32 * (CONSUMER_WARPS + 1 + TABLE_WARPS);      // consumers, producer, column tables
constexpr int SMEM_LIMIT = 227 * 1024 - 3328;           // dynamic; the static arrays take 3200 bytes
constexpr int STAGES = 8;
constexpr int STAGE_BYTES = 16384;          // two 8 KiB weight tiles: K block kb of both 128-row tiles

using namespace tc;

__device__ __forceinline__ void mma_s8u8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.u8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldmatrix4(uint32_t (&x)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(addr) : "memory");
}

template <int BITS, int NT>
__global__ void __launch_bounds__(THREADS, 1)
small_m_kernel(const SmallMParams p, const __grid_constant__ CUtensorMap w_map)
{
    extern __shared__ __align__(128) uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 511u) & ~511u;         // (the ring's swizzle repeats every 512 bytes)
    uint8_t* smem = smem_raw + (base - smem_u32(smem_raw));
    // ring | token codes (nibbles) | per unit: s_c / 16, step flags | barriers
    const int a_pitch = p.K_pad / 2 + (((p.K_pad / 2) & 127) ? 0 : 64);      // odd multiple of 64: two token rows fill the 32 banks
    uint8_t* ring = smem;
    uint8_t* act = ring + STAGES * STAGE_BYTES;
    float* unit_scale = reinterpret_cast<float*>(act + 8 * NT * a_pitch);    // [4 n_kb]
    uint8_t* unit_flags = reinterpret_cast<uint8_t*>(unit_scale + 4 * p.n_kb);
    uint64_t* bars = reinterpret_cast<uint64_t*>(unit_flags + (4 * p.n_kb + 7) / 8 * 8);       // full[STAGES], empty[STAGES]
    __shared__ int s_abort_flag;
    __shared__ float s_col[3][256];              // zero-point correction, s_w and bias of the block's channels
    volatile int* s_abort = &s_abort_flag;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);

    if (tid == 0) {
        s_abort_flag = 0;
        for (int s = 0; s < STAGES; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8 * s) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(empty0 + 8 * s), "r"(CONSUMER_WARPS) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // (the layout's own tables)
    for (int u = tid; u < 4 * p.n_kb; u += THREADS) { unit_scale[u] = __ldg(&p.unit_sz[u].x) * 0.0625f; unit_flags[u] = __ldg(p.step_flags + u); }
    const int tileA = p.tiles_per_block * (int)blockIdx.x;
    const bool haveB = p.tiles_per_block == 2 && tileA + 1 < p.n_wtiles;
    __syncthreads();
    pdl_trigger();
    pdl_wait();

    float R[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) R[nt][e] = 0.f;

    if (warp == CONSUMER_WARPS) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            // the weights as rows of 64 bytes: K block kb of tile t is rows 128 (t n_kb + kb) ..
            const int rowA = tileA * p.n_kb * 128, rowB = rowA + p.n_kb * 128;
            const uint32_t bytes = haveB ? STAGE_BYTES : STAGE_BYTES / 2;      // (the second tile's half of a stage stays empty)
            int issued = 0;
            for (int kb = 0; kb < p.n_kb; ++kb) {
                const int s = kb % STAGES;
                if (kb >= STAGES && !mbar_wait(empty0 + 8 * s, (uint32_t)(kb / STAGES - 1) & 1u, s_abort)) break;
                if (*s_abort) break;
                const uint32_t dst = smem_u32(ring + s * STAGE_BYTES), bar = full0 + 8 * s;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
                auto load = [&](uint32_t to, int row) {
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(to), "l"(&w_map), "r"(0), "r"(row), "r"(bar) : "memory");
                };
                load(dst, rowA + 128 * kb);
                if (haveB) load(dst + 8192, rowB + 128 * kb);
                issued = kb + 1;
            }
            // After a give-up the consumers no longer wait for the copies still in flight: they must have
            // landed before the block's shared memory goes away (bounded like every other wait).
            if (*s_abort) {
                for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb) mbar_wait(full0 + 8 * (kb % STAGES), (uint32_t)(kb / STAGES) & 1u, s_abort, false);
            }
        }
    } else if (warp > CONSUMER_WARPS) {
        // ------------------------------------------------------------ column tables: two warps, four channels a lane (in the consumers'
        // own code the loads of the g clusters took 3 us at the end of the kernel)
        const int at = 128 * (warp - CONSUMER_WARPS - 1) + lane, n = tileA * 128 + at;      // my channels: n + 32 e
        float corr[4] = {0.f, 0.f, 0.f, 0.f};
        if (p.corr) {
#pragma unroll
            for (int e = 0; e < 4; ++e) if (n + 32 * e < p.N) corr[e] = p.corr[n + 32 * e];
        } else {
#pragma unroll 4
            for (int c = 0; c < p.g; ++c) {
                const float sz = __ldg(p.cl_sz + c);
#pragma unroll
                for (int e = 0; e < 4; ++e) corr[e] = __fmaf_rn(sz, n + 32 * e < p.N ? (float)__ldg(p.wsum + (int64_t)c * p.ld_w + n + 32 * e) : 0.f, corr[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool in = n + 32 * e < p.N;
            s_col[0][at + 32 * e] = corr[e];
            s_col[1][at + 32 * e] = in ? __ldg(p.s_w + n + 32 * e) : 0.f;
            s_col[2][at + 32 * e] = in && p.bias ? __ldg(p.bias + n + 32 * e) : 0.f;
        }
        asm volatile("bar.arrive 2, %0;" ::"n"(32 * (CONSUMER_WARPS + TABLE_WARPS)) : "memory");
    } else {
        // ------------------------------------------------------------ consumers
        // (the producer is already streaming weights while the consumers prepare their tables)
        const int tile_sel = warp >> 3;                       // which of the block's two tiles
        const bool active = tile_sel == 0 || haveB;
        const int n0 = (tileA + tile_sel) * 128 + 16 * (warp & 7);
        // The tokens' codes as nibbles: word j of a unit holds positions 8j..8j+3 in the low and 8j+4..8j+7 in the high nibbles
        // of its bytes (the packed format of 4-bit codes). Word j of the four units of a K block are stored side by side. Rows >= M
        // are zero. Four units a thread at a time, their loads first.
        {
            constexpr int SPLIT = 2 / NT;                     // warps of a row
            const int r = warp / SPLIT;
            const uint32_t* row = reinterpret_cast<const uint32_t*>(p.a + (int64_t)(r < p.M ? r : 0) * p.a_row_bytes);
#pragma unroll 1
            for (int u0 = lane + 32 * (warp % SPLIT); u0 < p.n_units; u0 += 4 * 32 * SPLIT) {
                uint32_t q[4][BITS];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int u = u0 + k * 32 * SPLIT;
                    const bool in = r < p.M && u < p.n_units;
#pragma unroll
                    for (int e = 0; e < BITS; ++e) q[k][e] = in ? row[u * BITS + e] : 0u;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int u = u0 + k * 32 * SPLIT;
                    if (u >= p.n_units) break;
                    uint32_t o[8];
                    unpack_act32<BITS>(q[k], o);
                    uint32_t* d = reinterpret_cast<uint32_t*>(act + r * a_pitch + 64 * (u >> 2) + 4 * (u & 3));
#pragma unroll
                    for (int e = 0; e < 4; ++e) d[4 * e] = o[2 * e] | (o[2 * e + 1] << 4);
                }
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * CONSUMER_WARPS) : "memory");
        // lane i hands ldmatrix row i % 8 of matrix (unit) i / 8; piece c of row r lies at c ^ ((r / 2) & 3)
        const uint32_t w_at = smem_u32(ring) + tile_sel * 8192 + (16 * (warp & 7) + (lane & 7)) * 64 + 16 * ((lane >> 3) ^ ((lane >> 1) & 3));
        const uint8_t* arow = act + g8 * a_pitch + 16 * t4;
        int acc0[NT][4], acc1[NT][4];                         // the two accumulators (as in the large kernel, the layout says which)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) { acc0[nt][e] = 0; acc1[nt][e] = 0; }

        for (int kb = 0; kb < p.n_kb; ++kb) {
            const int s = kb % STAGES;
            const uint32_t f4 = __shfl_sync(0xffffffffu, *reinterpret_cast<const uint32_t*>(unit_flags + 4 * kb), 0);
            uint4 B[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) B[nt] = *reinterpret_cast<const uint4*>(arow + 8 * nt * a_pitch + 64 * kb);
            // (when a wait has given up, the remaining K blocks multiply what lies in the ring, and nothing is written out)
            mbar_sleep_or_abort(full0 + 8 * s, (uint32_t)(kb / STAGES) & 1u, s_abort);
            __syncwarp();
            if (!active) {
                if (lane == 0) mbar_arrive(empty0 + 8 * s);
                continue;
            }
            uint32_t x0[4], x1[4];                            // rows g8, g8 + 8: word t4 of the four units
            ldmatrix4(x0, w_at + s * STAGE_BYTES);
            ldmatrix4(x1, w_at + s * STAGE_BYTES + 512);
            __syncwarp();
            if (lane == 0) mbar_arrive(empty0 + 8 * s);       // the stage's bytes are in registers
            auto multiply = [&](int j, int (&acc)[NT][4]) {   // unit j
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const uint32_t b = j == 0 ? B[nt].x : j == 1 ? B[nt].y : j == 2 ? B[nt].z : B[nt].w;
                    mma_s8u8(acc[nt], (x0[j] << 4) & 0xF0F0F0F0u, (x1[j] << 4) & 0xF0F0F0F0u, x0[j] & 0xF0F0F0F0u, x1[j] & 0xF0F0F0F0u,
                             b & 0x0F0F0F0Fu, (b >> 4) & 0x0F0F0F0Fu);
                }
            };
            constexpr uint32_t ALL = 0x01010101u;
            if ((f4 & (ALL * (STEP_LAST | STEP_SKIP | STEP_BUF))) == 0u) {
#pragma unroll
                for (int j = 0; j < 4; ++j) multiply(j, acc0);
            } else if ((f4 & (ALL * (STEP_LAST | STEP_SKIP | STEP_BUF))) == ALL * STEP_BUF) {
#pragma unroll
                for (int j = 0; j < 4; ++j) multiply(j, acc1);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t f = f4 >> (8 * j);
                    if (f & STEP_SKIP) continue;
                    auto unit = [&](int (&acc)[NT][4]) {
                        multiply(j, acc);
                        if (f & STEP_LAST) {
                            const float sc = unit_scale[4 * kb + j];
#pragma unroll
                            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                                for (int e = 0; e < 4; ++e) { R[nt][e] = __fmaf_rn(sc, (float)acc[nt][e], R[nt][e]); acc[nt][e] = 0; }
                        }
                    };
                    if (f & STEP_BUF) unit(acc1); else unit(acc0);
                }
            }
        }

        // -------------------------------------------------------- epilogue: y = s_w (R - corr) + bias
        asm volatile("bar.sync 2, %0;" ::"n"(32 * (CONSUMER_WARPS + TABLE_WARPS)) : "memory");
        if (active && n0 < p.N && !__any_sync(0xffffffffu, *s_abort)) {
            const float corr = s_col[0][n0 - 128 * tileA + (lane & 15)], sw = s_col[1][n0 - 128 * tileA + (lane & 15)], bs = s_col[2][n0 - 128 * tileA + (lane & 15)];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {             // rows g (accumulator entries 0, 1) and g + 8 (entries 2, 3)
                const int src = g8 + 8 * hh, n = n0 + src;
                const float c = __shfl_sync(0xffffffffu, corr, src), s = __shfl_sync(0xffffffffu, sw, src), b = __shfl_sync(0xffffffffu, bs, src);
                if (n >= p.N) continue;
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int m = 8 * nt + 2 * t4 + e;
                        if (m >= p.M) continue;
                        float v = __fmaf_rn(s, R[nt][2 * hh + e] - c, b);
                        if (p.act == RPTQ_ACT_RELU) v = fmaxf(v, 0.f);
                        if (p.y_dtype == RPTQ_OUT_F32) static_cast<float*>(p.y)[(int64_t)m * p.ldy + n] = v;
                        else static_cast<__half*>(p.y)[(int64_t)m * p.ldy + n] = __float2half_rn(v);
                    }
            }
        }
    }
    __syncthreads();
    if (tid == 0 && *s_abort && p.status) atomicExch(p.status, RPTQ_ERR_DEVICE_TIMEOUT);
}

static int smem_bytes(int nt, int K_pad)
{
    const int a_pitch = K_pad / 2 + (((K_pad / 2) & 127) ? 0 : 64);
    return 512 + STAGES * STAGE_BYTES + 8 * nt * a_pitch + (K_pad / 32) * 4 + (K_pad / 32 + 7) / 8 * 8 + 2 * STAGES * 8;
}

// The packed weights as a matrix of 64-byte rows, copied 128 rows (one tile's K block) at a time with the 64-byte swizzle, so
// that ldmatrix reads eight rows without a bank conflict.
static int weight_map(const SmallMParams& p, CUtensorMap* map)
{
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) fn = nullptr;
        return reinterpret_cast<Encode>(fn);
    }();
    if (!encode) return RPTQ_ERR_CUDA;
    const cuuint64_t dims[2] = {64, (cuuint64_t)p.n_wtiles * p.n_kb * 128}, strides[1] = {64};
    const cuuint32_t box[2] = {64, 128}, step[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t*>(p.w), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? RPTQ_OK : RPTQ_ERR_CUDA;
}

template <int BITS, int NT>
static int launch_one(SmallMParams p, int device, cudaStream_t st)
{
    const int smem = smem_bytes(NT, p.K_pad);
    static SmemAllowed done;
    if (allow_smem(reinterpret_cast<const void*>(small_m_kernel<BITS, NT>), device, SMEM_LIMIT, done) != RPTQ_OK) return RPTQ_ERR_CUDA;
    // a block per 128 channels where the SMs suffice: the call then takes as long as one tile's stream
    const int n_sm = sm_count(device);
    if (n_sm == 0) return RPTQ_ERR_CUDA;
    p.tiles_per_block = p.n_wtiles <= n_sm ? 1 : 2;
    const int blocks = (p.n_wtiles + p.tiles_per_block - 1) / p.tiles_per_block;
    CUtensorMap map;
    if (weight_map(p, &map) != RPTQ_OK) return RPTQ_ERR_CUDA;
    return launch_kernel(small_m_kernel<BITS, NT>, dim3((unsigned)blocks), THREADS, (size_t)smem, 0, st, p, map);
}

bool fits(int M, int bits, int K_pad)
{
    return M <= 16 && (bits == 3 || bits == 4) && smem_bytes(M <= 8 ? 1 : 2, K_pad) <= SMEM_LIMIT;
}

int launch(const SmallMParams& p, int bits, int device, cudaStream_t st)
{
    if (p.M <= 8) return bits == 3 ? launch_one<3, 1>(p, device, st) : launch_one<4, 1>(p, device, st);
    return bits == 3 ? launch_one<3, 2>(p, device, st) : launch_one<4, 2>(p, device, st);
}

}  // namespace smallm
}  // namespace rptq
