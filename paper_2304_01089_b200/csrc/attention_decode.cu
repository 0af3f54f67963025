// Attention for a few queries per sequence (decode steps): rptq_attention and rptq_attention_kv route
// calls with at most 7 (8) queries here.
//
// With one query per head the products are matrix-vector products and the call is bound by reading the
// quantised cache once; the prefill kernels would fill one row of their query tile and walk the keys
// serially in one block per (sequence, head). Here the KEYS are the M dimension of mma.sync:
//   - a thread-block cluster of 1, 2, 4 or 8 blocks shares one (sequence, head), each block takes a
//     contiguous range of keys, each of its four warps every fourth 32-key tile of it. Row maxima, sums and
//     the partial outputs meet through distributed shared memory, so there is no workspace and no
//     second kernel;
//   - packed K and V rows arrive by cp.async in a private ring of each warp (no block-wide barrier in the
//     loops); 3-bit rows are expanded to nibbles once per tile;
//   - scores: K codes are operand A (16 keys x 32 or 16 positions), the queries operand B, held in registers
//     for the whole range. Three modes:
//       INT   everything quantised: bytes, m16n8k32. Column 7 of the queries is all ones, so the same
//             product gives the per-key code sums of the zero-point term;
//       LIMB  fp16 query, at most two of them: the kernel is bound by the instructions that turn codes into
//             operands (1.5 per code for fp16 operands, 0.4 for bytes), and a query fills one column of
//             eight. So the QUERY becomes four signed bytes in four columns: q = X 2^-k, X an integer of 31 bits, with
//             one k per cluster (exact unless |q| is below 2^-19 of the cluster's largest: then it is off by 2^-32 of
//             that at most, less than fp32 sums lose), and the sums are exact integers. (Three bytes and one k per
//             head took the same time, but where a head's clusters differ by 10^4 in the query's magnitude and the keys'
//             scale undoes that, the small queries kept four bits.) The probabilities become three unsigned bytes (24
//             bits, at least fp16's precision everywhere);
//       HALF  fp16 query, three to eight: fp16 operands, m16n8k16. A nibble n moved to mantissa bits 6-9 of
//             16.0 is 16 + n, one packed addition makes it n - 8 (bytes: 1024 + n, n - 128). The centre is a
//             constant of the query row in the scores (it cancels in the softmax) and part of the zero
//             point in the outputs. (Codes as fp16 subnormals would need no arithmetic, but the tensor
//             core aligns products by their exponent fields: their leading zeros were lost from the fp32
//             sums, 1e-3 at scores of 67);
//   - the scores of the block's keys stay in shared memory; the softmax parameters follow from them (for
//     integer calls from the whole cluster's, since the 8-bit codes need the finished sums);
//   - outputs: V^T is operand A (positions x keys; pairs or quads of keys are brought together with byte
//     permutes on the packed words), the probabilities operand B.
// Measured (72 heads of 128 channels, eight sequences, one query, 2011 keys, 4-bit cache, KV-only):
// 1072 us before (prefill kernel), 65 to 67 us here.
#include <type_traits>

#include "attn_common.cuh"

namespace rptq {
namespace attn_decode {

using namespace attn;

constexpr int WARPS = 4, THREADS = 32 * WARPS;
constexpr int TILE = 32;                       // keys per tile of a warp
constexpr int STAGES = 3;
constexpr int MAX_Q = 8;                       // columns of operand B
constexpr int LIMB_Q = 2;                      // queries of the LIMB mode (columns 4 q + limb)
constexpr float P_UNITS = 16776192.0f;         // LIMB: 2^24 - 2^10, so that P = 1 stays below 2^24 by more than ex2's error (2^-22)
constexpr int MAX_CLUSTER = 8;
constexpr int SCORE_BYTES_MAX = 96 * 1024;     // of the block's keys
// shared memory of a block besides the dynamic part: the kernel's static arrays and the system's 1 KiB, rounded up
constexpr int static_smem(bool half_mode) { return half_mode ? 10 * 1024 : 6 * 1024; }
constexpr int SM_BYTES = 227 * 1024;                          // shared memory of an SM that blocks can have
constexpr int dynamic_smem_max(bool half_mode) { return SM_BYTES - static_smem(half_mode); }

__device__ __forceinline__ void mma_u8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.u8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_u8s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 32 bits at this shared-memory address of block `rank` of the cluster
__device__ __forceinline__ uint32_t ld_peer(uint32_t addr, uint32_t rank)
{
    uint32_t v;
    asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\tld.shared::cluster.u32 %0, [ra];\n\t}"
                 : "=r"(v) : "r"(addr), "r"(rank) : "memory");
    return v;
}

__host__ __device__ inline int nibble_pitch(int units) { return 16 * (units | 1); }

struct SmemPlan { int ring_stage, ring, expand, expand_all, scores, score_pitch, total; };
__host__ __device__ inline SmemPlan smem_plan(int bits_k, int bits_v, int units_k, int units_v, int n_q, int keys_block)
{
    SmemPlan s;
    const int pk = raw_pitch(bits_k, units_k), pv = raw_pitch(bits_v, units_v);
    s.ring_stage = TILE * (pk > pv ? pk : pv);
    s.ring = WARPS * STAGES * s.ring_stage;
    const int red = WARPS * n_q * 32 * units_v * 4;           // partial outputs of the four warps, after the loops
    if (s.ring < red) s.ring = red;
    const int ek = bits_k == 3 ? nibble_pitch(units_k) : 0, ev = bits_v == 3 ? nibble_pitch(units_v) : 0;
    s.expand = TILE * (ek > ev ? ek : ev);
    s.expand_all = WARPS * s.expand;
    s.score_pitch = keys_block + 8;
    s.scores = n_q * s.score_pitch * 4;
    s.total = s.ring + s.expand_all + s.scores;
    return s;
}

enum { INT = 0, HALF = 1, LIMB = 2 };
// BK, BV: bits of a code as the inner loops see it (4 or 8; 3-bit rows are expanded to nibbles first).
template <int MODE, int BK, int BV>
__global__ void __launch_bounds__(THREADS)
decode_kernel(const AttnParams p, int keys_block, int units_k_max, int units_v_max)
{
    constexpr bool KV = MODE != INT;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ float s_coef[MODE == LIMB ? LIMB_Q : 1][MAX_UNITS], s_czq[MAX_UNITS];      // (LIMB: times the 2^-k of the query's cluster)
    __shared__ uint32_t s_top[LIMB_Q][MAX_UNITS];             // LIMB: the largest |q| of a unit, as fp16 bits
    __shared__ uint8_t s_last[MAX_UNITS];
    __shared__ float s_wm[WARPS][MAX_Q], s_wl[WARPS][MAX_Q];
    __shared__ float s_m[MAX_Q], s_l[MAX_Q];                  // this block's row maxima and sums (read by its peers)
    __shared__ int s_wrs[WARPS][MAX_Q], s_rs[MAX_Q];
    // the queries in K's position order: fp16 (HALF) or 31-bit integers (LIMB)
    __shared__ __align__(16) uint32_t s_q[MODE == HALF ? MAX_Q * 16 * MAX_UNITS : MODE == LIMB ? LIMB_Q * 32 * MAX_UNITS : 4];
    __shared__ __align__(16) uint32_t s_qb[32 * MAX_UNITS][MODE == HALF ? 4 : 2];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g8 = lane >> 2, t4 = lane & 3;
    const int h = blockIdx.y;
    const uint32_t rank = cluster_rank(), n_ranks = cluster_size();
    const int64_t q_row0 = (int64_t)blockIdx.z * p.Tq, k_row0 = (int64_t)blockIdx.z * p.Tk;
    const int uk0 = __ldg(p.cl_unit0_k + h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (h + 1) * p.gh_k) - uk0;
    const int uv0 = __ldg(p.cl_unit0_v + h * p.gh_v), nuv = __ldg(p.cl_unit0_v + (h + 1) * p.gh_v) - uv0;
    const SmemPlan sp = smem_plan(p.bits_k, p.bits_v, units_k_max, units_v_max, p.Tq, keys_block);
    uint8_t* ring = smem + warp * STAGES * sp.ring_stage;
    uint8_t* expand = smem + sp.ring + warp * sp.expand;
    float* S = reinterpret_cast<float*>(smem + sp.ring + sp.expand_all);       // [Tq][score_pitch]

    const int j0 = (int)rank * keys_block, j1 = min(p.Tk, j0 + keys_block);    // my keys
    const int n_tiles = j1 > j0 ? (j1 - j0 + TILE - 1) / TILE : 0;
    const int my_tiles = n_tiles > warp ? (n_tiles - warp + WARPS - 1) / WARPS : 0;

    // Start the copies of my i-th tile's rows into stage i % STAGES; rows past the last key are zero-filled.
    // Four lanes per row, so that a warp-wide copy touches eight rows and its addresses need no division.
    auto stage_tile = [&](int i, const uint8_t* base, int64_t row_bytes, int bits, int u0, int nu, int pitch) {
        if (i < my_tiles) {
            const int win = (4 * bits * u0) & ~15, n16 = ((4 * bits * u0 - win) + 4 * bits * nu + 15) >> 4;
            const int j = j0 + TILE * (warp + WARPS * i), n_rows = min(TILE, j1 - j);
            const int r0 = lane >> 2, c0 = lane & 3;
            const uint8_t* src = base + (k_row0 + j + r0) * row_bytes + win + 16 * c0;
            uint32_t dst = smem_u32(ring + (i % STAGES) * sp.ring_stage) + r0 * pitch + 16 * c0;
#pragma unroll
            for (int rg = 0; rg < TILE / 8; ++rg) {
                const bool ok = r0 + 8 * rg < n_rows;
                const uint8_t* from = ok ? src : base;             // (an address that is not read)
#pragma unroll
                for (int c = 0; c < 4; ++c) {                      // at most 16 chunks per row
                    if (c0 + 4 * c < n16) cp_async16(dst + 64 * c, ok ? from + 64 * c : from, ok);
                    if (4 * c + 4 >= n16) break;
                }
                src += 8 * row_bytes; dst += 8 * pitch;
            }
        }
        cp_async_commit();
    };
    // 3-bit rows of the staged tile -> nibble rows
    auto expand_tile = [&](const uint8_t* raw, int raw_p, int off, int nu) {
        const int ep = nibble_pitch(nu);
        for (int it = lane; it < TILE * nu; it += 32) {
            const int r = it & (TILE - 1), u = it / TILE;
            const uint32_t* w = reinterpret_cast<const uint32_t*>(raw + r * raw_p + off) + 3 * u;
            const uint32_t a = w[0], b = w[1], c = w[2];
            const uint32_t tail = ((a >> 3) & 0x11111111u) | (((b >> 3) & 0x11111111u) << 1) | (((c >> 3) & 0x11111111u) << 2);
            *reinterpret_cast<uint4*>(expand + r * ep + 16 * u) = make_uint4(a & 0x77777777u, b & 0x77777777u, c & 0x77777777u, tail);
        }
        __syncwarp();
    };

    pdl_trigger();
    pdl_wait();
    const int pk = raw_pitch(p.bits_k, units_k_max), pv = raw_pitch(p.bits_v, units_v_max);
#pragma unroll 1
    for (int i = 0; i < STAGES - 1; ++i) stage_tile(i, p.k, p.k_row_bytes, p.bits_k, uk0, nuk, pk);

    // ---------------------------------------------------------------- the queries, as operand B of every unit
    if (tid < nuk) {
        const float2 k = __ldg(p.unit_sz_k + uk0 + tid);
        if constexpr (MODE == HALF) {
            s_coef[0][tid] = k.x * p.qk_scale_log2e;
        } else if constexpr (MODE == INT) {
            const float2 q = __ldg(p.unit_sz_q + uk0 + tid);
            const float c = q.x * k.x * p.qk_scale_log2e;
            s_coef[0][tid] = c;
            s_czq[tid] = -c * q.y;
        }
        s_last[tid] = (tid == nuk - 1) || (__ldg(p.unit_cluster_k + uk0 + tid + 1) != __ldg(p.unit_cluster_k + uk0 + tid));
    }
    if constexpr (MODE == HALF) {
        __half* sq = reinterpret_cast<__half*>(s_q);
        for (int it = tid; it < p.Tq * 32 * nuk; it += THREADS) {
            const int q = it / (32 * nuk), pp = it - q * (32 * nuk), pos = 32 * uk0 + pp;
            sq[q * 32 * MAX_UNITS + pp] = __ldg(p.jidx_k + pos) >= 0 ? p.q_f16[(q_row0 + q) * p.ldq + __ldg(p.src_k + pos)] : __ushort_as_half(0);
        }
    } else if constexpr (MODE == LIMB) {
        // my positions of the queries: lane of unit warp + 4 k
        uint32_t raw[LIMB_Q][MAX_UNITS / WARPS];
#pragma unroll
        for (int k = 0; k < MAX_UNITS / WARPS; ++k) {
            const int u = warp + WARPS * k, pos = 32 * (uk0 + u) + lane;
            const int ch = u < nuk && __ldg(p.jidx_k + pos) >= 0 ? (int)__ldg(p.src_k + pos) : -1;
#pragma unroll
            for (int q = 0; q < LIMB_Q; ++q) {
                raw[q][k] = ch >= 0 && q < p.Tq ? (uint32_t)__half_as_ushort(p.q_f16[(q_row0 + q) * p.ldq + ch]) : 0u;
                const uint32_t top = __reduce_max_sync(0xffffffffu, raw[q][k] & 0x7FFFu);
                if (lane == 0) s_top[q][u] = top;
            }
        }
        __syncthreads();
        const int cl = lane < nuk ? __ldg(p.unit_cluster_k + uk0 + lane) : -1;
        const float c = lane < nuk ? __ldg(&p.unit_sz_k[uk0 + lane].x) * p.qk_scale_log2e : 0.f;
#pragma unroll
        for (int q = 0; q < LIMB_Q; ++q) {
            // lane = unit: the largest |q| of its cluster
            const uint32_t mine = lane < MAX_UNITS ? s_top[q][lane] : 0u;
            uint32_t top = mine;
#pragma unroll
            for (int i = 0; i < MAX_UNITS; ++i) {
                const uint32_t t = __shfl_sync(0xffffffffu, mine, i);
                if (__shfl_sync(0xffffffffu, cl, i) == cl) top = max(top, t);
            }
            // its exponent field e: |q| < 2^(e - 126), so |q| 2^(156 - e) < 2^30 (no fp16 number is below 2^-24)
            const bool finite = top < 0x7C00u;
            const int e = finite ? max(__float_as_int(__half2float(__ushort_as_half((unsigned short)top))) >> 23, 103) : 103;
            // a query that is not finite makes its scores, and so its outputs, not a number
            if (warp == 0 && lane < nuk) s_coef[q][lane] = finite ? c * __int_as_float((e - 29) << 23) : __int_as_float(0x7FC00000);
            const float to_int = finite ? __int_as_float((283 - e) << 23) : 0.f;
#pragma unroll
            for (int k = 0; k < MAX_UNITS / WARPS; ++k) {
                const int u = warp + WARPS * k;
                const float f = __shfl_sync(0xffffffffu, to_int, u);
                // (0 times infinity is converted to 0)
                reinterpret_cast<int*>(s_q)[q * 32 * MAX_UNITS + 32 * u + lane] = __float2int_rn(__half2float(__ushort_as_half((unsigned short)raw[q][k])) * f);
            }
        }
    }
    __syncthreads();
    // operand B of unit u for lane l, the same for all warps: written once by the block, then held in registers
    constexpr int QW = MODE == HALF ? 4 : 2;
#pragma unroll 1
    for (int it = tid; it < nuk * 32; it += THREADS) {
        const int u = it >> 5, l = it & 31, col = l >> 2, w = l & 3;           // column; word of the unit (codes 8 w .. 8 w + 7)
        uint32_t b[QW] = {};
        if constexpr (MODE == HALF) {
            // register i pairs codes (0, 2), (1, 3), (4, 6), (5, 7) as nib_half does
            if (col < p.Tq) {
                const uint4 v = *reinterpret_cast<const uint4*>(s_q + col * 16 * MAX_UNITS + 16 * u + 4 * w);
                b[0] = __byte_perm(v.x, v.y, 0x5410); b[1] = __byte_perm(v.x, v.y, 0x7632);
                b[2] = __byte_perm(v.z, v.w, 0x5410); b[3] = __byte_perm(v.z, v.w, 0x7632);
            }
        } else if constexpr (MODE == LIMB) {
            // column 4 q + limb: X = d0 + 2^8 d1 + 2^16 d2 + 2^24 d3 with signed bytes d; adding half of every lower
            // digit's range turns the arithmetic shift into the balanced digit
            const int q = col >> 2, limb = col & 3;
            if (q < p.Tq) {
                const int* x = reinterpret_cast<const int*>(s_q) + q * 32 * MAX_UNITS + 32 * u + 8 * w;
                const int half = limb == 0 ? 0 : limb == 1 ? 128 : limb == 2 ? 128 + 32768 : 128 + 32768 + 8388608;
#pragma unroll
                for (int i = 0; i < 8; ++i) b[i >> 2] |= ((uint32_t)((x[i] + half) >> (8 * limb)) & 255u) << (8 * (i & 3));
            }
        } else if (col == 7) {
            b[0] = b[1] = 0x01010101u;                                         // code sums of the keys
        } else if (col < p.Tq) {
            const uint8_t* row = p.q + (q_row0 + col) * p.q_row_bytes;
            const int unit = uk0 + u;
            if (p.bits_q == 8) {
                const uint2 v = reinterpret_cast<const uint2*>(row + 32 * unit)[w];
                b[0] = v.x; b[1] = v.y;
            } else if (p.bits_q == 4) {
                const uint32_t v = reinterpret_cast<const uint32_t*>(row + 16 * unit)[w];
                b[0] = v & 0x0F0F0F0Fu; b[1] = (v >> 4) & 0x0F0F0F0Fu;
            } else {
                const uint32_t* v = reinterpret_cast<const uint32_t*>(row + 12 * unit);
                const uint32_t q3[3] = {v[0], v[1], v[2]};
                uint32_t o[8];
                unpack_act32<3>(q3, o);
                b[0] = w == 0 ? o[0] : w == 1 ? o[2] : w == 2 ? o[4] : o[6];
                b[1] = w == 0 ? o[1] : w == 1 ? o[3] : w == 2 ? o[5] : o[7];
            }
        }
#pragma unroll
        for (int i = 0; i < QW; ++i) s_qb[u * 32 + l][i] = b[i];
    }
    __syncthreads();
    uint32_t qb[MAX_UNITS][QW];
#pragma unroll
    for (int u = 0; u < MAX_UNITS; ++u) {
#pragma unroll
        for (int i = 0; i < QW; ++i) qb[u][i] = u < nuk ? s_qb[u * 32 + lane][i] : 0u;
    }

    // ---------------------------------------------------------------- scores of my keys
    const int off = p.Tk - p.Tq;
    const int q0 = MODE == LIMB ? t4 >> 1 : 2 * t4, q1 = q0 + 1;               // the queries of my columns of the score fragments
    // LIMB: my two columns' weights (the two lanes of a query hold digits 0, 1 and digits 2, 3)
    const float w0 = (t4 & 1) ? 65536.0f : 1.0f, w1 = (t4 & 1) ? 16777216.0f : 256.0f;
    const float* coef = s_coef[MODE == LIMB ? q0 : 0];
    const int vis0 = p.causal ? min(p.Tk - 1, q0 + off) : p.Tk - 1, vis1 = p.causal ? min(p.Tk - 1, q1 + off) : p.Tk - 1;
    float m0 = NEG_BIG, m1 = NEG_BIG;
    uint32_t last_mask = 0u;
    for (int u = 0; u < nuk; ++u) last_mask |= (uint32_t)s_last[u] << u;
    const int offK = (4 * p.bits_k * uk0) & 15;
    for (int i = 0; i < my_tiles; ++i) {
        stage_tile(i + STAGES - 1, p.k, p.k_row_bytes, p.bits_k, uk0, nuk, pk);
        cp_async_wait<STAGES - 1>();
        __syncwarp();
        const uint8_t* rows = ring + (i % STAGES) * sp.ring_stage + offK;
        int pitch = pk;
        if (BK == 4 && p.bits_k == 3) {
            expand_tile(rows - offK, pk, offK, nuk);
            rows = expand; pitch = nibble_pitch(nuk);
        }
        const int jt = TILE * (warp + WARPS * i);                              // first key of the tile within my range
        const bool all_visible = j0 + jt + TILE <= j1 && (!p.causal || j0 + jt + TILE - 1 <= off);
        const uint8_t* r0 = rows + g8 * pitch + (BK == 4 ? 4 : 8) * t4;        // my word of keys g8, g8 + 8, g8 + 16, g8 + 24
        typename std::conditional<MODE == HALF, float, int>::type acc[2][4] = {};
        float Sv[2][4] = {}, col[2][2] = {};
#pragma unroll
        for (int u = 0; u < MAX_UNITS; ++u) {
            if (u < nuk) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint8_t* ra = r0 + 16 * half * pitch, *rb = ra + 8 * pitch;
                    if constexpr (BK == 4) {
                        const uint32_t a = *reinterpret_cast<const uint32_t*>(ra + 16 * u), b = *reinterpret_cast<const uint32_t*>(rb + 16 * u);
                        if constexpr (MODE == HALF) {
                            mma_f16(acc[half], nib_half<0>(a), nib_half<0>(b), nib_half<8>(a), nib_half<8>(b), qb[u][0], qb[u][1]);
                            mma_f16(acc[half], nib_half<4>(a), nib_half<4>(b), nib_half<12>(a), nib_half<12>(b), qb[u][2], qb[u][3]);
                        } else if constexpr (MODE == LIMB) {
                            mma_u8s8(acc[half], a & 0x0F0F0F0Fu, b & 0x0F0F0F0Fu, (a >> 4) & 0x0F0F0F0Fu, (b >> 4) & 0x0F0F0F0Fu, qb[u][0], qb[u][1]);
                        } else {
                            mma_u8(acc[half], a & 0x0F0F0F0Fu, b & 0x0F0F0F0Fu, (a >> 4) & 0x0F0F0F0Fu, (b >> 4) & 0x0F0F0F0Fu, qb[u][0], qb[u][1]);
                        }
                    } else {
                        const uint2 a = *reinterpret_cast<const uint2*>(ra + 32 * u), b = *reinterpret_cast<const uint2*>(rb + 32 * u);
                        if constexpr (MODE == HALF) {
                            mma_f16(acc[half], byte_half<0>(a.x), byte_half<0>(b.x), byte_half<8>(a.x), byte_half<8>(b.x), qb[u][0], qb[u][1]);
                            mma_f16(acc[half], byte_half<0>(a.y), byte_half<0>(b.y), byte_half<8>(a.y), byte_half<8>(b.y), qb[u][2], qb[u][3]);
                        } else if constexpr (MODE == LIMB) {
                            mma_u8s8(acc[half], a.x, b.x, a.y, b.y, qb[u][0], qb[u][1]);
                        } else {
                            mma_u8(acc[half], a.x, b.x, a.y, b.y, qb[u][0], qb[u][1]);
                        }
                    }
                }
                if ((last_mask >> u) & 1u) {
                    const float c = coef[u];
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        if constexpr (MODE == LIMB) {                          // entries 0 and 2: keys g8 and g8 + 8
                            Sv[half][0] = __fmaf_rn(c, __fmaf_rn(w1, (float)acc[half][1], w0 * (float)acc[half][0]), Sv[half][0]);
                            Sv[half][2] = __fmaf_rn(c, __fmaf_rn(w1, (float)acc[half][3], w0 * (float)acc[half][2]), Sv[half][2]);
                        } else {
                            if constexpr (MODE == INT) {                       // column 7 where t4 == 3
                                const float cz = s_czq[u];
                                col[half][0] = __fmaf_rn(cz, (float)acc[half][1], col[half][0]);
                                col[half][1] = __fmaf_rn(cz, (float)acc[half][3], col[half][1]);
                            }
#pragma unroll
                            for (int e = 0; e < 4; ++e) Sv[half][e] = __fmaf_rn(c, (float)acc[half][e], Sv[half][e]);
                        }
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[half][e] = 0;
                    }
                }
            }
        }
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if constexpr (MODE == LIMB) {
                Sv[half][0] += __shfl_xor_sync(0xffffffffu, Sv[half][0], 1);
                Sv[half][2] += __shfl_xor_sync(0xffffffffu, Sv[half][2], 1);
            }
            if constexpr (MODE == INT) {
                const float c0 = __shfl_sync(0xffffffffu, col[half][0], lane | 3), c1 = __shfl_sync(0xffffffffu, col[half][1], lane | 3);
                Sv[half][0] += c0; Sv[half][1] += c0; Sv[half][2] += c1; Sv[half][3] += c1;
            }
            const int ja = jt + 16 * half + g8, jb = ja + 8;                   // within my range
            float v0 = Sv[half][0], v1 = Sv[half][1], v2 = Sv[half][2], v3 = Sv[half][3];
            if (!all_visible) {
                v0 = j0 + ja <= vis0 && j0 + ja < j1 ? v0 : NEG_BIG; v1 = j0 + ja <= vis1 && j0 + ja < j1 ? v1 : NEG_BIG;
                v2 = j0 + jb <= vis0 && j0 + jb < j1 ? v2 : NEG_BIG; v3 = j0 + jb <= vis1 && j0 + jb < j1 ? v3 : NEG_BIG;
            }
            const bool mine0 = q0 < p.Tq && (MODE != LIMB || (t4 & 1) == 0), mine1 = MODE != LIMB && q1 < p.Tq;
            if (mine0) { S[q0 * sp.score_pitch + ja] = v0; S[q0 * sp.score_pitch + jb] = v2; m0 = fmaxf(m0, fmaxf(v0, v2)); }
            if (mine1) { S[q1 * sp.score_pitch + ja] = v1; S[q1 * sp.score_pitch + jb] = v3; m1 = fmaxf(m1, fmaxf(v1, v3)); }
        }
        __syncwarp();                                                          // the stage (and the expanded rows) may be overwritten
    }
    cp_async_wait<0>();
    __syncwarp();
    // the V tiles of the first stages travel while the maxima meet
#pragma unroll 1
    for (int i = 0; i < STAGES - 1; ++i) stage_tile(i, p.v, p.v_row_bytes, p.bits_v, uv0, nuv, pv);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
        m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    if (lane < 4) {
        if constexpr (MODE == LIMB) { if ((t4 & 1) == 0) s_wm[warp][q0] = m0; }
        else { s_wm[warp][q0] = m0; s_wm[warp][q1] = m1; }
    }
    __syncthreads();
    if (tid < MAX_Q) {
        float m = s_wm[0][tid];
#pragma unroll
        for (int w = 1; w < WARPS; ++w) m = fmaxf(m, s_wm[w][tid]);
        s_m[tid] = m;
    }
    __syncthreads();
    const int qc = MODE == LIMB ? g8 >> 2 : g8;                // the query of my column of operand B
    const bool on = qc < p.Tq;
    float mq = on ? s_m[qc] : 0.f;
    float fq = 0.f;                                            // INT: code = rne(2^(S - m) f)
    if constexpr (!KV) {
        // row sums relative to the block's maximum, then the whole cluster's maximum and sum
        for (int q = warp; q < p.Tq; q += WARPS) {
            const float m = s_m[q];
            float l = 0.f;
            for (int j = lane; j < j1 - j0; j += 32) l += ex2(S[q * sp.score_pitch + j] - m);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            if (lane == 0) s_l[q] = l;
        }
        cluster_sync();
        if (on) {
            const uint32_t am = smem_u32(s_m + g8), al = smem_u32(s_l + g8);
            float M = NEG_BIG, l = 0.f;
            for (uint32_t r = 0; r < n_ranks; ++r) M = fmaxf(M, __uint_as_float(ld_peer(am, r)));
            for (uint32_t r = 0; r < n_ranks; ++r) {
                const float mr = __uint_as_float(ld_peer(am, r));
                if (mr > 0.5f * NEG_BIG) l = __fmaf_rn(ex2(mr - M), __uint_as_float(ld_peer(al, r)), l);   // (a block that sees no key adds nothing)
            }
            mq = M;
            fq = p.inv_sP / l;
        }
    }

    // ---------------------------------------------------------------- outputs: V^T times the probabilities
    // Lane (g8, t4) reads word g8 of a pair of units (8 codes: positions 8 g8 .. 8 g8 + 7 of the 64) of keys
    // 2 t4, 2 t4 + 1, 2 t4 + 8, 2 t4 + 9 of every 16; accumulator i of the pair holds code i in row g8 and code i + 4 in row g8 + 8.
    using Acc = typename std::conditional<MODE == HALF, float, int>::type;
    Acc O[MAX_UNITS / 2][4][4];
#pragma unroll
    for (int a = 0; a < MAX_UNITS / 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int e = 0; e < 4; ++e) O[a][b][e] = (Acc)0;
    float lsum = 0.f;
    int rsum = 0;
    const int offV = (4 * p.bits_v * uv0) & 15;
    const float* Sq = S + (on ? qc : 0) * sp.score_pitch;
    const uint32_t limb_sel = MODE == LIMB ? (uint32_t)(g8 & 3) * 0x11u + 0x40u : 0u;     // byte `limb` of two words
    for (int i = 0; i < my_tiles; ++i) {
        stage_tile(i + STAGES - 1, p.v, p.v_row_bytes, p.bits_v, uv0, nuv, pv);
        // this tile's probabilities first: they do not wait for the copies
        const int jt = TILE * (warp + WARPS * i);
        uint32_t pb[2][2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const float2 x = *reinterpret_cast<const float2*>(Sq + jt + 16 * half + 2 * t4), y = *reinterpret_cast<const float2*>(Sq + jt + 16 * half + 8 + 2 * t4);
            if constexpr (MODE == LIMB) {
                // 24-bit integers: P in units of 1 / P_UNITS (the row sum counts in the same unit). The maximum is subtracted before the
                // scaling: folded into the exponent, the shift would be rounded to the maximum's own grid, and from 2^11 on P = 1 would
                // need a 25th bit
                uint32_t X[4];
                const float v[4] = {x.x, x.y, y.x, y.y};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float f = ex2(v[e] - mq) * P_UNITS;
                    lsum += f;
                    X[e] = on ? __float2uint_rn(f) : 0u;
                }
                pb[half][0] = __byte_perm(__byte_perm(X[0], X[1], limb_sel), __byte_perm(X[2], X[3], limb_sel), 0x5410);   // digit 3 is zero
                pb[half][1] = 0u;
            } else if constexpr (MODE == HALF) {
                const uint32_t w0 = on ? pack_half2(ex2(x.x - mq), ex2(x.y - mq)) : 0u, w1 = on ? pack_half2(ex2(y.x - mq), ex2(y.y - mq)) : 0u;
                const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&w0)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&w1));
                lsum += (f0.x + f0.y) + (f1.x + f1.y);         // the rounded values: the division normalises what was multiplied
                pb[half][0] = w0; pb[half][1] = w1;
            } else {
                const float v[4] = {x.x, x.y, y.x, y.y};
                uint32_t w = 0u;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int c = on ? min(__float2int_rn(ex2(v[e] - mq) * fq), 255) : 0;
                    rsum += c;
                    w |= (uint32_t)c << (8 * e);
                    if (p.p_dbg && on) {
                        const int j = j0 + jt + 16 * half + 2 * t4 + (e & 1) + 8 * (e >> 1);
                        if (j < j1) p.p_dbg[(((int64_t)blockIdx.z * p.H + h) * p.Tq + g8) * p.Tk + j] = (uint8_t)c;
                    }
                }
                pb[half][0] = w; pb[half][1] = 0u;
            }
        }
        cp_async_wait<STAGES - 1>();
        __syncwarp();
        const uint8_t* rows = ring + (i % STAGES) * sp.ring_stage + offV;
        int pitch = pv;
        if (BV == 4 && p.bits_v == 3) {
            expand_tile(rows - offV, pv, offV, nuv);
            rows = expand; pitch = nibble_pitch(nuv);
        }
#pragma unroll
        for (int a = 0; a < MAX_UNITS / 2; ++a) {
            if (2 * a < nuv) {
                // (words of a unit past the head's last one are not read: the last unit's go into rows that are never written out)
                const int word = min(8 * a + g8, 4 * nuv - 1);
                uint32_t ph[2][8];                             // INT, LIMB: [16 keys][code]: codes of four keys as bytes
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint8_t* r0 = rows + (16 * half + 2 * t4) * pitch;
                    if constexpr (BV == 4) {
                        const uint8_t* c = r0 + 4 * word;
                        const uint32_t wa = *reinterpret_cast<const uint32_t*>(c), wb = *reinterpret_cast<const uint32_t*>(c + pitch);
                        const uint32_t wc = *reinterpret_cast<const uint32_t*>(c + 8 * pitch), wd = *reinterpret_cast<const uint32_t*>(c + 9 * pitch);
                        if constexpr (MODE == HALF) {
                            // low and high halves of a pair of keys: codes (0, 4, 1, 5) and (2, 6, 3, 7) by shifting
                            const uint32_t x0 = __byte_perm(wa, wb, 0x5410), y0 = __byte_perm(wa, wb, 0x7632);
                            const uint32_t x1 = __byte_perm(wc, wd, 0x5410), y1 = __byte_perm(wc, wd, 0x7632);
                            mma_f16(O[a][0], nib_half<0>(x0), nib_half<4>(x0), nib_half<0>(x1), nib_half<4>(x1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][1], nib_half<8>(x0), nib_half<12>(x0), nib_half<8>(x1), nib_half<12>(x1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][2], nib_half<0>(y0), nib_half<4>(y0), nib_half<0>(y1), nib_half<4>(y1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][3], nib_half<8>(y0), nib_half<12>(y0), nib_half<8>(y1), nib_half<12>(y1), pb[half][0], pb[half][1]);
                        } else {
                            const uint32_t x01l = __byte_perm(wa, wb, 0x5140), x01h = __byte_perm(wa, wb, 0x7362);
                            const uint32_t x23l = __byte_perm(wc, wd, 0x5140), x23h = __byte_perm(wc, wd, 0x7362);
                            const uint32_t b[4] = {__byte_perm(x01l, x23l, 0x5410), __byte_perm(x01l, x23l, 0x7632),
                                                   __byte_perm(x01h, x23h, 0x5410), __byte_perm(x01h, x23h, 0x7632)};
#pragma unroll
                            for (int e = 0; e < 4; ++e) { ph[half][e] = b[e] & 0x0F0F0F0Fu; ph[half][e + 4] = (b[e] >> 4) & 0x0F0F0F0Fu; }
                        }
                    } else {
                        const uint8_t* c = r0 + 8 * word;
                        const uint2 wa = *reinterpret_cast<const uint2*>(c), wb = *reinterpret_cast<const uint2*>(c + pitch);
                        const uint2 wc = *reinterpret_cast<const uint2*>(c + 8 * pitch), wd = *reinterpret_cast<const uint2*>(c + 9 * pitch);
                        if constexpr (MODE == HALF) {
                            const uint32_t x0 = __byte_perm(wa.x, wb.x, 0x5410), x1 = __byte_perm(wc.x, wd.x, 0x5410);      // codes 0, 1
                            const uint32_t y0 = __byte_perm(wa.x, wb.x, 0x7632), y1 = __byte_perm(wc.x, wd.x, 0x7632);      // codes 2, 3
                            const uint32_t u0 = __byte_perm(wa.y, wb.y, 0x5410), u1 = __byte_perm(wc.y, wd.y, 0x5410);      // codes 4, 5
                            const uint32_t v0 = __byte_perm(wa.y, wb.y, 0x7632), v1 = __byte_perm(wc.y, wd.y, 0x7632);      // codes 6, 7
                            mma_f16(O[a][0], byte_half<0>(x0), byte_half<0>(u0), byte_half<0>(x1), byte_half<0>(u1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][1], byte_half<8>(x0), byte_half<8>(u0), byte_half<8>(x1), byte_half<8>(u1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][2], byte_half<0>(y0), byte_half<0>(v0), byte_half<0>(y1), byte_half<0>(v1), pb[half][0], pb[half][1]);
                            mma_f16(O[a][3], byte_half<8>(y0), byte_half<8>(v0), byte_half<8>(y1), byte_half<8>(v1), pb[half][0], pb[half][1]);
                        } else {
#pragma unroll
                            for (int w = 0; w < 2; ++w) {
                                const uint32_t A = w ? wa.y : wa.x, B = w ? wb.y : wb.x, C = w ? wc.y : wc.x, D = w ? wd.y : wd.x;
                                const uint32_t x01l = __byte_perm(A, B, 0x5140), x01h = __byte_perm(A, B, 0x7362);
                                const uint32_t x23l = __byte_perm(C, D, 0x5140), x23h = __byte_perm(C, D, 0x7362);
                                ph[half][4 * w] = __byte_perm(x01l, x23l, 0x5410); ph[half][4 * w + 1] = __byte_perm(x01l, x23l, 0x7632);
                                ph[half][4 * w + 2] = __byte_perm(x01h, x23h, 0x5410); ph[half][4 * w + 3] = __byte_perm(x01h, x23h, 0x7632);
                            }
                        }
                    }
                }
                if constexpr (MODE != HALF) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) mma_u8(O[a][e], ph[0][e], ph[0][e + 4], ph[1][e], ph[1][e + 4], pb[0][0], pb[1][0]);
                }
            }
        }
        __syncwarp();
    }
    cp_async_wait<0>();
    __syncthreads();                                           // the rings are free: they hold the partial outputs from here on

    // ---------------------------------------------------------------- the warps' and the blocks' parts meet
    uint32_t* red = reinterpret_cast<uint32_t*>(smem);         // [WARPS][Tq][32 nuv]
    const int n_pos = 32 * nuv, part = p.Tq * n_pos;
#pragma unroll
    for (int a = 0; a < MAX_UNITS / 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int q = MODE == LIMB ? t4 >> 1 : 2 * t4 + (e & 1), pos = 64 * a + 8 * g8 + b + 4 * (e >> 1);
                if constexpr (MODE == LIMB) {
                    if (e & 1) continue;
                    // the three digits' sums (each below 2^31: a block's keys are bounded) as one number, P counted in 1 / P_UNITS
                    float v = (t4 & 1) ? 65536.0f * (float)O[a][b][e] : __fmaf_rn(256.0f, (float)O[a][b][e + 1], (float)O[a][b][e]);
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    if (q < p.Tq && pos < n_pos && (t4 & 1) == 0) red[warp * part + q * n_pos + pos] = __float_as_uint(v);
                } else if (q < p.Tq && pos < n_pos) {
                    if constexpr (KV) red[warp * part + q * n_pos + pos] = __float_as_uint(O[a][b][e]);
                    else red[warp * part + q * n_pos + pos] = (uint32_t)O[a][b][e];
                }
            }
    if constexpr (KV) {
        lsum += __shfl_xor_sync(0xffffffffu, lsum, 1); lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
        if (t4 == 0 && (MODE != LIMB || (g8 & 3) == 0)) s_wl[warp][qc] = lsum;
    } else {
        rsum += __shfl_xor_sync(0xffffffffu, rsum, 1); rsum += __shfl_xor_sync(0xffffffffu, rsum, 2);
        if (t4 == 0) s_wrs[warp][g8] = rsum;
    }
    __syncthreads();
    for (int i = tid; i < part; i += THREADS) {
        if constexpr (KV) {
            float v = __uint_as_float(red[i]);
#pragma unroll
            for (int w = 1; w < WARPS; ++w) v += __uint_as_float(red[w * part + i]);
            red[i] = __float_as_uint(v);
        } else {
            uint32_t v = red[i];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) v += red[w * part + i];
            red[i] = v;
        }
    }
    if (tid < MAX_Q) {
        if constexpr (KV) { float l = 0.f; for (int w = 0; w < WARPS; ++w) l += s_wl[w][tid]; s_l[tid] = l; }
        else { int r = 0; for (int w = 0; w < WARPS; ++w) r += s_wrs[w][tid]; s_rs[tid] = r; }
    }
    cluster_sync();
    const uint32_t a_red = smem_u32(red), a_m = smem_u32(s_m), a_l = smem_u32(s_l), a_rs = smem_u32(s_rs);
    for (int i = (int)rank * THREADS + tid; i < part; i += (int)n_ranks * THREADS) {
        const int q = i / n_pos, pos = 32 * uv0 + (i - q * n_pos);
        if (__ldg(p.jidx_v + pos) < 0) continue;
        const float2 sz = __ldg(p.unit_sz_v + (pos >> 5));
        float o;
        if constexpr (KV) {
            float M = NEG_BIG, l = 0.f, acc = 0.f;
            for (uint32_t r = 0; r < n_ranks; ++r) M = fmaxf(M, __uint_as_float(ld_peer(a_m + 4 * q, r)));
            for (uint32_t r = 0; r < n_ranks; ++r) {
                const float w = ex2(__uint_as_float(ld_peer(a_m + 4 * q, r)) - M);          // 0 for a block that sees no key
                l = __fmaf_rn(w, __uint_as_float(ld_peer(a_l + 4 * q, r)), l);
                acc = __fmaf_rn(w, __uint_as_float(ld_peer(a_red + 4 * i, r)), acc);
            }
            o = sz.x * (acc * (1.0f / l) - (sz.y - (MODE == LIMB ? 0.0f : BV == 4 ? 8.0f : 128.0f)));
        } else {
            int acc = 0, rs = 0;
            for (uint32_t r = 0; r < n_ranks; ++r) {
                acc += (int)ld_peer(a_red + 4 * i, r);
                rs += (int)ld_peer(a_rs + 4 * q, r);
            }
            o = p.s_P * sz.x * (float)(acc - (int)sz.y * rs);
        }
        p.out[(q_row0 + q) * p.ldo + __ldg(p.src_v + pos)] = __float2half_rn(o);
    }
    cluster_sync();                                            // the peers have read what they need from my shared memory
}

// Blocks per (sequence, head) and keys per block. The blocks run in waves of what the SMs hold (at most four per SM
// by registers), and a block costs about as much as FIXED_KEYS keys before and after its loops (8 us + 17 us per 1000
// keys alone, 8 + 31 with four blocks per SM): of the splits whose scores fit, the one with the smallest
// waves x (keys + FIXED_KEYS). Measured, us for 1 / 2 / 4 / 8 blocks (4 bits): 576 pairs of 2011 keys 72 / 77 / 95 / 122,
// 72 pairs 44 / 25 / 19 / 25, 12 pairs 44 / 25 / 16 / 12, 576 pairs of 300 keys 20 / 27 / 45 / 82; 3 bits (three blocks
// per SM), 576 pairs of 2011 keys 131 / 109 / 125 / 173.
constexpr int FIXED_KEYS = 400;
static int keys_of_split(int Tk, int n_ranks) { return ((Tk + n_ranks - 1) / n_ranks + TILE - 1) / TILE * TILE; }
// Dynamic shared memory of a block with `keys` keys; 0 where it or the scores are more than a block may have. (The largest, eight
// units of 8 bits in one tensor and of 3 bits in the other: 104448 bytes of rings, 18432 to expand, 98304 of scores.)
static int smem_of_split(const AttnParams& p, bool half_mode, int units_k, int units_v, int keys)
{
    if ((int64_t)p.Tq * (keys + 8) * 4 > SCORE_BYTES_MAX) return 0;
    const int bytes = smem_plan(p.bits_k, p.bits_v, units_k, units_v, p.Tq, keys).total;
    return bytes <= dynamic_smem_max(half_mode) ? bytes : 0;
}
static bool half_mode_of(const AttnParams& p, bool kv) { return kv && p.Tq > LIMB_Q; }
static bool plan(const AttnParams& p, bool half_mode, int units_k, int units_v, int n_seq, int n_sm, int* n_ranks, int* keys_block, int* smem)
{
    const int64_t pairs = (int64_t)p.H * n_seq;
    int64_t best = -1;
    for (int c = 1; c <= MAX_CLUSTER; c *= 2) {
        const int keys = keys_of_split(p.Tk, c), bytes = smem_of_split(p, half_mode, units_k, units_v, keys);
        if (bytes == 0) continue;
        if (c > 1 && keys < WARPS * TILE && best >= 0) break;
        int per_sm = SM_BYTES / (bytes + static_smem(half_mode));
        per_sm = per_sm > 4 ? 4 : per_sm;
        int64_t slots = (int64_t)n_sm * per_sm;
        if (c >= 4) slots -= slots / 8;                          // clusters of this size do not fill every GPC
        const int64_t waves = (pairs * c + slots - 1) / slots;
        const int64_t cost = waves * (keys + FIXED_KEYS);
        if (best < 0 || cost < best) { best = cost; *n_ranks = c; *keys_block = keys; *smem = bytes; }
    }
    return best >= 0;
}

bool fits(const AttnParams& p, bool kv, int units_k, int units_v)
{
    // (what a block needs must fit when eight blocks share the keys)
    return p.Tq <= (kv ? MAX_Q : MAX_Q - 1) && smem_of_split(p, half_mode_of(p, kv), units_k, units_v, keys_of_split(p.Tk, MAX_CLUSTER)) > 0;
}

template <int MODE, int BK, int BV>
static int launch_one(const AttnParams& p, int units_k, int units_v, int n_seq, int dev, int n_sm, cudaStream_t st)
{
    int n_ranks = 1, keys_block = 0, smem = 0;
    if (!plan(p, MODE == HALF, units_k, units_v, n_seq, n_sm, &n_ranks, &keys_block, &smem)) return RPTQ_ERR_UNSUPPORTED;
    static SmemAllowed done;
    if (allow_smem(reinterpret_cast<const void*>(decode_kernel<MODE, BK, BV>), dev, dynamic_smem_max(MODE == HALF), done) != RPTQ_OK) return RPTQ_ERR_CUDA;
    return launch_kernel(decode_kernel<MODE, BK, BV>, dim3((unsigned)n_ranks, (unsigned)p.H, (unsigned)n_seq), THREADS, (size_t)smem, (unsigned)n_ranks, st,
                         p, keys_block, units_k, units_v);
}

int launch(const AttnParams& p, bool kv, int units_k, int units_v, int n_seq, int dev, int n_sm, cudaStream_t st)
{
    const bool k8 = p.bits_k == 8, v8 = p.bits_v == 8;
    auto pick = [&](auto mode) {
        constexpr int MODE = decltype(mode)::value;
        if (k8) return v8 ? launch_one<MODE, 8, 8>(p, units_k, units_v, n_seq, dev, n_sm, st) : launch_one<MODE, 8, 4>(p, units_k, units_v, n_seq, dev, n_sm, st);
        return v8 ? launch_one<MODE, 4, 8>(p, units_k, units_v, n_seq, dev, n_sm, st) : launch_one<MODE, 4, 4>(p, units_k, units_v, n_seq, dev, n_sm, st);
    };
    if (!kv) return pick(std::integral_constant<int, INT>());
    return half_mode_of(p, true) ? pick(std::integral_constant<int, HALF>()) : pick(std::integral_constant<int, LIMB>());
}

}  // namespace attn_decode
}  // namespace rptq
