// Attention for more queries than a decode step has: rptq_attention and rptq_attention_kv on the tcgen05 tensor cores.
//
// A persistent block works on 128 queries of one head at a time. The softmax output is needed with the row's final maximum
// (and, where it is quantised at 8 bits, its final sum), so the keys are walked twice: pass 1 finds the row maxima
// (integer calls: and the row sums), pass 2 forms the probabilities and multiplies them with V. Nothing is
// rescaled on the way. Scores are computed in both passes; the tensor cores have room for that.
//
// What bounds it: one exponential per score and pass (the special-function unit gives 16 per clock and SM), then the
// issue slots of the softmax warps: a score costs one multiply-add per cluster of the head, and five or six
// instructions more. So everything else is kept off those warps:
//   warp 0        issues the MMAs: per key tile, one accumulator per CLUSTER of the head (the scales differ), handed over
//                 slot by slot through a ring in tensor memory; then, in pass 2, P V of the previous tile into the
//                 head's output accumulator, which stays in tensor memory over the whole pass
//   warps 4-7     keys: packed rows arrive by cp.async one tile ahead, are unpacked into the swizzled operand tile; integer
//                 calls: with the per-key zero-point term -sum_c s^Q s^K z^Q sum_p K_q. They also lay out the queries.
//   warps 8-11    values: unpacked and transposed into [position][key] (byte permutes on the packed words)
//   warps 12-19   softmax: thread = (query row, half of the tile's keys); S = sum_c coef_c acc_c in registers
// Operand types (MODE):
//   I8   bytes, kind::i8, int32 sums
//   F8   both codes of at most four bits: a nibble n as an 8-bit E4M3 pattern IS the number n 2^-9, so the same bytes
//        multiply as kind::f8f6f4 and the sums (below 2^16 units) come out as exact fp32: no conversion per score and
//        cluster
//   KV   fp16 query; codes as fp16 integers n - 8 (n - 128): the centre is a constant per row in the scores and part of the
//        zero point in the outputs
// P V is u8 x u8 -> s32 for I8 and F8 (exact), fp16 x fp16 -> fp32 for KV.
// Key order inside a tile of the second product (both operands are written in it, so the sums do not change):
// KEYS = 128: byte b of word w is key w + 32 b; KV, 64 keys: see v_tile. It lets the V loader read and
// write shared memory without bank conflicts.
//
// Measured: MEASURED_PREFILL
#include <type_traits>

#include "attn_common.cuh"
#include "pack.cuh"
#include "tc.cuh"

namespace rptq {
namespace attn_prefill {

using namespace attn;
using tc::mbar_arrive;
using tc::mbar_init;
using tc::mbar_wait;
using tc::mbar_wait_warp;

enum { I8 = 0, F8 = 1, KV = 2 };
constexpr int BM = 128, THREADS = 640;
constexpr int K_WARP0 = 4, V_WARP0 = 8, S_WARP0 = 12;
// registers per thread of the five warpgroups (the block is launched with 96 each)
constexpr int REGS_MMA = 48, REGS_LOAD = 72, REGS_SOFTMAX = 144;
static_assert(REGS_MMA + 2 * REGS_LOAD + 2 * REGS_SOFTMAX <= 5 * 96, "register pool");
constexpr int O_COLS = 32 * MAX_UNITS;                    // tensor memory: the output accumulator, then the score slots
constexpr int ATOM_Q = BM * 128;                          // 128 rows of 128 bytes

__host__ __device__ constexpr int keys_of(int mode) { return mode == KV ? 64 : 128; }

// Shared memory of a launch (sizes follow the widest head of the layouts).
struct Plan {
    int n_items, n_qt, n_seq;
    int off_k, k_stage, off_v, v_stage, v_stages, off_p, off_rawk, pitch_k, off_rawv, pitch_v, off_col, off_x, off_bar, total;
    int local_v;          // V's heads own their channels and the output tile fits the V region: rows leave through shared memory
    int out_pitch;
    int* status;
};

// Row pitch of a staged packed tile: an odd number of 16-byte chunks, so that eight rows read at one column lie in
// different banks.
static int raw_pitch_of(int bits, int units)
{
    const int c = (4 * bits * units + 15) / 16 + (bits == 3 ? 1 : 0);
    return 16 * (c | 1);
}

__device__ __forceinline__ void ld8(uint32_t taddr, uint32_t* v)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)), "l"(reinterpret_cast<uint64_t&>(c)));
    return d;
}
// The whole warp executes these in converged control flow; one elected lane issues.
template <int KIND>       // 0 i8, 1 f8f6f4, 2 f16
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    if constexpr (KIND == 0)
        asm volatile("{\n\t.reg .pred p, q;\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
    else if constexpr (KIND == 1)
        asm volatile("{\n\t.reg .pred p, q;\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
    else
        asm volatile("{\n\t.reg .pred p, q;\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar)
{
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}
// The nibbles (bytes) at bit B of the two halves of w as fp16 numbers n - 8 (n - 128).
template <int B>
__device__ __forceinline__ uint32_t nib_half(uint32_t w)
{
    const uint32_t t = ((B <= 6 ? w << (6 - B) : w >> (B - 6)) & 0x03C003C0u) | 0x4C004C00u;      // 16 + n
    const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&t), __float2half2_rn(-24.0f));
    return *reinterpret_cast<const uint32_t*>(&r);
}
template <int B>
__device__ __forceinline__ uint32_t byte_half(uint32_t w)
{
    const uint32_t t = ((w >> B) & 0x00FF00FFu) | 0x64006400u;                                    // 1024 + n
    const __half2 r = __hadd2(*reinterpret_cast<const __half2*>(&t), __float2half2_rn(-1152.0f));
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t a) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory"); }
__device__ __forceinline__ void sts16(uint32_t addr, uint16_t a) { asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(a) : "memory"); }
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint16_t lds16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.b16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}
// Unit u of a staged packed row of 3- or 4-bit codes as nibble words (the 4-bit format).
__device__ __forceinline__ uint4 nibbles(uint32_t row, int u, int bits)
{
    if (bits == 4) return lds128(row + 16 * u);
    const uint32_t a = lds32(row + 12 * u), b = lds32(row + 12 * u + 4), c = lds32(row + 12 * u + 8);
    const uint32_t tail = ((a >> 3) & 0x11111111u) | ((b >> 2) & 0x22222222u) | ((c >> 1) & 0x44444444u);
    return make_uint4(a & 0x77777777u, b & 0x77777777u, c & 0x77777777u, tail);
}

// Units of a head in K's (and Q's) layout as the kernel sees them: a head without channels has one unit of zeros, so that its
// scores are zero like any others.
__device__ __forceinline__ int units_seen(int nu) { return nu > 0 ? nu : 1; }

// One block's walk over its work: item = (query tile, head, sequence), the tiles with the most visible keys first.
struct Item { int qt, h, seq, n_kt; };
__device__ __forceinline__ Item item_of(const AttnParams& p, const Plan& g, int idx, int keys)
{
    Item it;
    const int per = p.H * g.n_seq, q = idx / per, r = idx - q * per;
    it.qt = g.n_qt - 1 - q;
    it.seq = r / p.H;
    it.h = r - it.seq * p.H;
    const int last = p.causal ? min(p.Tk - 1, it.qt * BM + BM - 1 + p.Tk - p.Tq) : p.Tk - 1;
    it.n_kt = last / keys + 1;
    return it;
}

template <int MODE>
__global__ void __launch_bounds__(THREADS, 1)
prefill_kernel(const AttnParams p, const Plan g)
{
    constexpr int KEYS = keys_of(MODE), N_SLOTS = (512 - O_COLS) / KEYS;
    constexpr int K_ATOM = KEYS * 128;                    // operand tile of the keys: KEYS rows of 128 bytes per atom
    constexpr int UNITS_PER_ATOM = MODE == KV ? 2 : 4;    // 64 bytes (fp16) or 32 bytes per unit
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - smem_u32(smem_raw));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + g.off_bar);
    constexpr int B_QFULL = 0, B_QEMPTY = 1, B_KFULL = 2, B_KEMPTY = 4, B_SFULL = 6, B_SEMPTY = B_SFULL + N_SLOTS, B_PFULL = B_SEMPTY + N_SLOTS,
                  B_PEMPTY = B_PFULL + 1, B_VFULL = B_PEMPTY + 1, B_VEMPTY = B_VFULL + 2, B_OFULL = B_VEMPTY + 2, B_OEMPTY = B_OFULL + 1,
                  B_OUT = B_OEMPTY + 1, B_XS = B_OUT + 1, B_XV = B_XS + 1, B_DRAIN = B_XV + 1, N_BARS = B_DRAIN + 1;
    static_assert(N_BARS * 8 + 16 <= 256, "barrier block");
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + N_BARS);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        mbar_init(bar(B_QFULL), 4); mbar_init(bar(B_QEMPTY), 1);
        for (int i = 0; i < 2; ++i) { mbar_init(bar(B_KFULL + i), 4); mbar_init(bar(B_KEMPTY + i), 1); mbar_init(bar(B_VFULL + i), 4); mbar_init(bar(B_VEMPTY + i), 1); }
        for (int i = 0; i < N_SLOTS; ++i) { mbar_init(bar(B_SFULL + i), 1); mbar_init(bar(B_SEMPTY + i), 8); }
        mbar_init(bar(B_PFULL), 8); mbar_init(bar(B_PEMPTY), 1);
        mbar_init(bar(B_OFULL), 1); mbar_init(bar(B_OEMPTY), 8); mbar_init(bar(B_OUT), 8);
        mbar_init(bar(B_XS), 8); mbar_init(bar(B_XV), 4); mbar_init(bar(B_DRAIN), 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *s_tmem;
    const int off = p.Tk - p.Tq;
    float* s_col = reinterpret_cast<float*>(smem + g.off_col);            // [4][KEYS]
    float2* s_x = reinterpret_cast<float2*>(smem + g.off_x);              // [2][2][BM]: the halves' row statistics

    if (warp < K_WARP0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_MMA));
        if (warp == 0) {
            // ------------------------------------------------------------ MMA issuer
            constexpr uint32_t FMT = MODE == I8 ? (2u << 4) : (1u << 4);                          // D: s32 or f32; A, B: u8 / E4M3 / f16
            constexpr uint32_t ID_QK = FMT | ((uint32_t)(KEYS >> 3) << 17) | (8u << 24);
            constexpr uint32_t ID_PV = (MODE == KV ? (1u << 4) : (2u << 4)) | (8u << 24);
            const uint64_t dq = tc::smem_desc_sw128(base), dk = tc::smem_desc_sw128(base + g.off_k), dv = tc::smem_desc_sw128(base + g.off_v),
                           dp = tc::smem_desc_sw128(base + g.off_p);
            uint32_t n_k = 0, n_s = 0, n_v = 0, n_item = 0;
            bool ok = true;
            for (int idx = blockIdx.x; idx < g.n_items && ok; idx += gridDim.x, ++n_item) {
                const Item it = item_of(p, g, idx, KEYS);
                const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0;
                const int nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - __ldg(p.cl_unit0_v + it.h * p.gh_v);
                // bit u: unit u is the last of its cluster
                const int cl = lane < nuk ? __ldg(p.unit_cluster_k + uk0 + lane) : -1;
                const int cl_next = __shfl_down_sync(0xffffffffu, cl, 1);
                const uint32_t last = __ballot_sync(0xffffffffu, lane < units_seen(nuk) && (lane >= nuk - 1 || cl != cl_next));
                const uint32_t id_pv = ID_PV | ((uint32_t)(4 * nuv) << 17);
                if (!mbar_wait_warp(bar(B_QFULL), n_item & 1, s_abort)) { ok = false; break; }
                auto scores = [&]() {
                    const uint32_t st = n_k & 1;
                    if (!mbar_wait_warp(bar(B_KFULL + st), (n_k >> 1) & 1, s_abort)) return false;
                    tc::tc_fence_after();
                    const uint64_t kb = dk + (uint64_t)(st * (uint32_t)(g.k_stage >> 4));
                    bool first = true;
#pragma unroll 1
                    for (int u = 0; u < units_seen(nuk); ++u) {
                        const uint32_t slot = n_s % N_SLOTS, d = tmem + O_COLS + slot * KEYS;
                        if (first) {
                            if (!mbar_wait_warp(bar(B_SEMPTY + slot), ((n_s / N_SLOTS) & 1) ^ 1, s_abort)) return false;
                            tc::tc_fence_after();
                        }
                        const uint32_t atom = (uint32_t)u / UNITS_PER_ATOM, in = (uint32_t)u % UNITS_PER_ATOM;
                        const uint64_t a = dq + (uint64_t)(atom * (ATOM_Q >> 4)), b = kb + (uint64_t)(atom * (K_ATOM >> 4));
                        if constexpr (MODE == KV) {
                            mma<2>(d, a + 4 * in, b + 4 * in, ID_QK, first ? 0u : 1u);
                            mma<2>(d, a + 4 * in + 2, b + 4 * in + 2, ID_QK, 1u);
                        } else {
                            mma<MODE == F8 ? 1 : 0>(d, a + 2 * in, b + 2 * in, ID_QK, first ? 0u : 1u);
                        }
                        first = false;
                        if ((last >> u) & 1u) { commit(bar(B_SFULL + slot)); ++n_s; first = true; }
                    }
                    commit(bar(B_KEMPTY + st));
                    ++n_k;
                    return true;
                };
                auto outputs = [&](bool first) {
                    const uint32_t st = g.v_stages == 2 ? n_v & 1 : 0u, ph = g.v_stages == 2 ? (n_v >> 1) & 1 : n_v & 1;
                    if (!mbar_wait_warp(bar(B_VFULL + st), ph, s_abort)) return false;
                    if (!mbar_wait_warp(bar(B_PFULL), n_v & 1, s_abort)) return false;
                    tc::tc_fence_after();
                    const uint64_t b = dv + (uint64_t)(st * (uint32_t)(g.v_stage >> 4));
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (nuv > 0) mma<MODE == KV ? 2 : 0>(tmem, dp + 2 * k, b + 2 * k, id_pv, (first && k == 0) ? 0u : 1u);
                    commit(bar(B_PEMPTY));
                    commit(bar(B_VEMPTY + st));
                    ++n_v;
                    return true;
                };
                for (int kt = 0; kt < it.n_kt && ok; ++kt) ok = scores();
                for (int kt = 0; kt < it.n_kt && ok; ++kt) {
                    ok = scores();
                    if (!ok) break;
                    if (kt == it.n_kt - 1) commit(bar(B_QEMPTY));              // the item's last score product has been issued
                    if (kt == 1) {                                             // the item's first output product comes next
                        ok = mbar_wait_warp(bar(B_OEMPTY), (n_item & 1) ^ 1, s_abort);
                        tc::tc_fence_after();
                    }
                    if (kt > 0 && ok) ok = outputs(kt == 1);
                }
                if (ok && it.n_kt == 1) { ok = mbar_wait_warp(bar(B_OEMPTY), (n_item & 1) ^ 1, s_abort); tc::tc_fence_after(); }
                if (ok) ok = outputs(it.n_kt == 1);
                if (ok) commit(bar(B_OFULL));
            }
            if (!ok) {
                commit(bar(B_DRAIN));
                mbar_wait(bar(B_DRAIN), 0, s_abort, false);
            }
        }
    } else if (warp < V_WARP0) {
        // ---------------------------------------------------------------- keys (and queries)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LOAD));
        const int kw = warp - K_WARP0, kt_id = tid - 32 * K_WARP0;             // 0..3, 0..127
        constexpr int ROWS_W = KEYS / 4;                                       // key rows that a warp copies and unpacks
        const bool direct = MODE != KV && p.bits_k == 8;                       // bytes already: copied straight into the operand tile
        // copies of a tile's packed rows (eight lanes per row), into the raw buffer or, swizzled, into operand stage st
        auto copy_rows = [&](const Item& it, int kt, uint32_t st) {
            const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0;
            const int win = (4 * p.bits_k * uk0) & ~15, n16 = ((4 * p.bits_k * uk0 - win) + 4 * p.bits_k * nuk + 15) >> 4;
            const int r0 = lane >> 3, c0 = lane & 7;
#pragma unroll 2
            for (int i = 0; i < ROWS_W / 4; ++i) {
                const int r = ROWS_W * kw + 4 * i + r0, j = kt * KEYS + r;
                const bool okr = j < p.Tk;
                const uint8_t* src = p.k + ((int64_t)it.seq * p.Tk + (okr ? j : 0)) * p.k_row_bytes + win;
                for (int c = c0; c < n16; c += 8) {
                    const uint32_t dst = direct ? base + g.off_k + st * g.k_stage + (c >> 3) * K_ATOM + r * 128 + (((c & 7) ^ (r & 7)) << 4)
                                                : base + g.off_rawk + r * g.pitch_k + 16 * c;
                    cp_async16(dst, src + 16 * c, okr ? 16 : 0);
                }
            }
        };
        uint32_t n_k = 0, n_item = 0;
        bool ok = true;
        int idx = blockIdx.x;
        if (idx < g.n_items) copy_rows(item_of(p, g, idx, KEYS), 0, 0u);       // (stage 0 is free at the start)
        cp_async_commit();
        for (; idx < g.n_items && ok; idx += gridDim.x, ++n_item) {
            const Item it = item_of(p, g, idx, KEYS);
            const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0;
            const int off_b = (4 * p.bits_k * uk0) & 15;
            // ---- the item's queries
            if (!mbar_wait(bar(B_QEMPTY), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
            const int i0 = it.qt * BM;
            if constexpr (MODE == KV) {
                // a lane takes up to four pairs of positions (operand order: codes 0, 2, 1, 3, 4, 6, 5, 7 of every eight, the order
                // in which the key codes come out of their words) and gathers their channels row by row
                int ca[4], cb[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int p2 = lane + 32 * k, code = (p2 >> 2) * 8 + (p2 & 1) + 4 * ((p2 >> 1) & 1), pos = 32 * uk0 + code;
                    const bool in = p2 < 16 * nuk;            // (a head without channels: no pair is, zeros are written)
                    ca[k] = in && __ldg(p.jidx_k + pos) >= 0 ? (int)__ldg(p.src_k + pos) : -1;
                    cb[k] = in && __ldg(p.jidx_k + pos + 2) >= 0 ? (int)__ldg(p.src_k + pos + 2) : -1;
                }
#pragma unroll 2
                for (int r = kw; r < BM; r += 4) {
                    const bool okr = i0 + r < p.Tq;
                    const __half* row = p.q_f16 + ((int64_t)it.seq * p.Tq + (okr ? i0 + r : 0)) * p.ldq;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int p2 = lane + 32 * k;
                        if (p2 < 16 * units_seen(nuk)) {
                            const uint32_t lo = okr && ca[k] >= 0 ? (uint32_t)__half_as_ushort(row[ca[k]]) : 0u;
                            const uint32_t hi = okr && cb[k] >= 0 ? (uint32_t)__half_as_ushort(row[cb[k]]) : 0u;
                            sts32(base + k * ATOM_Q + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + 4 * (lane & 3), lo | (hi << 16));
                        }
                    }
                }
            } else {
#pragma unroll 2
                for (int i = kt_id; i < BM * units_seen(nuk); i += 128) {
                    const int r = i / units_seen(nuk), u = i - r * units_seen(nuk);
                    uint32_t o[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                    if (u < nuk && i0 + r < p.Tq) load_unit(p.q + ((int64_t)it.seq * p.Tq + i0 + r) * p.q_row_bytes, uk0 + u, p.bits_q, o);
                    const uint32_t d = base + (u >> 2) * ATOM_Q + r * 128, c = 2 * (u & 3), sw = r & 7;
                    sts128(d + ((c ^ sw) << 4), o[0], o[1], o[2], o[3]);
                    sts128(d + (((c + 1) ^ sw) << 4), o[4], o[5], o[6], o[7]);
                }
            }
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_QFULL));
            // integer calls: -s^Q s^K z^Q qk_scale log2(e) of unit `lane`
            float czq = 0.f;
            if constexpr (MODE != KV) {
                if (lane < nuk) {
                    const float2 q = __ldg(p.unit_sz_q + uk0 + lane), k = __ldg(p.unit_sz_k + uk0 + lane);
                    czq = -(q.x * k.x * p.qk_scale_log2e) * q.y;
                }
            }
            // ---- the key tiles, twice
            const int n_tiles = 2 * it.n_kt;
#pragma unroll 1
            for (int t = 0; t < n_tiles; ++t, ++n_k) {
                const uint32_t st = n_k & 1;
                const uint32_t tile = base + g.off_k + st * g.k_stage;
                // the copies of the tile after this one (of the next item after the last)
                auto copy_next = [&]() {
                    if (t + 1 < n_tiles) copy_rows(it, t + 1 < it.n_kt ? t + 1 : t + 1 - it.n_kt, st ^ 1u);
                    else if (idx + (int)gridDim.x < g.n_items) copy_rows(item_of(p, g, idx + gridDim.x, KEYS), 0, st ^ 1u);
                    cp_async_commit();
                };
                if constexpr (MODE == KV) {
                    // thread = (row, parity of the unit): up to four units, as nibble words or bytes
                    const int r = kt_id >> 1, odd = kt_id & 1;
                    const uint32_t raw = base + g.off_rawk + r * g.pitch_k + off_b;
                    uint4 w[4][2];
                    cp_async_wait<0>();
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int u = 2 * i + odd;
                        w[i][0] = w[i][1] = make_uint4(0u, 0u, 0u, 0u);
                        if (u < nuk) {
                            if (p.bits_k == 8) { w[i][0] = lds128(raw + 32 * u); w[i][1] = lds128(raw + 32 * u + 16); }
                            else w[i][0] = nibbles(raw, u, p.bits_k);
                        }
                    }
                    __syncwarp();
                    copy_next();
                    if (!mbar_wait(bar(B_KEMPTY + st), ((n_k >> 1) & 1) ^ 1, s_abort)) { ok = false; break; }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (2 * i + odd < units_seen(nuk)) {
                            const uint32_t d = tile + i * K_ATOM + r * 128, sw = r & 7;
                            const uint32_t a[8] = {w[i][0].x, w[i][0].y, w[i][0].z, w[i][0].w, w[i][1].x, w[i][1].y, w[i][1].z, w[i][1].w};
#pragma unroll
                            for (int c = 0; c < 4; ++c) {                          // eight codes = one chunk
                                const uint32_t at = d + (((4 * odd + c) ^ sw) << 4);
                                if (p.bits_k == 8) sts128(at, byte_half<0>(a[2 * c]), byte_half<8>(a[2 * c]), byte_half<0>(a[2 * c + 1]), byte_half<8>(a[2 * c + 1]));
                                else sts128(at, nib_half<0>(a[c]), nib_half<8>(a[c]), nib_half<4>(a[c]), nib_half<12>(a[c]));
                            }
                        }
                    }
                } else {
                    const int r = kt_id, sw = r & 7;
                    float col = 0.f;
                    if (direct) {
                        // the next tile's copies go into the other stage: its products must have read it
                        const bool more = t + 1 < n_tiles || idx + (int)gridDim.x < g.n_items;
                        if (more && !mbar_wait(bar(B_KEMPTY + (st ^ 1u)), (((n_k + 1) >> 1) & 1) ^ 1, s_abort)) { ok = false; break; }
                        copy_next();
                        cp_async_wait<1>();
                        __syncwarp();
#pragma unroll 1
                        for (int u = 0; u < nuk; ++u) {
                            const uint32_t d = tile + (u >> 2) * K_ATOM + r * 128, c = 2 * (u & 3);
                            const uint4 a = lds128(d + ((c ^ sw) << 4)), b = lds128(d + (((c + 1) ^ sw) << 4));
                            unsigned s = __dp4a(a.x, 0x01010101u, 0u);
                            s = __dp4a(a.y, 0x01010101u, s); s = __dp4a(a.z, 0x01010101u, s); s = __dp4a(a.w, 0x01010101u, s);
                            s = __dp4a(b.x, 0x01010101u, s); s = __dp4a(b.y, 0x01010101u, s); s = __dp4a(b.z, 0x01010101u, s); s = __dp4a(b.w, 0x01010101u, s);
                            col = __fmaf_rn(__shfl_sync(0xffffffffu, czq, u), (float)s, col);
                        }
                    } else {
                        const uint32_t raw = base + g.off_rawk + r * g.pitch_k + off_b;
                        uint4 w[MAX_UNITS];
                        cp_async_wait<0>();
                        __syncwarp();
#pragma unroll
                        for (int u = 0; u < MAX_UNITS; ++u) w[u] = u < nuk ? nibbles(raw, u, p.bits_k) : make_uint4(0u, 0u, 0u, 0u);
                        __syncwarp();
                        copy_next();
                        if (!mbar_wait(bar(B_KEMPTY + st), ((n_k >> 1) & 1) ^ 1, s_abort)) { ok = false; break; }
#pragma unroll
                        for (int u = 0; u < MAX_UNITS; ++u) {
                            if (u < units_seen(nuk)) {
                                const uint32_t d = tile + (u >> 2) * K_ATOM + r * 128, c = 2 * (u & 3);
                                const uint32_t o[8] = {w[u].x & 0x0F0F0F0Fu, (w[u].x >> 4) & 0x0F0F0F0Fu, w[u].y & 0x0F0F0F0Fu, (w[u].y >> 4) & 0x0F0F0F0Fu,
                                                       w[u].z & 0x0F0F0F0Fu, (w[u].z >> 4) & 0x0F0F0F0Fu, w[u].w & 0x0F0F0F0Fu, (w[u].w >> 4) & 0x0F0F0F0Fu};
                                sts128(d + ((c ^ sw) << 4), o[0], o[1], o[2], o[3]);
                                sts128(d + (((c + 1) ^ sw) << 4), o[4], o[5], o[6], o[7]);
                                unsigned s = 0u;
#pragma unroll
                                for (int e = 0; e < 8; ++e) s = __dp4a(o[e], 0x01010101u, s);
                                col = __fmaf_rn(__shfl_sync(0xffffffffu, czq, u), (float)s, col);
                            }
                        }
                    }
                    s_col[(n_k & 3) * KEYS + r] = col;
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_KFULL + st));
            }
        }
        cp_async_wait<0>();
    } else if (warp < S_WARP0) {
        // ---------------------------------------------------------------- values
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LOAD));
        const int vw = warp - V_WARP0;
        constexpr int ROWS_W = KEYS / 4;
        auto copy_rows = [&](const Item& it, int kt) {
            const int uv0 = __ldg(p.cl_unit0_v + it.h * p.gh_v), nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - uv0;
            const int win = (4 * p.bits_v * uv0) & ~15, n16 = ((4 * p.bits_v * uv0 - win) + 4 * p.bits_v * nuv + 15) >> 4;
            const int r0 = lane >> 3, c0 = lane & 7;
#pragma unroll 2
            for (int i = 0; i < ROWS_W / 4; ++i) {
                const int r = ROWS_W * vw + 4 * i + r0, j = kt * KEYS + r;
                const bool okr = j < p.Tk;
                const uint8_t* src = p.v + ((int64_t)it.seq * p.Tk + (okr ? j : 0)) * p.v_row_bytes + win;
                for (int c = c0; c < n16; c += 8) cp_async16(base + g.off_rawv + r * g.pitch_v + 16 * c, src + 16 * c, okr ? 16 : 0);
            }
        };
        uint32_t n_v = 0, n_x = 0, n_item = 0;
        bool ok = true;
        // all four warps have passed this point (bounded, unlike a named barrier)
        auto group_sync = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_XV));
            const bool done = mbar_wait(bar(B_XV), n_x & 1, s_abort);
            ++n_x;
            return done;
        };
        int idx = blockIdx.x;
        if (idx < g.n_items) copy_rows(item_of(p, g, idx, KEYS), 0);
        cp_async_commit();
        for (; idx < g.n_items && ok; idx += gridDim.x, ++n_item) {
            const Item it = item_of(p, g, idx, KEYS);
            const int uv0 = __ldg(p.cl_unit0_v + it.h * p.gh_v), nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - uv0;
            const int off_b = (4 * p.bits_v * uv0) & 15;
            // the previous item's output rows have left the region
            if (!mbar_wait(bar(B_OUT), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
#pragma unroll 1
            for (int kt = 0; kt < it.n_kt; ++kt, ++n_v) {
                const uint32_t st = g.v_stages == 2 ? n_v & 1 : 0u, ph = g.v_stages == 2 ? (n_v >> 1) & 1 : n_v & 1;
                cp_async_wait<0>();
                if (!group_sync()) { ok = false; break; }                      // everyone's copies of the tile have landed
                if (!mbar_wait(bar(B_VEMPTY + st), ph ^ 1, s_abort)) { ok = false; break; }
                const uint32_t tile = base + g.off_v + st * g.v_stage, raw = base + g.off_rawv + off_b;
                if constexpr (MODE == KV) {
                    // lane = (chunk c8 = 4 hf + v of the 64 slots, word j of the unit): keys 16 a + 8 hf + 2 v + {0, 1}, a = 0..3
                    const int c8 = lane & 7, j = lane >> 3, key0 = 8 * (c8 >> 2) + 2 * (c8 & 3);
#pragma unroll 1
                    for (int u = vw; u < nuv; u += 4) {
                        uint32_t lo[8], hi[8];                                 // my eight codes of the eight keys (hi: bytes 4..7 of 8-bit codes)
#pragma unroll
                        for (int a = 0; a < 8; ++a) {
                            const uint32_t row = raw + (16 * (a >> 1) + key0 + (a & 1)) * g.pitch_v;
                            hi[a] = 0u;
                            if (p.bits_v == 8) { lo[a] = lds32(row + 32 * u + 8 * j); hi[a] = lds32(row + 32 * u + 8 * j + 4); }
                            else if (p.bits_v == 4) lo[a] = lds32(row + 16 * u + 4 * j);
                            else {
                                const uint32_t x = lds32(row + 12 * u), y = lds32(row + 12 * u + 4), z = lds32(row + 12 * u + 8);
                                const uint32_t tail = ((x >> 3) & 0x11111111u) | ((y >> 2) & 0x22222222u) | ((z >> 1) & 0x44444444u);
                                lo[a] = j == 3 ? tail : (j == 0 ? x : j == 1 ? y : z) & 0x77777777u;
                            }
                        }
                        const uint32_t d = tile + (32 * u + 8 * j) * 128;
                        // codes e and e + 4 (nibbles) or e (bytes) of the four key pairs = one chunk of position row 8 j + e; row & 7 = e
                        auto put = [&](int e, const uint32_t (&h4)[4]) { sts128(d + e * 128 + ((c8 ^ e) << 4), h4[0], h4[1], h4[2], h4[3]); };
                        if (p.bits_v == 8) {
#pragma unroll
                            for (int half = 0; half < 4; ++half) {             // codes 2 half, 2 half + 1
                                uint32_t x[4], h0[4], h1[4];
#pragma unroll
                                for (int a = 0; a < 4; ++a) {
                                    const uint32_t p0 = half < 2 ? lo[2 * a] : hi[2 * a], p1 = half < 2 ? lo[2 * a + 1] : hi[2 * a + 1];
                                    x[a] = __byte_perm(p0, p1, (half & 1) ? 0x7632 : 0x5410);
                                    h0[a] = byte_half<0>(x[a]); h1[a] = byte_half<8>(x[a]);
                                }
                                put(2 * half, h0); put(2 * half + 1, h1);
                            }
                        } else {
#pragma unroll
                            for (int half = 0; half < 2; ++half) {             // codes 2 half, 2 half + 1 and those + 4
                                uint32_t x[4], h0[4], h1[4], h4[4], h5[4];
#pragma unroll
                                for (int a = 0; a < 4; ++a) {
                                    x[a] = __byte_perm(lo[2 * a], lo[2 * a + 1], half ? 0x7632 : 0x5410);
                                    h0[a] = nib_half<0>(x[a]); h4[a] = nib_half<4>(x[a]); h1[a] = nib_half<8>(x[a]); h5[a] = nib_half<12>(x[a]);
                                }
                                put(2 * half, h0); put(2 * half + 1, h1); put(2 * half + 4, h4); put(2 * half + 5, h5);
                            }
                        }
                    }
                } else {
                    // lane w: keys w, w + 32, w + 64, w + 96 of unit u; word w of the 32 positions' rows
                    const uint32_t wc = (uint32_t)lane >> 2, wo = 4 * ((uint32_t)lane & 3);
#pragma unroll 1
                    for (int u = vw; u < nuv; u += 4) {
                        const uint32_t d = tile + 32 * u * 128 + wo;
                        auto put = [&](int pos, uint32_t x) { sts32(d + pos * 128 + ((wc ^ (pos & 7)) << 4), x); };
                        // 4 x 4 byte transpose: out[i] = byte i of the four rows
                        auto transpose = [](uint32_t a, uint32_t b, uint32_t c, uint32_t e, uint32_t (&out)[4]) {
                            const uint32_t x01l = __byte_perm(a, b, 0x5140), x01h = __byte_perm(a, b, 0x7362);
                            const uint32_t x23l = __byte_perm(c, e, 0x5140), x23h = __byte_perm(c, e, 0x7362);
                            out[0] = __byte_perm(x01l, x23l, 0x5410); out[1] = __byte_perm(x01l, x23l, 0x7632);
                            out[2] = __byte_perm(x01h, x23h, 0x5410); out[3] = __byte_perm(x01h, x23h, 0x7632);
                        };
                        if (p.bits_v == 8) {
#pragma unroll
                            for (int half = 0; half < 2; ++half) {
                                uint4 rw[4];
#pragma unroll
                                for (int b = 0; b < 4; ++b) rw[b] = lds128(raw + (lane + 32 * b) * g.pitch_v + 32 * u + 16 * half);
                                const uint32_t a[4][4] = {{rw[0].x, rw[0].y, rw[0].z, rw[0].w}, {rw[1].x, rw[1].y, rw[1].z, rw[1].w},
                                                          {rw[2].x, rw[2].y, rw[2].z, rw[2].w}, {rw[3].x, rw[3].y, rw[3].z, rw[3].w}};
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    uint32_t o[4];
                                    transpose(a[0][k], a[1][k], a[2][k], a[3][k], o);
#pragma unroll
                                    for (int i = 0; i < 4; ++i) put(16 * half + 4 * k + i, o[i]);
                                }
                            }
                        } else {
                            uint4 rw[4];
#pragma unroll
                            for (int b = 0; b < 4; ++b) rw[b] = nibbles(raw + (lane + 32 * b) * g.pitch_v, u, p.bits_v);
                            const uint32_t a[4][4] = {{rw[0].x, rw[0].y, rw[0].z, rw[0].w}, {rw[1].x, rw[1].y, rw[1].z, rw[1].w},
                                                      {rw[2].x, rw[2].y, rw[2].z, rw[2].w}, {rw[3].x, rw[3].y, rw[3].z, rw[3].w}};
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                uint32_t o[4];
                                transpose(a[0][k], a[1][k], a[2][k], a[3][k], o);
#pragma unroll
                                for (int i = 0; i < 4; ++i) { put(8 * k + i, o[i] & 0x0F0F0F0Fu); put(8 * k + 4 + i, (o[i] >> 4) & 0x0F0F0F0Fu); }
                            }
                        }
                    }
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_VFULL + st));
                if (!group_sync()) { ok = false; break; }                      // the raw rows have been read
                if (kt + 1 < it.n_kt) copy_rows(it, kt + 1);
                else if (idx + (int)gridDim.x < g.n_items) copy_rows(item_of(p, g, idx + gridDim.x, KEYS), 0);
                cp_async_commit();
            }
        }
        cp_async_wait<0>();
    } else {
        // ---------------------------------------------------------------- softmax
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
        const int sw_ = warp - S_WARP0, q4 = sw_ & 3, hf = sw_ >> 2;           // lane quarter of the accumulators, half of the keys
        const int row = 32 * q4 + lane;                                        // query row within the tile
        constexpr int RUN = KEYS / 8;                                          // my keys: KEYS / 4 * b + RUN * hf + 0 .. RUN - 1, b = 0..3
        const uint32_t t_lane = tmem + ((uint32_t)(32 * q4) << 16);
        uint32_t n_k = 0, n_s = 0, n_p = 0, n_x = 0, n_item = 0;
        bool ok = true;
        auto group_sync = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_XS));
            const bool done = mbar_wait(bar(B_XS), n_x & 1, s_abort);
            ++n_x;
            return done;
        };
        for (int idx = blockIdx.x; idx < g.n_items && ok; idx += gridDim.x, ++n_item) {
            const Item it = item_of(p, g, idx, KEYS);
            const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0;
            const int uv0 = __ldg(p.cl_unit0_v + it.h * p.gh_v), nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - uv0;
            const int i0 = it.qt * BM, i = i0 + row;
            const bool live = i0 + 32 * q4 < p.Tq;                             // some row of my warp exists
            const int vis = p.causal ? min(p.Tk - 1, i + off) : p.Tk - 1;      // my last visible key
            const int vis_all = p.causal ? min(p.Tk - 1, i0 + 32 * q4 + off) : p.Tk - 1;    // of the warp's first row
            // coefficient of unit `lane`'s cluster; bit u of last: unit u is the last of its cluster
            float coef = 0.f;
            int cl = -1;
            if (lane < nuk) {
                cl = __ldg(p.unit_cluster_k + uk0 + lane);
                coef = __ldg(&p.unit_sz_k[uk0 + lane].x) * p.qk_scale_log2e;
                if constexpr (MODE != KV) coef = __ldg(&p.unit_sz_q[uk0 + lane].x) * __ldg(&p.unit_sz_k[uk0 + lane].x) * p.qk_scale_log2e;
                if constexpr (MODE == F8) coef *= 262144.0f;                   // both operands are n 2^-9
            }
            const int cl_next = __shfl_down_sync(0xffffffffu, cl, 1);
            const uint32_t last = __ballot_sync(0xffffffffu, lane < units_seen(nuk) && (lane >= nuk - 1 || cl != cl_next));

            float2 S[4][RUN / 2];
            // scores of my row against my keys of tile kt, times log2(e); hidden keys at NEG_BIG
            auto scores = [&](int kt) {
                const float* col = s_col + (n_k & 3) * KEYS;
                bool first = true;
                uint32_t m = last;                                             // (at least one bit)
                do {
                    const uint32_t slot = n_s % N_SLOTS;
                    const float c = __shfl_sync(0xffffffffu, coef, __ffs(m) - 1);
                    if (!mbar_wait(bar(B_SFULL + slot), (n_s / N_SLOTS) & 1, s_abort)) return false;
                    ++n_s;
                    __syncwarp();
                    tc::tc_fence_after();
                    if (live) {
                        if (first) {
                            if constexpr (MODE == KV) {
#pragma unroll
                                for (int b = 0; b < 4; ++b)
#pragma unroll
                                    for (int e = 0; e < RUN / 2; ++e) S[b][e] = make_float2(0.f, 0.f);
                            } else {
#pragma unroll
                                for (int b = 0; b < 4; ++b)
#pragma unroll
                                    for (int e = 0; e < RUN / 2; e += 2) {
                                        const float4 v = *reinterpret_cast<const float4*>(col + KEYS / 4 * b + RUN * hf + 2 * e);
                                        S[b][e] = make_float2(v.x, v.y); S[b][e + 1] = make_float2(v.z, v.w);
                                    }
                            }
                        }
                        const float2 c2 = make_float2(c, c);
                        const uint32_t ta = t_lane + O_COLS + slot * KEYS + RUN * hf;
                        uint32_t v[2][RUN];
                        auto load = [&](int b) {
                            if constexpr (RUN == 16) tc::tc_ld16(ta + KEYS / 4 * b, reinterpret_cast<uint32_t(&)[16]>(v[b & 1]));
                            else ld8(ta + KEYS / 4 * b, v[b & 1]);
                        };
                        load(0);
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            tc::tc_wait_ld();
                            if (b < 3) load(b + 1);
#pragma unroll
                            for (int e = 0; e < RUN / 2; ++e) {
                                float2 x;
                                if constexpr (MODE == I8) x = make_float2((float)(int)v[b & 1][2 * e], (float)(int)v[b & 1][2 * e + 1]);
                                else x = make_float2(__uint_as_float(v[b & 1][2 * e]), __uint_as_float(v[b & 1][2 * e + 1]));
                                S[b][e] = fma2(c2, x, S[b][e]);
                            }
                        }
                    }
                    first = false;
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_SEMPTY + slot));
                    m &= m - 1;
                } while (m);
                ++n_k;
                const int j0 = kt * KEYS;
                if (live && j0 + KEYS - 1 > vis_all) {
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int e = 0; e < RUN / 2; ++e) {
                            const int j = j0 + KEYS / 4 * b + RUN * hf + 2 * e;
                            if (j > vis) S[b][e].x = NEG_BIG;
                            if (j + 1 > vis) S[b][e].y = NEG_BIG;
                        }
                }
                return true;
            };

            // ---- pass 1: row maximum (integer calls: and row sum) over my keys
            float m = NEG_BIG, l = 0.f;
            for (int kt = 0; kt < it.n_kt; ++kt) {
                if (!scores(kt)) { ok = false; break; }
                if (live) {
                    float x0 = NEG_BIG, x1 = NEG_BIG;
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int e = 0; e < RUN / 2; e += 2) {
                            x0 = fmaxf(x0, fmaxf(S[b][e].x, S[b][e].y));
                            x1 = fmaxf(x1, fmaxf(S[b][e + 1].x, S[b][e + 1].y));
                        }
                    const float n = fmaxf(m, fmaxf(x0, x1));
                    if constexpr (MODE != KV) {
                        const float2 nn = make_float2(-n, -n);
                        float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
                        for (int b = 0; b < 4; ++b)
#pragma unroll
                            for (int e = 0; e < RUN / 2; e += 2) {
                                const float2 y = add2(S[b][e], nn), z = add2(S[b][e + 1], nn);
                                a0 = add2(a0, make_float2(ex2(y.x), ex2(y.y)));
                                a1 = add2(a1, make_float2(ex2(z.x), ex2(z.y)));
                            }
                        l = l * ex2(m - n) + ((a0.x + a0.y) + (a1.x + a1.y));
                    }
                    m = n;
                }
            }
            if (!ok) break;
            s_x[hf * BM + row] = make_float2(m, l);
            if (!group_sync()) { ok = false; break; }
            {
                const float2 o = s_x[(hf ^ 1) * BM + row];
                const float n = fmaxf(m, o.x);
                if constexpr (MODE != KV) l = l * ex2(m - n) + o.y * ex2(o.x - n);     // (a half without a visible key weighs 0)
                m = n;
            }
            // ---- pass 2: probabilities
            const float2 nm = make_float2(-m, -m);
            const float f = MODE == KV ? 0.f : p.inv_sP / l * 1.7763568394002505e-15f;   // times 2^-49: see below
            const float2 f2 = make_float2(f, f), k100 = make_float2(7.888609052210118e-31f, 7.888609052210118e-31f);   // 2^-100
            float lsum = 0.f;
            uint32_t rsum = 0u;
            const uint32_t p_row = base + g.off_p + row * 128, p_sw = row & 7;
            for (int kt = 0; kt < it.n_kt; ++kt, ++n_p) {
                if (!scores(kt)) { ok = false; break; }
                uint32_t w[16];
                if (live) {
                    if constexpr (MODE == KV) {
#pragma unroll
                        for (int b = 0; b < 4; ++b)
#pragma unroll
                            for (int e = 0; e < RUN / 2; ++e) {
                                const float2 y = add2(S[b][e], nm);
                                w[4 * e + b] = pack_half2(ex2(y.x), ex2(y.y));         // chunk e: the four pairs b
                                const float2 r = __half22float2(*reinterpret_cast<const __half2*>(&w[4 * e + b]));
                                lsum += r.x + r.y;           // the rounded values: the division normalises what was multiplied
                            }
                    } else {
                        // code = min(rne(2^(S - m) / (s_P l)), 255): the product scaled by 2^-149 is rounded once, half to even, to the
                        // grid of the subnormals, whose bit pattern is the integer itself; the saturating pack clamps it
#pragma unroll
                        for (int e = 0; e < RUN / 2; ++e) {
                            int q[4][2];
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const float2 y = add2(S[b][e], nm);
                                const float2 t = mul2(mul2(make_float2(ex2(y.x), ex2(y.y)), f2), k100);
                                q[b][0] = __float_as_int(t.x); q[b][1] = __float_as_int(t.y);
                            }
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                w[2 * e + k] = sat_pack_u8(q[1][k], q[0][k], sat_pack_u8(q[3][k], q[2][k], 0u));
                                rsum = __dp4a(w[2 * e + k], 0x01010101u, rsum);
                            }
                        }
                        if (p.p_dbg && i < p.Tq) {
                            uint8_t* dst = p.p_dbg + (((int64_t)it.seq * p.H + it.h) * p.Tq + i) * p.Tk;
#pragma unroll
                            for (int e = 0; e < 16; ++e)
#pragma unroll
                                for (int b = 0; b < 4; ++b) {
                                    const int j = kt * KEYS + KEYS / 4 * b + RUN * hf + e;
                                    if (j < p.Tk) dst[j] = (uint8_t)(w[e] >> (8 * b));
                                }
                        }
                    }
                }
                if (!mbar_wait(bar(B_PEMPTY), (n_p & 1) ^ 1, s_abort)) { ok = false; break; }
                if (live) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) sts128(p_row + (((4 * hf + c) ^ p_sw) << 4), w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                }
                tc::fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_PFULL));
            }
            if (!ok) break;
            // ---- outputs
            s_x[2 * BM + hf * BM + row] = make_float2(lsum, __uint_as_float(rsum));
            if (!group_sync()) { ok = false; break; }
            const float2 part = s_x[2 * BM + (hf ^ 1) * BM + row];
            const float inv_l = MODE == KV ? 1.0f / (lsum + part.x) : 0.f;
            const int rs = (int)(rsum + __float_as_uint(part.y));
            if (!mbar_wait(bar(B_OFULL), n_item & 1, s_abort)) { ok = false; break; }
            __syncwarp();
            tc::tc_fence_after();
            const uint32_t stage = base + g.off_v, o_row = stage + row * g.out_pitch;
            __half* out_row = p.out + ((int64_t)it.seq * p.Tq + i) * p.ldo;
            for (int u = hf; u < nuv; u += 2) {
                // channel of position `lane` of the unit
                const int pos = 32 * (uv0 + u) + lane;
                const int ch = __ldg(p.jidx_v + pos) >= 0 ? (int)__ldg(p.src_v + pos) : -1;
                const float2 sz = __ldg(p.unit_sz_v + uv0 + u);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t v[16];
                    if (live) { tc::tc_ld16(t_lane + 32 * u + 16 * half, v); tc::tc_wait_ld(); }
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int c = __shfl_sync(0xffffffffu, ch, 16 * half + e);
                        if (!live || c < 0) continue;
                        float o;
                        if constexpr (MODE == KV) o = sz.x * (__uint_as_float(v[e]) * inv_l - (sz.y - (p.bits_v == 8 ? 128.0f : 8.0f)));
                        else o = p.s_P * sz.x * (float)((int)v[e] - (int)sz.y * rs);
                        const __half oh = __float2half_rn(o);
                        if (g.local_v) sts16(o_row + 2 * (c - it.h * p.hd), __half_as_ushort(oh));
                        else if (i < p.Tq) out_row[c] = oh;
                    }
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_OEMPTY));
            if (g.local_v) {
                if (!group_sync()) { ok = false; break; }                      // (a row's units are spread over both halves)
                __half* out0 = p.out + ((int64_t)it.seq * p.Tq + i0) * p.ldo + it.h * p.hd;
                const int n_rows = min(BM, p.Tq - i0);
                const bool pairs = (((uintptr_t)p.out & 3u) == 0) && (p.ldo & 1) == 0 && (p.hd & 1) == 0;
                for (int r = sw_; r < n_rows; r += 8) {
                    const uint32_t src = stage + r * g.out_pitch;
                    if (pairs) {
                        uint32_t* dst = reinterpret_cast<uint32_t*>(out0 + (int64_t)r * p.ldo);
                        for (int c = lane; c < p.hd / 2; c += 32) dst[c] = lds32(src + 4 * c);
                    } else {
                        for (int c = lane; c < p.hd; c += 32) out0[(int64_t)r * p.ldo + c] = __ushort_as_half(lds16(src + 2 * c));
                    }
                }
                __syncwarp();
            }
            if (lane == 0) mbar_arrive(bar(B_OUT));
        }
    }

    // ---------------------------------------------------------------- teardown
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    if (tid == 0 && *s_abort && g.status) atomicExch(g.status, RPTQ_ERR_DEVICE_TIMEOUT);
}

template <int MODE>
static int launch_one(const AttnParams& p, int units_k, int units_v, int n_seq, bool v_heads_local, int dev, int n_sm, cudaStream_t st)
{
    constexpr int KEYS = keys_of(MODE);
    Plan g{};
    g.n_qt = (p.Tq + BM - 1) / BM;
    g.n_seq = n_seq;
    const int64_t items = (int64_t)g.n_qt * p.H * n_seq;
    if (items > 2147483647ll) return RPTQ_ERR_UNSUPPORTED;
    g.n_items = (int)items;
    const int atoms = MODE == KV ? (units_k + 1) / 2 : (units_k + 3) / 4;
    g.off_k = atoms * ATOM_Q;
    g.k_stage = atoms * KEYS * 128;
    g.off_v = g.off_k + 2 * g.k_stage;
    g.v_stage = units_v * 32 * 128;
    const int raw_k = MODE != KV && p.bits_k == 8 ? 0 : KEYS * raw_pitch_of(p.bits_k, units_k);
    g.pitch_k = raw_pitch_of(p.bits_k, units_k);
    g.pitch_v = raw_pitch_of(p.bits_v, units_v);
    const int rest = BM * 128 + raw_k + KEYS * g.pitch_v + 4 * KEYS * 4 + 4 * BM * 8 + 256;
    constexpr int LIMIT = 226 * 1024;                     // (with 1 KiB for the alignment: the most a block may have)
    g.v_stages = g.off_v + 2 * g.v_stage + rest <= LIMIT ? 2 : 1;
    g.off_p = g.off_v + g.v_stages * g.v_stage;
    g.off_rawk = g.off_p + BM * 128;
    g.off_rawv = g.off_rawk + raw_k;
    g.off_col = g.off_rawv + KEYS * g.pitch_v;
    g.off_x = g.off_col + 4 * KEYS * 4;
    g.off_bar = g.off_x + 4 * BM * 8;
    g.total = g.off_bar + 256;
    if (g.total > LIMIT) return RPTQ_ERR_UNSUPPORTED;
    // an output tile in the V and P region: an odd number of words per row keeps a warp's rows in different banks
    const int words = (p.hd + 1) / 2;
    g.out_pitch = 4 * (words | 1);
    g.local_v = v_heads_local && BM * g.out_pitch <= g.v_stages * g.v_stage + BM * 128;
    g.status = device_status_word();
    const void* fn = reinterpret_cast<const void*>(prefill_kernel<MODE>);
    static std::atomic<uint64_t> done{0}, pool_ok{0};
    if (!(pool_ok.load(std::memory_order_acquire) >> (dev & 63) & 1u)) {
        cudaFuncAttributes attr;
        if (cudaFuncGetAttributes(&attr, fn) != cudaSuccess) return RPTQ_ERR_CUDA;
        // the register re-partition (setmaxnreg) draws on what the block is launched with
        if (attr.numRegs * THREADS < 128 * (REGS_MMA + 2 * REGS_LOAD + 2 * REGS_SOFTMAX)) return RPTQ_ERR_UNSUPPORTED;
        if (dev >= 0 && dev < 64) pool_ok.fetch_or(uint64_t(1) << dev, std::memory_order_release);
    }
    if (allow_smem(fn, dev, 227 * 1024, done) != RPTQ_OK) return RPTQ_ERR_CUDA;
    const int grid = g.n_items < n_sm ? g.n_items : n_sm;
    return launch_kernel(prefill_kernel<MODE>, dim3((unsigned)grid), THREADS, (size_t)g.total + 1024, 0, st, p, g);
}

int launch(const AttnParams& p, bool kv, int units_k, int units_v, int n_seq, bool v_heads_local, int dev, int n_sm, cudaStream_t st)
{
    if (kv) return launch_one<KV>(p, units_k, units_v, n_seq, v_heads_local, dev, n_sm, st);
    if (p.bits_q <= 4 && p.bits_k <= 4) return launch_one<F8>(p, units_k, units_v, n_seq, v_heads_local, dev, n_sm, st);
    return launch_one<I8>(p, units_k, units_v, n_seq, v_heads_local, dev, n_sm, st);
}

}  // namespace attn_prefill
}  // namespace rptq
