// Attention for more queries than a decode step has: rptq_attention and rptq_attention_kv on the tcgen05 tensor cores.
//
// A persistent block works on 128 queries of one head at a time. Where the softmax output is quantised at 8 bits it is needed with the
// row's final maximum and sum, so integer calls walk the keys twice: pass 1 finds the row maxima and sums, pass 2 forms the
// probabilities and multiplies them with V. Nothing is rescaled on the way. Scores are computed in both passes; the tensor cores
// have room for that. KV calls walk the keys once: probabilities are relative to a reference that follows the row's maximum, and
// the output accumulator is brought to a new reference where it moves (3 x 1100 queries on 1337 keys, 32 heads of 128 channels: two walks
// 345 us, one 310).
//
// What bounds it: one exponential per score and pass (the special-function unit gives 16 per clock and SM), then the
// issue slots of the softmax warps: a score costs one multiply-add per cluster of the head, and five or six
// instructions more. So everything else is kept off those warps:
//   warps 0, 1    issue the score MMAs of two STREAMS (integer calls: the halves of a 128-key tile; KV: even and odd tiles
//                 of 64 keys): one accumulator per CLUSTER of the head (the scales differ), handed over slot by slot
//                 through the stream's own ring in tensor memory. The streams run on their own, so that one's drains
//                 fall under the other's exponentials
//   warp 2        issues P V (integer calls: in pass 2) into the head's output accumulator, which stays in tensor memory
//   warps 4-7     keys: packed rows arrive by cp.async one tile ahead, are unpacked into the swizzled operand tile; they
//                 also lay out the queries: integer calls store q - z^Q where that fits the operand type (a byte; 16 in
//                 magnitude for E4M3), otherwise q, and form the per-key term -sum_c s^Q s^K z^Q sum_p K_q
//   warps 8-11    values: unpacked and transposed into [position][key] (byte permutes on the packed words); and the
//                 output of an item, while the next item's pass 1 runs (they have nothing else to do there)
//   warps 12-19   softmax, four per stream: thread = query row, 64 keys; S = sum_c coef_c acc_c in registers; KV: rescaling
// Operand types (MODE):
//   I8   bytes, kind::i8, int32 sums
//   F8   both codes of at most four bits: a nibble n as an 8-bit E4M3 pattern IS the number n 2^-9, so the same bytes
//        multiply as kind::f8f6f4 and the sums (below 2^16 units) come out as exact fp32: no conversion per score and
//        cluster
//   KV   fp16 query; codes as fp16 integers n - 8 (n - 128): the centre is a constant per row in the scores and part of the
//        zero point in the outputs
// P V is u8 x u8 -> s32 for I8 and F8 (exact), fp16 x fp16 -> fp32 for KV.
// Key order inside a tile of the second product (both operands are written in it, so the sums do not change): within a
// quarter of 32 keys, byte b of word w is key w + 8 b; KV, quarters of 16 keys: fp16 pair b of chunk y is keys
// 4 b + 2 y + {0, 1}. It lets the V loader read and write shared memory without bank conflicts.
//
// Measured, us, against a mma.sync kernel with 64 (KV: 128) queries per block (72 heads of 128 channels, four clusters each,
// causal, two sequences of 2048 tokens): 3 bits 2321 -> 735; KV, 32 heads, three sequences, 1100 queries on 1337 keys, 4 bits
// 945 -> 310. What bounds it is the latency of the hand-overs between the roles: of the 9.7 warp cycles an issue (37 heads, 2048
// tokens), 3.7 are long scoreboards (tensor-memory loads, barrier waits), 1.7 fixed latencies, 0.4 instruction fetch (cache-only, of
// 11.3: 4.7, 1.5, 1.7); issue slots are 52 % (44 %) busy, the tensor pipe 11 %. Code that runs at the same time is worth keeping short all the
// same: the compiler told that the warp index is uniform 916 -> 790 (93 -> 83 KB of code), the output rows' store loops not
// unrolled 790 -> 772; a first cluster's drain of its own (two copies of the loop) 790 -> 830. The order in which items are dealt
// out: see item_index (767 -> 735).
#include <type_traits>

#include "attn_common.cuh"
#include "pack.cuh"

namespace rptq {
namespace attn_prefill {

using namespace attn;

enum { I8 = 0, F8 = 1, KV = 2 };
// Eight softmax warps, four for each stream. Sixteen of 32 keys a thread measured the same (773 and 770 us), KV 3 % slower: the loaders
// then have 56 registers.
constexpr int BM = 128, THREADS = 640, STREAMS = 2;
constexpr int K_WARP0 = 4, V_WARP0 = 8, S_WARP0 = 12;
constexpr int COLS = 64;                                  // keys of a stream's piece of work = columns of a score slot
constexpr int N_SLOTS = 2;                                // score slots of each stream
constexpr int S_WARPS = 4 * STREAMS;                      // softmax warps
// registers per thread of the warpgroups: MMA issuers, two of loaders, two of softmax (the block is launched with 96 each)
constexpr int REGS_MMA = 48, REGS_LOAD = 72, REGS_SOFTMAX = 144;
constexpr int REGS_ALL = REGS_MMA + 2 * REGS_LOAD + STREAMS * REGS_SOFTMAX;
static_assert(REGS_ALL <= 5 * 96, "register pool");
constexpr int O_COLS = 32 * MAX_UNITS;                    // tensor memory: the output accumulator, then the score slots
constexpr int ATOM_Q = BM * 128;                          // 128 rows of 128 bytes

__host__ __device__ constexpr int keys_of(int mode) { return mode == KV ? 64 : 128; }

// Shared memory of a launch (sizes follow the widest head of the layouts).
struct Plan {
    int n_items, n_qt, per_qt;        // per_qt: items of a query tile (heads x sequences)
    uint32_t inv_per_qt, inv_h;       // ceil(2^32 / per_qt), ceil(2^32 / H)
    int off_k, k_stage, off_v, v_stage, v_stages, off_p, p_tiles, off_rawk, rawk_stage, rawk_stages, pitch_k, off_rawv, pitch_v, off_col, off_ml, off_sum, off_bar, total;
    int local_v;          // V's heads own their channels and the output tile fits the V and P region: rows leave through shared memory
    int out_pitch;
    int q_staged;         // KV (whose heads own their channels): a head's queries are copied in rows of its own channels, in pieces of 16 bytes
    int folded;           // integer calls: the queries are stored as q - z^Q (it fits the operand type): no per-key term
    int* status;
};

__device__ __forceinline__ void ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void st32(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};"
        ::"r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]), "r"(taddr) : "memory");
}
// The whole warp executes these in converged control flow; one elected lane issues. a, b: the low words of the operands'
// descriptors (the high words are the same for every tile).
constexpr uint32_t DESC_HI = (uint32_t)(1024 >> 4) | (1u << 14) | (2u << 29);       // of smem_desc_sw128
template <int KIND>       // 0 i8, 1 f8f6f4, 2 f16
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc)
{
    if constexpr (KIND == 0)
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::i8 [%0], da, db, %3, p;\n\t}" ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(DESC_HI) : "memory");
    else if constexpr (KIND == 1)
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %3, p;\n\t}" ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(DESC_HI) : "memory");
    else
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\tmov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\telect.sync _|q, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "@q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(DESC_HI) : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar)
{
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void sts16_if(bool p, uint32_t addr, uint16_t a)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.shared.b16 [%0], %1;\n\t}" ::"r"(addr), "h"(a), "r"((int)p) : "memory");
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
// Every other round of items is dealt out backwards, so that no block gets the dearer one of every round (37 heads, 2048 tokens, causal:
// items of 16, 12, 8 and 4 tiles on one block, of 13, 9, 5 and 1 on another).
__device__ __forceinline__ int item_index(uint32_t n)
{
    return (int)(n * gridDim.x + ((n & 1u) ? gridDim.x - 1u - blockIdx.x : blockIdx.x));
}
struct Item { int qt, h, seq, n_kt; };
__device__ __forceinline__ Item item_of(const AttnParams& p, const Plan& g, int idx, int keys)
{
    Item it;
    // quotients by multiplication with ceil(2^32 / divisor): at most one too large
    auto divide = [](int n, int d, uint32_t inv, int& rest) {
        int q = d == 1 ? n : (int)__umulhi((uint32_t)n, inv);
        rest = n - q * d;
        if (rest < 0) { --q; rest += d; }
        return q;
    };
    int r;
    it.qt = g.n_qt - 1 - divide(idx, g.per_qt, g.inv_per_qt, r);
    it.seq = divide(r, p.H, g.inv_h, it.h);
    const int last = p.causal ? min(p.Tk - 1, it.qt * BM + BM - 1 + p.Tk - p.Tq) : p.Tk - 1;
    it.n_kt = last / keys + 1;
    return it;
}

// K8, V8: 8-bit key / value codes (otherwise 3 or 4 bits). Separate instances keep each one's code well inside the instruction
// cache, which this kernel's five roles share (at 188 KB of code every warp issued one instruction per 10 to 15 clocks:
// 1285 us against 886).
template <int MODE, bool K8, bool V8>
__global__ void __launch_bounds__(THREADS, 1)
prefill_kernel(const AttnParams p, const Plan g)
{
    constexpr int KEYS = keys_of(MODE);
    constexpr bool ALT = MODE == KV;                      // the streams take tiles by turns (otherwise halves of every tile)
    constexpr int PASSES = MODE == KV ? 1 : 2;            // over the keys
    static_assert(O_COLS + 2 * N_SLOTS * COLS <= 512, "tensor memory");
    constexpr int K_ATOM = KEYS * 128;                    // operand tile of the keys: KEYS rows of 128 bytes per atom
    constexpr int Q_LOADERS = MODE == KV ? 8 : 4;         // warps that lay out the queries
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (base - smem_u32(smem_raw));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + g.off_bar);
    constexpr int B_QFULL = 0, B_QEMPTY = 1, B_KFULL = 2, B_KEMPTY = 4, B_SFULL = 6, B_SEMPTY = B_SFULL + 2 * N_SLOTS, B_PFULL = B_SEMPTY + 2 * N_SLOTS,
                  B_PEMPTY = B_PFULL + 2, B_VFULL = B_PEMPTY + 2, B_VEMPTY = B_VFULL + 2, B_OFULL = B_VEMPTY + 2, B_OEMPTY = B_OFULL + 1,
                  B_OUT = B_OEMPTY + 1, B_SUM = B_OUT + 1, B_XS = B_SUM + 1, B_XV = B_XS + 1, B_DRAIN = B_XV + 1, B_REF = B_DRAIN + 3, N_BARS = B_REF + (ALT ? 16 : 0);
    static_assert(N_BARS * 8 + 16 <= 512, "barrier block");
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + N_BARS);
    volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
    const uint32_t bar0 = smem_u32(bars);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

    if (tid == 0) {
        mbar_init(bar(B_QFULL), Q_LOADERS); mbar_init(bar(B_QEMPTY), 2);
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(B_KFULL + i), 4); mbar_init(bar(B_KEMPTY + i), ALT ? 1 : 2); mbar_init(bar(B_VFULL + i), 4); mbar_init(bar(B_VEMPTY + i), 1);
            mbar_init(bar(B_PFULL + i), 4); mbar_init(bar(B_PEMPTY + i), 1);
        }
        for (int i = 0; i < 2 * N_SLOTS; ++i) { mbar_init(bar(B_SFULL + i), 1); mbar_init(bar(B_SEMPTY + i), 4); }
        mbar_init(bar(B_OFULL), 1); mbar_init(bar(B_OEMPTY), 4); mbar_init(bar(B_OUT), 4);
        mbar_init(bar(B_SUM), S_WARPS); mbar_init(bar(B_XV), 4);
        if constexpr (PASSES == 2) mbar_init(bar(B_XS), S_WARPS);
        for (int i = 0; i < 3; ++i) mbar_init(bar(B_DRAIN + i), 1);
        if constexpr (ALT) for (int i = 0; i < 16; ++i) mbar_init(bar(B_REF + i), 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    pdl_trigger();
    pdl_wait();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    float* s_col = reinterpret_cast<float*>(smem + g.off_col);            // [4][KEYS]
    float2* s_ml = reinterpret_cast<float2*>(smem + g.off_ml);            // [2][STREAMS][BM]: row maxima and sums over a stream's keys; KV: references
    uint32_t* s_sum = reinterpret_cast<uint32_t*>(smem + g.off_sum);      // [STREAMS][BM]: sums of probabilities (codes)

    if (warp < K_WARP0) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_MMA));
        auto desc = [&](int off) { return ((base + (uint32_t)off) & 0x3FFFFu) >> 4 | 1u << 16; };
        bool ok = true;
        if (warp < 2) {
            // ------------------------------------------------------------ scores of one stream
            const int stream = warp;
            constexpr uint32_t ID = (MODE == I8 ? (2u << 4) : (1u << 4)) | ((uint32_t)(COLS >> 3) << 17) | (8u << 24);   // D: s32 or f32; A, B: u8 / E4M3 / f16
            constexpr uint32_t LOG_ATOM = ALT ? 1 : 2, STEP = ALT ? 4 : 2;                   // units per atom; a unit's bytes / 16
            const uint32_t dq = desc(0), dk = desc(g.off_k + (ALT ? 0 : stream * COLS * 128)), k_step = (uint32_t)(g.k_stage >> 4);
            const uint32_t d0 = tmem + O_COLS + stream * (N_SLOTS * COLS);
            const uint32_t id = MODE == I8 && g.folded ? ID | (1u << 7) : ID;                // (signed bytes)
            const uint32_t b_full0 = bar(B_SFULL + stream * N_SLOTS), b_empty0 = bar(B_SEMPTY + stream * N_SLOTS);
            uint32_t n_k = 0, slot = 0, par = 1, n_item = 0;                    // n_k: my tiles so far
            for (int idx; ok && (idx = item_index(n_item)) < g.n_items; ++n_item) {
                const Item it = item_of(p, g, idx, KEYS);
                const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0, nu = units_seen(nuk);
                // bit u: unit u is the last of its cluster
                const int cl = lane < nuk ? __ldg(p.unit_cluster_k + uk0 + lane) : -1;
                const int cl_next = __shfl_down_sync(0xffffffffu, cl, 1);
                const uint32_t last = __ballot_sync(0xffffffffu, lane < nu && (lane >= nuk - 1 || cl != cl_next));
                if (!mbar_sleep_warp(bar(B_QFULL), n_item & 1, s_abort)) { ok = false; break; }
#pragma unroll 1
                for (int pass = 0; pass < PASSES && ok; ++pass) {
#pragma unroll 1
                    for (int kt = ALT ? stream : 0; kt < it.n_kt && ok; kt += ALT ? 2 : 1, ++n_k) {
                        const uint32_t st = ALT ? stream : n_k & 1;            // (KV: a stage belongs to a stream, which so sees all its phases)
                        if (!mbar_sleep_warp(bar(B_KFULL + st), (ALT ? n_k : n_k >> 1) & 1, s_abort)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t kb = dk + st * k_step;
                        uint32_t acc = 0u;
#pragma unroll 1
                        for (uint32_t u = 0; u < (uint32_t)nu; ++u) {
                            if (acc == 0u) {
                                if (!mbar_sleep_warp(b_empty0 + 8 * slot, par, s_abort)) { ok = false; break; }
                                tc_fence_after();
                            }
                            const uint32_t d = d0 + slot * COLS, in = (u & ((1u << LOG_ATOM) - 1u)) * STEP;
                            const uint32_t a = dq + (u >> LOG_ATOM) * (ATOM_Q >> 4) + in, b = kb + (u >> LOG_ATOM) * (K_ATOM >> 4) + in;
                            if constexpr (MODE == KV) {
                                mma<2>(d, a, b, id, acc);
                                mma<2>(d, a + 2, b + 2, id, 1u);
                            } else {
                                mma<MODE == F8 ? 1 : 0>(d, a, b, id, acc);
                            }
                            acc = 1u;
                            if ((last >> u) & 1u) {
                                commit(b_full0 + 8 * slot);
                                acc = 0u;
                                slot ^= 1u;
                                par ^= slot ^ 1u;
                            }
                        }
                        if (ok) commit(bar(B_KEMPTY + st));
                    }
                }
                if (ok) commit(bar(B_QEMPTY));
            }
        } else if (warp == 2) {
            // ------------------------------------------------------------ outputs
            constexpr uint32_t ID = (MODE == KV ? (1u << 4) : (2u << 4)) | (8u << 24);
            const uint32_t dv = desc(g.off_v), dp = desc(g.off_p), v_step = (uint32_t)(g.v_stage >> 4);
            uint32_t n_v = 0, n_item = 0, n_p0 = 0, n_p1 = 0;                  // (KV: tiles of each stream so far)
            for (int idx; ok && (idx = item_index(n_item)) < g.n_items; ++n_item) {
                const Item it = item_of(p, g, idx, KEYS);
                const int nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - __ldg(p.cl_unit0_v + it.h * p.gh_v);
                const uint32_t id = ID | ((uint32_t)(4 * nuv) << 17);
                if (!mbar_sleep_warp(bar(B_OEMPTY), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
                uint32_t acc = 0u;
#pragma unroll 1
                for (int kt = 0; kt < it.n_kt && ok; ++kt, ++n_v) {
                    const uint32_t st = g.v_stages == 2 ? n_v & 1 : 0u, ph = g.v_stages == 2 ? (n_v >> 1) & 1 : n_v & 1;
                    if (!mbar_sleep_warp(bar(B_VFULL + st), ph, s_abort)) { ok = false; break; }
                    const uint32_t b0 = dv + st * v_step;
                    if constexpr (ALT) {
                        const uint32_t stream = kt & 1, n_p = stream ? n_p1 : n_p0;
                        if (!mbar_sleep_warp(bar(B_PFULL + stream), n_p & 1, s_abort)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t a0 = dp + (g.p_tiles == 2 ? stream * (BM * 128 >> 4) : 0u);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (nuv > 0) mma<2>(tmem, a0 + 2 * k, b0 + 2 * k, id, k == 0 ? acc : 1u);
                        if (stream) ++n_p1; else ++n_p0;
                        // one buffer for both streams: it goes to the stream of the tile that follows
                        commit(bar(B_PEMPTY + (g.p_tiles == 2 ? stream : kt + 1 < it.n_kt ? stream ^ 1u : 0u)));
                    } else {
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            if (!mbar_sleep_warp(bar(B_PFULL + half), n_v & 1, s_abort)) { ok = false; break; }
                            tc_fence_after();
                            if (nuv > 0) {
                                mma<0>(tmem, dp + 4 * half, b0 + 4 * half, id, half == 0 ? acc : 1u);
                                mma<0>(tmem, dp + 4 * half + 2, b0 + 4 * half + 2, id, 1u);
                            }
                            commit(bar(B_PEMPTY + half));
                        }
                    }
                    acc = 1u;
                    if (ok) commit(bar(B_VEMPTY + st));
                }
                if (ok) commit(bar(B_OFULL));
            }
        }
        if (warp < 3 && !ok) {
            commit(bar(B_DRAIN + warp));
            mbar_wait(bar(B_DRAIN + warp), 0, s_abort, false);
        }
    } else if (warp < S_WARP0) {
        // ---------------------------------------------------------------- loaders: keys and queries (warps 4-7), values and outputs (8-11)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_LOAD));
        constexpr int ROWS_W = KEYS / 4;                                       // rows of a tile that a warp copies
        const int lw = warp & 3, lt = tid & 127;
        const int r0 = ROWS_W * lw + (lane >> 3), c0 = lane & 7;               // eight lanes per row; my rows are r0 + 4 i
        bool ok = true;
        // The tile that is being fetched (`nx`) and the one that is being worked on (`cu`), one tile behind
        struct Tile { uint32_t n; int t, n_t, kt; Item it; int u0, nu; };       // (n: the block's n-th item)
        const bool is_k = warp < V_WARP0;
        Tile nx, cu;
        nx.n = 0xFFFFFFFFu; nx.t = 0; nx.n_t = 1; nx.kt = 0;
        // keys: every item's tiles once a pass; values: once
        auto advance = [&]() {
            ++nx.kt;
            if (++nx.t == nx.n_t) {
                const int idx = item_index(++nx.n);
                nx.t = 0;
                if (idx >= g.n_items) return false;
                nx.it = item_of(p, g, idx, KEYS);
                nx.n_t = is_k ? PASSES * nx.it.n_kt : nx.it.n_kt;
                const int32_t* u = is_k ? p.cl_unit0_k + nx.it.h * p.gh_k : p.cl_unit0_v + nx.it.h * p.gh_v;
                nx.u0 = __ldg(u);
                nx.nu = __ldg(u + (is_k ? p.gh_k : p.gh_v)) - nx.u0;
            }
            if (nx.t == 0 || nx.kt == nx.it.n_kt) nx.kt = 0;
            return true;
        };
        const uint8_t* const codes = is_k ? p.k : p.v;
        const int64_t row_bytes = is_k ? p.k_row_bytes : p.v_row_bytes;
        const int bits = is_k ? p.bits_k : p.bits_v;
        // Copies of the packed rows of the tile to fetch: row r goes to dst(r, c), chunk c of 16 bytes. Rows past the last key: zeros.
        auto copy_rows = [&](const Tile& nx, auto dst) {
            const int win = (4 * bits * nx.u0) & ~15, n16 = ((4 * bits * nx.u0 - win) + 4 * bits * nx.nu + 15) >> 4;
            const int rows = p.Tk - nx.kt * KEYS;
            const uint8_t* from = codes + ((int64_t)nx.it.seq * p.Tk + nx.kt * KEYS + r0) * row_bytes + win + 16 * c0;
            const uint32_t rb = (uint32_t)row_bytes;
#pragma unroll 1
            for (int c = c0; c < n16; c += 8, from += 128) {
#pragma unroll
                for (int i = 0; i < ROWS_W / 4; ++i) {
                    const bool in = r0 + 4 * i < rows;
                    cp_async16(dst(r0 + 4 * i, c), in ? from + (uint64_t)(4 * i) * rb : codes, in);
                }
            }
        };
        // KV: the queries as fp16 in operand order (codes 0, 2, 1, 3, 4, 6, 5, 7 of every eight positions, the order in which
        // the key codes come out of their words). Eight warps of 16 rows; a lane takes up to four pairs of positions. The head's
        // channels of a row are copied as they are into the row's own place in the operand tile and permuted there, four rows at
        // a time (read, then written): gathered from global memory they took 22700 clocks an item, every load's latency in turn.
        auto gather_queries = [&](const Item& it, uint32_t n_item) {
            const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0, nu = units_seen(nuk);
            const int r0 = (warp - K_WARP0) * 16, rows = p.Tq - it.qt * BM - r0;               // rows: how many of my rows exist
            const __half* q_rows = p.q_f16 + ((int64_t)it.seq * p.Tq + it.qt * BM + r0) * p.ldq;
            int ca[4], cb[4];                                 // channels of my pairs (staged: their place in the row), -1: none
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int p2 = lane + 32 * k, code = (p2 >> 2) * 8 + (p2 & 1) + 4 * ((p2 >> 1) & 1), pos = 32 * uk0 + code;
                const bool in = p2 < 16 * nuk;                // (a head without channels: no pair is, zeros are written)
                auto place = [&](int at) {
                    if (!in || __ldg(p.jidx_k + at) < 0) return -1;
                    const int c = (int)__ldg(p.src_k + at);
                    return g.q_staged ? ((c - it.h * p.hd) >> 6) * ATOM_Q + 2 * ((c - it.h * p.hd) & 63) : c;
                };
                ca[k] = place(pos);
                cb[k] = place(pos + 2);
            }
            if (!mbar_sleep_warp(bar(B_QEMPTY), (n_item & 1) ^ 1, s_abort)) return false;
            if (g.q_staged) {
                const int per_row = p.hd / 8;                 // 16-byte chunks
#pragma unroll 1
                for (int i = lane; i < 16 * per_row; i += 32) {
                    const int r = i / per_row, c = i - r * per_row;
                    cp_async16(base + (c >> 3) * ATOM_Q + (r0 + r) * 128 + 16 * (c & 7), r < rows ? q_rows + r * p.ldq + it.h * p.hd + 8 * c : p.q_f16, r < rows);
                }
                cp_async_commit();
                cp_async_wait<0>();
                __syncwarp();
            }
#pragma unroll 1
            for (int r4 = 0; r4 < 16; r4 += 4) {
                uint32_t v[4][4];
#pragma unroll
                for (int rr = 0; rr < 4; ++rr)
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint16_t x = 0, y = 0;
                        if (g.q_staged) {
                            const uint32_t row = base + (r0 + r4 + rr) * 128;
                            if (ca[k] >= 0) x = lds16(row + ca[k]);
                            if (cb[k] >= 0) y = lds16(row + cb[k]);
                        } else if (r4 + rr < rows) {          // (layouts whose heads share channels, rows without alignment)
                            const uint16_t* row = reinterpret_cast<const uint16_t*>(q_rows) + (r4 + rr) * p.ldq;
                            if (ca[k] >= 0) x = row[ca[k]];
                            if (cb[k] >= 0) y = row[cb[k]];
                        }
                        v[rr][k] = x | ((uint32_t)y << 16);
                    }
                __syncwarp();
#pragma unroll
                for (int rr = 0; rr < 4; ++rr)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (lane + 32 * k < 16 * nu)
                            sts32(base + k * ATOM_Q + (r0 + r4 + rr) * 128 + (((lane >> 2) ^ ((r4 + rr) & 7)) << 4) + 4 * (lane & 3), v[rr][k]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_QFULL));
            return true;
        };
        bool have = advance();
        uint32_t n_item = 0;
        if (is_k) {
            // ------------------------------------------------------------ keys
            constexpr bool direct = MODE != KV && K8;                   // bytes already: copied straight into the operand tile
            float czq = 0.f;                      // integer calls: -s^Q s^K z^Q qk_scale log2(e) of unit `lane`
            uint32_t seq[2] = {0, 0};             // KV: tiles of each stage (stream) so far
            // iteration n fetches tile n and works on tile n - 1
#pragma unroll 1
            for (uint32_t n = 0; ok; ++n) {
                // (with one raw buffer a tile is fetched just before it is worked on)
                const bool ahead = direct || g.rawk_stages == 2;
                if (ahead ? have : n > 0) {
                    if constexpr (direct) {
                        // (copied into the operand tile itself: its products must have read it)
                        if (!mbar_sleep_warp(bar(B_KEMPTY + (n & 1)), ((n >> 1) & 1) ^ 1, s_abort)) { ok = false; break; }
                        const uint32_t to = base + g.off_k + (n & 1) * g.k_stage;
                        copy_rows(nx, [&](int r, int c) { return to + (c >> 3) * K_ATOM + r * 128 + (((c & 7) ^ (r & 7)) << 4); });
                    } else {
                        const uint32_t to = base + g.off_rawk + (ahead ? (n & 1) * g.rawk_stage : 0);
                        copy_rows(ahead ? nx : cu, [&](int r, int c) { return to + r * g.pitch_k + 16 * c; });
                    }
                }
                cp_async_commit();
                if (n > 0) {
                    const uint32_t m = n - 1, st = ALT ? cu.kt & 1 : m & 1, ph = ALT ? (st ? seq[1]++ : seq[0]++) : m >> 1;
                    const uint32_t tile = base + g.off_k + st * g.k_stage;
                    const int nuk = cu.nu, nu = units_seen(nuk);
                    if (cu.t == 0) {
                        // ---- a new item's queries
                        if constexpr (MODE == KV) {
                            if (!gather_queries(cu.it, n_item)) { ok = false; break; }
                        } else {
                            const int i = cu.it.qt * BM + lt;
                            const uint8_t* q_row = p.q + ((int64_t)cu.it.seq * p.Tq + (i < p.Tq ? i : 0)) * p.q_row_bytes;
                            czq = 0.f;
                            if (lane < nuk) {
                                const float2 q = __ldg(p.unit_sz_q + cu.u0 + lane), k = __ldg(p.unit_sz_k + cu.u0 + lane);
                                czq = -(q.x * k.x * p.qk_scale_log2e) * q.y;
                            }
                            if (!mbar_sleep_warp(bar(B_QEMPTY), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
#pragma unroll 2
                            for (int u = 0; u < nu; ++u) {
                                uint32_t o[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                                if (u < nuk && i < p.Tq) {
                                    load_unit(q_row, cu.u0 + u, p.bits_q, o);
                                    if (g.folded) {
                                        // 128 + q - z of every byte, then two's complement (I8), or sign and magnitude: the E4M3 pattern of
                                        // (q - z) 2^-9. Pads hold some constant; the keys' pads are 0
                                        const uint32_t z4 = (uint32_t)(int)__ldg(&p.unit_sz_q[cu.u0 + u].y) * 0x01010101u;
#pragma unroll
                                        for (int e = 0; e < 8; ++e) {
                                            if (MODE == I8 && p.bits_q == 8) { o[e] ^= 0x80808080u; continue; }          // (z = 128)
                                            const uint32_t t = (o[e] | 0x80808080u) - z4;
                                            if constexpr (MODE == I8) o[e] = t ^ 0x80808080u;
                                            else {
                                                const uint32_t neg = ~t & 0x80808080u, one = neg >> 7;
                                                o[e] = ((t ^ 0x80808080u ^ (one * 255u)) + one) | neg;
                                            }
                                        }
                                    }
                                }
                                const uint32_t d = base + (u >> 2) * ATOM_Q + lt * 128, c = 2 * (u & 3), sw = lt & 7;
                                sts128(d + ((c ^ sw) << 4), o[0], o[1], o[2], o[3]);
                                sts128(d + (((c + 1) ^ sw) << 4), o[4], o[5], o[6], o[7]);
                            }
                            fence_proxy_async();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(bar(B_QFULL));
                        }
                        ++n_item;
                    }
                    if (ahead && have) cp_async_wait<1>(); else cp_async_wait<0>();
                    __syncwarp();                                              // (a warp unpacks the rows that it copied)
                    if (!direct && !mbar_sleep_warp(bar(B_KEMPTY + st), (ph & 1) ^ 1, s_abort)) { ok = false; break; }
                    const uint32_t raw0 = base + g.off_rawk + (ahead ? (m & 1) * g.rawk_stage : 0) + ((4 * p.bits_k * cu.u0) & 15);
                    if constexpr (MODE == KV) {
                        // thread = (row, parity of the unit)
                        const int r = lt >> 1, odd = lt & 1, sw = r & 7;
                        const uint32_t raw = raw0 + r * g.pitch_k, d = tile + r * 128;
                        if constexpr (K8) {
#pragma unroll 2
                            for (int u = odd; u < nu; u += 2) {
                                uint4 w[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
                                if (u < nuk) { w[0] = lds128(raw + 32 * u); w[1] = lds128(raw + 32 * u + 16); }
                                const uint32_t a[8] = {w[0].x, w[0].y, w[0].z, w[0].w, w[1].x, w[1].y, w[1].z, w[1].w};
#pragma unroll
                                for (int c = 0; c < 4; ++c)                        // eight codes = one chunk
                                    sts128(d + (u >> 1) * K_ATOM + (((4 * odd + c) ^ sw) << 4),
                                           byte_half<0>(a[2 * c]), byte_half<8>(a[2 * c]), byte_half<0>(a[2 * c + 1]), byte_half<8>(a[2 * c + 1]));
                            }
                        } else {
                            uint4 w[4];                                        // (all loads first: a warp on its own is bound by latency)
#pragma unroll
                            for (int i = 0; i < 4; ++i) w[i] = 2 * i + odd < nuk ? nibbles(raw, 2 * i + odd, p.bits_k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                if (2 * i + odd < nu) {
                                    const uint32_t a[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
                                    for (int c = 0; c < 4; ++c)
                                        sts128(d + i * K_ATOM + (((4 * odd + c) ^ sw) << 4), nib_half<0>(a[c]), nib_half<8>(a[c]), nib_half<4>(a[c]), nib_half<12>(a[c]));
                                }
                            }
                        }
                    } else {
                        const int r = lt, sw = r & 7;
                        const uint32_t raw = raw0 + r * g.pitch_k, d = tile + r * 128;
                        if constexpr (!direct) {
#pragma unroll
                            for (int h = 0; h < 2; ++h) {                      // one atom: four units, all loads first
                                uint4 w[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) w[i] = 4 * h + i < nuk ? nibbles(raw, 4 * h + i, p.bits_k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    if (4 * h + i < nu) {
                                        const uint32_t at = d + h * K_ATOM;
                                        sts128(at + (((2 * i) ^ sw) << 4), w[i].x & 0x0F0F0F0Fu, (w[i].x >> 4) & 0x0F0F0F0Fu, w[i].y & 0x0F0F0F0Fu, (w[i].y >> 4) & 0x0F0F0F0Fu);
                                        sts128(at + (((2 * i + 1) ^ sw) << 4), w[i].z & 0x0F0F0F0Fu, (w[i].z >> 4) & 0x0F0F0F0Fu, w[i].w & 0x0F0F0F0Fu, (w[i].w >> 4) & 0x0F0F0F0Fu);
                                    }
                                }
                            }
                        }
                        if (!g.folded) {
                            float col = 0.f;
#pragma unroll 1
                            for (int u = 0; u < nu; ++u) {
                                const uint32_t at = d + (u >> 2) * K_ATOM, c = 2 * (u & 3);
                                const uint4 a = lds128(at + ((c ^ sw) << 4)), b = lds128(at + (((c + 1) ^ sw) << 4));
                                unsigned s0 = __dp4a(a.x, 0x01010101u, 0u), s1 = __dp4a(b.x, 0x01010101u, 0u);
                                s0 = __dp4a(a.y, 0x01010101u, s0); s1 = __dp4a(b.y, 0x01010101u, s1);
                                s0 = __dp4a(a.z, 0x01010101u, s0); s1 = __dp4a(b.z, 0x01010101u, s1);
                                s0 = __dp4a(a.w, 0x01010101u, s0); s1 = __dp4a(b.w, 0x01010101u, s1);
                                col = __fmaf_rn(__shfl_sync(0xffffffffu, czq, u), (float)(s0 + s1), col);
                            }
                            s_col[(m & 3) * KEYS + r] = col;
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_KFULL + st));
                }
                if (!have) break;
                cu = nx;
                have = advance();
            }
        } else {
            // ------------------------------------------------------------ values and outputs
            // KV: row r of the tile is staged at row blk + 4 y + 8 (2 b + s), r = 16 blk + 4 b + 2 y + s (see v_tile below)
            auto staged_row = [](int r) { return MODE == KV ? (r >> 4) + 4 * ((r >> 1) & 1) + 8 * (2 * ((r >> 2) & 3) + (r & 1)) : r; };
            uint32_t n_x = 0;
            // all four warps have passed this point (bounded, unlike a named barrier)
            auto group_sync = [&]() {
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_XV));
                const bool done = mbar_sleep_warp(bar(B_XV), n_x & 1, s_abort);
                ++n_x;
                return done;
            };
            // iteration n works on tile n - 1, then fetches tile n
#pragma unroll 1
            for (uint32_t n = 0; ok; ++n) {
                const int uv0 = cu.u0, nuv = cu.nu;
                const Item& it = cu.it;
                if (n > 0) {
                    const uint32_t raw = base + g.off_rawv + ((4 * p.bits_v * uv0) & 15), n_v = n - 1;
                    const uint32_t st = g.v_stages == 2 ? n_v & 1 : 0u, ph = g.v_stages == 2 ? (n_v >> 1) & 1 : n_v & 1;
                    cp_async_wait<0>();
                    if (!group_sync()) { ok = false; break; }                  // everyone's copies of the tile have landed
                    if (!mbar_sleep_warp(bar(B_VEMPTY + st), ph ^ 1, s_abort)) { ok = false; break; }
                    const uint32_t tile = base + g.off_v + st * g.v_stage;
                    if constexpr (MODE == KV) {
                        // lane = (chunk c8 of the 64 slots, word j of the unit). Chunk c8 = 2 blk + y holds the pairs b = 0..3 of keys
                        // 16 blk + 4 b + 2 y + {0, 1}: staged rows blk + 4 y + 8 (2 b + s), so the eight chunks' rows are in different banks
                        const int c8 = lane & 7, j = lane >> 3;
                        const uint32_t rows = raw + ((c8 >> 1) + 4 * (c8 & 1)) * g.pitch_v;
#pragma unroll 1
                        for (int u = lw; u < nuv; u += 4) {
                            const uint32_t d = tile + (32 * u + 8 * j) * 128;
                            // one chunk of position row 8 j + e; row & 7 = e
                            auto put = [&](int e, const uint32_t (&h4)[4]) { sts128(d + e * 128 + ((c8 ^ e) << 4), h4[0], h4[1], h4[2], h4[3]); };
                            if constexpr (V8) {
#pragma unroll
                                for (int half = 0; half < 2; ++half) {             // codes 4 half .. 4 half + 3
                                    uint32_t x[8];
#pragma unroll
                                    for (int a = 0; a < 8; ++a) x[a] = lds32(rows + 8 * a * g.pitch_v + 32 * u + 8 * j + 4 * half);
#pragma unroll
                                    for (int q = 0; q < 2; ++q) {
                                        uint32_t h0[4], h1[4];
#pragma unroll
                                        for (int b = 0; b < 4; ++b) {
                                            const uint32_t y = __byte_perm(x[2 * b], x[2 * b + 1], q ? 0x7632 : 0x5410);
                                            h0[b] = byte_half<0>(y); h1[b] = byte_half<8>(y);
                                        }
                                        put(4 * half + 2 * q, h0); put(4 * half + 2 * q + 1, h1);
                                    }
                                }
                            } else {
                                uint32_t x[8];
#pragma unroll
                                for (int a = 0; a < 8; ++a) {
                                    const uint32_t row = rows + 8 * a * g.pitch_v;
                                    if (p.bits_v == 4) x[a] = lds32(row + 16 * u + 4 * j);
                                    else {
                                        const uint32_t w0 = lds32(row + 12 * u), w1 = lds32(row + 12 * u + 4), w2 = lds32(row + 12 * u + 8);
                                        const uint32_t tail = ((w0 >> 3) & 0x11111111u) | ((w1 >> 2) & 0x22222222u) | ((w2 >> 1) & 0x44444444u);
                                        x[a] = j == 3 ? tail : (j == 0 ? w0 : j == 1 ? w1 : w2) & 0x77777777u;
                                    }
                                }
#pragma unroll
                                for (int q = 0; q < 2; ++q) {                      // codes 2 q, 2 q + 1 and those + 4
                                    uint32_t y[4], h[4];
#pragma unroll
                                    for (int b = 0; b < 4; ++b) y[b] = __byte_perm(x[2 * b], x[2 * b + 1], q ? 0x7632 : 0x5410);
#pragma unroll
                                    for (int b = 0; b < 4; ++b) h[b] = nib_half<0>(y[b]);
                                    put(2 * q, h);
#pragma unroll
                                    for (int b = 0; b < 4; ++b) h[b] = nib_half<8>(y[b]);
                                    put(2 * q + 1, h);
#pragma unroll
                                    for (int b = 0; b < 4; ++b) h[b] = nib_half<4>(y[b]);
                                    put(2 * q + 4, h);
#pragma unroll
                                    for (int b = 0; b < 4; ++b) h[b] = nib_half<12>(y[b]);
                                    put(2 * q + 5, h);
                                }
                            }
                        }
                    } else {
                        // lane = word w of the positions' rows: keys 32 (w / 8) + w % 8 + 8 b
                        const uint32_t wc = (uint32_t)lane >> 2, wo = 4 * ((uint32_t)lane & 3);
                        const uint32_t rows = raw + (32 * (lane >> 3) + (lane & 7)) * g.pitch_v;
#pragma unroll 1
                        for (int u = lw; u < nuv; u += 4) {
                            // position 8 k + i of the unit: row base at[i] + 1024 k (the swizzle depends on i alone)
                            uint32_t at[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) at[i] = tile + 32 * u * 128 + wo + i * 128 + ((wc ^ i) << 4);
                            auto put = [&](int pos, uint32_t x) { sts32(at[pos & 7] + (pos >> 3) * 1024, x); };
                            // 4 x 4 byte transpose: out[i] = byte i of the four rows
                            auto transpose = [](uint32_t a, uint32_t b, uint32_t c, uint32_t e, uint32_t (&out)[4]) {
                                const uint32_t x01l = __byte_perm(a, b, 0x5140), x01h = __byte_perm(a, b, 0x7362);
                                const uint32_t x23l = __byte_perm(c, e, 0x5140), x23h = __byte_perm(c, e, 0x7362);
                                out[0] = __byte_perm(x01l, x23l, 0x5410); out[1] = __byte_perm(x01l, x23l, 0x7632);
                                out[2] = __byte_perm(x01h, x23h, 0x5410); out[3] = __byte_perm(x01h, x23h, 0x7632);
                            };
                            if constexpr (V8) {
#pragma unroll
                                for (int half = 0; half < 2; ++half) {
                                    uint4 rw[4];
#pragma unroll
                                    for (int b = 0; b < 4; ++b) rw[b] = lds128(rows + 8 * b * g.pitch_v + 32 * u + 16 * half);
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
                                for (int b = 0; b < 4; ++b) rw[b] = nibbles(rows + 8 * b * g.pitch_v, u, p.bits_v);
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
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_VFULL + st));
                    if (!group_sync()) { ok = false; break; }                  // the raw rows have been read
                }
                if (have) copy_rows(nx, [&](int r, int c) { return base + g.off_rawv + staged_row(r) * g.pitch_v + 16 * c; });
                cp_async_commit();
                if constexpr (MODE == KV) {
                    if (have && nx.t == 0 && !gather_queries(nx.it, n == 0 ? 0u : n_item + 1)) { ok = false; break; }
                }
                if (n > 0 && cu.t == cu.n_t - 1) {
                // ---- the item's output rows: warp = lane quarter of the accumulator, thread = row
                // channel of position `lane` of every unit, asked for before the wait
                int chs[MAX_UNITS];
#pragma unroll
                for (int u = 0; u < MAX_UNITS; ++u) {
                    const int pos = 32 * (uv0 + u) + lane;
                    chs[u] = u < nuv && __ldg(p.jidx_v + pos) >= 0 ? (int)__ldg(p.src_v + pos) : -1;
                }
                if (!mbar_sleep_warp(bar(B_SUM), n_item & 1, s_abort) || !mbar_sleep_warp(bar(B_OFULL), n_item & 1, s_abort)) { ok = false; break; }
                tc_fence_after();
                const int row = 32 * lw + lane, i0 = it.qt * BM, i = i0 + row;
                const bool live = i0 + 32 * lw < p.Tq;                         // some row of my warp exists
                if (live) {
                    float inv_l = 0.f;
                    int rs = 0;
                    if constexpr (MODE == KV) {
                        // (the later reference, in which the accumulator is, is the larger one)
                        const float2* ml = s_ml + (n_item & 1) * STREAMS * BM + row;
                        const float ref = fmaxf(ml[0].y, ml[BM].y);
                        // (products rounded before they are added, as a stream rounds them that has one more tile, all of it hidden from this row:
                        // how far the tile's last row sees changes no bit)
                        inv_l = 1.0f / __fadd_rn(__fmul_rn(__uint_as_float(s_sum[row]), ex2(ml[0].y - ref)),
                                                 __fmul_rn(__uint_as_float(s_sum[BM + row]), ex2(ml[BM].y - ref)));
                    } else {
#pragma unroll
                        for (int q = 0; q < STREAMS; ++q) rs += (int)s_sum[q * BM + row];
                    }
                    const uint32_t stage = base + g.off_v, o_row = stage + row * g.out_pitch;
                    __half* out_row = p.out + ((int64_t)it.seq * p.Tq + i) * p.ldo;
#pragma unroll 1
                    for (int u = 0; u < nuv; ++u) {
                        // channel of position `lane` of the unit
                        int ch = chs[0];
#pragma unroll
                        for (int v = 0; v + 1 < MAX_UNITS; ++v) chs[v] = chs[v + 1];      // (a queue: the loop is not unrolled)
                        const float2 sz = __ldg(p.unit_sz_v + uv0 + u);
                        const float sc = MODE == KV ? sz.x * inv_l : p.s_P * sz.x, zf = sz.x * (sz.y - (V8 ? 128.0f : 8.0f));
                        const int zi = (int)sz.y * rs;
                        if (g.local_v && ch >= 0) ch = 2 * (ch - it.h * p.hd);         // its byte within a staged row
                        auto value = [&](uint32_t v) {
                            if constexpr (MODE == KV) return __half_as_ushort(__float2half_rn(__fmaf_rn(__uint_as_float(v), sc, -zf)));
                            else return __half_as_ushort(__float2half_rn(sc * (float)((int)v - zi)));
                        };
                        const uint32_t t_unit = tmem + ((uint32_t)(32 * lw) << 16) + 32 * u;
                        if (!g.local_v) {                                      // straight to the channel, column by column (rare layouts)
#pragma unroll 1
                            for (int e = 0; e < 32; ++e) {
                                const int c = __shfl_sync(0xffffffffu, ch, e);
                                uint32_t v;
                                asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(v) : "r"(t_unit + e) : "memory");
                                tc_wait_ld();
                                if (c >= 0 && i < p.Tq) out_row[c] = __ushort_as_half(value(v));
                            }
                            continue;
                        }
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            uint32_t v[16];
                            tc_ld16(t_unit + 16 * h, v);
                            tc_wait_ld();
                            // (the staged words of row r are exchanged by r & 31: no bank conflicts)
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                const int c = __shfl_sync(0xffffffffu, ch, 16 * h + e);
                                sts16_if(c >= 0, o_row + ((uint32_t)c ^ ((uint32_t)lane << 2)), value(v[e]));
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_OEMPTY));
                    if (g.local_v) {
                        const int n_rows = min(32, p.Tq - i0 - 32 * lw);
                        const uint32_t src = stage + 32 * lw * g.out_pitch;
                        __half* dst = p.out + ((int64_t)it.seq * p.Tq + i0 + 32 * lw) * p.ldo + it.h * p.hd;
                        const bool pairs = (((uintptr_t)p.out & 3u) == 0) && (p.ldo & 1) == 0 && (p.hd & 1) == 0;
                        if (pairs) {
#pragma unroll 1
                            for (int r = 0; r < n_rows; ++r, dst += p.ldo)
#pragma unroll 1
                                for (int c = lane; c < p.hd / 2; c += 32) reinterpret_cast<uint32_t*>(dst)[c] = lds32(src + r * g.out_pitch + ((c ^ r) << 2));
                        } else {
                            #pragma unroll 1
                            for (int r = 0; r < n_rows; ++r, dst += p.ldo)
#pragma unroll 1
                                for (int c = lane; c < p.hd; c += 32) dst[c] = __ushort_as_half(lds16(src + r * g.out_pitch + (((c >> 1) ^ r) << 2) + 2 * (c & 1)));
                        }
                    }
                } else if (lane == 0) {
                    mbar_arrive(bar(B_OEMPTY));
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_OUT));
                ++n_item;
                }
                if (!have) break;
                cu = nx;
                have = advance();
            }
        }
        cp_async_wait<0>();
    } else {
        // ---------------------------------------------------------------- softmax
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX));
        const int q4 = warp & 3, stream = (warp - S_WARP0) >> 2;              // q4: lane quarter of the accumulators
        const int row = 32 * q4 + lane;                                        // query row within the tile
        const uint32_t t_col = tmem + ((uint32_t)(32 * q4) << 16) + O_COLS + stream * (N_SLOTS * COLS);
        const uint32_t b_full0 = bar(B_SFULL + stream * N_SLOTS), b_empty0 = bar(B_SEMPTY + stream * N_SLOTS);
        uint32_t n_k0 = 0, slot = 0, par = 0, n_s = 0, n_item = 0;   // n_s: my tiles multiplied with V so far
        uint32_t ref_par = 0, n_other = 0;                           // KV: phases of the other stream's references (one bit for each set), its tiles so far
        bool ok = true;
        for (int idx; ok && (idx = item_index(n_item)) < g.n_items; ++n_item) {
            const Item it = item_of(p, g, idx, KEYS);
            const int i0 = it.qt * BM, i = i0 + row, off = p.Tk - p.Tq;
            const bool live = i0 + 32 * q4 < p.Tq;                             // some row of my warp exists
            const int vis = p.causal ? min(p.Tk - 1, i + off) : p.Tk - 1;      // my last visible key
            const int vis_all = p.causal ? min(p.Tk - 1, i0 + 32 * q4 + off) : p.Tk - 1;    // of the warp's first row
            // coefficient of unit `lane`'s cluster; bit u of last: unit u is the last of its cluster
            float coef = 0.f;
            uint32_t last;
            {
                const int uk0 = __ldg(p.cl_unit0_k + it.h * p.gh_k), nuk = __ldg(p.cl_unit0_k + (it.h + 1) * p.gh_k) - uk0;
                int cl = -1;
                if (lane < nuk) {
                    cl = __ldg(p.unit_cluster_k + uk0 + lane);
                    if constexpr (MODE == KV) coef = __ldg(&p.unit_sz_k[uk0 + lane].x) * p.qk_scale_log2e;
                    else coef = __ldg(&p.unit_sz_q[uk0 + lane].x) * __ldg(&p.unit_sz_k[uk0 + lane].x) * p.qk_scale_log2e;
                    if constexpr (MODE == F8) coef *= 262144.0f;               // both operands are n 2^-9
                }
                const int cl_next = __shfl_down_sync(0xffffffffu, cl, 1);
                last = __ballot_sync(0xffffffffu, lane < units_seen(nuk) && (lane >= nuk - 1 || cl != cl_next));
            }
            float m = NEG_BIG, l = 0.f, f = 0.f, lsum = 0.f;
            uint32_t rsum = 0u;
#pragma unroll 1
            for (int pass = 2 - PASSES; pass < 2 && ok; ++pass, n_k0 += it.n_kt) {
                if constexpr (PASSES == 2) if (pass == 1) {
                    // the streams' statistics meet (two sets by turns: a warp may be an item ahead of another)
                    float2* ml = s_ml + (n_item & 1) * STREAMS * BM + row;
                    ml[stream * BM] = make_float2(m, l);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_XS));
                    if (!mbar_sleep_warp(bar(B_XS), n_item & 1, s_abort)) { ok = false; break; }
                    l = 0.f;
#pragma unroll
                    for (int q = 0; q < STREAMS; ++q) m = fmaxf(m, ml[q * BM].x);
#pragma unroll
                    for (int q = 0; q < STREAMS; ++q) l = __fmaf_rn(ml[q * BM].y, ex2(ml[q * BM].x - m), l);     // (a stream without a visible key weighs 0)
                    f = p.inv_sP / l * 1.7763568394002505e-15f;                // times 2^-49: see below
                }
#pragma unroll 1
                for (int kt = ALT ? stream : 0; kt < it.n_kt; kt += ALT ? 2 : 1) {
                    // ---- scores of my row against my keys of the tile, times log2(e); hidden keys at NEG_BIG
                    float2 S[COLS / 2];
                    const float* col = s_col + ((n_k0 + kt) & 3) * KEYS + stream * COLS;
                    bool first = true;
                    uint32_t left = last;                                      // (at least one bit)
                    do {
                        const float c = __shfl_sync(0xffffffffu, coef, __ffs(left) - 1);
                        if (!mbar_sleep_warp(b_full0 + 8 * slot, par, s_abort)) { ok = false; break; }
                        tc_fence_after();
                        if (live) {
                            uint32_t v[32];
                            ld32(t_col + slot * COLS, v);
                            if (first) {
#pragma unroll
                                for (int e = 0; e < COLS / 2; ++e) S[e] = make_float2(0.f, 0.f);
                                if (MODE != KV && !g.folded) {
#pragma unroll
                                    for (int e = 0; e < COLS / 2; e += 2) {
                                        const float4 x = *reinterpret_cast<const float4*>(col + 2 * e);
                                        S[e] = make_float2(x.x, x.y); S[e + 1] = make_float2(x.z, x.w);
                                    }
                                }
                            }
                            const float2 c2 = make_float2(c, c);
#pragma unroll
                            for (int h = 0; h < COLS / 32; ++h) {
                                tc_wait_ld();
#pragma unroll
                                for (int e = 0; e < 16; ++e) {
                                    float2 x;
                                    if constexpr (MODE == I8) x = make_float2((float)(int)v[2 * e], (float)(int)v[2 * e + 1]);
                                    else x = make_float2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
                                    S[16 * h + e] = fma2(c2, x, S[16 * h + e]);
                                }
                                if (h + 1 < COLS / 32) ld32(t_col + slot * COLS + 32, v);
                            }
                        }
                        first = false;
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(b_empty0 + 8 * slot);
                        slot ^= 1u;
                        par ^= slot ^ 1u;
                        left &= left - 1;
                    } while (left);
                    if (!ok) break;
                    const int j0 = kt * KEYS + (ALT ? 0 : stream * COLS);
                    if (live && j0 + COLS - 1 > vis_all) {
                        const int n_vis = vis - j0;                            // my last visible column
#pragma unroll
                        for (int e = 0; e < COLS / 2; ++e) {
                            if (2 * e > n_vis) S[e].x = NEG_BIG;
                            if (2 * e + 1 > n_vis) S[e].y = NEG_BIG;
                        }
                    }
                    if constexpr (PASSES == 2) if (pass == 0) {
                        // ---- pass 1: row maximum and sum over my keys
                        if (live) {
                            float x0 = NEG_BIG, x1 = NEG_BIG;
#pragma unroll
                            for (int e = 0; e < COLS / 2; e += 2) {
                                x0 = fmaxf(x0, fmaxf(S[e].x, S[e].y));
                                x1 = fmaxf(x1, fmaxf(S[e + 1].x, S[e + 1].y));
                            }
                            const float n = fmaxf(m, fmaxf(x0, x1));
                            const float2 nn = make_float2(-n, -n);
                            float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
                            for (int e = 0; e < COLS / 2; e += 2) {
                                const float2 y = add2(S[e], nn), z = add2(S[e + 1], nn);
                                a0 = add2(a0, make_float2(ex2(y.x), ex2(y.y)));
                                a1 = add2(a1, make_float2(ex2(z.x), ex2(z.y)));
                            }
                            l = l * ex2(m - n) + ((a0.x + a0.y) + (a1.x + a1.y));
                            m = n;
                        }
                        continue;
                    }
                    // ---- KV: the reference that the row's probabilities are relative to: its maximum so far. References are handed from tile to tile,
                    // and so from stream to stream, in two sets by turns, since a stream may be an item ahead of the other (no more: see
                    // B_OUT below). Each row moves for itself: with the other rows of its warp, as the pass over the accumulator would allow, its bits
                    // would depend on the queries beside it. Error against 64 bits of 24 calls (level, rising and falling scores), ratio to that of
                    // two walks: 0.996 to 1.000; with moves of more than a power of two only: 0.9985 to 1.0004, and at most 2 % faster.
                    float down = 1.f;                                          // what the sums so far are worth in the new reference
                    bool moved = false;
                    if constexpr (MODE == KV) {
                        if (live) {
                            const uint32_t set = n_item & 1;
                            float2* ml = s_ml + set * STREAMS * BM + row;
                            float x0 = NEG_BIG, x1 = NEG_BIG;
#pragma unroll
                            for (int e = 0; e < COLS / 2; e += 2) {
                                x0 = fmaxf(x0, fmaxf(S[e].x, S[e].y));
                                x1 = fmaxf(x1, fmaxf(S[e + 1].x, S[e + 1].y));
                            }
                            float ref = fmaxf(x0, x1);
                            if (kt > 0) {
                                if (!mbar_sleep_warp(bar(B_REF + 8 * set + 2 * q4 + (stream ^ 1)), (ref_par >> set) & 1, s_abort)) { ok = false; break; }
                                ref_par ^= 1u << set;
                                const float before = ml[(stream ^ 1) * BM].x;
                                moved = ref > before;
                                if (moved) down = ex2(before - ref);
                                else ref = before;
                            }
                            if (kt + 1 < it.n_kt) {
                                ml[stream * BM].x = ref;
                                __syncwarp();
                                if (lane == 0) mbar_arrive(bar(B_REF + 8 * set + 2 * q4 + stream));
                            }
                            lsum *= ex2(m - ref);
                            m = ref;
                        }
                    }
                    // ---- probabilities (integer calls: pass 2). P's region also stages the previous item's output
                    if (kt < 2 && !mbar_sleep_warp(bar(B_OUT), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
                    // the buffer's previous tile has been multiplied
                    // (one buffer for both streams: stream 1's first tile waits for stream 0's)
                    const uint32_t behind = ALT && g.p_tiles == 1 && stream == 1 ? 0u : 1u;
                    if (!mbar_sleep_warp(bar(B_PEMPTY + stream), (n_s & 1) ^ behind, s_abort)) { ok = false; break; }
                    ++n_s;
                    if constexpr (MODE == KV) {
                        if (live && __any_sync(0xffffffffu, moved)) {
                            // the output accumulator of my rows in the new reference, when the tile before has been multiplied (with one buffer for both
                            // streams that is what has just been waited for) and before mine is. What it costs, us, scores that fall along the keys and so
                            // hardly move, rise, and show no trend: heads of 128 channels (32 heads, 3 x 1100 queries on 1337 keys) 292, 301, 304
                            // (two walks: 326); of 64 (32 heads, 2 x 2048 tokens) 283, 347, 349 (two walks: 355). 32 columns a wait instead of 16:
                            // 64 queries on 3000 keys 114 -> 112.
                            const uint32_t n_before = stream == 0 ? n_other + (kt >> 1) : n_other + ((kt + 1) >> 1);
                            if (g.p_tiles == 2 && !mbar_sleep_warp(bar(B_PEMPTY + (stream ^ 1)), (n_before - 1) & 1, s_abort)) { ok = false; break; }
                            tc_fence_after();
                            const int nuv = __ldg(p.cl_unit0_v + (it.h + 1) * p.gh_v) - __ldg(p.cl_unit0_v + it.h * p.gh_v);
                            const uint32_t t_out = tmem + ((uint32_t)(32 * q4) << 16);
#pragma unroll 1
                            for (int u = 0; u < nuv; ++u) {
                                uint32_t v[32];
                                ld32(t_out + 32 * u, v);
                                tc_wait_ld();
#pragma unroll
                                for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * down);
                                st32(t_out + 32 * u, v);
                            }
                            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                            tc_fence_before();
                        }
                    }
                    if (live) {
                        const float2 nm = make_float2(-m, -m);
                        if constexpr (MODE == KV) {
                            const uint32_t p_row = base + g.off_p + (g.p_tiles == 2 ? stream * (BM * 128) : 0) + row * 128;
#pragma unroll
                            for (int blk = 0; blk < COLS / 16; ++blk)
#pragma unroll
                                for (int y = 0; y < 2; ++y) {                  // chunk 2 blk + y: keys 16 blk + 4 b + 2 y + {0, 1}
                                    uint32_t w[4];
#pragma unroll
                                    for (int b = 0; b < 4; ++b) {
                                        const float2 x = add2(S[8 * blk + 2 * b + y], nm);
                                        w[b] = pack_half2(ex2(x.x), ex2(x.y));
                                        const float2 r = __half22float2(*reinterpret_cast<const __half2*>(&w[b]));
                                        lsum += r.x + r.y;   // the rounded values: the division normalises what was multiplied
                                    }
                                    sts128(p_row + (((2 * blk + y) ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
                                }
                        } else {
                            // code = min(rne(2^(S - m) / (s_P l)), 255): the product scaled by 2^-149 is rounded once, half to even, to the
                            // grid of the subnormals, whose bit pattern is the integer itself; the saturating pack clamps it
                            const float2 f2 = make_float2(f, f), k100 = make_float2(7.888609052210118e-31f, 7.888609052210118e-31f);   // 2^-100
                            const uint32_t p_row = base + g.off_p + row * 128;
#pragma unroll
                            for (int blk = 0; blk < COLS / 32; ++blk) {          // 32 keys: word x has keys x + 8 b
                                uint32_t w[8];
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    int q[4][2];
#pragma unroll
                                    for (int b = 0; b < 4; ++b) {
                                        const float2 y = add2(S[16 * blk + 4 * b + e], nm);
                                        const float2 t = mul2(mul2(make_float2(ex2(y.x), ex2(y.y)), f2), k100);
                                        q[b][0] = __float_as_int(t.x); q[b][1] = __float_as_int(t.y);
                                    }
#pragma unroll
                                    for (int k = 0; k < 2; ++k) {
                                        w[2 * e + k] = sat_pack_u8(q[1][k], q[0][k], sat_pack_u8(q[3][k], q[2][k], 0u));
                                        rsum = __dp4a(w[2 * e + k], 0x01010101u, rsum);
                                    }
                                }
                                const int c = 4 * stream + 2 * blk;
                                sts128(p_row + ((c ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
                                sts128(p_row + (((c + 1) ^ (row & 7)) << 4), w[4], w[5], w[6], w[7]);
                            }
                            if (p.p_dbg && i < p.Tq) {                         // key k of the stream: byte (k & 31) / 8 of word k & 7 of block k / 32
                                uint8_t* dst = p.p_dbg + (((int64_t)it.seq * p.H + it.h) * p.Tq + i) * p.Tk;
#pragma unroll 1
                                for (int k = 0; k < COLS && j0 + k < p.Tk; ++k) {
                                    const int c = 4 * stream + 2 * (k >> 5) + ((k & 7) >> 2);
                                    dst[j0 + k] = (uint8_t)(lds32(p_row + ((c ^ (row & 7)) << 4) + 4 * (k & 3)) >> (8 * ((k & 31) >> 3)));
                                }
                            }
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(B_PFULL + stream));
                }
            }
            if (!ok) break;
            // (a stream without a tile of its own has not waited for the previous item's sums to be read)
            if (ALT && it.n_kt == 1 && !mbar_sleep_warp(bar(B_OUT), (n_item & 1) ^ 1, s_abort)) { ok = false; break; }
            if constexpr (MODE == KV) {
                s_ml[((n_item & 1) * STREAMS + stream) * BM + row].y = m;
                n_other += (uint32_t)(stream == 0 ? it.n_kt / 2 : (it.n_kt + 1) / 2);
            }
            s_sum[stream * BM + row] = MODE == KV ? __float_as_uint(lsum) : rsum;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_SUM));
        }
    }

    // ---------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    if (tid == 0 && *s_abort && g.status) atomicExch(g.status, RPTQ_ERR_DEVICE_TIMEOUT);
}

template <int MODE, bool K8, bool V8>
static int launch_one(const AttnParams& p, int zq_min, int zq_max, int units_k, int units_v, int n_seq, bool v_heads_local, int dev, int n_sm, cudaStream_t st)
{
    constexpr int KEYS = keys_of(MODE);
    const int qmax_q = (1 << p.bits_q) - 1;
    Plan g{};
    g.n_qt = (p.Tq + BM - 1) / BM;
    const int64_t items = (int64_t)g.n_qt * p.H * n_seq;
    if (items > 2147483647ll) return RPTQ_ERR_UNSUPPORTED;
    g.n_items = (int)items;
    g.per_qt = p.H * n_seq;
    auto inverse = [](uint32_t d) { return (uint32_t)(((uint64_t(1) << 32) + d - 1) / d); };       // (d = 1 is not divided by)
    g.inv_per_qt = inverse((uint32_t)g.per_qt);
    g.inv_h = inverse((uint32_t)p.H);
    const int atoms = MODE == KV ? (units_k + 1) / 2 : (units_k + 3) / 4;
    g.off_k = atoms * ATOM_Q;
    g.k_stage = atoms * KEYS * 128;
    g.off_v = g.off_k + 2 * g.k_stage;
    g.v_stage = units_v * 32 * 128;
    g.pitch_k = raw_pitch(p.bits_k, units_k);
    g.pitch_v = raw_pitch(p.bits_v, units_v);
    g.rawk_stage = MODE != KV && p.bits_k == 8 ? 0 : KEYS * g.pitch_k;
    const int rest = BM * 128 + KEYS * g.pitch_v + 4 * KEYS * 4 + 2 * STREAMS * BM * 8 + STREAMS * BM * 4 + 512;
    constexpr int LIMIT = 226 * 1024;                     // (with 1 KiB for the alignment: the most a block may have)
    // a second packed key tile first (the copies of a tile then have a whole tile's time), then (KV) a probability tile for each
    // stream, then a second value tile
    int used = g.off_v + g.v_stage + g.rawk_stage + rest;
    g.rawk_stages = used + g.rawk_stage <= LIMIT ? 2 : 1;
    used += (g.rawk_stages - 1) * g.rawk_stage;
    g.p_tiles = MODE == KV && used + BM * 128 <= LIMIT ? 2 : 1;
    used += (g.p_tiles - 1) * BM * 128;
    g.v_stages = used + g.v_stage <= LIMIT ? 2 : 1;
    g.off_p = g.off_v + g.v_stages * g.v_stage;
    g.off_rawk = g.off_p + g.p_tiles * BM * 128;
    g.off_rawv = g.off_rawk + g.rawk_stages * g.rawk_stage;
    g.off_col = g.off_rawv + KEYS * g.pitch_v;
    g.off_ml = g.off_col + 4 * KEYS * 4;
    g.off_sum = g.off_ml + 2 * STREAMS * BM * 8;
    g.off_bar = g.off_sum + STREAMS * BM * 4;
    g.total = g.off_bar + 512;
    if (g.total > LIMIT) return RPTQ_ERR_UNSUPPORTED;
    // the output tile is staged in the V and P region (rows of a multiple of 128 bytes: see the staging stores)
    g.out_pitch = (2 * p.hd + 127) / 128 * 128;
    g.local_v = v_heads_local && BM * g.out_pitch <= g.v_stages * g.v_stage + g.p_tiles * BM * 128;
    g.q_staged = MODE == KV && p.hd % 8 == 0 && p.ldq % 8 == 0 && aligned16(p.q_f16);
    g.folded = MODE == F8 ? zq_min >= qmax_q - 16 && zq_max <= 16 : MODE == I8 ? zq_min >= qmax_q - 127 && zq_max <= 128 : 0;
    g.status = device_status_word();
    if (!g.status) return RPTQ_ERR_ALLOC;
    const void* fn = reinterpret_cast<const void*>(prefill_kernel<MODE, K8, V8>);
    static SmemAllowed done;
    static std::atomic<uint64_t> pool_ok{0};
    if (!(pool_ok.load(std::memory_order_acquire) >> (dev & 63) & 1u)) {
        cudaFuncAttributes attr;
        if (cudaFuncGetAttributes(&attr, fn) != cudaSuccess) return RPTQ_ERR_CUDA;
        // the register re-partition (setmaxnreg) draws on what the block is launched with
        if (attr.numRegs * THREADS < 128 * REGS_ALL) return RPTQ_ERR_UNSUPPORTED;
        if (dev >= 0 && dev < 64) pool_ok.fetch_or(uint64_t(1) << dev, std::memory_order_release);
    }
    if (allow_smem(fn, dev, 227 * 1024, done) != RPTQ_OK) return RPTQ_ERR_CUDA;
    const int grid = g.n_items < n_sm ? g.n_items : n_sm;
    return launch_kernel(prefill_kernel<MODE, K8, V8>, dim3((unsigned)grid), THREADS, (size_t)g.total + 1024, 0, st, p, g);
}

int launch(const AttnParams& p, bool kv, int zq_min, int zq_max, int units_k, int units_v, int n_seq, bool v_heads_local, int dev, int n_sm, cudaStream_t st)
{
    const bool k8 = p.bits_k == 8, v8 = p.bits_v == 8;
    auto go = [&](auto mode, auto ek, auto ev) {
        return launch_one<decltype(mode)::value, decltype(ek)::value, decltype(ev)::value>(p, zq_min, zq_max, units_k, units_v, n_seq, v_heads_local, dev, n_sm, st);
    };
    using std::false_type;
    using std::true_type;
    if (kv) {
        const std::integral_constant<int, KV> mode;
        if (k8) return v8 ? go(mode, true_type(), true_type()) : go(mode, true_type(), false_type());
        return v8 ? go(mode, false_type(), true_type()) : go(mode, false_type(), false_type());
    }
    if (p.bits_q <= 4 && !k8) {
        const std::integral_constant<int, F8> mode;
        return v8 ? go(mode, false_type(), true_type()) : go(mode, false_type(), false_type());
    }
    const std::integral_constant<int, I8> mode;
    if (k8) return v8 ? go(mode, true_type(), true_type()) : go(mode, true_type(), false_type());
    return v8 ? go(mode, false_type(), true_type()) : go(mode, false_type(), false_type());
}

}  // namespace attn_prefill
}  // namespace rptq
