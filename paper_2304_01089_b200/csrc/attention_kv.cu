// rptq_attention_kv: attention with only the key / value cache quantised (Sec. 5.2: the W4A4KV, W4A3KV and W3A3KV schemes).
// The query and the probabilities stay 16-bit floating point; K and V are the per-cluster codes of the per-head layouts (Sec.
// 4.2, 5.1), written by the projections' epilogues. Argument checks and the choice of the kernel: attention_decode.cu
// for a few queries per sequence, attention_prefill.cu for more.
#include "attn_common.cuh"

extern "C" int rptq_attention_kv(const rptq_layout_t* LK, const rptq_layout_t* LV, int n_heads,
                                 const void* q_f16, int64_t ldq, int Tq, const void* k_codes, const void* v_codes, int Tk, int n_seq,
                                 float qk_scale, int causal, void* out_f16, int64_t ldo, void* stream)
{
    using namespace rptq;
    using namespace rptq::attn;
    if (!LK || !LV || !q_f16 || !k_codes || !v_codes || !out_f16) return RPTQ_ERR_INVALID_ARG;
    if (n_heads < 1 || Tq < 0 || Tk < Tq || n_seq < 0 || !(qk_scale >= 0.f)) return RPTQ_ERR_INVALID_ARG;
    if (LK->g % n_heads || LV->g % n_heads || LK->C != LV->C || LK->C % n_heads || ldq < LK->C || ldo < LV->C) return RPTQ_ERR_INVALID_ARG;
    if (!aligned16(k_codes) || !aligned16(v_codes) || (reinterpret_cast<uintptr_t>(q_f16) & 1u) || (reinterpret_cast<uintptr_t>(out_f16) & 1u))
        return RPTQ_ERR_INVALID_ARG;
    if (n_heads > 65535 || n_seq > 65535) return RPTQ_ERR_UNSUPPORTED;
    if (!LK->in_cluster_order || !LV->in_cluster_order) return RPTQ_ERR_UNSUPPORTED;
    const int units_k = max_units_per_head(LK, n_heads), units_v = max_units_per_head(LV, n_heads);
    if (units_k > MAX_UNITS || units_v > MAX_UNITS) return RPTQ_ERR_UNSUPPORTED;
    if (!heads_own_their_channels(LK, n_heads)) return RPTQ_ERR_INVALID_ARG;
    if (Tq == 0 || n_seq == 0) return RPTQ_OK;
    int dev = -1;
    if (LK->device < 0 || cudaGetDevice(&dev) != cudaSuccess) return RPTQ_ERR_CUDA;
    if (dev != LK->device || dev != LV->device) return RPTQ_ERR_INVALID_ARG;

    AttnParams p{};
    p.q_f16 = static_cast<const __half*>(q_f16); p.ldq = ldq;
    p.k = static_cast<const uint8_t*>(k_codes); p.v = static_cast<const uint8_t*>(v_codes);
    p.k_row_bytes = LK->row_bytes; p.v_row_bytes = LV->row_bytes; p.bits_k = LK->bits; p.bits_v = LV->bits;
    p.Tq = Tq; p.Tk = Tk; p.H = n_heads; p.hd = LK->C / n_heads; p.gh_k = LK->g / n_heads; p.gh_v = LV->g / n_heads; p.causal = causal ? 1 : 0;
    p.cl_unit0_k = LK->d_cl_unit0; p.cl_unit0_v = LV->d_cl_unit0; p.unit_cluster_k = LK->d_unit_cluster;
    p.unit_sz_k = LK->d_unit_sz; p.unit_sz_v = LV->d_unit_sz;
    p.src_k = LK->d_src; p.src_v = LV->d_src; p.jidx_k = LK->d_jidx; p.jidx_v = LV->d_jidx;
    p.qk_scale_log2e = qk_scale * 1.4426950408889634f;
    p.out = static_cast<__half*>(out_f16); p.ldo = ldo;

    auto st = static_cast<cudaStream_t>(stream);
    const int n_sm = sm_count(dev);
    if (n_sm == 0) return RPTQ_ERR_CUDA;
    if (attn_decode::fits(p, true, units_k, units_v)) return attn_decode::launch(p, true, units_k, units_v, n_seq, dev, n_sm, st);
    return attn_prefill::launch(p, true, 0, 0, units_k, units_v, n_seq, heads_own_their_channels(LV, n_heads), dev, n_sm, st);
}
