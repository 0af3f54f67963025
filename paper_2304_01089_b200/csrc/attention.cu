// rptq_attention: self-attention on quantised Q, K and V (Sec. 4.2: Q and K share one reorder index; Sec. 5.1: the reorders of
// the attention sites are per head with their own clusters, the softmax output is quantised at 8 bits). Argument checks and
// the choice of the kernel: attention_decode.cu for a few queries per sequence, attention_prefill.cu for more.
//
// Of the four terms of (Q_q - z^Q)(K_q - z^K) the two that depend only on the query row shift a whole row of scores and
// cancel in the softmax; what is left is sum_c s^Q_c s^K_c sum_p (Q_q - z^Q_c) K_q.
#include "attn_common.cuh"

extern "C" int rptq_attention(const rptq_layout_t* LQ, const rptq_layout_t* LK, const rptq_layout_t* LV, int n_heads,
                              const void* q_codes, int Tq, const void* k_codes, const void* v_codes, int Tk, int n_seq,
                              float s_P, int z_P, float qk_scale, int causal,
                              void* out_f16, int64_t ldo, uint8_t* p_codes_out, void* stream)
{
    using namespace rptq;
    using namespace rptq::attn;
    if (!LQ || !LK || !LV || !q_codes || !k_codes || !v_codes || !out_f16) return RPTQ_ERR_INVALID_ARG;
    if (n_heads < 1 || Tq < 0 || Tk < Tq || n_seq < 0 || !(s_P > 0.f) || !(qk_scale >= 0.f)) return RPTQ_ERR_INVALID_ARG;
    if (LQ->g % n_heads || LK->g != LQ->g || LV->g % n_heads || ldo < LV->C) return RPTQ_ERR_INVALID_ARG;
    if (!aligned16(q_codes) || !aligned16(k_codes) || !aligned16(v_codes) || (reinterpret_cast<uintptr_t>(out_f16) & 1u)) return RPTQ_ERR_INVALID_ARG;
    // Q and K pair equal positions: same reorder index, same cluster sizes (the placement follows from them and the unit order)
    if (LQ->C != LK->C || LQ->in_cluster_order != LK->in_cluster_order || LQ->size != LK->size || LQ->perm != LK->perm) return RPTQ_ERR_INVALID_ARG;
    if (z_P != 0 || n_heads > 65535 || n_seq > 65535) return RPTQ_ERR_UNSUPPORTED;
    if (!LQ->in_cluster_order || !LV->in_cluster_order) return RPTQ_ERR_UNSUPPORTED;
    const int units_k = max_units_per_head(LQ, n_heads), units_v = max_units_per_head(LV, n_heads);
    if (units_k > MAX_UNITS || units_v > MAX_UNITS) return RPTQ_ERR_UNSUPPORTED;
    if ((int64_t)Tk * 255 * 255 > 2147483647ll) return RPTQ_ERR_UNSUPPORTED;      // the int32 sums of the second product
    if (Tq == 0 || n_seq == 0) return RPTQ_OK;
    int dev = -1;
    if (LQ->device < 0 || cudaGetDevice(&dev) != cudaSuccess) return RPTQ_ERR_CUDA;
    if (dev != LQ->device || dev != LK->device || dev != LV->device) return RPTQ_ERR_INVALID_ARG;

    AttnParams p{};
    p.q = static_cast<const uint8_t*>(q_codes); p.k = static_cast<const uint8_t*>(k_codes); p.v = static_cast<const uint8_t*>(v_codes);
    p.q_row_bytes = LQ->row_bytes; p.k_row_bytes = LK->row_bytes; p.v_row_bytes = LV->row_bytes;
    p.bits_q = LQ->bits; p.bits_k = LK->bits; p.bits_v = LV->bits;
    p.Tq = Tq; p.Tk = Tk; p.H = n_heads; p.hd = LV->C / n_heads; p.gh_k = LQ->g / n_heads; p.gh_v = LV->g / n_heads; p.causal = causal ? 1 : 0;
    p.cl_unit0_k = LQ->d_cl_unit0; p.cl_unit0_v = LV->d_cl_unit0; p.unit_cluster_k = LQ->d_unit_cluster;
    p.unit_sz_q = LQ->d_unit_sz; p.unit_sz_k = LK->d_unit_sz; p.unit_sz_v = LV->d_unit_sz;
    p.src_v = LV->d_src; p.jidx_v = LV->d_jidx;
    p.inv_sP = 1.0f / s_P; p.s_P = s_P; p.qk_scale_log2e = qk_scale * 1.4426950408889634f;
    p.out = static_cast<__half*>(out_f16); p.ldo = ldo; p.p_dbg = p_codes_out;

    auto st = static_cast<cudaStream_t>(stream);
    const int n_sm = sm_count(dev);
    if (n_sm == 0) return RPTQ_ERR_CUDA;
    if (attn_decode::fits(p, false, units_k, units_v)) return attn_decode::launch(p, false, units_k, units_v, n_seq, dev, n_sm, st);
    return attn_prefill::launch(p, false, LQ->z_min, LQ->z_max, units_k, units_v, n_seq, heads_own_their_channels(LV, n_heads), dev, n_sm, st);
}
