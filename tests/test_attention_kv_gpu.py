"""rptq_attention_kv (key / value cache quantised only, Sec. 5.2) against the oracle's definition.

The kernel multiplies fp16 operands with fp32 sums: the query is fp16 as given, the K and V codes are exact
in fp16, the scores' error is that of fp32 sums (~1e-6 relative), and the probabilities are rounded to fp16
before the second product. A probability moves by at most 2^-11 of itself, so
    |O - O_oracle| <= 2^-10 sum_j P[i][j] |V^[j][p]|  +  2^-11 |O|  +  1e-5 max|V^|
(the first term with a factor 2 for the exp2 approximation and the score error, the second for the fp16
result); the oracle computes in fp64 from the same fp16 query values.
"""
import numpy as np
import pytest

import oracle
from test_attention_gpu import Case, channel_of_oracle_position

pytestmark = pytest.mark.gpu


def _check(c, q16, causal, n_seq=1):
    """c: a Case (its K layout is LK, V layout LV); q16: fp16 [n_seq * Tq][C] in the original channel order."""
    import torch
    from scipy.special import softmax
    from paper_2304_01089_b200 import binding
    Tq, Tk, H, hd, gh = c.Tq // n_seq, c.Tk // n_seq, c.H, c.hd, c.gh
    Cn = H * hd
    out = torch.full((n_seq * Tq + 1, Cn + 8), float("nan"), dtype=torch.float16, device="cuda")
    qd = torch.from_numpy(q16).cuda()
    binding.attention_kv(c.LK, c.LV, H, qd, c.dk, c.dv, out, c.qk_scale, causal, Tq=Tq, Tk=Tk, n_seq=n_seq)
    torch.cuda.synchronize()
    o = out.float().cpu().numpy()
    assert np.isnan(o[n_seq * Tq]).all() and np.isnan(o[:, Cn:]).all()
    o = o[:n_seq * Tq, :Cn].astype(np.float64)
    ch_k = channel_of_oracle_position(c.perm_qk, c.size_qk).astype(np.int32)
    ch_v = channel_of_oracle_position(c.perm_v, c.size_v)
    real_v = ch_v >= 0
    off_v, _ = oracle.segment_offsets(c.size_v)
    Vh = np.zeros(c.v.shape)
    for cl in range(len(c.size_v)):
        sl = slice(off_v[cl], off_v[cl] + c.size_v[cl])
        Vh[:, sl] = float(c.sV[cl]) * (c.v[:, sl].astype(np.float64) - c.zV[cl])
    off_k, _ = oracle.segment_offsets(c.size_qk)
    for s in range(n_seq):
        qs, ks = slice(s * Tq, (s + 1) * Tq), slice(s * Tk, (s + 1) * Tk)
        q64 = q16[qs].astype(np.float64)
        want = oracle.attention_kv(q64, ch_k, c.k[ks], c.v[ks], H, gh, c.size_qk, c.sK.astype(np.float64), c.zK,
                                   c.size_v, c.sV.astype(np.float64), c.zV, c.qk_scale, causal)
        got = np.zeros_like(want)
        got[:, real_v] = o[qs][:, ch_v[real_v]]
        # the bound needs P: recomputed here from the oracle's own inputs (test-side arithmetic for the bound only)
        for h in range(H):
            lo, hi = off_k[h * gh], off_k[(h + 1) * gh]
            real_k = ch_k[lo:hi] >= 0
            Kh = np.zeros((Tk, hi - lo))
            for cl in range(h * gh, (h + 1) * gh):
                sl = slice(off_k[cl] - lo, off_k[cl] - lo + c.size_qk[cl])
                Kh[:, sl] = float(c.sK[cl]) * (c.k[ks][:, off_k[cl]:off_k[cl] + c.size_qk[cl]].astype(np.float64) - c.zK[cl])
            A = c.qk_scale * q64[:, ch_k[lo:hi][real_k]] @ Kh[:, real_k].T
            if causal:
                A = np.where(np.arange(Tk)[None, :] <= np.arange(Tq)[:, None] + (Tk - Tq), A, -np.inf)
            P = softmax(A, axis=1)
            vs = slice(off_v[h * gh], off_v[(h + 1) * gh])
            bound = 2.0 ** -10 * (P @ np.abs(Vh[ks][:, vs])) + 2.0 ** -11 * np.abs(want[:, vs]) + 1e-5 * np.abs(Vh).max()
            assert np.all(np.abs(got[:, vs] - want[:, vs]) <= bound), (s, h, np.abs(got[:, vs] - want[:, vs]).max())
        assert np.abs(want).max() > 0


def _query(rng, T, Cn, scale=1.0):
    return (rng.normal(size=(T, Cn)) * scale).astype(np.float16)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("bits", [(4, 4, 4), (4, 3, 3), (4, 8, 8)])
def test_small_heads_ragged_tiles(causal, bits):
    c = Case(41, H=3, hd=40, gh=4, Tq=150, Tk=150, bits=bits)
    _check(c, _query(np.random.default_rng(1), 150, 120), causal)


@pytest.mark.parametrize("causal", [False, True])
def test_head_of_128_channels_four_clusters(causal):
    c = Case(42, H=2, hd=128, gh=4, Tq=200, Tk=200, allow_empty=False)
    _check(c, _query(np.random.default_rng(2), 200, 256, 0.5), causal)


@pytest.mark.parametrize("Tq,Tk", [(1, 1), (1, 130), (70, 200), (65, 129)])
def test_queries_are_the_last_tokens_of_the_cache(Tq, Tk):
    c = Case(43 + Tq, H=2, hd=64, gh=4, Tq=Tq, Tk=Tk)
    _check(c, _query(np.random.default_rng(3), Tq, 128), True)


def test_several_sequences_and_empty_clusters():
    c = Case(44, H=2, hd=48, gh=4, Tq=3 * 40, Tk=3 * 70)
    _check(c, _query(np.random.default_rng(4), 120, 96), True, n_seq=3)


def test_refusals_and_empty_calls():
    import torch
    from paper_2304_01089_b200 import binding
    c = Case(45, H=2, hd=32, gh=2, Tq=8, Tk=8)
    q = torch.zeros((8, 64), dtype=torch.float16, device="cuda")
    out = torch.full((8, 64), 7.0, dtype=torch.float16, device="cuda")
    binding.attention_kv(c.LK, c.LV, 2, q, c.dk, c.dv, out, c.qk_scale, True, Tq=0, Tk=8)
    binding.attention_kv(c.LK, c.LV, 2, q, c.dk, c.dv, out, c.qk_scale, True, Tq=8, Tk=8, n_seq=0)
    torch.cuda.synchronize()
    assert bool((out == 7.0).all())
    with pytest.raises(binding.RptqError) as e:      # more queries than keys
        binding.attention_kv(c.LK, c.LV, 2, q, c.dk, c.dv, out, c.qk_scale, True, Tq=8, Tk=4)
    assert e.value.status == binding.ERR_INVALID_ARG
    with pytest.raises(binding.RptqError) as e:      # heads that do not divide the clusters
        binding.attention_kv(c.LK, c.LV, 3, q, c.dk, c.dv, out, c.qk_scale, True)
    assert e.value.status == binding.ERR_INVALID_ARG


def test_layouts_whose_heads_do_not_own_their_channels_are_refused():
    import torch
    from paper_2304_01089_b200 import binding
    from helpers import random_layout_params
    rng = np.random.default_rng(9)
    perm, size, scale, zero = random_layout_params(rng, 64, 4, 4, allow_empty=False)     # one permutation across both heads
    L = binding.Layout(perm, size, scale, zero, 4)
    q = torch.zeros((8, 64), dtype=torch.float16, device="cuda")
    codes = torch.zeros((8, L.row_bytes), dtype=torch.uint8, device="cuda")
    with pytest.raises(binding.RptqError) as e:
        binding.attention_kv(L, L, 2, q, codes, codes, torch.zeros_like(q), 0.1, True)
    assert e.value.status == binding.ERR_INVALID_ARG


def test_opt66b_heads_sampled_rows():
    """72 heads of 128 channels, 2048 tokens, 4-bit cache, causal; sampled (head, query) rows against the oracle
    run on that head and that query alone."""
    import torch
    from paper_2304_01089_b200 import binding
    H, hd, gh, T = 72, 128, 4, 2048
    c = Case(46, H=H, hd=hd, gh=gh, Tq=T, Tk=T, allow_empty=False)
    rng = np.random.default_rng(6)
    q16 = _query(rng, T, H * hd, 0.5)
    out = torch.empty((T, H * hd), dtype=torch.float16, device="cuda")
    binding.attention_kv(c.LK, c.LV, H, torch.from_numpy(q16).cuda(), c.dk, c.dv, out, c.qk_scale, True)
    torch.cuda.synchronize()
    o = out.float().cpu().numpy().astype(np.float64)
    off_k, _ = oracle.segment_offsets(c.size_qk)
    off_v, _ = oracle.segment_offsets(c.size_v)
    ch_k = channel_of_oracle_position(c.perm_qk, c.size_qk)
    ch_v = channel_of_oracle_position(c.perm_v, c.size_v)
    pad = lambda a: np.pad(a, ((0, 0), (0, (-a.shape[1]) % 128)))
    for h, i in [(0, 0), (71, T - 1), (35, 63), (35, 64)] + [(int(rng.integers(H)), int(rng.integers(T))) for _ in range(8)]:
        cl = slice(h * gh, (h + 1) * gh)
        ks = slice(off_k[h * gh], off_k[(h + 1) * gh]); vs = slice(off_v[h * gh], off_v[(h + 1) * gh])
        chk = ch_k[ks] - h * hd                                  # channels of the head, relative; pads stay negative
        chk = np.where(ch_k[ks] >= 0, chk, -1)
        chk = np.pad(chk, (0, (-len(chk)) % 128), constant_values=-1).astype(np.int32)
        want = oracle.attention_kv(q16[i:i + 1, h * hd:(h + 1) * hd].astype(np.float64), chk, pad(c.k[:i + 1, ks]), pad(c.v[:i + 1, vs]),
                                   1, gh, c.size_qk[cl], c.sK[cl].astype(np.float64), c.zK[cl],
                                   c.size_v[cl], c.sV[cl].astype(np.float64), c.zV[cl], c.qk_scale, True)
        chans = ch_v[vs]
        real = chans >= 0
        got, w = o[i, chans[real]], want[0, :vs.stop - vs.start][real]
        vmax = float(c.sV[cl].max()) * 15
        assert np.all(np.abs(got - w) <= 2.0 ** -10 * vmax + 2.0 ** -11 * np.abs(w) + 1e-5 * vmax)


# The kernel for at most eight queries: see test_attention_gpu.py::test_few_queries.
@pytest.mark.parametrize("bits", [(4, 4, 4), (4, 3, 3), (4, 8, 8), (4, 8, 3), (4, 4, 8)])
@pytest.mark.parametrize("Tq,Tk,n_seq,causal", [(1, 31, 1, True), (8, 33, 3, True), (2, 128, 1, False), (8, 1000, 1, True), (1, 2500, 2, True)])
def test_few_queries(Tq, Tk, n_seq, causal, bits):
    c = Case(900 + Tk + 10 * bits[1] + bits[2], H=2, hd=72, gh=4, Tq=Tq * n_seq, Tk=Tk * n_seq, bits=bits)
    _check(c, _query(np.random.default_rng(3), Tq * n_seq, 144), causal, n_seq=n_seq)


# See test_attention_gpu.py::test_few_queries_splits; one or two queries and three or more take different operand types.
@pytest.mark.parametrize("bits", [(4, 4, 4), (4, 3, 8)])
@pytest.mark.parametrize("Tk", [300, 600, 1030])
@pytest.mark.parametrize("Tq", [1, 2, 3, 7])
def test_few_queries_splits(Tq, Tk, bits):
    c = Case(930 + Tk + Tq, H=2, hd=72, gh=4, Tq=Tq, Tk=Tk, bits=bits)
    _check(c, _query(np.random.default_rng(15), Tq, 144), True)


@pytest.mark.parametrize("Tq", [1, 3])
def test_few_queries_of_many_heads_take_one_block_per_head(Tq):
    c = Case(951 + Tq, H=300, hd=16, gh=4, Tq=Tq, Tk=700)
    _check(c, _query(np.random.default_rng(16), Tq, 300 * 16), True)


# The kernel for more queries: see test_attention_gpu.py::test_tile_edges; tiles of 64 keys that two streams take by turns.
@pytest.mark.parametrize("Tq,Tk,n_seq,causal", [(9, 9, 1, True), (64, 65, 1, True), (128, 128, 2, False), (129, 257, 1, True), (200, 400, 1, True)])
@pytest.mark.parametrize("bits", [(4, 4, 4), (4, 3, 8), (4, 8, 3)])
def test_tile_edges(Tq, Tk, n_seq, causal, bits):
    c = Case(700 + Tq + 10 * bits[1] + bits[2], H=2, hd=72, gh=4, Tq=Tq * n_seq, Tk=Tk * n_seq, bits=bits)
    _check(c, _query(np.random.default_rng(7), Tq * n_seq, 144), causal, n_seq=n_seq)


def test_many_items_and_wide_heads():
    c = Case(730, H=90, hd=16, gh=2, Tq=140, Tk=200)
    _check(c, _query(np.random.default_rng(8), 140, 90 * 16), True)
    c = Case(731, H=2, hd=256, gh=1, Tq=130, Tk=140, bits=(4, 8, 8))
    _check(c, _query(np.random.default_rng(9), 130, 512), True)


@pytest.mark.parametrize("hd,Tq", [(36, 140), (20, 129), (8, 256), (136, 140)])
def test_query_rows_of_any_width(hd, Tq):
    """Heads whose rows are whole pieces of 16 bytes are staged and permuted in place, others are gathered channel by channel."""
    c = Case(740 + hd, H=2, hd=hd, gh=2, Tq=Tq, Tk=Tq + 61)
    _check(c, _query(np.random.default_rng(hd), Tq, 2 * hd), True)


def _rebuild_keys(c, bits):
    import torch
    c.dk = torch.from_numpy(oracle.pack(np.ascontiguousarray(c.k[:, c.LK.contiguous_position()]), bits)).cuda()


@pytest.mark.parametrize("Tq", [1, 2, 3])
@pytest.mark.parametrize("q_offset", [300.0, -300.0, 700.0])
def test_scores_far_from_zero(Tq, q_offset):
    """An offset of the query that is the same for every key: the scores as the kernel forms them lie near +-2600 (6000) in units
    of log2 (the row-constant zero-point term is left out), their differences are ordinary. Key positions 2 i and 2 i + 1 hold
    codes that add up to 15."""
    c = Case(60, H=2, hd=64, gh=1, Tq=Tq, Tk=300)
    c.sK[:] = 0.1
    from paper_2304_01089_b200 import binding
    c.LK = binding.Layout(c.perm_qk, c.size_qk, c.sK, c.zK, 4)
    c.k[:, 1::2] = 15 - c.k[:, 0::2]
    _rebuild_keys(c, 4)
    q = q_offset + np.round(4 * np.random.default_rng(11).normal(size=(Tq, 128))) / 4
    _check(c, q.astype(np.float16), True)


@pytest.mark.parametrize("Tq", [1, 2])
def test_scores_far_apart(Tq):
    """Row maxima of a few thousand (in units of log2): one key has all the weight."""
    c = Case(61, H=2, hd=64, gh=1, Tq=Tq, Tk=300)
    _check(c, _query(np.random.default_rng(12), Tq, 128, 1000.0), True)


@pytest.mark.parametrize("Tq", [1, 2, 3])
def test_clusters_of_different_magnitudes(Tq):
    """A head's clusters differ by 10^4 in the query's magnitude and by as much the other way in the keys' scale: the small
    queries count as much as the large ones."""
    from paper_2304_01089_b200 import binding
    c = Case(62, H=2, hd=64, gh=2, Tq=Tq, Tk=300, allow_empty=False)
    c.sK = np.tile(np.array([1e-3, 30.0], np.float32), 2)
    c.LK = binding.Layout(c.perm_qk, c.size_qk, c.sK, c.zK, 4)
    q = np.random.default_rng(13).normal(size=(Tq, 128))
    at = 0
    for cl, n in enumerate(c.size_qk):
        q[:, c.perm_qk[at:at + n]] *= (200.0, 0.02)[cl % 2]
        at += n
    _check(c, q.astype(np.float16), True)


@pytest.mark.parametrize("bits,Tq,Tk", [((4, 8, 3), 8, 24000), ((4, 3, 8), 8, 24000), ((4, 8, 3), 1, 23600)])
def test_few_queries_of_heads_of_eight_units(bits, Tq, Tk):
    """The most shared memory that the kernel for few queries can need: rings for one cache tensor's 8-bit rows, room to expand the
    other's 3-bit rows, and the scores of as many keys as a block may have."""
    c = Case(970 + Tq, H=2, hd=256, gh=1, Tq=Tq, Tk=Tk, bits=bits)
    _check(c, _query(np.random.default_rng(14), Tq, 512, 0.2), True)


@pytest.mark.parametrize("hd,bits,Tq,Tk,n_seq,causal", [(64, (4, 4, 4), 130, 700, 1, True), (64, (4, 4, 4), 200, 200, 2, False), (72, (4, 3, 8), 9, 129, 3, True),
                                                        (256, (4, 8, 8), 130, 330, 1, True)])
def test_scores_that_rise_along_the_keys(hd, bits, Tq, Tk, n_seq, causal):
    """Row maxima that grow by more than 2^8 from tile to tile for some rows, by less for others, and not at all for the rest (one walk
    over the keys: the sums so far are brought to a new reference where that happens). Heads of eight units leave room for one
    tile of probabilities only."""
    rng = np.random.default_rng(15)
    top = (1 << bits[1]) - 1
    c = Case(980 + hd + Tk, H=2, hd=hd, gh=1 if hd == 256 else 2, Tq=Tq * n_seq, Tk=Tk * n_seq, bits=bits)
    ramp = np.tile(np.arange(Tk) / (Tk - 1.0), n_seq)[:, None] * top
    real = np.arange(c.k.shape[1])
    codes = np.clip(np.rint(ramp + 0.05 * top * rng.normal(size=c.k.shape)), 0, top).astype(c.k.dtype)
    off, _ = oracle.segment_offsets(c.size_qk)
    for cl, n in enumerate(c.size_qk):
        at = real[off[cl]:off[cl] + n]
        c.k[:, at] = codes[:, at]
    _rebuild_keys(c, bits[1])
    step = float(np.dot(c.size_qk, c.sK)) / 2 * top * c.qk_scale          # what a query of ones gains from the first key to the last
    rise = rng.choice([-300.0, -20.0, 0.0, 3.0, 12.0, 60.0, 300.0], size=(Tq * n_seq, 1)) / step
    _check(c, (rise * (1 + 0.1 * rng.normal(size=(Tq * n_seq, 2 * hd)))).astype(np.float16), causal, n_seq=n_seq)


def _rising(seed, H, hd, Tq, Tk, n_seq, bits):
    """A case whose keys' codes grow from the first key of a sequence to the last, and queries of which some gain hundreds of powers of two on
    the way, some a few, some nothing."""
    rng = np.random.default_rng(seed)
    top = (1 << bits[1]) - 1
    c = Case(seed, H=H, hd=hd, gh=1 if hd == 256 else 2, Tq=Tq * n_seq, Tk=Tk * n_seq, bits=bits)
    ramp = np.tile(np.arange(Tk) / (Tk - 1.0), n_seq)[:, None] * top
    off, _ = oracle.segment_offsets(c.size_qk)
    for cl, n in enumerate(c.size_qk):
        sl = slice(off[cl], off[cl] + n)
        c.k[:, sl] = np.clip(np.rint(ramp + 0.1 * top * rng.normal(size=(Tk * n_seq, n))), 0, top)
    _rebuild_keys(c, bits[1])
    step = float(np.dot(c.size_qk, c.sK)) / H * top * c.qk_scale
    rise = rng.choice([-100.0, -5.0, 0.0, 1.5, 6.0, 40.0, 200.0], size=(Tq * n_seq, 1)) / step
    return c, (rise * (1 + 0.3 * rng.normal(size=(Tq * n_seq, H * hd)))).astype(np.float16)


def _outputs(c, q16, causal, n_seq=1, Tk=None):
    """fp16 [rows of q16][C]: these queries on the case's cache, or on its first Tk keys."""
    import torch
    from paper_2304_01089_b200 import binding
    Tq, Tk = q16.shape[0] // n_seq, Tk or c.Tk // n_seq
    out = torch.full((q16.shape[0], c.H * c.hd), 7.0, dtype=torch.float16, device="cuda")
    binding.attention_kv(c.LK, c.LV, c.H, torch.from_numpy(np.ascontiguousarray(q16)).cuda(), c.dk, c.dv, out, c.qk_scale,
                         causal, Tq=Tq, Tk=Tk, n_seq=n_seq)
    torch.cuda.synchronize()
    assert binding.get_device_status() == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("hd,bits", [(64, (4, 4, 4)), (256, (4, 8, 8))])
def test_a_row_depends_on_nothing_but_itself_and_its_keys(hd, bits):
    """The same bits whatever the other queries of the block are (other magnitudes, infinite ones among them), and whether a prompt comes
    whole or in chunks, whose rows lie elsewhere in their blocks and see other tiles hidden."""
    Tq, Tk = 300, 700
    c, q = _rising(990 + hd, 2, hd, Tq, Tk, 1, bits)
    whole = _outputs(c, q, True)
    assert np.isfinite(whole).all()
    rng = np.random.default_rng(17)
    others = (q * rng.choice([0.0, 0.3, 3.0], size=(Tq, 1))).astype(np.float16)
    others[::11] = np.inf
    keep = np.arange(Tq) % 5 == 2
    others[keep] = q[keep]
    np.testing.assert_array_equal(_outputs(c, others, True)[keep].view(np.uint16), whole[keep].view(np.uint16))
    cuts = [0, 40, 57, 190, 213, Tq]
    for lo, hi in zip(cuts, cuts[1:]):
        part = _outputs(c, q[lo:hi], True, Tk=Tk - Tq + hi)
        np.testing.assert_array_equal(part.view(np.uint16), whole[lo:hi].view(np.uint16))


@pytest.mark.parametrize("H,hd,bits,Tq,Tk,n_seq", [(12, 16, (4, 4, 4), 300, 330, 14), (12, 16, (4, 4, 4), 250, 390, 20), (4, 256, (4, 8, 8), 300, 330, 40),
                                                   (24, 16, (4, 4, 4), 50, 60, 24)])
def test_blocks_with_several_items_of_rising_scores(H, hd, bits, Tq, Tk, n_seq):
    """Three items and more to every block, of which one prompt's have odd and even numbers of key tiles (or one tile each): the state that a block
    carries from item to item (barrier phases, two sets of references) against calls of one prompt, whose blocks have one item.
    Heads of 256 channels leave room for one tile of probabilities only."""
    import torch
    per_prompt = H * ((Tq + 127) // 128)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert per_prompt <= sms and per_prompt * n_seq >= 3 * sms
    c, q = _rising(1200 + hd + Tk, H, hd, Tq, Tk, n_seq, bits)
    whole = _outputs(c, q, True, n_seq=n_seq)
    k, v = c.dk, c.dv
    for s in range(n_seq):
        c.dk, c.dv = k[s * Tk:(s + 1) * Tk], v[s * Tk:(s + 1) * Tk]
        alone = _outputs(c, q[s * Tq:(s + 1) * Tq], True, Tk=Tk)
        np.testing.assert_array_equal(whole[s * Tq:(s + 1) * Tq].view(np.uint16), alone.view(np.uint16))
    c.dk, c.dv = k, v
    if hd == 16:
        _check(c, q, True, n_seq=n_seq)
