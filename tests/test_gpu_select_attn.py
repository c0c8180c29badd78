"""adapshot_select_attn (the paper's attention-based relevance ranking, Sec. 4.2) against the oracle's
relevance_attention: scores within 1e-3 relative (bf16 inputs are shared; the differences are fp32
accumulation and the exponential), indices bit-exact wherever the oracle's scores are further apart
than that, ties by the lower shot id."""
import numpy as np
import pytest
import torch

from oracle import adapshot_oracle as orc
from paper_2605_03644_b200 import workloads as wl
from tests import helpers as hp

pytestmark = pytest.mark.gpu
SCORE_REL = 1e-3


def _run(ab, model, dp, layer, q, k, per_token=False):
    B = q.shape[0]
    sel = torch.full((B, k), -1, dtype=torch.int32, device="cuda")
    score = torch.zeros((B, k), dtype=torch.float32, device="cuda")
    ws = torch.empty(max(256, ab.adapshot_select_attn_workspace_bytes(model, dp, B, q.shape[1], k)), dtype=torch.uint8,
                     device="cuda")
    st = hp.new_status()
    ab.adapshot_select_attn(model, dp, layer, q.cuda(), k, sel, score, ws, st, per_token=per_token)
    torch.cuda.synchronize()
    assert st.item() == 0
    return sel.cpu().numpy(), score.cpu().numpy()


def _check(w, nl, layer, k, per_token=False, q_gain=1.0):
    ab = hp.gpu_binding()
    pool = wl.make_pool(w, n_layers=nl)
    qs = wl.make_queries(w, n_layers=nl, n_probes=1)
    q = (qs["q"][:, layer, 0].float() * q_gain).to(torch.bfloat16).contiguous()      # [B][T_q][Hq][d] as stored
    dp = hp.dev_pool(ab, pool)
    model = hp.model_of(ab, w, n_layers=nl)
    sel, score = _run(ab, model, dp, layer, q, k, per_token)
    k_layer = hp.f64(pool["k"][layer])
    for b in range(w.batch):
        s = orc.relevance_attention(hp.f64(q[b]), k_layer, pool["shot_off"], per_token=per_token)
        # scores of the shots the kernel chose, against the oracle's values for those shots
        assert np.all(np.abs(score[b] - s[sel[b]]) <= SCORE_REL * np.abs(s[sel[b]]) + 1e-30), b
        # the choice itself: the oracle's order, up to pairs the tolerance cannot tell apart
        order = np.argsort(-s, kind="stable")
        assert len(set(sel[b].tolist())) == k
        for r in range(k):
            if sel[b, r] != order[r]:
                assert abs(s[sel[b, r]] - s[order[r]]) <= 2 * SCORE_REL * abs(s[order[r]]), (b, r)
        # nothing better was left out: the weakest chosen shot is within the tolerance of rank k
        assert s[sel[b]].min() >= s[order[k - 1]] * (1 - 2 * SCORE_REL)
    return sel, score


def test_tiny_pool_one_tile():
    w = wl.CONFIGS["cfg1"].scaled(dtype="bf16", n_shots=12, len_lo=5, len_hi=5, t_q=7, seed=81)
    _check(w, 1, 0, 5)


def test_8b_shape_many_tiles_and_splits():
    # 8B head shape, 96 shots of 30-200 tokens (about 11 K pool tokens: 86 key tiles, several ranges per unit),
    # T_q * G = 192 rows: two M tiles, the second half empty; the third of three layers is the representative one
    w = wl.CONFIGS["cfg2"].scaled(n_shots=96, len_lo=30, len_hi=200, batch=2, k=24, t_q=48, seed=82)
    _check(w, 3, 2, 24)
    _check(w, 3, 2, 24, per_token=True)


def test_head_dim_64_group_of_three_and_one_token_shots():
    w = wl.CONFIGS["cfg2"].scaled(n_shots=300, len_lo=1, len_hi=9, batch=3, k=300, t_q=5, head_dim=64, n_q_heads=6,
                                  n_kv_heads=2, seed=83)
    _check(w, 1, 0, 300)


def test_peaked_queries_single_out_their_shot():
    # queries five times larger: the softmax over the pool concentrates on a few keys
    w = wl.CONFIGS["cfg2"].scaled(n_shots=64, len_lo=20, len_hi=90, batch=2, k=8, t_q=16, seed=84)
    sel, score = _check(w, 1, 0, 8, q_gain=5.0)
    assert (score[:, 0] > 1.5 / 64).all()                 # well above the uniform share of 1 / 64


def test_identical_shots_get_equal_masses():
    # a pool made of one shot repeated: every shot gets the same mass (the order among them is decided by the
    # last bits of the fp64 sums, which depend on how the keys fall into warps: only exact ties go by shot id,
    # and that rule is the top-k kernel's, tested with the embedding selector)
    ab = hp.gpu_binding()
    w = wl.CONFIGS["cfg2"].scaled(n_shots=1, len_lo=17, len_hi=17, batch=1, k=1, t_q=8, seed=85)
    pool = wl.make_pool(w, n_layers=1)
    n_rep = 9
    pool["k"] = pool["k"].repeat(1, n_rep, 1, 1).contiguous()
    pool["v"] = pool["v"].repeat(1, n_rep, 1, 1).contiguous()
    pool["shot_off"] = np.arange(n_rep + 1, dtype=np.int64) * 17
    pool["emb"] = pool["emb"].repeat(n_rep, 1).contiguous()
    qs = wl.make_queries(w, n_layers=1, n_probes=1)
    q = qs["q"][:, 0, 0].contiguous()
    dp = hp.dev_pool(ab, pool)
    sel, score = _run(ab, hp.model_of(ab, w, n_layers=1), dp, 0, q, n_rep)
    assert np.allclose(score, 1.0 / n_rep, rtol=1e-4)
    assert sorted(sel[0].tolist()) == list(range(n_rep))


@pytest.mark.parametrize("lens,n_shots,t_q,batch", [((128, 128), 40, 3, 1), ((1, 1), 700, 2, 2), ((15, 17), 130, 33, 1),
                                                   ((900, 1100), 9, 1, 3)])
def test_masses_per_shot_at_tile_and_range_edges(lens, n_shots, t_q, batch):
    # shots that end with the 128-key tiles, shots of one key, shots around the 16-key groups, shots that span several
    # ranges of keys
    w = wl.CONFIGS["cfg2"].scaled(n_shots=n_shots, len_lo=lens[0], len_hi=lens[1], batch=batch, k=n_shots, t_q=t_q,
                                  n_q_heads=8, n_kv_heads=2, seed=86)
    _check(w, 1, 0, n_shots)


def test_rows_in_several_batches():
    # 8 KV heads, 20000 one-token shots: a tile of 128 rows leaves 82 MB of pieces, so the four M tiles go two by two:
    # each query's two tiles apart from the other's
    w = wl.CONFIGS["cfg2"].scaled(n_shots=20000, len_lo=1, len_hi=1, batch=2, k=64, t_q=40, n_q_heads=32, n_kv_heads=8,
                                  head_dim=64, seed=87)
    _check(w, 1, 0, 64)


def test_a_query_whose_rows_are_cut_by_a_batch():
    # as above with three M tiles per query: batches of two tiles, so a query's masses are summed over two launches
    w = wl.CONFIGS["cfg2"].scaled(n_shots=24000, len_lo=1, len_hi=1, batch=1, k=64, t_q=70, n_q_heads=32, n_kv_heads=8,
                                  head_dim=64, seed=88)
    _check(w, 1, 0, 64)


@pytest.mark.parametrize("t_q,batch", [(200, 1), (20, 2), (64, 1), (100, 3)])
def test_m_tiles_and_ranges_per_cta(t_q, batch):
    # 7 M tiles (two CTAs of four, one place empty), 2 M tiles (they share a CTA with two ranges), 2 and 12
    w = wl.CONFIGS["cfg2"].scaled(n_shots=70, len_lo=10, len_hi=120, batch=batch, k=30, t_q=t_q, n_q_heads=8,
                                  n_kv_heads=2, seed=89)
    _check(w, 1, 0, 30)


def _scores_and_masses(gain, t_q):
    """Keys and queries that lean towards a common direction: logits of about ten times the gain with many shots close to
    the largest.  Returns the call's scores and the oracle's, in the call's order."""
    ab = hp.gpu_binding()
    w = wl.CONFIGS["cfg2"].scaled(n_shots=200, len_lo=16, len_hi=80, batch=1, k=200, t_q=t_q, n_q_heads=8, n_kv_heads=2,
                                  channel_scale=False, seed=90)
    pool, qs = wl.make_pool(w, n_layers=1), wl.make_queries(w, n_layers=1, n_probes=1)
    lean = torch.nn.functional.normalize(torch.randn(2, 128, generator=torch.Generator().manual_seed(3)), dim=1)
    pool["k"] = (pool["k"].float() + 8.0 * lean).to(torch.bfloat16)
    q = (qs["q"][:, 0, 0].float() + 8.0 * gain * lean.repeat_interleave(4, 0)).to(torch.bfloat16).contiguous()
    sel, score = _run(ab, hp.model_of(ab, w, n_layers=1), hp.dev_pool(ab, pool), 0, q, 200)
    s = orc.relevance_attention(hp.f64(q[0]), hp.f64(pool["k"][0]), pool["shot_off"])
    return score[0], s[sel[0]]


@pytest.mark.parametrize("t_q", [8, 40])
def test_masses_of_peaked_rows(t_q):
    # Logits of about 40.  The exponentials are good to 2.6e-6 and so is the normaliser; a score of 40 / ln 2 = 58 carries an
    # fp32 sum's rounding, 2^-24 * 58 = 3.4e-6 at a time.  (Seen: 4e-7 of the norm.)
    score, want = _scores_and_masses(4.0, t_q)
    assert np.linalg.norm(score - want) <= 5e-6 * np.linalg.norm(want)


@pytest.mark.parametrize("big", [0.0, 128.0])
def test_masses_do_not_carry_the_rounding_of_large_scores(big):
    # whole numbers, so that the scores are exact; with big = 128 all of them are 2048 larger, which the masses must not show:
    # the exponentials (2.6e-6) are all that is rounded
    ab = hp.gpu_binding()
    w = wl.CONFIGS["cfg2"].scaled(n_shots=150, len_lo=16, len_hi=40, batch=1, k=150, t_q=6, n_q_heads=4, n_kv_heads=2,
                                  head_dim=64, seed=91)
    pool = wl.make_pool(w, n_layers=1)
    g = torch.Generator().manual_seed(4)
    pool["k"] = torch.randint(-1, 2, pool["k"].shape, generator=g).to(torch.bfloat16)
    q = torch.randint(-2, 3, (1, 6, 4, 64), generator=g).to(torch.bfloat16)
    pool["k"][..., 0], q[..., 0] = big, big
    sel, score = _run(ab, hp.model_of(ab, w, n_layers=1), hp.dev_pool(ab, pool), 0, q, 150)
    s = orc.relevance_attention(hp.f64(q[0]), hp.f64(pool["k"][0]), pool["shot_off"])
    assert np.all(np.abs(score[0] - s[sel[0]]) <= 3e-6 * s[sel[0]])


@pytest.mark.parametrize("batch,t_q", [(1, 3), (2, 130)])
def test_many_shots_of_one_token(batch, t_q):
    # 66000 shots of one token: two passes, all heads at once; two M tiles per query at 130 tokens
    w = wl.CONFIGS["cfg2"].scaled(n_shots=66000, len_lo=1, len_hi=1, batch=batch, k=32, t_q=t_q, n_q_heads=8,
                                  n_kv_heads=8, head_dim=64, emb_dim=8, seed=92)
    _check(w, 1, 0, 32)


@pytest.mark.parametrize("n_shots,lens,t_q,batch", [(5, (40, 70), 300, 1), (64, (16, 48), 17, 2), (700, (100, 140), 3, 1)])
def test_warps_per_shot_and_many_ranges(n_shots, lens, t_q, batch):
    # eight warps per shot over nineteen M tiles, over one, and more ranges than a thread of the merge takes at a time
    w = wl.CONFIGS["cfg2"].scaled(n_shots=n_shots, len_lo=lens[0], len_hi=lens[1], batch=batch, k=n_shots, t_q=t_q, n_q_heads=8,
                                  n_kv_heads=1, seed=93)
    _check(w, 1, 0, n_shots)


@pytest.mark.parametrize("lens,n_shots,t_q,batch,hq,hkv", [
    ((11, 11), 300, 33, 2, 8, 2),       # just below the line of twelve tokens: two passes; K tiles two by two
    ((12, 12), 300, 33, 2, 8, 2),       # on it: one pass
    ((1, 6), 9000, 40, 3, 8, 8),        # every CTA keeps four K tiles; two M tiles per query; queries in parts
    ((1, 3), 50, 5, 1, 4, 1),           # one K tile
    ((1, 40), 200, 150, 1, 8, 1),       # nineteen M tiles of one query in front of 32 K tiles
])
def test_short_shots(lens, n_shots, t_q, batch, hq, hkv):
    w = wl.CONFIGS["cfg2"].scaled(n_shots=n_shots, len_lo=lens[0], len_hi=lens[1], batch=batch, k=min(n_shots, 50), t_q=t_q,
                                  n_q_heads=hq, n_kv_heads=hkv, head_dim=64 if hkv == 8 else 128, seed=94)
    _check(w, 1, 0, w.k)


def test_short_shots_with_queries_in_batches():
    # 210 K keys x 8 heads x 4 bytes: 39 queries at a time, so 40 queries go as two times twenty; those at the seam and the ends
    ab = hp.gpu_binding()
    w = wl.CONFIGS["cfg2"].scaled(n_shots=42000, len_lo=5, len_hi=5, batch=40, k=64, t_q=1, n_q_heads=8, n_kv_heads=8,
                                  head_dim=64, emb_dim=8, seed=95)
    pool, qs = wl.make_pool(w, n_layers=1), wl.make_queries(w, n_layers=1, n_probes=1)
    q = qs["q"][:, 0, 0].contiguous()
    sel, score = _run(ab, hp.model_of(ab, w, n_layers=1), hp.dev_pool(ab, pool), 0, q, 64)
    k_layer = hp.f64(pool["k"][0])
    for b in (0, 19, 20, 39):
        s = orc.relevance_attention(hp.f64(q[b]), k_layer, pool["shot_off"])
        assert np.all(np.abs(score[b] - s[sel[b]]) <= SCORE_REL * s[sel[b]])
        assert s[sel[b]].min() >= np.sort(s)[-64] * (1 - 2 * SCORE_REL)


@pytest.mark.parametrize("n_shots,t_q,hq,hkv", [
    (66000, 2, 8, 8),                   # the pieces of one M tile are more than 256 MB: the KV heads go four by four
    (4000, 550, 32, 8),                 # eighteen M tiles of one query in two batches
])
def test_pieces_in_batches(n_shots, t_q, hq, hkv):
    w = wl.CONFIGS["cfg2"].scaled(n_shots=n_shots, len_lo=12, len_hi=12, batch=1, k=32, t_q=t_q, n_q_heads=hq, n_kv_heads=hkv,
                                  head_dim=64, emb_dim=8, seed=96)
    _check(w, 1, 0, 32)
