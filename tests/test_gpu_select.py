"""adapshot_select vs the fp64 oracle: indices bit-exact (ties -> lowest shot id)."""
import numpy as np
import pytest
import torch

from oracle import adapshot_oracle as orc
from paper_2605_03644_b200 import workloads as wl
from tests import helpers as hp

pytestmark = pytest.mark.gpu


def _check(ab, emb, q_emb, k):
    so = torch.arange(emb.shape[0] + 1, dtype=torch.int64, device="cuda")
    pool = ab.Pool(so, None, None, emb.cuda().contiguous())
    sel, score, st = hp.run_select(ab, pool, q_emb, k)
    want, want_sc = orc.select_topk(hp.f64(q_emb), hp.f64(emb), k)
    assert st == 0
    assert np.array_equal(sel.cpu().numpy(), want), "top-k indices must be bit-exact"
    assert np.allclose(score.cpu().numpy(), want_sc, atol=1e-6)


@pytest.mark.parametrize("name", ["cfg1", "cfg2", "cfg3", "cfg5"])
def test_select_matches_oracle_on_the_configs(name):
    ab = hp.gpu_binding()
    w = wl.CONFIGS[name]
    g = torch.Generator().manual_seed(w.seed)
    emb = torch.randn(w.n_shots, w.emb_dim, generator=g)
    emb = emb / emb.norm(dim=1, keepdim=True)
    q = torch.randn(w.batch, w.emb_dim, generator=g)
    q = q / q.norm(dim=1, keepdim=True)
    assert orc.min_adjacent_gap(hp.f64(q), hp.f64(emb), w.k) > 1e-12
    _check(ab, emb, q, w.k)


@pytest.mark.parametrize("N,E,B,k", [(1, 4, 1, 1), (5, 3, 2, 5), (33, 130, 3, 7), (1000, 64, 2, 1000),
                                     (8192, 16, 1, 8192), (8193, 16, 2, 100), (20000, 32, 2, 4096)])
def test_select_edge_shapes(N, E, B, k):
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(N + E)
    _check(ab, torch.randn(N, E, generator=g), torch.randn(B, E, generator=g), k)


def test_select_ties_and_zero_norm():
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(5)
    emb = torch.randn(300, 64, generator=g)
    emb[200] = emb[7]; emb[100] = emb[7]; emb[250] = emb[7]     # exact duplicates
    emb[13] = 0.0                                              # zero norm -> score 0
    emb[40:60] = emb[40]                                       # a run of equal rows
    q = torch.cat([emb[7:8], emb[40:41], torch.randn(1, 64, generator=g)])
    _check(ab, emb, q, 300)
    _check(ab, emb, q, 5)
    sel, _, _ = hp.run_select(ab, ab.Pool(torch.arange(301, device="cuda"), None, None, emb.cuda()), q, 4)
    assert sel[0].tolist() == [7, 100, 200, 250]
    assert sel[1, :4].tolist() == [40, 41, 42, 43]


@pytest.mark.parametrize("k", [1, 33, 128, 512, 1000])
@pytest.mark.parametrize("copies", [1, 31, 33, 127, 129, 700])       # below and above what a bin of candidates may hold; more than k of them
def test_select_by_bins_and_by_sorting(copies, k):
    # a pool large enough for the selection, whose best shots are copies of one another and whose scores span many octaves
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(copies + k)
    emb = torch.randn(9000, 32, generator=g)
    q = torch.randn(4, 32, generator=g)
    emb[:3000] += 3.0 * q[0]
    at = torch.randperm(9000, generator=g)[:copies]
    emb[at] = q[0] + 0.01 * torch.randn(32, generator=g)
    _check(ab, emb, q, k)


def test_nested_probes_are_prefixes():
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(6)
    emb, q = torch.randn(500, 32, generator=g), torch.randn(2, 32, generator=g)
    pool = ab.Pool(torch.arange(501, device="cuda"), None, None, emb.cuda())
    full, _, _ = hp.run_select(ab, pool, q, 128)
    for n in (1, 16, 64):
        part, _, _ = hp.run_select(ab, pool, q, n)
        assert torch.equal(part, full[:, :n])


@pytest.mark.parametrize("N,E,B,k", [(33, 16, 3, 33), (97, 48, 8, 13), (3001, 64, 9, 1500), (4096, 768, 17, 1025),
                                     (8192, 32, 4, 5000), (9000, 112, 33, 1024), (2048, 64, 32, 1000), (2100, 32, 16, 1024)])
def test_select_batches(N, E, B, k):
    # fp64 matrix tiles: remainders of 32 shots, 8 and 16 queries, embeddings of one step, of fewer steps than warps
    # and of unequal shares; rank counting and radix selection with few and with many candidates; k beyond the
    # positive scores (half of them are)
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(N + E)
    _check(ab, torch.randn(N, E, generator=g), torch.randn(B, E, generator=g), k)


@pytest.mark.parametrize("n_same,k", [(6000, 700), (6000, 1500), (1025, 900)])
def test_radix_selection_cuts_equal_scores_by_id(n_same, k):
    # more equal scores around rank k than the candidate area takes, in front of them a few better ones
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(n_same)
    emb = torch.randn(6100, 32, generator=g)
    same = torch.randperm(6100, generator=g)[:n_same]
    emb[same] = emb[same[0]].clone()
    _check(ab, emb, torch.cat([emb[same[:1]] + 0.3 * torch.randn(1, 32, generator=g), torch.randn(2, 32, generator=g)]), k)
    zero = torch.zeros(6100, 32)
    zero[17], zero[5000] = 1.0, -1.0
    _check(ab, zero, torch.ones(1, 32), k)


@pytest.mark.parametrize("N,B,k", [(2, 1, 2), (31, 2, 31), (2047, 1, 2047), (2049, 1, 300), (3741, 1, 3741), (3742, 1, 3742)])
def test_rank_counting_with_ties(N, B, k):
    # odd and even counts (a last pair of one key), one and two tiles of keys; every embedding occurs about three times, so that equal scores lie in front of and behind each other
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(N)
    base = torch.randn((N + 2) // 3, 32, generator=g)
    emb = base[torch.randint(0, base.shape[0], (N,), generator=g)]
    _check(ab, emb, torch.randn(B, 32, generator=g), k)


@pytest.mark.parametrize("N,B,k", [(3751, 1, 64), (3752, 1, 64), (6100, 1, 600), (6400, 1, 600), (8192, 1, 4096), (8192, 3, 4096),
                                   (4171, 1, 64), (4172, 1, 64), (5160, 1, 600), (5161, 1, 600), (5401, 1, 1024), (5402, 1, 1024),
                                   (7758, 1, 1025), (7759, 1, 1025)])
def test_both_sides_of_the_line_between_counting_and_selection(N, B, k):
    # N^2 B against 11 million and what k adds, up to 1024 and beyond; every embedding occurs about three times
    ab = hp.gpu_binding()
    g = torch.Generator().manual_seed(N + B)
    base = torch.randn((N + 2) // 3, 32, generator=g)
    emb = base[torch.randint(0, base.shape[0], (N,), generator=g)]
    _check(ab, emb, torch.randn(B, 32, generator=g), k)
