"""ReusePath.run: what it reads and writes is what the object and the call hold at that moment."""
import ctypes

import pytest
import torch

from paper_2605_03644_b200 import workloads as wl
from tests import helpers as hp

pytestmark = pytest.mark.gpu

VARIANTS = {"full": dict(vpool=False), "vpool": dict(vpool=True), "fused": dict(fused=True, vpool=False)}
BUFFERS = ("sel_idx", "sel_score", "ctx_off", "H", "first_ok", "status", "ws_select", "ws_attn", "ws_entropy")


def _workload(seed):
    return wl.CONFIGS["cfg2"].scaled(n_layers=3, n_q_heads=4, n_kv_heads=2, n_shots=20, len_lo=20, len_hi=20, len_dist="const",
                                     batch=3, k=6, probes=(2, 6), t_q=9, vocab=1000, emb_dim=64, seed=seed)


def _path(w, variant, **kw):
    from paper_2605_03644_b200 import binding as ab
    from paper_2605_03644_b200.pipeline import ReusePath
    pool = hp.dev_pool(ab, wl.make_pool(w))
    return ReusePath(hp.model_of(ab, w), pool, w.batch, w.k, w.probes, w.t_q, w.vocab, w.k * w.len_hi, 2, **VARIANTS[variant], **kw)


def _inputs(path, qs):
    chunk = lambda x: [x[:, lb:le].contiguous().cuda() for lb, le in path.chunks]
    return qs["q_emb"].cuda(), chunk(qs["q"]), chunk(qs["kq"]), chunk(qs["vq"]), qs["logits"].cuda(), 6.0


@pytest.mark.parametrize("variant", VARIANTS)
def test_a_pass_uses_the_tensors_and_the_pool_it_has_now(variant):
    w, other = _workload(41), _workload(42)
    path, fresh = _path(w, variant), _path(other, variant)
    args = _inputs(path, wl.make_queries(w))
    path.run(*args)
    want_out, want_H, want_ok = ([t.clone() for t in fresh.run(*args)[0]], fresh.H.clone(), fresh.first_ok.clone())
    torch.cuda.synchronize()
    # everything the object holds is replaced, the pool among it
    held = {name: getattr(path, name) for name in BUFFERS}
    held.update({f"{name}[{i}]": t for name in ("k_bufs", "v_bufs", "out") for i, t in enumerate(getattr(path, name))})
    for name in BUFFERS:
        setattr(path, name, torch.zeros_like(held[name]))
    for name in ("k_bufs", "v_bufs", "out"):
        setattr(path, name, [torch.zeros_like(t) for t in getattr(path, name)])
    path.pool, path.model = fresh.pool, fresh.model
    before = {name: t.clone() for name, t in held.items()}
    out, H, ok = path.run(*args)
    torch.cuda.synchronize()
    assert path.status.item() == 0 and fresh.status.item() == 0
    assert H is path.H and ok is path.first_ok and torch.equal(H, want_H) and torch.equal(ok, want_ok)
    assert torch.equal(path.sel_idx, fresh.sel_idx) and torch.equal(path.ctx_off, fresh.ctx_off)
    assert all(torch.equal(a, b) for a, b in zip(out, want_out))
    for name, t in held.items():
        assert torch.equal(t, before[name]), name
    # probes are read at the call, too
    path.probes = fresh.probes = [1, 5]
    a, b = path.run(*args)[0], fresh.run(*args)[0]
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b)) and not any(torch.equal(x, y) for x, y in zip(a, want_out))


@pytest.mark.parametrize("lens", [(20, 20), (90, 150)])
@pytest.mark.parametrize("variant", VARIANTS)
def test_what_unselected_shots_hold_does_not_matter(variant, lens):
    # contexts that end within a 128-key tile, in a pool whose other shots are not numbers (slots that nothing has
    # filled yet, for instance)
    w = _workload(43).scaled(len_lo=lens[0], len_hi=lens[1], len_dist="uniform")
    path = _path(w, variant)
    args = _inputs(path, wl.make_queries(w))
    want = [t.clone() for t in path.run(*args)[0]]
    shot_off, chosen = path.pool.shot_off.tolist(), set(path.sel_idx.flatten().tolist())
    assert len(chosen) < w.n_shots
    for i in range(w.n_shots):
        if i not in chosen:
            path.pool.k[:, shot_off[i]:shot_off[i + 1]] = float("nan")
            path.pool.v[:, shot_off[i]:shot_off[i + 1]] = float("inf") if i % 2 else float("nan")
    got = path.run(*args)[0]
    torch.cuda.synchronize()
    assert path.status.item() == 0
    assert all(torch.isfinite(b).all() and torch.equal(a, b) for a, b in zip(want, got))


@pytest.mark.parametrize("overlap", [dict(), dict(entropy_overlap=True)])
@pytest.mark.parametrize("variant", VARIANTS)
def test_fewer_and_shorter_queries_than_planned(variant, overlap):
    # two of three queries, five of nine tokens: what a path planned for just that gives
    w = _workload(44)
    small = w.scaled(batch=2, t_q=5)
    path, fresh = _path(w, variant, **overlap), _path(small, variant)
    path.run(*_inputs(path, wl.make_queries(w)))              # (every query has a selection)
    args = _inputs(fresh, wl.make_queries(small))
    out, H, ok = path.run(*args)
    want_out, want_H, want_ok = fresh.run(*args)
    torch.cuda.synchronize()
    assert path.status.item() == 0 and fresh.status.item() == 0
    assert torch.equal(path.sel_idx[:2], fresh.sel_idx) and torch.equal(path.ctx_off[:2], fresh.ctx_off)
    assert all(torch.equal(a.flatten()[:b.numel()], b.flatten()) for a, b in zip(out, want_out))
    assert torch.equal(H[:want_H.numel()], want_H) and torch.equal(ok[:2], want_ok)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("vocab", [7, 1000, 20003])          # less than a vector, one slice per row, several with a ragged tail
@pytest.mark.parametrize("variant", VARIANTS)
def test_entropy_beside_the_attention_equals_its_own_call(variant, vocab, dtype):
    # own workspaces: beside the attention; one workspace for every step: after it, as calls in turn would have it
    w = _workload(47).scaled(vocab=vocab, t_q=70)
    path, steps = _path(w, variant), _path(w, variant)
    args = list(_inputs(path, wl.make_queries(w)))
    stride = -(-vocab // 8) * 8
    args[4] = torch.nn.functional.pad(args[4].to(dtype), (0, stride - vocab))[:, :vocab]
    tau = 0.9 * torch.log(torch.tensor(float(vocab))).item()
    steps.select(args[0])
    if variant == "fused":
        steps.plan()
    for i, (lb, le) in enumerate(steps.chunks):
        if variant == "fused":
            steps.attend_fused(args[1][i], args[2][i], args[3][i], steps.out[i], lb, le)
        else:
            steps.assemble(lb, le, keep_plan=i > 0)
            steps.attend(args[1][i], args[2][i], args[3][i], steps.out[i], lb, le)
    steps.entropy(args[4], tau)
    for shared in (False, True):
        if shared:
            path.ws_entropy = path.ws_select = path.ws_attn
        path.H.fill_(-1)
        path.first_ok.fill_(-7)
        out, H, ok = path.run(*args[:5], tau)
        torch.cuda.synchronize()
        assert path.status.item() == 0 and steps.status.item() == 0
        assert torch.equal(H, steps.H) and torch.equal(ok, steps.first_ok)
        assert all(torch.equal(a, b) for a, b in zip(out, steps.out))


@pytest.mark.parametrize("batch,t_q", [(1, 9), (4, 9), (5, 9), (13, 40)])      # one column of the merge's grid holds 4 queries, or 8
def test_every_query_of_a_pass_has_its_entropy(batch, t_q):
    w = _workload(52).scaled(batch=batch, t_q=t_q)
    path = _path(w, "full")
    args = _inputs(path, wl.make_queries(w))
    p = torch.softmax(args[4].double(), 1)
    want = -(p * p.log()).sum(1)
    tau = float(want.view(batch, -1).max(1).values.median()) + 1e-4
    path.H.fill_(-1)
    path.first_ok.fill_(-7)
    _, H, ok = path.run(*args[:5], tau)
    torch.cuda.synchronize()
    torch.testing.assert_close(H.double(), want, rtol=1e-5, atol=1e-5)
    good = (H <= tau).view(batch, -1)
    assert torch.equal(ok, torch.where(good.any(1), good.int().argmax(1), -1).int())


def _launches(path, args):
    """Kernels of one pass, counted in a captured graph."""
    path.run(*args)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        path.run(*args)
    n = ctypes.c_size_t()
    assert ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("variant", VARIANTS)
def test_entropy_has_launches_of_its_own_only_where_it_has_to(variant):
    # two chunks of layers: scores, top-k, per chunk (gather,) preparation, attention and merge; the fused form has a plan instead
    w = _workload(49)
    path = _path(w, variant)
    args = _inputs(path, wl.make_queries(w))
    beside = 2 + (1 + 2 * 3 if variant == "fused" else 1 + 2 * 4)
    assert _launches(path, args) == beside
    # a tensor of the entropy step in memory that the last attention call reads or writes: the calls in turn
    shared = {"ws_attn": path.ws_attn, "out": path.out[-1], "q": args[1][-1], "kq": args[2][-1], "vq": args[3][-1],
              "sel_idx": path.sel_idx, "ctx_off": path.ctx_off}
    if variant != "fused":
        shared["k_ctx"] = path.k_bufs[0]
    if variant == "full":
        shared["v_ctx"] = path.v_bufs[0]
    for name, n_bytes in (("H", 4), ("first_ok", 4), ("ws_entropy", 256)):
        own = getattr(path, name)
        for where, memory in shared.items():
            room = memory.flatten().view(torch.uint8)
            if room.numel() < max(n_bytes, own.nbytes):
                continue
            setattr(path, name, room[:own.nbytes].view(own.dtype))
            assert _launches(path, args) == beside + 2, (name, where)
        setattr(path, name, own)
    assert _launches(path, args) == beside


@pytest.mark.parametrize("vocab,own", [(699048, 0), (699056, 2)])          # 16 MB of logits less 64 bytes, and 128 bytes more
def test_entropy_of_large_logits_comes_after_the_attention(vocab, own):
    w = _workload(50).scaled(vocab=8)
    path = _path(w, "full")
    path.ws_entropy = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    args = list(_inputs(path, wl.make_queries(w)))
    args[4] = torch.randn(w.batch * len(w.probes), vocab, generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    assert _launches(path, args) == 11 + own
    p = torch.softmax(args[4].double(), 1)
    torch.testing.assert_close(path.H.double(), -(p * p.log()).sum(1), rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("variant,where", [("full", "out"), ("full", "k_ctx"), ("full", "v_ctx"), ("vpool", "out"), ("vpool", "k_ctx"),
                                           ("fused", "out")])
def test_logits_that_the_pass_writes_are_read_behind_it(variant, where):
    # logits in the cache or in the last output: what the pass leaves there, as the calls in turn have it
    w = _workload(51)
    path, steps = _path(w, variant), _path(w, variant)
    args = list(_inputs(path, wl.make_queries(w)))

    def logits_of(p):
        memory = {"out": p.out[-1], "k_ctx": p.k_bufs and p.k_bufs[0], "v_ctx": p.v_bufs and p.v_bufs[0]}[where]
        memory.zero_()
        return memory.flatten()[:w.batch * len(w.probes) * w.vocab].view(-1, w.vocab)

    args[4] = logits_of(steps)
    steps.select(args[0])
    if variant == "fused":
        steps.plan()
    for i, (lb, le) in enumerate(steps.chunks):
        if variant == "fused":
            steps.attend_fused(args[1][i], args[2][i], args[3][i], steps.out[i], lb, le)
        else:
            steps.assemble(lb, le, keep_plan=i > 0)
            steps.attend(args[1][i], args[2][i], args[3][i], steps.out[i], lb, le)
    steps.entropy(args[4], 6.0)
    args[4] = logits_of(path)
    out, H, ok = path.run(*args[:5], 6.0)
    torch.cuda.synchronize()
    assert path.status.item() == 0 and steps.status.item() == 0
    assert torch.equal(H, steps.H) and torch.equal(ok, steps.first_ok) and H.std() > 0
    assert all(torch.equal(a, b) for a, b in zip(out, steps.out))


@pytest.mark.parametrize("variant,tensor", [("vpool", "v"), ("fused", "v"), ("fused", "k")])
def test_entropy_states_in_the_pool_do_not_meet_the_attention(variant, tensor):
    # a workspace that lies on a selected shot of the last layer: written after the attention has read the shot
    w = _workload(48).scaled(vocab=20003, t_q=70)
    path = _path(w, variant)
    args = list(_inputs(path, wl.make_queries(w)))
    args[4] = torch.nn.functional.pad(args[4], (0, 20008 - w.vocab))[:, :w.vocab]
    want = [t.clone() for t in path.run(*args)[0]]
    want_H, want_ok = path.H.clone(), path.first_ok.clone()
    shot = path.sel_idx[0, 0].item()
    path.ws_entropy = getattr(path.pool, tensor)[w.n_layers - 1, path.pool.shot_off[shot].item():].flatten().view(torch.uint8)
    got, H, ok = path.run(*args)
    torch.cuda.synchronize()
    assert path.status.item() == 0 and torch.equal(H, want_H) and torch.equal(ok, want_ok)
    assert all(torch.equal(a, b) for a, b in zip(want, got))


@pytest.mark.parametrize("batch", [1, 2])
def test_rounds_of_probes_use_the_tensors_they_have_now(batch):
    from paper_2605_03644_b200 import binding as ab
    from paper_2605_03644_b200.adaptive import ProbeRounds
    w = _workload(45).scaled(batch=batch, n_shots=12)
    make = lambda seed: ProbeRounds(hp.model_of(ab, w), hp.dev_pool(ab, wl.make_pool(w.scaled(seed=seed))), batch, 1, 2, 2, 2,
                                    w.t_q, w.vocab, 160)
    driver, fresh = make(45), make(46)
    qs = [wl.make_queries(w.scaled(seed=50 + r)) for r in range(2)]
    inputs = lambda r, probes: tuple(qs[r][name].cuda() for name in ("q", "kq", "vq", "logits"))
    q_emb = qs[0]["q_emb"].cuda()
    tau = float(torch.softmax(qs[1]["logits"].double(), 1).log().mul(-torch.softmax(qs[1]["logits"].double(), 1)).sum(1).max()) + 0.01
    driver.run(q_emb, inputs, 0.0)
    want = fresh.run(q_emb, inputs, tau)
    for name in ("sel_idx", "sel_score", "status", "first_ok", "H", "out", "k_ctx", "v_ctx", "_ctx_off"):
        setattr(driver, name, torch.zeros_like(getattr(driver, name)))
    driver.pool = fresh.pool
    assert driver.run(q_emb, inputs, tau) == want and want["n_star"][0] > 0
    torch.cuda.synchronize()
    assert torch.equal(driver.sel_idx, fresh.sel_idx) and torch.equal(driver.out, fresh.out)
    assert torch.equal(driver.first_ok, fresh.first_ok)
    # an error is seen in the status word it was written to
    driver.ctx_cap = 32
    with pytest.raises(RuntimeError, match="capacity"):
        driver.run(q_emb, inputs, 0.0)
