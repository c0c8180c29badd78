"""The work that users of this library have it do, as measurable cases.

Each case is one pass through the public entry points: the whole reuse path of a batch of queries
(`ReusePath`), rounds of probes (`ProbeRounds`), one decoding step over the chosen prefix, and the ranking
and entropy steps alone at the sizes where they are called by themselves.  Shapes are those of the
repository's configurations (`paper_2605_03644_b200.workloads.CONFIGS`) with fewer layers, so that several
copies of a pool fit one GPU, or generic ones around them.
"""
from __future__ import annotations

import math

import torch

from paper_2605_03644_b200 import binding as ab
from paper_2605_03644_b200.adaptive import ProbeRounds
from paper_2605_03644_b200.pipeline import ReusePath

DEV = "cuda"
TAU = 0.65                       # the paper's threshold
# (query heads, KV heads, head dimension): the configurations' three shapes, a 3B-sized one and one of d = 64
HEADS = [(4, 1, 64), (24, 8, 128), (32, 8, 128), (32, 8, 64), (64, 8, 128)]


# ------------------------------------------------------------------------------------------ the cases
def _pass(name, heads, layers, shots, lens, batch, k, probes, t_q, vocab, emb=1024, logits="bf16", dist="uniform",
          variant="auto", graph=False, pos_mode=0, base=5e5):
    return dict(name=name, kind="pass", hq=heads[0], hkv=heads[1], d=heads[2], layers=layers, shots=shots,
                len_lo=lens[0], len_hi=lens[1], dist=dist, emb=emb, batch=batch, k=k,
                probes=",".join(str(p) for p in probes), t_q=t_q, vocab=vocab, logits=logits, variant=variant,
                graph=graph, pos_mode=pos_mode, base=base)


def _decode(name, heads, layers, shots, lens, batch, k, t_new, t_own, base=5e5):
    return dict(name=name, kind="decode", hq=heads[0], hkv=heads[1], d=heads[2], layers=layers, shots=shots,
                len_lo=lens[0], len_hi=lens[1], dist="uniform", batch=batch, k=k, t_new=t_new, t_own=t_own, base=base)


def listed():
    return [
        # The smallest pool anyone keeps (cfg1 in the storage type that attention takes): an interactive
        # query over eight short shots, where launches and host work are all there is.
        _pass("small_query", (4, 1, 64), 1, 64, (32, 32), 1, 8, (8,), 16, 1024, emb=128, logits="fp32", base=1e4),
        # cfg2: one layer of an 8B-shaped model, one query with four nested probes, replayed as a CUDA graph
        # (how a server runs a latency-bound pass).
        _pass("layer_graph", (32, 8, 128), 1, 2048, (64, 256), 1, 128, (16, 32, 64, 128), 128, 32000, logits="fp32",
              graph=True),
        # cfg3: a batch of eight queries, each over 256 shots (about 33 K tokens), here four layers.
        _pass("batch", (32, 8, 128), 4, 4096, (64, 192), 8, 256, (256,), 128, 128256),
        # cfg5: thirty-two queries with seven nested probes up to 512 shots, lognormal lengths, here one layer.
        _pass("nested_probes", (32, 8, 128), 1, 8192, (40, 400), 32, 512, (8, 16, 32, 64, 128, 256, 512), 64, 128256,
              dist="lognormal"),
        # cfg4: one long query (64 heads: 2048 query rows per KV head) over a context of about 64 K tokens.
        _pass("long_context", (64, 8, 128), 3, 320, (128, 512), 1, 200, (200,), 256, 128256),
        # A caller that has no memory for an assembled cache; keys stored as prefilled (the paper's own form).
        _pass("no_cache", (32, 8, 128), 2, 1024, (64, 192), 2, 128, (64, 128), 100, 128256, variant="fused",
              pos_mode=1),
        # The paper's case study: shot counts 4-16, then 20-32, on one query, with the model's layers in one call.
        dict(name="probe_rounds", kind="rounds", hq=32, hkv=8, d=128, layers=16, shots=256, len_lo=64, len_hi=192,
             dist="uniform", emb=1024, batch=1, n0=4, step=4, m=4, rounds=2, t_q=64, vocab=128256, logits="bf16",
             base=5e5),
        # Decoding one token of one request, layer by layer as a model does it (the next layer's query does not
        # exist before this layer has run).
        _decode("decode_one", (32, 8, 128), 4, 512, (64, 192), 1, 128, 1, 77),
        # Decoding one token of a batch of requests, each over the prefix its own probes chose.
        _decode("decode_batch", (32, 8, 128), 2, 512, (64, 192), 32, 128, 1, 160),
        # The paper's own ranking (attention mass at one representative layer) over a pool of 2048 shots.
        dict(name="rank_by_attention", kind="rank", hq=32, hkv=8, d=128, layers=1, shots=2048, len_lo=64, len_hi=256,
             dist="uniform", batch=2, t_q=128, k=128, per_token=False, base=5e5),
        # Ranking a large pool by embeddings for a batch of queries (more shots than one sort takes, 768-wide
        # sentence embeddings).
        dict(name="select_large_pool", kind="select", shots=20000, emb=768, batch=16, k=512),
        # The confidence probe on the last-token logits of many probes.
        dict(name="entropy_logits", kind="entropy", rows=1024, vocab=128256, logits="bf16", group=4, form="full"),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of lo .. hi, odd ones among them."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _draw_once(rng):
    kind = rng.choice(["pass"] * 5 + ["decode"] * 2 + ["rounds", "rank", "select", "entropy"])
    if kind == "select":
        shots = _log_int(rng, 64, 65536)
        return dict(kind=kind, shots=shots, emb=rng.choice([128, 384, 768, 1024]), batch=_log_int(rng, 1, 32),
                    k=_log_int(rng, 1, min(shots, 1024)))
    if kind == "entropy":
        group = _log_int(rng, 1, 8)
        return dict(kind=kind, rows=group * _log_int(rng, 1, 512), vocab=rng.choice([32000, 50257, 128256, 151936]),
                    logits=rng.choice(["fp32", "bf16"]), group=group, form=rng.choice(["full", "full", "subset", "static"]))
    hq, hkv, d = rng.choice(HEADS)
    lo = rng.choice([16, 32, 64, 128])
    hi = lo * rng.choice([2, 3, 4])
    c = dict(kind=kind, hq=hq, hkv=hkv, d=d, len_lo=lo, len_hi=hi, dist="uniform", base=rng.choice([1e4, 5e5]))
    if kind == "rank":
        shots = _log_int(rng, 64, 4096)
        return dict(c, layers=1, shots=shots, batch=_log_int(rng, 1, 8), t_q=_log_int(rng, 8, 256),
                    k=_log_int(rng, 1, shots // 2), per_token=rng.random() < 0.3)
    if kind == "decode":
        t_new = rng.choice([1, 1, 1, _log_int(rng, 2, 256)])
        shots = _log_int(rng, 32, 1024)
        return dict(c, layers=rng.choice([1, 2, 4]), shots=shots, batch=_log_int(rng, 1, 64),
                    k=_log_int(rng, 2, min(shots, 512)), t_new=t_new, t_own=t_new + _log_int(rng, 1, 400))
    c.update(layers=rng.choice([1, 1, 2, 4, 8]), emb=rng.choice([128, 384, 768, 1024]), t_q=_log_int(rng, 8, 320),
             vocab=rng.choice([32000, 50257, 128256, 151936]), logits=rng.choice(["fp32", "bf16"]))
    if kind == "rounds":
        return dict(c, shots=_log_int(rng, 96, 512), batch=_log_int(rng, 1, 4), n0=rng.choice([1, 2, 4]),
                    step=rng.choice([1, 2, 4, 8]), m=rng.choice([2, 4]), rounds=rng.choice([2, 3]))
    shots = _log_int(rng, 64, 8192)
    k = _log_int(rng, 4, min(shots, 512))
    n_probes = rng.choice([1, 1, 2, 4, 7])
    probes = sorted({max(1, k >> i) for i in range(n_probes)})
    return dict(c, shots=shots, batch=_log_int(rng, 1, 32), k=k, probes=",".join(str(p) for p in probes),
                dist=rng.choice(["uniform", "lognormal"]), variant=rng.choice(["auto"] * 5 + ["fused"]),
                graph=rng.random() < 0.3, pos_mode=rng.choice([0, 0, 0, 1]))


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        c = _draw_once(rng)
        if _cost(c) <= top * (0.2 if c.get("variant") == "fused" else 1.0) and _state_bytes(c) <= 24e9:
            return c


# -------------------------------------------------------------------------------------- sizes of a case
def _lens(c):
    """Mean and standard deviation of a shot's length (lognormal: of its unclipped law, around the geometric mean)."""
    lo, hi = c["len_lo"], c["len_hi"]
    if c["dist"] == "lognormal":
        med = math.sqrt(lo * hi) * 0.95
        mean = med * math.exp(0.08)
        return mean, mean * 0.417
    return (lo + hi) / 2.0, math.sqrt(((hi - lo + 1) ** 2 - 1) / 12.0)


def _cap(c, k):
    """Cache capacity a user plans for k shots: the mean context plus eight standard deviations (a query that
    outgrew it would be reported in `status`), never more than k shots of the longest length; whole tiles."""
    mean, sd = _lens(c)
    need = min(k * c["len_hi"], k * mean * 1.02 + 8 * sd * math.sqrt(k))
    return int(-(-need // 128) * 128)


def _probes(c):
    if c["kind"] == "rounds":
        return [c["n0"] + i * c["step"] for i in range(c["m"] * c["rounds"])]
    return [int(p) for p in c["probes"].split(",")]


def _k(c):
    return _probes(c)[-1] if c["kind"] == "rounds" else c["k"]


def _logit_bytes(c):
    return 4 if c["logits"] == "fp32" else 2


def work(c):
    """Each input read once and each output written once; the multiplications of the attention (or score) rows."""
    if c["kind"] == "select":
        return {"bytes": 4.0 * c["emb"] * (c["shots"] + c["batch"]) + 8.0 * c["batch"] * c["k"],
                "flops": 2.0 * c["batch"] * c["shots"] * c["emb"]}
    if c["kind"] == "entropy":
        return {"bytes": float(c["rows"]) * (c["vocab"] * _logit_bytes(c) + 4), "flops": 6.0 * c["rows"] * c["vocab"]}
    mean = _lens(c)[0]
    hq, hkv, d = c["hq"], c["hkv"], c["d"]
    row_kv, row_q = 2.0 * hkv * d, 2.0 * hq * d            # bytes of one token's K (or V), of its Q (or output)
    if c["kind"] == "rank":
        tokens = c["shots"] * mean
        return {"bytes": tokens * row_kv + c["batch"] * c["t_q"] * row_q + 8.0 * c["batch"] * c["k"],
                "flops": 2.0 * d * hq * c["batch"] * c["t_q"] * tokens}
    if c["kind"] == "decode":
        ctx = mean * 0.75 * c["k"]                         # each request keeps between half of its shots and all
        per_layer = c["batch"] * (2 * row_kv * (ctx + c["t_own"]) + 2 * row_q * c["t_new"])
        return {"bytes": c["layers"] * per_layer,
                "flops": c["layers"] * c["batch"] * 4.0 * c["t_new"] * hq * d * (ctx + c["t_own"])}
    probes, k, b, t = _probes(c), _k(c), c["batch"], c["t_q"]
    distinct = c["shots"] * (1.0 - (1.0 - k / c["shots"]) ** b) * mean      # pool tokens that some query selects
    rows = b * len(probes)
    nbytes = (4.0 * c["emb"] * (c["shots"] + b) + c["layers"] * (2 * row_kv * distinct + rows * t * (2 * row_q + 2 * row_kv))
              + rows * c["vocab"] * _logit_bytes(c))
    flops = c["layers"] * b * sum(4.0 * t * hq * d * (mean * n + (t + 1) / 2.0) for n in probes)
    return {"bytes": nbytes, "flops": flops + 2.0 * b * c["shots"] * c["emb"]}


def _cost(c):
    w = work(c)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.4e15)


def _state_bytes(c):
    """About what prepare() holds on the GPU."""
    if c["kind"] == "select":
        return 4.0 * c["emb"] * c["shots"] + 16.0 * c["batch"] * c["shots"]
    if c["kind"] == "entropy":
        return c["rows"] * c["vocab"] * 6.0
    row_kv = 2.0 * c["hkv"] * c["d"]
    pool = 2 * row_kv * c["shots"] * _lens(c)[0] * c["layers"]
    if c["kind"] == "rank":
        return 2 * pool
    k = _k(c)
    rows = c["batch"] * (1 if c["kind"] == "decode" else len(_probes(c))) * c.get("t_q", c.get("t_new", 1))
    return pool + c["batch"] * _cap(c, k) * 2 * row_kv * c["layers"] + 8.0 * rows * c["hq"] * c["d"] * c["layers"]


def tolerance(c):
    """About four times what was seen against a 64-bit evaluation of the same inputs.

    Ranking by embeddings is decided in 64 bits (the scores are those values rounded to fp32: 2.6e-8).
    Entropies are 32-bit sums (7e-8 of the norm; 2.3e-6 over two tokens, where the sum is small against its
    terms), masses too (2.5e-6; of neighbouring ones a few are closer than that).  Attention outputs are bf16
    rows of sums whose operands (rotated Q and K, the probabilities) are rounded to bf16 (4.1e-3; the three
    forms of the attention call differ by 6e-4 among each other)."""
    if c["kind"] == "select":
        return {"rel": 1e-7}
    if c["kind"] == "entropy":
        return {"rel": 1e-5 if c["form"] == "subset" else 1e-6}
    if c["kind"] == "rank":
        return {"rel": 2e-5, "differ": 0.01}
    return {"rel": 1e-2}


# ------------------------------------------------------------------------------------------- the inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _randn(g, *shape, dtype=torch.bfloat16):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _shot_off(c, g):
    lo, hi = c["len_lo"], c["len_hi"]
    if c["dist"] == "lognormal":
        z = torch.randn(c["shots"], generator=g, device=DEV)
        t = torch.round(math.sqrt(lo * hi) * 0.95 * torch.exp(0.4 * z)).clamp(lo, hi)
    else:
        t = torch.randint(lo, hi + 1, (c["shots"],), generator=g, device=DEV)
    off = torch.zeros(c["shots"] + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(t.to(torch.int64), 0, out=off[1:])
    return off


def _channels(c, g):
    """Cached keys and values have channels of unlike size: one scale per layer, head and channel."""
    shape = (c["layers"], 1, c["hkv"], c["d"])
    return torch.empty(shape, device=DEV).uniform_(0.5, 2.0, generator=g).to(torch.bfloat16)


def _embeddings(n, e, g):
    x = _randn(g, n, e, dtype=torch.float32)
    return x / x.norm(dim=1, keepdim=True)


def _pool(c, g, with_v=True):
    off = _shot_off(c, g)
    tokens = int(off[-1])
    sk, sv = _channels(c, g), _channels(c, g)
    k = _randn(g, c["layers"], tokens, c["hkv"], c["d"]).mul_(sk)
    v = _randn(g, c["layers"], tokens, c["hkv"], c["d"]).mul_(sv) if with_v else None
    emb = _embeddings(c["shots"], c["emb"], g) if "emb" in c else None
    return ab.Pool(off, k, v, emb), sk, sv


def _query_emb(c, g, emb):
    """A query resembles some of the cached shots."""
    near = torch.randint(0, emb.shape[0], (c["batch"],), generator=g, device=DEV)
    x = _embeddings(c["batch"], c["emb"], g) + 0.5 * emb[near]
    return (x / x.norm(dim=1, keepdim=True)).contiguous()


def _logits(rows, vocab, dtype, g, confident):
    """Last-token logits: a broad bulk and one token that stands out the more, the more confident the row
    (0 .. 1: from an entropy of several nats to nearly none)."""
    stride = -(-vocab // 8) * 8
    x = torch.randn(rows, stride, generator=g, device=DEV) * 2.0
    top = torch.randint(0, vocab, (rows, 1), generator=g, device=DEV)
    bump = 8.0 + 16.0 * confident.view(-1, 1) + 2.0 * torch.rand(rows, 1, generator=g, device=DEV)
    x.scatter_(1, top, bump)
    return x.to(torch.float32 if dtype == "fp32" else torch.bfloat16)[:, :vocab]


def _model(c):
    return ab.make_model(c["layers"], c["hq"], c["hkv"], c["d"], "bf16", c["base"], k_pos_mode=c.get("pos_mode", 0))


def _queries(c, g, layers, n_probes, sk, sv):
    """Un-rotated Q, K_q and V_q of the probes' tokens at `layers` layers."""
    b, t, d = c["batch"], c["t_q"], c["d"]
    per_layer = (1, layers, 1, 1, c["hkv"], d)
    return (_randn(g, b, layers, n_probes, t, c["hq"], d),
            _randn(g, b, layers, n_probes, t, c["hkv"], d).mul_(sk.view(per_layer)),
            _randn(g, b, layers, n_probes, t, c["hkv"], d).mul_(sv.view(per_layer)))


def _prepare_pass(c, g):
    pool, sk, sv = _pool(c, g)
    probes = _probes(c)
    fused = c["variant"] == "fused"
    path = ReusePath(_model(c), pool, c["batch"], c["k"], probes, c["t_q"], c["vocab"], _cap(c, c["k"]), fused=fused,
                     vpool=False if fused else None)
    q, kq, vq = _queries(c, g, c["layers"], len(probes), sk, sv)
    step = torch.linspace(0.1, 1.0, len(probes), device=DEV).repeat(c["batch"])
    s = dict(case=c, path=path, q_emb=_query_emb(c, g, pool.emb), q=[q], kq=[kq], vq=[vq],
             logits=_logits(c["batch"] * len(probes), c["vocab"], c["logits"], g, step))
    if c["graph"]:
        path.capture(s["q_emb"], s["q"], s["kq"], s["vq"], s["logits"], TAU)
    return s


def _prepare_rounds(c, g):
    pool, sk, sv = _pool(c, g)
    k_max = _k(c)
    driver = ProbeRounds(_model(c), pool, c["batch"], c["n0"], c["step"], c["m"], c["rounds"], c["t_q"], c["vocab"],
                         _cap(c, k_max))
    driver.k_ctx.zero_()              # decoding goes on over this cache; what no shot fills stays zero
    driver.v_ctx.zero_()
    inputs = []
    for r in range(c["rounds"]):      # no probe is confident enough before the last round
        last = r == c["rounds"] - 1
        conf = (torch.linspace(0.5, 1.0, c["m"], device=DEV) if last else torch.zeros(c["m"], device=DEV)).repeat(c["batch"])
        q, kq, vq = _queries(c, g, c["layers"], c["m"], sk, sv)
        inputs.append((q, kq, vq, _logits(c["batch"] * c["m"], c["vocab"], c["logits"], g, conf)))
    return dict(case=c, driver=driver, q_emb=_query_emb(c, g, pool.emb), inputs=inputs)


def _prepare_decode(c, g):
    """The assembled cache of every layer, as the passes before left it, and one step's tensors."""
    pool, sk, sv = _pool(c, g)
    b, k, cap, n_own = c["batch"], c["k"], _cap(c, c["k"]), c["t_own"]
    model = _model(c)
    sel = torch.stack([torch.randperm(c["shots"], generator=g, device=DEV)[:k] for _ in range(b)]).to(torch.int32)
    off = torch.empty(b, k + 1, dtype=torch.int64, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    caches = []
    for layer in range(c["layers"]):
        kc = torch.empty(b, 1, cap, c["hkv"], c["d"], dtype=torch.bfloat16, device=DEV)
        vc = torch.empty_like(kc)
        ab.adapshot_assemble_kv(model, pool, sel, layer, layer + 1, kc, vc, cap, off, status)
        caches.append((kc, vc))
    per_layer = [(_randn(g, b, 1, c["t_new"], c["hq"], c["d"]), _randn(g, b, 1, n_own, c["hkv"], c["d"]).mul_(sk[layer]),
                  _randn(g, b, 1, n_own, c["hkv"], c["d"]).mul_(sv[layer]),
                  torch.empty(b, 1, c["t_new"], c["hq"], c["d"], dtype=torch.bfloat16, device=DEV))
                 for layer in range(c["layers"])]
    ws = torch.empty(max(256, ab.adapshot_decode_workspace_bytes(model, b, c["t_new"], n_own, 1)), dtype=torch.uint8,
                     device=DEV)
    return dict(case=c, model=model, caches=caches, off=off, cap=cap, status=status, ws=ws, per_layer=per_layer,
                n_shots=torch.randint((k + 1) // 2, k + 1, (b,), generator=g, device=DEV, dtype=torch.int32))


def _prepare_rank(c, g):
    pool, _, _ = _pool(c, g, with_v=False)
    b, t, hq = c["batch"], c["t_q"], c["hq"]
    # some shots speak to the queries more than others: their keys lean towards a direction that the queries share
    # (a log-normal spread of the masses, as relevance has it)
    lean = _randn(g, c["hkv"], c["d"], dtype=torch.float32)
    lean /= lean.norm(dim=1, keepdim=True)
    owner = torch.repeat_interleave(torch.arange(c["shots"], device=DEV), pool.shot_off[1:] - pool.shot_off[:-1])
    much = torch.randn(c["shots"], generator=g, device=DEV)[owner]
    for a in range(0, owner.numel(), 1 << 18):
        pool.k[0, a:a + (1 << 18)] += (much[a:a + (1 << 18), None, None] * lean).to(torch.bfloat16)
    q = _randn(g, b, t, hq, c["d"])
    q += (8.0 * lean.repeat_interleave(hq // c["hkv"], 0)).to(torch.bfloat16)
    model = _model(c)
    ws = torch.empty(max(256, ab.adapshot_select_attn_workspace_bytes(model, pool, b, t, c["k"])), dtype=torch.uint8,
                     device=DEV)
    return dict(case=c, model=model, pool=pool, q=q, ws=ws, **_selection(c))


def _selection(c):
    return dict(sel=torch.empty(c["batch"], c["k"], dtype=torch.int32, device=DEV),
                score=torch.empty(c["batch"], c["k"], dtype=torch.float32, device=DEV),
                status=torch.zeros(1, dtype=torch.int32, device=DEV))


def _prepare_select(c, g):
    emb = _embeddings(c["shots"], c["emb"], g)
    pool = ab.Pool(torch.arange(c["shots"] + 1, dtype=torch.int64, device=DEV), None, None, emb)
    ws = torch.empty(max(256, ab.adapshot_select_workspace_bytes(c["shots"], c["batch"], c["k"])), dtype=torch.uint8,
                     device=DEV)
    return dict(case=c, pool=pool, q_emb=_query_emb(c, g, emb), ws=ws, **_selection(c))


def _prepare_entropy(c, g):
    rows = c["rows"]
    conf = torch.rand(rows, generator=g, device=DEV)
    return dict(case=c, logits=_logits(rows, c["vocab"], c["logits"], g, conf),
                H=torch.empty(rows, dtype=torch.float32, device=DEV),
                ok=torch.empty(rows // c["group"], dtype=torch.int32, device=DEV),
                ids=torch.randint(0, c["vocab"], (2,), generator=g, device=DEV, dtype=torch.int32),   # "Yes" and "No"
                ws=torch.empty(max(256, ab.adapshot_entropy_workspace_bytes(rows, c["vocab"])), dtype=torch.uint8, device=DEV),
                status=torch.zeros(1, dtype=torch.int32, device=DEV))


PREPARE = {"pass": _prepare_pass, "rounds": _prepare_rounds, "decode": _prepare_decode, "rank": _prepare_rank,
           "select": _prepare_select, "entropy": _prepare_entropy}


def prepare(case, seed):
    return PREPARE[case["kind"]](case, _gen(seed))


# --------------------------------------------------------------------------------------------- the pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "pass":
        path = s["path"]
        if c["graph"]:
            out, H, ok = path.replay()
        else:
            out, H, ok = path.run(s["q_emb"], s["q"], s["kq"], s["vq"], s["logits"], TAU)
        return dict(sel=path.sel_idx, score=path.sel_score, off=path.ctx_off, out=out, H=H, first_ok=ok, status=path.status)
    if kind == "rounds":
        d = s["driver"]
        entropies = []
        got = d.run(s["q_emb"], lambda r, probes: s["inputs"][r], TAU, on_round=lambda r, drv: entropies.append(drv.H.clone()))
        return dict(sel=d.sel_idx, out=d.out, k_ctx=d.k_ctx, v_ctx=d.v_ctx, H=entropies,
                    n_star=got["n_star"], rounds=got["rounds_run"])
    if kind == "decode":
        for (kc, vc), (q, ko, vo, out) in zip(s["caches"], s["per_layer"]):
            ab.adapshot_decode_attn(s["model"], kc, vc, s["cap"], s["off"], c["k"], s["n_shots"], q, ko, vo, 0, 1, out,
                                    None, s["ws"], s["status"])
        return dict(out=[t[3] for t in s["per_layer"]], status=s["status"])
    if kind == "rank":
        ab.adapshot_select_attn(s["model"], s["pool"], 0, s["q"], c["k"], s["sel"], s["score"], s["ws"], s["status"],
                                per_token=c["per_token"])
        return dict(sel=s["sel"], score=s["score"], status=s["status"])
    if kind == "select":
        ab.adapshot_select(s["pool"], s["q_emb"], c["k"], s["sel"], s["score"], s["ws"], s["status"])
        return dict(sel=s["sel"], score=s["score"], status=s["status"])
    rows = c["group"]
    if c["form"] == "subset":
        ab.adapshot_entropy_subset(s["logits"], s["ids"], s["H"], TAU, rows, s["ok"], s["ws"], s["status"], renorm=True)
    elif c["form"] == "static":
        ab.adapshot_entropy_static(s["logits"], s["H"], TAU, rows, s["ok"], s["status"])
    else:
        ab.adapshot_entropy(s["logits"], s["H"], TAU, rows, s["ok"], s["ws"], s["status"])
    return dict(H=s["H"], first_ok=s["ok"], status=s["status"])
