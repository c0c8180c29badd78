"""What the ctypes binding refuses before it calls into the library: tensors of another size or type than the call reads.
No device: tensors that say they are on the GPU, and a library call that notes that it was reached."""
import pytest
import torch


class OnGpu(torch.Tensor):
    is_cuda = True


def _t(*shape, dtype=torch.bfloat16):
    return torch.zeros(*shape, dtype=dtype).as_subclass(OnGpu)


@pytest.fixture
def ab(monkeypatch):
    from paper_2605_03644_b200 import build
    build.build()
    from paper_2605_03644_b200 import binding
    binding.calls = []
    for name in ("_reuse_pass", "_select", "_entropy"):
        monkeypatch.setattr(binding, name, lambda *a, name=name: binding.calls.append(name) or 0)
    monkeypatch.setattr(binding, "_stream", lambda: 0)
    yield binding
    del binding.calls


def _pass_args(ab, B=3, P=2, k=4, t_q=5):
    hq, hkv, d, ends = 4, 2, 64, [2, 3]
    pool = ab.Pool(_t(9, dtype=torch.int64), _t(3, 80, hkv, d), _t(3, 80, hkv, d), _t(8, 16, dtype=torch.float32))
    i32, u8, f32 = dict(dtype=torch.int32), dict(dtype=torch.uint8), dict(dtype=torch.float32)
    rows = lambda h: [_t(B, le - lb, P, t_q, h, d) for lb, le in ((0, 2), (2, 3))]
    return dict(model=ab.make_model(3, hq, hkv, d, "bf16", 1e4), pool=pool, probe_nshots=[2, k], layer_end=ends,
                variant=ab.PASS_FULL, k=k, ctx_cap=40, q_emb=_t(B, 16, **f32), q=rows(hq), kq=rows(hkv),
                vq=rows(hkv), out=rows(hq), logits=_t(B * P, 24, **f32), tau=0.5, sel_idx=_t(B, k, **i32),
                sel_score=_t(B, k, **f32), ctx_off=_t(B, k + 1, dtype=torch.int64), k_ctx=_t(B * 2 * 40 * hkv * d),
                v_ctx=_t(B * 2 * 40 * hkv * d), H=_t(B * P, **f32), first_ok=_t(B, **i32), ws_select=_t(256, **u8),
                ws_attn=_t(256, **u8), ws_entropy=_t(256, **u8), status=_t(1, **i32))


def test_a_pass_of_the_right_sizes_is_called(ab):
    args = _pass_args(ab)
    ab.adapshot_reuse_pass(**args)
    args["logits"] = args["logits"].to(torch.bfloat16)
    ab.adapshot_reuse_pass(**args)
    assert ab.calls == ["_reuse_pass"] * 2


@pytest.mark.parametrize("name,make", [
    ("q_emb", lambda t: t[:2]), ("q_emb", lambda t: t[:, :8].contiguous()), ("q_emb", lambda t: t.to(torch.bfloat16)),
    ("q_emb", lambda t: t.to(torch.float16)), ("logits", lambda t: t[:4]), ("logits", lambda t: t.to(torch.float16)),
    ("q", lambda t: [t[0], t[0][:, :1, :, :4].contiguous()]), ("kq", lambda t: [t[0].to(torch.float8_e4m3fn), t[1]]),
    ("vq", lambda t: t[:1]), ("out", lambda t: [t[0], t[1].to(torch.int8)]),
])
def test_a_pass_over_tensors_it_would_read_out_of_range_is_refused(ab, name, make):
    args = _pass_args(ab)
    args[name] = make(args[name])
    with pytest.raises(ValueError):
        ab.adapshot_reuse_pass(**args)
    assert ab.calls == []


def test_select_and_entropy_refuse_other_shapes_and_types(ab):
    a = _pass_args(ab)
    for q_emb in (a["q_emb"][:, :8].contiguous(), a["q_emb"].to(torch.bfloat16), _t(4, 16, dtype=torch.float32)):
        with pytest.raises(ValueError):
            ab.adapshot_select(a["pool"], q_emb, a["k"], a["sel_idx"], None, a["ws_select"], a["status"])
    with pytest.raises(ValueError):
        ab.adapshot_entropy(a["logits"].to(torch.float16), a["H"], 0.5, 2, None, a["ws_entropy"], a["status"])
    assert ab.calls == []
    ab.adapshot_select(a["pool"], a["q_emb"], a["k"], a["sel_idx"], None, a["ws_select"], a["status"])
    ab.adapshot_entropy(a["logits"], a["H"], 0.5, 2, None, a["ws_entropy"], a["status"])
    assert ab.calls == ["_select", "_entropy"]


def test_a_prefix_of_the_selection_is_taken_of_one_query_alone(ab, monkeypatch):
    got = []
    monkeypatch.setattr(ab, "_assemble_from", lambda *a: got.append((a[3], a[4])) or 0)
    a = _pass_args(ab)
    call = lambda sel, k: ab.adapshot_assemble_kv_from(a["model"], a["pool"], sel, 0, 0, 3, a["k_ctx"], a["v_ctx"], 40,
                                                       a["ctx_off"], a["status"], k=k)
    one, three = a["sel_idx"][:1].contiguous(), a["sel_idx"]
    call(one, 2), call(one, None), call(three, 4), call(three, None)
    assert got == [(1, 2), (1, 4), (3, 4), (3, 4)]
    for sel, k in ((one, 5), (three, 2)):
        with pytest.raises(ValueError):
            call(sel, k)
