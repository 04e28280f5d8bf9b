"""The native argument marshalling refuses what the entry points have always refused, before anything is launched."""
import pytest
import torch

from paper_2608_21836_b200 import binding as l4l
from paper_2608_21836_b200 import build


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def test_a_module_for_another_torch_is_rebuilt_and_not_loaded(monkeypatch, tmp_path):
    assert not build.marshal_is_stale() and l4l._load_native().BUILT_FOR == build.marshal_tag()
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    assert build.marshal_is_stale()
    monkeypatch.setattr(l4l, "_native", None)
    with pytest.raises(ImportError, match="9.9.9.*build it with"):
        l4l._load_native()
    monkeypatch.setattr(build, "MARSHAL", str(tmp_path / "missing.so"))
    with pytest.raises(FileNotFoundError, match="build it with"):
        l4l._load_native()


def calls(t4, t3, i):
    """Every call of the native module, its tensors all of one kind."""
    t2 = torch.zeros(4, 32)
    return {
        "prefill": lambda: l4l.l4l_attn_prefill(t4, t4, t4, t4, i, 1.0, i),
        "chunk": lambda: l4l.l4l_attn_prefill_chunk(t4, t4, t4, t4, i, i, 1.0, i),
        "chunk_append": lambda: l4l.l4l_attn_prefill_chunk_append(t4, t4, t4, t4, t4, t4, i, i, 1.0, i),
        "rope": lambda: l4l.l4l_rope_kv_append(t4, t4, t4, t4, t4, i, i, t2, t2),
        "decode": lambda: l4l.l4l_attn_decode(t3, t3, t4, t4, i, 4, 1.0, i),
        "decode_append": lambda: l4l.l4l_attn_decode_append(t3, t3, t4, t4, t4, t4, i, 4, 1.0, i),
        "decode_paged": lambda: l4l.l4l_attn_decode_paged(t3, t3, t4, t4, i, i, 4, 1.0, i),
        "decode_paged_append": lambda: l4l.l4l_attn_decode_paged_append(t3, t3, t4, t4, i, t4, t4, i, 4, 1.0, i),
        "decode_rope": lambda: l4l.l4l_attn_decode_rope_append(t3, t3, t4, t4, t4, t4, i, 4, 1.0, t2, t2, i),
        "decode_paged_rope": lambda: l4l.l4l_attn_decode_paged_rope_append(t3, t3, t4, t4, i, t4, t4, i, 4, 1.0, t2, t2, i),
        "decode_fp8": lambda: l4l.l4l_attn_decode_fp8(t3, t3, t4, t4, t2, t2, i, 4, 1.0, i),
        "decode_paged_fp8": lambda: l4l.l4l_attn_decode_paged_fp8(t3, t3, t4, t4, t2, t2, i, i, 4, 1.0, i),
        "decode_append_fp8": lambda: l4l.l4l_attn_decode_append_fp8(t3, t3, t4, t4, t2, t2, t4, t4, i, 4, 1.0, i),
        "decode_rope_fp8": lambda: l4l.l4l_attn_decode_rope_append_fp8(t3, t3, t4, t4, t2, t2, t4, t4, i, 4, 1.0, t2, t2, i),
        "scan": lambda: l4l.l4l_rglru_scan(t3, t3, t3, t2, t2, t3, i),
    }


NAMES = sorted(calls(None, None, None))


@pytest.mark.parametrize("name", NAMES)
def test_host_tensors_and_other_objects_are_type_errors(name):
    t4, t3, i = torch.zeros(1, 4, 2, 64, dtype=torch.bfloat16), torch.zeros(1, 2, 64, dtype=torch.bfloat16), torch.zeros(1, dtype=torch.int32)
    with pytest.raises(TypeError):
        calls(t4, t3, i)[name]()
    with pytest.raises(TypeError):
        calls(7, 7, 7)[name]()


def decode_calls(device):
    """Every decode entry point, by name, with arguments that it accepts."""
    B, Hq, Hkv, D, page = 2, 4, 2, 128, 16
    z = lambda *s, dtype=torch.bfloat16: torch.zeros(*s, dtype=dtype, device=device)  # noqa: E731
    # caches [B, Hkv, slots, D] and pools [pages, Hkv, slots, D] of one shape: within bounds whichever way they are read
    k, v, k8, v8 = (z(B, Hkv, page, D, dtype=t) for t in (torch.bfloat16,) * 2 + (torch.uint8,) * 2)
    ones, table = torch.ones(Hkv, device=device), torch.arange(B, dtype=torch.int32, device=device).view(B, 1)
    step = dict(q=z(B, Hq, D), o=z(B, Hq, D), kv_lens=torch.full((B,), 5, dtype=torch.int32, device=device), max_kv_len=page,
                scale=1.0, workspace=z(8 << 20, dtype=torch.uint8))
    kv, pool = dict(cache_k=k, cache_v=v), dict(pool_k=k, pool_v=v, block_table=table)
    kv8 = dict(cache_k8=k8, cache_v8=v8, k_scale=ones, v_scale=ones)
    pool8 = dict(pool_k8=k8, pool_v8=v8, k_scale=ones, v_scale=ones, block_table=table)
    append = dict(k_new=z(B, 1, Hkv, D), v_new=z(B, 1, Hkv, D))
    rope = dict(append, cos=z(page, D // 2, dtype=torch.float32), sin=z(page, D // 2, dtype=torch.float32))
    forms = dict(decode=kv, decode_append=kv | append, decode_rope_append=kv | rope, decode_paged=pool,
                 decode_paged_append=pool | append, decode_paged_rope_append=pool | rope, decode_fp8=kv8,
                 decode_append_fp8=kv8 | append, decode_rope_append_fp8=kv8 | rope, decode_paged_fp8=pool8)
    return {name: (getattr(l4l, "l4l_attn_" + name), step | args) for name, args in forms.items()}


DECODES = decode_calls("cpu")


# without one of these the call would be another operation
@pytest.mark.parametrize("name,argument", [(n, a) for n in DECODES for a in ("k_new", "v_new", "block_table", "cos") if a in DECODES[n][1]])
def test_an_argument_left_out_is_named(name, argument):
    """Refused by name, ahead of any look at the tensors: the entry point says what the operation is, not its arguments."""
    call, args = DECODES[name]
    with pytest.raises(TypeError, match=f"^{argument} must be a tensor"):
        call(**{**args, argument: None})


@pytest.mark.gpu
@pytest.mark.parametrize("name", DECODES)
def test_every_decode_argument_is_required(name):
    call, args = decode_calls("cuda")[name]
    call(**args)
    for argument in set(args) - {"max_kv_len", "scale"}:
        with pytest.raises((TypeError, l4l.L4LError)):
            call(**{**args, argument: None})
    if name.endswith("fp8"):                                   # without scales it is no call over a bf16 cache
        bf16 = {a: t.to(torch.bfloat16) for a, t in args.items() if a.endswith("8")}
        with pytest.raises(TypeError):
            call(**{**args, **bf16, "k_scale": None, "v_scale": None})
    torch.cuda.synchronize()


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_float32_on_the_device_is_a_type_error(name):
    t4, t3 = torch.zeros(1, 4, 2, 64, device="cuda"), torch.zeros(1, 2, 64, device="cuda")
    with pytest.raises(TypeError):
        calls(t4, t3, torch.zeros(1, dtype=torch.int32, device="cuda"))[name]()


@pytest.mark.gpu
def test_shapes_are_value_errors_and_statuses_are_raised():
    q, o = torch.zeros(2, 4, 64, dtype=torch.bfloat16, device="cuda"), torch.zeros(2, 4, 64, dtype=torch.bfloat16, device="cuda")
    ck, lens = torch.zeros(2, 2, 8, 64, dtype=torch.bfloat16, device="cuda"), torch.ones(2, dtype=torch.int32, device="cuda")
    new = torch.zeros(2, 1, 2, 64, dtype=torch.bfloat16, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_DECODE, 2, 4, 2, 64, 8)
    with pytest.raises(ValueError):
        l4l.l4l_attn_decode(q, o[:1], ck, ck, lens, 8, 1.0, ws)
    with pytest.raises(ValueError):
        l4l.l4l_attn_decode_append(q, o, ck, ck, new[:, :, :1], new, lens, 8, 1.0, ws)
    with pytest.raises(ValueError):
        l4l.l4l_attn_decode(q, o, ck, ck[:, :, :4], lens, 8, 1.0, ws)
    with pytest.raises(TypeError):
        l4l.l4l_attn_decode(q, o, ck, ck, lens, 8, 1.0, ws, lse=torch.zeros(2, 3, device="cuda"))
    with pytest.raises(l4l.L4LError):
        l4l.l4l_attn_decode(q, o, ck, ck, lens, 9, 1.0, ws)        # more than the cache's slots
    l4l.l4l_attn_decode(q, o, ck, ck.clone(), lens, 8, 1.0, ws)
