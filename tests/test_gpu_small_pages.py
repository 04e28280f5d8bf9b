"""Pools of small pages (a load per page) against pools of 64-token pages and the contiguous cache, which take the general
path: the arithmetic and its order are the same, so the outputs are equal bit for bit, whatever the strides of the pool."""
import pytest
import torch

from paper_2608_21836_b200 import binding as l4l

pytestmark = pytest.mark.gpu


def pool_of(cache, page, table, n_pages, layout):
    """The contiguous cache [B, Hkv, slots, D] as a pool of pages [n_pages, Hkv, page, D] in one of three memory layouts."""
    B, Hkv, slots, D = cache.shape
    if layout == "head":                                   # dense
        pool = torch.full((n_pages, Hkv, page, D), float("nan"), dtype=cache.dtype, device="cuda")
    elif layout == "token":                                # [page, token, head, D]
        pool = torch.full((n_pages, page, Hkv, D), float("nan"), dtype=cache.dtype, device="cuda").transpose(1, 2)
    else:                                                  # padded rows, heads outermost
        pool = torch.full((Hkv, n_pages, page, D + 64), float("nan"), dtype=cache.dtype, device="cuda")[..., :D].transpose(0, 1)
    for b in range(B):
        for i in range(slots // page):
            pool[table[b, i]] = cache[b, :, i * page:(i + 1) * page]
    return pool


@pytest.mark.parametrize("cluster", [0, -1])
@pytest.mark.parametrize("layout", ["head", "token", "padded"])
@pytest.mark.parametrize("Hq,Hkv,D", [(4, 1, 128), (12, 3, 128), (16, 2, 128), (32, 2, 128), (3, 3, 64)])
@pytest.mark.parametrize("page", [16, 32])
def test_small_pages_equal_the_contiguous_cache(page, Hq, Hkv, D, layout, cluster):
    slots, lens = 640, [1, 15, 16, 17, 31, 33, 95, 97, 127, 128, 129, 200, 255, 257, 500, 640, 0]
    B = len(lens)
    g = torch.Generator(device="cuda").manual_seed(page + Hq + D)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, ck, cv, kn, vn = mk(B, Hq, D), mk(B, Hkv, slots, D), mk(B, Hkv, slots, D), mk(B, 1, Hkv, D), mk(B, 1, Hkv, D)
    kv_lens = torch.tensor(lens, dtype=torch.int32, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_DECODE, B, Hq, Hkv, D, slots)
    n = slots // page
    table = torch.randperm(B * n + 3, generator=g, device="cuda")[:B * n].view(B, n).to(torch.int32)
    pk, pv = (pool_of(c, page, table, B * n + 3, layout) for c in (ck, cv))
    with l4l.decode_override(cluster=cluster, warp=0):
        want, got = torch.empty_like(q), torch.empty_like(q)
        l4l.l4l_attn_decode(q, want, ck, cv, kv_lens, slots, D ** -0.5, ws)
        l4l.l4l_attn_decode_paged(q, got, pk, pv, table, kv_lens, slots, D ** -0.5, ws)
        assert torch.equal(want.view(torch.int16), got.view(torch.int16))
        l4l.l4l_attn_decode_append(q, want, ck, cv, kn, vn, kv_lens, slots, D ** -0.5, ws)
        l4l.l4l_attn_decode_paged_append(q, got, pk, pv, table, kn, vn, kv_lens, slots, D ** -0.5, ws)
    assert l4l.l4l_last_device_error(ws) == 0
    assert torch.equal(want.view(torch.int16), got.view(torch.int16))
    for c, p in ((ck, pk), (cv, pv)):                      # the newest row went to the right page, and nothing else changed
        assert torch.equal(c.view(torch.int16), torch.stack([p[table[b].long()].transpose(0, 1).flatten(1, 2) for b in range(B)]).view(torch.int16))


@pytest.mark.parametrize("cluster", [0, -1])
@pytest.mark.parametrize("Hkv", [1, 2])
@pytest.mark.parametrize("page", [16, 32])
def test_a_pool_of_one_page(page, Hkv, cluster):
    """Outer extents of 1, whose strides address nothing: whatever they are, the map is a valid one."""
    g = torch.Generator(device="cuda").manual_seed(page + Hkv)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, ck, cv = mk(1, 4 * Hkv, 128), mk(1, Hkv, page, 128), mk(1, Hkv, page, 128)
    lens, table = torch.tensor([page - 3], dtype=torch.int32, device="cuda"), torch.zeros(1, 1, dtype=torch.int32, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_DECODE, 1, 4 * Hkv, Hkv, 128, page)
    strides = [(0, 8), (8, 16), (1 << 40, 1 << 41)] if Hkv == 1 else [(0, page * 128), (1 << 41, page * 128)]
    with l4l.decode_override(cluster=cluster, warp=0):
        want, got = torch.empty_like(q), torch.empty_like(q)
        l4l.l4l_attn_decode(q, want, ck, cv, lens, page, 128 ** -0.5, ws)
        for sp, sh in strides:
            pk, pv = (c.as_strided((1, Hkv, page, 128), (sp, sh, 128, 1)) for c in (ck, cv))
            l4l.l4l_attn_decode_paged(q, got.zero_(), pk, pv, table, lens, page, 128 ** -0.5, ws)
            assert torch.equal(want.view(torch.int16), got.view(torch.int16))
