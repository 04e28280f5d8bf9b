"""Chunks over caches of different lengths run their row blocks in the order of their work: every block exactly once, whatever
the mix of lengths. Checked bit for bit against one launch per sequence, which has nothing to order."""
import numpy as np
import pytest
import torch

from paper_2608_21836_b200 import binding as l4l

pytestmark = pytest.mark.gpu
SENTINEL = 0x4D4D
i32 = lambda a: torch.from_numpy(np.asarray(a, np.int32)).cuda()  # noqa: E731


# ranked launches from just beyond two blocks per SM (B = 31: 310) to many, head pairs and single heads; by place: few blocks, B > 32
@pytest.mark.parametrize("page", [0, 16, 256])
@pytest.mark.parametrize("B,Hq,Hkv,D", [(2, 4, 2, 64), (2, 64, 8, 64), (31, 4, 2, 64), (32, 5, 5, 64), (32, 4, 2, 128), (33, 3, 1, 64),
                                         (70, 2, 1, 128), (128, 5, 5, 64), (129, 4, 2, 64)])
def test_row_blocks_by_work_cover_every_row_once(B, Hq, Hkv, D, page):
    r = np.random.default_rng(B)
    S, slots = 520, 1280
    past, qlen = r.integers(0, slots - S + 1, B).astype(np.int32), r.integers(0, S + 1, B).astype(np.int32)
    past[r.integers(0, B, B // 2)] = 256                       # equal weights, and sequences with nothing to do
    qlen[r.integers(0, B, B // 4)] = 0
    past[0], qlen[0] = 0, S
    by_work = l4l.l4l_prefill_row_block_order(i32(past), i32(qlen), S, slots, Hq, Hkv, D) is not None
    assert by_work == ((B, Hq) in ((2, 64), (31, 4), (32, 5), (32, 4)))
    g = torch.Generator(device="cuda").manual_seed(B)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, kn, vn = mk(B, S, Hq, D), mk(B, S, Hkv, D), mk(B, S, Hkv, D)
    if page:
        n = slots // page
        ck, cv = mk(B * n, Hkv, page, D), mk(B * n, Hkv, page, D)
        table = torch.randperm(B * n, generator=g, device="cuda").view(B, n).to(torch.int32)
    else:
        ck, cv, table = mk(B, Hkv, slots, D), mk(B, Hkv, slots, D), None
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    outs = []
    for step in (B, 1):
        o, k2, v2 = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16), ck.clone(), cv.clone()
        pa, ql = i32(past), i32(qlen)
        for b in range(0, B, step):
            e = slice(b, b + step)
            c = slice(None) if page else e
            l4l.l4l_attn_prefill_chunk_append(q[e], kn[e], vn[e], o[e], k2[c], v2[c], pa[e], ql[e], D ** -0.5, ws,
                                              block_table=table[e] if page else None)
        assert l4l.l4l_last_device_error(ws) == 0
        outs.append([t.view(torch.int16) for t in (o, k2, v2)])
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    if not page:      # the chunk read back from the cache by the other entry point, without the write
        o = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16)
        l4l.l4l_attn_prefill_chunk(q, o, outs[0][1].view(torch.bfloat16), outs[0][2].view(torch.bfloat16), pa, ql, D ** -0.5, ws)
        assert torch.equal(o.view(torch.int16), outs[0][0])


# the kernel with a block per item (S <= 512) ranks its row blocks too
@pytest.mark.parametrize("page", [0, 64])
@pytest.mark.parametrize("B,Hq,Hkv,D", [(12, 32, 8, 128), (32, 10, 2, 64), (31, 5, 5, 128)])
def test_ranked_short_chunks(B, Hq, Hkv, D, page):
    """The same bits as one launch per sequence, which has nothing to order."""
    r = np.random.default_rng(B)
    S, slots = 500, 1280
    past, qlen = r.integers(0, slots - S + 1, B).astype(np.int32), r.integers(0, S + 1, B).astype(np.int32)
    past[: B // 3], qlen[: B // 6], past[-1], qlen[-1] = 256, 0, 0, S
    assert l4l.l4l_prefill_row_block_order(i32(past), i32(qlen), S, slots, Hq, Hkv, D) is not None
    g = torch.Generator(device="cuda").manual_seed(B)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, kn, vn = mk(B, S, Hq, D), mk(B, S, Hkv, D), mk(B, S, Hkv, D)
    n = slots // page if page else 0
    ck, cv = (mk(B * n, Hkv, page, D) if page else mk(B, Hkv, slots, D) for _ in range(2))
    table = torch.randperm(B * n, generator=g, device="cuda").view(B, n).to(torch.int32) if page else None
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    outs = []
    for step in (B, 1):
        o, k2, v2 = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16), ck.clone(), cv.clone()
        for b in range(0, B, step):
            e = slice(b, b + step)
            c = slice(None) if page else e
            l4l.l4l_attn_prefill_chunk_append(q[e], kn[e], vn[e], o[e], k2[c], v2[c], i32(past)[e], i32(qlen)[e], D ** -0.5, ws,
                                              block_table=table[e] if page else None)
        assert l4l.l4l_last_device_error(ws) == 0
        outs.append([t.view(torch.int16) for t in (o, k2, v2)])
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("G", [2, 3])
@pytest.mark.parametrize("B", [2, 7, 31, 32])
def test_the_order_is_by_work(B, G):
    """Every row block that holds rows once, heaviest first (equal weights by sequence), none after the last."""
    r = np.random.default_rng(10 * B + G)
    S, slots, Hq = 900, 8192, 60 * G
    rows, shift = (128, 0) if G % 2 == 0 else (256, 1)
    for kind in ("spread", "few", "groups"):
        past, qlen = r.integers(0, slots - S, B), r.integers(0, S + 1, B)
        if kind == "few":
            past, qlen = r.integers(0, 3, B) * 128, r.choice([0, 1, 128, 129, S], B)
            past[0], past[-1] = 0, 256
        if kind == "groups":
            past = np.where(np.arange(B) < B // 2, 0, 4000)
        order = l4l.l4l_prefill_row_block_order(i32(past), i32(qlen), S, slots, Hq, Hq // G, 64).cpu().numpy().tolist()
        want = sorted((-(-(-p // 128) + ((qb + 1) << shift)), b, qb) for b, (p, n) in enumerate(zip(past.tolist(), qlen.tolist()))
                      for qb in range(-(-n // rows)))
        assert order[:len(want)] == [[b, qb] for _, b, qb in want] and all(e == [-1, -1] for e in order[len(want):])


@pytest.mark.parametrize("past", [0, 640])
def test_equal_pasts_keep_the_order_of_places(past):
    B, S, G = 9, 700, 4
    qlen = [700, 1, 129, 0, 300, 128, 699, 512, 257]
    order = l4l.l4l_prefill_row_block_order(i32([past] * B), i32(qlen), S, 4096, 32, 8, 128).cpu().numpy().tolist()
    assert order == [[b, qb] if qb * 128 < qlen[b] else [-1, -1] for qb in reversed(range(6)) for b in range(B)]


def test_where_the_order_is_by_place():
    lens = lambda B: (i32(np.arange(B) * 100), i32([500] * B))  # noqa: E731
    order = lambda B, slots, Hq=32: l4l.l4l_prefill_row_block_order(*lens(B), 500, slots, Hq, Hq // 4, 128)  # noqa: E731
    assert order(8, 8192) is not None
    assert order(8, 627) is None and order(8, 628) is not None       # no room for a tile ahead of the chunk
    assert order(1, 8192, 256) is None                                # one sequence
    assert order(33, 8192) is None and order(32, 8192) is not None
    assert order(4, 8192) is None                                     # 256 blocks: less than two per SM


# several items per CTA (S > 512: a CTA goes on with blocks that have not started; B = 33: empty row blocks are passed over one by one), and a
# block per item, against launches of at most one block per SM
@pytest.mark.parametrize("B,Hq,Hkv,D,S", [(7, 32, 8, 128, 520), (32, 6, 2, 128, 700), (33, 12, 4, 64, 300), (33, 12, 4, 64, 530), (32, 12, 12, 64, 513),
                                          (2, 64, 8, 128, 2000)])
def test_prompts_of_uneven_length_in_one_launch(B, Hq, Hkv, D, S):
    """Fresh prompts, empty and short ones among them, with the cache written in the same launch (whole tiles and ragged ends, room behind
    the prompt and too little of it): the same bits as one launch per sequence and group of heads."""
    r = np.random.default_rng(B + S)
    lens = r.integers(0, S + 1, B).astype(np.int32)
    lens[:2] = S, 0 if B > 2 else 1
    lens[-1] = min(256, S)
    g = torch.Generator(device="cuda").manual_seed(B)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, k, v = mk(B, S, Hq, D), mk(B, S, Hkv, D), mk(B, S, Hkv, D)
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    G, ln = Hq // Hkv, i32(lens)
    assert B * (-(-S // 128) * Hq // 2 if G % 2 == 0 else -(-S // 256) * Hq) > torch.cuda.get_device_properties(0).multi_processor_count
    for slots in (S + 37, S - 70):
        outs = []
        for whole in (True, False):
            o = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16)
            ck, cv = (torch.full((B, Hkv, slots, D), SENTINEL, dtype=torch.int16, device="cuda").view(torch.bfloat16) for _ in range(2))
            if whole:
                l4l.l4l_attn_prefill(q, k, v, o, ln, D ** -0.5, ws, cache_k=ck, cache_v=cv)
            else:
                for b in range(B):
                    for h in range(Hkv):
                        e, hq, hk = slice(b, b + 1), slice(h * G, (h + 1) * G), slice(h, h + 1)
                        l4l.l4l_attn_prefill(q[e, :, hq], k[e, :, hk], v[e, :, hk], o[e, :, hq], ln[e], D ** -0.5, ws, cache_k=ck[e, hk],
                                             cache_v=cv[e, hk])
            assert l4l.l4l_last_device_error(ws) == 0
            outs.append([t.view(torch.int16) for t in (o, ck, cv)])
        for a, b in zip(*outs):
            assert torch.equal(a, b)
