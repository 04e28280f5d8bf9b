"""Prefill launches whose CTAs go on with blocks that have not started (more than 512 new tokens, more blocks than SMs):
what the short launches of the other prefill tests check, on the kernel that those do not reach."""
import math

import numpy as np
import pytest
import torch

from oracle import l4l_oracle as orc
from paper_2608_21836_b200 import binding as l4l
from helpers import Guarded, assert_close_to_oracle, bits_equal, nan_bf16
from test_gpu_prefill import check_prefill, poison_padding, rand_qkv, sentinel_bf16
from test_gpu_prefill_chunk_append import as_bf16, check_outputs, make_chunk

pytestmark = pytest.mark.gpu
S = 530


def items(B, Hq, Hkv):
    """The launch's blocks; the tests below are about launches that have more of them than the GPU has SMs."""
    n = B * (-(-S // 128) * Hq // 2 if (Hq // Hkv) % 2 == 0 else -(-S // 256) * Hq)
    assert n > torch.cuda.get_device_properties(0).multi_processor_count
    return n


PAST = [0, 1, 127, 128, 129, 300, 511, 64, 700, 5, 256, 90]
QLEN = [257, 128, 1, 129, 200, 5, 130, 0, 64, S, 256, 383]


# a page of 0: a contiguous cache. Groups of query heads that share the rows of a key tile evenly and unevenly, in pairs and singly; ranked
# launches (more than two blocks per SM) and others
@pytest.mark.parametrize("page", [0, 16, 64, 256])
@pytest.mark.parametrize("Hq,Hkv,D", [(8, 2, 128), (20, 2, 128), (5, 1, 128), (16, 1, 64), (5, 5, 64)])
def test_chunks_append_every_row_and_attend(Hq, Hkv, D, page):
    """Chunks over caches that hold NaN from their past on, in pages whose table maps what is used and no more."""
    past, qlen, B, Lmax = PAST, QLEN, len(PAST), 1280
    items(B, Hq, Hkv)
    (q, kn, vn), g = make_chunk(B, S, Hq, Hkv, D, qlen, seed=40 + page + Hq)
    dead = torch.arange(Lmax).view(1, 1, Lmax, 1) >= torch.tensor(past).view(B, 1, 1, 1)
    ck, cv = (torch.where(dead, nan_bf16((1,)), torch.randn(B, Hkv, Lmax, D, generator=g).to(torch.bfloat16)) for _ in range(2))
    pa, ql, scale = np.array(past, np.int32), np.array(qlen, np.int32), 1.0 / math.sqrt(D)
    ek, ev = orc.kv_append(ck, cv, kn, vn, pa, ql)
    ref, ref_lse = orc.prefill_chunk(q, as_bf16(ek), as_bf16(ev), pa, ql, scale)
    table = None
    if page:
        n = Lmax // page
        table = torch.randperm(B * n + 3, generator=g)[:B * n].view(B, n).to(torch.int32)
        for b in range(B):
            table[b, -(-(past[b] + qlen[b]) // page):] = -1 if b % 2 else 10 ** 6
        pool = [nan_bf16((B * n + 3, Hkv, page, D)).clone() for _ in range(2)]
        for b in range(B):
            for i, at in enumerate(table[b].tolist()):
                if 0 <= at < B * n + 3:
                    for dst, src in zip(pool, (ck, cv)):
                        dst[at] = src[b, :, i * page:(i + 1) * page]
        ck, cv = pool
        ek, ev = orc.kv_append_paged(ck, cv, table.numpy(), kn, vn, pa, ql)
    gq, gkn, gvn, gk, gv = (Guarded(t.contiguous()) for t in (q, kn, vn, ck, cv))
    go = Guarded(sentinel_bf16((B, S, Hq, D)))
    lse = torch.full((B, Hq, S), -12345.0, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    l4l.l4l_attn_prefill_chunk_append(gq.t, gkn.t, gvn.t, go.t, gk.t, gv.t, torch.from_numpy(pa).cuda(), torch.from_numpy(ql).cuda(),
                                      scale, ws, lse=lse, block_table=table.cuda() if page else None)
    torch.cuda.synchronize()
    assert l4l.l4l_last_device_error(ws) == 0
    assert all(x.margins_intact() for x in (gq, gkn, gvn, gk, gv, go))
    assert bits_equal(gk.t, ek) and bits_equal(gv.t, ev)                     # exactly the chunks' rows were written
    check_outputs(go.t, lse, ref, ref_lse, qlen, B, S, Hq, "chunks")


RAGGED = [0, 1, 2, 63, 64, 65, 127, 128, 129, 200, 255, 256, 257, 300, 383, 384, 385, 511, 512, 513, S]


@pytest.mark.parametrize("token_major", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D", [(4, 2, 64), (3, 3, 64), (4, 1, 128), (5, 1, 128), (3, 3, 128)])
def test_prompts_of_ragged_lengths(Hq, Hkv, D, token_major):
    """NaN in every row past a length, margins around every buffer, log-sum-exp, caches of both orders of heads and tokens."""
    B = len(RAGGED)
    items(B, Hq, Hkv)
    q, k, v = (poison_padding(x, RAGGED) for x in rand_qkv(B, S, Hq, Hkv, D, seed=50 + D + Hq))
    check_prefill(q, k, v, RAGGED, 1.0 / math.sqrt(D), Lmax=560, token_major_cache=token_major)


# a cache that a tensor map describes, and one whose stride between sequences (there is one) no map can hold
@pytest.mark.parametrize("mapped", [True, False])
def test_views_of_a_fused_projection(mapped):
    B, Hq, Hkv, D, slots = 1, 64, 8, 128, 600
    items(B, Hq, Hkv)
    g = torch.Generator().manual_seed(61)
    qkv = torch.randn(B, S, Hq + 2 * Hkv, D, generator=g).to(torch.bfloat16)
    q, k, v = (x.contiguous() for x in qkv.split([Hq, Hkv, Hkv], 2))
    ref, _ = orc.prefill(q, k, v, np.array([S], np.int32), 0.09)
    dq, dk, dv = qkv.cuda().split([Hq, Hkv, Hkv], 2)
    o = torch.zeros(B, S, Hq, D, dtype=torch.bfloat16, device="cuda")
    bufs = [Guarded(sentinel_bf16((Hkv, slots, D))) for _ in range(2)]
    ck, cv = (x.t[None] if mapped else x.t.as_strided((1, Hkv, slots, D), (1 << 41, slots * D, D, 1), x.t.storage_offset()) for x in bufs)
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    l4l.l4l_attn_prefill(dq, dk, dv, o, torch.tensor([S], dtype=torch.int32, device="cuda"), 0.09, ws, cache_k=ck, cache_v=cv)
    torch.cuda.synchronize()
    assert l4l.l4l_last_device_error(ws) == 0
    assert_close_to_oracle(o.cpu(), ref, "fused projection")
    for x, want in zip(bufs, (k, v)):
        assert x.margins_intact() and bits_equal(x.t[:, :S], want[0].transpose(0, 1).contiguous())
        assert (x.t[:, S:].cpu().view(torch.int16) == 0x4D4D).all()


def big_call(seed):
    """Twelve ragged prompts, with room for their outputs: (call, fill with new data, outputs)."""
    B, Hq, Hkv, D = 12, 8, 2, 128
    items(B, Hq, Hkv)
    g = torch.Generator(device="cuda").manual_seed(seed)
    new = lambda h: torch.zeros(B, S, h, D, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    q, k, v, o = new(Hq), new(Hkv), new(Hkv), new(Hq)
    ck, cv = (torch.zeros(B, Hkv, S, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    n = torch.tensor(QLEN, dtype=torch.int32, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)

    def fill():
        for x in (q, k, v):
            x.normal_(generator=g)
        for x in (o, ck, cv):
            x.zero_()

    return (lambda: l4l.l4l_attn_prefill(q, k, v, o, n, D ** -0.5, ws, cache_k=ck, cache_v=cv)), fill, (o, ck, cv)


def test_in_a_cuda_graph():
    """Captured once, replayed over new data twice in a row: the bits of the same call outside a graph."""
    call, fill, outs = big_call(71)
    fill(), call(), torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
        call()
    for _ in range(3):
        fill(), call()
        want = [x.clone() for x in outs]
        for x in outs:
            x.zero_()
        graph.replay()
        assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(outs, want))


def test_two_streams_at_once():
    """Launches of two streams share the GPU: the blocks that one claims are its own."""
    calls = [big_call(seed) for seed in (81, 82)]
    wants = []
    for call, fill, outs in calls:
        fill(), call()
        wants.append([x.clone() for x in outs])
        for x in outs:
            x.zero_()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    for _ in range(10):
        for s, (call, _, _) in zip(streams, calls):
            with torch.cuda.stream(s):
                call()
    torch.cuda.synchronize()
    for (_, _, outs), want in zip(calls, wants):
        assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(outs, want))
