"""Prefill launches whose CTAs go on with blocks that have not started (more than 512 new tokens, more blocks than SMs):
what the short launches of the other prefill tests check, on the kernel that those do not reach."""
import math

import numpy as np
import pytest
import torch

from oracle import l4l_oracle as orc
from paper_2608_21836_b200 import binding as l4l
from helpers import Guarded, bits_equal, nan_bf16
from test_gpu_prefill import sentinel_bf16
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
