"""Chunks over caches of different lengths run their row blocks in the order of their work: every block exactly once, whatever
the mix of lengths. Checked bit for bit against one launch per sequence, which has nothing to order."""
import numpy as np
import pytest
import torch

from paper_2608_21836_b200 import binding as l4l

pytestmark = pytest.mark.gpu
SENTINEL = 0x4D4D


@pytest.mark.parametrize("B,Hq,Hkv,D", [(2, 4, 2, 64), (31, 4, 2, 64), (33, 3, 1, 64), (70, 2, 1, 128), (128, 5, 5, 64), (129, 4, 2, 64)])
def test_row_blocks_by_work_cover_every_row_once(B, Hq, Hkv, D):
    r = np.random.default_rng(B)
    S, slots = 520, 1200
    past, qlen = r.integers(0, slots - S + 1, B).astype(np.int32), r.integers(0, S + 1, B).astype(np.int32)
    past[r.integers(0, B, B // 2)] = 256                       # equal weights, and sequences with nothing to do
    qlen[r.integers(0, B, B // 4)] = 0
    past[0], qlen[0] = 0, S
    g = torch.Generator(device="cuda").manual_seed(B)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.bfloat16)  # noqa: E731
    q, kn, vn, ck, cv = mk(B, S, Hq, D), mk(B, S, Hkv, D), mk(B, S, Hkv, D), mk(B, Hkv, slots, D), mk(B, Hkv, slots, D)
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, B, Hq, Hkv, D, S)
    outs = []
    for step in (B, 1):
        o, k2, v2 = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16), ck.clone(), cv.clone()
        pa, ql = torch.from_numpy(past).cuda(), torch.from_numpy(qlen).cuda()
        for b in range(0, B, step):
            e = slice(b, b + step)
            l4l.l4l_attn_prefill_chunk_append(q[e], kn[e], vn[e], o[e], k2[e], v2[e], pa[e], ql[e], D ** -0.5, ws)
        assert l4l.l4l_last_device_error(ws) == 0
        outs.append([t.view(torch.int16) for t in (o, k2, v2)])
    for a, b in zip(*outs):
        assert torch.equal(a, b)
    # the chunk read back from the cache by the other entry point, without the write
    o = torch.full_like(q.view(torch.int16), SENTINEL).view(torch.bfloat16)
    l4l.l4l_attn_prefill_chunk(q, o, outs[0][1].view(torch.bfloat16), outs[0][2].view(torch.bfloat16), pa, ql, D ** -0.5, ws)
    assert torch.equal(o.view(torch.int16), outs[0][0])
