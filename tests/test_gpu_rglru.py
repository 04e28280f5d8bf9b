"""l4l_rglru_scan (gated linear recurrence of the RecurrentGemma block) against the fp64 oracle.

Tolerance. y is rounded to bf16 (2^-9 relative) and the kernel uses hardware approximations (tanh.approx for the two
sigmoids: ~2.5e-4 absolute each; ex2.approx). An error d in the recurrence gate changes ln a by 8 softplus(a_param) d;
over the state's memory horizon (about 1 / |ln a| steps) that accumulates to a relative error of about d / r in the
carried state, i.e. below 1e-3 unless the gate is nearly closed. For the O(1) data used here the attention tolerances
(max-abs 2e-2, mean-abs 2e-3) hold with margin and are asserted tighter: max-abs 1e-2, mean-abs 1.5e-3."""
import numpy as np
import pytest
import torch

from oracle import l4l_oracle as orc
from paper_2608_21836_b200 import binding as l4l
from helpers import Guarded, nan_bf16

pytestmark = pytest.mark.gpu
SENTINEL = 0x4D4D


def make(B, T, W, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(B, T, W, generator=g).to(torch.bfloat16)
    gx = (torch.randn(B, T, W, generator=g) * 2).to(torch.bfloat16)
    ga = (torch.randn(B, T, W, generator=g) * 2).to(torch.bfloat16)
    # a^8-style initialisation: a at r = 1 between 0.9 and 0.999  ->  softplus(a_param) = -ln(a) / 8
    a_max = torch.rand(W, generator=g) * 0.099 + 0.9
    sp = -torch.log(a_max) / 8
    a_param = torch.log(torch.expm1(sp))
    h0 = torch.randn(B, W, generator=g)
    return x, gx, ga, a_param.float(), h0.float()


def check(y_gpu, st_gpu, y_ref, st_ref, valid):
    got = y_gpu.float().cpu().double().numpy()
    err = np.abs(got - y_ref)[valid]
    assert np.isfinite(got[valid]).all()
    assert err.max() <= 1e-2, f"max-abs {err.max():.3g}"
    assert err.mean() <= 1.5e-3, f"mean-abs {err.mean():.3g}"
    assert torch.isfinite(st_gpu).all()
    serr = np.abs(st_gpu.cpu().double().numpy() - st_ref)
    assert serr.max() <= 5e-3, f"state max-abs {serr.max():.3g}"


@pytest.mark.parametrize("B,T,W", [(2, 300, 2560), (1, 1237, 200), (3, 65, 40), (1, 1, 64), (5, 1000, 96), (1, 16, 64), (2, 17, 128),
                                   (4, 300, 2560), (4, 600, 2560), (5, 520, 2440), (19, 530, 512)])
def test_rglru_matches_oracle(B, T, W):
    """Sequences of many tiles (eight warps hand the state on from tile to tile), of exactly one tile (sixteen steps, which
    have a kernel of their own) and just past it; a second segment inside a sequence, ragged lengths, a channel count that does not fill
    the last strip; launches of 149 to 200 strips, which the library cuts into 32- or 16-channel strips (a warp
    then owns two or four consecutive time tiles)."""
    if (B, W) in ((4, 2560), (5, 2440), (19, 512)):                    # 160, 195 and 152 strips at 64 channels
        assert l4l.l4l_rglru_strip_channels(B, T, W) in (16, 32)
        assert l4l.l4l_rglru_strip_channels(4, 600, 2560) == 16 and l4l.l4l_rglru_strip_channels(4, 300, 2560) == 32
    x, gx, ga, ap, h0 = make(B, T, W, 1100 + T)
    pos = torch.arange(T, dtype=torch.int32).repeat(B, 1)
    if T > 40:
        pos[0, 37:] = torch.arange(T - 37, dtype=torch.int32)        # a second segment inside sequence 0
    lens = [T] + [max(1, T - 7 * i) for i in range(1, B)]
    # rows past a sequence's length are caller memory that may hold anything: NaN there must reach neither y nor the state
    dead = torch.arange(T).view(1, T, 1) >= torch.tensor(lens).view(B, 1, 1)
    nan = nan_bf16((1,))
    x, gx, ga = torch.where(dead, nan, x), torch.where(dead, nan, gx), torch.where(dead, nan, ga)
    y_ref, st_ref = orc.rglru(x, gx, ga, ap.numpy(), state=h0.double().numpy(), position=pos.numpy(), seq_len=lens)
    gy = Guarded(torch.full((B, T, W), SENTINEL, dtype=torch.int16).view(torch.bfloat16))
    gs = Guarded(h0)
    ws = l4l.new_rglru_workspace(B, T, W)
    l4l.l4l_rglru_scan(x.cuda(), gx.cuda(), ga.cuda(), ap.cuda(), gs.t, gy.t, ws, position=pos.cuda(),
                       seq_lens=torch.tensor(lens, dtype=torch.int32).cuda())
    torch.cuda.synchronize()
    assert l4l.l4l_last_device_error(ws) == 0
    assert gy.margins_intact() and gs.margins_intact()
    valid = np.arange(T)[None, :, None] < np.array(lens)[:, None, None]
    valid = np.broadcast_to(valid, (B, T, W))
    check(gy.t, gs.t, y_ref, st_ref, valid)
    assert (gy.t.cpu().view(torch.int16).numpy()[~valid] == SENTINEL).all()          # rows past seq_len untouched


@pytest.mark.parametrize("B,T,W", [(1, 1, 8), (3, 1, 264), (70, 1, 256), (4, 2, 2560), (3, 7, 264), (3, 8, 256), (3, 9, 1032), (5, 16, 520)])
def test_rglru_few_steps(B, T, W):
    """Decode steps and short chunks (no tiles, a thread per channel pair): around the eight steps taken at once and the 128 pairs of a
    block, with empty and ragged sequences, resets inside and rows past the end that hold NaN."""
    x, gx, ga, ap, h0 = make(B, T, W, 77 + T)
    # halved, so that all |y| < 4: half a bf16 ulp is 7.8e-3 there and 1.6e-2 above, beyond the absolute bound of check()
    h0, x = 0.5 * h0, 0.5 * x
    pos = torch.arange(5, 5 + T, dtype=torch.int32).repeat(B, 1)
    pos[0] = torch.arange(T)
    pos[-1, T // 2:] = torch.arange(T - T // 2)
    lens = [T] + [(T - 2 * i) % (T + 1) if T > 1 else i % 2 for i in range(1, B)]    # (one step: empty and not in turn)
    lens[-1] = 0 if B > 2 and T == 1 else lens[-1]
    dead = torch.arange(T).view(1, T, 1) >= torch.tensor(lens).view(B, 1, 1)
    nan = nan_bf16((1,))
    x, gx, ga = torch.where(dead, nan, x), torch.where(dead, nan, gx), torch.where(dead, nan, ga)
    y_ref, st_ref = orc.rglru(x, gx, ga, ap.numpy(), state=h0.double().numpy(), position=pos.numpy(), seq_len=lens)
    gy = Guarded(torch.full((B, T, W), SENTINEL, dtype=torch.int16).view(torch.bfloat16))
    gs = Guarded(h0)
    ws = l4l.new_rglru_workspace(B, T, W)
    l4l.l4l_rglru_scan(x.cuda(), gx.cuda(), ga.cuda(), ap.cuda(), gs.t, gy.t, ws, position=pos.cuda(),
                       seq_lens=torch.tensor(lens, dtype=torch.int32).cuda())
    torch.cuda.synchronize()
    assert gy.margins_intact() and gs.margins_intact()
    valid = np.broadcast_to(np.arange(T)[None, :, None] < np.array(lens)[:, None, None], (B, T, W))
    check(gy.t, gs.t, y_ref, st_ref, valid)
    assert (gy.t.cpu().view(torch.int16).numpy()[~valid] == SENTINEL).all()


def test_rglru_chunks_carry_the_state():
    """A prompt of 200 steps, then single steps (the decode regime): same as one pass over all of it."""
    B, T, W = 2, 205, 128
    x, gx, ga, ap, h0 = make(B, T, W, 7)
    y_ref, st_ref = orc.rglru(x, gx, ga, ap.numpy(), state=np.zeros((B, W)),
                              position=np.tile(np.arange(T, dtype=np.int32), (B, 1)))
    dx, dgx, dga, dap = x.cuda(), gx.cuda(), ga.cuda(), ap.cuda()
    state = torch.zeros(B, W, device="cuda")
    y = torch.zeros(B, T, W, dtype=torch.bfloat16, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, 1, 1, 1, 64, 1)
    pos = torch.arange(200, dtype=torch.int32, device="cuda").repeat(B, 1)
    y0 = torch.zeros(B, 200, W, dtype=torch.bfloat16, device="cuda")
    l4l.l4l_rglru_scan(dx[:, :200].contiguous(), dgx[:, :200].contiguous(), dga[:, :200].contiguous(), dap, state, y0, ws,
                       position=pos)
    y[:, :200] = y0
    for t in range(200, T):
        y1 = torch.zeros(B, 1, W, dtype=torch.bfloat16, device="cuda")
        l4l.l4l_rglru_scan(dx[:, t:t + 1].contiguous(), dgx[:, t:t + 1].contiguous(), dga[:, t:t + 1].contiguous(), dap,
                           state, y1, ws)
        y[:, t] = y1[:, 0]
    torch.cuda.synchronize()
    assert l4l.l4l_last_device_error(ws) == 0
    check(y, state, y_ref, st_ref, np.ones((B, T, W), bool))


def test_rglru_rejects_bad_shapes():
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, 1, 1, 1, 64, 1)
    x = torch.zeros(1, 4, 12, dtype=torch.bfloat16, device="cuda")                  # W not a multiple of 8
    with pytest.raises(l4l.L4LError):
        l4l.l4l_rglru_scan(x, x.clone(), x.clone(), torch.zeros(12, device="cuda"), torch.zeros(1, 12, device="cuda"),
                           x.clone(), ws)


def test_rglru_empty_inputs_are_a_no_op():
    ws = l4l.new_workspace(l4l.L4L_OP_PREFILL, 1, 1, 1, 64, 1)
    state = torch.full((2, 64), 7.0, device="cuda")
    e = torch.zeros(2, 0, 64, dtype=torch.bfloat16, device="cuda")
    l4l.l4l_rglru_scan(e, e.clone(), e.clone(), torch.zeros(64, device="cuda"), state, e.clone(), ws)
    # all sequences of length 0: the state comes back unchanged
    x = torch.randn(2, 8, 64, device="cuda").to(torch.bfloat16)
    y = torch.full((2, 8, 64), 3.0, device="cuda").to(torch.bfloat16)
    l4l.l4l_rglru_scan(x, x.clone(), x.clone(), torch.zeros(64, device="cuda"), state, y, ws,
                       seq_lens=torch.zeros(2, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert (state == 7.0).all() and (y == 3.0).all() and l4l.l4l_last_device_error(ws) == 0


def segment_steps(T, channels, segments):
    steps = 16 * (64 // channels)                                  # whole rounds of 8 warps' tiles
    return -(-(-(-T // steps)) // (8 * segments)) * 8 * steps


# every kernel that is built for cut launches, two and four segments, with positions and without
@pytest.mark.parametrize("B,T,W,positions,shape", [
    (4, 8192, 2560, True, (32, 4)), (5, 8007, 2048, True, (32, 4)), (6, 2049, 4096, True, (32, 2)), (6, 6000, 4096, False, (32, 4)),
    (2, 5133, 2560, True, (16, 4)), (2, 8192, 2560, False, (16, 4)), (16, 2048, 2560, True, (64, 2)), (8, 4096, 2560, True, (64, 4))])
def test_rglru_time_segments(B, T, W, positions, shape):
    """Launches that the library cuts into segments of the time axis (a workspace with room for the counters) against the
    same launch uncut (a workspace of the status block alone), which takes the same steps in the same order: equal bit
    for bit. Lengths: all, the end of a segment and one past it, none, one step, all but one; resets; a second call finds the
    counters at zero."""
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert l4l.l4l_rglru_launch_shape(B, T, W, positions) == shape
    assert l4l.l4l_rglru_launch_shape(B, T, W, positions)[1] > 1 and l4l.l4l_rglru_launch_shape(B, T, W, positions, 256)[1] == 1
    x, gx, ga, ap, h0 = (t.cuda() for t in make(B, T, W, 1900 + T))
    seg = segment_steps(T, *shape)
    assert (T - 1) // seg + 1 == shape[1]
    lens = ([T, seg + 1, seg, 0, 1, T - 1] + [T] * B)[:B]
    none = 3 if B > 3 else None
    lens = torch.tensor(lens, dtype=torch.int32, device="cuda")
    pos = torch.arange(T, dtype=torch.int32, device="cuda").repeat(B, 1) if positions else None
    if positions:
        pos[0, seg:] -= seg                                        # a reset on the first step of a segment, and one inside
        pos[0, seg + 900:] -= 900
    cut = l4l.new_rglru_workspace(B, T, W).view(torch.uint8)
    uncut = cut[:256].clone()
    outs = []
    for ws in (uncut, cut, cut):
        y, st = torch.zeros_like(x), h0.clone()
        l4l.l4l_rglru_scan(x, gx, ga, ap, st, y, ws, position=pos, seq_lens=lens)
        assert l4l.l4l_last_device_error(ws) == 0
        outs.append((y, st))
    assert int(cut[256:].max()) == 0
    for y, st in outs[1:]:
        assert torch.equal(y.view(torch.int16), outs[0][0].view(torch.int16)) and torch.equal(st, outs[0][1])
    assert torch.isfinite(outs[0][0]).all() and (none is None or torch.equal(outs[0][1][none], h0[none]))


@pytest.mark.parametrize("B,T,W,positions", [(2, 5133, 2560, True), (6, 2049, 4096, True), (2, 8192, 2560, False)])
def test_rglru_cut_launches_match_the_oracle(B, T, W, positions):
    assert l4l.l4l_rglru_launch_shape(B, T, W, positions)[1] > 1
    x, gx, ga, ap, h0 = make(B, T, W, 2100 + T)
    pos = torch.arange(T, dtype=torch.int32).repeat(B, 1) + (0 if positions else 1)     # no position 0: no resets
    if positions:
        pos[0, 1900:] -= 1900
    lens = [T] + [T - 400 * i for i in range(1, B)]
    y_ref, st_ref = orc.rglru(x, gx, ga, ap.numpy(), state=h0.double().numpy(), position=pos.numpy(), seq_len=lens)
    y, st = torch.zeros(B, T, W, dtype=torch.bfloat16, device="cuda"), h0.cuda()
    ws = l4l.new_rglru_workspace(B, T, W)
    l4l.l4l_rglru_scan(x.cuda(), gx.cuda(), ga.cuda(), ap.cuda(), st, y, ws, position=pos.cuda() if positions else None,
                       seq_lens=torch.tensor(lens, dtype=torch.int32).cuda())
    assert l4l.l4l_last_device_error(ws) == 0
    check(y, st, y_ref, st_ref, np.broadcast_to(np.arange(T)[None, :, None] < np.array(lens)[:, None, None], (B, T, W)))
