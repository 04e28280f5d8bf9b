"""The order of the sums in the decode kernels is part of their results: builds stay comparable bit for bit. Inputs on which the
order decides, so that every other order is off by far more than a rounding."""
import math

import pytest
import torch

from paper_2608_21836_b200 import binding as l4l

pytestmark = pytest.mark.gpu
KERNELS = {"split": dict(cluster=0, warp=0), "cluster": dict(cluster=1, warp=0), "warp": dict(cluster=0, warp=1)}
SHAPES = [(8, 2, 128), (24, 2, 128), (10, 2, 128), (4, 4, 64), (18, 2, 64)]


def decode(kernel, fp8, Hq, Hkv, D, q, k, v, scale):
    """q [D], k, v [16, D] as every query head of one sequence of 16 tokens sees them; o [Hq, D] and lse [Hq]."""
    lens = torch.tensor([16], dtype=torch.int32, device="cuda")
    q = q.to(torch.bfloat16).cuda().expand(1, Hq, D).contiguous()
    k, v = (t.to(torch.float8_e4m3fn if fp8 else torch.bfloat16).cuda().expand(1, Hkv, 16, D).contiguous() for t in (k, v))
    o, lse = torch.empty_like(q), torch.empty(1, Hq, device="cuda")
    ws = l4l.new_workspace(l4l.L4L_OP_DECODE, 1, Hq, Hkv, D, 16)
    with l4l.decode_override(**KERNELS[kernel]):
        if fp8:
            ones = torch.ones(Hkv, device="cuda")
            l4l.l4l_attn_decode_fp8(q, o, k, v, ones, ones, lens, 16, scale, ws, lse=lse)
        else:
            l4l.l4l_attn_decode(q, o, k, v, lens, 16, scale, ws, lse=lse)
    assert l4l.l4l_last_device_error(ws) == 0
    return o[0].float().cpu(), lse[0].cpu()


def cases(f):
    return pytest.mark.parametrize("kernel,fp8", [(k, f8) for f8 in (False, True) for k in KERNELS])(
        pytest.mark.parametrize("Hq,Hkv,D", SHAPES)(f))


@cases
def test_scores_are_one_sum_over_the_head_dims_in_order(kernel, fp8, Hq, Hkv, D):
    """A large product in the first 16 head dims, a small one in the second and the large one's negative in the third: summed in
    order in 24 bits the small one is lost (it lies 29 bits or more below), whatever the token, and all weights are equal."""
    q, k, v = torch.zeros(D), torch.zeros(16, D), torch.arange(16.0).repeat(D, 1).T.clone()
    q[0] = q[32] = 2.0 ** 13
    k[:, 0], k[:, 32] = 256.0, -256.0                          # products of 2^21
    q[16] = 2.0 ** -8
    k[:, 16] = torch.arange(16.0) / 16                         # products below 2^-8
    o, lse = decode(kernel, fp8, Hq, Hkv, D, q, k, v, 2.0 ** 12)   # ... which the scale would make scores of up to 15
    assert torch.equal(o, torch.full_like(o, 7.5))
    assert (lse - math.log(16)).abs().max() < 1e-5


@cases
def test_denominators_are_sums_of_the_tokens_of_a_fragment(kernel, fp8, Hq, Hkv, D):
    """Weights 1 at token 0 and 2^-24 at tokens 1 and 9, 0 elsewhere. A lane sums tokens 2c, 2c + 1, 2c + 8 and 2c + 9 of a block: 2^-24 is
    half a unit in the last place of 1 and is lost twice. Token 1 and token 9 added to one another first would make 1 + 2^-23, whose
    logarithm is 1.2e-7."""
    q, k, v = torch.zeros(D), torch.zeros(16, D), torch.ones(16, D)
    q[0] = 1.0
    k[:, 0] = -448.0
    k[0, 0], k[1, 0], k[9, 0] = 0.0, -24.0, -24.0
    o, lse = decode(kernel, fp8, Hq, Hkv, D, q, k, v, math.log(2.0))
    assert torch.equal(o, torch.ones_like(o)) and (lse == 0).all()
