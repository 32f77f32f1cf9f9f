"""The row sums that normalise O come out of the same contraction as O (a column of ones behind V).  With V constant along the
keys every O is that constant times sum / sum: exact for powers of two, whatever the keys, masks, splits and raises of the
running maximum were.  With V zero but for one dominant key O shows the sums themselves."""
import math

import pytest
import torch

from paper_2505_21036_b200 import api, layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 96, 128])
@pytest.mark.parametrize("B,H,T,fh,fw,L", [(1, 1, 2, 5, 7, 0), (1, 1, 1, 16, 16, 1), (2, 3, 5, 11, 13, 29), (1, 9, 6, 20, 23, 77), (2, 30, 7, 16, 17, 40)])
def test_constant_values_come_back(D, B, H, T, fh, fw, L):
    shape = api.make_shape(B, H, D, T, fh, fw, L)
    params = api.make_params(max(T // 4, 1), fh * fw // 4, sample_stride=3)
    N = T * fh * fw + L
    g = torch.Generator("cuda").manual_seed(D + N)
    q, k = (torch.randn(B, H, N, D, device="cuda", generator=g) for _ in range(2))
    k *= torch.linspace(0.5, 12.0, N, device="cuda")[None, None, :, None]       # later keys raise the running maximum
    v = (2.0 ** (torch.arange(D, device="cuda") % 5 - 2)).expand(B, H, N, D)
    q, k, v = (x.to(torch.bfloat16).contiguous() for x in (q, k, v))
    attn = layer.RainFusionAttention(shape, params, "cuda")
    for step, lse in ((0, None), (0, True), (9, None), (9, True)):              # dense and sparse, both instances of the kernel
        o = torch.full_like(q, float("nan"))
        l = torch.full((B, H, N), float("nan"), device="cuda") if lse else None
        attn(q, k, v, o, lse=l, step=step, num_steps=10)
        attn.check()
        assert torch.equal(o, v), (step, lse)
        assert l is None or bool(torch.isfinite(l).all())


@pytest.mark.parametrize("D,lse", [(64, False), (64, True), (96, False), (128, True)])
def test_many_small_weights_beside_a_large_one(D, lse):
    """One key of weight 1, 262 143 of about 2^-19: together they weigh 0.2 to 1.2.  Added up tile by tile in fp32 the row sum
    is off by half a unit of its last place a tile at most, 2048 * 2^-24 = 1.2e-4; in an accumulator that holds the whole row every
    small weight is cut off at that place, 2.6e-3 in all."""
    N = 1 << 18
    shape = api.make_shape(1, 1, D, 4, 256, 256, 0)
    g = torch.Generator("cuda").manual_seed(D)
    sc = 1.4426950408889634 / math.sqrt(D)
    x = (7.5 + torch.rand(N, device="cuda", generator=g)).to(torch.bfloat16)          # queries and keys along one dimension
    y = (-9.5 / (8 * sc) + 0.3 * torch.randn(N, device="cuda", generator=g)).to(torch.bfloat16)
    y[0] = 9.5 / (8 * sc)
    q, k, v = (torch.zeros(1, 1, N, D, device="cuda", dtype=torch.bfloat16) for _ in range(3))
    q[0, 0, :, 0], k[0, 0, :, 0] = x, y
    v[0, 0, 0] = 1 + torch.arange(D, device="cuda") / D
    o = torch.full_like(q, float("nan"))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.rf_dense_attn_fwd(shape, q, k, v, o, torch.empty(1, 1, N, device="cuda") if lse else None, status)
    rows = torch.arange(N // 2, N, N // 1024, device="cuda")      # of items that are not cut into pieces (those are the first ones)
    exponent = x[rows].double()[:, None] * (y.double() - y[0].double())[None] * sc
    ref = v[0, 0, 0].double()[None] / torch.exp2(exponent).sum(1, keepdim=True)
    assert int(status.item()) == 0
    # against the rounded reference: both round alike where the sums agree
    bias = float((o[0, 0][rows].double() / ref.to(torch.bfloat16).double() - 1).mean())
    assert abs(bias) < 1.5e-4, bias
