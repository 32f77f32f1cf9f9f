"""The row sums that normalise O come out of the same contraction as O (a column of ones behind V).  With V constant along the
keys every O is that constant times sum / sum: exact for powers of two, whatever the keys, masks, splits and raises of the
running maximum were."""
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
