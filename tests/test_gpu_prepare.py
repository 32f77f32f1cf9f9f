"""rf_sparse_call takes the decision, the tile schedule and the reordered copies in one launch; the entry points it stands for
take a launch each.  Both ways have to give the same classes, windows, lists and output bits."""
import pytest
import torch

import gpu_util as gu
from paper_2505_21036_b200 import api

pytestmark = pytest.mark.gpu

BW = [0.125, 0.5]


def call(shape, params, q, k, v, bw, ws_bytes, one):
    """(classes, windows, count, lists, kv_len, bitmap, o, lse, status) by one call, or by three."""
    mem = gu.Guarded()
    B, H, N, D = q.shape
    ws = mem.alloc((ws_bytes,), torch.uint8, 255, "ws")
    sched = api.Schedule(shape, params, "cuda", with_bitmap=True)
    cls, win, status = (mem.alloc(s, torch.int32, f, n) for s, f, n in (((B, H), -9, "class"), ((B, H), -9, "window"), ((1,), 0, "status")))
    o, lse = mem.alloc((B, H, N, D), torch.bfloat16, float("nan"), "o"), mem.alloc((B, H, N), torch.float32, float("nan"), "lse")
    w = win if bw else None
    if one:
        api.rf_sparse_call(shape, params, bw, q, k, v, cls, w, sched, o, lse, ws, status)
    else:
        if bw:
            api.rf_arm_classify_plus(shape, params, bw, q, k, cls, win, None, ws, status)
        else:
            api.rf_arm_classify(shape, params, q, k, cls, None, ws, status)
        api.rf_build_block_mask_plus(shape, params, cls, w, sched, status)
        api.rf_sparse_attn_fwd_plus(shape, params, q, k, v, cls, w, sched, o, lse, ws, status)
    torch.cuda.synchronize()
    mem.check("one call" if one else "three calls")
    listed = torch.arange(sched.nKmax, device="cuda") < sched.count[..., None]
    return cls, win, sched.count, sched.kv_tile * listed, sched.kv_len, sched.bitmap, o, lse, status


@pytest.mark.parametrize("bw", [None, BW])
@pytest.mark.parametrize("B,H,D,T,fh,fw,L,omega,opt", [
    (1, 1, 64, 1, 7, 9, 0, 1, {}),                                     # one query tile, one score CTA
    (1, 3, 96, 10, 12, 16, 226, 10, {}),                               # fewer items than SMs: tickets
    (2, 5, 128, 7, 19, 27, 77, 7, dict(textural_stride=3)),
    (1, 40, 64, 5, 11, 23, 16, 300, dict(sample_mode=api.RF_SAMPLE_GLOBAL)),
    (1, 6, 128, 40, 9, 14, 3, 2, dict(temporal_permute=0, two_mask=1)),  # stride sample of many score CTAs
    (1, 6, 64, 9, 45, 61, 0, 9, dict(spatial_key_first_frame=1)),
    (1, 3, 96, 6, 20, 21, 40, 5, dict(temporal_window_2d=(5, 6))),
    (2, 48, 64, 5, 20, 21, 9, 6, {}),                                  # a copying CTA takes several steps
    (2, 48, 64, 9, 20, 21, 9, 6, {}),                                  # more copying CTAs than a head's share, four steps each
])
def test_one_call_gives_what_three_give(B, H, D, T, fh, fw, L, omega, opt, bw):
    if bw and "temporal_window_2d" in opt:
        bw = None
    shape = api.make_shape(B, H, D, T, fh, fw, L)
    params = api.make_params(max(T // 4, 1), fh * fw // 4, sample_stride=omega, **opt)
    S, N = fh * fw, T * fh * fw + L
    g = torch.Generator("cuda").manual_seed(N + D)
    q, k, v = (torch.randn(B, H, N, D, device="cuda", generator=g) for _ in range(3))
    for h in range(H):                                                 # a frame's tokens alike, a position's, or neither
        p = torch.randn((T, 1, D) if h % 3 == 0 else (1, S, D), device="cuda", generator=g) * (1.8 if h % 3 < 2 else 0.0)
        for x in (q, k):
            x[:, h, :T * S].view(B, T, S, D).add_(p)
    q, k, v = (x.to(torch.bfloat16).contiguous() for x in (q, k, v))
    full = api.rf_workspace_bytes(shape, params)
    first = call(shape, params, q, k, v, bw, full, False)
    assert int(first[-1]) == 0 and bool(((first[0] >= 0) & (first[0] < 3)).all())
    for size in (full, full + 4096):
        for a, b in zip(first, call(shape, params, q, k, v, bw, size, True)):
            assert torch.equal(a, b) or (a.is_floating_point() and torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(), b.nan_to_num()))


@pytest.mark.parametrize("bw", [None, BW])
@pytest.mark.parametrize("B,H,D,T,fh,fw,L,omega", [(1, 3, 64, 4, 8, 8, 16, 4), (2, 5, 96, 7, 19, 27, 77, 7)])
def test_a_sparse_call_reports_a_score_kernel_that_gave_up(B, H, D, T, fh, fw, L, omega, bw):
    """The call's launches with the score kernel's failure flag set in place of that kernel: the merged launch must hand the code on,
    write class and window -1, list every tile, reorder nothing and leave a call that ends; the next call is a normal one."""
    shape = api.make_shape(B, H, D, T, fh, fw, L)
    params = api.make_params(max(T // 4, 1), fh * fw // 4, sample_stride=omega)
    N = T * fh * fw + L
    g = torch.Generator("cuda").manual_seed(N)
    q, k, v = (torch.randn(B, H, N, D, device="cuda", generator=g).to(torch.bfloat16) for _ in range(3))
    mem = gu.Guarded()
    ws = mem.alloc((api.rf_workspace_bytes(shape, params),), torch.uint8, 0x5A, "ws")
    sched = api.Schedule(shape, params, "cuda")
    cls, win, status = (mem.alloc(s, torch.int32, f, n) for s, f, n in (((B, H), -9, "class"), ((B, H), -9, "window"), ((1,), 0, "status")))
    o, lse = mem.alloc((B, H, N, D), torch.bfloat16, float("nan"), "o"), mem.alloc((B, H, N), torch.float32, float("nan"), "lse")
    w = win if bw else None
    api.rf_selftest_sparse_call_abandoned(shape, params, bw, q, k, v, cls, w, sched, o, lse, ws, status)
    torch.cuda.synchronize()
    mem.check("abandoned call")
    assert int(status.item()) == 5                                     # RF_ERR_TIMEOUT
    assert bool((cls == -1).all()) and bool((win == (-1 if bw else -9)).all())
    assert bool((sched.count == sched.nKmax).all()) and bool((sched.kv_len == N).all())
    assert torch.equal((sched.kv_tile & 0x7FFFFFFF).reshape(-1, sched.nKmax),
                       torch.arange(sched.nKmax, device="cuda", dtype=torch.int32).expand(B * H * sched.nQ, -1))
    copies = 3 * (-(-B * H * N * D * 2 // 256) * 256)
    assert bool((ws[:copies] == 0x5A).all())
    dense, dense_lse = torch.empty_like(q), torch.empty_like(lse)      # (its pieces may be cut elsewhere: equal but for rounding)
    api.rf_dense_attn_fwd(shape, q, k, v, dense, dense_lse)
    assert float((o.float() - dense.float()).abs().max()) < 2 * gu.O_MAX_ABS and float((lse - dense_lse).abs().max()) < 2 * gu.LSE_ABS
    status.zero_()
    full = ws.numel()
    for a, b in zip(call(shape, params, q, k, v, bw, full, False), call(shape, params, q, k, v, bw, full, True)):
        assert torch.equal(a, b) or (a.is_floating_point() and torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(), b.nan_to_num()))
    api.rf_sparse_call(shape, params, bw, q, k, v, cls, w, sched, o, lse, ws, status)
    assert int(status.item()) == 0 and bool((cls >= 0).all())
