"""Split items of the attention kernel: shapes of few items, whose tile lists are cut into pieces that several CTAs work
off and one joins.  Sizes at the edges of the plan: fewer items than SMs, an odd number of query tiles, no text rows, a
partial last wave whose tail begins inside a row of heads."""
import ctypes as C

import numpy as np
import pytest
import torch

import gpu_util as gu
from oracle import rainfusion_oracle as orc
from paper_2505_21036_b200 import api, synth
from paper_2505_21036_b200.layer import RainFusionAttention

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,D,T,fh,fw,L,omega", [
    (1, 3, 96, 10, 12, 16, 226, 10),
    (2, 3, 64, 9, 13, 17, 61, 9),
    (1, 5, 128, 8, 16, 24, 0, 8),
    (1, 7, 64, 16, 24, 29, 77, 40),
])
def test_split_items_match_the_oracle(B, H, D, T, fh, fw, L, omega):
    wl = synth.Workload(name="split", B=B, H=H, D=D, T=T, frame_h=fh, frame_w=fw, L_text=L, frame_window=T // 4,
                        spatial_window=fh * fw // 4, textural_stride=2, sample_mode=0, sample_stride=omega, alpha=0.9, amp=2.0,
                        config_id=9)
    run = gu.Run(wl)
    cls, _ = run.arm()
    run.build()
    sparse, again, dense = run.sparse(), run.sparse(), run.dense()
    assert all(np.array_equal(x, y) for x, y in zip(sparse, again))     # pieces are joined in order, whoever joins them
    rows = np.unique(np.concatenate([np.random.default_rng(5).choice(wl.N, 96, replace=False), [0, 127, 128, wl.N - 1]]))
    for (o, lse), classes in ((sparse, cls), (dense, np.full_like(cls, orc.DENSE))):
        for b in range(B):
            for h in range(H):
                ref, lref = orc.masked_attention(run.q_bits[b, h], run.k_bits[b, h], run.v_bits[b, h], int(classes[b, h]),
                                                 gu.geom(wl), gu.pparams(wl), rows=rows)
                gu.check_attention(o[b, h][rows], lse[b, h][rows], ref, lref, f"head {b},{h}", strict=False)
        assert np.isfinite(o).all() and np.isfinite(lse).all()


def test_pairs_that_list_no_tile_between_others():
    """A caller's schedule may leave query tiles without any key tile: their rows are not written, and the items before and
    after such a pair on the same CTA (more pairs than SMs, so a CTA works off several) give the bits they give without it."""
    wl = synth.small_workload("empty", H=64, D=64, T=6, fh=12, fw=11, L=37, wf=1, ws=20, tau=2, mode=0, omega=6)
    run = gu.Run(wl)
    run.force_classes([h % 4 for h in range(wl.H)])
    run.build()
    o, lse = run.sparse()
    none = np.zeros((wl.H, run.sched.nQ), dtype=bool)
    rng = np.random.default_rng(3)
    for h in range(wl.H):
        for pair in range(-(-run.sched.nQ // 2)):
            kind = rng.integers(4)                     # both tiles, one of them, or neither keeps its list
            none[h, 2 * pair:2 * pair + 2] = {0: True, 1: [True, False][:run.sched.nQ - 2 * pair], 2: False, 3: False}[int(kind)]
    run.sched.count[0, torch.from_numpy(none).cuda()] = 0
    o2, lse2 = run.outputs()
    api.rf_sparse_attn_fwd(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.sched, o2, lse2, run.ws, run.status)
    torch.cuda.synchronize()
    assert int(run.status.item()) == 0
    run.mem.check("attention with empty lists")
    slot = np.arange(wl.N)
    for h in range(wl.H):
        tok = slot.copy()
        if h % 4 == orc.TEMPORAL:                      # position-major slots
            tok[:wl.Nv] = (slot[:wl.Nv] % wl.T) * wl.S + slot[:wl.Nv] // wl.T
        written = np.empty(wl.N, dtype=bool)
        written[tok] = ~none[h, slot // 128]
        got_o, got_l = o2[0, h].float().cpu().numpy(), lse2[0, h].cpu().numpy()
        assert np.isnan(got_o[~written]).all() and np.isnan(got_l[~written]).all(), h
        assert np.array_equal(got_o[written], o[0, h][written]) and np.array_equal(got_l[written], lse[0, h][written]), h


def small_split(**kw):
    """The first shape above: 27 items of 9 tiles, every one of them in two pieces."""
    base = dict(name="split", B=1, H=3, D=96, T=10, frame_h=12, frame_w=16, L_text=226, frame_window=2, spatial_window=48,
                textural_stride=2, sample_mode=0, sample_stride=10, alpha=0.9, amp=2.0, config_id=9)
    base.update(kw)
    return synth.Workload(**base)


def attention(run, call, params=None, windows=None):
    """One call of an entry point that takes the sparse arguments; (o, lse) as the bits they hold."""
    o, lse = run.outputs()
    call(run.shape, params or run.params, run.q, run.k, run.v, run.head_class, windows, run.sched, o, lse, run.ws, run.status)
    torch.cuda.synchronize()
    assert int(run.status.item()) == 0
    return gu.bits_of(o).copy(), lse.cpu().numpy().view(np.uint32).copy()


def same_bits(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def test_one_reordering_serves_calls_of_other_sampling_parameters():
    """rf_sparse_attn_reordered depends on the copies alone: neither the sampling stride of the reordering nor what the rest
    of the workspace holds may matter, and a second call finds what the first one found."""
    run = gu.Run(small_split())
    run.force_classes([0, 1, 2])
    run.build()
    ref = attention(run, api.rf_sparse_attn_fwd_plus)
    other = api.params_of(small_split(sample_stride=5))
    run.ws = run.mem.alloc((max(api.rf_workspace_bytes(run.shape, p) for p in (run.params, other)),), torch.uint8, 0x5A, "ws")
    api.rf_reorder_tokens(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.ws)
    for _ in range(2):
        assert same_bits(attention(run, api.rf_sparse_attn_reordered, other), ref)
    run.mem.check("rf_sparse_attn_reordered")


def test_a_dense_call_leaves_the_workspace_it_is_given_alone():
    """rf_dense_attn_fwd takes a workspace for the sake of one calling form and uses none of it: copies that
    rf_reorder_tokens left there survive.  The form with a scratch block of its own gives the same attention."""
    run = gu.Run(small_split())
    run.force_classes([0, 1, 2])
    run.build()
    ref = attention(run, api.rf_sparse_attn_fwd_plus)
    lib, n = api.load(), api.load().rf_dense_workspace_bytes(C.byref(run.shape))
    assert n > 0
    run.ws = run.mem.alloc((run.ws.numel() + n,), torch.uint8, name="ws")
    scratch = run.mem.alloc((n,), torch.uint8, 0x5A, "scratch")

    def dense(call, block):
        o, lse = run.outputs()
        code = call(C.byref(run.shape), run.q.data_ptr(), run.k.data_ptr(), run.v.data_ptr(), o.data_ptr(), lse.data_ptr(),
                    block.data_ptr(), block.numel(), run.status.data_ptr(), None)
        torch.cuda.synchronize()
        assert code == 0 and int(run.status.item()) == 0
        return o.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64)

    api.rf_reorder_tokens(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.ws)
    before = run.ws.clone()
    plain, split = dense(lib.rf_dense_attn_fwd, run.ws), dense(lib.rf_dense_attn_fwd_split, scratch)
    assert torch.equal(run.ws, before)
    assert same_bits(attention(run, api.rf_sparse_attn_reordered), ref)
    for h in range(run.wl.H):
        gu.check_attention(split[0][0, h], split[1][0, h], plain[0][0, h], plain[1][0, h], f"head {h}", strict=False)
    run.mem.check("dense calls")


def test_a_workspace_without_room_for_pieces_still_serves():
    """A block sized for seven heads (224 items: none is split) serves six (192 items, the last 44 in pieces), although six
    need more for themselves: the copies and ARM's scratch fit."""
    shapes = [small_split(H=h, D=64, T=16, frame_h=16, frame_w=32, L_text=0, sample_stride=16, frame_window=4, spatial_window=128)
              for h in (7, 6)]
    seven, six = (api.rf_workspace_bytes(api.shape_of(w), api.params_of(w)) for w in shapes)
    assert seven < six
    run = gu.Run(shapes[1])
    ref_cls, ref_rec = run.arm()
    run.build()
    ref = run.sparse()
    run.ws = run.mem.alloc((seven,), torch.uint8, 0x5A, "ws")
    cls, rec = run.arm()
    assert np.array_equal(cls, ref_cls) and np.array_equal(rec, ref_rec)
    whole = run.sparse()
    for h in range(run.wl.H):
        gu.check_attention(whole[0][0, h], whole[1][0, h], ref[0][0, h], ref[1][0, h], f"head {h}", strict=False)
    bits = attention(run, api.rf_sparse_attn_fwd_plus)
    api.rf_reorder_tokens(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.ws)
    assert same_bits(attention(run, api.rf_sparse_attn_reordered), bits)
    run.mem.check("workspace without pieces")
    # the host pipeline's block: without the room the groups' pieces would take, the call's bits are those of whole items
    lib, pipe = api.load(), C.c_void_p()
    full = lib.rf_host_pipeline_staging_bytes(C.byref(run.shape), C.byref(run.params), 2)
    staging = torch.empty(full, dtype=torch.uint8, device="cuda")
    assert lib.rf_host_pipeline_create(C.byref(run.shape), C.byref(run.params), 2, staging.data_ptr(), full - (1 << 20), C.byref(pipe)) == 0
    q, k, v, o = (t.cpu().pin_memory() for t in (run.q, run.k, run.v, torch.zeros_like(run.q)))
    assert lib.rf_host_pipeline_run(pipe, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), None) == 0
    lib.rf_host_pipeline_destroy(pipe)                 # waits
    assert np.array_equal(gu.bits_of(o), bits[0])
    run.ws = run.ws[:3 * run.q.numel() * 2]            # no room for ARM's scratch either: refused as ever
    with pytest.raises(api.RainFusionError, match="workspace"):
        run.arm()


def test_rows_that_list_no_tile_are_not_written_in_a_split_item_either():
    """One query tile of a split pair without an entry: its rows stay as they are, the other tile's are what they were."""
    run = gu.Run(small_split())
    run.force_classes([orc.SPATIAL, orc.SPATIAL, orc.TEXTURAL])   # original order: a tile's rows are its tokens
    run.build()
    o, lse = run.sparse()
    run.sched.count[0, :, 3] = 0
    o2, lse2 = run.outputs()
    api.rf_sparse_attn_fwd(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.sched, o2, lse2, run.ws, run.status)
    torch.cuda.synchronize()
    assert int(run.status.item()) == 0
    got_o, got_l = o2.float().cpu().numpy(), lse2.cpu().numpy()
    none = np.zeros(run.wl.N, dtype=bool)
    none[3 * 128:4 * 128] = True
    assert np.isnan(got_o[:, :, none]).all() and np.isnan(got_l[:, :, none]).all()
    assert np.array_equal(got_o[:, :, ~none], o[:, :, ~none]) and np.array_equal(got_l[:, :, ~none], lse[:, :, ~none])


def test_a_dense_call_does_without_scratch(monkeypatch):
    """The scratch of a dense call is no necessity: with none left in torch's allocator, or with a tensor of the caller's
    that is too small, the items stay whole; a tensor that is large enough gives the bits of the default."""
    run = gu.Run(small_split())
    n = api.load().rf_dense_workspace_bytes(C.byref(run.shape))
    own, none = run.mem.alloc((n,), torch.uint8, 0x5A, "scratch"), run.mem.alloc((0,), torch.uint8, name="none")

    def dense(**kw):
        o, lse = run.outputs()
        api.rf_dense_attn_fwd(run.shape, run.q, run.k, run.v, o, lse, run.status, **kw)
        torch.cuda.synchronize()
        assert int(run.status.item()) == 0
        run.mem.check("rf_dense_attn_fwd")
        return gu.bits_of(o).copy(), lse.cpu().numpy().view(np.uint32).copy()

    split = dense()

    def exhausted(*args, **kw):
        raise torch.OutOfMemoryError("none left")
    monkeypatch.setattr(torch, "empty", exhausted)
    without = dense()
    assert same_bits(dense(scratch=own), split) and same_bits(dense(scratch=none), without) and not same_bits(split, without)


def check_rows(run, out, classes, windows=None, key_first=False, t2d=None):
    """96 rows of every head and the last one against the oracle."""
    wl = run.wl
    rows = np.unique(np.concatenate([np.random.default_rng(5).choice(wl.N, 96, replace=False), [wl.N - 1]]))
    for h in range(wl.H):
        pp = gu.pparams(wl, key_first, t2d)
        if windows is not None:
            w = int(windows[h])
            pp = orc.PatternParams(w if classes[h] == orc.SPATIAL else wl.frame_window,
                                   w if classes[h] == orc.TEMPORAL else wl.spatial_window, wl.textural_stride)
        ref, lref = orc.masked_attention(run.q_bits[0, h], run.k_bits[0, h], run.v_bits[0, h], int(classes[h]), gu.geom(wl), pp,
                                         rows=rows)
        gu.check_attention(out[0][0, h][rows], out[1][0, h][rows], ref, lref, f"head {h} class {classes[h]}", strict=False)


@pytest.mark.parametrize("permute", [0, 1])
@pytest.mark.parametrize("D", [64, 128])
def test_split_items_with_the_other_readings_of_the_patterns(D, permute):
    run = gu.Run(small_split(D=D), temporal_permute=permute, t2d=(3, 4), key_first=1)
    classes = [orc.SPATIAL, orc.TEMPORAL, orc.TEXTURAL]
    run.force_classes(classes)
    run.build()
    check_rows(run, run.sparse(), classes, key_first=True, t2d=(3, 4))


def test_split_items_with_a_window_per_head():
    run = gu.Run(small_split())
    classes, windows, _ = run.arm_plus([0.125, 0.25, 0.5])
    run.build_plus()
    check_rows(run, run.sparse_plus(), classes[0], windows[0])


@pytest.mark.parametrize("shape", [dict(), dict(T=4, L_text=37)])      # in pieces, whole
@pytest.mark.parametrize("D", [64, 96, 128])
def test_output_without_lse_is_the_output_with_it(D, shape):
    run = gu.Run(small_split(D=D, **shape))
    run.force_classes([0, 1, 2])
    run.build()
    o, lse = run.outputs()

    def both(call):
        bits = []
        for wanted in (lse, None):
            o.fill_(float("nan"))
            call(wanted)
            torch.cuda.synchronize()
            assert int(run.status.item()) == 0
            bits.append(gu.bits_of(o).copy())
        assert np.array_equal(*bits) and np.isfinite(o.float().cpu().numpy()).all()
    both(lambda l: api.rf_sparse_attn_fwd(run.shape, run.params, run.q, run.k, run.v, run.head_class, run.sched, o, l, run.ws, run.status))
    both(lambda l: api.rf_dense_attn_fwd(run.shape, run.q, run.k, run.v, o, l, run.status))


# four heads: every item in pieces; six: the last 44 of 192, which begin inside the second of two groups
FOUR = small_split(H=4)
SIX = small_split(H=6, D=64, T=16, frame_h=16, frame_w=32, L_text=0, sample_stride=16, frame_window=4, spatial_window=128)
# a group of one head has no pieces by itself but those of the call, and ARM's scratch is so small (50 tokens a frame, three
# sampled tokens) that the pieces' tickets lie where the sums of its recalls do: they cannot be cleared by the launch that reads those
MEETING = small_split(H=2, D=64, T=624, frame_h=5, frame_w=10, L_text=226, sample_stride=12384, frame_window=156, spatial_window=12)


def test_the_shapes_here_have_items_in_pieces():
    """Their workspaces hold more than the reordered copies and ARM's rows, else the tests around this one show little."""
    for wl in (small_split(), FOUR, SIX):
        rows = -(-max(wl.S, -(-wl.Nv // wl.sample_stride)) // 64) * 64
        others = 3 * wl.H * wl.N * wl.D * 2 + 2 * wl.H * 9 * rows * 4
        piece = 2 * 128 * (wl.D + 4) * 4
        assert api.rf_workspace_bytes(api.shape_of(wl), api.params_of(wl)) > others + 2 * piece


@pytest.mark.parametrize("bandwidths", [None, [0.125, 0.25, 0.5]])
@pytest.mark.parametrize("wl,groups", [(FOUR, 1), (FOUR, 2), (FOUR, 4), (SIX, 2), (SIX, 3), (SIX, 6), (MEETING, 2)])
def test_split_items_of_a_call_in_groups_of_heads(wl, groups, bandwidths):
    """The plan is the whole call's, whichever heads a group holds: the output's bits are the resident call's."""
    shape, params = api.shape_of(wl), api.params_of(wl)
    host = [torch.from_numpy(x.view(np.int16)).view(torch.bfloat16).pin_memory() for x in synth.make_qkv(wl)]
    oh = torch.full(host[0].shape, float("nan"), dtype=torch.bfloat16).pin_memory()
    pipe = api.HostPipeline(shape, params, "cuda", groups)
    pipe.set_bandwidths(bandwidths or [])
    for _ in range(2):
        pipe.run(*host, oh)
    assert pipe.status() == 0
    resident = RainFusionAttention(shape, params, "cuda", dense_fraction=0.0, bandwidths=bandwidths)
    q, k, v = (t.cuda() for t in host)
    o = torch.empty_like(q)
    resident(q, k, v, o)
    resident.check()
    assert torch.equal(oh.view(torch.int16), o.cpu().view(torch.int16))
    pipe.close()


def test_split_items_in_a_replayed_graph():
    shape, params = api.shape_of(FOUR), api.params_of(FOUR)
    eager, graphed = (RainFusionAttention(shape, params, "cuda", dense_fraction=0.0, graph=g) for g in (False, True))
    q, k, v = (gu.to_dev(x) for x in synth.make_qkv(FOUR))
    og, oe = torch.empty_like(q), torch.empty_like(q)
    for _ in range(3):
        graphed(q, k, v, og)
        eager(q, k, v, oe)
        torch.cuda.synchronize()
        assert torch.equal(og.view(torch.int16), oe.view(torch.int16))
        q.copy_(torch.roll(q.clone(), 1, dims=1))          # other classes, other lists, other pieces
    eager.check()
    graphed.check()
