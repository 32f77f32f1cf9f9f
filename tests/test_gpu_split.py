"""Split items of the attention kernel: shapes of few items, whose tile lists are cut into pieces that several CTAs work
off and one joins.  Sizes at the edges of the plan: fewer items than SMs, an odd number of query tiles, no text rows, a
partial last wave whose tail begins inside a row of heads."""
import numpy as np
import pytest

import gpu_util as gu
from oracle import rainfusion_oracle as orc
from paper_2505_21036_b200 import synth

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
