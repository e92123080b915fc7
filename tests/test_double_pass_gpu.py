"""The double-precision pass over flagged frames at the edges of its tiles (eight query rows, eight keys, eight warps), against the
oracle: a margin that no frame passes sends all of them through it."""
import numpy as np
import pytest
import torch

from oracle import mukv_oracle as O
from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3])                      # (a single frame is split over the device)
@pytest.mark.parametrize("q_heads,kv_heads,head_dim,tokens,bf16,over", [
    (1, 1, 128, 2, True, {}),                              # one tile of two rows, seven warps without a key
    (4, 2, 64, 9, False, {}),                              # a row more than a tile
    (2, 2, 64, 63, False, dict(attn_causal=1)),            # eight tiles, the last one ragged
    (6, 2, 64, 65, True, dict(attn_causal=1)),             # two tiles in one warp; causal: shares without a visible key
    (6, 2, 64, 65, True, dict(path=1)),                    # flagged by the multiply-add kernel
    (28, 4, 128, 196, True, {}),
    (16, 2, 128, 256, False, dict(keep_low_freq=1)),       # all tiles full
    (4, 4, 64, 100, True, dict(past_frames=3)),            # 175 keys, the cached ones first
])
def test_flagged_frames(n, q_heads, kv_heads, head_dim, tokens, bf16, over):
    spec = StreamSpec(seed=91, n_layers=2, n_q_heads=q_heads, n_kv_heads=kv_heads, head_dim=head_dim, tokens_per_frame=tokens,
                      bf16=bf16, n_outlier=1, n_frames=6, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    options = {B.OPT_FLAG_MARGIN: 4.0, B.OPT_SCORE_PATH: over.get("path", 0)}
    over = {k: v for k, v in over.items() if k != "path"}
    run = H.GpuRun(dict(spec=spec, keep=max(1, tokens // 4), fseg=4, chunk=n, alpha=0.7), options=options, **over).compress()
    st = O.Store(H.oracle_cfg(run.cfg))
    for t0 in range(0, 6, n):
        kv = [spec.frame_kv(t) for t in range(t0, t0 + n)]
        O.compress_chunk(st, np.stack([spec.frame_q(t) for t in range(t0, t0 + n)]), np.stack([x[0] for x in kv], axis=1),
                         np.stack([x[1] for x in kv], axis=1))
    H.check_frames_against_oracle(run, st, range(6), full_layers=True)
    for t in range(6):
        for s in range(3):
            # exact up to the rounding to single precision, half a unit in the last place of 24 bits; the fused score
            # cancels against the minimum, so its error is one of values up to 1 in double precision
            np.testing.assert_allclose(run.scores[s, t], st.scores[t][s], rtol=2.0 ** -24 * 1.01, atol=1e-12)
    stats = run.ctx.mukv_get_stats()
    assert stats.refined_frames == 6 and stats.device_status == 0
    seg = run.ctx.region(3).cpu().numpy()
    for u in range(st.n_segments):
        sk, sv = st.segment_entry(u)
        H.close(seg[u][:, 0], sk, f"segment entry K {u}")
        H.close(seg[u][:, 1], sv, f"segment entry V {u}")
    torch.cuda.synchronize()
