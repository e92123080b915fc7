"""fp32 chunks on the tensor cores (every value as three bf16 terms), against the oracle."""
import numpy as np
import pytest

from oracle import mukv_oracle as O  # noqa: F401  (the harness compares with it)
from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q_heads,kv_heads,head_dim,tokens,over", [
    (2, 1, 64, 17, {}),                                    # one ragged tile, fewer key rows than DFT rows
    (28, 4, 128, 196, {}),                                 # ragged query tiles (18 tokens x 7 heads), two DFT tiles
    (16, 2, 128, 256, {}),                                 # the largest key tile: four slots of 32 KB, the rings at their smallest
    (6, 2, 64, 128, dict(attn_causal=1)),                  # exactly one DFT tile
    (8, 8, 64, 130, dict(keep_low_freq=1)),                # one query head per key head, two rows in the second tile
])
def test_fp32_chunks_in_bf16_terms(q_heads, kv_heads, head_dim, tokens, over):
    spec = StreamSpec(seed=61, n_layers=2, n_q_heads=q_heads, n_kv_heads=kv_heads, head_dim=head_dim, tokens_per_frame=tokens,
                      bf16=False, n_outlier=2, n_frames=5, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=3)
    run = H.GpuRun(dict(spec=spec, keep=max(1, tokens // 4), fseg=2, chunk=3, alpha=0.7), **over).compress()
    st = H.oracle_stream(spec, H.oracle_cfg(run.cfg), range(5), last_only=False, workers=1)
    # Ids and bytes as the oracle has them.  The bound on the fused scores is what the library's choice between single and
    # double precision rests on: the kept set cannot change below half the margin.
    worst = H.check_frames_against_oracle(run, st, range(5), full_layers=True)
    assert worst < H.FLAG_MARGIN / 2
    assert run.ctx.mukv_get_stats().device_status == 0


def test_fp32_values_that_are_not_finite():
    spec = StreamSpec(seed=62, n_layers=1, n_q_heads=4, n_kv_heads=2, head_dim=64, tokens_per_frame=40, bf16=False, n_outlier=0,
                      n_frames=2)
    run = H.GpuRun(dict(spec=spec, keep=10, fseg=2, chunk=2, alpha=0.7))
    q, k, v = run.gs.chunk(0, 2)
    k[0, 1, 5, 0, 3] = float("inf")
    kept = H.torch.zeros((2, 10), dtype=H.torch.int32, device=run.device)
    run.ctx.mukv_compress_chunk(q, k, v, 2, 0, kept)
    assert kept[1].tolist() == list(range(10))             # no ranking: the lowest ids
    assert run.ctx.mukv_get_stats().device_status == 7
    st = H.oracle_stream(spec, H.oracle_cfg(run.cfg), range(1), last_only=False, workers=1)
    assert kept[0].tolist() == np.asarray(st.kept[0]).tolist()
    assert B.FP32 == run.cfg.dtype
