"""fp32 chunks on the tensor cores (every value as three bf16 terms), against the oracle."""
import numpy as np
import pytest

from oracle import mukv_oracle as O
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


def test_fp32_five_scoring_layers_up_to_what_the_terms_may_take_and_beyond():
    # 24.1 MB of terms per frame: eleven frames fit the 256 MB, a call of twelve is scored by the multiply-add kernel (a kernel
    # less: no splitting)
    spec = StreamSpec(seed=63, n_layers=5, n_q_heads=28, n_kv_heads=4, head_dim=128, tokens_per_frame=196, bf16=False, n_outlier=2,
                      n_frames=12, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=49, fseg=4, chunk=12, alpha=0.7), n_score_layers=5)
    gen = H.torch.Generator(device=run.device).manual_seed(64)
    q0, k, v = run.gs.chunk(0, 12)
    q = H.torch.stack([q0] + [H.torch.randn(q0.shape, device=run.device, generator=gen) for _ in range(4)])
    st = O.Store(H.oracle_cfg(run.cfg))
    O.compress_chunk(st, *(H.to_numpy_bits(x) for x in (q, k, v)))
    before = 0
    for n, kernels in ((11, 4), (12, 3), (3, 4)):
        run.ctx.mukv_reset()
        kept = H.torch.full((n, 49), -1, dtype=H.torch.int32, device=run.device)
        sc = H.torch.zeros((3, n, 196), device=run.device)
        run.ctx.mukv_compress_chunk(q[:, :n].contiguous(), k[:, :n].contiguous(), v[:, :n].contiguous(), n, 0, kept, sc)
        run.kept, run.scores = kept.cpu().numpy(), sc.cpu().numpy()
        assert H.check_frames_against_oracle(run, st, range(n), full_layers=True) < H.FLAG_MARGIN / 2
        stats = run.ctx.mukv_get_stats()
        assert stats.device_status == 0 and stats.kernel_launches - before == kernels
        before = stats.kernel_launches
