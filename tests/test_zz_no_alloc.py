"""mukv_score_frames_noalloc against mukv_compress_chunk and against the CPU oracle.

The entry point under test serves callers that cannot allocate device memory (everything was given
to another pool at start-up, or the allocator is off limits while they run): its scratch is a
fixed array inside the library.  The array is shared by all calls and keeps the previous call's
contents, so the check runs two different calls back to back and both must agree with the regular
entry point: kept token ids bit-exact, scores within the tolerance of the parity tests.
This file is collected last on purpose, so that a failure here cannot hide any other test.
"""
import numpy as np
import pytest
import torch

from oracle import mukv_oracle as O
from paper_2605_22269_b200 import binding as B
from tests import harness as H

pytestmark = pytest.mark.gpu


def _both_ways(name, n_frames, first):
    run = H.GpuRun(name, n_frames=first + n_frames)
    c = run.cfg
    dev = run.device
    q, k, v = run.gs.chunk(first, n_frames)
    kept_ref = torch.full((n_frames, c.keep_per_frame), -1, dtype=torch.int32, device=dev)
    sc_ref = torch.zeros((3, n_frames, c.tokens_per_frame), dtype=torch.float32, device=dev)
    # the regular entry point: frames must continue the stream, so store `first` frames before them
    if first:
        q0, k0, v0 = run.gs.chunk(0, first)
        run.ctx.mukv_compress_chunk(q0, k0, v0, first, 0)
    run.ctx.mukv_compress_chunk(q, k, v, n_frames, first, kept_ref, sc_ref)
    kept = torch.full_like(kept_ref, -2)
    sc = torch.full_like(sc_ref, -2.0)
    B.mukv_score_frames_noalloc(c, q, k[c.n_layers - 1], n_frames, kept, sc)
    torch.cuda.synchronize()
    assert kept.cpu().numpy().tolist() == kept_ref.cpu().numpy().tolist(), f"{name}: kept ids differ"
    H.close(sc.cpu().numpy(), sc_ref.cpu().numpy(), f"{name}: scores")


def test_noalloc_matches_compress_chunk_twice_in_a_row():
    _both_ways("chunk7b", 5, 0)          # bf16, 28 query heads over 4 key heads
    _both_ways("chunk7b", 3, 2)          # fewer frames than the call before: stale scratch must not matter
    _both_ways("tiny", 8, 0)             # fp32


def test_noalloc_against_the_oracle_with_another_context_created_in_between():
    # the oracle decides, not the other entry point; and a context of a smaller shape created
    # between two calls must not take the scoring kernels' shared memory away
    wl = H.workload("chunk7b")
    spec = wl["spec"]
    cfg = H.spec_config(spec, wl)
    n = 5
    from paper_2605_22269_b200.synth.gpu import GpuStream
    gs = GpuStream(spec, "cuda:0")
    q, k, v = gs.chunk(0, n)
    st = O.Store(dict(H.oracle_cfg(cfg), n_layers=1))
    O.compress_chunk(st, H.to_numpy_bits(q), H.to_numpy_bits(k[-1:]), H.to_numpy_bits(v[-1:]))
    for round_ in range(2):
        kept = torch.full((n, cfg.keep_per_frame), -2, dtype=torch.int32, device="cuda:0")
        sc = torch.full((3, n, cfg.tokens_per_frame), -2.0, dtype=torch.float32, device="cuda:0")
        B.mukv_score_frames_noalloc(cfg, q, k[cfg.n_layers - 1], n, kept, sc)
        torch.cuda.synchronize()
        for f in range(n):
            assert kept[f].cpu().numpy().tolist() == st.kept[f].tolist(), f"round {round_}: kept ids differ at frame {f}"
            for i in range(3):
                H.close(sc[i, f].cpu().numpy(), st.scores[f][i], f"round {round_}: score[{i}] frame {f}")
        if round_ == 0:
            small = H.GpuRun("tiny")                 # fp32, P = 64, D = 64: the smallest shared-memory need
            small.compress()
            B.MukvContext(H.spec_config(H.StreamSpec(seed=5, n_layers=1, n_q_heads=4, n_kv_heads=4, head_dim=64,
                                                     tokens_per_frame=196, bf16=True, n_outlier=0, n_frames=2),
                                        dict(keep=9, fseg=2, chunk=2, alpha=0.7)), "cuda:0").close()


def test_noalloc_rejects_what_does_not_fit():
    wl = H.workload("chunk7b")
    cfg = H.spec_config(wl["spec"], wl)
    x = torch.zeros(64, dtype=torch.bfloat16, device="cuda:0")
    out = torch.zeros(64, dtype=torch.int32, device="cuda:0")
    with pytest.raises(B.MukvError) as e:
        B.mukv_score_frames_noalloc(cfg, x, x, B.NOALLOC_MAX_FRAMES + 1, out, None)
    assert e.value.status == -5 and "static scratch" in str(e.value)
    with pytest.raises(B.MukvError) as e:
        B.mukv_score_frames_noalloc(cfg, x, x, 1, None, None)
    assert e.value.status == -1


def _inputs(hq, hkv, d, tokens, n, bf16, seed):
    spec = H.StreamSpec(seed=seed, n_layers=1, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, tokens_per_frame=tokens, bf16=bf16,
                        n_outlier=1, n_frames=n, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    q, k, _ = spec.chunk(0, n)
    return spec, q, k[0]


def _against_oracle(spec, q, k, n, keep, exact=(), **over):
    """exact: frames that go through the double-precision pass; their scores are the rounded exact ones."""
    cfg = H.spec_config(spec, dict(keep=keep, fseg=1, chunk=n, alpha=0.7), **over)
    kept = torch.full((n, keep), -2, dtype=torch.int32, device="cuda:0")
    sc = torch.full((3, n, spec.tokens_per_frame), -2.0, dtype=torch.float32, device="cuda:0")
    B.mukv_score_frames_noalloc(cfg, H.to_device(q, spec.bf16), H.to_device(k, spec.bf16), n, kept, sc)
    kept, sc = kept.cpu().numpy(), sc.cpu().numpy()
    for f in range(n):
        ref = O.score_frame(q[f], k[f], float(cfg.alpha), bool(over.get("attn_causal")), bool(over.get("keep_low_freq")))
        assert kept[f].tolist() == O.select_tokens(ref[2], keep).tolist(), f
        assert np.abs(sc[2, f] - ref[2]).max() < H.FLAG_MARGIN / 2, f
        for i in range(3):
            H.close(sc[i, f], ref[i], f"score[{i}] frame {f}")
            if f in exact:                                 # (one rounding to float: half a unit in the last place)
                assert (np.abs(sc[i, f] - ref[i]) <= 2.0 ** -24 * np.abs(ref[i]) + 1e-12).all(), (i, f)


def test_noalloc_shapes_back_to_back():
    # other head sizes, tilings and matrix tables, each behind a call of another shape and length
    for i, (hq, hkv, d, tokens, n, bf16, over) in enumerate([
            (8, 8, 64, 130, 1, True, dict(attn_causal=1)),
            (28, 4, 128, 196, 16, True, dict(keep_low_freq=1)),
            (8, 8, 64, 130, 16, True, dict(attn_causal=1, keep_low_freq=1)),
            (2, 1, 64, 17, 5, True, {}),
            (32, 8, 128, 256, 16, True, {}),
            (14, 2, 64, 77, 3, False, {}),
            (14, 2, 64, 77, 16, True, dict(attn_causal=1))]):
        spec, q, k = _inputs(hq, hkv, d, tokens, n, bf16, 90 + i)
        _against_oracle(spec, q, k, n, max(1, tokens // 4), **over)


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("paired", [[3], [0, 5, 9, 15], [0, 1, 2, 5, 15], [0, 1, 2, 4, 5, 6, 8, 10, 12, 14]])
def test_noalloc_frames_in_double_precision(bf16, paired):
    # Every token of a paired frame stands there twice, and an odd number is kept: a pair lies across the boundary and the
    # frame is scored again in double precision.  Up to four such frames of 28 heads share a head between blocks, more do not.
    spec, q, k = _inputs(28, 4, 128, 196, 16, bf16, 97)
    for f in paired:
        q[f, 1::2], k[f, 1::2] = q[f, ::2], k[f, ::2]
    _against_oracle(spec, q, k, 16, 49, exact=paired)
