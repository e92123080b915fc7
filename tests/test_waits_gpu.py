"""Waits between blocks of one kernel: what is left when one runs out."""
import numpy as np
import pytest

from oracle import mukv_oracle as O
from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H
from tests import internals as I

pytestmark = pytest.mark.gpu


@pytest.fixture
def lib(monkeypatch):
    monkeypatch.setattr(B, "_LIB", I.load())
    return B._LIB


@pytest.mark.parametrize("bf16", [True, False])
def test_a_wait_that_ran_out_does_not_reach_the_next_calls(lib, bf16):
    # Every frame is flagged.  The waits of the first and of the fourth call are given no time, those of the others the usual one:
    # these store what the oracle stores.
    spec = StreamSpec(seed=84, n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, tokens_per_frame=40, bf16=bf16, n_outlier=1,
                      n_frames=18, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=10, fseg=3, chunk=3, alpha=0.7), options={B.OPT_FLAG_MARGIN: 4.0})
    dev = run.device
    kept = H.torch.full((18, 10), -7, dtype=H.torch.int32, device=dev)
    scores = H.torch.zeros((6, 3, 3, 40), device=dev)
    for call in range(6):
        lib.internals_wait_limit(run.ctx.handle, 0 if call in (0, 3) else 1_500_000_000)
        run.ctx.mukv_compress_chunk(*run.gs.chunk(3 * call, 3), 3, 3 * call, kept[3 * call:3 * call + 3], scores[call])
        assert run.ctx.mukv_get_stats().device_status == 6
    st = H.oracle_stream(spec, H.oracle_cfg(run.cfg), range(18), last_only=False, workers=1)
    run.kept = kept.cpu().numpy()
    run.scores = scores.permute(1, 0, 2, 3).reshape(3, 18, 40).cpu().numpy()
    good = [t for t in range(18) if t // 3 not in (0, 3)]
    sub = O.Store(H.oracle_cfg(run.cfg))
    for name in ("kept", "page_k", "page_v", "sum_k", "sum_v", "scores"):
        getattr(sub, name).extend(getattr(st, name)[t] for t in good)
    H.check_frames_against_oracle(run, sub, good, full_layers=True)
    seg = run.ctx.region(3).cpu().numpy()
    for u in (1, 2, 4, 5):                                 # (segment u holds the frames of call u)
        sk, sv = st.segment_entry(u)
        H.close(seg[u][:, 0], sk, f"segment entry K {u}")
        H.close(seg[u][:, 1], sv, f"segment entry V {u}")
    assert run.ctx.mukv_get_stats().refined_frames >= 12
    # a reset forgets it
    run.ctx.mukv_reset()
    run.compress()
    H.check_frames_against_oracle(run, st, range(18), full_layers=True)
    stats = run.ctx.mukv_get_stats()
    assert stats.device_status == 0 and stats.refined_frames == 18


@pytest.mark.parametrize("bf16", [True, False])
def test_two_contexts_on_two_streams_with_every_frame_flagged(bf16):
    # Calls whose copies alone fill the device.  Each context's flagged frames find places held by the other's.
    spec = StreamSpec(seed=85, n_layers=14, n_q_heads=28, n_kv_heads=4, head_dim=128, tokens_per_frame=196, bf16=bf16, n_outlier=2,
                      n_frames=64, scene_sigma=1.0, frame_sigma=0.5, scene_min=10, scene_max=20)
    wl = dict(spec=spec, keep=49, fseg=16, chunk=16, alpha=0.7)
    runs = [H.GpuRun(wl, options={B.OPT_FLAG_MARGIN: 4.0}) for _ in range(3)]
    dev = runs[0].device
    kept = H.torch.full((3, 64, 49), -7, dtype=H.torch.int32, device=dev)
    chunks = []
    for t0 in range(0, 64, 16):
        chunks.append(runs[0].gs.alloc(16))
        runs[0].gs.fill(t0, 16, *chunks[-1])
    for c, x in enumerate(chunks):                         # alone
        runs[2].ctx.mukv_compress_chunk(*x, 16, 16 * c, kept[2, 16 * c:16 * c + 16])
    H.torch.cuda.synchronize()
    streams = [H.torch.cuda.Stream() for _ in range(2)]
    for rep in range(3):
        for i, s in enumerate(streams):
            runs[i].ctx.mukv_reset(stream=s)
        for c, x in enumerate(chunks):
            for i, s in enumerate(streams):
                runs[i].ctx.mukv_compress_chunk(*x, 16, 16 * c, kept[i, 16 * c:16 * c + 16], stream=s)
        H.torch.cuda.synchronize()
        for i in range(2):
            stats = runs[i].ctx.mukv_get_stats()
            assert stats.device_status == 0 and stats.refined_frames == 64
            assert H.torch.equal(kept[i], kept[2])
            for region in (0, 1, 2, 3, 4, 5):
                assert H.torch.equal(runs[i].ctx.region(region), runs[2].ctx.region(region)), region
        kept[:2] = -7
    st = H.oracle_stream(spec, H.oracle_cfg(runs[2].cfg), range(2), last_only=True, workers=1)
    assert kept[2, :2].tolist() == [x.tolist() for x in st.kept]


def test_scoring_without_a_workspace_takes_back_what_it_could_not_decide(lib):
    # frames 3 and 9 hold every token twice and keep an odd number: only double precision decides them
    spec = StreamSpec(seed=86, n_layers=1, n_q_heads=28, n_kv_heads=4, head_dim=128, tokens_per_frame=196, bf16=True, n_outlier=1,
                      n_frames=16, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    q, k, _ = spec.chunk(0, 16)
    for f in (3, 9):
        q[f, 1::2], k[0, f, 1::2] = q[f, ::2], k[0, f, ::2]
    cfg = H.spec_config(spec, dict(keep=49, fseg=1, chunk=16, alpha=0.7))
    ref = [O.score_frame(q[f], k[0, f], float(cfg.alpha)) for f in range(16)]
    ids = [O.select_tokens(r[2], 49).tolist() for r in ref]
    dq, dk = H.to_device(q, True), H.to_device(k[0], True)
    kept = H.torch.full((16, 49), -7, dtype=H.torch.int32, device="cuda:0")
    scores = H.torch.zeros((3, 16, 196), device="cuda:0")
    for ns in (0, 1_500_000_000, 0, 1_500_000_000):
        kept.fill_(-7)
        assert lib.internals_score_noalloc(B.C.byref(cfg), dq.data_ptr(), dk.data_ptr(), 16, kept.data_ptr(), scores.data_ptr(),
                                           B._stream(None), ns) == 0
        got, sc = kept.tolist(), scores.cpu().numpy()
        back = [f for f in range(16) if got[f] == [-1] * 49 and np.isnan(sc[:, f]).all()]
        assert bool(back) == (ns == 0)
        for f in range(16):
            if f not in back:
                assert got[f] == ids[f], f
                for i in range(3):
                    H.close(sc[i, f], ref[f][i], f"score[{i}] frame {f}")
