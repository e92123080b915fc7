"""A stream from its reset to a question, captured once and replayed as a graph."""
import pytest
import torch

from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls", [1, 2, 3])               # (the library alternates between two sets of sums from call to call)
@pytest.mark.parametrize("bf16,over", [(True, {}), (False, {}), (True, dict(keep_per_segment=40)), (True, dict(past_frames=1))])
def test_replays_of_a_captured_stream(calls, bf16, over):
    T = 4 * calls
    spec = StreamSpec(seed=81, n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64, tokens_per_frame=40, bf16=bf16, n_outlier=1,
                      n_frames=T, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=10, fseg=4, chunk=4, alpha=0.7), **over)
    dev, ctx = run.device, run.ctx
    chunks = []
    for c in range(calls):
        chunks.append(run.gs.alloc(4))
        run.gs.fill(4 * c, 4, *chunks[-1])
    kept = torch.full((T, 40 if "keep_per_segment" in over else 10), -1, dtype=torch.int32, device=dev)
    scores = torch.zeros((calls, 3, 4, 40), device=dev)
    qtok, offs, _ = spec.questions(3, 4, 9)
    qtok = H.to_device(qtok, bf16, dev)
    seg, frm = (torch.full((3, k), -9, dtype=torch.int32, device=dev) for k in (2, 3))
    counts = torch.zeros((3, 2), dtype=torch.int32, device=dev)

    def stream():
        ctx.mukv_reset()
        for c, (q, k, v) in enumerate(chunks):
            ctx.mukv_compress_chunk(q, k, v, 4, 4 * c, kept[4 * c:4 * c + 4], scores[c])
        ctx.mukv_retrieve(qtok, offs, None, 2, 3, 0, 0.3, B.RETR_SEMI, seg, frm, None, None, counts)

    outs = [kept, scores, seg, frm, counts] + [ctx.region(i) for i in (0, 2, 3, 4, 5)]
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        stream()
        side.synchronize()
        first = [x.clone() for x in outs]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            stream()
        for _ in range(3):
            for x in outs:
                x.zero_()
            graph.replay()
            side.synchronize()
            for x, y in zip(outs, first):
                assert torch.equal(x, y)
    assert ctx.mukv_get_stats().device_status == 0


@pytest.mark.parametrize("bf16", [True, False])
def test_replays_of_scoring_without_a_workspace(bf16):
    # (the first call on a device is made outside the capture); a call of another length between two replays leaves its own scratch
    spec = StreamSpec(seed=82, n_layers=1, n_q_heads=8, n_kv_heads=2, head_dim=64, tokens_per_frame=40, bf16=bf16, n_outlier=1,
                      n_frames=5, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=10, fseg=4, chunk=5, alpha=0.7))
    q, k, _ = run.gs.chunk(0, 5)
    kept = torch.full((5, 10), -1, dtype=torch.int32, device=run.device)
    scores = torch.zeros((3, 5, 40), device=run.device)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        def call(n):
            B.mukv_score_frames_noalloc(run.cfg, q, k[0], n, kept, scores)
        call(5)
        side.synchronize()
        first = [kept.clone(), scores.clone()]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            call(5)
        for _ in range(3):
            call(2)
            kept.fill_(-1)
            scores.zero_()
            graph.replay()
            side.synchronize()
            assert torch.equal(kept, first[0]) and torch.equal(scores, first[1])
