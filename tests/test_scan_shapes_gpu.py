"""The scan at the edges of its tiles (eight rows, eight questions, blocks of one row tile or many, warps of one to eight question
tiles), against the oracle."""
import ctypes as C

import numpy as np
import pytest

from oracle import mukv_oracle as O
from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H
from tests import internals as I
from tests.test_parity_gpu import retrieval_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [9, 16, 17, 33, 64, 65, 97, 128])       # (up to eight questions have a kernel of their own)
@pytest.mark.parametrize("T,kv_heads,head_dim", [(7, 1, 64), (41, 2, 128)])
def test_scan_of_many_questions(nq, T, kv_heads, head_dim):
    spec = StreamSpec(seed=95, n_layers=1, n_q_heads=2 * kv_heads, n_kv_heads=kv_heads, head_dim=head_dim, tokens_per_frame=16,
                      bf16=True, n_outlier=1, n_frames=T, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=4, fseg=4, chunk=T, alpha=0.7)).compress()
    st = H.oracle_stream(spec, H.oracle_cfg(run.cfg), range(T), last_only=True, workers=1)
    qtok, offs, _ = spec.questions(nq, 1, 5)
    limit = np.random.default_rng(nq).integers(1, T + 1, nq)
    # (with fewer places than frames and with a place for each: every score is an output)
    retrieval_check(run, st, qtok, offs, 2, 5, 0.3, B.RETR_SEMI, t_limit=limit.astype(np.int64))
    retrieval_check(run, st, qtok, offs, 3, T, 0.0, B.RETR_PARALLEL)
    assert run.ctx.mukv_get_stats().device_status == 0


# frames of one key head of 64 channels and sixteen patch-level blocks each, questions, question tiles of a warp
MANY_ROWS = [(50, 9, 1), (50, 33, 2), (110, 80, 4), (431, 16, 2), (431, 24, 1), (431, 33, 4), (431, 97, 8), (770, 9, 2), (770, 64, 8),
             (770, 128, 8), (2000, 24, 4)]


def check_every_score(T, nq):
    """Compresses T frames, asks nq questions and compares what the scan left in the workspace."""
    spec = StreamSpec(seed=96, n_layers=1, n_q_heads=2, n_kv_heads=1, head_dim=64, tokens_per_frame=16, bf16=True, n_outlier=1,
                      n_frames=T, scene_sigma=1.0, frame_sigma=0.5, scene_min=2, scene_max=4)
    run = H.GpuRun(dict(spec=spec, keep=4, fseg=4, chunk=T, alpha=0.7), patch_split=4, grid_width=4, want_scores=False).compress()
    qtok, offs, _ = spec.questions(nq, 1, 5)
    i32, dev = H.torch.int32, run.device
    seg, frm, pat = (H.torch.full((nq, 3), -9, dtype=i32, device=dev) for _ in range(3))
    counts = H.torch.zeros((nq, 3), dtype=i32, device=dev)
    run.ctx.mukv_retrieve3(H.to_device(qtok, True, dev), offs, None, B.MukvRetrParams(3, 3, 3, 0.3, 0.3, 0.0, 0, B.RETR_SEMI), seg, frm,
                           pat, None, None, None, counts)
    where = (C.c_longlong * 12)()
    B._LIB.internals_scores(run.ctx.handle, where)
    ws = run.ctx.workspace
    held = run.ctx.region(9).cpu().numpy().reshape(-1) > 0
    for level, n in enumerate((T, (T + 3) // 4, 16 * T)):
        keys = run.ctx.region((4, 5, 8)[level]).cpu().numpy().reshape(-1, 64)[:n].astype(np.float64)
        for single in (0, 1):
            off, stride = where[6 * single + 2 * level], where[6 * single + 2 * level + 1]
            got = ws[off:off + (8, 4)[single] * stride * nq].view((H.torch.float64, H.torch.float32)[single]).view(nq, stride)[:, :n].cpu().numpy()
            for i in range(nq):
                ref = O.cosine(O.pool_question(qtok[offs[i]:offs[i + 1]], 1), keys)
                if not single:                             # sums of 64 products in double precision, (64 + a few) 2^-53 of the norms
                    assert np.abs(got[i] - ref).max() < 1e-13, (level, i)
                else:                                      # rounded once
                    there = held if level == 2 else np.ones(n, bool)
                    assert np.abs(got[i][there] - ref[there]).max() < 2.0 ** -24 + 1e-13 and (got[i][~there] == -np.inf).all(), (level, i)
    assert counts[:, 0].min() >= min(3, (T + 3) // 4) and counts[:, 1:].min() >= 3


@pytest.mark.parametrize("T,nq,tiles", MANY_ROWS)
def test_every_score_of_blocks_of_several_row_tiles(monkeypatch, T, nq, tiles):
    monkeypatch.setattr(B, "_LIB", I.load())
    rows = T + (T + 3) // 4 + 16 * T
    shape = I.scan_shape(rows, nq, H.torch.cuda.get_device_properties(0).multi_processor_count)
    assert shape[0] == tiles and shape[2] > 1 and rows % (8 * shape[2]) != 0          # (a last block that is not full)
    check_every_score(T, nq)


@pytest.mark.parametrize("T,nq,by_rows", [(3, 1, 1), (742, 1, 1), (743, 1, 0), (155, 2, 1), (156, 2, 0), (122, 3, 1), (123, 3, 0), (89, 4, 1),
                                          (90, 4, 0), (74, 5, 1), (75, 5, 0), (46, 8, 1), (47, 8, 0), (431, 2, 0), (431, 7, 0)])
def test_every_score_on_both_sides_of_the_line_between_the_scans(monkeypatch, T, nq, by_rows):
    monkeypatch.setattr(B, "_LIB", I.load())
    assert B._LIB.internals_scan_by_rows(T + (T + 3) // 4 + 16 * T, nq, 64) == by_rows
    check_every_score(T, nq)
