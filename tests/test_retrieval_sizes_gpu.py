"""Retrieval where the dispatch changes: numbers of questions around the scan for few, numbers of blocks around the sizes at
which all scores are ranked directly or through a histogram, numbers of candidates up to what the short ranking holds."""
import numpy as np
import pytest

from oracle import mukv_oracle as O
from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H

pytestmark = pytest.mark.gpu

SPEC = StreamSpec(seed=71, n_layers=1, n_q_heads=4, n_kv_heads=2, head_dim=64, tokens_per_frame=16, bf16=True, n_outlier=1,
                  n_frames=530, scene_sigma=1.0, frame_sigma=0.5, scene_min=3, scene_max=9)


@pytest.mark.parametrize("frames,fseg,n_q,k_seg,k_frm,mode", [
    (128, 2, 1, 3, 5, B.RETR_SEMI),                        # the most frames that are ranked directly, one row per warp in the scan
    (129, 1, 2, 3, 5, B.RETR_SEMI),                        # the histogram for frames and segments, two rows per warp, an odd row left
    (133, 7, 8, 2, 64, B.RETR_SEMI),                       # the most questions of the small scan; 128 candidates of 133
    (133, 7, 9, 2, 64, B.RETR_PARALLEL),                   # more than a few questions
    (530, 4, 3, 5, 200, B.RETR_SEMI),                      # 400 candidates and their second ranking
    (530, 4, 3, 140, 256, B.RETR_SEMI),                    # 512 candidates and some ties: more than the short list may hold
    (530, 4, 3, 9, 30, B.RETR_HIER),
])
def test_sizes_of_a_retrieval(frames, fseg, n_q, k_seg, k_frm, mode):
    run = H.GpuRun(dict(spec=SPEC, keep=4, fseg=fseg, chunk=40, alpha=0.7), n_frames=frames, want_scores=False).compress()
    st = H.oracle_stream(SPEC, H.oracle_cfg(run.cfg), range(frames), last_only=False, workers=1)
    qtok, offs, _ = SPEC.questions(n_q, 1, 6)
    ret = run.retrieve(qtok, offs, k_seg, k_frm, 0, 0.3, mode)
    dec, _ = run.gather(ret, k_frm)
    omode = {B.RETR_SEMI: O.MODE_SEMI, B.RETR_PARALLEL: O.MODE_PARALLEL, B.RETR_HIER: O.MODE_HIER}[mode]
    seg, frm, counts = (ret[n].cpu().numpy() for n in ("seg_idx", "frm_idx", "counts"))
    bits = H.to_numpy_bits(dec)
    for i in range(n_q):
        r = O.retrieve(st, qtok[offs[i]:offs[i + 1]], k_seg, k_frm, 0, 0.3, omode)
        n_seg, n_frm = len(r["seg_idx"]), len(r["frm_idx"])
        assert counts[i].tolist() == [n_seg, n_frm]
        assert seg[i, :n_seg].tolist() == np.asarray(r["seg_idx"]).tolist() and (seg[i, n_seg:] == -1).all()
        assert frm[i, :n_frm].tolist() == np.asarray(r["frm_idx"]).tolist() and (frm[i, n_frm:] == -1).all()
        ref, _ = O.gather(st, r["frm_idx"])
        assert bits[i][:, :, :n_frm * 4].tobytes() == ref.tobytes()


@pytest.mark.parametrize("frames,n_q,k_seg,k_frm,mode", [
    (60, 3, 2, 3, B.RETR_SEMI),                            # few blocks, all ranked directly
    (60, 3, 12, 40, B.RETR_SEMI),                          # the segment without a score is among the top N; 60 candidates of 60
    (300, 9, 70, 4, B.RETR_SEMI),                          # the histogram
    (300, 2, 3, 8, B.RETR_PARALLEL),
    (300, 2, 75, 256, B.RETR_HIER),                        # every segment selected
])
def test_blocks_and_questions_that_are_not_finite(frames, n_q, k_seg, k_frm, mode):
    # An Inf among a frame's keys is accepted input (the frame keeps its lowest ids).  Its frame, segment and one patch-level
    # block have no cosine: they rank last and stay out of the global query.  The last question holds a NaN: no block has a
    # score for it, the lowest ids are taken.  Ids only: nothing is gathered.
    wl = dict(spec=SPEC, keep=4, fseg=4, chunk=60, alpha=0.7)
    run = H.GpuRun(wl, n_frames=frames, want_scores=False, patch_split=2, grid_width=4)
    st = O.Store(H.oracle_cfg(run.cfg))
    for t0 in range(0, frames, 60):
        q, k, v = SPEC.chunk(t0, 60)
        if t0 == 0:
            k[0, 9, 2, 1, 5] = 0x7F80
        run.ctx.mukv_compress_chunk(*(H.to_device(x, True, run.device) for x in (q, k, v)), 60, t0)
        O.compress_chunk(st, q, k, v)
    qtok, offs, _ = SPEC.questions(n_q, 1, 6)
    qtok[offs[n_q - 1], 0, 0] = 0x7FC0
    dev, i32 = run.device, H.torch.int32
    k_pat = 2 * k_frm if k_frm < 128 else 256
    seg, frm, pat = (H.torch.full((n_q, k), -9, dtype=i32, device=dev) for k in (k_seg, k_frm, k_pat))
    sc = [H.torch.full(x.shape, float("nan"), device=dev) for x in (seg, frm, pat)]
    counts = H.torch.zeros((n_q, 3), dtype=i32, device=dev)
    omode = {B.RETR_SEMI: O.MODE_SEMI, B.RETR_PARALLEL: O.MODE_PARALLEL, B.RETR_HIER: O.MODE_HIER}[mode]
    for lam_seg in (0.0, 0.3):
        run.ctx.mukv_retrieve3(H.to_device(qtok, True, dev), offs, None,
                               B.MukvRetrParams(k_pat, k_frm, k_seg, 0.3, 0.3, lam_seg, 0, mode), seg, frm, pat, *sc, counts)
        for i in range(n_q):
            r = O.retrieve3(st, qtok[offs[i]:offs[i + 1]], (k_pat, k_frm, k_seg), (0.3, 0.3, lam_seg), 0, omode)
            for got, score, name, n in zip((seg, frm, pat), sc, ("seg", "frm", "patch"), counts[i].tolist()):
                ref = np.asarray(r[name + "_idx"]).tolist()
                assert n == len(ref) and got[i, :n].tolist() == ref and (got[i, n:] == -1).all(), (lam_seg, i, name)
                H.close(score[i, :n].cpu().numpy(), r[name + "_score"], name)
