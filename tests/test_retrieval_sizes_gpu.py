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
    (133, 7, 9, 2, 64, B.RETR_PARALLEL),                   # one more: the tile of 64 questions
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
