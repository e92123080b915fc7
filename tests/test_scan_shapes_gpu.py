"""The scan at the edges of its tiles (eight rows, eight questions, warps of one to eight question tiles), against the oracle."""
import numpy as np
import pytest

from paper_2605_22269_b200 import binding as B
from paper_2605_22269_b200.synth.cpu import StreamSpec
from tests import harness as H
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
