"""Rules of the host side that pick a kernel or its tiles."""
import ctypes as C

from paper_2605_22269_b200 import binding as B
from tests import internals as I


def test_every_shape_fits():
    # 227 KB of shared memory and 20 warps to a block; the columns of a block are columns of the pooled questions (128)
    seen = set()
    for rows in [1, 7, 8, 9, 63, 64, 107, 850, 1913, 4000, 7438, 8288, 11475, 21250, 44625, 400_000, 60_000_000]:
        for nq in range(1, 129):
            T, groups, tiles = I.scan_shape(rows, nq)
            assert T in (1, 2, 4, 8) and 1 <= groups <= 4 and tiles >= 1 and groups * tiles <= 20
            assert nq <= 8 * T * groups <= 128
            assert 2 * (32 * (8 * T * groups + 4) * 8 + 8 * tiles * 36 * 4) + 1024 <= 227 * 1024
            seen.add((T, tiles > 1))
    assert seen >= {(T, True) for T in (1, 2, 4, 8)} | {(1, False)}      # (blocks of one row tile, of many)


def test_blocks_do_not_multiply_the_fetched_questions():
    # a block fetches every question: 128 of them on 8,288 rows once went to 1,036 blocks of a single row tile
    for rows in range(7000, 15500, 500):
        for nq in (97, 100, 128):
            assert (rows + 7) // 8 // I.scan_shape(rows, nq)[2] <= 444, (rows, nq)


def test_every_bf16_frame_without_past_keys_is_scored_on_the_tensor_cores():
    # (scoring without a workspace has no other path for bf16)
    lib = I.load()
    n = 0
    for q_heads, kv_heads in [(1, 1), (2, 1), (7, 1), (28, 4), (32, 1), (32, 8), (31, 1), (24, 8), (12, 2)]:
        for d in (64, 128):
            for tokens in range(1, 257):
                cfg = B.make_config(n_layers=1, n_q_heads=q_heads, n_kv_heads=kv_heads, head_dim=d, tokens_per_frame=tokens,
                                    keep_per_frame=1, frames_per_segment=1, max_frames_per_chunk=1, max_frames=1)
                if lib.mukv_workspace_bytes(C.byref(cfg)):
                    n += 1
                    assert lib.internals_on_tensor_cores(C.byref(cfg)), (q_heads, kv_heads, d, tokens)
    assert n > 3000
