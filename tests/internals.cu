// The library once more, with what its tests need to reach from outside.
#include "../paper_2605_22269_b200/csrc/mukv.cu"

// limit of the waits between blocks of this context's calls; 0: every such wait is a single look
extern "C" void internals_wait_limit(mukv_ctx* ctx, unsigned long long ns) { ctx->wait_ns = ns; }

// mukv_score_frames_noalloc with the limit of its waits
extern "C" mukv_status internals_score_noalloc(const mukv_config* cfg, const void* q, const void* k, int32_t n, int32_t* kept,
                                               float* scores, mukv_stream stream, unsigned long long ns) {
  return score_frames_noalloc(cfg, q, k, n, kept, scores, stream, ns);
}

// tiles of the scan: {question tiles of a warp, question groups, row tiles of a block}
extern "C" void internals_scan_shape(long long rows, int nq, int n_sms, int* out) {
  const ScanShape s = scan_shape(rows, nq, n_sms);
  out[0] = s.T; out[1] = s.q_groups; out[2] = s.row_tiles;
}

extern "C" int internals_scan_by_rows(long long rows, int nq, int channels) { return scan_by_rows(rows, nq, channels); }

// where the last retrieval left the scores of every question with every frame, segment and patch-level block: byte offset in the
// workspace and question stride, doubles first, then their single-precision copies
extern "C" void internals_scores(const mukv_ctx* ctx, long long* out) {
  const long long T = ctx->cfg.max_frames, S = (long long)ctx->cfg.patch_split * ctx->cfg.patch_split;
  const long long v[12] = {(long long)ctx->wl.s_frm, T, (long long)ctx->wl.s_seg, ctx->sl.max_segs, (long long)ctx->wl.s_pat, T * S,
                           (long long)ctx->wl.f_frm, pad4(T), (long long)ctx->wl.f_seg, pad4(ctx->sl.max_segs), (long long)ctx->wl.f_pat,
                           pad4(T * S)};
  for (int i = 0; i < 12; ++i) out[i] = v[i];
}

// whether a bf16 chunk of this shape is scored on the tensor cores
extern "C" int internals_on_tensor_cores(const mukv_config* cfg) { return tc_shape(*cfg).ok; }
