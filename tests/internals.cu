// The library once more, with what its tests need to reach from outside.
#include "../paper_2605_22269_b200/csrc/mukv.cu"

// limit of the waits between blocks of this context's calls; 0: every such wait is a single look
extern "C" void internals_wait_limit(mukv_ctx* ctx, unsigned long long ns) { ctx->wait_ns = ns; }

// mukv_score_frames_noalloc with the limit of its waits
extern "C" mukv_status internals_score_noalloc(const mukv_config* cfg, const void* q, const void* k, int32_t n, int32_t* kept,
                                               float* scores, mukv_stream stream, unsigned long long ns) {
  return score_frames_noalloc(cfg, q, k, n, kept, scores, stream, ns);
}
