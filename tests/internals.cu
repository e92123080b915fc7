// The library once more, with what its tests need to reach from outside.
#include "../paper_2605_22269_b200/csrc/mukv.cu"

// limit of the waits between blocks of this context's calls; 0: every such wait is a single look
extern "C" void internals_wait_limit(mukv_ctx* ctx, unsigned long long ns) { ctx->wait_ns = ns; }
