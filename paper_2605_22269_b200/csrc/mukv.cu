// Host side of the MuKV library: context, store layout, argument checks, kernel launches.
// Built for sm_100a only.  No device memory is allocated here: the store and the workspace
// belong to the caller.
#include "../../include/mukv.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "compact.cuh"
#include "retrieve.cuh"
#include "score.cuh"
#include "score64.cuh"
#include "score_ps.cuh"
#include "segsel.cuh"

using namespace mukv;

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct StoreLayout {
  size_t pages, kept, frame_entry, seg_entry, frame_key, seg_key, frame_ts, page_table, frame_ksum, patch_key, patch_cnt,
      kept_count, total;
  size_t pages_bytes, kept_stride;
  size_t page_bytes;
  long long max_segs;
};

struct WorkLayout {
  size_t q_terms, k_terms; // fp32 chunks: queries and keys of the scoring layers as three bf16 terms
  size_t colsum_f, ifft_f, colsum_d, ifft_d, frame_counter, head_counter, flagged, n_flagged, tail_ctr, sel_flag,
      seg_flag, stat_refined, dev_status, att_acc;
  size_t q64, qnorm, s_frm, s_seg, s_pat, f_frm, f_seg, f_pat, wtab, total;
  size_t zero_begin, zero_end;          // region that must start as zeros
};

// Tiling of the tensor-core scoring kernel.
struct TcShape {
  bool ok;                 // bf16 chunk scored on the tensor cores (every supported bf16 shape fits)
  int tpt, tiles, npad, n_mt, ps_stages;
  int own_rows, past_pad;  // key-tile rows of the frame's own keys; rows reserved per cached past frame (0: none)
  size_t smem_ps;
  bool split;              // fp32 chunk scored on the tensor cores in three bf16 terms (ok is false: it has a path of its own)
  int split_frames;        // most frames of a call for that (what the terms of a call may take is limited)
  int n_a, n_b, b_slot;    // its operand rings
};

thread_local std::string g_create_error;

}  // namespace

struct mukv_ctx {
  mukv_config cfg;
  StoreLayout sl;
  WorkLayout wl;
  unsigned char* store;
  unsigned char* ws;
  long long frames;
  long long launches;
  int parity = 0;                        // which of the two flagged counters and sets of column sums this chunk uses
  long long att_dirty[2] = {0, 0};       // values of a set that the last call on it has written
  unsigned epoch = 0;                    // compress calls so far (tags the per-frame selection flags)
  int C, G, esize, nc, Ls;
  int key_rows;                          // key rows of the multiply-add scoring kernel: P + past_frames * kappa
  float flag_margin, flat_ratio;
  bool force_fma = false;                // MUKV_OPT_SCORE_PATH 1: multiply-add scoring for every dtype
  bool failed = false;                   // a compress call broke off half way: only reset / stats / destroy
  TcShape tcs;                           // tcs.ok: the chunk is scored on the tensor cores
  int n_sms;
  unsigned long long wait_ns = kWaitNs;  // limit of the waits inside compact_kernel and tail_kernel
  int places = 1;                        // blocks of compact_kernel that an empty device holds at once
  CUtensorMap wmap;                      // DFT matrix terms [3*D][D] bf16
  CUtensorMap pmap;                      // the page region as [frame][plane][kept row][key head][D] (past_frames > 0)
  // Segment entries a compress call left to whoever comes next (see flush_segments): the frames whose
  // segments still have to be pooled, and the stream that call ran on
  mutable bool seg_pending = false;
  mutable long long seg_first = 0;
  mutable int seg_n = 0;
  mutable cudaStream_t seg_stream = nullptr;
  std::string err;
  // optional per-kernel timing (host objects only)
  bool prof_on = false;
  std::vector<cudaEvent_t> prof_ev;      // pairs: start, stop
  std::vector<int> prof_kind;            // kind of each used pair
};

namespace {

mukv_status fail(mukv_ctx* ctx, mukv_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (ctx) ctx->err = buf; else g_create_error = buf;
  return st;
}

// A launch failed after part of a compress call was enqueued: the chunk is half stored and the
// device-side counters no longer match the host's, so the context stops until mukv_reset.
mukv_status broke_off(mukv_ctx* ctx, const char* what, cudaError_t e) {
  ctx->failed = true;
  return fail(ctx, MUKV_E_CUDA, "%s: %s (the chunk is half stored: call mukv_reset)", what, cudaGetErrorString(e));
}

// Brackets one kernel launch with a pair of events when profiling is on.
struct ProfScope {
  mukv_ctx* c;
  cudaStream_t st;
  cudaEvent_t stop = nullptr;
  ProfScope(mukv_ctx* ctx, int kind, cudaStream_t s) : c(ctx), st(s) {
    if (!c->prof_on) return;
    const size_t used = c->prof_kind.size();
    while (c->prof_ev.size() < 2 * (used + 1)) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return;
      c->prof_ev.push_back(e);
    }
    c->prof_kind.push_back(kind);
    cudaEventRecord(c->prof_ev[2 * used], st);
    stop = c->prof_ev[2 * used + 1];
  }
  ~ProfScope() {
    if (stop) cudaEventRecord(stop, st);
  }
};

bool is_pow2(long long x) { return x > 0 && (x & (x - 1)) == 0; }
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

// Returns nullptr if the configuration is supported, else the reason.
const char* check_config(const mukv_config* c) {
  if (!c) return "null config";
  if (c->dtype != MUKV_BF16 && c->dtype != MUKV_FP32) return "dtype must be MUKV_BF16 or MUKV_FP32";
  if (c->n_layers < 1 || c->n_kv_heads < 1 || c->n_q_heads < 1) return "layer/head counts must be positive";
  if (c->n_q_heads % c->n_kv_heads != 0) return "n_q_heads must be a multiple of n_kv_heads";
  if (c->head_dim != 64 && c->head_dim != 128) return "head_dim must be 64 or 128";
  if (c->tokens_per_frame < 1 || c->tokens_per_frame > MUKV_MAX_TOKENS) return "tokens_per_frame out of range";
  if (c->keep_per_frame < 1 || c->keep_per_frame > c->tokens_per_frame) return "keep_per_frame out of range";
  if (c->frames_per_segment < 1) return "frames_per_segment must be positive";
  if (c->max_frames_per_chunk < 1 || c->max_frames_per_chunk > 4096) return "max_frames_per_chunk out of range";
  if (c->max_frames < 1) return "max_frames must be positive";
  if (!(c->alpha >= 0.f && c->alpha <= 1.f)) return "alpha must lie in [0, 1]";
  if (!(c->tie_eps >= 0.f)) return "tie_eps must be >= 0";
  if (c->patch_split < 0 || c->patch_split > MUKV_MAX_PATCH_SPLIT) return "patch_split out of range";
  if (c->patch_split > 0 && (c->grid_width < 1 || c->tokens_per_frame % c->grid_width != 0))
    return "grid_width must divide tokens_per_frame when patch_split > 0";
  if (c->reserved != 0) return "reserved fields must be 0";
  if (c->past_frames < 0) return "past_frames must be >= 0";
  if (c->past_frames > 0) {
    if (c->keep_per_segment > 0) return "past keys are not combined with segment-level selection";
    if ((long long)c->past_frames * c->keep_per_frame + c->tokens_per_frame > MUKV_MAX_TOKENS)
      return "past_frames * keep_per_frame + tokens_per_frame must be <= 256";
  }
  if (c->keep_per_segment < 0) return "keep_per_segment must be >= 0";
  if (c->keep_per_segment > 0) {
    if (c->patch_split != 0) return "segment-level selection has no patch level";
    if ((long long)c->frames_per_segment * c->tokens_per_frame > kSegSelMaxTokens)
      return "segment-level selection: frames_per_segment * tokens_per_frame must be <= 4096";
    if (c->keep_per_segment > c->frames_per_segment * c->tokens_per_frame) return "keep_per_segment out of range";
  }
  if (c->n_score_layers < 0 || c->score_layer_offset < 0 ||
      (c->n_score_layers > 1 ? c->n_score_layers : 1) + c->score_layer_offset > c->n_layers)
    return "scoring layers must lie inside the model: n_score_layers + score_layer_offset <= n_layers";
  if ((long long)(c->n_score_layers > 1 ? c->n_score_layers : 1) * c->n_q_heads > 4096) return "too many scoring layers";
  const long long esize = c->dtype == MUKV_BF16 ? 2 : 4;
  const long long row_vec = (long long)c->n_kv_heads * c->head_dim * esize / 16;
  if (!is_pow2(row_vec) || row_vec > 256) return "Hkv*D*sizeof(element)/16 must be a power of two <= 256";
  // the scoring kernel keeps one key head of a frame in shared memory
  const int key_rows = c->tokens_per_frame + c->past_frames * c->keep_per_frame;
  const size_t smem = c->dtype == MUKV_BF16 ? score_smem_bytes<__nv_bfloat16>(key_rows, c->head_dim)
                                            : score_smem_bytes<float>(key_rows, c->head_dim);
  if (smem > 227 * 1024) return "tokens_per_frame * head_dim too large for shared memory";
  return nullptr;
}

StoreLayout store_layout(const mukv_config& c) {
  StoreLayout s;
  const size_t esize = c.dtype == MUKV_BF16 ? 2 : 4;
  const size_t C = (size_t)c.n_kv_heads * c.head_dim;
  const size_t T = (size_t)c.max_frames;
  s.max_segs = (c.max_frames + c.frames_per_segment - 1) / c.frames_per_segment;
  s.page_bytes = (size_t)c.n_layers * 2 * c.keep_per_frame * C * esize;
  size_t off = 0;
  // segment-level selection: a segment's pages share kappa_v token slots; kept ids are padded to P per frame
  const bool seg_scope = c.keep_per_segment > 0;
  s.pages_bytes = seg_scope ? (size_t)s.max_segs * c.keep_per_segment * c.n_layers * 2 * C * esize : T * s.page_bytes;
  s.kept_stride = seg_scope ? (size_t)c.tokens_per_frame : (size_t)c.keep_per_frame;
  s.pages = off;        off = align_up(off + s.pages_bytes);
  s.kept = off;         off = align_up(off + T * s.kept_stride * sizeof(int));
  s.frame_entry = off;  off = align_up(off + T * c.n_layers * 2 * C * sizeof(float));
  s.seg_entry = off;    off = align_up(off + (size_t)s.max_segs * c.n_layers * 2 * C * sizeof(float));
  s.frame_key = off;    off = align_up(off + T * C * sizeof(float));
  s.seg_key = off;      off = align_up(off + (size_t)s.max_segs * C * sizeof(float));
  s.frame_ts = off;     off = align_up(off + T * sizeof(long long));
  s.page_table = off;   off = align_up(off + T * sizeof(long long));
  s.frame_ksum = off;   off = align_up(off + T * C * sizeof(double));
  const size_t S = (size_t)c.patch_split * c.patch_split;
  s.patch_key = off;    off = align_up(off + T * S * C * sizeof(float));
  s.patch_cnt = off;    off = align_up(off + T * S * sizeof(int));
  s.kept_count = off;   off = align_up(off + (seg_scope ? T * sizeof(int) : 0));
  s.total = off;
  return s;
}

TcShape tc_shape(const mukv_config& c) {
  TcShape t;
  memset(&t, 0, sizeof t);
  const int G = c.n_q_heads / c.n_kv_heads;
  if (G > 128) return t;
  t.tpt = 128 / G;
  t.tiles = (c.tokens_per_frame + t.tpt - 1) / t.tpt;
  t.npad = (c.tokens_per_frame + 15) / 16 * 16;
  t.own_rows = t.npad;
  if (c.past_frames > 0) {
    // the cached keys of a past frame start on a multiple of eight rows of the key tile (one swizzle
    // atom), behind the frame's own keys
    t.own_rows = (c.tokens_per_frame + 7) / 8 * 8;
    t.past_pad = (c.keep_per_frame + 7) / 8 * 8;
    t.npad = (t.own_rows + c.past_frames * t.past_pad + 15) / 16 * 16;
    if (c.keep_per_segment > 0) return t;               // pages of different lengths are not one regular tensor
  }
  t.n_mt = (c.tokens_per_frame + 127) / 128;
  if (c.dtype != MUKV_BF16) {
    // fp32: frame-level selection without past keys.  (Segment-level selection ranks fp32 chunks in double precision,
    // and past keys are stored as fp32 rows.)  The terms of a call take 6 bytes per value of the scoring layers' queries
    // and keys, 4.8 MB per frame of 28 x 196 x 128 queries.  256 MB is what a workspace is given for them (a choice, not a
    // measurement: 55 such frames); longer calls keep the multiply-add kernel, about five times slower.
    if (c.past_frames > 0 || c.keep_per_segment > 0) return t;
    const long long ls = c.n_score_layers > 1 ? c.n_score_layers : 1;
    const long long per_frame = 6LL * ls * c.tokens_per_frame * (c.n_q_heads + c.n_kv_heads) * c.head_dim;
    const long long most = (256LL << 20) / per_frame;
    t.split_frames = (int)(most < c.max_frames_per_chunk ? most : c.max_frames_per_chunk);
    t.split = t.split_frames > 0 && t.npad <= kPsSplit * kPsAccCols &&
              score_ps_split_rings(t.npad, c.head_dim, 227 * 1024, &t.n_a, &t.n_b, &t.b_slot, &t.smem_ps);
    return t;
  }
  t.ps_stages = score_ps_stages(t.npad, c.head_dim, 227 * 1024);
  t.smem_ps = score_ps_smem_bytes(t.npad, c.head_dim, t.ps_stages < 2 ? 2 : t.ps_stages);
  t.ok = t.ps_stages >= 2 && t.npad <= kPsSplit * kPsAccCols;
  return t;
}

constexpr int kRefineSplit = 4;     // blocks per query head where whole segments are scored in double precision
// Rows of P doubles that the column sums of the double-precision pass have room for: one for every (frame, head, part) of a
// call of segment-level selection, and for a head of a single flagged frame to be split over the device (see score64_split).
size_t refine_rows(const mukv_config& c) {
  const size_t rows = (size_t)c.max_frames_per_chunk * (c.n_score_layers > 1 ? c.n_score_layers : 1) * c.n_q_heads * kRefineSplit;
  return rows > 512 ? rows : 512;
}
// Single precision decides a frame only when its lowest kept and highest dropped fused score are
// further apart than tie_eps + kFlagMargin; a signal whose range is below kFlatRatio of its
// magnitude (the min-max division then amplifies rounding noise) also sends the frame to the
// double-precision pass.
constexpr float kFlagMargin = 3e-6f;
constexpr float kFlatRatio = 1e-3f;

// rows of single-precision scores start on 16 bytes
inline long long pad4(long long n) { return (n + 3) / 4 * 4; }

// the DFT matrix in three bf16 terms, see DftTerms
constexpr size_t dft_bytes(int D) { return (size_t)3 * D * D * sizeof(uint16_t); }

WorkLayout work_layout(const mukv_config& c) {
  WorkLayout w;
  const size_t F = c.max_frames_per_chunk, P = c.tokens_per_frame;
  const size_t C = (size_t)c.n_kv_heads * c.head_dim;
  const size_t max_segs = (c.max_frames + c.frames_per_segment - 1) / c.frames_per_segment;
  size_t off = 0;
  const TcShape ts = tc_shape(c);
  const size_t Ls = c.n_score_layers > 1 ? c.n_score_layers : 1;
  w.colsum_f = off;       off = align_up(off + F * Ls * (size_t)c.n_q_heads * P * sizeof(float));
  w.ifft_f = off;         off = align_up(off + F * Ls * c.n_kv_heads * P * sizeof(float));
  w.colsum_d = off;       off = align_up(off + refine_rows(c) * P * sizeof(double));
  w.ifft_d = off;         off = align_up(off + F * Ls * c.n_kv_heads * P * sizeof(double));
  w.zero_begin = off;
  w.frame_counter = off;  off = align_up(off + F * sizeof(int));
  w.head_counter = off;   off = align_up(off + F * Ls * c.n_q_heads * sizeof(int));
  w.flagged = off;        off = align_up(off + F * sizeof(int));
  w.n_flagged = off;      off = align_up(off + 2 * sizeof(int));   // alternate between chunks
  w.tail_ctr = off;       off = align_up(off + 2 * kTailWords * sizeof(int));   // alternate, too
  w.sel_flag = off;       off = align_up(off + F * sizeof(unsigned));
  w.seg_flag = off;       off = align_up(off + F * sizeof(int));
  w.stat_refined = off;   off = align_up(off + sizeof(long long));
  w.dev_status = off;     off = align_up(off + sizeof(int));
  w.att_acc = off;        off = align_up(off + (ts.ok || ts.split ? 2 * F * P * sizeof(unsigned long long) : 0));   // alternate, too
  w.zero_end = off;
  w.q64 = off;            off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * C * sizeof(double));
  w.qnorm = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * c.n_kv_heads * sizeof(double));
  w.s_frm = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * c.max_frames * sizeof(double));
  w.s_seg = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * max_segs * sizeof(double));
  w.s_pat = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * c.max_frames * c.patch_split * c.patch_split *
                                               sizeof(double));
  w.f_frm = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * pad4(c.max_frames) * sizeof(float));
  w.f_seg = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * pad4(max_segs) * sizeof(float));
  w.f_pat = off;          off = align_up(off + (size_t)MUKV_MAX_QUESTIONS * pad4(c.max_frames * c.patch_split * c.patch_split) *
                                               sizeof(float));
  w.wtab = off;           off = align_up(off + (ts.ok || ts.split ? dft_bytes(c.head_dim) : 0));
  const size_t tf = ts.split ? (size_t)ts.split_frames * Ls * P * 6 : 0;
  w.q_terms = off;        off = align_up(off + tf * c.n_q_heads * c.head_dim);
  w.k_terms = off;        off = align_up(off + tf * C);
  w.total = off;
  return w;
}

int pick_nc(int P) { return P <= 64 ? 2 : P <= 128 ? 4 : P <= 224 ? 7 : 8; }

// Launches a kernel; with `dependent` it may be scheduled while the previous kernel of the stream
// still runs (programmatic dependent launch: the kernel itself waits in pdl_wait()).  cluster > 1: that many
// neighbouring blocks form a cluster.
template <typename... KArgs, typename... Args>
cudaError_t launch_c(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                     bool dependent, unsigned cluster, Args... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  if (dependent) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster;
    attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                     bool dependent, Args... args) {
  return launch_c(kernel, grid, block, smem, st, dependent, 1u, args...);
}

// Zeros `bytes` (a multiple of eight, below 16 GB) on the stream.  Where no kernel can be launched (a stream of another device than
// the current one) it is a memset, which can.
cudaError_t zero_async(void* p, size_t bytes, cudaStream_t st, bool dependent) {
  const int n = (int)(bytes / 8), blocks = (n + kCompactThreads - 1) / kCompactThreads;
  if (n <= 0) return cudaSuccess;
  cudaError_t e = launch_k(zero_kernel, dim3(blocks < 148 ? blocks : 148), kCompactThreads, 0, st, dependent,
                           static_cast<unsigned long long*>(p), n);
  if (e == cudaSuccess) return e;
  cudaGetLastError();
  return cudaMemsetAsync(p, 0, bytes, st);
}

template <typename T>
cudaError_t launch_score(const ScoreParams& sp, int nc, dim3 grid, size_t smem, cudaStream_t st, bool dependent) {
  switch (nc) {
    case 2: return launch_k(score_kernel<T, 2>, grid, kScoreThreads, smem, st, dependent, sp);
    case 4: return launch_k(score_kernel<T, 4>, grid, kScoreThreads, smem, st, dependent, sp);
    case 7: return launch_k(score_kernel<T, 7>, grid, kScoreThreads, smem, st, dependent, sp);
    default: return launch_k(score_kernel<T, 8>, grid, kScoreThreads, smem, st, dependent, sp);
  }
}

// Raises a kernel's dynamic shared-memory limit to everything the device allows beside the
// kernel's static shared memory.
cudaError_t raise_smem_limit(const void* fn, int optin) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, fn);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

template <typename T>
cudaError_t raise_score_limits(int optin) {
  cudaError_t e = raise_smem_limit((const void*)score_kernel<T, 2>, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_kernel<T, 4>, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_kernel<T, 7>, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_kernel<T, 8>, optin);
  return e;
}

constexpr int kMaxDevices = 64;
std::mutex g_dev_mutex;
bool g_limits_raised[kMaxDevices];
int g_compact_per_sm[kMaxDevices];

// Once per device (that device current): the dynamic shared-memory limit of every kernel that
// needs more than the default goes to the device's maximum.  The limit belongs to the kernel,
// not to a context, so it is never set to one context's need: a second context of another
// shape, or the allocation-free entry point, would otherwise find it too low.
// places: blocks of compact_kernel, whichever form of it, that the device holds at once when nothing else runs.
cudaError_t raise_kernel_limits(int* n_sms, int* places) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(n_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  if (places) *places = g_compact_per_sm[dev] * *n_sms;
  if (g_limits_raised[dev]) return cudaSuccess;
  int optin = 0;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = raise_score_limits<__nv_bfloat16>(optin);
  if (e == cudaSuccess) e = raise_score_limits<float>(optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)rank_kernel, optin);
  for (const void* fn : {(const void*)scan_kernel<1>, (const void*)scan_kernel<2>, (const void*)scan_kernel<4>, (const void*)scan_kernel<8>})
    if (e == cudaSuccess) e = raise_smem_limit(fn, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)segsel_kernel, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_ps_kernel<false, false>, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_ps_kernel<true, false>, optin);
  if (e == cudaSuccess) e = raise_smem_limit((const void*)score_ps_kernel<false, true>, optin);
  if (e == cudaSuccess) {
    typedef __nv_bfloat16 B16;
    int least = 1 << 30;
    for (const void* fn : {(const void*)compact_kernel<B16, false, false>, (const void*)compact_kernel<B16, false, true>,
                           (const void*)compact_kernel<B16, true, false>, (const void*)compact_kernel<B16, true, true>}) {
      int per_sm = 0;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCompactThreads, 0);
      least = std::min(least, per_sm);
    }
    if (e == cudaSuccess && least < 1) e = cudaErrorInvalidConfiguration;
    g_compact_per_sm[dev] = least;
    if (places) *places = least * *n_sms;
  }
  if (e == cudaSuccess) g_limits_raised[dev] = true;
  return e;
}

// ---------------------------------------------------------------- TMA descriptors
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// bf16 tensor [rows][mid][D] (D contiguous) seen as a rank-3 map; the box is box_rows x box_mid x 64
// channels, written to shared memory with the 128-byte swizzle.  Out-of-range rows read as zero.
bool encode_map3(CUtensorMap* m, const void* base, int D, int mid, long long rows, int box_mid, int box_rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)mid, (cuuint64_t)rows};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)mid * D * 2};
  const cuuint32_t box[3] = {64u, (cuuint32_t)box_mid, (cuuint32_t)box_rows};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The pages of a store with frame-level selection, bf16: [frames][2L planes][kappa rows][Hkv][D] as a
// rank-5 map; the box is the kappa rows of one key head in one plane of one page, 64 channels wide.
bool encode_map_pages(CUtensorMap* m, const void* pages, int D, int Hkv, int kappa, int planes, long long frames,
                      long long page_bytes) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t row = (cuuint64_t)Hkv * D * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)D, (cuuint64_t)Hkv, (cuuint64_t)kappa, (cuuint64_t)planes, (cuuint64_t)frames};
  const cuuint64_t strides[4] = {(cuuint64_t)D * 2, row, row * kappa, (cuuint64_t)page_bytes};
  const cuuint32_t box[5] = {64u, 1u, (cuuint32_t)kappa, 1u, 1u};
  const cuuint32_t estr[5] = {1u, 1u, 1u, 1u, 1u};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(pages), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_map2(CUtensorMap* m, const void* base, int cols, long long rows, int box_rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1u, 1u};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

uint16_t bf16_rne(float x) {
  uint32_t b;
  memcpy(&b, &x, 4);
  b += 0x7FFFu + ((b >> 16) & 1u);
  return (uint16_t)(b >> 16);
}
float bf16_val(uint16_t h) {
  const uint32_t b = (uint32_t)h << 16;
  float x;
  memcpy(&x, &b, 4);
  return x;
}

// The D-point DFT as a matrix, rows = output column n, columns = input channel d (the layout of
// a K-major B operand): n <= D/2 holds cos(2 pi n d / D), n > D/2 holds -sin(2 pi (n - D/2) d / D).
// Each entry is split into three bf16 terms, hi + mid + lo, stored as [3][D][D].
template <int D>
struct DftTerms {
  uint16_t w[3 * D * D];
  DftTerms() {
    const double pi = 3.14159265358979323846;
    for (int n = 0; n < D; ++n)
      for (int d = 0; d < D; ++d) {
        const int b = n <= D / 2 ? n : n - D / 2;
        const int m = (int)(((long long)b * d) % D);
        const double ang = 2.0 * pi * (double)m / (double)D;
        const double x = n <= D / 2 ? std::cos(ang) : -std::sin(ang);
        const uint16_t hi = bf16_rne((float)x);
        const double r1 = x - (double)bf16_val(hi);
        const uint16_t mid = bf16_rne((float)r1);
        const double r2 = r1 - (double)bf16_val(mid);
        w[(0 * D + n) * D + d] = hi;
        w[(1 * D + n) * D + d] = mid;
        w[(2 * D + n) * D + d] = bf16_rne((float)r2);
      }
  }
};

// Worked out once per process and head size (for every context: 80 us of mukv_create at D = 64, 300 us at D = 128).
const uint16_t* dft_terms(int D) {
  if (D == 64) {
    static const DftTerms<64> t;
    return t.w;
  }
  static const DftTerms<128> t;
  return t.w;
}

// The pooling of segment entries (Eq. 5 at segment level) for frames first .. first + n - 1.
SegmentArgs segment_args_of(const mukv_ctx* ctx, long long first, int n) {
  const mukv_config& c = ctx->cfg;
  SegmentArgs a;
  memset(&a, 0, sizeof a);
  a.L = c.n_layers; a.kappa = c.keep_per_frame; a.C = ctx->C; a.fseg = c.frames_per_segment;
  a.n_frames = n; a.first_frame = first;
  a.frame_entry = reinterpret_cast<const float*>(ctx->store + ctx->sl.frame_entry);
  a.frame_ksum = reinterpret_cast<const double*>(ctx->store + ctx->sl.frame_ksum);
  a.seg_entry = reinterpret_cast<float*>(ctx->store + ctx->sl.seg_entry);
  a.seg_key = reinterpret_cast<float*>(ctx->store + ctx->sl.seg_key);
  if (c.keep_per_segment > 0) a.kept_count = reinterpret_cast<const int*>(ctx->store + ctx->sl.kept_count);
  return a;
}

// A compress call does not pool the segment entries of its chunk itself: the next compress call does it with blocks that do
// not wait for that call's
// scoring kernel (more rows in its compaction kernel, one plane per block; with segment-level selection, extra blocks of its
// first segsel_kernel launch).  Whoever else needs the entries first
// (retrieval, a gather with summary tokens, a view of the store, an export) pools them with one launch here.
cudaError_t flush_segments(const mukv_ctx* ctx, cudaStream_t st) {
  if (!ctx->seg_pending) return cudaSuccess;
  CompactParams cp;
  memset(&cp, 0, sizeof cp);
  const SegmentArgs a = segment_args_of(ctx, ctx->seg_first, ctx->seg_n);
  cp.L = a.L; cp.kappa = a.kappa; cp.C = a.C; cp.fseg = a.fseg; cp.n_frames = a.n_frames; cp.first_frame = a.first_frame;
  cp.frame_entry = const_cast<float*>(a.frame_entry); cp.frame_ksum = const_cast<double*>(a.frame_ksum);
  cp.seg_entry = a.seg_entry; cp.seg_key = a.seg_key; cp.kept_count = a.kept_count;
  const cudaError_t e = launch_k(segment_kernel, dim3(2 * a.L), kCompactThreads, 0, st, !ctx->prof_on, cp);
  if (e == cudaSuccess) ctx->seg_pending = false;
  return e;
}

// What a launch of the persistent scoring kernel needs beside the scoring parameters.
struct PsLaunch {
  const TcShape* t;
  int n_sms;
  const CUtensorMap* wmap;
  const CUtensorMap* pmap;       // stored pages (past keys), or null
  unsigned long long* att_acc;   // [frames][P], zero
  int* status;
  int kappa;
  bool dependent;
  __nv_bfloat16 *q_terms, *k_terms;   // SPLIT: room for the terms of an fp32 chunk
};

// Scores a chunk on the tensor cores (Eq. 1-3; Eq. 4 and the selection follow in compact_kernel).
cudaError_t launch_score_ps(PsLaunch& l, const ScoreParams& sp, cudaStream_t st, const char** why) {
  const TcShape& t = *l.t;
  const int P = sp.P, D = sp.D, n = sp.n_frames;
  CUtensorMap qmap, kmap, kmap128;
  const long long rows = (long long)sp.Ls * n * P;
  const void *q = sp.q, *k = sp.k_last;
  bool maps = true;
  if (t.split) {
    SplitParams s;
    s.src[0] = reinterpret_cast<const float*>(sp.q); s.src[1] = reinterpret_cast<const float*>(sp.k_last);
    s.dst[0] = l.q_terms; s.dst[1] = l.k_terms;
    s.n[0] = rows * sp.Hq * D; s.n[1] = rows * sp.Hkv * D;
    const long long blocks = ((s.n[0] + s.n[1]) / 8 + 255) / 256, most = 8LL * l.n_sms;   // eight blocks per SM are resident
    *why = "split_terms kernel";
    const cudaError_t e = launch_k(split_terms_kernel, dim3((unsigned)(blocks < most ? blocks : most)), 256u, 0, st, l.dependent, s);
    if (e != cudaSuccess) return e;
    q = l.q_terms;
    k = l.k_terms;
    maps = encode_map3(&kmap128, k, D, sp.Hkv, 3 * rows, 1, 128);
  }
  const long long map_rows = t.split ? 3 * rows : rows;
  if (!maps || !encode_map3(&qmap, q, D, sp.Hq, map_rows, sp.G, t.tpt) ||
      !encode_map3(&kmap, k, D, sp.Hkv, map_rows, 1, t.own_rows)) {
    *why = "cuTensorMapEncodeTiled failed";
    return cudaErrorInvalidValue;
  }
  ScorePsParams pp;
  memset(&pp, 0, sizeof pp);
  pp.sp = sp;
  pp.att_acc = l.att_acc;
  pp.tiles = t.tiles; pp.tpt = t.tpt; pp.npad = t.npad; pp.n_mt = t.n_mt; pp.n_stages = t.ps_stages;
  pp.own_rows = t.own_rows; pp.n_past = sp.n_past_frames; pp.past_pad = t.past_pad; pp.kappa = l.kappa;
  pp.past_plane0 = 2 * sp.first_score_layer; pp.past_first = sp.past_first;
  pp.ipu = t.n_mt + t.tiles;
  pp.ipf = sp.Ls * sp.Hkv * pp.ipu;
  pp.n_items = n * pp.ipf;
  pp.exp2_scale = (float)(1.4426950408889634 / std::sqrt((double)D));
  pp.status = l.status;
  int blocks = l.n_sms < kPsMaxBlocks ? l.n_sms : kPsMaxBlocks;
  if (blocks > pp.n_items) blocks = pp.n_items;
  *why = "score_ps kernel";
  const bool past = sp.n_past_frames > 0;
  if (t.split) {
    pp.n_a = t.n_a; pp.n_b = t.n_b; pp.b_slot = t.b_slot; pp.term_rows = (int)rows;
    return launch_k(score_ps_kernel<false, true>, dim3(blocks), kPsThreads, t.smem_ps, st, l.dependent, pp, qmap, kmap,
                    *l.wmap, kmap128);
  }
  return launch_k(past ? score_ps_kernel<true, false> : score_ps_kernel<false, false>, dim3(blocks), kPsThreads, t.smem_ps,
                  st, l.dependent, pp, qmap, kmap, *l.wmap, past ? *l.pmap : kmap);
}

unsigned long long* att_acc_of(const mukv_ctx* ctx, int parity) {
  return reinterpret_cast<unsigned long long*>(ctx->ws + ctx->wl.att_acc) +
         (size_t)parity * ctx->cfg.max_frames_per_chunk * ctx->cfg.tokens_per_frame;
}

PsLaunch ps_launch_of(mukv_ctx* ctx) {
  PsLaunch l;
  memset(&l, 0, sizeof l);
  l.t = &ctx->tcs; l.n_sms = ctx->n_sms; l.wmap = &ctx->wmap; l.pmap = &ctx->pmap;
  l.att_acc = att_acc_of(ctx, ctx->parity);
  l.status = reinterpret_cast<int*>(ctx->ws + ctx->wl.dev_status);
  l.kappa = ctx->cfg.keep_per_frame;
  l.dependent = !ctx->prof_on;
  l.q_terms = reinterpret_cast<__nv_bfloat16*>(ctx->ws + ctx->wl.q_terms);
  l.k_terms = reinterpret_cast<__nv_bfloat16*>(ctx->ws + ctx->wl.k_terms);
  return l;
}

template <typename T>
mukv_status compress_impl(mukv_ctx* ctx, const void* d_q, const float* d_ext, const void* d_k, const void* d_v, int n,
                          long long t0, int* d_kept_out, float* d_scores_out, cudaStream_t st) {
  const mukv_config& c = ctx->cfg;
  const int P = c.tokens_per_frame, L = c.n_layers, C = ctx->C;
  const bool seg_scope = c.keep_per_segment > 0;
  if (seg_scope) {
    if (d_ext) return fail(ctx, MUKV_E_UNSUPPORTED, "caller-supplied scores are ranked per frame only");
    if (t0 % c.frames_per_segment != 0)
      return fail(ctx, MUKV_E_STATE, "segment-level selection: first_frame must be a multiple of frames_per_segment");
  }
  ScoreParams sp;
  memset(&sp, 0, sizeof sp);
  sp.P = P; sp.Hq = c.n_q_heads; sp.Hkv = c.n_kv_heads; sp.D = c.head_dim; sp.G = ctx->G;
  sp.kappa = c.keep_per_frame; sp.n_frames = n; sp.causal = c.attn_causal; sp.keep_low = c.keep_low_freq;
  sp.alpha = c.alpha; sp.tie_eps = c.tie_eps; sp.flag_margin = ctx->flag_margin; sp.flat_ratio = ctx->flat_ratio;
  sp.first_frame = t0;
  sp.q = d_q;
  sp.Ls = ctx->Ls;
  sp.q_layer_stride = (long long)n * P * c.n_q_heads * c.head_dim;
  sp.k_layer_stride = (long long)n * P * C;
  sp.k_last = reinterpret_cast<const T*>(d_k) + (long long)(L - c.score_layer_offset - ctx->Ls) * n * P * C;
  sp.colsum_part = ctx->ws + ctx->wl.colsum_f;
  sp.ifft_part = ctx->ws + ctx->wl.ifft_f;
  sp.frame_counter = reinterpret_cast<int*>(ctx->ws + ctx->wl.frame_counter);
  sp.head_counter = reinterpret_cast<int*>(ctx->ws + ctx->wl.head_counter);
  sp.flagged = reinterpret_cast<int*>(ctx->ws + ctx->wl.flagged);
  sp.n_flagged = reinterpret_cast<int*>(ctx->ws + ctx->wl.n_flagged) + ctx->parity;
  sp.kept_store = reinterpret_cast<int*>(ctx->store + ctx->sl.kept);
  sp.kept_out = d_kept_out;
  sp.scores_out = d_scores_out;
  sp.frame_ts = reinterpret_cast<long long*>(ctx->store + ctx->sl.frame_ts);
  sp.page_table = reinterpret_cast<long long*>(ctx->store + ctx->sl.page_table);
  sp.pages_off = (long long)ctx->sl.pages;
  sp.page_bytes = (long long)ctx->sl.page_bytes;
  sp.status = reinterpret_cast<int*>(ctx->ws + ctx->wl.dev_status);
  sp.store = ctx->store;
  sp.first_score_layer = L - c.score_layer_offset - ctx->Ls;
  sp.past_first = t0 - c.past_frames > 0 ? t0 - c.past_frames : 0;
  sp.n_past_frames = c.past_frames > 0 ? (int)(t0 - sp.past_first) : 0;
  sp.refine = 0;
  sp.row_split = 1;
  const dim3 grid(ctx->Ls * c.n_q_heads, n);
  cudaError_t e = cudaSuccess;
  const char* what = "score kernel";
  bool on_tc = false;                                    // scored by the persistent kernel, selected by compact_kernel
  int n_launch = 0;
  if (seg_scope) {
    // One block per segment ranks all its tokens.  A bf16 chunk is first scored on the tensor cores and
    // ranked from those single-precision sums; segments that are too close to call are scored and
    // ranked again in double precision (both launches of that pass return at once for the others).
    // Any other chunk goes through the double-precision pass as a whole.
    const bool tc_first = ctx->tcs.ok && !ctx->force_fma;
    const int n_seg = (n + c.frames_per_segment - 1) / c.frames_per_segment;
    const int seg_tokens = (n < c.frames_per_segment ? n : c.frames_per_segment) * P;
    const bool dep = !ctx->prof_on;
    SegSelParams gp;
    memset(&gp, 0, sizeof gp);
    gp.fseg = c.frames_per_segment; gp.kappa_v = c.keep_per_segment;
    gp.token_bytes = (long long)L * 2 * C * ctx->esize;
    gp.kept_count = reinterpret_cast<int*>(ctx->store + ctx->sl.kept_count);
    gp.seg_flag = reinterpret_cast<int*>(ctx->ws + ctx->wl.seg_flag);
    gp.n_seg = n_seg;
    // Segment entries the previous call left behind: pooled by extra blocks of the first segsel_kernel launch
    // (that kernel uses one SM per segment); with per-kernel timing on, by a launch of their own
    if (ctx->seg_pending && ctx->prof_on) {
      ProfScope ps(ctx, 3, st);
      e = flush_segments(ctx, st);
      if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "segment kernel: %s", cudaGetErrorString(e));
      ++n_launch;
    }
    int extra = 0;
    if (ctx->seg_pending) {
      gp.prev = segment_args_of(ctx, ctx->seg_first, ctx->seg_n);
      extra = 2 * L;
    }
    gp.stat_refined = reinterpret_cast<unsigned long long*>(ctx->ws + ctx->wl.stat_refined);
    if (tc_first) {
      PsLaunch pl = ps_launch_of(ctx);
      {
        ProfScope ps(ctx, 0, st);
        e = launch_score_ps(pl, sp, st, &what);
        ctx->att_dirty[ctx->parity] = (long long)n * P;
      }
      if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
      n_launch += 2;
      gp.sp = sp;
      gp.att_acc = pl.att_acc;
      gp.src32 = 1;
      {
        ProfScope ps(ctx, 1, st);
        e = launch_k(segsel_kernel, dim3(n_seg + extra), kSegSelThreads, segsel_smem_bytes(seg_tokens), st, dep, gp);
      }
      if (e != cudaSuccess) return broke_off(ctx, "segment selection kernel", e);
      ctx->seg_pending = false;
      extra = 0;
      memset(&gp.prev, 0, sizeof gp.prev);
    }
    ScoreParams sd = sp;
    sd.no_select = 1;
    sd.row_split = kRefineSplit;
    sd.colsum_part = ctx->ws + ctx->wl.colsum_d;
    sd.ifft_part = ctx->ws + ctx->wl.ifft_d;
    if (tc_first) {
      sd.seg_gate = gp.seg_flag;
      sd.gate_fseg = c.frames_per_segment;
    }
    {
      ProfScope ps(ctx, tc_first ? 1 : 0, st);
      const long long units = (long long)ctx->Ls * c.n_q_heads * kRefineSplit * (tc_first ? 1 : n), most = 3LL * ctx->n_sms;
      const dim3 grid_d((unsigned)(units < most ? units : most));
      e = launch_k(score64_kernel<T>, grid_d, kScoreThreads, 0, st, tc_first && dep, sd);
    }
    if (e != cudaSuccess) {
      if (tc_first) return broke_off(ctx, "score kernel", e);
      return fail(ctx, MUKV_E_CUDA, "score kernel: %s", cudaGetErrorString(e));
    }
    gp.sp = sd;
    gp.src32 = 0;
    gp.only_flagged = tc_first ? 1 : 0;
    {
      ProfScope ps(ctx, 1, st);
      e = launch_k(segsel_kernel, dim3(n_seg + extra), kSegSelThreads, segsel_smem_bytes(seg_tokens), st, tc_first && dep,
                   gp);
    }
    if (e != cudaSuccess) return broke_off(ctx, "segment selection kernel", e);
    ctx->seg_pending = false;
    n_launch += 2;
  } else if (!d_ext) {
    ProfScope ps(ctx, 0, st);
    if ((ctx->tcs.ok || (ctx->tcs.split && n <= ctx->tcs.split_frames)) && !ctx->force_fma) {
      n_launch += ctx->tcs.split ? 1 : 0;
      PsLaunch pl = ps_launch_of(ctx);
      e = launch_score_ps(pl, sp, st, &what);
      ctx->att_dirty[ctx->parity] = (long long)n * P;
      on_tc = true;
    } else
      e = launch_score<T>(sp, ctx->nc, grid, score_smem_bytes<T>(ctx->key_rows, c.head_dim), st, !ctx->prof_on);
    ++n_launch;
  }
  if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "%s: %s", what, cudaGetErrorString(e));

  // Compaction of every frame that single precision decides; after the persistent scoring kernel
  // its blocks also do the selection (Eq. 4, top-kappa) from that kernel's partial sums.
  CompactParams cp;
  memset(&cp, 0, sizeof cp);
  cp.L = L; cp.kappa = c.keep_per_frame; cp.C = C; cp.P = P; cp.n_frames = n; cp.first_frame = t0;
  cp.k = d_k; cp.v = d_v;
  cp.store = ctx->store;
  cp.frame_entry = reinterpret_cast<float*>(ctx->store + ctx->sl.frame_entry);
  cp.frame_key = reinterpret_cast<float*>(ctx->store + ctx->sl.frame_key);
  cp.frame_ksum = reinterpret_cast<double*>(ctx->store + ctx->sl.frame_ksum);
  cp.stat_refined = reinterpret_cast<long long*>(ctx->ws + ctx->wl.stat_refined);
  cp.tail_ctr = reinterpret_cast<int*>(ctx->ws + ctx->wl.tail_ctr) + ctx->parity * kTailWords;
  cp.tail_next = reinterpret_cast<int*>(ctx->ws + ctx->wl.tail_ctr) + (ctx->parity ^ 1) * kTailWords;
  cp.wait_ns = ctx->wait_ns;
  cp.sel_flag = reinterpret_cast<unsigned*>(ctx->ws + ctx->wl.sel_flag);
  cp.epoch = (++ctx->epoch) & 0x7fffffffu;
  cp.n_flagged_next = reinterpret_cast<int*>(ctx->ws + ctx->wl.n_flagged) + (ctx->parity ^ 1);
  cp.fseg = c.frames_per_segment;
  cp.seg_entry = reinterpret_cast<float*>(ctx->store + ctx->sl.seg_entry);
  cp.seg_key = reinterpret_cast<float*>(ctx->store + ctx->sl.seg_key);
  cp.patch_split = c.patch_split; cp.grid_width = c.grid_width;
  cp.patch_key = reinterpret_cast<float*>(ctx->store + ctx->sl.patch_key);
  cp.patch_cnt = reinterpret_cast<int*>(ctx->store + ctx->sl.patch_cnt);
  cp.sel_mode = seg_scope ? 3 : d_ext ? 2 : on_tc ? 1 : 0;
  cp.kept_count = seg_scope ? reinterpret_cast<const int*>(ctx->store + ctx->sl.kept_count) : nullptr;
  cp.ext_scores = d_ext;
  cp.att_acc = att_acc_of(ctx, ctx->parity);
  cp.att_clear = att_acc_of(ctx, ctx->parity ^ 1);       // (nobody reads the previous call's sums any more)
  cp.n_clear = ctx->att_dirty[ctx->parity ^ 1];
  ctx->att_dirty[ctx->parity ^ 1] = 0;
  cp.sp = sp;
  // segment entries the previous call left behind: more rows of blocks (with per-kernel timing on,
  // a launch of their own, so that each kernel is timed doing its own work only)
  if (ctx->seg_pending && ctx->prof_on) {
    ProfScope ps(ctx, 3, st);
    e = flush_segments(ctx, st);
    if (e != cudaSuccess) return broke_off(ctx, "segment kernel", e);
    ++n_launch;
  }
  if (ctx->seg_pending) {
    cp.prev = segment_args_of(ctx, ctx->seg_first, ctx->seg_n);
    cp.prev_rows = (2 * L + n - 1) / n;
  }
  // A plane of a frame is three round trips of rows for one block.  While the planes of a short call leave most of the
  // device idle (three blocks per SM are resident), two or four blocks share one by columns, which leaves one trip; a part
  // of a row stays at least 256 bytes.  (Sixteen one-frame calls of 28 layers and a question: 352 us with one block per plane,
  // 300 with parts; calls of 7 frames and 24 layers, which get two parts: no difference.)
  cp.parts = 1;
  while (cp.parts < 4 && 4LL * n * L * cp.parts <= 3LL * ctx->n_sms && C * ctx->esize / (2 * cp.parts) >= 256) cp.parts *= 2;
  // Flagged frames (frame-level selection by Eq. 1-4 only): blocks that redo them, as many as an empty device has places for
  // beside the copies, or has in all (any number of them does the work, see redo_flagged; a block per SM would find its
  // places three on some SMs and none on others), and no more than a frame has units.
  // They are blocks of the compaction kernel, which spares the calls that flag nothing a launch.  fp32 calls keep the launch:
  // a hundredth of their time, behind a kernel of twice the bytes.
  int redo = 0;
  if (!seg_scope && !d_ext) {
    const int units = ctx->Ls * c.n_q_heads * ((P + 7) / 8), planes = 4 * L + 1;
    const int others = n * (L * 2 * cp.parts + (c.patch_split > 0 ? 1 : 0) + cp.prev_rows), room = ctx->places - others;
    redo = std::min(std::max(units, planes), sizeof(T) == 4 ? ctx->n_sms : room <= 0 ? ctx->places : std::max(room, ctx->n_sms));
    cp.colsum_d = reinterpret_cast<double*>(ctx->ws + ctx->wl.colsum_d);
    cp.ifft_d = reinterpret_cast<double*>(ctx->ws + ctx->wl.ifft_d);
    cp.sp.scratch_rows = (int)std::min<size_t>(refine_rows(c), 0x7fffffff);
    cp.sp.n_selected = cp.tail_ctr + 1;
    if (sizeof(T) == 2) cp.redo_blocks = redo;
  }
  {
    ProfScope ps(ctx, 2, st);
    const int rows = L * 2 * cp.parts + (c.patch_split > 0 ? 1 : 0) + cp.prev_rows + (cp.redo_blocks + n - 1) / n;
    const bool sel = cp.sel_mode == 1;
    cp.later_blocks = (long long)n * rows > ctx->places;
    e = launch_k(cp.parts > 1 ? (sel ? compact_kernel<T, true, true> : compact_kernel<T, true, false>)
                              : (sel ? compact_kernel<T, false, true> : compact_kernel<T, false, false>),
                 dim3(n, rows), kCompactThreads, 0, st, !ctx->prof_on, cp);
  }
  if (e != cudaSuccess) return broke_off(ctx, "compact kernel", e);
  ctx->seg_pending = false;

  // (The segment entries need every frame of the chunk.  They are left to the next call, see flush_segments.)
  if constexpr (sizeof(T) == 4) {
    if (redo > 0) {
      ProfScope ps(ctx, 1, st);
      e = launch_k(tail_kernel<T>, dim3(redo), kCompactThreads, 0, st, !ctx->prof_on, cp);
      ++n_launch;
    }
  }
  if (e != cudaSuccess) return broke_off(ctx, "tail kernel", e);
  ctx->seg_pending = true;
  ctx->seg_first = t0;
  ctx->seg_n = n;
  ctx->seg_stream = st;

  ctx->launches += n_launch + 1;                          // + compact_kernel
  ctx->parity ^= 1;
  ctx->frames = t0 + n;
  return MUKV_OK;
}

mukv_status create_impl(const mukv_config* cfg, void* d_store, size_t store_bytes, void* d_workspace,
                        size_t workspace_bytes, long long frames0, mukv_ctx** out);

mukv_status retrieve_impl(mukv_ctx* ctx, const void* d_qtok, const int32_t* h_q_offsets, const int64_t* h_t_limit,
                          int32_t nq, const mukv_retr_params& prm, int32_t* d_seg_idx, int32_t* d_frm_idx,
                          int32_t* d_pat_idx, float* d_seg_score, float* d_frm_score, float* d_pat_score,
                          int32_t* d_counts, int counts_stride, mukv_stream stream) {
  try {
    const int k_seg = prm.k_seg, k_frm = prm.k_frm, k_pat = prm.k_patch, top_n = prm.top_n, mode = prm.mode;
    if (ctx->failed) return fail(ctx, MUKV_E_STATE, "an earlier call broke off half way: call mukv_reset");
    if (!d_qtok || !h_q_offsets || !d_seg_idx || !d_frm_idx || !d_counts)
      return fail(ctx, MUKV_E_INVALID, "null argument");
    if (!aligned16(d_qtok) || !aligned4(d_seg_idx) || !aligned4(d_frm_idx) || !aligned4(d_seg_score) ||
        !aligned4(d_frm_score) || !aligned4(d_counts))
      return fail(ctx, MUKV_E_ALIGN, "d_qtok must be 16-byte aligned, the outputs 4-byte aligned");
    if (nq < 1) return fail(ctx, MUKV_E_INVALID, "nq must be >= 1");
    if (nq > MUKV_MAX_QUESTIONS) return fail(ctx, MUKV_E_CAPACITY, "nq %d exceeds %d", nq, MUKV_MAX_QUESTIONS);
    if (k_seg < 1 || k_frm < 1 || k_pat < 0 || top_n < 0)
      return fail(ctx, MUKV_E_INVALID, "k_seg, k_frm must be >= 1, k_patch and top_n >= 0");
    if (k_seg > MUKV_MAX_TOPK || k_frm > MUKV_MAX_TOPK || k_pat > MUKV_MAX_TOPK || top_n > MUKV_MAX_TOPK)
      return fail(ctx, MUKV_E_CAPACITY, "k_seg / k_frm / k_patch / top_n exceed %d", MUKV_MAX_TOPK);
    if (k_pat > 0 && ctx->cfg.patch_split == 0) return fail(ctx, MUKV_E_STATE, "the store has no patch level");
    if (k_pat > 0 && !d_pat_idx) return fail(ctx, MUKV_E_INVALID, "d_patch_idx is null");
    if (!aligned4(d_pat_idx) || !aligned4(d_pat_score)) return fail(ctx, MUKV_E_ALIGN, "outputs must be 4-byte aligned");
    if (mode != MUKV_RETR_PARALLEL && mode != MUKV_RETR_HIER && mode != MUKV_RETR_SEMI)
      return fail(ctx, MUKV_E_INVALID, "unknown retrieval mode %d", mode);
    for (float lam : {prm.lambda_patch, prm.lambda_frm, prm.lambda_seg})
      if (!(lam >= 0.f && lam <= 1.f)) return fail(ctx, MUKV_E_INVALID, "every lambda must lie in [0, 1]");
    if (ctx->frames < 1) return fail(ctx, MUKV_E_STATE, "the store is empty");
    if (ctx->seg_pending) {                                // the last chunk's segment entries are read below
      const cudaError_t ef = flush_segments(ctx, static_cast<cudaStream_t>(stream));
      if (ef != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "segment kernel: %s", cudaGetErrorString(ef));
      ctx->launches += 1;
    }
    QMeta meta;
    if (h_q_offsets[0] != 0) return fail(ctx, MUKV_E_INVALID, "q_offsets[0] must be 0");
    for (int i = 0; i < nq; ++i) {
      if (h_q_offsets[i + 1] <= h_q_offsets[i])
        return fail(ctx, MUKV_E_INVALID, "question %d has no tokens (offsets must ascend)", i);
      if (h_t_limit && h_t_limit[i] < 0) return fail(ctx, MUKV_E_INVALID, "t_limit[%d] is negative", i);
    }
    for (int i = 0; i <= nq; ++i) meta.off[i] = h_q_offsets[i];
    for (int i = 0; i < nq; ++i) meta.t_limit[i] = h_t_limit ? (long long)h_t_limit[i] : ctx->frames;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const mukv_config& c = ctx->cfg;
    const int C = ctx->C;
    double* q64 = reinterpret_cast<double*>(ctx->ws + ctx->wl.q64);
    double* qnorm = reinterpret_cast<double*>(ctx->ws + ctx->wl.qnorm);
    double* s_frm = reinterpret_cast<double*>(ctx->ws + ctx->wl.s_frm);
    double* s_seg = reinterpret_cast<double*>(ctx->ws + ctx->wl.s_seg);
    const float* frame_key = reinterpret_cast<const float*>(ctx->store + ctx->sl.frame_key);
    const float* seg_key = reinterpret_cast<const float*>(ctx->store + ctx->sl.seg_key);
    const long long n_frm = ctx->frames;
    const long long n_seg = (n_frm + c.frames_per_segment - 1) / c.frames_per_segment;
    const int S = c.patch_split * c.patch_split;
    const long long n_pat = k_pat > 0 ? n_frm * S : 0;
    const long long rows = n_frm + n_seg + n_pat;
    const bool few = scan_by_rows(rows, nq, C);
    cudaError_t e = cudaSuccess;
    {
      ProfScope ps(ctx, 4, st);
      const dim3 grid(nq, c.n_kv_heads);
      const int cs = few ? 1 : MUKV_MAX_QUESTIONS, qs = few ? C : 1;
      if (c.dtype == MUKV_BF16)
        e = launch_k(qpool_kernel<__nv_bfloat16>, grid, kPoolThreads, 0, st, !ctx->prof_on,
                     reinterpret_cast<const __nv_bfloat16*>(d_qtok), meta, c.n_q_heads, c.n_kv_heads, c.head_dim, q64, cs, qs, qnorm, (int)few);
      else
        e = launch_k(qpool_kernel<float>, grid, kPoolThreads, 0, st, !ctx->prof_on, reinterpret_cast<const float*>(d_qtok), meta,
                     c.n_q_heads, c.n_kv_heads, c.head_dim, q64, cs, qs, qnorm, (int)few);
    }
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "qpool kernel: %s", cudaGetErrorString(e));
    double* s_pat = reinterpret_cast<double*>(ctx->ws + ctx->wl.s_pat);
    const float* patch_key = reinterpret_cast<const float*>(ctx->store + ctx->sl.patch_key);
    {
      ProfScope ps(ctx, 5, st);
      ScanParams sc;
      memset(&sc, 0, sizeof sc);
      sc.frame_key = frame_key; sc.seg_key = seg_key; sc.patch_key = patch_key;
      sc.n_frm = n_frm; sc.n_seg = n_seg; sc.n_pat = n_pat;
      sc.C = C; sc.nq = nq; sc.Hkv = c.n_kv_heads; sc.q64t = q64; sc.qn2 = qnorm;
      sc.s_frm = s_frm; sc.s_seg = s_seg; sc.s_pat = s_pat;
      sc.frm_stride = c.max_frames; sc.seg_stride = ctx->sl.max_segs; sc.pat_stride = (long long)c.max_frames * S;
      sc.f_frm = reinterpret_cast<float*>(ctx->ws + ctx->wl.f_frm); sc.f_frm_stride = pad4(c.max_frames);
      sc.f_seg = reinterpret_cast<float*>(ctx->ws + ctx->wl.f_seg); sc.f_seg_stride = pad4(ctx->sl.max_segs);
      sc.f_pat = reinterpret_cast<float*>(ctx->ws + ctx->wl.f_pat); sc.f_pat_stride = pad4((long long)c.max_frames * S);
      sc.patch_cnt = reinterpret_cast<const int*>(ctx->store + ctx->sl.patch_cnt);
      if (few) {
        const int per_block = nq > 1 ? 16 : 8;                 // a row or two per warp, up to eight blocks per SM
        const long long want = (rows + per_block - 1) / per_block, most = 8LL * ctx->n_sms;
        const dim3 grid((unsigned)(want < most ? want : most));
        e = launch_k(nq == 1 ? scan_few_kernel<1> : nq <= 4 ? scan_few_kernel<4> : scan_few_kernel<kScanFew>, grid, 256, 0, st,
                     !ctx->prof_on, sc);
      } else {
        const ScanShape sh = scan_shape(rows, nq, ctx->n_sms);
        sc.q_groups = sh.q_groups; sc.row_tiles = sh.row_tiles;
        const dim3 grid((unsigned)(((rows + 7) / 8 + sh.row_tiles - 1) / sh.row_tiles));
        e = launch_k(sh.T == 1 ? scan_kernel<1> : sh.T == 2 ? scan_kernel<2> : sh.T == 4 ? scan_kernel<4> : scan_kernel<8>, grid,
                     32u * sh.q_groups * sh.row_tiles, sh.smem, st, !ctx->prof_on, sc);
      }
    }
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "scan kernel: %s", cudaGetErrorString(e));
    RankParams rp;
    memset(&rp, 0, sizeof rp);
    rp.nq = nq; rp.C = C; rp.fseg = c.frames_per_segment;
    rp.k_seg = k_seg; rp.k_frm = k_frm; rp.k_pat = k_pat; rp.top_n = top_n; rp.mode = mode; rp.S = S;
    rp.lam_seg = (double)prm.lambda_seg; rp.lam_frm = (double)prm.lambda_frm; rp.lam_pat = (double)prm.lambda_patch;
    rp.delta = (double)c.tie_eps;
    rp.n_frm = n_frm; rp.n_seg = n_seg;
    rp.s_frm = s_frm; rp.s_seg = s_seg; rp.s_pat = s_pat;
    rp.frm_stride = c.max_frames; rp.seg_stride = ctx->sl.max_segs; rp.pat_stride = (long long)c.max_frames * S;
    rp.frame_key = frame_key; rp.seg_key = seg_key; rp.patch_key = patch_key;
    rp.patch_cnt = reinterpret_cast<const int*>(ctx->store + ctx->sl.patch_cnt);
    rp.seg_idx = d_seg_idx; rp.frm_idx = d_frm_idx; rp.pat_idx = d_pat_idx;
    rp.seg_score = d_seg_score; rp.frm_score = d_frm_score; rp.pat_score = d_pat_score;
    rp.counts = d_counts; rp.counts_stride = counts_stride;
    {
      ProfScope ps(ctx, 6, st);
      size_t rank_smem = (size_t)C * sizeof(double);
      rp.f_frm = reinterpret_cast<const float*>(ctx->ws + ctx->wl.f_frm); rp.f_frm_stride = pad4(c.max_frames);
      rp.f_seg = reinterpret_cast<const float*>(ctx->ws + ctx->wl.f_seg); rp.f_seg_stride = pad4(ctx->sl.max_segs);
      rp.f_pat = reinterpret_cast<const float*>(ctx->ws + ctx->wl.f_pat); rp.f_pat_stride = pad4((long long)c.max_frames * S);
      // (of each granularity the copies that fit, in its own block; none where a question sees too few for it)
      const size_t room = (size_t)kRankStageBytes - rank_smem;
      size_t stage = 0;
      const long long counts[3] = {n_seg, n_frm, n_pat};
      for (int i = 0; i < 3; ++i) {
        const size_t b = (size_t)pad4(counts[i]) * sizeof(float);
        if (counts[i] <= kRankFew || b > room || (i > 0 && mode == MUKV_RETR_HIER)) continue;
        rp.stage |= 1 << i;
        stage = std::max(stage, b);
      }
      rp.roles = rank_roles(mode, k_pat);
      e = launch_c(rank_kernel, dim3(nq * rp.roles), kRankThreads, rank_smem + stage, st, !ctx->prof_on, rp.roles, rp, meta);
    }
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "rank kernel: %s", cudaGetErrorString(e));
    ctx->launches += 4;
    return MUKV_OK;
  } catch (...) {
    return fail(ctx, MUKV_E_INVALID, "unexpected exception");
  }
}



mukv_status check_chunk_args(mukv_ctx* ctx, int n_frames, long long first_frame) {
  if (n_frames < 1) return fail(ctx, MUKV_E_INVALID, "n_frames must be >= 1");
  if (n_frames > ctx->cfg.max_frames_per_chunk)
    return fail(ctx, MUKV_E_CAPACITY, "n_frames %d exceeds max_frames_per_chunk %d", n_frames,
                ctx->cfg.max_frames_per_chunk);
  if (first_frame != ctx->frames)
    return fail(ctx, MUKV_E_STATE, "first_frame %lld does not continue the stream (%lld frames stored)", first_frame,
                ctx->frames);
  if (first_frame + n_frames > ctx->cfg.max_frames)
    return fail(ctx, MUKV_E_CAPACITY, "store full: %lld + %d frames > max_frames %lld", ctx->frames, n_frames,
                (long long)ctx->cfg.max_frames);
  return MUKV_OK;
}

}  // namespace

extern "C" {

size_t mukv_store_bytes(const mukv_config* cfg) {
  if (check_config(cfg)) return 0;
  return store_layout(*cfg).total;
}

size_t mukv_workspace_bytes(const mukv_config* cfg) {
  if (check_config(cfg)) return 0;
  return work_layout(*cfg).total;
}

mukv_status mukv_create(const mukv_config* cfg, void* d_store, size_t store_bytes, void* d_workspace,
                        size_t workspace_bytes, mukv_ctx** out) {
  return create_impl(cfg, d_store, store_bytes, d_workspace, workspace_bytes, 0, out);
}

// Host readers of the store (a view of a region, an export): segment entries still owed by the last
// compress call are pooled on that call's stream, and the stream is waited for.
static cudaError_t settle_store(const mukv_ctx* ctx) {
  if (!ctx->seg_pending) return cudaSuccess;
  const cudaStream_t st = ctx->seg_stream;
  cudaError_t e = flush_segments(ctx, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

mukv_status mukv_export_header(const mukv_ctx* ctx, mukv_store_header* out) {
  if (!ctx || !out) return MUKV_E_INVALID;
  if (settle_store(ctx) != cudaSuccess) return MUKV_E_CUDA;
  memset(out, 0, sizeof *out);
  out->magic = MUKV_STORE_MAGIC;
  out->version = MUKV_STORE_VERSION;
  out->cfg = ctx->cfg;
  out->frames = ctx->frames;
  out->store_bytes = ctx->sl.total;
  return MUKV_OK;
}

mukv_status mukv_import(const mukv_store_header* header, void* d_store, size_t store_bytes, void* d_workspace,
                        size_t workspace_bytes, mukv_ctx** out) {
  if (!out) return fail(nullptr, MUKV_E_INVALID, "out is null");
  *out = nullptr;
  if (!header) return fail(nullptr, MUKV_E_INVALID, "null header");
  if (header->magic != MUKV_STORE_MAGIC || header->version != MUKV_STORE_VERSION)
    return fail(nullptr, MUKV_E_INVALID, "not a store header of this library version");
  if (header->frames < 0 || header->frames > header->cfg.max_frames)
    return fail(nullptr, MUKV_E_INVALID, "header: frame count out of range");
  if (check_config(&header->cfg) == nullptr && header->store_bytes != store_layout(header->cfg).total)
    return fail(nullptr, MUKV_E_INVALID, "header: store size does not match its configuration");
  return create_impl(&header->cfg, d_store, store_bytes, d_workspace, workspace_bytes, header->frames, out);
}

}  // extern "C"

namespace {
mukv_status create_impl(const mukv_config* cfg, void* d_store, size_t store_bytes, void* d_workspace,
                        size_t workspace_bytes, long long frames0, mukv_ctx** out) {
  if (!out) return fail(nullptr, MUKV_E_INVALID, "out is null");
  *out = nullptr;
  if (!cfg || !d_store || !d_workspace) return fail(nullptr, MUKV_E_INVALID, "null argument");
  if (const char* why = check_config(cfg))
    return fail(nullptr, (cfg->dtype != MUKV_BF16 && cfg->dtype != MUKV_FP32) ? MUKV_E_DTYPE : MUKV_E_SHAPE, "%s", why);
  if (!aligned16(d_store) || !aligned16(d_workspace))
    return fail(nullptr, MUKV_E_ALIGN, "store and workspace must be 16-byte aligned");
  mukv_ctx* ctx = new (std::nothrow) mukv_ctx();
  if (!ctx) return fail(nullptr, MUKV_E_INVALID, "out of host memory");
  ctx->cfg = *cfg;
  ctx->sl = store_layout(*cfg);
  ctx->wl = work_layout(*cfg);
  if (store_bytes < ctx->sl.total || workspace_bytes < ctx->wl.total) {
    const size_t need_s = ctx->sl.total, need_w = ctx->wl.total;
    delete ctx;
    return fail(nullptr, MUKV_E_CAPACITY, "store needs %zu bytes (got %zu), workspace needs %zu bytes (got %zu)",
                need_s, store_bytes, need_w, workspace_bytes);
  }
  ctx->store = static_cast<unsigned char*>(d_store);
  ctx->ws = static_cast<unsigned char*>(d_workspace);
  ctx->frames = frames0;
  ctx->launches = 0;
  ctx->C = cfg->n_kv_heads * cfg->head_dim;
  ctx->G = cfg->n_q_heads / cfg->n_kv_heads;
  ctx->Ls = cfg->n_score_layers > 1 ? cfg->n_score_layers : 1;
  ctx->esize = cfg->dtype == MUKV_BF16 ? 2 : 4;
  ctx->key_rows = cfg->tokens_per_frame + cfg->past_frames * cfg->keep_per_frame;
  ctx->nc = pick_nc(ctx->key_rows);
  ctx->tcs = tc_shape(*cfg);
  ctx->n_sms = 1;
  ctx->flag_margin = kFlagMargin;
  ctx->flat_ratio = kFlatRatio;
  const int D = cfg->head_dim;
  cudaError_t e = raise_kernel_limits(&ctx->n_sms, &ctx->places);
  if (e == cudaSuccess && (ctx->tcs.ok || ctx->tcs.split)) {
    e = cudaMemcpy(ctx->ws + ctx->wl.wtab, dft_terms(D), dft_bytes(D), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !encode_map2(&ctx->wmap, ctx->ws + ctx->wl.wtab, D, 3LL * D, D)) e = cudaErrorInvalidValue;
    if (e == cudaSuccess && ctx->tcs.ok && cfg->past_frames > 0 &&
        !encode_map_pages(&ctx->pmap, ctx->store + ctx->sl.pages, D, cfg->n_kv_heads, cfg->keep_per_frame, 2 * cfg->n_layers,
                          cfg->max_frames, (long long)ctx->sl.page_bytes))
      e = cudaErrorInvalidValue;
  }
  if (e == cudaSuccess)
    e = cudaMemset(ctx->ws + ctx->wl.zero_begin, 0, ctx->wl.zero_end - ctx->wl.zero_begin);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    fail(nullptr, MUKV_E_CUDA, "mukv_create: %s", cudaGetErrorString(e));
    delete ctx;
    return MUKV_E_CUDA;
  }
  *out = ctx;
  return MUKV_OK;
}
}  // namespace

extern "C" {

void mukv_destroy(mukv_ctx* ctx) {
  if (!ctx) return;
  for (cudaEvent_t e : ctx->prof_ev) cudaEventDestroy(e);
  delete ctx;
}

mukv_status mukv_profile_enable(mukv_ctx* ctx, int32_t on) {
  if (!ctx) return MUKV_E_INVALID;
  ctx->prof_on = on != 0;
  ctx->prof_kind.clear();
  return MUKV_OK;
}

mukv_status mukv_profile_read(mukv_ctx* ctx, double* ms, int64_t* launches) {
  if (!ctx || !ms || !launches) return MUKV_E_INVALID;
  for (int i = 0; i < MUKV_PROF_KINDS; ++i) { ms[i] = 0.0; launches[i] = 0; }
  for (size_t i = 0; i < ctx->prof_kind.size(); ++i) {
    float t = 0.f;
    cudaError_t e = cudaEventSynchronize(ctx->prof_ev[2 * i + 1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&t, ctx->prof_ev[2 * i], ctx->prof_ev[2 * i + 1]);
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "mukv_profile_read: %s", cudaGetErrorString(e));
    ms[ctx->prof_kind[i]] += (double)t;
    launches[ctx->prof_kind[i]] += 1;
  }
  ctx->prof_kind.clear();
  return MUKV_OK;
}

mukv_status mukv_reset(mukv_ctx* ctx, mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  // Arrival counters, flagged lists, selection flags, statistics, the event word and the column sums start over, and so does
  // the alternation between the two sets: calls captured into a graph behind a reset are replayed with the sets that they were
  // captured with, so the reset has to leave both in the same state every time.
  cudaError_t e = zero_async(ctx->ws + ctx->wl.zero_begin, ctx->wl.zero_end - ctx->wl.zero_begin, static_cast<cudaStream_t>(stream),
                             !ctx->prof_on);
  if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "mukv_reset: %s", cudaGetErrorString(e));
  ctx->frames = 0;
  ctx->parity = 0;
  ctx->att_dirty[0] = ctx->att_dirty[1] = 0;
  ctx->failed = false;
  ctx->seg_pending = false;
  return MUKV_OK;
}

mukv_status mukv_set_option(mukv_ctx* ctx, int32_t option, double value) {
  if (!ctx) return MUKV_E_INVALID;
  switch (option) {
    case MUKV_OPT_FLAG_MARGIN:
      if (!(value >= (double)kFlagMargin) || !(value <= 4.0))
        return fail(ctx, MUKV_E_INVALID, "the safety margin can only be raised above %g (got %g)", (double)kFlagMargin, value);
      ctx->flag_margin = (float)value;
      return MUKV_OK;
    case MUKV_OPT_SCORE_PATH:
      if (value != 0.0 && value != 1.0) return fail(ctx, MUKV_E_INVALID, "score path must be 0 or 1");
      ctx->force_fma = value == 1.0;
      return MUKV_OK;
    default:
      return fail(ctx, MUKV_E_INVALID, "unknown option %d", option);
  }
}

mukv_status mukv_compress_chunk(mukv_ctx* ctx, const void* d_q, const void* d_k, const void* d_v, int32_t n_frames,
                                int64_t first_frame, int32_t* d_kept_out, float* d_scores_out,
                                mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  try {
    if (ctx->failed) return fail(ctx, MUKV_E_STATE, "an earlier call broke off half way: call mukv_reset");
    if (!d_q || !d_k || !d_v) return fail(ctx, MUKV_E_INVALID, "null input pointer");
    if (!aligned16(d_q) || !aligned16(d_k) || !aligned16(d_v) || !aligned4(d_kept_out) || !aligned4(d_scores_out))
      return fail(ctx, MUKV_E_ALIGN, "d_q, d_k, d_v must be 16-byte aligned, the outputs 4-byte aligned");
    if (const mukv_status st = check_chunk_args(ctx, n_frames, first_frame)) return st;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (ctx->cfg.dtype == MUKV_BF16)
      return compress_impl<__nv_bfloat16>(ctx, d_q, nullptr, d_k, d_v, n_frames, first_frame, d_kept_out, d_scores_out, st);
    return compress_impl<float>(ctx, d_q, nullptr, d_k, d_v, n_frames, first_frame, d_kept_out, d_scores_out, st);
  } catch (...) {
    return fail(ctx, MUKV_E_INVALID, "unexpected exception");
  }
}

mukv_status mukv_compress_chunk_scored(mukv_ctx* ctx, const float* d_select_scores, const void* d_k, const void* d_v,
                                       int32_t n_frames, int64_t first_frame, int32_t* d_kept_out,
                                       mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  try {
    if (ctx->failed) return fail(ctx, MUKV_E_STATE, "an earlier call broke off half way: call mukv_reset");
    if (!d_select_scores || !d_k || !d_v) return fail(ctx, MUKV_E_INVALID, "null input pointer");
    if (!aligned4(d_select_scores) || !aligned16(d_k) || !aligned16(d_v) || !aligned4(d_kept_out))
      return fail(ctx, MUKV_E_ALIGN, "d_k, d_v must be 16-byte aligned, scores and outputs 4-byte aligned");
    if (const mukv_status st = check_chunk_args(ctx, n_frames, first_frame)) return st;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (ctx->cfg.dtype == MUKV_BF16)
      return compress_impl<__nv_bfloat16>(ctx, nullptr, d_select_scores, d_k, d_v, n_frames, first_frame, d_kept_out,
                                          nullptr, st);
    return compress_impl<float>(ctx, nullptr, d_select_scores, d_k, d_v, n_frames, first_frame, d_kept_out, nullptr, st);
  } catch (...) {
    return fail(ctx, MUKV_E_INVALID, "unexpected exception");
  }
}

mukv_status mukv_retrieve(mukv_ctx* ctx, const void* d_qtok, const int32_t* h_q_offsets, const int64_t* h_t_limit,
                          int32_t nq, int32_t k_seg, int32_t k_frm, int32_t top_n, float lambda_frm, int32_t mode,
                          int32_t* d_seg_idx, int32_t* d_frm_idx, float* d_seg_score, float* d_frm_score,
                          int32_t* d_counts, mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  mukv_retr_params rp;
  memset(&rp, 0, sizeof rp);
  rp.k_seg = k_seg; rp.k_frm = k_frm; rp.k_patch = 0;
  rp.lambda_frm = lambda_frm; rp.top_n = top_n; rp.mode = mode;
  return retrieve_impl(ctx, d_qtok, h_q_offsets, h_t_limit, nq, rp, d_seg_idx, d_frm_idx, nullptr, d_seg_score,
                       d_frm_score, nullptr, d_counts, 2, stream);
}

mukv_status mukv_retrieve3(mukv_ctx* ctx, const void* d_qtok, const int32_t* h_q_offsets, const int64_t* h_t_limit,
                           int32_t nq, const mukv_retr_params* params, int32_t* d_seg_idx, int32_t* d_frm_idx,
                           int32_t* d_patch_idx, float* d_seg_score, float* d_frm_score, float* d_patch_score,
                           int32_t* d_counts, mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  if (!params) return fail(ctx, MUKV_E_INVALID, "null params");
  return retrieve_impl(ctx, d_qtok, h_q_offsets, h_t_limit, nq, *params, d_seg_idx, d_frm_idx, d_patch_idx, d_seg_score,
                       d_frm_score, d_patch_score, d_counts, 3, stream);
}

int64_t mukv_decode3_tokens(const mukv_ctx* ctx, int32_t k_seg, int32_t k_frm, int32_t k_patch) {
  if (!ctx || k_seg < 0 || k_frm < 0 || k_patch < 0) return 0;
  const mukv_config& c = ctx->cfg;
  long long pmax = 0;
  if (c.patch_split > 0) {
    const int rows = c.tokens_per_frame / c.grid_width;
    pmax = (long long)((rows + c.patch_split - 1) / c.patch_split) * ((c.grid_width + c.patch_split - 1) / c.patch_split);
    if (pmax > c.keep_per_frame) pmax = c.keep_per_frame;
  }
  long long per_frame = c.keep_per_frame;
  if (c.keep_per_segment > 0)                            // a frame may hold up to a whole segment's budget
    per_frame = c.keep_per_segment < c.tokens_per_frame ? c.keep_per_segment : c.tokens_per_frame;
  return (long long)k_seg + (long long)k_frm * per_frame + (long long)k_patch * pmax;
}

mukv_status mukv_gather3(mukv_ctx* ctx, const int32_t* d_seg_idx, const int32_t* d_frm_idx, const int32_t* d_patch_idx,
                         const int32_t* d_counts, int32_t nq, int32_t k_seg, int32_t k_frm, int32_t k_patch,
                         void* d_decode, int64_t decode_stride_bytes, int32_t* d_ntok, int32_t* d_tok_meta,
                         mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  try {
    if (ctx->failed) return fail(ctx, MUKV_E_STATE, "an earlier call broke off half way: call mukv_reset");
    if (!d_seg_idx || !d_frm_idx || !d_counts || !d_decode || !d_ntok) return fail(ctx, MUKV_E_INVALID, "null argument");
    if (k_patch > 0 && !d_patch_idx) return fail(ctx, MUKV_E_INVALID, "d_patch_idx is null");
    if (!aligned4(d_seg_idx) || !aligned4(d_frm_idx) || !aligned4(d_patch_idx) || !aligned4(d_counts) ||
        !aligned16(d_decode) || !aligned4(d_ntok) || !aligned4(d_tok_meta))
      return fail(ctx, MUKV_E_ALIGN, "d_decode must be 16-byte aligned, index arrays 4-byte aligned");
    if (nq < 1 || k_seg < 1 || k_frm < 1 || k_patch < 0) return fail(ctx, MUKV_E_INVALID, "nq, k_seg, k_frm must be >= 1");
    if (nq > MUKV_MAX_QUESTIONS || k_seg > MUKV_MAX_TOPK || k_frm > MUKV_MAX_TOPK || k_patch > MUKV_MAX_TOPK)
      return fail(ctx, MUKV_E_CAPACITY, "nq or a k too large");
    const mukv_config& c = ctx->cfg;
    if (k_patch > 0 && c.patch_split == 0) return fail(ctx, MUKV_E_STATE, "the store has no patch level");
    const long long tok_cap = mukv_decode3_tokens(ctx, k_seg, k_frm, k_patch);
    const long long need = (long long)c.n_layers * 2 * tok_cap * ctx->C * ctx->esize;
    if (decode_stride_bytes < need)
      return fail(ctx, MUKV_E_CAPACITY, "decode_stride_bytes %lld < %lld needed per question",
                  (long long)decode_stride_bytes, need);
    if (decode_stride_bytes % 16 != 0) return fail(ctx, MUKV_E_ALIGN, "decode_stride_bytes must be a multiple of 16");
    if (ctx->seg_pending) {                                // the summary tokens are segment entries
      const cudaError_t ef = flush_segments(ctx, static_cast<cudaStream_t>(stream));
      if (ef != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "segment kernel: %s", cudaGetErrorString(ef));
      ctx->launches += 1;
    }
    Gather3Params gp;
    memset(&gp, 0, sizeof gp);
    gp.nq = nq; gp.k_seg = k_seg; gp.k_frm = k_frm; gp.k_pat = k_patch; gp.L = c.n_layers; gp.kappa = c.keep_per_frame;
    gp.C = ctx->C; gp.P = c.tokens_per_frame; gp.S = c.patch_split * c.patch_split; gp.grid_width = c.grid_width;
    gp.patch_split = c.patch_split; gp.tok_cap = (int)tok_cap; gp.esize = ctx->esize;
    gp.seg_idx = d_seg_idx; gp.frm_idx = d_frm_idx; gp.pat_idx = d_patch_idx; gp.counts = d_counts;
    gp.store = ctx->store;
    gp.page_table = reinterpret_cast<const long long*>(ctx->store + ctx->sl.page_table);
    gp.kept_store = reinterpret_cast<const int*>(ctx->store + ctx->sl.kept);
    gp.seg_entry = reinterpret_cast<const float*>(ctx->store + ctx->sl.seg_entry);
    gp.patch_cnt = reinterpret_cast<const int*>(ctx->store + ctx->sl.patch_cnt);
    gp.kept_count = c.keep_per_segment > 0 ? reinterpret_cast<const int*>(ctx->store + ctx->sl.kept_count) : nullptr;
    gp.kept_stride = (int)ctx->sl.kept_stride;
    gp.decode = static_cast<unsigned char*>(d_decode);
    gp.decode_stride = decode_stride_bytes;
    gp.ntok = d_ntok; gp.tok_meta = d_tok_meta;
    const long long units = (long long)nq * c.n_layers * 2 * (k_frm + 1);
    const unsigned blocks = (unsigned)(units < 0x7fffffffLL ? units : 0x7fffffffLL);   // one run per block, see gather_kernel
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    {
      ProfScope ps(ctx, 7, st);
      e = launch_k(c.dtype == MUKV_BF16 ? gather3_kernel<__nv_bfloat16> : gather3_kernel<float>, dim3(blocks), 256, 0, st,
                   !ctx->prof_on, gp);
    }
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "gather3 kernel: %s", cudaGetErrorString(e));
    ctx->launches += 1;
    return MUKV_OK;
  } catch (...) {
    return fail(ctx, MUKV_E_INVALID, "unexpected exception");
  }
}

mukv_status mukv_gather(mukv_ctx* ctx, const int32_t* d_frm_idx, const int32_t* d_counts, int32_t nq, int32_t k_frm,
                        void* d_decode, int64_t decode_stride_bytes, int32_t* d_tok_meta, mukv_stream stream) {
  if (!ctx) return MUKV_E_INVALID;
  try {
    if (ctx->failed) return fail(ctx, MUKV_E_STATE, "an earlier call broke off half way: call mukv_reset");
    if (!d_frm_idx || !d_counts || !d_decode) return fail(ctx, MUKV_E_INVALID, "null argument");
    if (!aligned4(d_frm_idx) || !aligned4(d_counts) || !aligned16(d_decode) || !aligned4(d_tok_meta))
      return fail(ctx, MUKV_E_ALIGN, "d_decode must be 16-byte aligned, index arrays 4-byte aligned");
    if (ctx->cfg.keep_per_segment > 0)
      return fail(ctx, MUKV_E_UNSUPPORTED, "pages have different lengths (segment-level selection): use mukv_gather3");
    if (nq < 1 || k_frm < 1) return fail(ctx, MUKV_E_INVALID, "nq and k_frm must be >= 1");
    if (nq > MUKV_MAX_QUESTIONS || k_frm > MUKV_MAX_TOPK)
      return fail(ctx, MUKV_E_CAPACITY, "nq or k_frm too large");
    const mukv_config& c = ctx->cfg;
    const long long run = (long long)c.keep_per_frame * ctx->C * ctx->esize;
    const long long need = (long long)c.n_layers * 2 * k_frm * run;
    if (decode_stride_bytes < need)
      return fail(ctx, MUKV_E_CAPACITY, "decode_stride_bytes %lld < %lld needed per question",
                  (long long)decode_stride_bytes, need);
    if (decode_stride_bytes % 16 != 0) return fail(ctx, MUKV_E_ALIGN, "decode_stride_bytes must be a multiple of 16");
    GatherParams gp;
    gp.nq = nq; gp.k_frm = k_frm; gp.L = c.n_layers; gp.kappa = c.keep_per_frame;
    gp.run_bytes = run;
    gp.frm_idx = d_frm_idx; gp.counts = d_counts;
    gp.store = ctx->store;
    gp.page_table = reinterpret_cast<const long long*>(ctx->store + ctx->sl.page_table);
    gp.kept_store = reinterpret_cast<const int*>(ctx->store + ctx->sl.kept);
    gp.decode = static_cast<unsigned char*>(d_decode);
    gp.decode_stride = decode_stride_bytes;
    gp.tok_meta = d_tok_meta;
    const long long units = (long long)nq * c.n_layers * 2 * k_frm;
    const unsigned blocks = (unsigned)(units < 0x7fffffffLL ? units : 0x7fffffffLL);   // one run per block, see gather_kernel
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    {
      ProfScope ps(ctx, 7, st);
      const bool wide = run >= 16 * 1024;
      e = launch_k(wide ? gather_kernel<512> : gather_kernel<128>, dim3(blocks), wide ? 512u : 128u, 0, st, !ctx->prof_on, gp);
    }
    if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "gather kernel: %s", cudaGetErrorString(e));
    ctx->launches += 1;
    return MUKV_OK;
  } catch (...) {
    return fail(ctx, MUKV_E_INVALID, "unexpected exception");
  }
}

void* mukv_store_region(const mukv_ctx* ctx, int32_t which, size_t* bytes) {
  if (!ctx) return nullptr;
  if (settle_store(ctx) != cudaSuccess) return nullptr;
  const mukv_config& c = ctx->cfg;
  const StoreLayout& s = ctx->sl;
  const size_t T = (size_t)c.max_frames, C = (size_t)ctx->C;
  size_t off = 0, sz = 0;
  switch (which) {
    case 0: off = s.pages; sz = s.pages_bytes; break;
    case 1: off = s.kept; sz = T * s.kept_stride * sizeof(int); break;
    case 10: if (c.keep_per_segment <= 0) return nullptr; off = s.kept_count; sz = T * sizeof(int); break;
    case 2: off = s.frame_entry; sz = T * c.n_layers * 2 * C * sizeof(float); break;
    case 3: off = s.seg_entry; sz = (size_t)s.max_segs * c.n_layers * 2 * C * sizeof(float); break;
    case 4: off = s.frame_key; sz = T * C * sizeof(float); break;
    case 5: off = s.seg_key; sz = (size_t)s.max_segs * C * sizeof(float); break;
    case 6: off = s.frame_ts; sz = T * sizeof(long long); break;
    case 7: off = s.page_table; sz = T * sizeof(long long); break;
    case 8: off = s.patch_key; sz = T * c.patch_split * c.patch_split * C * sizeof(float); break;
    case 9: off = s.patch_cnt; sz = T * c.patch_split * c.patch_split * sizeof(int); break;
    default: return nullptr;
  }
  if (bytes) *bytes = sz;
  return ctx->store + off;
}

mukv_status mukv_get_stats(mukv_ctx* ctx, mukv_stats* out, mukv_stream stream) {
  if (!ctx || !out) return MUKV_E_INVALID;
  memset(out, 0, sizeof *out);
  long long refined = 0;
  int dev_status = 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(&refined, ctx->ws + ctx->wl.stat_refined, sizeof refined, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&dev_status, ctx->ws + ctx->wl.dev_status, sizeof dev_status, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(ctx, MUKV_E_CUDA, "mukv_get_stats: %s", cudaGetErrorString(e));
  const mukv_config& c = ctx->cfg;
  out->frames = ctx->frames;
  out->segments = (ctx->frames + c.frames_per_segment - 1) / c.frames_per_segment;
  out->kept_tokens = ctx->frames * c.keep_per_frame;
  out->page_bytes = (long long)ctx->sl.page_bytes;
  out->store_bytes_used = ctx->frames * (long long)ctx->sl.page_bytes;
  if (c.keep_per_segment > 0) {
    const long long fs = c.frames_per_segment, full = ctx->frames / fs, rest = ctx->frames % fs;
    out->kept_tokens = full * c.keep_per_segment + (long long)c.keep_per_segment * rest / fs;
    out->page_bytes = 0;                                 // pages have different lengths
    out->store_bytes_used = out->kept_tokens * c.n_layers * 2 * ctx->C * ctx->esize;
  }
  out->refined_frames = refined;
  out->kernel_launches = ctx->launches;
  out->device_status = dev_status;
  return MUKV_OK;
}

const char* mukv_last_error(const mukv_ctx* ctx) { return ctx ? ctx->err.c_str() : g_create_error.c_str(); }

}  // extern "C"

// =====================================================================================
// Scoring without a workspace.
//
// Everything above works in memory the caller hands over (store, workspace).  Some callers
// cannot produce such a buffer: a plug-in that runs inside a serving process whose start-up
// code has already given the whole device to its KV-cache pool, or a control loop that is
// forbidden to touch the allocator once it is running (cudaMalloc may fail there, and it
// synchronises the device when it does not).  For them the scratch of the scoring kernel lives
// in the array below, which is part of the loaded library image on every device.
// =====================================================================================
namespace {

constexpr int kNaFrames = MUKV_NOALLOC_MAX_FRAMES, kNaHq = MUKV_NOALLOC_MAX_Q_HEADS;
constexpr int kNaHkv = MUKV_NOALLOC_MAX_KV_HEADS, kNaP = MUKV_MAX_TOKENS;
constexpr size_t kNaColF = 0;
constexpr size_t kNaFftF = kNaColF + (size_t)kNaFrames * kNaHq * kNaP * sizeof(float);
constexpr size_t kNaColD = kNaFftF + (size_t)kNaFrames * kNaHkv * kNaP * sizeof(float);
constexpr size_t kNaFftD = kNaColD + (size_t)kNaFrames * kNaHq * kNaP * sizeof(double);
constexpr size_t kNaKept = kNaFftD + (size_t)kNaFrames * kNaHkv * kNaP * sizeof(double);
constexpr size_t kNaTs = kNaKept + (size_t)kNaFrames * kNaP * sizeof(int);
constexpr size_t kNaPt = kNaTs + 256;
constexpr size_t kNaW128 = kNaPt + 256;                  // DFT matrix terms, D = 128 and D = 64
constexpr size_t kNaW64 = kNaW128 + 3 * 128 * 128 * 2;
constexpr size_t kNaCtrl = kNaW64 + 3 * 64 * 64 * 2;     // frame_counter[16], flagged[16], n_flagged, status; at 256: sel_flag, at 512:
                                                         // head_counter
constexpr size_t kNaCtrlBytes = 512 + (size_t)kNaFrames * kNaHq * sizeof(int);
constexpr size_t kNaAtt = kNaCtrl + kNaCtrlBytes;        // column sums of the tensor-core path: zeroed together with the words
constexpr size_t kNaTotal = kNaAtt + (size_t)kNaFrames * kNaP * sizeof(unsigned long long);

// In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaTotal];

struct NoallocDevice {
  unsigned char* ptr;                                    // device address of the array
  int n_sms;
  CUtensorMap wmap128, wmap64;
};
NoallocDevice g_noalloc[kMaxDevices];

// Once per device, with that device current: resolves the array's device address and makes sure the
// scoring kernels may use the shared memory the largest supported frame needs.  Allocates nothing.
cudaError_t noalloc_setup(int dev, const NoallocDevice** out) {
  NoallocDevice& d = g_noalloc[dev];
  {
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (d.ptr) { *out = &d; return cudaSuccess; }
  }
  int n_sms = 0;
  cudaError_t e = raise_kernel_limits(&n_sms, nullptr);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  if (!d.ptr) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    unsigned char* base = static_cast<unsigned char*>(ptr);
    for (int D : {64, 128}) {
      unsigned char* dst = base + (D == 128 ? kNaW128 : kNaW64);
      e = cudaMemcpy(dst, dft_terms(D), dft_bytes(D), cudaMemcpyHostToDevice);
      if (e == cudaSuccess && !encode_map2(D == 128 ? &d.wmap128 : &d.wmap64, dst, D, 3LL * D, D)) e = cudaErrorInvalidValue;
      if (e != cudaSuccess) return e;
    }
    // (a copy from pageable memory may return before it has arrived, and the caller's stream need not wait for it)
    e = cudaStreamSynchronize(cudaStreamLegacy);
    if (e != cudaSuccess) return e;
    d.n_sms = n_sms;
    d.ptr = base;
  }
  *out = &d;
  return cudaSuccess;
}

template <typename T>
mukv_status noalloc_impl(const mukv_config& c, const void* d_q, const void* d_k_last, int n, int* d_kept_out,
                         float* d_scores_out, cudaStream_t st, unsigned long long wait_ns) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return fail(nullptr, MUKV_E_CAPACITY, "device index %d not supported", dev);
  const int P = c.tokens_per_frame, D = c.head_dim;
  const TcShape ts = tc_shape(c);
  if (sizeof(T) == 2 && !ts.ok) return fail(nullptr, MUKV_E_UNSUPPORTED, "no tiling of the scoring kernel for this shape");   // (none)
  const NoallocDevice* nd = nullptr;
  e = noalloc_setup(dev, &nd);
  if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "set-up of the static scratch: %s", cudaGetErrorString(e));
  unsigned char* base = nd->ptr;
  ScoreParams sp;
  memset(&sp, 0, sizeof sp);
  sp.P = P; sp.Hq = c.n_q_heads; sp.Hkv = c.n_kv_heads; sp.D = D; sp.G = c.n_q_heads / c.n_kv_heads;
  sp.kappa = c.keep_per_frame; sp.n_frames = n; sp.causal = c.attn_causal; sp.keep_low = c.keep_low_freq;
  sp.alpha = c.alpha; sp.tie_eps = c.tie_eps; sp.flag_margin = kFlagMargin; sp.flat_ratio = kFlatRatio;
  sp.Ls = 1;                                             // one scoring layer: the one the caller passes
  sp.q_layer_stride = (long long)n * P * c.n_q_heads * D;
  sp.k_layer_stride = (long long)n * P * c.n_kv_heads * D;
  sp.first_frame = 0;
  sp.q = d_q;
  sp.k_last = d_k_last;
  sp.colsum_part = base + kNaColF;
  sp.ifft_part = base + kNaFftF;
  sp.frame_counter = reinterpret_cast<int*>(base + kNaCtrl);
  sp.head_counter = reinterpret_cast<int*>(base + kNaCtrl + 512);
  sp.flagged = reinterpret_cast<int*>(base + kNaCtrl) + kNaFrames;
  sp.n_flagged = reinterpret_cast<int*>(base + kNaCtrl) + 2 * kNaFrames;
  sp.kept_store = d_kept_out ? d_kept_out : reinterpret_cast<int*>(base + kNaKept);
  sp.kept_out = nullptr;
  sp.scores_out = d_scores_out;
  sp.frame_ts = reinterpret_cast<long long*>(base + kNaTs);
  sp.page_table = reinterpret_cast<long long*>(base + kNaPt);
  sp.refine = 0;
  sp.row_split = 1;
  // The array keeps what the last call left, be it one that broke off or raced with another: the arrival counters, the flagged
  // count, the status word and (tensor-core path) the column sums start at zero in every call.  (Left clean by the
  // call before they could be spoilt for good.)
  e = zero_async(base + kNaCtrl, kNaCtrlBytes + (ts.ok ? (size_t)n * P * sizeof(unsigned long long) : 0), st, true);
  if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "clearing the scratch: %s", cudaGetErrorString(e));
  const int units = n * c.n_q_heads * ((P + 7) / 8);
  if constexpr (sizeof(T) == 2) {
    // bf16: scored on the tensor cores like a chunk of a context, then one block per frame selects.
    PsLaunch pl;
    memset(&pl, 0, sizeof pl);
    pl.t = &ts; pl.n_sms = nd->n_sms; pl.wmap = D == 128 ? &nd->wmap128 : &nd->wmap64;
    pl.att_acc = reinterpret_cast<unsigned long long*>(base + kNaAtt);
    pl.status = sp.n_flagged + 1;
    pl.kappa = c.keep_per_frame;
    pl.dependent = true;
    const char* why = "";
    e = launch_score_ps(pl, sp, st, &why);
    if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "%s: %s", why, cudaGetErrorString(e));
    CompactParams cp;
    memset(&cp, 0, sizeof cp);
    cp.sp = sp;
    cp.att_acc = pl.att_acc;
    cp.sel_flag = reinterpret_cast<unsigned*>(base + kNaCtrl + 256);
    cp.colsum_d = reinterpret_cast<double*>(base + kNaColD);
    cp.ifft_d = reinterpret_cast<double*>(base + kNaFftD);
    cp.sp.scratch_rows = kNaFrames * kNaHq;
    cp.wait_ns = wait_ns;
    // (blocks for the flagged frames: two per SM are resident beside one another; they wait for the first n only)
    e = launch_k(select_kernel, dim3(n + std::min(units, 2 * nd->n_sms)), kCompactThreads, 0, st, true, cp, (const int*)pl.status);
    if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "select kernel: %s", cudaGetErrorString(e));
  } else {
    e = launch_score<T>(sp, pick_nc(P), dim3(c.n_q_heads, n), score_smem_bytes<T>(P, D), st, true);
    if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "score kernel: %s", cudaGetErrorString(e));
    // Flagged frames in double precision.  The scratch holds the partial sums of 16 frames with one block per head; while
    // few frames are flagged the same room lets several blocks share a head.
    sp.refine = 1;
    sp.scratch_rows = kNaFrames * kNaHq;
    sp.colsum_part = base + kNaColD;
    sp.ifft_part = base + kNaFftD;
    e = launch_k(score64_kernel<T>, dim3(std::min(units, nd->n_sms)), kScoreThreads, 0, st, true, sp);
    if (e != cudaSuccess) return fail(nullptr, MUKV_E_CUDA, "refine kernel: %s", cudaGetErrorString(e));
  }
  return MUKV_OK;
}

// wait_ns: limit of the waits inside select_kernel
mukv_status score_frames_noalloc(const mukv_config* cfg, const void* d_q, const void* d_k_last, int32_t n_frames,
                                 int32_t* d_kept_out, float* d_scores_out, mukv_stream stream, unsigned long long wait_ns) {
  try {
    if (!cfg || !d_q || !d_k_last) return fail(nullptr, MUKV_E_INVALID, "null argument");
    if (!d_kept_out && !d_scores_out) return fail(nullptr, MUKV_E_INVALID, "no output requested");
    mukv_config c = *cfg;
    c.max_frames = 1;                                            // fields this entry point ignores
    c.max_frames_per_chunk = 1;
    c.n_layers = 1;
    c.frames_per_segment = 1;
    c.n_score_layers = 0;
    c.score_layer_offset = 0;
    c.patch_split = 0;
    c.keep_per_segment = 0;
    c.past_frames = 0;
    c.reserved = 0;
    if (const char* why = check_config(&c))
      return fail(nullptr, (c.dtype != MUKV_BF16 && c.dtype != MUKV_FP32) ? MUKV_E_DTYPE : MUKV_E_SHAPE, "%s", why);
    if (n_frames < 1) return fail(nullptr, MUKV_E_INVALID, "n_frames must be >= 1");
    if (n_frames > kNaFrames || c.n_q_heads > kNaHq || c.n_kv_heads > kNaHkv)
      return fail(nullptr, MUKV_E_CAPACITY,
                  "the static scratch holds at most %d frames, %d query heads and %d key heads per call "
                  "(got %d, %d, %d)", kNaFrames, kNaHq, kNaHkv, n_frames, c.n_q_heads, c.n_kv_heads);
    if (!aligned16(d_q) || !aligned16(d_k_last) || !aligned4(d_kept_out) || !aligned4(d_scores_out))
      return fail(nullptr, MUKV_E_ALIGN, "d_q, d_k_last must be 16-byte aligned, the outputs 4-byte aligned");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (c.dtype == MUKV_BF16)
      return noalloc_impl<__nv_bfloat16>(c, d_q, d_k_last, n_frames, d_kept_out, d_scores_out, st, wait_ns);
    return noalloc_impl<float>(c, d_q, d_k_last, n_frames, d_kept_out, d_scores_out, st, wait_ns);
  } catch (...) {
    return fail(nullptr, MUKV_E_INVALID, "unexpected exception");
  }
}

}  // namespace

extern "C" mukv_status mukv_score_frames_noalloc(const mukv_config* cfg, const void* d_q, const void* d_k_last,
                                                 int32_t n_frames, int32_t* d_kept_out, float* d_scores_out,
                                                 mukv_stream stream) {
  return score_frames_noalloc(cfg, d_q, d_k_last, n_frames, d_kept_out, d_scores_out, stream, kWaitNs);
}
