// KV compaction into the paged store and block pooling (Sec. 3.3 "selected KV slices ... are
// stored", Sec. 3.4 Eq. 5), and the in-block selection that feeds it (Eq. 4 and the top-kappa rule).
//
// compact_kernel<T>: one thread block per (layer, K|V, frame).  The kappa kept rows of that
// plane (C = Hkv*D elements each, one contiguous run in the input) are copied, in ascending
// token order, to the frame's page; the same registers feed the mean over the kept rows.
// The last-layer key plane is summed in double: its mean is the retrieval key (Eq. 5) that
// later ranks blocks, so it is kept free of accumulation-order noise.
//
// Where do the kept ids come from?  After the persistent tensor-core scoring kernel every block
// works them out itself (sel_mode 1): it reads the column sums of its frame, adds the key heads'
// frequency sums in a fixed order, applies Eq. 4 and selects, all in single precision; the blocks of a frame run
// the same arithmetic on the same numbers, so they agree, and the one with plane 0 writes the ids
// and the index.  That costs a few microseconds at the start of each block, in parallel on the
// whole device, where a selection inside the scoring kernel left one block per frame working while
// all others had finished.  After the other scoring kernels the ids are read from the store
// (sel_mode 0).  Either way a frame whose lowest kept and highest dropped score are closer than
// tie_eps + flag_margin is skipped here: redo_flagged decides it in double precision and compacts it.
//
// Flagged frames (about one chunk in fifty on the synthetic streams): redo_flagged.  Blocks behind those of the copies (bf16
// calls; p.redo_blocks of them) wait until the ids of every frame of the chunk are published or the frame is on the list, and
// leave if the list is empty; else they score its frames in double precision (score64.cuh), and when the selections have all been
// made they compact those frames.  Units of both are taken by ticket: a block waits for units that other blocks have taken, never
// for a block that has not started, so nothing depends on how many of them the device has a place for (another context's blocks,
// or a kernel of the caller's, may hold places).  fp32 calls have tail_kernel<T> for it, a launch behind compact_kernel.
// The segment entries (Eq. 5 at segment level; one (layer, K|V) plane per block, mean over the frames
// present) of the common case are not written by the call itself.  The next call pools them with a row
// of compact_kernel blocks that does not wait for its scoring kernel (CompactParams::prev), or the first
// reader launches segment_kernel for them.  (As the last launch of every call that kernel cost 6 us;
// pooling by the compaction block that finishes a plane last was measured too: the fence every block
// then needs before it signs off costs more than a launch.)
#pragma once
#include "common.cuh"
#include "score64.cuh"

namespace mukv {

constexpr int kCompactThreads = 256;
constexpr int kTailWords = 2;
static_assert(kCompactThreads == kScoreThreads, "redo_flagged runs the scoring and the compaction code in one block");

struct CompactParams {
  int L, kappa, C, P;             // C = Hkv*D elements per row
  int n_frames;
  long long first_frame;
  const void* k;                  // [L][n][P][C]
  const void* v;
  unsigned char* store;           // store base
  float* frame_entry;             // [max_frames][L][2][C]
  float* frame_key;               // [max_frames][C]
  double* frame_ksum;             // [max_frames][C]  exact sums of the last-layer kept keys
  long long* stat_refined;        // device counter
  // Words of redo_flagged.  Two sets of them (and of the flagged count) alternate from call to call, and a call clears those of
  // the next one: whatever a call leaves behind, a wait that ran out included, is nothing that a later one starts from.
  int* n_flagged_next;            // the flagged count of the next call
  int* tail_ctr;                  // [kTailWords] next unit, frames selected (sp.n_selected)
  int* tail_next;                 // the next call's
  int redo_blocks;                // compact_kernel: blocks at the end of the grid that redo flagged frames (0: none)
  double *colsum_d, *ifft_d;      // their partial sums, see score64_frame_block
  // segment entries (Eq. 5 at segment level)
  int fseg;                       // frames per segment
  float* seg_entry;               // [max_segs][L][2][C]
  float* seg_key;                 // [max_segs][C]
  // selection
  // patch-level blocks (Sec. 3.2; Eq. 5 "similarly"): S = patch_split^2 super patches per frame
  int patch_split, grid_width;    // 0: no patch level
  float* patch_key;               // [max_frames][S][C]
  int* patch_cnt;                 // [max_frames][S]
  // compact_kernel: with prev.n_frames > 0 the grid has prev_rows more rows of blocks (behind the first one), which
  // pool the segment entries the previous call left to this one.  prev_rows = ceil(2L / n_frames), one (layer, K|V)
  // plane per block: a plane is a chain of L2 round trips of about 5 us, so that a single row of n_frames blocks
  // with several planes each kept one-frame calls waiting for 70 us (28 layers) behind 8 us of copying
  SegmentArgs prev;
  int prev_rows;
  int parts;                      // compact_kernel: blocks that share a (layer, K|V) plane of a frame, by columns
  int sel_mode;                   // 0: kept ids are in the store; 1: select here from the partial sums;
                                  // 2: select here by the caller's scores; 3: ids and counts are in the store
                                  // (segment-level selection)
  const float* ext_scores;        // [n_frames][P] (sel_mode 2)
  const int* kept_count;          // [max_frames] (sel_mode 3: a frame's page holds that many tokens; ids in
                                  // kept_store with a stride of P), else null
  const unsigned long long* att_acc;  // [F][P] column sums of the persistent scoring kernel (sel_mode 1)
  unsigned long long* att_clear;  // sums of the call before, cleared for the next one
  long long n_clear;
  int later_blocks;               // 1: the grid is larger than what is resident at once
  unsigned* sel_flag;             // [F] (epoch << 1 | risky) once the plane-0 block has published its frame's ids
  unsigned epoch;                 // number of this call, never repeated
  unsigned long long wait_ns;     // limit of a wait for other blocks of the grid
  ScoreParams sp;                 // partial sums, Eq. 4 parameters, index and flag outputs
};

// a token id read back from memory, forced into the frame (row addresses are computed from it)
__device__ __forceinline__ int token_id(int id, int P) { return (unsigned)id < (unsigned)P ? id : 0; }

struct SelectScratch {
  unsigned mm[kCompactThreads / 32][4];   // per-warp min / max keys of the two signals
  int hist[256];
  int list[256];                  // keys of the scores in the bin that holds the kappa-th largest
  int cnt[kCompactThreads / 32][4];
  unsigned ab[kCompactThreads / 32][2];
  int bin, rank, n_list;
  float tau;
  // scratch of select_by_score (ranking by the caller's scores)
  double sc64[MUKV_MAX_TOKENS];
  double misc64[4 * (kCompactThreads / 32)];
  int cnt64[kCompactThreads / 32 + 1];
};

// Eq. 4 and the top-kappa rule for frame f from the partial sums of the persistent scoring kernel,
// run by a whole block of kCompactThreads threads (thread t owns token t; P <= 256).  The kept ids
// go to s_kept in ascending order; with `write` also to the store and to the caller's outputs.
// Returns true when single precision cannot decide the frame safely (see select_frame): nothing
// of the frame may then be used, and with `write` the frame has been put on the flagged list.
// Everything is single precision; scores lie in [0, 1], so their bit patterns order like the
// values and the reductions run on them as integers.
__device__ inline bool select_from_partials(const CompactParams& p, int f, bool write, int* s_kept, SelectScratch* sc) {
  const ScoreParams& sp = p.sp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = kCompactThreads / 32;
  const int P = sp.P, Hkv = sp.Hkv * sp.Ls, kappa = sp.kappa;   // key heads of all scoring layers
  const bool valid = tid < P;
  float att = 0.f, fft = 0.f;
  if (valid) {
    const float* fp = reinterpret_cast<const float*>(sp.ifft_part) + (long long)f * Hkv * P + tid;
    const unsigned long long a64 = __ldcg(p.att_acc + (long long)f * P + tid);
    float f32 = 0.f;
#pragma unroll 1
    for (int g = 0; g < Hkv; g += 8) {                     // (eight key heads in flight)
      float y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = g + i < Hkv ? __ldcg(fp + (long long)(g + i) * P) : 0.f;
#pragma unroll
      for (int w = 4; w >= 1; w >>= 1)
#pragma unroll
        for (int i = 0; i < w; ++i) y[i] += y[i + w];
      f32 += y[0];
    }
    // (divisions: a rounded reciprocal would shift all scores of a frame alike, I_att of 28 heads x 196 tokens by 4e-8)
    att = att_value(a64) / (float)((long long)sp.Hq * sp.Ls * P);
    fft = f32 / (float)((long long)Hkv * sp.D);
  }
  // ---- min / max of both signals over the frame (both are sums of non-negative terms)
  {
    const unsigned ka = __float_as_uint(att), kf = __float_as_uint(fft);
    const unsigned v0 = __reduce_min_sync(kFull, valid ? ka : 0xffffffffu), v1 = __reduce_max_sync(kFull, valid ? ka : 0u);
    const unsigned v2 = __reduce_min_sync(kFull, valid ? kf : 0xffffffffu), v3 = __reduce_max_sync(kFull, valid ? kf : 0u);
    if (lane == 0) { sc->mm[warp][0] = v0; sc->mm[warp][1] = v1; sc->mm[warp][2] = v2; sc->mm[warp][3] = v3; }
    sc->hist[tid] = 0;
    if (tid == 0) sc->n_list = 0;
  }
  // a frame with a score that is not a number has no ranking: every score counts as 0 below, so
  // that the lowest kappa ids are kept (every block of the frame sees the same sums and agrees)
  const bool bad = __syncthreads_or(valid && !(isfinite(att) && isfinite(fft))) != 0;
  const int wl = lane < NW ? lane : 0;                     // lanes past the warp count repeat warp 0
  const unsigned m0 = __reduce_min_sync(kFull, sc->mm[wl][0]), m1 = __reduce_max_sync(kFull, sc->mm[wl][1]);
  const unsigned m2 = __reduce_min_sync(kFull, sc->mm[wl][2]), m3 = __reduce_max_sync(kFull, sc->mm[wl][3]);
  const float amin = __uint_as_float(m0), amax = __uint_as_float(m1);
  const float fmin_ = __uint_as_float(m2), fmax_ = __uint_as_float(m3);
  // ---- Eq. 4
  // (one reciprocal per signal, the same in every thread, instead of a division per token)
  const float inv_a = (amax == amin) ? 0.f : 1.f / (amax - amin);
  const float inv_f = (fmax_ == fmin_) ? 0.f : 1.f / (fmax_ - fmin_);
  const float an = (att - amin) * inv_a;
  float fn = (fft - fmin_) * inv_f;
  if (sp.keep_low) fn = 1.f - fn;
  const float s = bad ? 0.f : sp.alpha * an + (1.f - sp.alpha) * fn;
  const int key = __float_as_int(s);
  // ---- tau = kappa-th largest score: a 256-bin histogram finds its bin, the scores of that bin
  // are ranked among themselves
  int bin = (int)(s * 256.f);
  bin = bin < 0 ? 0 : (bin > 255 ? 255 : bin);
  if (valid) atomicAdd(&sc->hist[bin], 1);
  __syncthreads();
  if (warp == 0) {
    int c[8], T = 0;                                     // lane l owns bins 8l .. 8l+7
#pragma unroll
    for (int i = 0; i < 8; ++i) { c[i] = sc->hist[8 * lane + i]; T += c[i]; }
    int incl = T;                                        // scores in this lane's bins and all higher ones
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_down_sync(kFull, incl, o);
      if (lane + o < 32) incl += v;
    }
    const int above = incl - T;
    if (above < kappa && kappa <= above + T) {           // true for exactly one lane
      int r = kappa - above, b = 7;
      for (; b > 0; --b) {
        if (r <= c[b]) break;
        r -= c[b];
      }
      sc->bin = 8 * lane + b;
      sc->rank = r;
    }
  }
  __syncthreads();
  const bool member = valid && bin == sc->bin;
  if (member) sc->list[atomicAdd(&sc->n_list, 1)] = key;
  __syncthreads();
  if (member) {
    const int n = sc->n_list, r = sc->rank;
    int gt = 0, ge = 0;
    for (int i = 0; i < n; ++i) {
      const int o = sc->list[i];
      gt += (o > key);
      ge += (o >= key);
    }
    if (gt < r && r <= ge) sc->tau = s;                  // every writer holds the same value
  }
  __syncthreads();
  const float tau = sc->tau;
  const float delta = sp.tie_eps;
  const bool sure = valid && (s > tau + delta);
  const bool band = valid && !sure && (s >= tau - delta);
  const unsigned lt = (1u << lane) - 1u;
  const unsigned b_sure = __ballot_sync(kFull, sure), b_band = __ballot_sync(kFull, band);
  if (lane == 0) { sc->cnt[warp][0] = __popc(b_sure); sc->cnt[warp][1] = __popc(b_band); }
  __syncthreads();
  int n_sure = 0, band_rank = __popc(b_band & lt);
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    n_sure += sc->cnt[w][0];
    if (w < warp) band_rank += sc->cnt[w][1];
  }
  const bool keep = sure || (band && band_rank < kappa - n_sure);
  const unsigned b_keep = __ballot_sync(kFull, keep);
  {
    // lowest kept and highest dropped score, for the safety test below
    const unsigned ks = (unsigned)key;
    const unsigned a = __reduce_min_sync(kFull, keep ? ks : 0xffffffffu);
    const unsigned b = __reduce_max_sync(kFull, (valid && !keep) ? ks : 0u);
    if (lane == 0) { sc->cnt[warp][2] = __popc(b_keep); sc->ab[warp][0] = a; sc->ab[warp][1] = b; }
  }
  __syncthreads();
  int pos = __popc(b_keep & lt);
  unsigned ka = 0xffffffffu, kb = 0u;
  bool any_dropped = false;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    if (w < warp) pos += sc->cnt[w][2];
    ka = min(ka, sc->ab[w][0]);
    kb = max(kb, sc->ab[w][1]);
  }
  any_dropped = kappa < P;
  // does single precision decide this frame safely?  (see select_frame)
  const float a = __uint_as_float(ka), b = any_dropped ? __uint_as_float(kb) : -3.0e38f;
  bool risky = any_dropped && (a - b <= delta + sp.flag_margin);
  const float aabs = fmaxf(amax, -amin), fabs_ = fmaxf(fmax_, -fmin_);
  if (amax != amin && (amax - amin) < sp.flat_ratio * aabs && sp.alpha != 0.f) risky = true;
  if (fmax_ != fmin_ && (fmax_ - fmin_) < sp.flat_ratio * fabs_ && sp.alpha != 1.f) risky = true;
  // column sums too close together for their fixed-point step (see kAttFine); equal ones only when they are small as well
  const float fine = kAttFine / (float)((long long)sp.Hq * sp.Ls * P);
  if (amax - amin < fine && (amax != amin || amax < fine)) risky = true;
  if (bad) risky = false;                                 // double precision would not rank it either
  if (keep) s_kept[pos] = tid;
  if (write) {
    const long long f_abs = sp.first_frame + f;
    if (keep) {
      sp.kept_store[f_abs * kappa + pos] = tid;
      if (sp.kept_out) sp.kept_out[(long long)f * kappa + pos] = tid;
    }
    if (sp.scores_out && valid) {
      const long long np = (long long)sp.n_frames * P;
      sp.scores_out[0 * np + (long long)f * P + tid] = att;
      sp.scores_out[1 * np + (long long)f * P + tid] = fft;
      sp.scores_out[2 * np + (long long)f * P + tid] = s;
    }
    if (tid == 0) {
      sp.frame_ts[f_abs] = f_abs;
      sp.page_table[f_abs] = sp.pages_off + f_abs * sp.page_bytes;
      if (risky) sp.flagged[atomicAdd(sp.n_flagged, 1)] = f;
      if (bad && sp.status) atomicCAS(sp.status, 0, kStatusNonFinite);
    }
  }
  __syncthreads();
  return risky;
}

__device__ __forceinline__ SegmentArgs segment_args(const CompactParams& p) {
  SegmentArgs a;
  a.L = p.L; a.kappa = p.kappa; a.C = p.C; a.fseg = p.fseg; a.n_frames = p.n_frames; a.first_frame = p.first_frame;
  a.frame_entry = p.frame_entry; a.frame_ksum = p.frame_ksum; a.seg_entry = p.seg_entry; a.seg_key = p.seg_key;
  a.kept_count = p.kept_count;
  return a;
}

// Segment entries (Eq. 5 at segment level) of one (layer, K|V) plane for every segment the chunk
// touches: mean over the frames present, added in frame order.  Run by one whole block.  The loads
// of up to 16 frames (and, in single precision, of two columns) are in flight together: the
// work is a chain of L2 round trips and little else.
__device__ __noinline__ void compact_segment_plane(const SegmentArgs p, int l, int kv) {
  const int tid = threadIdx.x;
  const int C = p.C, kappa = p.kappa;
  const bool exact = (l == p.L - 1) && (kv == 0);
  const long long frames_total = p.first_frame + p.n_frames;
  const long long first_seg = p.first_frame / p.fseg, last_seg = (frames_total - 1) / p.fseg;
  for (long long u = first_seg; u <= last_seg; ++u) {
    const long long t0 = u * p.fseg;
    long long t1 = t0 + p.fseg;
    if (t1 > frames_total) t1 = frames_total;
    const int nf = (int)(t1 - t0);
    if (p.kept_count) {
      // frames keep different numbers of tokens (segment-level selection): the mean over all kept
      // tokens of the segment is the count-weighted mean of the frame entries
      for (int col = tid; col < C; col += kCompactThreads) {
        long long n_tok = 0;
        double td = 0.0;
        float tf = 0.f;
        for (long long ff = t0; ff < t1; ff += 16) {
          int cn[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) cn[i] = ff + i < t1 ? __ldcg(p.kept_count + ff + i) : 0;
          if (exact) {
            double x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) x[i] = ff + i < t1 ? __ldcg(p.frame_ksum + (ff + i) * C + col) : 0.0;
#pragma unroll
            for (int i = 0; i < 16; ++i) td += x[i];
          } else {
            float x[16];
#pragma unroll
            for (int i = 0; i < 16; ++i)
              x[i] = ff + i < t1 ? __ldcg(p.frame_entry + (((ff + i) * p.L + l) * 2 + kv) * C + col) : 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i) tf += (float)cn[i] * x[i];
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) n_tok += cn[i];
        }
        if (exact) {
          const float m = n_tok ? (float)(td / (double)n_tok) : 0.f;
          p.seg_key[u * C + col] = m;
          p.seg_entry[((u * p.L + l) * 2 + kv) * C + col] = m;
        } else {
          p.seg_entry[((u * p.L + l) * 2 + kv) * C + col] = n_tok ? tf / (float)n_tok : 0.f;
        }
      }
      continue;
    }
    if (exact) {
      for (int col = tid; col < C; col += kCompactThreads) {
        double t = 0.0;
        for (long long ff = t0; ff < t1; ff += 16) {
          double x[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) x[i] = ff + i < t1 ? __ldcg(p.frame_ksum + (ff + i) * C + col) : 0.0;
#pragma unroll
          for (int i = 0; i < 16; ++i) t += x[i];
        }
        const float m = (float)(t / ((double)nf * (double)kappa));
        p.seg_key[u * C + col] = m;
        p.seg_entry[((u * p.L + l) * 2 + kv) * C + col] = m;
      }
    } else {
      for (int col = tid; col < C; col += 2 * kCompactThreads) {
        const int col1 = col + kCompactThreads;
        const bool two = col1 < C;
        float ta = 0.f, tb = 0.f;
        for (long long ff = t0; ff < t1; ff += 16) {
          float xa[16], xb[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float* src = p.frame_entry + (((ff + i) * p.L + l) * 2 + kv) * C;
            xa[i] = ff + i < t1 ? __ldcg(src + col) : 0.f;
            xb[i] = (two && ff + i < t1) ? __ldcg(src + col1) : 0.f;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) { ta += xa[i]; tb += xb[i]; }
        }
        float* dst = p.seg_entry + ((u * p.L + l) * 2 + kv) * C;
        dst[col] = ta / (float)nf;
        if (two) dst[col1] = tb / (float)nf;
      }
    }
  }
}

// Rows in flight per thread.  With 4 row groups per pass, 5 covers the 49 kept rows of the 7B shape in
// three trips (20 + 20 + 9) where 4 needs a fourth trip for a single row; the kernel then takes 80
// registers and three blocks per SM instead of four, which measured faster all the same.
constexpr int kRowsInFlight = 5;

struct CompactScratch {
  union {
    struct {
      float red[kCompactThreads * 8];
      double red64[kCompactThreads * 8];
    };
    struct {                                               // compact_plane_part
      uint4 rows[kRowsInFlight * kCompactThreads];
      double sums[kCompactThreads * 4];
    };
    Score64Scratch s64;                                    // redo_flagged
  };
  int kept[MUKV_MAX_TOKENS];
};

// Copies the kappa kept rows (ids in sc->kept, ascending) of plane (l, kv) of chunk frame f to the
// frame's page (planes of kappa rows each, starting at `page`) and writes the plane's frame entry
// (Eq. 5; zeros for a frame that keeps nothing).  Run by a whole block.
// NV = 16-byte vectors per row; the block covers 256/NV rows per pass.
template <typename T>
__device__ inline void compact_plane(const CompactParams& p, int plane, int f, CompactScratch* sc, int kappa,
                                     unsigned char* page) {
  constexpr int VE = 16 / sizeof(T);
  const int tid = threadIdx.x;
  const int l = plane >> 1, kv = plane & 1;
  const long long f_abs = p.first_frame + f;
  const int C = p.C;
  const int NV = C / VE;                        // vectors per row (power of two, <= 256)
  const int rows_per_pass = kCompactThreads / NV;
  const T* src_base = reinterpret_cast<const T*>(kv ? p.v : p.k) + ((long long)l * p.n_frames + f) * p.P * C;
  T* dst_base = reinterpret_cast<T*>(page) + (long long)plane * kappa * C;
  const int c = tid % NV, r0 = tid / NV;
  const bool exact = (l == p.L - 1) && (kv == 0);
  float acc[VE];
  double acc64[VE];
#pragma unroll
  for (int e = 0; e < VE; ++e) { acc[e] = 0.f; acc64[e] = 0.0; }
  for (int r = r0; r < kappa; r += rows_per_pass * kRowsInFlight) {
    uint4 x[kRowsInFlight];
#pragma unroll
    for (int u = 0; u < kRowsInFlight; ++u) {
      const int rr = r + u * rows_per_pass;
      if (rr < kappa) x[u] = ld_stream(src_base + (long long)sc->kept[rr] * C + c * VE);
    }
#pragma unroll
    for (int u = 0; u < kRowsInFlight; ++u) {
      const int rr = r + u * rows_per_pass;
      if (rr < kappa) {
        st_stream(dst_base + (long long)rr * C + c * VE, x[u]);
        const uint32_t w[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
        float e[VE];
        if constexpr (sizeof(T) == 2) {
#pragma unroll
          for (int i = 0; i < 4; ++i) { e[(2 * i) % VE] = bf16_lo(w[i]); e[(2 * i + 1) % VE] = bf16_hi(w[i]); }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i % VE] = __uint_as_float(w[i]);
        }
        if (exact) {
#pragma unroll
          for (int i = 0; i < VE; ++i) acc64[i] += (double)e[i];
        } else {
#pragma unroll
          for (int i = 0; i < VE; ++i) acc[i] += e[i];
        }
      }
    }
  }
  // reduce the row groups (fixed order) and write the mean
  if (exact) {
#pragma unroll
    for (int i = 0; i < VE; ++i) sc->red64[tid * VE + i] = acc64[i];
  } else {
#pragma unroll
    for (int i = 0; i < VE; ++i) sc->red[tid * VE + i] = acc[i];
  }
  __syncthreads();
  float* fe = p.frame_entry + ((f_abs * p.L + l) * 2 + kv) * C;
  for (int col = tid; col < C; col += kCompactThreads) {
    const int cv = col / VE, ce = col % VE;
    if (exact) {
      double t = 0.0;
      for (int g = 0; g < rows_per_pass; ++g) t += sc->red64[(g * NV + cv) * VE + ce];
      p.frame_ksum[f_abs * C + col] = t;
      const float m = kappa ? (float)(t / (double)kappa) : 0.f;
      fe[col] = m;
      p.frame_key[f_abs * C + col] = m;
    } else {
      float t = 0.f;
      for (int g = 0; g < rows_per_pass; ++g) t += sc->red[(g * NV + cv) * VE + ce];
      fe[col] = kappa ? t / (float)kappa : 0.f;
    }
  }
}

// The same for part `part` of `parts` (2 or 4) of the plane's columns: NV = C / VE / parts vectors per row, parts times the rows
// per pass, which takes short calls from three round trips of rows to one or two (see compact_kernel).  The rows of a trip
// go through shared memory and are added up in the order of compact_plane (256 / (C / VE) groups of rows, each ascending,
// then the groups), so that a frame's entry is the same bit for bit however the stream is cut into calls.  (Adding them up in
// the order of the copy was 0.6 us of 18 faster in a one-frame call; a thread per vector of 256 / parts threads, 13 rows each
// in flight, 9 us slower: two warps then fetch all the code.)
template <typename T>
__device__ inline void compact_plane_part(const CompactParams& p, int plane, int f, CompactScratch* sc, int kappa,
                                          unsigned char* page, int part, int parts) {
  constexpr int VE = 16 / sizeof(T), WE = VE / 2;          // elements per vector, per half of one
  const int tid = threadIdx.x;
  const int l = plane >> 1, kv = plane & 1;
  const long long f_abs = p.first_frame + f;
  const int C = p.C;
  const int NV = C / VE / parts, c_off = part * NV * VE;
  const int groups = kCompactThreads / (C / VE), rows_per_pass = groups * parts;
  const T* src_base = reinterpret_cast<const T*>(kv ? p.v : p.k) + ((long long)l * p.n_frames + f) * p.P * C + c_off;
  T* dst_base = reinterpret_cast<T*>(page) + (long long)plane * kappa * C + c_off;
  const int c = tid % NV, r0 = tid / NV;
  const bool exact = (l == p.L - 1) && (kv == 0);
  // sums: thread (row group, half vector)
  const int halves = 2 * kCompactThreads / parts;          // of a group of rows
  const int g = tid / (2 * NV);
  float acc[WE];
  double acc64[WE];
#pragma unroll
  for (int e = 0; e < WE; ++e) { acc[e] = 0.f; acc64[e] = 0.0; }
  const uint2* half = reinterpret_cast<const uint2*>(sc->rows);
  auto elem = [](const uint2& x, int e) {
    const uint32_t w = WE == 4 ? (e < 2 ? x.x : x.y) : (e == 0 ? x.x : x.y);
    return WE == 4 ? ((e & 1) ? bf16_hi(w) : bf16_lo(w)) : __uint_as_float(w);
  };
  for (int base = 0; base < kappa; base += rows_per_pass * kRowsInFlight) {
    uint4 x[kRowsInFlight];
#pragma unroll
    for (int u = 0; u < kRowsInFlight; ++u) {
      const int rr = base + u * rows_per_pass + r0;
      if (rr < kappa) x[u] = ld_stream(src_base + (long long)sc->kept[rr] * C + c * VE);
    }
    if (base) __syncthreads();                             // the previous trip's rows have been added
#pragma unroll
    for (int u = 0; u < kRowsInFlight; ++u) {
      const int rr = base + u * rows_per_pass + r0;
      if (rr < kappa) {
        st_stream(dst_base + (long long)rr * C + c * VE, x[u]);
        sc->rows[u * kCompactThreads + tid] = x[u];
      }
    }
    __syncthreads();
    const int n = min(kappa - base, rows_per_pass * kRowsInFlight);
    if (tid < halves) {
      if (exact) {
        for (int r = g, o = tid; r < n; r += groups, o += halves) {
          const uint2 y = half[o];
#pragma unroll
          for (int e = 0; e < WE; ++e) acc64[e] += (double)elem(y, e);
        }
      } else {
#pragma unroll 4
        for (int r = g, o = tid; r < n; r += groups, o += halves) {
          const uint2 y = half[o];
#pragma unroll
          for (int e = 0; e < WE; ++e) acc[e] += elem(y, e);
        }
      }
    }
  }
  float* sums = reinterpret_cast<float*>(sc->sums);        // [groups][NV * VE]
  if (tid < halves) {
#pragma unroll
    for (int e = 0; e < WE; ++e) {
      if (exact) sc->sums[tid * WE + e] = acc64[e];
      else sums[tid * WE + e] = acc[e];
    }
  }
  __syncthreads();
  const int cols = NV * VE;
  float* fe = p.frame_entry + ((f_abs * p.L + l) * 2 + kv) * C + c_off;
  for (int col = tid; col < cols; col += kCompactThreads) {
    if (exact) {
      double t = 0.0;
      for (int g = 0; g < groups; ++g) t += sc->sums[g * cols + col];
      p.frame_ksum[f_abs * C + c_off + col] = t;
      const float m = kappa ? (float)(t / (double)kappa) : 0.f;
      fe[col] = m;
      p.frame_key[f_abs * C + c_off + col] = m;
    } else {
      float t = 0.f;
      for (int g = 0; g < groups; ++g) t += sums[g * cols + col];
      fe[col] = kappa ? t / (float)kappa : 0.f;
    }
  }
}

// Patch-level block keys of chunk frame f (Eq. 5 on the kept tokens of each super patch): mean of
// their last-layer keys, summed in double like the frame key; kept ids in sc->kept.  Run by a
// whole block; the kept rows are first grouped by super patch, then every thread sums its channels
// of each group in ascending row order.  sc->red is used as scratch.
template <typename T>
__device__ __noinline__ void pool_patches(const CompactParams& p, int f, CompactScratch* sc) {
  constexpr int EW = ElemTraits<T>::kPerWord;
  const int tid = threadIdx.x;
  const int S = p.patch_split * p.patch_split, C = p.C, kappa = p.kappa;
  const long long f_abs = p.first_frame + f;
  int* order = reinterpret_cast<int*>(sc->red);          // kept ids grouped by super patch, ascending inside a group
  int* start = order + MUKV_MAX_TOKENS;                  // [S + 1] first entry of every group
  int* sp_of = start + 32;                               // [kappa] super patch of each kept row
  static_assert(sizeof(sc->red) >= (2 * MUKV_MAX_TOKENS + 32) * sizeof(int), "scratch too small");
  static_assert(MUKV_MAX_PATCH_SPLIT * MUKV_MAX_PATCH_SPLIT < 32, "group starts do not fit");
  __syncthreads();
  for (int r = tid; r < kappa; r += kCompactThreads) sp_of[r] = super_patch_index(sc->kept[r], p.P, p.grid_width, p.patch_split);
  __syncthreads();
  if (tid <= S) {
    int c = 0;
    for (int r = 0; r < kappa; ++r) c += (sp_of[r] < tid);
    start[tid] = c;
  }
  __syncthreads();
  for (int r = tid; r < kappa; r += kCompactThreads) {
    const int s = sp_of[r];
    int pos = start[s];
    for (int q = 0; q < r; ++q) pos += (sp_of[q] == s);
    order[pos] = sc->kept[r];
  }
  __syncthreads();
  // a thread owns one 32-bit word of the row (one or two channels); eight rows are in flight at a time
  const int wpr = C / EW;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(reinterpret_cast<const T*>(p.k) +
                                                          ((long long)(p.L - 1) * p.n_frames + f) * p.P * C);
  for (int w = tid; w < wpr; w += kCompactThreads) {
    for (int sp = 0; sp < S; ++sp) {
      const int b = start[sp], e = start[sp + 1];
      double t0 = 0.0, t1 = 0.0;
      for (int i = b; i < e; i += 8) {
        uint32_t x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = i + u < e ? __ldg(src + (long long)order[i + u] * wpr + w) : 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {                      // (a zero word adds +0.0)
          if (EW == 2) {
            t0 += (double)bf16_lo(x[u]);
            t1 += (double)bf16_hi(x[u]);
          } else {
            t0 += (double)__uint_as_float(x[u]);
          }
        }
      }
      const int cnt = e - b;
      float* dst = p.patch_key + ((f_abs * S) + sp) * C + (long long)w * EW;
      dst[0] = cnt ? (float)(t0 / (double)cnt) : 0.f;
      if (EW == 2) dst[1] = cnt ? (float)(t1 / (double)cnt) : 0.f;
    }
  }
  if (tid < S) p.patch_cnt[f_abs * S + tid] = start[tid + 1] - start[tid];
}

// is chunk frame f on the flagged list (of n entries)?
__device__ __forceinline__ bool frame_is_flagged(const int* flagged, int n, int f) {
  bool hit = false;
  for (int i = 0; i < n; ++i) hit |= (__ldcg(flagged + i) == f);
  return hit;
}

// Bounded wait until done() holds (other blocks of the same grid bring it about).  False after limit_ns; 0: one look.
constexpr unsigned long long kWaitNs = 1500000000ull;
template <typename Done>
__device__ __forceinline__ bool wait_until(unsigned long long limit_ns, Done done) {
  unsigned long long t0 = 0;
  for (long long spin = 0;; ++spin) {
    if (done()) return true;
    if (limit_ns == 0) return false;
    if ((spin & 63) == 63) {
      unsigned long long now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return false;
    }
    __nanosleep(100);
  }
}

constexpr int kStatusTailWait = 6;   // the wait for another block's ids or double-precision scores ran out

// The flagged frames of a call, run by any number of blocks.  `blocks`: how many were launched for it; it sets the size of the
// units only.  One counter hands out the units of both phases, so the first ticket of the second one is also the news that
// every scoring unit has been taken.  (A barrier of all blocks in place of the tickets was as fast with the device to itself: a
// flagged frame of a sixteen-frame call 75 us on top of it either way; all 64 frames of four calls 2,350 us, now 2,236.)
template <typename T>
__device__ __noinline__ void redo_flagged(const CompactParams& p, int blocks, CompactScratch* cs) {
  __shared__ int s_word;
  const ScoreParams& sp = p.sp;
  const int tid = threadIdx.x;
  const int n_fl = *reinterpret_cast<volatile int*>(sp.n_flagged);
  auto next_unit = [&] {
    __syncthreads();                                       // (the last unit is done with what the block shares)
    if (tid == 0) s_word = atomicAdd(p.tail_ctr, 1);
    __syncthreads();
    return s_word;
  };
  // ---- scores in double precision; the block that finishes a frame last selects
  const int heads = sp.Ls * sp.Hq, rs = score64_split(n_fl, heads, sp.P, blocks, sp.scratch_rows), units = heads * rs;
  int w = next_unit();
  for (; w < n_fl * units; w = next_unit()) {
    if (w == 0 && tid == 0) *p.stat_refined += n_fl;
    const int slot = w / units, u = w % units;
    score64_frame_block<T>(sp, p.colsum_d, p.ifft_d, u / rs, u % rs, rs, __ldcg(sp.flagged + slot), slot, &cs->s64);
  }
  // ---- the flagged frames' compaction, plane by plane; two blocks share one by columns while there are enough
  const int parts = n_fl * 4 * p.L <= blocks && p.C * (int)sizeof(T) >= 512 ? 2 : 1;
  const int per = 2 * p.L * parts + (p.patch_split > 0 ? 1 : 0);
  w -= n_fl * units;
  if (w >= n_fl * per) return;
  // every scoring unit has been taken by a block that runs: all selections are made before long
  __syncthreads();
  if (tid == 0) {
    const volatile int* done = sp.n_selected;
    s_word = wait_until(p.wait_ns, [&] { return *done >= n_fl; }) ? 1 : 0;
    __threadfence();
  }
  __syncthreads();
  if (!s_word) {
    if (tid == 0 && sp.status) atomicCAS(sp.status, 0, kStatusTailWait);
    return;
  }
  for (; w < n_fl * per; w = next_unit() - n_fl * units) {
    const int f = __ldcg(sp.flagged + w / per), x = w % per;
    const long long f_abs = p.first_frame + f;
    unsigned char* page = p.store + sp.pages_off + f_abs * sp.page_bytes;
    for (int r = tid; r < p.kappa; r += kCompactThreads) cs->kept[r] = token_id(__ldcg(sp.kept_store + f_abs * p.kappa + r), p.P);
    __syncthreads();
    if (x >= 2 * p.L * parts) pool_patches<T>(p, f, cs);
    else if (parts == 1) compact_plane<T>(p, x, f, cs, p.kappa, page);
    else compact_plane_part<T>(p, x >> 1, f, cs, p.kappa, page, x & 1, 2);
  }
}

// PARTS: two or four blocks share a plane (p.parts).  SELECT: sel_mode 1; else the mode is looked up.  (A kernel for each, so that
// none carries the code of the others: a block's first pass through its code is instruction fetch more than anything else.)
template <typename T, bool PARTS, bool SELECT>
__global__ void __launch_bounds__(kCompactThreads, 3) compact_kernel(const __grid_constant__ CompactParams p) {
  __shared__ CompactScratch cs;
  __shared__ SelectScratch ss;
  const int tid = threadIdx.x;
  const int parts = PARTS ? p.parts : 1, sel_mode = SELECT ? 1 : p.sel_mode;
  // frame is the fast block index: the blocks that start first cover the low planes of every frame,
  // the plane-0 blocks among them
  const int f = blockIdx.x;
  // block row -> plane l*2 + kv; with a patch level its blocks (plane 2L) sit in row 1, so that they run
  // in the first wave beside the copy blocks instead of alone at the end
  int row = blockIdx.y;
  if (p.prev.n_frames > 0) {
    if (row >= 1 && row <= p.prev_rows) {
      // nothing of this call is needed for the entries of the previous one: no wait for the scoring kernel (which has
      // itself waited for the previous call's kernels; without a scoring kernel the wait is here)
      if (sel_mode == 2) pdl_wait();
      const int pl = (row - 1) * gridDim.x + blockIdx.x;
      if (pl < 2 * p.prev.L) compact_segment_plane(p.prev, pl >> 1, pl & 1);
      return;
    }
    if (row > p.prev_rows) row -= p.prev_rows;
  }
  if constexpr (sizeof(T) == 2) {
    const int first = 2 * p.L * parts + (p.patch_split > 0 ? 1 : 0);     // row of the first block for flagged frames
    if (p.redo_blocks > 0 && row >= first) {
      if ((row - first) * gridDim.x + blockIdx.x >= p.redo_blocks) return;
      pdl_wait();
      pdl_trigger();
      // Nothing is flagged any more once every frame's ids are out.  The blocks that publish them are earlier ones of the grid
      // and wait for nobody.
      if (sel_mode == 1) {
        bool ok = true;
        for (int i = tid; i < p.n_frames; i += kCompactThreads) {
          const volatile unsigned* flag = p.sel_flag + i;
          ok = wait_until(p.wait_ns, [&] { return (*flag >> 1) == p.epoch; }) && ok;
        }
        __threadfence();
        if (!__syncthreads_and(ok)) {
          if (tid == 0 && p.sp.status) atomicCAS(p.sp.status, 0, kStatusTailWait);
          return;
        }
      }
      if (*reinterpret_cast<volatile int*>(p.sp.n_flagged) != 0) redo_flagged<T>(p, p.redo_blocks, &cs);
      return;
    }
  }
  const bool patches = p.patch_split > 0 && row == 1;
  if (p.patch_split > 0 && row > 1) --row;
  const int plane = patches ? 2 * p.L : row / parts, part = patches ? 0 : row % parts;
  const bool writes = plane == 0 && part == 0;           // this block writes the ids and the index of its frame
  pdl_wait();
  pdl_trigger();
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid <= kTailWords) *(tid < kTailWords ? p.tail_next + tid : p.n_flagged_next) = 0;
  if (writes)
    for (long long i = (long long)f * kCompactThreads + tid; i < p.n_clear; i += (long long)gridDim.x * kCompactThreads) p.att_clear[i] = 0ull;
  const long long f_abs = p.first_frame + f;
  int kappa_f = p.kappa;
  unsigned char* page = p.store + p.sp.pages_off + f_abs * p.sp.page_bytes;
  bool risky;
  if (sel_mode == 1) {
    __shared__ unsigned s_seen;
    // A block that starts after its frame's plane-0 block has published the ids (the blocks beyond
    // the first wave do) reads them; every other block selects itself.  Nobody waits.
    // (A grid that is resident as a whole has no such blocks, and the look costs a round trip to L2: 0.5 us of a one-frame
    // call of 16.)
    unsigned seen = 0u;
    if (p.later_blocks) {
      if (tid == 0) {
        unsigned v = 0u;
        if (!writes) {
          v = *reinterpret_cast<volatile unsigned*>(p.sel_flag + f);
          __threadfence();
        }
        s_seen = v;
      }
      __syncthreads();
      seen = s_seen;
    }
    if ((seen >> 1) == p.epoch) {
      risky = (seen & 1u) != 0u;
      for (int r = tid; r < p.kappa; r += kCompactThreads) cs.kept[r] = token_id(__ldcg(p.sp.kept_store + f_abs * p.kappa + r), p.P);
      __syncthreads();
    } else {
      risky = select_from_partials(p, f, writes, cs.kept, &ss);
      if (writes) {
        __threadfence();                        // this thread's ids are visible before the flag is
        __syncthreads();
        if (tid == 0) *reinterpret_cast<volatile unsigned*>(p.sel_flag + f) = (p.epoch << 1) | (risky ? 1u : 0u);
      }
    }
  } else if (sel_mode == 2) {
    // Ranking by numbers the caller supplies (no Eq. 1-4): every block ranks its frame itself, in
    // double precision on exact inputs, so nothing is ever too close to call; plane 0 writes the ids.
    const double sx = tid < p.P ? (double)__ldg(p.ext_scores + (long long)f * p.P + tid) : 0.0;
    const bool bad = __syncthreads_or(tid < p.P && !isfinite(sx)) != 0;
    select_by_score(p.sp, f, bad ? 0.0 : sx, writes, cs.kept, ss.sc64, ss.cnt64, ss.misc64);
    if (bad && writes && tid == 0 && p.sp.status) atomicCAS(p.sp.status, 0, kStatusNonFinite);
    risky = false;
    __syncthreads();
  } else if (sel_mode == 3) {
    kappa_f = __ldcg(p.kept_count + f_abs);
    kappa_f = kappa_f < 0 ? 0 : (kappa_f > p.P ? p.P : kappa_f);
    page = p.store + __ldcg(p.sp.page_table + f_abs);
    for (int r = tid; r < kappa_f; r += kCompactThreads) cs.kept[r] = token_id(__ldcg(p.sp.kept_store + f_abs * p.P + r), p.P);
    risky = false;
    __syncthreads();
  } else {
    risky = frame_is_flagged(p.sp.flagged, *p.sp.n_flagged, f);
    for (int r = tid; r < p.kappa; r += kCompactThreads) cs.kept[r] = token_id(p.sp.kept_store[f_abs * p.kappa + r], p.P);
    __syncthreads();
  }
  if (risky) return;
  if (plane >= 2 * p.L) pool_patches<T>(p, f, &cs);
  else if constexpr (PARTS) compact_plane_part<T>(p, plane, f, &cs, kappa_f, page, part, parts);
  else compact_plane<T>(p, plane, f, &cs, kappa_f, page);
}

// Zeros n 64-bit words: what a reset and a call without a workspace start with.  (As a dependent launch it runs beside the start of
// the scoring kernel behind it: 28.1 us for sixteen frames scored without a workspace, 30.2 with a memset in its place.)
__global__ void __launch_bounds__(kCompactThreads) zero_kernel(unsigned long long* p, int n) {
  pdl_wait();
  pdl_trigger();
  for (int i = blockIdx.x * kCompactThreads + threadIdx.x; i < n; i += gridDim.x * kCompactThreads) p[i] = 0ull;
}

// Selection alone (scoring without a store, bf16): one block per frame, behind the persistent scoring kernel; the blocks behind
// those score the flagged frames again in double precision, once every frame's selection is out (a launch of its own for that cost
// calls that flag nothing 0.4 us of 31).  A code in *scoring (one of that kernel's bounded waits ran out) leaves no sums to trust:
// the ids are then -1 and the scores NaN.
// Nor does a block that waits too long for a frame leave ids that single precision could not decide: it gives the frame up, in
// the word that the frame's own block would publish in, and whoever finds that word so, all blocks behind the selection and the
// frame's own one, takes back what is not final: that frame, and the flagged ones.  (Either every one of these blocks
// finds all frames published, or none does.)
// Two blocks per SM: with three, 80 registers a thread, the double-precision scores spilled twice as much as in the compaction
// kernel for what the ways out take, and a call with a flagged frame 83.4 us; with two and none spilled 77.5, two flagged frames 94.0
// (106.8), eight 268 (369), sixteen 502 (587), nothing flagged 27.1 (27.8).  (Where the units of fewer blocks come out badly: three
// 131 (119), six 268 (219), eleven 501 (370); one or two are what a call of sixteen frames sees, a quarter of the time.)
constexpr unsigned kSelDone = 1u, kSelGivenUp = 2u, kSelRisky = 3u;
__global__ void __launch_bounds__(kCompactThreads, 2) select_kernel(const __grid_constant__ CompactParams p, const int* scoring) {
  __shared__ union {
    struct {
      SelectScratch ss;
      int kept[MUKV_MAX_TOKENS];
    };
    Score64Scratch s64;
  } sh;
  __shared__ unsigned s_word;
  const ScoreParams& sp = p.sp;
  const int n = sp.n_frames, tid = threadIdx.x;
  pdl_wait();
  pdl_trigger();
  const int failed = *scoring;
  int f0 = 0, f1 = 0;                                      // frames to take back: all of these, or
  bool only_risky = false;                                 // those that need the double-precision pass
  if ((int)blockIdx.x < n) {
    const int f = blockIdx.x;
    const bool risky = select_from_partials(p, f, true, sh.kept, &sh.ss);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_word = atomicCAS(p.sel_flag + f, 0u, risky ? kSelRisky : kSelDone);
    __syncthreads();
    if (!failed && s_word != kSelGivenUp) return;
    f0 = f;
    f1 = f + 1;
  } else {
    if (failed) return;
    unsigned word = kSelDone;
    if (tid < n) {                                         // (n <= MUKV_NOALLOC_MAX_FRAMES)
      const volatile unsigned* flag = p.sel_flag + tid;
      if (!wait_until(p.wait_ns, [&] { return (word = *flag) != 0u; })) {
        word = atomicCAS(p.sel_flag + tid, 0u, kSelGivenUp);
        if (word == 0u) word = kSelGivenUp;
      }
    }
    __threadfence();
    if (!__syncthreads_or(word == kSelGivenUp)) {
      const int n_fl = *reinterpret_cast<volatile int*>(sp.n_flagged), blocks = gridDim.x - n, heads = sp.Ls * sp.Hq;
      if (n_fl == 0) return;
      const int rs = score64_split(n_fl, heads, sp.P, blocks, sp.scratch_rows), units = heads * rs;
      for (int w = blockIdx.x - n; w < n_fl * units; w += blocks) {
        const int slot = w / units, u = w % units;
        score64_frame_block<__nv_bfloat16>(sp, p.colsum_d, p.ifft_d, u / rs, u % rs, rs, __ldcg(sp.flagged + slot), slot, &sh.s64);
        __syncthreads();
      }
      return;
    }
    f1 = n;
    only_risky = true;
  }
  const long long np = (long long)n * sp.P;
  for (int f = f0; f < f1; ++f) {
    if (only_risky && *reinterpret_cast<volatile unsigned*>(p.sel_flag + f) != kSelRisky) continue;   // (no word changes any more)
    for (int t = tid; t < sp.P; t += kCompactThreads) {
      if (t < sp.kappa) sp.kept_store[(long long)f * sp.kappa + t] = -1;
      for (int s = 0; s < 3 && sp.scores_out; ++s) sp.scores_out[s * np + (long long)f * sp.P + t] = __int_as_float(0x7fffffff);
    }
  }
}

// segment_kernel: one block per (layer, K|V) plane writes that plane of every segment entry the frames
// first_frame .. first_frame + n_frames - 1 touch.  Launched for the chunk of an earlier call when something is about to
// read its segment entries.
__global__ void __launch_bounds__(kCompactThreads) segment_kernel(const CompactParams p) {
  pdl_wait();
  pdl_trigger();
  for (int plane = blockIdx.x; plane < 2 * p.L; plane += gridDim.x)
    compact_segment_plane(segment_args(p), plane >> 1, plane & 1);
}

// The flagged frames as a launch of their own.
template <typename T>
__global__ void __launch_bounds__(kCompactThreads, 3) tail_kernel(const __grid_constant__ CompactParams p) {
  __shared__ CompactScratch cs;
  pdl_trigger();                                // the next call's scoring kernel may be scheduled (it waits for this one itself)
  pdl_wait();
  if (*p.sp.n_flagged == 0) return;             // the common case
  redo_flagged<T>(p, gridDim.x, &cs);
}

}  // namespace mukv
