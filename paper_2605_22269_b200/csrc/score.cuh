// Per-frame token scoring and selection (Sec. 3.3, Eq. 1-4 and the top-kappa rule).
//
// score_kernel<T, NC>: one thread block per (query head h, frame f), single precision on the multiply-add units (fp32 calls
// that the tensor cores do not hold; MUKV_OPT_SCORE_PATH 1).  The double-precision pass is in score64.cuh.
//   * Eq. 1: S = Q_h K_g^T / sqrt(D) over the frame's P tokens, row softmax, column sums.
//     Lanes own key columns (j = lane + 32c), a warp walks the query rows four at a time, so
//     the column sums stay in registers and only the row maximum / row sum cross lanes.
//     The attention matrix is never written anywhere.
//   * Eq. 2-3: the G query-head blocks that share key head g split that head's tokens and
//     transform each key vector along the feature axis; sum of the D bin magnitudes per token.
//   * The block that finishes a frame last (arrival counter, nobody waits) reduces the
//     per-head partials in a fixed order, applies Eq. 4 and selects the kappa tokens.
// T is the input element type.
#pragma once
#include "common.cuh"

namespace mukv {

constexpr int kScoreThreads = 256;
constexpr int kStatusNonFinite = 7;   // a frame's scores were not finite: its lowest kappa ids were kept
constexpr int kScoreWarps = kScoreThreads / 32;
constexpr int kRowsPerStep = 4;

struct ScoreParams {
  int P, Hq, Hkv, D, G, kappa;
  int Ls;                       // scoring layers (Eq. 1-3 are averaged over them); >= 1
  long long q_layer_stride;     // elements between the queries of two scoring layers (n * P * Hq * D)
  long long k_layer_stride;     // elements between the keys of two layers (n * P * Hkv * D)
  int n_frames;                 // frames in this chunk
  int causal, keep_low;
  float alpha, tie_eps, flag_margin, flat_ratio;
  long long first_frame;
  // inputs
  const void* q;                // [Ls][n][P][Hq][D]
  const void* k_last;           // [Ls][n][P][Hkv][D]  (the scoring layers of K; by default the last layer)
  // scratch
  void* colsum_part;            // A [F][Ls * Hq * row_split][P]
  void* ifft_part;              // A [F][Ls * Hkv][P]
  int* frame_counter;           // [F], zero between launches
  int* head_counter;            // [places][heads], too: see finish_frame
  int* flagged;                 // [F] frame slots needing the double pass
  int* n_flagged;               // count (written by the float pass, read by the double pass)
  // outputs
  int* kept_store;              // [max_frames][kappa]
  int* kept_out;                // [n][kappa] or null
  float* scores_out;            // [3][n][P] or null
  long long* frame_ts;          // [max_frames]
  long long* page_table;        // [max_frames]
  long long pages_off, page_bytes;
  int* n_selected;              // double-precision pass: counts the frames it has selected; or null
  int* status;                  // device event word (0 = nothing recorded); see mukv_stats.device_status
  // cached keys the queries also attend to (Sec. 3.2): the kept keys of the n_past_frames frames stored
  // just before the chunk, kappa rows each, read from their pages; n_past_frames = 0: none
  int n_past_frames;
  long long past_first;         // absolute index of the first of those frames
  int first_score_layer;        // layer of the model the first scoring layer is
  const unsigned char* store;   // store base (page_table holds byte offsets from it)
  int no_select;                // 1: only the partial sums are wanted (the selection runs over a whole segment elsewhere)
  int refine;                   // 1: frames come from the flagged list, no further flagging
  int row_split;                // blocks that share a query head, each a range of query rows (>= 1)
  int scratch_rows;             // double-precision pass over flagged frames: rows of P doubles that colsum_part has room for
                                // (see score64_split; a flagged frame's place is its place in the list)
  // segment-level selection, double-precision pass: only the frames of segments whose word is non-zero
  // are scored (segment of chunk frame f: f / gate_fseg); null: every frame
  const int* seg_gate;
  int gate_fseg;
};

struct FinishScratch {
  double part[kScoreWarps][256];
  double sc[256];
  double misc[64];
  int ints[64];
};

template <typename T>
__host__ __device__ constexpr int score_row_stride(int D) { return D + ElemTraits<T>::kPad; }

// P: key rows held in shared memory (the frame's tokens plus the past keys)
template <typename T>
__host__ inline size_t score_smem_bytes(int P, int D) {
  typedef float A;
  size_t ks = (size_t)P * score_row_stride<T>(D) * sizeof(T);
  size_t qs = (size_t)kScoreWarps * kRowsPerStep * D * sizeof(T);
  size_t tw = (size_t)D * 2 * sizeof(A);
  size_t red = (size_t)kScoreWarps * 256 * sizeof(A);
  const size_t all = ((ks + 15) / 16) * 16 + qs + tw + red;
  return (all > sizeof(FinishScratch) ? all : sizeof(FinishScratch)) + 64;
}

// The top-kappa rule for one frame on final scores (double), run by a whole block; thread t < P owns token t and gives its score s
// (P <= threads).  tau is the kappa-th largest score (rank counting); scores above tau + tie_eps are kept, the scores
// within tie_eps of tau share the remaining places by lowest token id.  Returns whether the thread's token stays; the kept ids go,
// ascending, to s_kept (shared memory, may be null) and, with `write`, to the store, to the caller's output and the frame's time
// stamp and page-table entry are set.
// s_sc (P doubles), s_int (one int per warp + 1), s_misc (4 doubles per warp) are shared scratch.
__device__ inline bool select_by_score(const ScoreParams& p, int f, double s, bool write, int* s_kept, double* s_sc, int* s_int,
                                       double* s_misc) {
  const int tid = threadIdx.x, P = p.P, kappa = p.kappa;
  const bool valid = tid < P;
  // (on order-preserving integers: a comparison of doubles takes sixteen clocks of a scheduler)
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(s_sc);
  const unsigned long long key = order_key(s);
  if (valid) s_key[tid] = key;
  __syncthreads();
  if (valid) {
    int gt = 0, ge = 0;
#pragma unroll 4
    for (int i = 0; i < P; ++i) {
      const unsigned long long o = s_key[i];
      gt += (o > key);
      ge += (o >= key);
    }
    if (gt < kappa && kappa <= ge) s_misc[0] = s;           // every writer holds the same value
  }
  __syncthreads();
  const double tau = s_misc[0];
  const double delta = (double)p.tie_eps;
  const bool sure = valid && (s > tau + delta);
  const bool band = valid && !sure && (s >= tau - delta);
  int n_sure, n_band, n_kept;
  block_excl_count(sure, s_int, n_sure);
  const int band_rank = block_excl_count(band, s_int, n_band);
  const bool keep = sure || (band && band_rank < kappa - n_sure);
  const long long f_abs = p.first_frame + f;
  const int pos = block_excl_count(keep, s_int, n_kept);
  if (keep) {
    if (s_kept) s_kept[pos] = tid;
    if (write) {
      p.kept_store[f_abs * kappa + pos] = tid;
      if (p.kept_out) p.kept_out[(long long)f * kappa + pos] = tid;
    }
  }
  if (write && tid == 0) {
    p.frame_ts[f_abs] = f_abs;
    p.page_table[f_abs] = p.pages_off + f_abs * p.page_bytes;
  }
  return keep;
}

// Eq. 4 and the top-kappa rule for one frame, run by a whole block; thread t < P owns token t, att_raw / fft_raw are its I_att and
// I_fft; s_sc (P doubles), s_int (one int per warp + 1), s_misc (4 doubles per warp) are shared scratch.
// With `refined` the frame is not put on the flagged list however close it is.
// The arithmetic here is always double: it is a few hundred operations per frame and keeps
// the normalisation from adding rounding noise of its own to the scores.
__device__ inline void select_frame(const ScoreParams& p, int f, double att_raw, double fft_raw, bool refined, double* s_sc, int* s_int,
                                    double* s_misc) {
  typedef double A;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = (int)blockDim.x >> 5;
  const int P = p.P;
  const bool valid = tid < P;
  const A big = (A)3.0e38;
  // ---- a frame with a score that is not a number has no ranking: every score counts as 0 below,
  // so that the lowest kappa ids are kept, and the event is recorded
  int n_bad;
  block_excl_count(valid && !(isfinite(att_raw) && isfinite(fft_raw)), s_int, n_bad);
  const bool bad = n_bad != 0;
  // ---- min / max of both signals over the frame
  A v[4] = {big, -big, big, -big};
  if (valid) {
    v[0] = att_raw < v[0] ? att_raw : v[0];
    v[1] = att_raw > v[1] ? att_raw : v[1];
    v[2] = fft_raw < v[2] ? fft_raw : v[2];
    v[3] = fft_raw > v[3] ? fft_raw : v[3];
  }
  v[0] = warp_min(v[0]); v[1] = warp_max(v[1]); v[2] = warp_min(v[2]); v[3] = warp_max(v[3]);
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) s_misc[warp * 4 + i] = v[i];
  }
  __syncthreads();
  A amin = big, amax = -big, fmin_ = big, fmax_ = -big;
  for (int w = 0; w < nwarp; ++w) {
    amin = s_misc[w * 4 + 0] < amin ? s_misc[w * 4 + 0] : amin;
    amax = s_misc[w * 4 + 1] > amax ? s_misc[w * 4 + 1] : amax;
    fmin_ = s_misc[w * 4 + 2] < fmin_ ? s_misc[w * 4 + 2] : fmin_;
    fmax_ = s_misc[w * 4 + 3] > fmax_ ? s_misc[w * 4 + 3] : fmax_;
  }
  __syncthreads();
  // ---- Eq. 4
  const A alpha = (A)p.alpha;
  const A an = (amax == amin) ? (A)0 : (att_raw - amin) / (amax - amin);
  A fn = (fmax_ == fmin_) ? (A)0 : (fft_raw - fmin_) / (fmax_ - fmin_);
  if (p.keep_low) fn = (A)1 - fn;
  const A s = bad ? (A)0 : alpha * an + ((A)1 - alpha) * fn;
  const bool keep = select_by_score(p, f, s, true, nullptr, s_sc, s_int, s_misc);
  if (p.scores_out && valid) {
    const long long np = (long long)p.n_frames * P;
    p.scores_out[0 * np + (long long)f * P + tid] = (float)att_raw;
    p.scores_out[1 * np + (long long)f * P + tid] = (float)fft_raw;
    p.scores_out[2 * np + (long long)f * P + tid] = (float)s;
  }
  if (tid == 0 && bad && p.status) atomicCAS(p.status, 0, kStatusNonFinite);
  // ---- does single precision decide this frame safely?
  // With a = lowest kept score and b = highest dropped score, the kept set is the same for every
  // perturbation of the scores below flag_margin / 2 as long as a - b > tie_eps + flag_margin: no
  // dropped token can then enter the tie band of the kappa-th score.  Anything closer is redone
  // in double precision.
  if (!refined && !bad) {
    const int kappa = p.kappa;
    const A delta = (A)p.tie_eps;
    A a = valid && keep ? s : big, b = valid && !keep ? s : -big;
    a = warp_min(a);
    b = warp_max(b);
    __syncthreads();
    if (lane == 0) { s_misc[warp * 4] = a; s_misc[warp * 4 + 1] = b; }
    __syncthreads();
    if (tid == 0) {
      for (int w = 1; w < nwarp; ++w) {
        a = s_misc[w * 4] < a ? s_misc[w * 4] : a;
        b = s_misc[w * 4 + 1] > b ? s_misc[w * 4 + 1] : b;
      }
      bool risky = (kappa < P) && (a - b <= delta + (A)p.flag_margin);
      // a nearly flat signal amplifies rounding noise through the min-max division
      const A fr = (A)p.flat_ratio;
      const A aabs = amax > -amin ? amax : -amin, fabs_ = fmax_ > -fmin_ ? fmax_ : -fmin_;
      if (amax != amin && (amax - amin) < fr * aabs && p.alpha != 0.f) risky = true;
      if (fmax_ != fmin_ && (fmax_ - fmin_) < fr * fabs_ && p.alpha != 1.f) risky = true;
      if (risky) {
        const int slot = atomicAdd(p.n_flagged, 1);
        p.flagged[slot] = f;
      }
    }
  }
}

// Sums over n rows of P values (`stride` rows apart), rows in order inside an eighth, then the eighths in order: thread t < P of a
// block of kScoreThreads gets column t.  A warp takes an eighth of the rows, a lane of it every 32nd column: all loads of a
// thread are independent (one thread per column walks n round trips to L2: 6 us for 112 rows).  part: [kScoreWarps][256].
template <typename A>
__device__ __noinline__ double column_sums(const A* rows, int n, int stride, int P, double (*part)[256]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (n + kScoreWarps - 1) / kScoreWarps, r0 = min(n, warp * per), r1 = min(n, r0 + per);
#pragma unroll 1
  for (int c0 = lane; c0 < P; c0 += 64) {                  // two columns at a time, eight rows in flight
    double t0 = 0.0, t1 = 0.0;
    const bool two = c0 + 32 < P;
    for (int r = r0; r < r1; r += 8) {
      A x0[8], x1[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        x0[i] = r + i < r1 ? __ldcg(rows + (long long)(r + i) * stride * P + c0) : (A)0;
        x1[i] = two && r + i < r1 ? __ldcg(rows + (long long)(r + i) * stride * P + c0 + 32) : (A)0;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) { t0 += (double)x0[i]; t1 += (double)x1[i]; }
    }
    part[warp][c0] = t0;
    if (two) part[warp][c0 + 32] = t1;
  }
  __syncthreads();
  double t = 0.0;
  if (tid < P)
    for (int w = 0; w < kScoreWarps; ++w) t += part[w][tid];
  __syncthreads();
  return t;
}

// true in every thread of the block that arrives last of n at *ctr, which is then zero again; what the others wrote before
// is visible to it
__device__ inline bool arrives_last(int* ctr, int n, int* s_flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const int old = atomicAdd(ctr, 1);
    *s_flag = old == n - 1;
    if (old == n - 1) *ctr = 0;                            // ready for the next launch
  }
  __syncthreads();
  const bool last = *s_flag != 0;
  if (last) __threadfence();
  __syncthreads();
  return last;
}

// Every block that has written its share of a frame's partial sums (column sums [heads][RS][P] and frequency sums [key
// heads][P], at place sf) calls this.  The last block of a head adds up its parts (in the row of the first; 392 rows of a frame
// split over the device took one block 15 us), the last one of the frame finishes Eq. 1 / Eq. 3 and selects.  Run by a whole
// block.  refined: the selection is final (see select_frame).
template <typename A>
__device__ inline void finish_frame(const ScoreParams& p, A* colsum, const A* ifft, int f, int sf, int hv, int RS, bool refined,
                                    FinishScratch* s) {
  if (p.no_select) return;
  const int tid = threadIdx.x, P = p.P, HqV = p.Ls * p.Hq, HkvV = p.Ls * p.Hkv;
  A* rows = colsum + (long long)sf * HqV * RS * P;
  if (RS > 1) {
    if (!arrives_last(p.head_counter + sf * HqV + hv, RS, s->ints)) return;
    const double t = column_sums(rows + (long long)hv * RS * P, RS, 1, P, s->part);
    if (tid < P) rows[(long long)hv * RS * P + tid] = (A)t;
  }
  if (!arrives_last(p.frame_counter + f, HqV, s->ints)) return;
  const double att = column_sums(rows, HqV, RS, P, s->part) / (double)((long long)HqV * P);
  const double fft = column_sums(ifft + (long long)sf * HkvV * P, HkvV, 1, P, s->part) / (double)((long long)HkvV * p.D);
  select_frame(p, f, att, fft, refined, s->sc, s->ints, s->misc);
  if (p.n_selected) {
    __threadfence();                                       // this thread's ids are visible before the frame counts
    __syncthreads();
    if (tid == 0) atomicAdd(p.n_selected, 1);
  }
}

// The work of one block: query head hv of frame f (a frame slot of the chunk); hv counts the query heads of all scoring
// layers, layer-major.
template <typename T, int NC>
__device__ __forceinline__ void score_frame_block(const ScoreParams& p, int hv, int f, unsigned char* smem_raw) {
  typedef float A;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int P = p.P, D = p.D, Hq = p.Hq, Hkv = p.Hkv, G = p.G;
  const int layer = hv / Hq, h = hv - layer * Hq;
  const int HqV = p.Ls * Hq, HkvV = p.Ls * Hkv;
  const int g = h / G;
  constexpr int EPW = ElemTraits<T>::kPerWord;
  const int DS = score_row_stride<T>(D);
  const int WS = DS / EPW;                         // words per padded K row
  const int DW = D / EPW;                          // words per vector

  // key rows: the past keys first, then the frame's own tokens
  const int n_past = p.n_past_frames * p.kappa, Pk = n_past + P;

  // ---- shared memory carve-up
  size_t off = 0;
  T* Ks = reinterpret_cast<T*>(smem_raw);
  off = (((size_t)Pk * DS * sizeof(T)) + 15) / 16 * 16;
  T* Qs = reinterpret_cast<T*>(smem_raw + off);
  off += (size_t)kScoreWarps * kRowsPerStep * D * sizeof(T);
  A* tw = reinterpret_cast<A*>(smem_raw + off);
  off += (size_t)D * 2 * sizeof(A);
  A* red = reinterpret_cast<A*>(smem_raw + off);
  FinishScratch* fin = reinterpret_cast<FinishScratch*>(smem_raw);   // (in the place of the keys, when all is done with them)

  // ---- stage K_g of this frame (rows padded so that 32 consecutive rows hit 32 banks)
  const T* Kg = reinterpret_cast<const T*>(p.k_last) + layer * p.k_layer_stride + ((long long)f * P * Hkv + g) * D;
  {
    constexpr int VE = 16 / sizeof(T);             // elements per 16-byte vector
    const int vec_per_row = D / VE;
    for (int v = tid; v < n_past * vec_per_row; v += kScoreThreads) {
      // row r of the past: kept row r % kappa of frame past_first + r / kappa, this layer's K plane of its page
      const int r = v / vec_per_row, c = v % vec_per_row;
      const long long t = p.past_first + r / p.kappa;
      const T* page = reinterpret_cast<const T*>(p.store + p.page_table[t]);
      const T* src = page + ((long long)(p.first_score_layer + layer) * 2 * p.kappa + r % p.kappa) * Hkv * D + g * D;
      const uint4 x = *reinterpret_cast<const uint4*>(src + c * VE);
      uint32_t* dst = reinterpret_cast<uint32_t*>(Ks + (size_t)r * DS + c * VE);
      dst[0] = x.x; dst[1] = x.y; dst[2] = x.z; dst[3] = x.w;
    }
    for (int v = tid; v < P * vec_per_row; v += kScoreThreads) {
      const int j = v / vec_per_row, c = v % vec_per_row;
      const uint4 x = *reinterpret_cast<const uint4*>(Kg + (long long)j * Hkv * D + c * VE);
      uint32_t* dst = reinterpret_cast<uint32_t*>(Ks + (size_t)(n_past + j) * DS + c * VE);
      dst[0] = x.x; dst[1] = x.y; dst[2] = x.z; dst[3] = x.w;
    }
    for (int d = tid; d < D; d += kScoreThreads) {
      double sn, cs;
      sincospi(2.0 * (double)d / (double)D, &sn, &cs);
      tw[2 * d] = (A)cs;
      tw[2 * d + 1] = (A)sn;
    }
  }
  __syncthreads();

  // ---- Eq. 1: column sums of the row softmax
  const uint32_t* Kw = reinterpret_cast<const uint32_t*>(Ks);
  uint32_t* Qw = reinterpret_cast<uint32_t*>(Qs) + (size_t)warp * kRowsPerStep * DW;
  const T* Qh = reinterpret_cast<const T*>(p.q) + layer * p.q_layer_stride + ((long long)f * P * Hq + h) * D;
  // 1/sqrt(D) as a two-term constant, so that single precision scales the logits without a
  // systematic relative error shared by every element
  const double scale_d = 1.0 / sqrt((double)D);
  const A scale = (A)scale_d;
  const A scale_lo = (A)(scale_d - (double)scale);
  A csum[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) csum[c] = (A)0;
  int jrow[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) jrow[c] = min(lane + 32 * c, Pk - 1) * WS;

  const int n_steps = (P + kRowsPerStep - 1) / kRowsPerStep;
  for (int rb = warp; rb < n_steps; rb += kScoreWarps) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kRowsPerStep; ++r) {
      const int i = rb * kRowsPerStep + r;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(Qh + (long long)min(i, P - 1) * Hq * D);
      for (int w = lane; w < DW; w += 32) Qw[r * DW + w] = (i < P) ? __ldg(src + w) : 0u;
    }
    __syncwarp();
    A acc[kRowsPerStep][NC];
#pragma unroll
    for (int r = 0; r < kRowsPerStep; ++r)
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[r][c] = (A)0;
#pragma unroll 2
    for (int w = 0; w < DW; ++w) {
      uint32_t qw[kRowsPerStep];
#pragma unroll
      for (int r = 0; r < kRowsPerStep; ++r) qw[r] = Qw[r * DW + w];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const uint32_t kw = Kw[jrow[c] + w];
#pragma unroll
        for (int r = 0; r < kRowsPerStep; ++r) acc[r][c] = dot_word<T>(qw[r], kw, acc[r][c]);
      }
    }
#pragma unroll
    for (int r = 0; r < kRowsPerStep; ++r) {
      const int i = rb * kRowsPerStep + r;
      A z[NC];
      A m = -INFINITY;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int j = lane + 32 * c;                     // past keys are visible to every query
        const bool ok = (j < Pk) && (!p.causal || j - n_past <= i);
        z[c] = ok ? fmaf(acc[r][c], scale, acc[r][c] * scale_lo) : -INFINITY;
        m = z[c] > m ? z[c] : m;
      }
      m = warp_max(m);
      A l = (A)0;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        z[c] = (z[c] == -INFINITY) ? (A)0 : expf(z[c] - m);
        l += z[c];
      }
      l = warp_sum(l);
      const A inv = (i < P) ? (A)1 / l : (A)0;
#pragma unroll
      for (int c = 0; c < NC; ++c) csum[c] += z[c] * inv;
    }
  }
  // cross-warp reduction in a fixed order
#pragma unroll
  for (int c = 0; c < NC; ++c) red[warp * 256 + lane + 32 * c] = csum[c];
  __syncthreads();
  if (tid < P) {                                       // the importance is that of the frame's own tokens
    A t = (A)0;
    for (int w = 0; w < kScoreWarps; ++w) t += red[w * 256 + n_past + tid];
    reinterpret_cast<A*>(p.colsum_part)[((long long)f * HqV + hv) * P + tid] = t;
  }

  // ---- Eq. 2-3: sum over the D bins of |DFT(k_j)| for this block's share of head g's tokens
  {
    const int hg = h % G;                            // the G blocks that hold key head g share its tokens
    const int half = D / 2;
    for (int j = hg + warp * G; j < P; j += kScoreWarps * G) {
      const T* kr = Ks + (size_t)(n_past + j) * DS;
      A total = (A)0;
      // bins 1 .. D/2-1 (twice, by conjugate symmetry) and bin 0
      for (int b = lane; b < half; b += 32) {
        A re = (A)0, im = (A)0;
        for (int d = 0; d < D; ++d) {
          const A x = (A)elem_to_float<T>(kr[d]);
          const int m = (b * d) & (D - 1);
          re += x * tw[2 * m];
          im -= x * tw[2 * m + 1];
        }
        const A mag = sqrtf(re * re + im * im);
        total += (b == 0) ? mag : (A)2 * mag;
      }
      // bin D/2: alternating sum
      A alt = (A)0;
      for (int d = lane; d < D; d += 32) {
        const A x = (A)elem_to_float<T>(kr[d]);
        alt += (d & 1) ? -x : x;
      }
      total = warp_sum(total);
      alt = warp_sum(alt);
      if (lane == 0)
        reinterpret_cast<A*>(p.ifft_part)[((long long)f * HkvV + layer * Hkv + g) * P + j] = total + (alt < (A)0 ? -alt : alt);
    }
  }

  finish_frame(p, reinterpret_cast<A*>(p.colsum_part), reinterpret_cast<const A*>(p.ifft_part), f, f, hv, 1, false, fin);
}

// Grid (query heads of all scoring layers, frames).
template <typename T, int NC>
__global__ void __launch_bounds__(kScoreThreads) score_kernel(const ScoreParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  pdl_trigger();
  score_frame_block<T, NC>(p, blockIdx.x, blockIdx.y, smem_raw);
}

}  // namespace mukv
