// Semi-hierarchical retrieval (Sec. 3.4, Eq. 6-8) and the gather of the retrieved context
// (Sec. 3.5, Eq. 9).
//
// All ranking arithmetic is double precision: the work is a few hundred MFLOP per batch of
// questions, tiny next to the gather, and it makes the selected indices independent of
// summation order.  Kernels:
//   qpool_kernel    Eq. 6   one block per (question, key head)
//   scan_kernel     Eq. 7   cosine of every question with every frame, segment and patch-level key (a skinny
//                           double-precision product on the fp64 tensor-core instruction)
//   scan_few_kernel         the same for at most eight questions on not too many rows, a warp per row or two
//   rank_kernel     stage-1 candidates, Eq. 8 rerank, final top-k; per question a cluster of blocks, one for each granularity
//   gather_kernel   Eq. 9   copies the selected pages into the per-question decode buffers
//   gather3_kernel          the same with summary tokens and the rows of patch-level blocks
#pragma once
#include "common.cuh"
#include "tc.cuh"

namespace mukv {

struct QMeta {
  int off[MUKV_MAX_QUESTIONS + 1];
  long long t_limit[MUKV_MAX_QUESTIONS];
};

// ------------------------------------------------------------------------------ Eq. 6
// One block per (question, key head).  Thread (slice, vector) sums one 16-byte vector of the head's
// channels over the tokens n = slice, slice + slices, ... and the G query heads of the group: every
// load is a full 16-byte vector and all of a thread's loads are independent.  The slices are added
// in a fixed order.  Channel c of question i is written to q64[c * cs + i * qs]: transposed (qs = 1) for
// scan_kernel, which stages it, a row per question (cs = 1) for scan_few_kernel; the head's share of the squared
// norm goes to qn2[question][key head] (the scans add the shares in head order).
constexpr int kPoolThreads = 512;
constexpr int kScanFew = 8;        // questions that scan_few_kernel takes at the most, see scan_by_rows
constexpr int kPoolSmemDoubles = 4096;

template <typename T>
__global__ void __launch_bounds__(kPoolThreads) qpool_kernel(const T* __restrict__ qtok, const QMeta meta, int Hq,
                                                             int Hkv, int D, double* __restrict__ q64, int cs, int qs,
                                                             double* __restrict__ qn2, int early) {
  constexpr int VE = 16 / sizeof(T);
  __shared__ double s_acc[kPoolSmemDoubles];
  __shared__ double s_part[kPoolThreads / 32];
  const int qi = blockIdx.x, g = blockIdx.y;
  const int G = Hq / Hkv;
  pdl_wait();
  // (In front of scan_few_kernel only, whose small blocks are all resident: those of scan_kernel pile up on the SMs that this kernel
  // leaves free.  With the trigger 8 questions on 11,475 rows of 512 channels took 36.0 us, without it 31.8; 48 on 107 rows 46.1
  // and 33.4; 9 to 24 on up to 11,475 rows the same within 0.3.)
  if (early) pdl_trigger();
  const int n0 = meta.off[qi], n1 = meta.off[qi + 1];
  const int DV = D / VE;                                    // vectors per head
  int nsl = kPoolThreads / DV;                              // token slices whose partial sums fit
  if (nsl > kPoolSmemDoubles / D) nsl = kPoolSmemDoubles / D;
  const int sl = threadIdx.x / DV, dv = threadIdx.x % DV;
  if (sl < nsl) {
    double tot[VE];
#pragma unroll
    for (int e = 0; e < VE; ++e) tot[e] = 0.0;
    for (int n = n0 + sl; n < n1; n += nsl) {
      const T* row = qtok + ((long long)n * Hq + (long long)g * G) * D + dv * VE;
#pragma unroll 1
      for (int j0 = 0; j0 < G; j0 += 8) {
        uint4 x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          x[j] = j0 + j < G ? *reinterpret_cast<const uint4*>(row + (long long)(j0 + j) * D) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t w[4] = {x[j].x, x[j].y, x[j].z, x[j].w};
          if constexpr (sizeof(T) == 2) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { tot[2 * i] += (double)bf16_lo(w[i]); tot[2 * i + 1] += (double)bf16_hi(w[i]); }
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) tot[i] += (double)__uint_as_float(w[i]);
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) s_acc[sl * D + dv * VE + e] = tot[e];
  }
  __syncthreads();
  double sq = 0.0;
  for (int col = threadIdx.x; col < D; col += kPoolThreads) {
    double t = 0.0;
    for (int k = 0; k < nsl; ++k) t += s_acc[k * D + col];
    t = t / (double)((long long)(n1 - n0) * G);
    q64[(long long)(g * D + col) * cs + (long long)qi * qs] = t;
    sq += t * t;
  }
  sq = warp_sum(sq);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kPoolThreads / 32; ++w) t += s_part[w];
    qn2[(long long)qi * Hkv + g] = t;
  }
}

// ------------------------------------------------------------------------------ Eq. 7
// Rows 0..n_frm-1 are frame keys, rows n_frm..n_frm+n_seg-1 segment keys, then n_pat patch-level
// keys (n_pat = 0 without a patch level).  The product [rows x C] . [C x questions] runs on the double-precision tensor-core
// instruction (mma.sync m8n8k4 f64; the scores have to be double because indices are ranked on them): a block owns
// row_tiles x 8 rows and all questions, a warp eight rows and T tiles of eight questions.  It walks the feature axis in
// chunks of 32 channels, the next chunk of the rows (float) and of the pooled questions (double) on its way to shared memory while
// one is multiplied.
// Bound by the fp64 tensor instruction, 64 multiply-adds per clock and SM: 21 us for 64 questions and the 11,475 rows of three
// hours.  scan_shape() picks the tiles so that all SMs get about the same share of them.  From launch to end, in the chain of
// dependent launches behind the pooling of the questions: 53 us with fixed blocks of 32 rows x 64 questions for that case, now 42;
// 1,913 rows (60 blocks for 148 SMs, which went in twos to what the pooling had left free; alone on the device both take 23)
// 51, now 26; 24 questions, padded to 64 then, and 5,313 rows 46, now 24.
constexpr int kScanCC = 32;                                  // channels of a chunk (C is a multiple of it)
constexpr int kScanRowPad = kScanCC + 4;                     // floats of a row, doubles of a question row: + 4 keeps the
constexpr int kScanQPad = 4;                                 // fragments' loads on different banks
constexpr int kScanMaxWarps = 20;

struct ScanShape {
  int T, q_groups, row_tiles;                                // tiles of a warp; warps side by side: question groups x row tiles
  size_t smem;
};
__host__ inline size_t scan_smem_bytes(int T, int q_groups, int row_tiles) {
  return 2 * ((size_t)kScanCC * (8 * T * q_groups + kScanQPad) * sizeof(double) + (size_t)8 * row_tiles * kScanRowPad * sizeof(float));
}
// The shape of least time, in clocks per chunk.  A wave of blocks takes what its warps take on the busiest scheduler (128 clocks a
// tile, 8 instructions of 16, and 40 for the rows' operands, which the tiles of a warp share) or its bytes at 32 a clock, the chunk's
// barrier and first operands (400) and the copies that one thread issues (50 each: a block of few warps is slow at fetching the
// chunk of all questions); then the bytes of all blocks, at 8,000 a clock of the device.  Blocks per SM as shared memory and
// registers (48 a thread for T = 1, up to 96 else) allow.
// Fitted to every shape at 1 to 8 KB per pooled question, 9 to 128 questions and 107 to 44,625 rows, keys in L2 and not: 0.7 % from the
// best one on average, 9 % at the most.  (Without residency, copies and the last term 5 % and 70 %: 128 questions on 8,288 rows
// went to 1,036 blocks of one row tile, each of which fetches all questions, 199 us; now 148.)
__host__ inline ScanShape scan_shape(long long rows, int nq, int n_sms) {
  const int nt = (nq + 7) / 8, tiles = (int)((rows + 7) / 8);      // (32-bit divisions: half a microsecond of the call)
  ScanShape best{0, 0, 0, 0};
  long long least = -1;
  for (int T = 1; T <= 8; T *= 2) {
    const int qg = (nt + T - 1) / T;
    if (qg > 4) continue;
    for (int rt = 1; rt * qg <= kScanMaxWarps; ++rt) {
      const int warps = rt * qg, smem = (int)scan_smem_bytes(T, qg, rt);
      const int by_smem = 227 * 1024 / (smem + 2048), by_regs = (T == 1 ? 40 : 20) / warps;      // (neither is 0)
      const int resident = by_smem < by_regs ? by_smem : by_regs;
      const int blocks = (tiles + rt - 1) / rt, per_sm = (blocks + n_sms - 1) / n_sms, full = per_sm / resident;
      const int bytes = kScanCC * 8 * 8 * T * qg + 8 * rt * kScanCC * 4, own = 400 + 50 * (bytes / 512) / warps;
      auto wave = [&](int b) {
        const int mma = (b * warps + 3) / 4 * (T * 128 + 40), load = b * bytes / 32;
        return (mma > load ? mma : load) + own;
      };
      const int rest = per_sm - full * resident;
      const long long t = (long long)full * wave(resident) + (rest ? wave(rest) : 0) + (long long)blocks * bytes / 8000;
      if (least < 0 || t < least) {
        least = t;
        best = {T, qg, rt, (size_t)smem};
      }
    }
  }
  return best;
}

struct ScanParams {
  const float* frame_key; const float* seg_key; const float* patch_key;
  long long n_frm, n_seg, n_pat;
  int C, nq, Hkv;
  const double* q64t; const double* qn2;
  double* s_frm; double* s_seg; double* s_pat;
  long long frm_stride, seg_stride, pat_stride;
  // the scores in single precision, which rank_kernel sifts; a patch-level block without tokens is marked kScanAbsent
  float* f_frm; float* f_seg; float* f_pat;
  long long f_frm_stride, f_seg_stride, f_pat_stride;         // multiples of four
  const int* patch_cnt;
  int q_groups, row_tiles;                                    // scan_kernel, see ScanShape
};
#define kScanAbsent (-INFINITY)
// The score of a block whose key, or of a question whose pooled vector, holds Inf or NaN: below every cosine and every mix
// of two.  Every score that is ranked is finite, so that a ranking of n members for k <= n places always fills all k (with a
// NaN for the k-th largest score no comparison holds and nothing was kept; the ids were then whatever lay in shared memory).
// (Both tests look at the high words: a comparison of doubles is slow, and these sit in chains that a question waits for.)
constexpr double kScoreNone = -2.0;
__device__ __forceinline__ bool no_score(double sc) { return __double2hiint(sc) == (int)0xc0000000; }   // (-2, cosines are above it)
__device__ __forceinline__ double finite_score(double sc) {
  return (__double2hiint(sc) & 0x7ff00000) == 0x7ff00000 ? kScoreNone : sc;
}

__device__ __forceinline__ void scan_store(const ScanParams& sp, int qi, long long row, double sc) {
  sc = finite_score(sc);
  if (row < sp.n_frm) {
    sp.s_frm[(long long)qi * sp.frm_stride + row] = sc;
    sp.f_frm[(long long)qi * sp.f_frm_stride + row] = (float)sc;
  } else if (row < sp.n_frm + sp.n_seg) {
    row -= sp.n_frm;
    sp.s_seg[(long long)qi * sp.seg_stride + row] = sc;
    sp.f_seg[(long long)qi * sp.f_seg_stride + row] = (float)sc;
  } else {
    row -= sp.n_frm + sp.n_seg;
    sp.s_pat[(long long)qi * sp.pat_stride + row] = sc;
    sp.f_pat[(long long)qi * sp.f_pat_stride + row] = sp.patch_cnt[row] > 0 ? (float)sc : kScanAbsent;
  }
}

template <int T>
__global__ void __launch_bounds__(32 * kScanMaxWarps) scan_kernel(const ScanParams sp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_qn[MUKV_MAX_QUESTIONS];
  const int C = sp.C, nq = sp.nq, nt = blockDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int QB = 8 * T * sp.q_groups, q_stride = QB + kScanQPad, R = 8 * sp.row_tiles;
  double* const s_q = reinterpret_cast<double*>(smem_raw);                        // [2][kScanCC][q_stride]
  float* const s_rows = reinterpret_cast<float*>(s_q + 2 * kScanCC * q_stride);   // [2][R][kScanRowPad]
  const long long row0 = (long long)blockIdx.x * R, n_rows = sp.n_frm + sp.n_seg + sp.n_pat;
  auto copy16 = [](void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst)), "l"(src) : "memory");
  };
  auto row_ptr = [&](long long row) {
    return row < sp.n_frm ? sp.frame_key + row * C
           : (row < sp.n_frm + sp.n_seg ? sp.seg_key + (row - sp.n_frm) * C
                                        : sp.patch_key + (row - sp.n_frm - sp.n_seg) * C);
  };
  auto fetch_rows = [&](int c0, int buf) {                   // (rows behind the last one repeat it: nobody stores their scores)
    for (int v = tid; v < R * (kScanCC / 4); v += nt) {
      const int r = v / (kScanCC / 4), c = v % (kScanCC / 4) * 4;
      copy16(s_rows + ((long long)buf * R + r) * kScanRowPad + c, row_ptr(min(row0 + r, n_rows - 1)) + c0 + c);
    }
  };
  auto fetch_questions = [&](int c0, int buf) {              // (columns behind the last question hold anything: a column of the
    for (int v = tid; v < kScanCC * (QB / 2); v += nt) {     // product depends on its own question only)
      const int c = v / (QB / 2), q = v % (QB / 2) * 2;
      copy16(s_q + ((long long)buf * kScanCC + c) * q_stride + q, sp.q64t + (long long)(c0 + c) * MUKV_MAX_QUESTIONS + q);
    }
  };
  // (The first keys are on their way before the wait: the kernel in front is qpool_kernel, which lets this one start only when
  // everything before it is complete.)
  fetch_rows(0, 0);
  pdl_wait();                                                // the pooled questions are complete
  // (No early start for the ranking: over 1,400 pairs of questions, rows and key widths it gained 0.4 us where the scan is one wave
  // of blocks, mostly nothing, and cost up to 4.5 us where it is longer.)
  fetch_questions(0, 0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int qq = tid; qq < nq; qq += nt) {                    // norms of the pooled questions (read after the barriers below)
    double t = 0.0;
    for (int g = 0; g < sp.Hkv; ++g) t += sp.qn2[(long long)qq * sp.Hkv + g];
    s_qn[qq] = sqrt(t);
  }
  const int rt = warp / sp.q_groups, q0 = warp % sp.q_groups * 8 * T;        // this warp's rows and questions
  const int fr = lane >> 2, fk = lane & 3;                   // fragment row / k (A), k / column (B)
  double acc[T][2], kk = 0.0;
#pragma unroll
  for (int i = 0; i < T; ++i) { acc[i][0] = 0.0; acc[i][1] = 0.0; }
  for (int c0 = 0, buf = 0; c0 < C; c0 += kScanCC, buf ^= 1) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();                                         // this chunk is there, the one before has been consumed
    if (c0 + kScanCC < C) {
      fetch_rows(c0 + kScanCC, buf ^ 1);
      fetch_questions(c0 + kScanCC, buf ^ 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const float* a_src = s_rows + ((long long)buf * R + rt * 8 + fr) * kScanRowPad + fk;
    const double* b_src = s_q + ((long long)buf * kScanCC + fk) * q_stride + q0 + fr;
#pragma unroll
    for (int k = 0; k < kScanCC; k += 4) {
      const double a = (double)a_src[k];                     // A[row fr][k fk]
      kk = fma(a, a, kk);
#pragma unroll
      for (int t = 0; t < T; ++t) dmma_m8n8k4(acc[t], a, b_src[k * q_stride + t * 8]);   // B[k fk][col fr]
    }
  }
  // the four lanes of a row hold the parts of its squared norm
  kk += __shfl_xor_sync(kFull, kk, 1);
  kk += __shfl_xor_sync(kFull, kk, 2);
  const double knorm = sqrt(kk);
  // accumulator tile: row fr, columns 2*fk and 2*fk + 1
  const long long row = row0 + rt * 8 + fr;
  if (row < n_rows) {
#pragma unroll
    for (int t = 0; t < T; ++t) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int qi = q0 + t * 8 + 2 * fk + e;
        if (qi >= nq) continue;
        double den = knorm * s_qn[qi];
        den = den > 1e-12 ? den : 1e-12;
        scan_store(sp, qi, row, acc[t][e] / den);
      }
    }
  }
}

// The same for at most kScanFew questions: a warp per row, plain double-precision multiply-adds; a row is one round trip to memory, 16
// doubles per lane and a butterfly.  scan_kernel goes through the feature axis in chunks, a barrier and the questions' operands
// each: 28 us for a few questions and half an hour of 512 channels, with pooling, ranking and a small gather, where this one
// takes 18 to 24.  But it takes eight questions in the time of one, and this one adds each question's product to every row, in loops
// made for one, for four and for eight questions.  Where the two take the same time was measured at 64 to 2,048 channels, 107 to
// 44,625 rows, with the keys in L2 and with L2 flushed (a chunk is then a round trip to memory, so that the tiles start to pay later);
// the line follows the flushed ones.  At 512 channels: 2 questions and 21,000 rows, 4 and 12,000, 5 and 10,000, 8 and 7,400 (in L2:
// 15,000, 9,600, 5,000 and 4,500); at 128 channels 2 and 6,000, 8 and 3,000; at 1,024 4 and 30,000, 8 and 10,000.  Eight questions
// on 11,475 rows of 512 channels: 55 us by rows, 48 by tiles (43 and 36); on 44,625 rows 107 and 66 (97 and 54).
__host__ inline bool scan_by_rows(long long rows, int nq, int C) {
  if (nq == 1) return rows <= 200LL * C;
  if (nq <= 4) return rows <= (60LL - 9 * nq) * C;
  return nq <= kScanFew && rows * nq <= 100LL * C && rows <= 12000;
}

template <int NQ>
__global__ void __launch_bounds__(256) scan_few_kernel(const ScanParams sp) {
  const int lane = threadIdx.x & 31;
  const int C = sp.C, nq = sp.nq;
  pdl_wait();                                                // the pooled questions are complete
  pdl_trigger();
  double qn = 0.0;                                           // lane i: norm of question i
  if (lane < nq) {
    for (int g = 0; g < sp.Hkv; ++g) qn += sp.qn2[(long long)lane * sp.Hkv + g];
    qn = sqrt(qn);
  }
  const long long n_rows = sp.n_frm + sp.n_seg + sp.n_pat;
  auto row_ptr = [&](long long row) {
    return row < sp.n_frm ? sp.frame_key + row * C
           : (row < sp.n_frm + sp.n_seg ? sp.seg_key + (row - sp.n_frm) * C
                                        : sp.patch_key + (row - sp.n_frm - sp.n_seg) * C);
  };
  constexpr int RW = NQ > 1 ? 2 : 1;                         // rows of a warp (they share the loads of the questions)
  for (long long row = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * RW; row < n_rows; row += (long long)gridDim.x * 8 * RW) {
    const float* src[RW];
    double dot[RW][NQ], kk[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      src[r] = row_ptr(row + r < n_rows ? row + r : row);
      kk[r] = 0.0;
#pragma unroll
      for (int i = 0; i < NQ; ++i) dot[r][i] = 0.0;
    }
    for (int c0 = 0; c0 < C; c0 += 512) {
      float4 x[RW][4];                                       // (C is a multiple of 32, not always of 512)
#pragma unroll
      for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = c0 + 128 * j + 4 * lane;
          x[r][j] = c < C ? __ldg(reinterpret_cast<const float4*>(src[r] + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + 128 * j + 4 * lane;
        double a[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          a[r][0] = (double)x[r][j].x; a[r][1] = (double)x[r][j].y; a[r][2] = (double)x[r][j].z; a[r][3] = (double)x[r][j].w;
          kk[r] = fma(a[r][0], a[r][0], fma(a[r][1], a[r][1], fma(a[r][2], a[r][2], fma(a[r][3], a[r][3], kk[r]))));
        }
        if (c < C) {
#pragma unroll
          for (int i = 0; i < NQ; ++i) {
            if (i < nq) {
              const double2* q = reinterpret_cast<const double2*>(sp.q64t + (long long)i * C + c);
              const double2 q0 = q[0], q1 = q[1];
#pragma unroll
              for (int r = 0; r < RW; ++r)
                dot[r][i] = fma(a[r][0], q0.x, fma(a[r][1], q0.y, fma(a[r][2], q1.x, fma(a[r][3], q1.y, dot[r][i]))));
            }
          }
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const double knorm = sqrt(warp_sum(kk[r]));
      double mine = 0.0;
#pragma unroll
      for (int i = 0; i < NQ; ++i) {
        const double d = warp_sum(dot[r][i]);
        if (lane == i) mine = d;
      }
      if (lane < nq && row + r < n_rows) {
        double den = knorm * qn;
        den = den > 1e-12 ? den : 1e-12;
        scan_store(sp, lane, row + r, mine / den);
      }
      __syncwarp();
    }
  }
}

// ------------------------------------------------------------------------------ ranking
constexpr int kRankList = 64;      // keys left in the radix select below which they are ranked directly
constexpr int kRankCand = 512;     // candidates that are ranked among themselves (at most one per thread)
constexpr int kRankBins = 512;     // bins of the linear histogram
constexpr int kRankFew = 128;      // scores that are all candidates at once (the histogram costs as much as ranking that many)

struct RankScratch {
  unsigned int hist[kRankBins];
  unsigned int wmin[32], wmax[32];
  int wcnt[32];
  int scan[40];
  unsigned long long prefix;
  double tau;
  int remaining;
  int bin, bin_count, list_n, cand_n;
  unsigned long long list[kRankList];
  __align__(16) unsigned long long cand_key[kRankCand];      // order keys, padded with 0 to a multiple of four
  __align__(16) int cand_idx[kRankCand];
  __align__(16) int kept_idx[kRankCand];                     // cand_idx of what is kept, INT_MAX of the rest
};

// order-preserving bits of a float and back
__device__ __forceinline__ unsigned order_key32(float x) {
  const unsigned b = __float_as_uint(x);
  return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float order_key32_inv(unsigned k) { return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k); }

// score(i) read from an array; every index a member.  One pair of types for the selections over
// segments, frames and candidates, so that they share one copy of block_topk_set (kept out of
// line: the ranking kernel is bound by instruction fetch, not by arithmetic).
struct ArrScore {
  const double* p;
  __device__ double operator()(int i) const { return p[i]; }
};
// every index takes part, or (patch-level blocks) those that hold tokens
struct Members {
  const int* cnt;
  __device__ bool operator()(int i) const { return !cnt || cnt[i] > 0; }
};

// The k best of the n_cand candidates in sc->cand_key / cand_idx (all: every one), with the tie band, ascending by
// index to out_idx / out_score; returns k.  n_cand <= kRankCand <= threads of the block.  Up to a quarter of the
// threads' number of candidates, four threads share one (the counting loops are what takes the time).
__device__ __noinline__ int rank_candidates(int n_cand, int k, bool all, double delta, int* out_idx, double* out_score,
                                            RankScratch* sc) {
  const int tid = threadIdx.x;
  const int sh = n_cand <= (int)blockDim.x / 4 ? 2 : 0, parts = 1 << sh, part = tid & (parts - 1), me = tid >> sh;
  const bool in = me < n_cand, first = part == 0;
  const unsigned long long key = in ? sc->cand_key[me] : 0ull;
  const int my_idx = in ? sc->cand_idx[me] : 0x7fffffff;
  const int n4 = (n_cand + 3) & ~3;
  if (tid >= n_cand && tid < n4) { sc->cand_key[tid] = 0ull; sc->kept_idx[tid] = 0x7fffffff; }
  __syncthreads();
  double tau = -1.0e300;
  if (!all) {
    int gt = 0, ge = 0;                                      // (the padding counts in neither: no score has key 0)
    for (int t = 4 * part; in && t < n_cand; t += 4 * parts) {
      const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(sc->cand_key + t);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(sc->cand_key + t + 2);
      gt += (a.x > key) + (a.y > key) + (b.x > key) + (b.y > key);
      ge += (a.x >= key) + (a.y >= key) + (b.x >= key) + (b.y >= key);
    }
    __syncwarp();
    if (sh) {                                                // (sh is the same in every thread)
      gt += __shfl_xor_sync(kFull, gt, 1);
      gt += __shfl_xor_sync(kFull, gt, 2);
      ge += __shfl_xor_sync(kFull, ge, 1);
      ge += __shfl_xor_sync(kFull, ge, 2);
    }
    if (in && gt < k && k <= ge) sc->tau = order_key_inv(key);   // every writer holds the same value
    __syncthreads();
    tau = sc->tau;
  }
  const double s = order_key_inv(key);
  const bool sure = in && (all || s > tau + delta);
  const bool band = in && !sure && s >= tau - delta;
  const int n_sure = __syncthreads_count(sure && first), n_band = __syncthreads_count(band && first);
  bool keep = sure || band;
  if (n_sure + n_band > k) {                                 // places inside the band go to the lowest indices
    if (in && first) sc->kept_idx[me] = band ? my_idx : 0x7fffffff;
    __syncthreads();
    if (band) {
      int before = 0;
      for (int t = 0; t < n_cand; ++t) before += sc->kept_idx[t] < my_idx ? 1 : 0;
      keep = before < k - n_sure;
    }
    __syncthreads();
  }
  if (in && first) sc->kept_idx[me] = keep ? my_idx : 0x7fffffff;
  __syncthreads();
  int pos = 0;
  for (int t = 4 * part; in && t < n_cand; t += 4 * parts) {
    const int4 a = *reinterpret_cast<const int4*>(sc->kept_idx + t);
    pos += (a.x < my_idx) + (a.y < my_idx) + (a.z < my_idx) + (a.w < my_idx);
  }
  __syncwarp();
  if (sh) {
    pos += __shfl_xor_sync(kFull, pos, 1);
    pos += __shfl_xor_sync(kFull, pos, 2);
  }
  if (keep && first) {
    out_idx[pos] = my_idx;
    if (out_score) out_score[pos] = s;
  }
  __syncthreads();
  return k;
}

// bins of the linear histogram: the bin number does not decrease with s, whatever is rounded
struct RankBins {
  float lo, scale;
  __device__ int operator()(float s) const {
    const int b = (int)((s - lo) * scale);
    return b < 0 ? 0 : (b < kRankBins ? b : kRankBins - 1);
  }
};
__device__ __forceinline__ RankBins rank_bins(const RankScratch* sc, int nwarp) {
  const int lane = threadIdx.x & 31, wl = lane < nwarp ? lane : 0;
  const float lo = order_key32_inv(__reduce_min_sync(kFull, sc->wmin[wl]));
  const float hi = order_key32_inv(__reduce_max_sync(kFull, sc->wmax[wl]));
  return {lo, hi > lo ? fminf((float)kRankBins / (hi - lo), 1e35f) : 0.f};
}
// the bin that holds the k-th largest score (the histogram is complete); two barriers
__device__ __forceinline__ int rank_find_bin(int k, RankScratch* sc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c = tid < kRankBins ? (int)sc->hist[kRankBins - 1 - tid] : 0;       // thread t: the bin t places from the top
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) sc->scan[warp] = incl;
  __syncthreads();
  const int above = __reduce_add_sync(kFull, lane < warp ? sc->scan[lane] : 0) + incl - c;
  if (above < k && k <= above + c) sc->bin = kRankBins - 1 - tid;               // true for exactly one thread
  __syncthreads();
  return sc->bin;
}

// Indices of the k highest scores among i in [0,n) with member(i) true, ascending by index, with
// the tie band: tau = k-th largest; scores above tau+delta are taken; those within delta of tau
// share the remaining places by lowest index.  Run by the whole block; returns the count
// (= min(k, number of members)).  score(i) must be cheap, pure and finite.
template <typename ScoreFn, typename MemberFn>
__device__ __noinline__ int block_topk_set(ScoreFn score, MemberFn member, int n, int k, double delta, int* out_idx,
                              double* out_score, RankScratch* sc) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  bool all = false;
  int n_mem = 0, bin = 0;
  RankBins bin_of{0.f, 0.f};
  __syncthreads();                                           // the scratch may still be read from a previous call
  if (tid == 0) sc->cand_n = 0;
  if (n > kRankFew) {
    // The k-th largest score tau lies in one bin of a linear histogram.  Whatever could be above it or within the tie
    // band of it is collected (any order) and ranked exactly: three sweeps over the scores instead of two for every
    // eight bits of a radix select, whose first passes see nothing but the common exponent.
    // ---- how many members, and the range of their scores (in single precision: it only places the bins)
    unsigned kmin = 0xffffffffu, kmax = 0u;
    int local = 0;
    for (int i = tid; i < n; i += nt) {
      if (!member(i)) continue;
      const float s = (float)score(i);
      const unsigned key = order_key32(s);
      kmin = min(kmin, key);
      kmax = max(kmax, key);
      ++local;
    }
    __syncwarp();
    kmin = __reduce_min_sync(kFull, kmin);
    kmax = __reduce_max_sync(kFull, kmax);
    local = __reduce_add_sync(kFull, local);
    if (lane == 0) { sc->wmin[warp] = kmin; sc->wmax[warp] = kmax; sc->wcnt[warp] = local; }
    for (int b = tid; b < kRankBins; b += nt) sc->hist[b] = 0u;
    __syncthreads();
    n_mem = __reduce_add_sync(kFull, lane < nwarp ? sc->wcnt[lane] : 0);
    if (k > n_mem) k = n_mem;
    if (k <= 0) return 0;
    all = (k == n_mem);
    bin_of = rank_bins(sc, nwarp);
    if (!all) {
      for (int i = tid; i < n; i += nt)
        if (member(i)) atomicAdd(&sc->hist[bin_of((float)score(i))], 1u);
      __syncthreads();
      bin = rank_find_bin(k, sc);
    }
  } else {
    __syncthreads();
  }
  const double slack = 2.0 * delta + 1e-12;
  for (int i = tid; i < n; i += nt) {
    if (!member(i)) continue;
    const double s = score(i);
    if (bin == 0 || bin_of((float)(s + slack)) >= bin) {
      const int c = atomicAdd(&sc->cand_n, 1);
      if (c < kRankCand) {
        sc->cand_idx[c] = i;
        sc->cand_key[c] = order_key(s);
      }
    }
  }
  __syncthreads();
  const int n_cand = sc->cand_n;
  if (n <= kRankFew) {
    n_mem = n_cand;
    if (k > n_mem) k = n_mem;
    if (k <= 0) return 0;
    all = (k == n_mem);
  }
  if (n_cand <= kRankCand) return rank_candidates(n_cand, k, all, delta, out_idx, out_score, sc);
  // ---- too many candidates (a large k, a crowded bin): radix select and an ordered walk
  double tau = -1.0e300;                                     // (all: everything is taken)
  __syncthreads();
  if (!all) {
    // radix select of the k-th largest order key, 8 bits per pass from the top
    if (tid == 0) { sc->prefix = 0ull; sc->remaining = k; }
    for (int pass = 0; pass < 8; ++pass) {
      const int shift = 56 - 8 * pass;
      for (int b = tid; b < 256; b += nt) sc->hist[b] = 0u;
      __syncthreads();
      const unsigned long long prefix = sc->prefix;
      const unsigned long long himask = pass == 0 ? 0ull : (~0ull << (shift + 8));
      for (int i = tid; i < n; i += nt) {
        if (!member(i)) continue;
        const unsigned long long key = order_key(score(i));
        if ((key & himask) == prefix) atomicAdd(&sc->hist[(unsigned)(key >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (tid < 32) {
        // warp 0 finds the bin that holds the remaining-th largest key: lane l owns bins 8l .. 8l+7
        int c[8], T = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) { c[i] = (int)sc->hist[8 * tid + i]; T += c[i]; }
        int incl = T;                                   // keys in this lane's bins and all higher ones
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_down_sync(kFull, incl, o);
          if (tid + o < 32) incl += v;
        }
        const int above = incl - T;
        const int rem = sc->remaining;
        __syncwarp();
        if (above < rem && rem <= above + T) {          // true for exactly one lane
          int r = rem - above, b = 7;
          for (; b > 0; --b) {
            if (r <= c[b]) break;
            r -= c[b];
          }
          sc->prefix = prefix | ((unsigned long long)(8 * tid + b) << shift);
          sc->remaining = r;
          sc->bin_count = c[b];
        }
      }
      __syncthreads();
      if (pass < 7 && sc->bin_count <= kRankList) {
        // few keys share the prefix found so far: collect them and rank them directly
        const unsigned long long pre = sc->prefix, mask = ~0ull << shift;
        if (tid == 0) sc->list_n = 0;
        __syncthreads();
        for (int i = tid; i < n; i += nt) {
          if (!member(i)) continue;
          const unsigned long long key = order_key(score(i));
          if ((key & mask) == pre) sc->list[atomicAdd(&sc->list_n, 1)] = key;
        }
        __syncthreads();
        const int m = sc->list_n, r = sc->remaining;
        if (tid < m) {
          const unsigned long long key = sc->list[tid];
          int gt = 0, ge = 0;
          for (int t = 0; t < m; ++t) {
            gt += (sc->list[t] > key);
            ge += (sc->list[t] >= key);
          }
          if (gt < r && r <= ge) sc->prefix = key;      // every writer holds the same value
        }
        __syncthreads();
        break;
      }
    }
    tau = order_key_inv(sc->prefix);
  }
  // count the sure ones
  int cnt = 0;
  for (int i = tid; i < n; i += nt)
    if (member(i) && !all && score(i) > tau + delta) ++cnt;
  __syncthreads();
  if (tid == 0) sc->remaining = 0;
  __syncthreads();
  cnt = warp_sum(cnt);
  if ((tid & 31) == 0 && cnt) atomicAdd(&sc->remaining, cnt);
  __syncthreads();
  const int need = k - sc->remaining;
  __syncthreads();
  // ordered emission
  int band_before = 0, out_before = 0;
  for (int base = 0; base < n; base += nt) {
    const int i = base + tid;
    bool sure = false, band = false;
    double s = 0.0;
    if (i < n && member(i)) {
      s = score(i);
      if (all) sure = true;
      else {
        sure = s > tau + delta;
        band = !sure && s >= tau - delta;
      }
    }
    int n_band, n_out;
    const int br = band_before + block_excl_count(band, sc->scan, n_band);
    const bool keep = sure || (band && br < need);
    const int pos = out_before + block_excl_count(keep, sc->scan, n_out);
    if (keep) {
      out_idx[pos] = i;
      if (out_score) out_score[pos] = s;
    }
    band_before += n_band;
    out_before += n_out;
  }
  __syncthreads();
  return k;
}

// block_topk_set for scores whose single-precision copies lie in shared memory (buf, 16-byte aligned, kScanAbsent where a
// score takes no part; up to three values behind the n-th are overwritten): range, histogram and collection run on the
// copies, four at a time, and only the candidates' doubles are read.  (On doubles the three sweeps were bound by
// instruction issue: 12 us for 10,800 scores; loading and converting them here took another 7.)
__device__ __noinline__ int staged_topk_set(const double* scores, const int* cnt, int n, int k, double delta, int* out_idx,
                                            double* out_score, float* buf, RankScratch* sc) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  int local = 0;
  const int n4 = (n + 3) & ~3;
  if (tid < n4 - n) buf[n + tid] = kScanAbsent;
  __syncthreads();                                           // (the scratch may still be read from a previous call, too)
  float lo = INFINITY, hi = -INFINITY;
  for (int v = tid; v < n4 >> 2; v += nt) {
    const float4 q = reinterpret_cast<const float4*>(buf)[v];
    const float s[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool absent = s[u] == kScanAbsent;
      lo = fminf(lo, absent ? INFINITY : s[u]);
      hi = fmaxf(hi, s[u]);
      local += absent ? 0 : 1;
    }
  }
  __syncwarp();
  unsigned kmin = order_key32(lo), kmax = order_key32(hi);
  kmin = __reduce_min_sync(kFull, kmin);
  kmax = __reduce_max_sync(kFull, kmax);
  local = __reduce_add_sync(kFull, local);
  if (lane == 0) { sc->wmin[warp] = kmin; sc->wmax[warp] = kmax; sc->wcnt[warp] = local; }
  for (int b = tid; b < kRankBins; b += nt) sc->hist[b] = 0u;
  if (tid == 0) sc->cand_n = 0;
  __syncthreads();
  const int n_mem = __reduce_add_sync(kFull, lane < nwarp ? sc->wcnt[lane] : 0);
  if (k > n_mem) k = n_mem;
  if (k <= 0) return 0;
  const bool all = (k == n_mem);
  const RankBins bin_of = rank_bins(sc, nwarp);
  int bin = 0;
  if (!all) {
    for (int v = tid; v < n4 >> 2; v += nt) {
      const float4 s = reinterpret_cast<const float4*>(buf)[v];
      atomicAdd(&sc->hist[bin_of(s.x)], 1u);
      atomicAdd(&sc->hist[bin_of(s.y)], 1u);
      atomicAdd(&sc->hist[bin_of(s.z)], 1u);
      atomicAdd(&sc->hist[bin_of(s.w)], 1u);
    }
    __syncthreads();
    bin = rank_find_bin(k, sc);
  }
  // within delta of a score of that bin, and what single precision may have moved (scores of magnitude 1 or less
  // by 6e-8; the range serves for others)
  const float span = bin_of.scale > 0.f ? (float)kRankBins / bin_of.scale : 0.f;
  const float slack = 2.f * (float)delta + 1e-6f * fmaxf(1.f, fmaxf(fabsf(bin_of.lo), fabsf(bin_of.lo + span)));
  for (int v = tid; v < n4 >> 2; v += nt) {
    const float4 q = reinterpret_cast<const float4*>(buf)[v];
    const float s[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (bin_of(s[u] + slack) >= bin && s[u] != kScanAbsent) {
        const int c = atomicAdd(&sc->cand_n, 1);
        if (c < kRankCand) sc->cand_idx[c] = 4 * v + u;
      }
    }
  }
  __syncthreads();
  const int n_cand = sc->cand_n;
  if (n_cand <= kRankCand) {
    if (tid < n_cand) sc->cand_key[tid] = order_key(scores[sc->cand_idx[tid]]);
    __syncthreads();
    return rank_candidates(n_cand, k, all, delta, out_idx, out_score, sc);
  }
  return block_topk_set(ArrScore{scores}, Members{cnt}, n, k, delta, out_idx, out_score, sc);
}

// the one of the two that fits (buf: null where there are no copies)
__device__ __forceinline__ int topk_set(const double* scores, const int* cnt, int n, int k, double delta, int* out_idx,
                                        double* out_score, float* buf, RankScratch* sc) {
  const int tid = threadIdx.x;
  if (n <= kRankFew && !cnt) {                               // every score is a candidate
    __syncthreads();                                         // (the scratch may still be read from a previous call)
    if (tid < n) { sc->cand_key[tid] = order_key(scores[tid]); sc->cand_idx[tid] = tid; }
    __syncthreads();
    k = min(k, n);
    return k > 0 ? rank_candidates(n, k, k == n, delta, out_idx, out_score, sc) : 0;
  }
  if (n > kRankFew && buf) return staged_topk_set(scores, cnt, n, k, delta, out_idx, out_score, buf, sc);
  return block_topk_set(ArrScore{scores}, Members{cnt}, n, k, delta, out_idx, out_score, sc);
}

struct RankParams {
  int nq, C, fseg;
  int k_seg, k_frm, k_pat, top_n, mode;
  int roles;                              // blocks per question, see rank_roles
  int S;                                  // patch-level blocks per frame (0: none)
  double lam_seg, lam_frm, lam_pat, delta;
  long long n_frm, n_seg;                 // stored
  const double* s_frm;                    // [nq][frm_stride]
  const double* s_seg;
  const double* s_pat;                    // [nq][pat_stride]
  long long frm_stride, seg_stride, pat_stride;
  const float* frame_key;
  const float* seg_key;
  const float* patch_key;
  const int* patch_cnt;                   // [frames][S]
  int* seg_idx; int* frm_idx; int* pat_idx; float* seg_score; float* frm_score; float* pat_score;
  int* counts; int counts_stride;         // 2 or 3 ints per question
  const float* f_frm; const float* f_seg; const float* f_pat;     // single-precision copies of the scores
  long long f_frm_stride, f_seg_stride, f_pat_stride;
  int stage;                              // bits 0, 1, 2: the copies of segments, frames, patch-level blocks fit in shared memory
};

constexpr int kRankThreads = 512;
constexpr int kRankStageBytes = 192 * 1024;       // dynamic shared memory the kernel may be given
constexpr int kMaxCand = 2 * MUKV_MAX_TOPK;

struct RankShared {
  RankScratch sc;
  int sel_seg[MUKV_MAX_TOPK];
  double sel_seg_score[MUKV_MAX_TOPK];
  int top[MUKV_MAX_TOPK];
  int cand[kMaxCand];
  double cand_score[kMaxCand];
  int pick[MUKV_MAX_TOPK];
  double pick_score[MUKV_MAX_TOPK];
  double gn[kRankThreads / 32];
  // what the block of the segments finds for the others
  double gnorm;
  int have_g, c_seg;
};

// Stage 1 + stage 2 of one granularity for one question, run by the whole block: top-2k candidates
// by cosine among the members, Eq. 8 against the global query gq (norm gnorm; have_g false: gamma = 0),
// then the k best by the calibrated score.  PARALLEL / HIER callers pass semi = false: the k best by
// cosine among the members.  Results (ascending ids) in sh->pick / sh->pick_score; returns the count.
// remote: the global query is fetched from the block of the segments between the stages, see rank_kernel.
__device__ __noinline__ int rank_level(const double* scores, const int* cnt, int n, int k, bool semi, double lambda,
                                       double delta, const float* keys, int C, double* gq, bool remote, RankShared* sh,
                                       float* buf) {
  const int tid = threadIdx.x;
  const int n_cand = topk_set(scores, cnt, n, semi ? 2 * k : k, delta, semi ? sh->cand : sh->pick,
                              semi ? sh->cand_score : sh->pick_score, buf, &sh->sc);
  if (!semi) return n_cand;
  if (remote) {
    tc::cluster_wait();
    for (int c = tid; c < C; c += kRankThreads) gq[c] = tc::cluster_ld_double(gq + c, 0);
    if (tid == 0) { sh->gnorm = tc::cluster_ld_double(&sh->gnorm, 0); sh->have_g = tc::cluster_ld_int(&sh->have_g, 0); }
    tc::cluster_arrive();                                    // that block may leave
    __syncthreads();
  }
  const double gnorm = sh->gnorm;
  const bool have_g = sh->have_g != 0;
  // Eq. 8 for every candidate: one warp per candidate
  const int lane = tid & 31, warp = tid >> 5;
  for (int ci = warp; ci < n_cand; ci += kRankThreads / 32) {
    const float* kr = keys + (long long)sh->cand[ci] * C;
    double dot = 0.0, kk = 0.0;
    for (int c0 = lane; c0 < C; c0 += 16 * 32) {             // (sixteen loads in flight)
      float x[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) x[u] = c0 + u * 32 < C ? __ldg(kr + c0 + u * 32) : 0.f;
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        if (c0 + u * 32 < C) {
          const double y = (double)x[u];
          dot = fma(y, gq[c0 + u * 32], dot);
          kk = fma(y, y, kk);
        }
      }
    }
    __syncwarp();
    dot = warp_sum(dot);
    kk = warp_sum(kk);
    if (lane == 0) {
      double gamma = 0.0;
      if (have_g) {
        double den = sqrt(kk) * gnorm;
        den = den > 1e-12 ? den : 1e-12;
        gamma = dot / den;
      }
      const double s1 = sh->cand_score[ci];
      sh->sc.cand_key[ci] = order_key(no_score(s1) ? kScoreNone : (1.0 - lambda) * s1 + lambda * gamma);
      sh->sc.cand_idx[ci] = ci;
    }
  }
  __syncthreads();
  // (at most 2 k candidates: no more than a thread each)
  const int c = min(k, n_cand);
  if (c > 0) rank_candidates(n_cand, c, c == n_cand, delta, sh->pick, sh->pick_score, &sh->sc);
  // pick holds positions in the candidate list (ascending position = ascending block id)
  for (int i = tid; i < c; i += kRankThreads) sh->pick[i] = sh->cand[sh->pick[i]];
  __syncthreads();
  return c;
}

__device__ __forceinline__ void rank_emit(int* idx, float* score, long long base, int k, int c, const RankShared* sh) {
  for (int i = threadIdx.x; i < k; i += kRankThreads) {
    idx[base + i] = i < c ? sh->pick[i] : -1;
    if (score) score[base + i] = i < c ? (float)sh->pick_score[i] : 0.f;
  }
}

// A cluster of two or three blocks per question, one for each granularity: block 0 ranks the segments and works out the global
// query, block 1 the frames, block 2 (k_pat > 0) the patch-level blocks.  Stage 1 needs nothing of the other blocks, stage 2 the
// global query, which is read from block 0's shared memory behind a cluster barrier.  (One block after the other: 14.5 us for
// one question on an hour of video, of which the segments and the global query were 5; bound by a chain of barriers, round
// trips to L2 and instruction fetch, so that blocks beside one another are what helps.)
// HIER looks at the frames of the selected segments only, so a block of the frames would wait for that of the segments from the
// start: block 0 ranks both, block 1 (k_pat > 0) the patch-level blocks beside its frames.  (With a block each, the hand-over cost
// one question on three hours of video 25.8 us with its gather, now 24.4; 64 on half an hour 65.2, now 64.3.)
__host__ __device__ inline int rank_roles(int mode, int k_pat) { return (mode == MUKV_RETR_HIER ? 1 : 2) + (k_pat > 0 ? 1 : 0); }
__global__ void __launch_bounds__(kRankThreads) rank_kernel(const RankParams p, const QMeta meta) {
  __shared__ RankShared sh;
  __shared__ __align__(8) uint64_t s_bar[1];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* gq = reinterpret_cast<double*>(smem_raw);               // [C] global query

  const int role = (int)tc::cluster_rank(), roles = p.roles;
  const int qi = blockIdx.x / roles, tid = threadIdx.x;
  if (role > 0) tc::cluster_arrive();                        // (phase 1: block 0 arrives when the others may go on)
  pdl_wait();                                                // the scores of the scan are complete
  // (No early start for the gather: 0.1 to 0.6 us slower for 1 to 128 questions on 100 to 10,800 frames, faster for none of them.)
  const int C = p.C;
  long long tl = meta.t_limit[qi];
  if (tl > p.n_frm) tl = p.n_frm;
  if (tl < 0) tl = 0;
  const int n_frm = (int)tl;
  // segment u is visible when its last stored frame is: min((u+1)*fseg, n_stored) <= t_limit
  int n_seg = (int)(tl / p.fseg);
  if (tl == p.n_frm && (p.n_frm % p.fseg) != 0) n_seg += 1;
  if (n_seg > p.n_seg) n_seg = (int)p.n_seg;
  const double* sf = p.s_frm + (long long)qi * p.frm_stride;
  const double* ss = p.s_seg + (long long)qi * p.seg_stride;
  const double* sp = p.s_pat + (long long)qi * p.pat_stride;
  const bool semi = p.mode == MUKV_RETR_SEMI, hier = p.mode == MUKV_RETR_HIER;
  // Single-precision copies of this block's scores.  (n4 values: what lies behind the n-th belongs to this question's row, too)
  const int n = role == 0 ? n_seg : role == 1 ? n_frm : n_frm * p.S, n4 = (n + 3) & ~3;
  float* buf = nullptr;
  // (few scores are all read as they are; HIER looks at the selected segments' frames only)
  if (((p.stage >> role) & 1) && n > kRankFew && !(hier && role > 0)) {
    buf = reinterpret_cast<float*>(gq + C);
    const float* src = role == 0 ? p.f_seg + (long long)qi * p.f_seg_stride
                       : role == 1 ? p.f_frm + (long long)qi * p.f_frm_stride : p.f_pat + (long long)qi * p.f_pat_stride;
    const uint32_t bar = tc::smem_u32(s_bar);
    if (tid == 0) {
      tc::mbar_init(bar, 1);
      tc::fence_mbar_init();
      tc::fence_proxy_async_smem();
      tc::mbar_expect_tx(bar, 4u * (uint32_t)n4);
      tc::bulk_load(tc::smem_u32(buf), src, 4u * (uint32_t)n4, bar);
    }
    __syncthreads();
    // a wait that runs out (it cannot, the copy needs nothing else) leaves the doubles in global memory to rank by
    if (!__syncthreads_and(tc::mbar_wait(bar, 0u))) buf = nullptr;
  }

  if (role == 0) {
    int c_seg = -1;
    if (semi) {
      // ---- global query = mean of the top-N segment keys (stage 1 order)
      const int N = p.top_n > 0 ? p.top_n : p.k_seg;
      // (without a lambda for segments the N = k_seg best are also the result: one ranking serves both)
      const bool same = N == p.k_seg && !(p.lam_seg > 0.0);
      int* top = same ? sh.pick : sh.top;
      double* top_score = same ? sh.pick_score : sh.cand_score;
      const int n_top = topk_set(ss, nullptr, n_seg, N, p.delta, top, top_score, buf, &sh.sc);
      if (same) c_seg = n_top;
      const int n_use = __syncthreads_count(tid < n_top && !no_score(top_score[tid]));    // (N <= threads of the block)
      if (n_use < n_top) {                                   // the list without those that have no score
        if (tid == 0)
          for (int i = 0, c = 0; i < n_top; ++i)
            if (!no_score(top_score[i])) sh.top[c++] = top[i];
        __syncthreads();
        top = sh.top;
      }
      double part = 0.0;
      for (int c = tid; c < C; c += kRankThreads) {
        double t = 0.0;
        for (int i = 0; i < n_use; i += 8) {                 // (eight loads in flight, added in order)
          float x[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            x[u] = i + u < n_use ? p.seg_key[(long long)top[i + u] * C + c] : 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u) t += (double)x[u];
        }
        t = n_use > 0 ? t / (double)n_use : 0.0;
        gq[c] = t;
        part += t * t;
      }
      __syncwarp();
      part = warp_sum(part);
      if ((tid & 31) == 0) sh.gn[tid >> 5] = part;
      __syncthreads();
      double gn = 0.0;
#pragma unroll
      for (int w = 0; w < kRankThreads / 32; ++w) gn += sh.gn[w];
      if (tid == 0) { sh.gnorm = sqrt(gn); sh.have_g = n_use > 0; }
    }
    if (!hier) tc::cluster_arrive();
    __syncthreads();
    // ---- segments (the paper's lambda for them is 0: final = stage-1 top-k)
    if (c_seg < 0)
      c_seg = rank_level(ss, nullptr, n_seg, p.k_seg, semi && p.lam_seg > 0.0, p.lam_seg, p.delta, p.seg_key, C, gq, false, &sh, buf);
    rank_emit(p.seg_idx, p.seg_score, (long long)qi * p.k_seg, p.k_seg, c_seg, &sh);
    if (tid == 0) p.counts[p.counts_stride * qi] = c_seg;
    if (!hier) {
      tc::cluster_wait();
      tc::cluster_arrive();                                  // phase 2: the others have read what they need
      tc::cluster_wait();
      return;
    }
    for (int i = tid; i < c_seg; i += kRankThreads) sh.sel_seg[i] = sh.pick[i];
    if (tid == 0) sh.c_seg = c_seg;
    if (roles > 1) tc::cluster_arrive();
    __syncthreads();
  }

  // ---- frames, or patch-level blocks: (frame, super patch) pairs that kept at least one token
  const bool frames = hier ? role == 0 : role == 1;
  const double* sc = frames ? sf : sp;
  const int* cnt = frames ? nullptr : p.patch_cnt;
  const int k = frames ? p.k_frm : p.k_pat;
  int c = 0;
  if (hier) {
    // Only what lies inside the selected segments is a candidate.  Those are few, so the ranking runs over positions in the
    // list "selected segments (ascending) x their blocks" and maps the winners back (ascending position = ascending block).
    if (role > 0) {
      tc::cluster_wait();
      const int c_seg = tc::cluster_ld_int(&sh.c_seg, 0);
      for (int i = tid; i < c_seg; i += kRankThreads) sh.sel_seg[i] = tc::cluster_ld_int(sh.sel_seg + i, 0);
      if (tid == 0) sh.c_seg = c_seg;
      tc::cluster_arrive();
      __syncthreads();
    }
    const int per_seg = p.fseg * (frames ? 1 : p.S), n_blocks = frames ? n_frm : n_frm * p.S;
    auto block_of = [&](int i) { return sh.sel_seg[i / per_seg] * per_seg + i % per_seg; };
    auto score_h = [&](int i) { return sc[block_of(i)]; };
    auto member_h = [&](int i) {
      const int b = block_of(i);
      return b < n_blocks && (!cnt || cnt[b] > 0);
    };
    c = block_topk_set(score_h, member_h, sh.c_seg * per_seg, k, p.delta, sh.pick, sh.pick_score, &sh.sc);
    for (int i = tid; i < c; i += kRankThreads) sh.pick[i] = block_of(sh.pick[i]);
    __syncthreads();
  } else {
    c = rank_level(sc, cnt, n, k, semi, frames ? p.lam_frm : p.lam_pat, p.delta, frames ? p.frame_key : p.patch_key, C, gq,
                   true, &sh, buf);
    if (!semi) {
      tc::cluster_wait();
      tc::cluster_arrive();
    }
  }
  if (frames) rank_emit(p.frm_idx, p.frm_score, (long long)qi * p.k_frm, p.k_frm, c, &sh);
  else rank_emit(p.pat_idx, p.pat_score, (long long)qi * p.k_pat, p.k_pat, c, &sh);
  if (tid == 0) {
    p.counts[p.counts_stride * qi + (frames ? 1 : 2)] = c;
    if (p.k_pat == 0 && p.counts_stride > 2) p.counts[p.counts_stride * qi + 2] = 0;
  }
  if (roles > 1) tc::cluster_wait();
  if (roles > 1 && role == 0) {                              // (HIER) phase 2: the other has read what it needs
    tc::cluster_arrive();
    tc::cluster_wait();
  }
}

// ------------------------------------------------------------------------------ Eq. 9
struct GatherParams {
  int nq, k_frm, L, kappa;
  long long run_bytes;                     // kappa * C * sizeof(T): one (frame, layer, K|V) run
  const int* frm_idx; const int* counts;
  const unsigned char* store; const long long* page_table; const int* kept_store;
  unsigned char* decode; long long decode_stride;
  int* tok_meta;
};

// unit = (question, plane = l*2+kv, slot): one contiguous run of the page goes to one contiguous
// run of the decode buffer.  Bound by memory.  One block per unit: with eight blocks per SM that walked the units the blocks
// drifted apart, and 64 questions (5.75 GB, 57,344 runs of 50 KB) took 1,002 us; blocks that start in the order of the
// units keep to neighbouring pages: 867 us with 256 threads, 855 with 512 (two thirds as many runs open at a time; 128
// threads: 904), 6.7 TB/s of algorithmic bytes; where two questions share a page its second reader finds it in L2.  Runs below 16 KB would leave 512 threads idle and take 128.  (A ring of bulk copies through
// shared memory: 961 us.)
template <int NT>
__global__ void __launch_bounds__(NT) gather_kernel(const GatherParams p) {
  pdl_wait();                                              // the selection may be the work of the kernel in front
  const long long planes = (long long)p.L * 2;
  const long long n_units = (long long)p.nq * planes * p.k_frm;
  for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
    const int slot = (int)(u % p.k_frm);
    const long long r = u / p.k_frm;
    const int plane = (int)(r % planes);
    const int qi = (int)(r / planes);
    if (slot >= p.counts[2 * qi + 1]) continue;
    const int f = p.frm_idx[(long long)qi * p.k_frm + slot];
    const unsigned char* src = p.store + p.page_table[f] + (long long)plane * p.run_bytes;
    unsigned char* dst = p.decode + (long long)qi * p.decode_stride +
                         ((long long)plane * p.k_frm + slot) * p.run_bytes;
    const long long nvec = p.run_bytes >> 4;
    long long v = threadIdx.x;
    for (; v + 3 * NT < nvec; v += 4 * NT) {
      uint4 x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = ld_stream(src + ((v + i * NT) << 4));
#pragma unroll
      for (int i = 0; i < 4; ++i) st_stream(dst + ((v + i * NT) << 4), x[i]);
    }
    for (; v < nvec; v += NT) st_stream(dst + (v << 4), ld_stream(src + (v << 4)));
    if (plane == 0 && p.tok_meta) {
      for (int t = threadIdx.x; t < p.kappa; t += NT) {
        int* m = p.tok_meta + (((long long)qi * p.k_frm + slot) * p.kappa + t) * 2;
        m[0] = f;
        m[1] = p.kept_store[(long long)f * p.kappa + t];
      }
    }
  }
}

// ------------------------------------------------------------------------------ Eq. 9, all granularities
struct Gather3Params {
  int nq, k_seg, k_frm, k_pat, L, kappa, C, P, S, grid_width, patch_split;
  int tok_cap;                             // token slots per (layer, K|V) plane of a decode buffer
  int esize;                               // bytes per element of the store dtype
  const int* seg_idx; const int* frm_idx; const int* pat_idx; const int* counts;   // counts [nq][3]
  const unsigned char* store; const long long* page_table; const int* kept_store;
  const float* seg_entry;                  // [segments][L][2][C]
  const int* patch_cnt;                    // [frames][S]
  const int* kept_count;                   // [frames] tokens in a frame's page, or null: kappa in every page
  int kept_stride;                         // ints per frame in kept_store
  unsigned char* decode; long long decode_stride;
  int* ntok; int* tok_meta;
};

// one contiguous run, copied by a block of 256 threads with four 16-byte vectors in flight per thread
__device__ __forceinline__ void copy_run16(unsigned char* dst, const unsigned char* src, long long bytes) {
  const long long nvec = bytes >> 4;
  long long v = threadIdx.x;
  for (; v + 3 * 256 < nvec; v += 4 * 256) {
    const uint4 x0 = ld_stream(src + (v << 4));
    const uint4 x1 = ld_stream(src + ((v + 256) << 4));
    const uint4 x2 = ld_stream(src + ((v + 512) << 4));
    const uint4 x3 = ld_stream(src + ((v + 768) << 4));
    st_stream(dst + (v << 4), x0);
    st_stream(dst + ((v + 256) << 4), x1);
    st_stream(dst + ((v + 512) << 4), x2);
    st_stream(dst + ((v + 768) << 4), x3);
  }
  for (; v < nvec; v += 256) st_stream(dst + (v << 4), ld_stream(src + (v << 4)));
}

constexpr int kGatherListCap = 1024;       // rows of patch-level blocks listed at a time (>= MUKV_MAX_TOKENS)

// Units, one per block: first, for every question and (layer, K|V) plane, the summary tokens and the patch-level rows
// (the longest ones: at the end of their plane's runs the last of them worked alone), then per question and plane k_frm
// frame runs (one contiguous run of the page each).  Token slots of a plane: summary
// tokens of the selected segments, kept tokens of the selected frames, kept tokens of the selected
// patch-level blocks.
template <typename T>
__global__ void __launch_bounds__(256) gather3_kernel(const Gather3Params p) {
  __shared__ int s_off[MUKV_MAX_TOPK + 1];                 // first row of each selected patch block
  __shared__ long long s_src[kGatherListCap];              // byte offset in the store of each listed row
  pdl_wait();
  const long long planes = (long long)p.L * 2;
  const long long n_rest = (long long)p.nq * planes;
  const long long n_units = n_rest * (p.k_frm + 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const long long row_bytes = (long long)p.C * p.esize;
  const long long run_bytes = (long long)p.kappa * row_bytes;
  for (long long u = blockIdx.x; u < n_units; u += gridDim.x) {
    const bool run = u >= n_rest;
    const int slot = run ? (int)((u - n_rest) % p.k_frm) : 0;
    const long long r = run ? (u - n_rest) / p.k_frm : u;
    const int plane = (int)(r % planes);
    const int qi = (int)(r / planes);
    const int c_seg = p.counts[3 * qi], c_frm = p.counts[3 * qi + 1], c_pat = p.counts[3 * qi + 2];
    unsigned char* dplane = p.decode + (long long)qi * p.decode_stride + (long long)plane * p.tok_cap * row_bytes;
    int* meta = p.tok_meta ? p.tok_meta + (long long)qi * p.tok_cap * 2 : nullptr;
    // kept tokens of the first n selected frames, with pages of different lengths (every warp adds them up itself)
    auto kept_before = [&](int n) {
      int t = 0;
      for (int i = lane; i < n; i += 32) t += p.kept_count[p.frm_idx[(long long)qi * p.k_frm + i]];
      __syncwarp();
      return warp_sum(t);
    };
    if (run) {
      if (slot >= c_frm) continue;
      const int f = p.frm_idx[(long long)qi * p.k_frm + slot];
      int row0 = c_seg + slot * p.kappa, rows = p.kappa;
      if (p.kept_count) {
        // pages of different lengths: this frame's rows start behind those of the frames before it
        row0 = c_seg + kept_before(slot);
        rows = p.kept_count[f];
      }
      const long long fbytes = (long long)rows * row_bytes;
      copy_run16(dplane + (long long)row0 * row_bytes, p.store + p.page_table[f] + (long long)plane * fbytes, fbytes);
      if (plane == 0 && meta) {
        for (int t = threadIdx.x; t < rows; t += blockDim.x) {
          meta[(row0 + t) * 2] = f;
          meta[(row0 + t) * 2 + 1] = p.kept_store[(long long)f * p.kept_stride + t];
        }
      }
      continue;
    }
    // ---- summary tokens: the segment's pooled entry of this plane, rounded to the store dtype
    for (int i = 0; i < c_seg; ++i) {
      const int useg = p.seg_idx[(long long)qi * p.k_seg + i];
      const float* e = p.seg_entry + ((long long)useg * planes + plane) * p.C;
      T* d = reinterpret_cast<T*>(dplane + (long long)i * row_bytes);
      for (int c = threadIdx.x; c < p.C; c += blockDim.x) {
        if constexpr (sizeof(T) == 2) d[c] = __float2bfloat16_rn(e[c]);
        else d[c] = e[c];
      }
      if (plane == 0 && meta && threadIdx.x == 0) { meta[i * 2] = -1 - useg; meta[i * 2 + 1] = -1; }
    }
    // ---- patch-level rows: block b = frame * S + super patch holds the frame's kept rows inside it
    __syncthreads();
    const int off0 = c_seg + (p.kept_count ? kept_before(c_frm) : c_frm * p.kappa);
    for (int i = threadIdx.x; i < c_pat; i += blockDim.x) s_off[i + 1] = p.patch_cnt[p.pat_idx[(long long)qi * p.k_pat + i]];
    __syncthreads();
    if (threadIdx.x == 0) {
      int off = off0;
      s_off[0] = off;
      for (int i = 1; i <= c_pat; ++i) {
        off += s_off[i];
        s_off[i] = off;
      }
      if (plane == 0 && p.ntok) p.ntok[qi] = off;
    }
    __syncthreads();
    // Patch blocks in batches whose rows fit the list.  One warp per block walks the frame's kept
    // list and notes where the rows of its super patch lie; then the whole block copies the rows.
    const int vpr = (int)(row_bytes >> 4);                 // 16-byte vectors per row
    for (int b0 = 0; b0 < c_pat;) {
      int b1 = b0 + 1;                                     // (one block has at most kappa <= list capacity rows)
      while (b1 < c_pat && s_off[b1 + 1] - s_off[b0] <= kGatherListCap) ++b1;
      for (int i = b0 + warp; i < b1; i += nwarp) {
        const int b = p.pat_idx[(long long)qi * p.k_pat + i];
        const int f = b / p.S, sp = b % p.S;
        const long long page = p.page_table[f] + (long long)plane * run_bytes;
        const int base = s_off[i] - s_off[b0], room = min(s_off[i + 1] - s_off[i], kGatherListCap - base);
        int pos = 0;
        for (int t0 = 0; t0 < p.kappa; t0 += 32) {
          const int t = t0 + lane;
          int tok = 0;
          bool hit = false;
          if (t < p.kappa) {
            tok = p.kept_store[(long long)f * p.kappa + t];
            hit = super_patch_index(tok, p.P, p.grid_width, p.patch_split) == sp;
          }
          const unsigned bal = __ballot_sync(kFull, hit);
          const int at = pos + __popc(bal & ((1u << lane) - 1u));
          if (hit && at < room) {
            s_src[base + at] = page + (long long)t * row_bytes;
            if (plane == 0 && meta) { meta[(s_off[i] + at) * 2] = f; meta[(s_off[i] + at) * 2 + 1] = tok; }
          }
          pos += __popc(bal);
        }
        // (a block with fewer rows than its count says, which a consistent store never has, repeats its first row)
        for (int at = pos + lane; at < room; at += 32) s_src[base + at] = page;
      }
      __syncthreads();
      const int nvec = min(s_off[b1] - s_off[b0], kGatherListCap) * vpr;
      unsigned char* dst = dplane + (long long)s_off[b0] * row_bytes;
      int v = threadIdx.x;
      for (; v + 3 * 256 < nvec; v += 4 * 256) {
        uint4 x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int vv = v + k * 256;
          x[k] = ld_stream(p.store + s_src[vv / vpr] + ((long long)(vv % vpr) << 4));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) st_stream(dst + ((long long)(v + k * 256) << 4), x[k]);
      }
      for (; v < nvec; v += 256)
        st_stream(dst + ((long long)v << 4), ld_stream(p.store + s_src[v / vpr] + ((long long)(v % vpr) << 4)));
      __syncthreads();                                     // the list is rewritten by the next batch
      b0 = b1;
    }
    __syncthreads();
  }
}

}  // namespace mukv
