// The double-precision scoring pass (Sec. 3.3, Eq. 1-4): frames whose selection single precision cannot decide, and
// whatever ranks whole segments in double precision.
//
// score64_frame_block<T>: one block of 256 threads scores some of the query rows of one head.  Eq. 1 and the DFT of
// Eq. 2-3 are products on the double-precision tensor-core instruction, operands converted exactly in registers.  A block
// takes its query rows eight at a time; each of the eight warps owns an eighth of the key columns, in tiles of eight, reads them
// from global memory (a key head of 50 KB stays in L1), keeps their column sums in registers over the row tiles and exchanges
// (maximum, sum) with the others once per row tile.
// Bound by the fp64 tensor instruction and the conversions: the 138 M multiply-adds of a frame of 28 heads x 196 tokens x 128
// channels are 7.6 us of the whole device; a flagged frame takes a call 75 us all the same, most of it code that comes from device
// memory.  (One multiply-add per lane and 32-bit word out of shared memory, with a conversion for each: 130 us.)  No more
// than 80 registers and no dynamic shared memory, so that the blocks of this pass can be blocks of compact_kernel: as a launch of
// its own behind every call it cost the calls that flag nothing 1 to 2 us (sixteen calls of one frame 297 us, now 271).
#pragma once
#include "common.cuh"
#include "score.cuh"

namespace mukv {

constexpr int kScore64Tiles = 4;          // key tiles of a warp at most: 256 keys / 8 / 8 warps

struct Score64Scratch {
  double2 tw[128];                        // cos, sin of 2 pi d / D
  double2 xch[2][8][8];                   // [parity][warp][row] (maximum, sum)
  double dft[8][8];                       // [warp][row]
  FinishScratch fin;
};

// element e of the 16 bytes in x, exactly
template <typename T>
__device__ __forceinline__ double elem64(const uint4& x, int e) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
  if constexpr (sizeof(T) == 2) return (double)((e & 1) ? bf16_hi(w[e >> 1]) : bf16_lo(w[e >> 1]));
  else return (double)__uint_as_float(w[e]);
}

// (Out of line, like the other long pieces of this pass: it runs for one call in fifty, and its instructions come from device
// memory then, a microsecond for every two or three hundred bytes in a row.)
__device__ __noinline__ double exp64(double x) { return exp(x); }

// The work of one block: part q (of RS) of the query rows of head hv of frame f (a frame slot of the chunk); hv counts the
// query heads of all scoring layers, layer-major.  The partial sums go to place sf of colsum [places][heads * RS][P] and ifft
// [places][key heads][P].  The block that finishes a frame last selects, unless no_select.  (Out of line: one copy for all that
// call it.  Their parameter blocks are __grid_constant__, so that the reference needs no copy.)
template <typename T>
__device__ __noinline__ void score64_frame_block(const ScoreParams& p, double* colsum, double* ifft, int hv, int q, int RS, int f,
                                                 int sf, Score64Scratch* sc) {
  constexpr int VE = 16 / sizeof(T);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int P = p.P, D = p.D, Hq = p.Hq, Hkv = p.Hkv, G = p.G;
  const int layer = hv / Hq, h = hv - layer * Hq, g = h / G;
  const int HqV = p.Ls * Hq, HkvV = p.Ls * Hkv;
  const int KB = D * (int)sizeof(T) / 64;                  // blocks of 64 bytes of a row: 16 bytes per lane of a quad
  const int fr = lane >> 2, fk = lane & 3;                 // fragment row (or column), place in the quad
  const int n_past = p.n_past_frames * p.kappa, Pk = n_past + P;   // key rows: the past keys first

  // key rows: the kept keys of the past frames (this layer's K plane of their pages), then the frame's own
  const T* Kg = reinterpret_cast<const T*>(p.k_last) + layer * p.k_layer_stride + ((long long)f * P * Hkv + g) * D;
  const long long k_row = (long long)Hkv * D;
  auto key_row = [&](int r) -> const T* {
    if (r >= n_past) return Kg + (long long)(r - n_past) * k_row;
    const T* page = reinterpret_cast<const T*>(p.store + p.page_table[p.past_first + r / p.kappa]);
    return page + ((long long)(p.first_score_layer + layer) * 2 * p.kappa + r % p.kappa) * k_row + g * D;
  };
  if (tid < D) {
    double sn, cs;
    sincospi(2.0 * (double)tid / (double)D, &sn, &cs);
    sc->tw[tid] = make_double2(cs, sn);
  }

  // ---- Eq. 1: column sums of the row softmax
  const unsigned char* Qh = reinterpret_cast<const unsigned char*>(
      reinterpret_cast<const T*>(p.q) + layer * p.q_layer_stride + ((long long)f * P * Hq + h) * D);
  const long long q_row = (long long)Hq * D * sizeof(T);
  const double scale = 1.0 / sqrt((double)D);
  const int n_ct = (Pk + 7) >> 3, ct_rem = n_ct & 7;
  const int ct0 = warp * (n_ct >> 3) + min(warp, ct_rem), my = (n_ct >> 3) + (warp < ct_rem ? 1 : 0);
  const T* krow[kScore64Tiles];
#pragma unroll
  for (int t = 0; t < kScore64Tiles; ++t) krow[t] = key_row(min((ct0 + t) * 8 + fr, Pk - 1)) + fk * VE;
  double csum[kScore64Tiles][2];
#pragma unroll
  for (int t = 0; t < kScore64Tiles; ++t) csum[t][0] = csum[t][1] = 0.0;
  const int n_rt = (P + 7) >> 3, n_per = (n_rt + RS - 1) / RS;
  const int rt_end = min((q + 1) * n_per, n_rt);
  int par = 0;
  for (int rt = q * n_per; rt < rt_end; ++rt, par ^= 1) {
    double acc[kScore64Tiles][2];
#pragma unroll
    for (int t = 0; t < kScore64Tiles; ++t) acc[t][0] = acc[t][1] = 0.0;
    const unsigned char* qrow = Qh + (long long)min(rt * 8 + fr, P - 1) * q_row + fk * 16;
    uint4 xa = __ldg(reinterpret_cast<const uint4*>(qrow));
    uint4 xb[kScore64Tiles];
#pragma unroll
    for (int t = 0; t < kScore64Tiles; ++t) xb[t] = t < my ? __ldg(reinterpret_cast<const uint4*>(krow[t])) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
    for (int kb = 0; kb < KB; ++kb) {
      // k step s takes channel s of every lane's sixteen bytes, for both operands; the next sixteen are on their way
      const int nb = kb + 1 < KB ? kb + 1 : 0;
      const uint4 ya = xa;
      xa = __ldg(reinterpret_cast<const uint4*>(qrow + nb * 64));
#pragma unroll
      for (int t = 0; t < kScore64Tiles; t += 2) {         // (two tiles at a time: their additions are independent)
        if (t < my) {
          const uint4 y0 = xb[t], y1 = xb[t + 1];
          xb[t] = __ldg(reinterpret_cast<const uint4*>(krow[t] + nb * 4 * VE));
          if (t + 1 < my) xb[t + 1] = __ldg(reinterpret_cast<const uint4*>(krow[t + 1] + nb * 4 * VE));
#pragma unroll
          for (int s = 0; s < VE; ++s) {
            const double a = elem64<T>(ya, s);
            dmma_m8n8k4(acc[t], a, elem64<T>(y0, s));
            if (t + 1 < my) dmma_m8n8k4(acc[t + 1], a, elem64<T>(y1, s));
          }
        }
      }
    }
    // this lane: row rt*8 + fr, columns (ct0 + t)*8 + 2 fk + e
    const int i = rt * 8 + fr;
    double m = -(double)INFINITY;
#pragma unroll
    for (int t = 0; t < kScore64Tiles; ++t)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int j = (ct0 + t) * 8 + 2 * fk + e;          // past keys are visible to every query
        const bool ok = t < my && j < Pk && (!p.causal || j - n_past <= i);
        acc[t][e] = ok ? acc[t][e] * scale : -(double)INFINITY;
        m = acc[t][e] > m ? acc[t][e] : m;
      }
    __syncwarp();
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const double u = __shfl_xor_sync(kFull, m, o);
      m = u > m ? u : m;
    }
    double l = 0.0;
#pragma unroll
    for (int t = 0; t < kScore64Tiles; ++t) {
      if (t < my) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          acc[t][e] = acc[t][e] == -(double)INFINITY ? 0.0 : exp64(acc[t][e] - m);
          l += acc[t][e];
        }
      }
    }
    __syncwarp();
    l += __shfl_xor_sync(kFull, l, 1);
    l += __shfl_xor_sync(kFull, l, 2);
    double2 (*x)[8] = sc->xch[par];                        // (a copy is rewritten two tiles later, behind the next barrier)
    if (fk == 0) x[warp][fr] = make_double2(m, l);
    __syncthreads();
    double mm = x[0][fr].x;
#pragma unroll
    for (int c = 1; c < 8; ++c) mm = x[c][fr].x > mm ? x[c][fr].x : mm;
    // lane fk of the row takes the shares of two warps
    double sum = 0.0;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const double2 v = x[2 * fk + c][fr];
      sum += v.y * (v.x == -(double)INFINITY ? 1.0 : exp64(v.x - mm));   // (a share without a visible key has the sum 0)
    }
    __syncwarp();
    sum += __shfl_xor_sync(kFull, sum, 1);
    sum += __shfl_xor_sync(kFull, sum, 2);
    const double w = (m == -(double)INFINITY ? 1.0 : exp64(m - mm)) / sum;
#pragma unroll
    for (int t = 0; t < kScore64Tiles; ++t) {
      if (t < my) {
        csum[t][0] = i < P ? fma(acc[t][0], w, csum[t][0]) : csum[t][0];
        csum[t][1] = i < P ? fma(acc[t][1], w, csum[t][1]) : csum[t][1];
      }
    }
    __syncwarp();
  }
  // the eight rows of a lane column, in a fixed order
#pragma unroll
  for (int t = 0; t < kScore64Tiles; ++t) {
    if (t < my) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        double v = csum[t][e];
        v += __shfl_xor_sync(kFull, v, 4);
        v += __shfl_xor_sync(kFull, v, 8);
        v += __shfl_xor_sync(kFull, v, 16);
        const int j = (ct0 + t) * 8 + 2 * fk + e - n_past;  // the importance is that of the frame's own tokens
        if (fr == 0 && j >= 0 && j < P) colsum[(((long long)sf * HqV + hv) * RS + q) * P + j] = v;
      }
    }
  }

  // ---- Eq. 2-3: sum over the D bins of |DFT(k_j)|; the G * RS blocks that hold key head g share its tokens.  Warp w of
  // the first D / 16 takes the real and the imaginary parts of bins 8 w .. 8 w + 7 (bin D/2, which is real, in the imaginary
  // place of bin 0)
  const int half = D >> 1, n_share = G * RS, per = (P + n_share - 1) / n_share;
  const int j0 = ((h % G) * RS + q) * per, j1 = min(j0 + per, P);
  __syncthreads();                                         // the twiddles are there
  for (int jt = j0; jt < j1; jt += 8) {
    if (warp < half / 8) {
      double re[2] = {0.0, 0.0}, im[2] = {0.0, 0.0};
      const T* kr = Kg + (long long)min(jt + fr, j1 - 1) * k_row + fk * VE;
      const int n = warp * 8 + fr;                         // the bin of this lane's matrix entries
      for (int kb = 0; kb < KB; ++kb) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(kr + kb * 4 * VE));
#pragma unroll
        for (int s = 0; s < VE; ++s) {
          const int d = (kb * 4 + fk) * VE + s;
          const double a = elem64<T>(x, s);
          const double2 t = sc->tw[(n * d) & (D - 1)];
          dmma_m8n8k4(re, a, t.x);
          dmma_m8n8k4(im, a, n == 0 ? ((d & 1) ? -1.0 : 1.0) : -t.y);
        }
      }
      double tot = 0.0;
#pragma unroll
      for (int e = 0; e < 2; ++e)
        tot += warp * 8 + 2 * fk + e == 0 ? fabs(re[e]) + fabs(im[e]) : 2.0 * sqrt(re[e] * re[e] + im[e] * im[e]);
      __syncwarp();
      tot += __shfl_xor_sync(kFull, tot, 1);
      tot += __shfl_xor_sync(kFull, tot, 2);
      if (fk == 0) sc->dft[warp][fr] = tot;
    }
    __syncthreads();
    if (tid < 8 && jt + tid < j1) {
      double t = 0.0;
      for (int w = 0; w < half / 8; ++w) t += sc->dft[w][tid];
      ifft[((long long)sf * HkvV + layer * Hkv + g) * P + jt + tid] = t;
    }
    __syncthreads();
  }
  finish_frame(p, colsum, ifft, f, sf, hv, RS, true, &sc->fin);
}

// Parts into which the query rows of a head are split: as many as give every one of `blocks` blocks something to do, while
// the scratch has a place for each (rows: P doubles each) and a part a row tile.
__host__ __device__ inline int score64_split(int frames, int heads, int P, int blocks, int rows) {
  const long long units = (long long)frames * heads;
  long long rs = (blocks < rows ? blocks : rows) / (units > 0 ? units : 1);
  if (rs > (P + 7) / 8) rs = (P + 7) / 8;
  return rs < 1 ? 1 : (int)rs;
}

// The pass over the flagged frames (refine: sp.flagged, sp.n_flagged), or, with seg_gate, over the frames of flagged segments,
// or over all: a one-dimensional grid walks the (frame, head, part) units.  With nothing flagged its blocks return at once.
template <typename T>
__global__ void __launch_bounds__(kScoreThreads, 3) score64_kernel(const __grid_constant__ ScoreParams p) {
  __shared__ Score64Scratch sc;
  pdl_wait();
  pdl_trigger();
  double* colsum = reinterpret_cast<double*>(p.colsum_part);
  double* ifft = reinterpret_cast<double*>(p.ifft_part);
  const int heads = p.Ls * p.Hq;
  if (p.refine) {
    const int n = *p.n_flagged, rs = score64_split(n, heads, p.P, gridDim.x, p.scratch_rows), units = heads * rs;
    for (int w = blockIdx.x; w < n * units; w += gridDim.x) {
      const int slot = w / units, u = w - slot * units;
      score64_frame_block<T>(p, colsum, ifft, u / rs, u % rs, rs, p.flagged[slot], slot, &sc);
      __syncthreads();
    }
    return;
  }
  // (the words of 32 segments are read at once: read frame by frame they were 6 us of a call of 16 frames)
  const int units = heads * p.row_split, n_seg = p.seg_gate ? (p.n_frames + p.gate_fseg - 1) / p.gate_fseg : 1;
  const int fseg = p.seg_gate ? p.gate_fseg : p.n_frames, lane = threadIdx.x & 31;
  for (int s0 = 0; s0 < n_seg; s0 += 32) {
    unsigned set = __ballot_sync(kFull, s0 + lane < n_seg && (!p.seg_gate || __ldcg(p.seg_gate + s0 + lane) != 0));
    for (; set; set &= set - 1) {
      const int f0 = (s0 + __ffs(set) - 1) * fseg, nf = min(fseg, p.n_frames - f0);
      for (int w = blockIdx.x; w < nf * units; w += gridDim.x) {
        const int f = f0 + w / units, u = w % units;
        score64_frame_block<T>(p, colsum, ifft, u / p.row_split, u % p.row_split, p.row_split, f, f, &sc);
        __syncthreads();
      }
    }
  }
}

}  // namespace mukv
