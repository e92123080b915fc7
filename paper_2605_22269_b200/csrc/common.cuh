// Shared device helpers of the MuKV kernels (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/mukv.h"

namespace mukv {

constexpr int kWarp = 32;
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- element access
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

template <typename T> struct ElemTraits;
template <> struct ElemTraits<__nv_bfloat16> {
  static constexpr int kPerWord = 2;      // elements in one 32-bit word
  static constexpr int kPad = 2;          // row padding (elements) that makes the word stride odd
};
template <> struct ElemTraits<float> {
  static constexpr int kPerWord = 1;
  static constexpr int kPad = 1;
};

template <typename T> __device__ __forceinline__ float elem_to_float(T x);
template <> __device__ __forceinline__ float elem_to_float<float>(float x) { return x; }
template <> __device__ __forceinline__ float elem_to_float<__nv_bfloat16>(__nv_bfloat16 x) {
  return __bfloat162float(x);
}

// acc += q.k over the elements packed in one 32-bit word
template <typename T> __device__ __forceinline__ float dot_word(uint32_t q, uint32_t k, float acc);
template <> __device__ __forceinline__ float dot_word<__nv_bfloat16>(uint32_t q, uint32_t k, float acc) {
  acc = fmaf(bf16_lo(q), bf16_lo(k), acc);
  return fmaf(bf16_hi(q), bf16_hi(k), acc);
}
template <> __device__ __forceinline__ float dot_word<float>(uint32_t q, uint32_t k, float acc) {
  return fmaf(__uint_as_float(q), __uint_as_float(k), acc);
}

// C += A B on the double-precision tensor-core instruction, 8 x 8 x 4: lane l holds A[l / 4][l % 4], B[l % 4][l / 4] and
// C[l / 4][2 (l % 4)], C[l / 4][2 (l % 4) + 1].  Measured: 64 multiply-adds per clock and SM, as its larger shapes and as
// plain double-precision multiply-adds, with a quarter of the operands to fetch and convert.
__device__ __forceinline__ void dmma_m8n8k4(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}

// order-preserving bits of a double and back
__device__ __forceinline__ unsigned long long order_key(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double order_key_inv(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
  return __longlong_as_double((long long)b);
}

// ---------------------------------------------------------------- warp / block reductions
template <typename A> __device__ __forceinline__ A warp_sum(A v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
template <typename A> __device__ __forceinline__ A warp_max(A v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    A u = __shfl_xor_sync(kFull, v, o);
    v = u > v ? u : v;
  }
  return v;
}
template <typename A> __device__ __forceinline__ A warp_min(A v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    A u = __shfl_xor_sync(kFull, v, o);
    v = u < v ? u : v;
  }
  return v;
}

// Exclusive prefix count of `flag` over the block in thread order, plus the block's total.
// scratch: at least (threads / 32 + 1) ints of shared memory.  Contains two barriers.
__device__ __forceinline__ int block_excl_count(bool flag, int* scratch, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = ((int)blockDim.x + 31) >> 5;
  const unsigned b = __ballot_sync(kFull, flag);
  const int in_warp = __popc(b & ((1u << lane) - 1u));
  __syncthreads();                       // scratch may still be read from a previous call
  if (lane == 0) scratch[warp] = __popc(b);
  __syncthreads();
  int before = 0, sum = 0;
  for (int w = 0; w < nwarp; ++w) {
    const int c = scratch[w];
    if (w < warp) before += c;
    sum += c;
  }
  total = sum;
  return before + in_warp;
}

// Programmatic dependent launch: a kernel launched with the programmatic-serialisation attribute may
// start while its predecessor in the stream still runs; pdl_wait() returns once that predecessor
// has completed and its writes are visible (a no-op for a normally launched kernel), pdl_trigger()
// tells the runtime that this block no longer minds the successor being scheduled.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// super patch (row-major, split x split) of token id j in a frame of P tokens laid out as a grid
// with grid_width tokens per row: rectangles of ceil(rows/split) x ceil(grid_width/split) tokens
__device__ __forceinline__ int super_patch_index(int j, int P, int grid_width, int split) {
  const int rows = P / grid_width;
  const int rh = (rows + split - 1) / split, cw = (grid_width + split - 1) / split;
  return (j / grid_width) / rh * split + (j % grid_width) / cw;
}

// Column sums of the softmax (Eq. 1), as the blocks of the persistent scoring kernel add them up: 23.40 fixed point in 64
// bits, so that the result does not depend on the order of the additions.  A column sum is at most the number of query
// rows that see the frame (layers x heads x tokens: 2^20 at the supported shapes).  Bit 63 marks a share that is not a
// number.
// A share is rounded to 2^-40, at most 256 blocks share a frame: a sum is off by 2^-33 at the most.  Eq. 4 divides by
// the range of the frame's sums, so a range below kAttFine = 2^-10 sends the frame to the double-precision pass; above it the
// rounding stays below 2^-23 of the range.  Without past keys the sums of a frame reach layers x heads at least, and the
// test for a flat signal flags such a frame already; with them a strong cached key can leave the frame's own columns next
// to nothing (at e^-30 of the mass every share rounds to 0).
constexpr float kAttFine = 1.f / 1024.f;
constexpr unsigned long long kAttPoison = 1ull << 63;
__device__ __forceinline__ void att_add(unsigned long long* acc, float v) {
  if (!(v < 1e30f)) atomicOr(acc, kAttPoison);
  else if (v > 0.f) atomicAdd(acc, __float2ull_rn(v * 1099511627776.f));
}
__device__ __forceinline__ float att_value(unsigned long long acc) {
  return (acc & kAttPoison) ? __int_as_float(0x7fffffff) : __ull2float_rn(acc) * (1.f / 1099511627776.f);
}

// sum of n doubles `stride` apart, added in order, sixteen loads in flight (one after the other each is a round trip to L2)
__device__ __forceinline__ double ordered_sum(const double* p, int n, long long stride) {
  double t = 0.0;
#pragma unroll 1
  for (int i0 = 0; i0 < n; i0 += 16) {
    double x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = i0 + i < n ? __ldcg(p + (i0 + i) * stride) : 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) t += x[i];
  }
  return t;
}

// ---------------------------------------------------------------- segment entries (Eq. 5 at segment level)
// What the pooling of segment entries needs, small enough to travel in registers (compact_segment_plane
// is kept out of line so that its 32 loads in flight do not set the register count of the kernels that
// call it; a reference to a kernel's parameter block would force a per-thread copy of the block instead).
struct SegmentArgs {
  int L, kappa, C, fseg, n_frames;
  long long first_frame;
  const float* frame_entry;
  const double* frame_ksum;
  float* seg_entry;
  float* seg_key;
  const int* kept_count;          // [max_frames] tokens kept per frame, or null: kappa in every frame
};

// 16-byte streaming copies
__device__ __forceinline__ uint4 ld_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ void st_stream(void* p, const uint4& v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

}  // namespace mukv
