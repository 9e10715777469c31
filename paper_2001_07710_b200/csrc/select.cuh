// Which mask of the library keeps most of a kernel's energy, and that energy (pattern selection, Section 4.1 / 5.1).
#pragma once
#include "common.cuh"

namespace pat {

// The exact answer: energies of all masks in fp64.
__device__ inline int best_mask_exact(const float* __restrict__ wk, const MaskTable& lib, double& best_e) {
  double sq[9];
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const double v = (double)wk[b];
    sq[b] = v * v;
  }
  best_e = -1.0;
  int best = 0;
  for (int j = 0; j < lib.K; ++j) {
    const unsigned m = lib.m[j];
    double e = 0.0;
#pragma unroll
    for (int b = 0; b < 9; ++b)
      if (m & (1u << b)) e += sq[b];
    if (e > best_e) { best_e = e; best = j; }
  }
  return best;
}

// The same by a whole warp for one kernel (the answer in every lane): the masks are spread over the lanes.
__device__ inline int best_mask_exact_warp(const float* __restrict__ wk, const MaskTable& lib) {
  double sq[9];
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const double v = (double)wk[b];
    sq[b] = v * v;
  }
  double best_e = -1.0;
  int best = 0x7FFFFFFF;
  for (int j = threadIdx.x & 31; j < lib.K; j += 32) {
    const unsigned m = lib.m[j];
    double e = 0.0;
#pragma unroll
    for (int b = 0; b < 9; ++b)
      if (m & (1u << b)) e += sq[b];
    if (e > best_e) { best_e = e; best = j; }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double oe = __shfl_xor_sync(0xFFFFFFFFu, best_e, off);
    const int oj = __shfl_xor_sync(0xFFFFFFFFu, best, off);
    if (oe > best_e || (oe == best_e && oj < best)) { best_e = oe; best = oj; }
  }
  return best == 0x7FFFFFFF ? 0 : best;          // (no comparison succeeds when an energy is not a number)
}

constexpr float kLead = 1.0f + 3.814697265625e-6f;     // 1 + 2^-18: an fp32 winner that leads by more is the exact one
constexpr float kFloor = 7.8886090522101181e-31f;      // 2^-100

// The best mask of the kernel whose nine fp32 weights wk holds (lowest id on ties) by its energy: squares of fp32 values
// are exact in fp64 and are added in ascending bit order, so the value is the same bits on any IEEE machine.
//
// The argmax is first taken in fp32.  Nine squares and a sum of at most nine non-negative terms carry a relative
// error below 2^-20 (nine roundings of 2^-24 each) as long as nothing overflows and the result is far above the
// subnormal range, so an fp32 winner that leads the runner-up by a factor of more than 1 + 2^-18 is the exact winner
// too.  Every other case - a lead inside the error bound (exact ties among them), a tiny, huge or non-finite energy -
// takes the exact path over all masks.  The winner's energy itself is always computed exactly.
// Returns -1 when the exact path has to decide.
__device__ inline int best_mask_fast(const float* __restrict__ wk, const MaskTable& lib) {
  float sqf[9];
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const float v = wk[b];
    sqf[b] = __fmul_rn(v, v);
  }
  float best32 = -1.0f, second32 = -1.0f;
  int best = 0;
  bool plain = true;                       // every fp32 energy is an ordinary finite number
#pragma unroll 4                           // (projection of 512 x 512 kernels, 126 masks: 62.8 -> 60.5 us)
  for (int j = 0; j < lib.K; ++j) {
    const unsigned m = lib.m[j];
    float e = 0.0f;
#pragma unroll
    for (int b = 0; b < 9; ++b)
      if (m & (1u << b)) e = __fadd_rn(e, sqf[b]);
    plain = plain && (e <= 3.0e38f);       // false for NaN and infinity
    if (e > best32) { second32 = best32; best32 = e; best = j; }
    else if (e > second32) second32 = e;   // e == best32 lands here: a tie is never a clear lead
  }
  const bool clear = plain && best32 >= kFloor && best32 > second32 * kLead;
  return clear ? best : -1;
}

// The best mask and its exact energy.
__device__ inline int best_mask(const float* __restrict__ wk, const MaskTable& lib, double& best_e) {
  const int best = best_mask_fast(wk, lib);
  if (best < 0) return best_mask_exact(wk, lib, best_e);
  best_e = 0.0;
  unsigned m = lib.m[best];
  while (m) {                              // ascending bit order
    const double v = (double)wk[__ffs(m) - 1];
    best_e += v * v;                       // the square of an fp32 value is exact in fp64
    m &= m - 1u;
  }
  return best;
}

// The same argmax over the full library of all 126 four-entry masks: the four largest squares.  Returns the winning mask (nine
// bits), or 0 when the exact path has to decide: no clear lead over the runner-up, which has the fifth largest square in
// place of the fourth, or an energy that is not an ordinary number.  Positions travel in the low four bits of the squares,
// which makes them wrong by less than 2^-19, so the lead has to be more than 1 + 2^-16.
__device__ __forceinline__ unsigned best_of_full_library(const float* __restrict__ wk) {
  unsigned v[9];
  float total = 0.0f;
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const float s = __fmul_rn(wk[b], wk[b]);
    total += s;
    v[b] = (__float_as_uint(s) & ~15u) | (unsigned)b;      // non-negative floats order like their bits
  }
  // the five largest to the front: five passes of a selection by exchanges (30 of them; their order does not matter inside)
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = 8; j > i; --j) {
      const unsigned hi = max(v[j - 1], v[j]), lo = min(v[j - 1], v[j]);
      v[j - 1] = hi;
      v[j] = lo;
    }
  const float top3 = __uint_as_float(v[0] & ~15u) + __uint_as_float(v[1] & ~15u) + __uint_as_float(v[2] & ~15u);
  const float best = top3 + __uint_as_float(v[3] & ~15u), second = top3 + __uint_as_float(v[4] & ~15u);
  const bool clear = total <= 3.0e38f && best >= kFloor && best > second * (1.0f + 1.52587890625e-5f);
  return clear ? (1u << (v[0] & 15u)) | (1u << (v[1] & 15u)) | (1u << (v[2] & 15u)) | (1u << (v[3] & 15u)) : 0u;
}

}  // namespace pat
