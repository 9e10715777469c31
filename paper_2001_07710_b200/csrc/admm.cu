// Primitives of the pattern-selection ADMM (Section 5.1) and of the library extraction (Algorithm 1, Section 5.2),
// batched over all kernels of a layer (or of a network): the training loop around them is not part of this library.
//
//   pat_simplex_project   u = [d - nu 1]_+ with nu the root of 1^T [d - nu 1]_+ = 1 (the proximal step's closed form)
//   pat_argmax_binarize   the one-hot vector closest to z: 1 at argmax_j z_j
//   pat_extract_library   "calculate the pattern distribution, remove the patterns with fewest occurrences"
//
// The first two stream n x K floats in and out once (8 and 4 - 8 bytes per element).  In the projection a vector is shared
// by the lanes of a warp (or of a group of lanes), strided over its entries so that loads and stores cover whole sectors.
#include "common.cuh"
#include "select.cuh"

namespace pat {
namespace {

constexpr int kVecMaxK = 256;              // entries per vector
constexpr int kVecWarps = 8;               // warps per block

// Sums over the L lanes that share a vector (L a power of two, groups aligned): the same bits in every lane of a group.
template <int L, typename T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
  for (int off = L / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

// The root is found without sorting.  g(nu) = sum_j max(d_j - nu, 0) is convex, piecewise linear and decreasing, and
// Newton's step for g(nu) = 1 from a point nu is nu' = (sum of the entries above nu - 1) / (their number): from any
// start with at least one entry above it the steps reach the root in finitely many rounds (after the first step they
// approach it from below and never pass it).  The sets {entries above nu} are nested whatever nu is, so two rounds
// with the same number of entries above nu have the same set, and then nu is the root of that piece: no set has
// to be stored, a round is one pass "compare, add, count" over the entries.  The rounds run in fp32 from a lower
// bound of the root (see the kernel) until the count repeats, then in fp64 from the fp32 result until the count repeats again - usually
// two or three rounds - so the final piece and its root are exact: the sums are exact to about 1e-16 relative (the
// inputs are fp32), and there is one rounding to fp32 at the end.
//
// L lanes share a vector, sixteen entries each (K <= 16 L), so a warp works on 32 / L vectors at once: a round is a
// chain of dependent steps (a sum over the group, a division, a comparison), and what the kernel needs is many such
// chains in flight, not many lanes per chain.  Entry j of a vector sits in lane j % L, slot j / L.  u may be d.  A thread that
// has a vector to itself exchanges nothing and wants registers for it rather than a fifth block per SM (131072 x 16: 16.1 ->
// 13.7 us, 262144 x 12: 17.7 -> 16.9).
constexpr int kVecQ = 16;
template <int L>
__global__ void __launch_bounds__(32 * kVecWarps, L == 1 ? 4 : 5) k_simplex_project(const float* d, long long n, int K, float* u) {
  constexpr int G = 32 / L;                // vectors per warp
  pdl_wait();
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), g = lane / L;
  const long long stride = (long long)gridDim.x * kVecWarps * G;
  const long long first = ((long long)blockIdx.x * kVecWarps + (threadIdx.x >> 5)) * G;
  if (first >= n) return;                  // whole warps leave together
  for (long long base = first; base < n; base += stride) {
    const bool valid = base + g < n;
    const long long i = valid ? base + g : n - 1;       // a group without a vector repeats the last one and stores nothing
    float x[kVecQ];                        // slots beyond K hold the lowest float: never above any nu
    const float* di = d + i * K + sl;
    const int nq = (K - sl + L - 1) / L;   // this lane's entries: slots 0 .. nq - 1
#pragma unroll
    for (int q = 0; q < kVecQ; ++q) x[q] = (q < nq) ? __ldcs(di + L * q) : -3.402823466e38f;
    // Start: for any set S of entries (sum of S - 1) / |S| is at most the root (the root is the largest such value,
    // taken over the sets of the k largest entries), so the largest entry of every lane gives a lower bound that lies
    // close below the root when few entries are active, and at least one entry is above it (the root is below the largest
    // entry).  Rounding may lift it past the root: the first Newton step from there lands below the root again.
    float top = x[0];
#pragma unroll
    for (int q = 1; q < kVecQ; ++q) top = fmaxf(top, x[q]);
    float nu32 = (group_sum<L>(top) - 1.0f) / (float)L;
    if (!(nu32 > -3.402823466e38f)) nu32 = -3.402823466e38f;   // overflow of the sum (or a NaN): start below every entry
    // Counts are kept as floats (exact up to 2^24): a pass is then one comparison and two predicated additions per entry.  (One
    // addition of a pair, the entry and a one, wants 32 registers where these take 16, and spilled 32 - 40 bytes: 262144 vectors
    // of 126, 56 and 24 entries took 74.8, 42.8 and 21.3 us; 63.7, 35.0 and 19.1 like this.)
    float before = -1.0f;
    bool done = false;
    for (int round = 0; round < K + 2; ++round) {       // fp32 rounds
      float s = 0.0f, c = 0.0f;
#pragma unroll
      for (int q = 0; q < kVecQ; ++q)
        if (x[q] > nu32) { s += x[q]; c += 1.0f; }
      s = group_sum<L>(s);
      c = group_sum<L>(c);
      if (!done) {
        if (c == before || c == 0.0f) { done = true; before = c; }   // the set repeats (or rounding has pushed nu past the largest entry)
        else { nu32 = (s - 1.0f) / c; before = c; }
      }
      if (__all_sync(0xFFFFFFFFu, done)) break;          // every vector of the warp is through
    }
    // `before` is now the number of entries above nu32 (when the rounds ended because the count repeated); if that holds
    // for every vector of the warp the first exact round needs no counting pass
    const float known = done ? before : 0.0f;
    const bool skip_first_count = __all_sync(0xFFFFFFFFu, known > 0.0f);
    // Exact rounds.  A float x is above a double nu exactly when it is above nu rounded down to a float, so the sets are
    // formed by fp32 comparisons; only the sum of a set is taken in fp64.  A round: count the entries above the
    // current threshold; the same count as before means the same set, whose root nu already is; otherwise its exact
    // sum gives the next nu.  After the fp32 rounds the first set is usually the final one: one fp64 sum, two counts.
    double nu = (double)nu32;
    float thr = nu32;
    before = -1.0f;
    done = false;
    for (int round = 0; round < K + 4; ++round) {
      float c = known;
      if (round > 0 || !skip_first_count) {
        c = 0.0f;
#pragma unroll
        for (int q = 0; q < kVecQ; ++q)
          if (x[q] > thr) c += 1.0f;
        c = group_sum<L>(c);
      }
      if (!done && c == before) done = true;
      if (__all_sync(0xFFFFFFFFu, done)) break;
      double s = 0.0;
#pragma unroll
      for (int q = 0; q < kVecQ; ++q)
        if (x[q] > thr) s += (double)x[q];
      s = group_sum<L>(s);
      if (!done) {
        if (c == 0.0f) { thr = -3.402823466e38f; before = -1.0f; }   // past the largest entry: start again from all entries (not the padding)
        else { nu = (s - 1.0) / (double)c; thr = __double2float_rd(nu); before = c; }
      }
    }
    if (valid) {
      float* ui = u + i * K + sl;
      // x - nu in fp64 is exact up to one rounding; an entry at or below the threshold is not above nu
#pragma unroll
      for (int q = 0; q < kVecQ; ++q)
        if (q < nq) __stcs(ui + L * q, x[q] > thr ? (float)((double)x[q] - nu) : 0.0f);
    }
  }
}

// Largest entry of every vector, the lowest index among equal ones; optionally the one-hot vector itself.  A block takes tiles
// of consecutive vectors: in and out as whole lines through shared memory (a vector's own lanes would touch pieces of
// sectors: 504-byte rows start anywhere), the maxima found in between, by a warp per vector (K > 32: two warp-wide
// reductions) or a thread per vector.  Several blocks per SM overlap each other's phases.  262144 x 126 with the
// one-hot vectors: 55 -> 48.5 us, 5.5 TB/s; 262144 x 12: 15 -> 6.5 us.
constexpr int kBinThreads = 256, kBinFloats = 4096;       // entries of a tile (at least one vector of up to 256)
__device__ __forceinline__ unsigned ordered(float v) {    // unsigned order = order of the values (finite; -0 = +0)
  const unsigned b = __float_as_uint(v + 0.0f);
  return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
// Q: entries per lane of a warp that shares a vector (0: K <= 32, a thread per vector)
template <int Q>
__global__ void __launch_bounds__(kBinThreads) k_argmax_binarize(const float* z, long long n, int K, int per_tile, FastDiv d_K,
                                                                 unsigned char* index_out, float* onehot_out) {
  __shared__ __align__(16) float s_z[kBinFloats];
  __shared__ uint8_t s_best[kBinFloats];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  pdl_wait();
  for (long long i0 = (long long)blockIdx.x * per_tile; i0 < n; i0 += (long long)gridDim.x * per_tile) {
    const int m = (int)(n - i0 < per_tile ? n - i0 : per_tile), e = m * K;
    const float* src = z + i0 * K;
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
      done = e & ~3;
      float4 v[kBinFloats / 4 / kBinThreads];
#pragma unroll
      for (int q = 0; q < kBinFloats / 4 / kBinThreads; ++q)
        if (4 * (t + q * kBinThreads) < done) v[q] = __ldcs(reinterpret_cast<const float4*>(src) + t + q * kBinThreads);
#pragma unroll
      for (int q = 0; q < kBinFloats / 4 / kBinThreads; ++q)
        if (4 * (t + q * kBinThreads) < done) reinterpret_cast<float4*>(s_z)[t + q * kBinThreads] = v[q];
    }
    for (int q = done + t; q < e; q += kBinThreads) s_z[q] = __ldcs(src + q);
    __syncthreads();
    if constexpr (Q > 0) {
      // four vectors of a warp at once: their reads and reductions overlap
      for (int v0 = 4 * wid; v0 < m; v0 += 4 * (kBinThreads / 32)) {
        unsigned best[4];
        int at[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float* zv = s_z + min(v0 + i, m - 1) * K;
          float x[Q];
#pragma unroll
          for (int q = 0; q < Q; ++q) x[q] = lane + 32 * q < K ? zv[lane + 32 * q] : -INFINITY;
          float top = x[0];
          at[i] = lane;
#pragma unroll
          for (int q = 1; q < Q; ++q)
            if (x[q] > top) { top = x[q]; at[i] = lane + 32 * q; }      // ascending: the first maximum stays
          best[i] = ordered(top);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const unsigned top = __reduce_max_sync(0xFFFFFFFFu, best[i]);
          at[i] = (int)__reduce_min_sync(0xFFFFFFFFu, best[i] == top ? (unsigned)at[i] : 0xFFFFu);
        }
        if (lane < 4 && v0 + lane < m) s_best[v0 + lane] = (uint8_t)(lane == 0 ? at[0] : lane == 1 ? at[1] : lane == 2 ? at[2] : at[3]);
      }
    } else {
      for (int v = t; v < m; v += kBinThreads) {
        const float* zv = s_z + v * K;
        float best = zv[0];
        int at = 0;
        for (int j = 1; j < K; ++j)
          if (zv[j] > best) { best = zv[j]; at = j; }
        s_best[v] = (uint8_t)at;
      }
    }
    __syncthreads();
    for (int v = t; v < m; v += kBinThreads) index_out[i0 + v] = s_best[v];
    if (onehot_out) {
      float* dst = onehot_out + i0 * K;
      auto hot = [&](int q) {
        const int v = d_K.div(q);
        return q - v * K == (int)s_best[v] ? 1.0f : 0.0f;
      };
      int out = 0;
      if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        out = e & ~3;
        for (int q = 4 * t; q < out; q += 4 * kBinThreads) {
          // a piece of four entries lies in one or two vectors when K >= 4: one division serves them all
          const int v = d_K.div(q), r = q - v * K;
          float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (K >= 4) {
            const int at = (int)s_best[v] - r, at2 = r + 4 > K ? (int)s_best[v + 1] + K - r : -1;   // v + 1 < m: q + 3 < out
            o = make_float4(at == 0 ? 1.0f : 0.0f, at == 1 || at2 == 1 ? 1.0f : 0.0f, at == 2 || at2 == 2 ? 1.0f : 0.0f, at == 3 || at2 == 3 ? 1.0f : 0.0f);
          } else {
            o = make_float4(hot(q), hot(q + 1), hot(q + 2), hot(q + 3));
          }
          __stcs(reinterpret_cast<float4*>(dst + q), o);
        }
      }
      for (int q = out + t; q < e; q += kBinThreads) __stcs(dst + q, hot(q));
    }
    __syncthreads();                         // the tile is free again
  }
}

// Pattern distribution: every kernel is given the mask that keeps most of its energy (as in pat_project) and the
// kernels per mask are counted, per block in shared memory first.  The counters are zeroed by a kernel of their own; this
// one is its programmatic dependent and does everything but the last additions before it waits for it.
// FULL: the library is all 126 masks, so the best one holds the four largest squares (the whole call at 262144
// kernels: 67 -> 11.8 us; a loop over 56 masks takes 18.8, so smaller libraries do not need a search of their own).
constexpr int kAssignThreads = 256, kFullK = 126;
__global__ void __launch_bounds__(256) k_zero_counts(unsigned long long* counts, int K) {
  pdl_wait();
  if ((int)threadIdx.x < K) counts[threadIdx.x] = 0ull;
}
// ROUNDS: kernels of a thread.  With one, twice as many blocks end and add their counts to the same few lines: for the full library, whose
// blocks are short, that costs more than it gives once all SMs have several (262144 kernels 16.6 us, 11.8 with two; 196608 13.0,
// 10.4; but 163840 8.9, 10.0 and 4096 6.6, 7.7).  Smaller libraries: one (262144 kernels, 56 masks 18.8, 22.3 with two; 12 masks 8.5, 9.1).
template <bool FULL, int ROUNDS>
__global__ void __launch_bounds__(kAssignThreads) k_assign_count(const float* __restrict__ w, long long n, MaskTable lib,
                                                                 unsigned long long* __restrict__ counts) {
  __shared__ unsigned int s_cnt[kMaxK + 1];
  __shared__ uint8_t s_id[FULL ? 512 : 1];                  // mask -> library id
  __shared__ __align__(16) float s_w[kAssignThreads * 9];
  const int t = threadIdx.x;
  for (int q = t; q <= kMaxK; q += kAssignThreads) s_cnt[q] = 0u;
  if (FULL && t < kFullK) s_id[lib.m[t]] = (uint8_t)t;
  for (int r = 0; r < ROUNDS; ++r) {
    const long long i0 = ((long long)blockIdx.x * ROUNDS + r) * kAssignThreads;
    __syncthreads();
    if (i0 >= n) break;
    const int m = (int)((n - i0 < kAssignThreads ? n - i0 : kAssignThreads) * 9);
    const float* src = w + i0 * 9;
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
      for (int q = t; q < (m >> 2); q += kAssignThreads) reinterpret_cast<float4*>(s_w)[q] = __ldg(reinterpret_cast<const float4*>(src) + q);
      for (int q = (m & ~3) + t; q < m; q += kAssignThreads) s_w[q] = __ldg(src + q);
    } else {
      for (int q = t; q < m; q += kAssignThreads) s_w[q] = __ldg(src + q);
    }
    __syncthreads();
    const bool in = i0 + t < n;
    int j = 0;                               // -1: undecided
    if (FULL) {
      const unsigned m = in ? best_of_full_library(s_w + 9 * t) : 0u;
      j = m ? (int)s_id[m] : -1;
    } else if (in) {
      j = best_mask_fast(s_w + 9 * t, lib);
    }
    if (in && j >= 0) atomicAdd(&s_cnt[j], 1u);
    // the undecided ones, each by the whole warp (one in ten thousand, but as one thread's loop over 126 masks in fp64 it
    // was half of the kernel's time)
    for (unsigned todo = __ballot_sync(0xFFFFFFFFu, in && j < 0); todo; todo &= todo - 1u) {
      const int k = best_mask_exact_warp(s_w + 9 * ((t & ~31) + __ffs(todo) - 1), lib);
      if ((t & 31) == 0) atomicAdd(&s_cnt[k], 1u);
    }
  }
  __syncthreads();
  pdl_wait();                                // the counters are zero
  for (int q = t; q < lib.K; q += kAssignThreads)
    if (s_cnt[q]) atomicAdd(&counts[q], (unsigned long long)s_cnt[q]);
}

// The K_out most frequent masks stay (equal counts: the lower id), in the order they have in the library.  One block:
// thread j ranks mask j among all masks, the survivors are written in id order.
__global__ void __launch_bounds__(256) k_pick_survivors(MaskTable lib, const unsigned long long* counts,
                                                        int K_out, unsigned short* __restrict__ masks_out) {
  pdl_wait();
  __shared__ unsigned long long s_c[kMaxK + 1];
  __shared__ int s_warp[8];
  const int j = threadIdx.x;
  s_c[j] = (j < lib.K) ? counts[j] : 0ull;
  __syncthreads();
  bool stays = false;
  if (j < lib.K) {
    int before = 0;
    const unsigned long long cj = s_c[j];
#pragma unroll 8
    for (int q = 0; q < lib.K; ++q) before += (s_c[q] > cj || (s_c[q] == cj && q < j)) ? 1 : 0;
    stays = before < K_out;
  }
  const unsigned ballot = __ballot_sync(0xFFFFFFFFu, stays);
  const int lane = j & 31, wid = j >> 5;
  if (lane == 0) s_warp[wid] = __popc(ballot);
  __syncthreads();
  int pos = __popc(ballot & ((1u << lane) - 1u));
  for (int q = 0; q < wid; ++q) pos += s_warp[q];
  if (stays) masks_out[pos] = lib.m[j];
}

// Blocks of the vector kernels: enough for eight resident blocks per SM, each warp then walks over its vectors.
unsigned vec_grid(int64_t n, int per_warp = 1) {
  static thread_local DeviceSlot slots[kMaxDevices];
  DeviceSlot* dv = device_slot(slots);
  const long long want = (long long)(dv ? dv->sms : 148) * 8;
  const long long need = (n + (long long)kVecWarps * per_warp - 1) / ((long long)kVecWarps * per_warp);
  return (unsigned)(need < want ? need : want);
}

}  // namespace
}  // namespace pat

using namespace pat;

extern "C" int pat_simplex_project(const float* d, int64_t n, int K, float* u, void* stream) {
  if (n == 0 && K >= 1 && K <= kVecMaxK) return PAT_OK;      // nothing to do (an empty batch may come with null pointers)
  if (!d || !u) return set_error(PAT_ERR_INVALID_ARG, "pat_simplex_project: null pointer");
  if (K < 1 || K > kVecMaxK) return set_error(PAT_ERR_SHAPE, "pat_simplex_project: K=%d outside 1..%d", K, kVecMaxK);
  if (n < 0 || n > 0x7FFFFFFFll * kVecWarps) return set_error(PAT_ERR_SHAPE, "pat_simplex_project: n=%lld out of range", (long long)n);
  if (!aligned(d, 4) || !aligned(u, 4)) return set_error(PAT_ERR_ALIGN, "pat_simplex_project: buffers must be 4-byte aligned");
  if (n == 0) return PAT_OK;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const auto fn = K <= 16 ? k_simplex_project<1> : K <= 32 ? k_simplex_project<2> : K <= 64 ? k_simplex_project<4> : K <= 128 ? k_simplex_project<8> : k_simplex_project<16>;
  const int per_warp = K <= 16 ? 32 : K <= 32 ? 16 : K <= 64 ? 8 : K <= 128 ? 4 : 2;
  const cudaError_t e = launch_dependent(fn, dim3(vec_grid(n, per_warp)), dim3(32 * kVecWarps), 0, st, d, (long long)n, K, u);
  if (e != cudaSuccess) return check_cuda(e, "pat_simplex_project launch");
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pat_simplex_project launch");
}

extern "C" int pat_argmax_binarize(const float* z, int64_t n, int K, uint8_t* index_out, float* onehot_out, void* stream) {
  if (n == 0 && K >= 1 && K <= kVecMaxK) return PAT_OK;
  if (!z || !index_out) return set_error(PAT_ERR_INVALID_ARG, "pat_argmax_binarize: null pointer");
  if (K < 1 || K > kVecMaxK) return set_error(PAT_ERR_SHAPE, "pat_argmax_binarize: K=%d outside 1..%d", K, kVecMaxK);
  if (n < 0 || n > 0x7FFFFFFFll * kVecWarps) return set_error(PAT_ERR_SHAPE, "pat_argmax_binarize: n=%lld out of range", (long long)n);
  if (!aligned(z, 4) || (onehot_out && !aligned(onehot_out, 4))) return set_error(PAT_ERR_ALIGN, "pat_argmax_binarize: buffers must be 4-byte aligned");
  if (n == 0) return PAT_OK;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // tiles of whole vectors; a multiple of four of them keeps every tile as well aligned as the first
  static thread_local DeviceSlot slots[kMaxDevices];
  DeviceSlot* dv = device_slot(slots);
  const long long most = (long long)(dv ? dv->sms : 148) * 8;
  int per_tile = kBinFloats / K;
  if (per_tile > 4) per_tile = per_tile / 4 * 4;
  FastDiv d_K;
  d_K.set(K);
  const long long tiles = (n + per_tile - 1) / per_tile;
  const auto fn = K <= 32 ? k_argmax_binarize<0> : K <= 64 ? k_argmax_binarize<2> : K <= 128 ? k_argmax_binarize<4> : k_argmax_binarize<8>;
  const cudaError_t e = launch_dependent(fn, dim3((unsigned)(tiles < most ? tiles : most)), dim3(kBinThreads), 0, st, z, (long long)n, K, per_tile, d_K, index_out, onehot_out);
  if (e != cudaSuccess) return check_cuda(e, "pat_argmax_binarize launch");
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pat_argmax_binarize launch");
}

extern "C" int pat_extract_library(const float* w, int64_t n, const uint16_t* masks_in, int K_in, int K_out,
                                   uint16_t* masks_out, uint64_t* counts_out, void* stream) {
  if (!w || !masks_out || !counts_out) return set_error(PAT_ERR_INVALID_ARG, "pat_extract_library: null pointer");
  if (int rc = check_library(masks_in, K_in)) return rc;
  if (K_out < 1 || K_out > K_in) return set_error(PAT_ERR_INVALID_ARG, "pat_extract_library: K_out=%d outside 1..%d", K_out, K_in);
  if (n < 0 || n > 0x7FFFFFFFll * 256) return set_error(PAT_ERR_SHAPE, "pat_extract_library: n=%lld out of range", (long long)n);
  if (!aligned(w, 4) || !aligned(counts_out, 8) || !aligned(masks_out, 2)) return set_error(PAT_ERR_ALIGN, "pat_extract_library: misaligned buffer");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  MaskTable lib;
  for (int j = 0; j <= kMaxK; ++j) lib.m[j] = (j < K_in) ? masks_in[j] : (uint16_t)0;
  lib.K = K_in;
  unsigned long long* counts = reinterpret_cast<unsigned long long*>(counts_out);
  cudaError_t le = launch_dependent(k_zero_counts, dim3(1), dim3(256), 0, st, counts, K_in);
  count_launches(1);
  if (n > 0 && le == cudaSuccess) {
    // 126 distinct masks of four entries are all there are; two kernels a thread from two and a half blocks per SM on (see k_assign_count)
    static thread_local DeviceSlot slots[kMaxDevices];
    DeviceSlot* dv = device_slot(slots);
    const bool full = K_in == kFullK;
    const int rounds = full && 2 * ((n + 2 * kAssignThreads - 1) / (2 * kAssignThreads)) >= 5ll * (dv ? dv->sms : 148) ? 2 : 1;
    const auto fn = !full ? k_assign_count<false, 1> : rounds == 1 ? k_assign_count<true, 1> : k_assign_count<true, 2>;
    const unsigned grid = (unsigned)((n + kAssignThreads * rounds - 1) / (kAssignThreads * rounds));
    le = launch_dependent(fn, dim3(grid), dim3(kAssignThreads), 0, st, w, (long long)n, lib, counts);
    count_launches(1);
  }
  if (le == cudaSuccess)
    le = launch_dependent(k_pick_survivors, dim3(1), dim3(256), 0, st, lib, static_cast<const unsigned long long*>(counts), K_out,
                          reinterpret_cast<unsigned short*>(masks_out));
  count_launches(1);
  if (le != cudaSuccess) return check_cuda(le, "pat_extract_library launch");
  return check_cuda(cudaGetLastError(), "pat_extract_library launch");
}
