// pat_project: per-kernel pattern selection and per-layer connectivity pruning, exact and deterministic.
//
// Pattern pruning multiplies each 3x3 kernel by one mask of the library (Section 4.1); the mask kept is the
// one that retains the largest squared L2 norm, the one-shot form of the argmax binarisation of Section 5.1.
// Connectivity pruning ranks kernels by their L2 norm (Section 6.1) and keeps the n_keep strongest of the layer.
//
// Exactness: squares of fp32 values are exact in fp64 and are added in ascending bit order, so the energies
// are the same bits on any IEEE machine.  The n_keep-th largest energy is found with a radix select over the
// (monotone) bit pattern of the non-negative doubles: a 16-bit digit by a histogram over the whole layer, then the keys
// that share it, by one cluster (k_select_cluster) or, in large layers, another 16-bit histogram and one thread block
// over a list (k_select_rest).  Four launches per layer, each a programmatic dependent of the one before: counters to
// zero, energies, threshold, output.
#include "common.cuh"
#include "select.cuh"

namespace pat {
namespace {

constexpr int kSelBlock = 256;               // kernels per block of the output kernel
constexpr int kBins = 65536;

struct SelectState {
  unsigned long long prefix;   // the threshold key
  unsigned int cut;            // kernels whose key equals the threshold are kept up to this index
  unsigned int pad;
};

// workspace layout
constexpr int kCoarse = 256;                 // coarse histogram: the upper 8 bits of a 16-bit digit
constexpr int kPasses = 2;                   // digits found with histograms over the whole layer (16 bits each)
constexpr size_t kHistWords = (size_t)kPasses * (kBins + kCoarse) + 4;   // one fine + one coarse histogram per pass, then two control words
constexpr int kListKeys = 32768;             // candidate keys kept beside their indices (longer lists look them up)
constexpr size_t kTicketWord = (size_t)kPasses * (kBins + kCoarse);     // hist[kTicketWord]: blocks of the running kernel that are done
constexpr size_t kListWord = kTicketWord + 1;                             // hist[kListWord]: length of the candidate list

struct ProjWs {
  unsigned long long* key;     // [FC] energy bit patterns
  unsigned char* pid;          // [FC] best pattern per kernel
  unsigned int* hist;          // [kPasses][65536 fine | 256 coarse], control words; zeroed by every call
  unsigned long long* cand_key;   // [kListKeys] the first of the keys that share the first digit with the threshold
  unsigned int* cand;          // [FC] indices of all of them, in the same (any) order
  SelectState* st;
  size_t bytes;
};

__device__ __forceinline__ bool aligned_dev(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

constexpr size_t ws_align(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t ws_bytes(int64_t FC) {
  return ws_align(8 * (size_t)FC) + ws_align((size_t)FC) + ws_align(4 * kHistWords) + ws_align(8 * (size_t)kListKeys) +
         ws_align(4 * (size_t)FC) + ws_align(sizeof(SelectState));
}

inline ProjWs carve(void* base, int64_t FC) {
  ProjWs w;
  char* p = static_cast<char*>(base);
  size_t o = 0;
  w.key = reinterpret_cast<unsigned long long*>(p + o); o += ws_align(8 * (size_t)FC);
  w.pid = reinterpret_cast<unsigned char*>(p + o);      o += ws_align((size_t)FC);
  w.hist = reinterpret_cast<unsigned int*>(p + o);      o += ws_align(4 * kHistWords);
  w.cand_key = reinterpret_cast<unsigned long long*>(p + o); o += ws_align(8 * (size_t)kListKeys);
  w.cand = reinterpret_cast<unsigned int*>(p + o);      o += ws_align(4 * (size_t)FC);
  w.st = reinterpret_cast<SelectState*>(p + o);         o += ws_align(sizeof(SelectState));
  w.bytes = o;
  return w;
}

// The selection kernels end with a step that needs the work of all their blocks (choosing the digit from the
// complete histogram, finishing the selection on the candidate list).  Instead of a launch of its own that step is done by
// whichever block finishes last: every block publishes its results, takes a ticket, and the block that draws the
// last ticket (which also puts the counter back to zero for the next kernel) goes on.  Returns true in every thread
// of that block; its reads of the other blocks' results must bypass L1 (__ldcg).
// One fence per block, not per thread: the block barrier orders every thread's writes and atomics before thread 0's
// fence, and a fence is cumulative - what thread 0 has observed is visible device-wide before its ticket is.  (A
// fence in every thread made each of them wait for its own atomics to return; with a quarter of a million threads
// that wait was most of the kernel.)
__device__ inline bool last_block_done(unsigned int* ticket) {
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// Histogram of one 16-bit digit (fine: all 16 bits, coarse: its upper 8 bits).  Identical digits inside a warp are
// merged into one atomic.  Called by all threads of a warp; `in` = this thread takes part.
__device__ inline void hist_add(unsigned int* fine, unsigned int* coarse, bool in, unsigned d) {
  const unsigned active = __ballot_sync(0xFFFFFFFFu, in);
  if (in) {
    const int lane = threadIdx.x & 31;
    const unsigned same = __match_any_sync(active, d);
    if ((int)(__ffs(same) - 1) == lane) atomicAdd(&fine[d], (unsigned)__popc(same));
    const unsigned same_c = __match_any_sync(active, d >> 8);
    if ((int)(__ffs(same_c) - 1) == lane) atomicAdd(&coarse[d >> 8], (unsigned)__popc(same_c));
  }
}

// Inclusive scan over the threads of a block (any size up to 1024; warp_tot: 32 words), thread 0 first.
__device__ inline unsigned long long block_scan_256(unsigned long long v, unsigned long long* warp_tot) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, v, off);
    if (lane >= off) v += u;
  }
  if (lane == 31) warp_tot[wid] = v;
  __syncthreads();
  unsigned long long add = 0;
  for (int q = 0; q < wid; ++q) add += warp_tot[q];
  __syncthreads();
  return v + add;
}

// Finds the digit d with  count(digit > d) < rem <= count(digit >= d), first in the coarse histogram, then among the
// 256 fine bins of the coarse bin found.  Called by a whole block, done by its first warp (eight bins a lane, shuffles: a
// scan over the block's warps took longer than the two reads).  Returns the digit in every thread and takes the keys above
// it off `rem`.  Counts fit 32 bits: a layer has fewer than 2^32 kernels.
__device__ inline unsigned pick_digit(const unsigned int* hist, int pass, unsigned long long& rem) {
  __shared__ unsigned s_digit, s_rest;
  const unsigned int* fine = hist + (size_t)pass * (kBins + kCoarse);
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    unsigned want = (unsigned)rem, digit = 0u;
#pragma unroll
    for (int level = 0; level < 2; ++level) {
      const unsigned int* bins = level == 0 ? fine + kBins : fine + 256u * digit;
      const int top = 255 - 8 * lane;          // the lane's bins: top, top - 1, .. top - 7
      const uint4 lo = __ldcg(reinterpret_cast<const uint4*>(bins + top - 7)), hi = __ldcg(reinterpret_cast<const uint4*>(bins + top - 3));
      const unsigned c[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
      unsigned sum = 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q) sum += c[q];
      unsigned above = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, above, off);
        if (lane >= off) above += u;
      }
      above -= sum;                            // keys in higher bins than this lane's
      unsigned found = 0u, rest = want;        // defined values even if no bin qualifies (a histogram that misses keys)
      const bool mine = want > above && want <= above + sum;
      if (mine) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (want > above && want <= above + c[q]) { found = (unsigned)(top - q); rest = want - above; }
          above += c[q];
        }
      }
      const unsigned who = __ballot_sync(0xFFFFFFFFu, mine);
      const int from = who ? __ffs(who) - 1 : 0;
      found = __shfl_sync(0xFFFFFFFFu, found, from);
      want = __shfl_sync(0xFFFFFFFFu, rest, from);
      digit = level == 0 ? found : 256u * digit + found;
    }
    if (lane == 0) { s_digit = digit; s_rest = want; }
  }
  __syncthreads();
  rem = s_rest;
  return s_digit;
}

// The counters of a call: both histograms and the two control words behind them.
constexpr int kZeroThreads = 256;
__global__ void __launch_bounds__(kZeroThreads) k_zero_counters(unsigned int* hist, int words) {
  pdl_wait();
  const int i = ((int)blockIdx.x * kZeroThreads + (int)threadIdx.x) * 4;
  if (i < words) *reinterpret_cast<uint4*>(hist + i) = make_uint4(0u, 0u, 0u, 0u);
}

// One kernel per thread: energies of all masks, argmax (lowest id on ties); histogram of the first digit of the
// energies' bit patterns.  do_select = false (everything or nothing is kept): pattern ids only.  A block's weights pass
// through shared memory, so that they are read as whole lines (nine strided reads a thread took half of the kernel).
//
// The first digit (sign, exponent, four mantissa bits) takes only a few dozen values in a layer, so its histogram is
// collected per block in shared memory and flushed with one global atomic per distinct value and block: atomics
// from a quarter of a million threads on those few addresses took longer than the rest of the projection.
//
// The energies are computed before the wait for the kernel that zeroes the counters: that one is launched as a dependent
// too and lets this one start only after its own wait, so whatever came before the call is complete.
constexpr int kPatBlock = 512;
constexpr int kSelSlots = 256;               // shared-memory counters, indexed by the digit's low bits and tagged with the digit
static_assert(kSelSlots == kCoarse && kPatBlock >= kCoarse, "one counter of each kind per thread of the first 256");
__global__ void __launch_bounds__(kPatBlock) k_select_pattern(const float* w, int64_t FC, MaskTable lib,
                                                              unsigned long long* __restrict__ key, unsigned char* __restrict__ pid,
                                                              unsigned int* hist, bool do_select) {
  if (!do_select) pdl_wait();                // no kernel of this call before this one
  __shared__ __align__(16) float s_w[kPatBlock * 9];
  __shared__ unsigned int s_tag[kSelSlots], s_cnt[kSelSlots], s_coarse[kCoarse];
  const int t = threadIdx.x;
  if (t < kSelSlots) { s_tag[t] = 0u; s_cnt[t] = 0u; s_coarse[t] = 0u; }
  const int64_t i0 = (int64_t)blockIdx.x * kPatBlock, i = i0 + t;
  const int n = (int)((FC - i0 < kPatBlock ? FC - i0 : kPatBlock) * 9);
  const float* src = w + i0 * 9;
  if (aligned_dev(src, 16)) {
    const int n4 = n >> 2;
    for (int q = t; q < n4; q += kPatBlock) reinterpret_cast<float4*>(s_w)[q] = reinterpret_cast<const float4*>(src)[q];
    for (int q = 4 * n4 + t; q < n; q += kPatBlock) s_w[q] = src[q];
  } else {
    for (int q = t; q < n; q += kPatBlock) s_w[q] = src[q];
  }
  __syncthreads();
  const bool in = i < FC;
  unsigned long long k = 0ull;
  if (in) {
    double best_e;
    const int best = best_mask(s_w + t * 9, lib, best_e);
    k = (unsigned long long)__double_as_longlong(best_e);   // e >= +0: bit pattern is monotone
    key[i] = k;
    pid[i] = (unsigned char)best;
  }
  if (!do_select) return;
  pdl_wait();                                // the counters are zero
  // identical digits inside the warp are merged first; the lane that speaks for a digit adds to the block's counters
  const unsigned d = (unsigned)(k >> 48);
  const unsigned active = __ballot_sync(0xFFFFFFFFu, in);
  if (in) {
    const int lane = t & 31;
    const unsigned same = __match_any_sync(active, d);
    if ((int)(__ffs(same) - 1) == lane) {
      const unsigned m = (unsigned)__popc(same);
      const unsigned slot = d & (unsigned)(kSelSlots - 1);
      const unsigned old = atomicCAS(&s_tag[slot], 0u, d + 1u);
      if (old == 0u || old == d + 1u) atomicAdd(&s_cnt[slot], m);
      else atomicAdd(&hist[d], m);           // the slot belongs to another digit: straight to the global histogram
      atomicAdd(&s_coarse[d >> 8], m);
    }
  }
  __syncthreads();
  if (t < kSelSlots) {
    if (s_cnt[t]) atomicAdd(&hist[s_tag[t] - 1u], s_cnt[t]);
    if (s_coarse[t]) atomicAdd(&hist[kBins + t], s_coarse[t]);
  }
}

// Among 256 counters (one per thread of the first 256; the others pass 0), the bin where the running count - taken
// from the highest bin down (DESCENDING) or from the lowest bin up - first reaches `rem`.  Returns the bin and sets
// `before` to the count of the bins passed on the way.  All threads of the block call it; `cnt` is this thread's bin
// (thread t owns bin 255 - t when descending, bin t otherwise).
template <bool DESCENDING>
__device__ inline int pick_bin_256(unsigned long long cnt, unsigned long long rem, unsigned long long* warp_tot,
                                   unsigned long long& before) {
  __shared__ int s_bin;
  __shared__ unsigned long long s_before;
  if (threadIdx.x == 0) { s_bin = 0; s_before = 0ull; }
  __syncthreads();
  const unsigned long long incl = block_scan_256(cnt, warp_tot);
  if (threadIdx.x < 256 && rem > incl - cnt && rem <= incl) { s_bin = DESCENDING ? 255 - (int)threadIdx.x : (int)threadIdx.x; s_before = incl - cnt; }
  __syncthreads();
  before = s_before;
  const int bin = s_bin;
  __syncthreads();                           // the shared results may be overwritten by the next call
  return bin;
}

// Threshold of larger layers.  All blocks: the first digit from its histogram (each block for itself: a launch or a ticket to do it once
// costs more than the two reads and scans), histogram of the second 16-bit digit over the keys whose first digit is the
// threshold's, and a list of those keys' indices (any order).  The last block picks the second digit
// and then works alone: it gathers from the list the keys that agree with the threshold in both digits - a handful
// for ordinary weights, which are ranked directly in shared memory.  If there are more than fit there (weights with
// few distinct values), it finds the remaining 32 bits of the threshold in four 8-bit passes over the list with a
// histogram in shared memory and then, among the keys equal to the threshold, the index below which `remaining` of
// them lie (four more passes, over the index bits).  Kernels whose key equals the threshold are kept in index order.
constexpr int kRestThreads = 1024;
constexpr int kShortList = 1536;
__global__ void __launch_bounds__(kRestThreads) k_select_rest(const unsigned long long* __restrict__ key, int64_t FC,
                                                              SelectState* st, long long n_keep, unsigned int* hist,
                                                              unsigned long long* cand_key, unsigned int* cand) {
  pdl_wait();
  __shared__ unsigned long long warp_tot[32];
  __shared__ unsigned int s_hist[256];
  __shared__ unsigned long long s_key[kShortList];
  __shared__ unsigned int s_idx[kShortList];
  __shared__ unsigned int s_n;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool in = i < FC;
  const unsigned long long my_key = in ? __ldcg(key + i) : 0ull;
  unsigned long long rem = (unsigned long long)n_keep;
  const unsigned long long first = pick_digit(hist, 0, rem);
  in = in && (my_key >> 48) == first;
  const unsigned d = (unsigned)((my_key >> 32) & 0xFFFFull);
  unsigned int* fine = hist + (size_t)(kBins + kCoarse);
  hist_add(fine, fine + kBins, in, d);
  {
    // a place in the list: one atomic per block (the warps' counts are added up in shared memory first)
    __shared__ unsigned int s_wcount[kRestThreads / 32], s_base;
    const unsigned active = __ballot_sync(0xFFFFFFFFu, in);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) s_wcount[wid] = (unsigned)__popc(active);
    __syncthreads();
    if (threadIdx.x < 32) {
      const unsigned c = s_wcount[lane];
      unsigned incl = c;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += u;
      }
      s_wcount[lane] = incl - c;
      if (lane == 31) s_base = incl ? atomicAdd(&hist[kListWord], incl) : 0u;
    }
    __syncthreads();
    if (in) {
      const unsigned pos = s_base + s_wcount[wid] + __popc(active & ((1u << lane) - 1u));
      cand[pos] = (unsigned)i;
      if (pos < (unsigned)kListKeys) cand_key[pos] = my_key;
    }
  }
  if (!last_block_done(hist + kTicketWord)) return;
  const int t = threadIdx.x;
  const unsigned n = __ldcg(&hist[kListWord]);
  if (t == 0) s_n = 0u;
  unsigned long long prefix = (first << 16) | pick_digit(hist, 1, rem);      // 32 bits decided
  // the keys that agree in both digits: read in order from the list (eight reads in flight), their indices only then
  const unsigned n_keys = min(n, (unsigned)kListKeys);
  auto take = [&](unsigned long long k, unsigned j) {
    if ((k >> 32) == prefix) {
      const unsigned pos = atomicAdd(&s_n, 1u);
      if (pos < (unsigned)kShortList) { s_key[pos] = k; s_idx[pos] = __ldcg(cand + j); }
    }
  };
  for (unsigned j0 = t; j0 < n_keys; j0 += 8 * kRestThreads) {
    unsigned long long k[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) k[q] = __ldcg(cand_key + min(j0 + q * kRestThreads, n_keys - 1u));
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (j0 + q * kRestThreads < n_keys) take(k[q], j0 + q * kRestThreads);
  }
  for (unsigned j = n_keys + t; j < n; j += kRestThreads) take(__ldcg(key + __ldcg(cand + j)), j);
  __syncthreads();
  const bool fits = s_n <= (unsigned)kShortList;
  const unsigned m = fits ? s_n : n;
  if (fits) {
    // The kept kernels of the short list are its first `rem` in the order (key descending, index ascending): the
    // entry with rem - 1 others before it carries the threshold and the last kept index.  A handful of entries: every
    // thread ranks its own against all others.
    for (unsigned j = t; j < m; j += kRestThreads) {
      const unsigned long long kj = s_key[j];
      const unsigned ij = s_idx[j];
      unsigned long long before = 0ull;
      for (unsigned q = 0; q < m; ++q) {
        const unsigned long long kq = s_key[q];
        before += (kq > kj || (kq == kj && s_idx[q] < ij)) ? 1ull : 0ull;
      }
      if (before + 1ull == rem) { st->prefix = kj; st->cut = ij; }
    }
    return;
  }
  // more entries than the short list holds (weights with few distinct values): digit by digit over the list itself
  auto entry = [&](unsigned j, unsigned long long& k, unsigned& idx) {
    idx = __ldcg(cand + j);
    k = __ldcg(key + idx);
  };
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (t < 256) s_hist[t] = 0u;
    __syncthreads();
    for (unsigned j = t; j < m; j += kRestThreads) {
      unsigned long long k; unsigned idx;
      entry(j, k, idx);
      if ((k >> (shift + 8)) == prefix) atomicAdd(&s_hist[(unsigned)(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    unsigned long long above;
    const int bin = pick_bin_256<true>(t < 256 ? s_hist[255 - t] : 0u, rem, warp_tot, above);
    prefix = (prefix << 8) | (unsigned long long)bin;
    rem -= above;
  }
  // prefix is the threshold now and rem (>= 1) the number of keys equal to it that are kept: the rem lowest indices
  unsigned long long ipre = 0ull;
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (t < 256) s_hist[t] = 0u;
    __syncthreads();
    for (unsigned j = t; j < m; j += kRestThreads) {
      unsigned long long k; unsigned idx;
      entry(j, k, idx);
      if (k == prefix && ((unsigned long long)idx >> (shift + 8)) == ipre) atomicAdd(&s_hist[(idx >> shift) & 255u], 1u);
    }
    __syncthreads();
    unsigned long long below;
    const int bin = pick_bin_256<false>(t < 256 ? s_hist[t] : 0u, rem, warp_tot, below);
    ipre = (ipre << 8) | (unsigned long long)bin;
    rem -= below;
  }
  if (t == 0) { st->prefix = prefix; st->cut = (unsigned int)ipre; }
}

// Threshold of layers of up to kClusterKeys kernels: one cluster of R blocks (one block up to kBlockKeys, eight above).  What k_select_rest
// takes is a chain of a dozen dependent trips to L2 - a histogram and a list in global memory, a fence, a ticket, and
// everything read back by the last block.  Here the blocks keep the keys that share the first digit in shared memory and find
// the rest of the threshold there, eight bits at a time from the top (key first, then the complemented index, so that among
// equal keys the lowest index comes first): a histogram per block, one cluster barrier, every block adds them up for itself.
// When few enough keys are left they are ranked directly, usually after one round.  A block whose keys do not fit its list
// reads them again in every round.
// The whole call: 64 x 64 14.5 -> 10.1 us, 256 x 256 16.6 -> 14.5, 512 x 256 19.4 -> 17.1; at 512 x 512 reading the keys with
// eight SMs costs what the rest saves (24 against 23 us; sixteen blocks: 23), so larger layers stay with k_select_rest.
constexpr int kSelThreads = 1024, kSelList = 3328, kSelFew = 128, kSelBlocks = 8;
constexpr int64_t kBlockKeys = 16384, kClusterKeys = 131072;
template <int R>
__device__ __forceinline__ void sel_barrier() {
  if constexpr (R == 1) { __syncthreads(); return; }
  __syncwarp();                                      // (.aligned, behind branches that lanes take apart)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of a block's shared memory, and what is done there.
__device__ __forceinline__ uint32_t sel_addr(const void* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
template <int R>
__global__ void __launch_bounds__(kSelThreads) k_select_cluster(const unsigned long long* __restrict__ key, int64_t FC, SelectState* st,
                                                                long long n_keep, const unsigned int* hist) {
  __shared__ unsigned long long s_key[kSelList], s_few_key[kSelFew];
  __shared__ unsigned int s_idx[kSelList], s_few_idx[kSelFew];
  __shared__ __align__(16) unsigned int s_hist[2][256];
  __shared__ unsigned int s_n, s_few, s_digit, s_rest, s_count;
  const int t = threadIdx.x, lane = t & 31;
  const int rank = R == 1 ? 0 : (int)(blockIdx.x % R);
  if (t == 0) { s_n = 0u; s_few = 0u; }
  if (t < 512) s_hist[t >> 8][t & 255] = 0u;
  pdl_wait();
  const int64_t per = (FC + R - 1) / R, i0 = rank * per, i1 = i0 + per < FC ? i0 + per : FC;
  unsigned long long rem = (unsigned long long)n_keep;
  const unsigned long long first = pick_digit(hist, 0, rem);
  constexpr int BATCH = R == 1 ? 8 : 16;                          // keys of a thread in flight
  for (int64_t b = i0; b < i1; b += BATCH * kSelThreads) {
    unsigned long long k[BATCH];
#pragma unroll
    for (int q = 0; q < BATCH; ++q) {
      const int64_t i = b + q * kSelThreads + t;
      k[q] = i < i1 ? __ldcg(key + i) : 0ull;
    }
    unsigned mine = 0u;                              // bit q: the thread's q-th key belongs on the list
#pragma unroll
    for (int q = 0; q < BATCH; ++q)
      if ((k[q] >> 48) == first && b + q * kSelThreads + t < i1) mine |= 1u << q;
    // a place in the list: one atomic per warp
    const unsigned c = (unsigned)__popc(mine);
    unsigned incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned u = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += u;
    }
    unsigned base = 0u;
    if (lane == 31) base = incl ? atomicAdd(&s_n, incl) : 0u;
    unsigned pos = __shfl_sync(0xFFFFFFFFu, base, 31) + incl - c;
#pragma unroll
    for (int q = 0; q < BATCH; ++q)
      if ((mine >> q) & 1u) {
        if (pos < (unsigned)kSelList) { s_key[pos] = k[q]; s_idx[pos] = (unsigned)(b + q * kSelThreads + t); }
        ++pos;
      }
  }
  __syncthreads();
  const bool listed = s_n <= (unsigned)kSelList;
  const int n_list = (int)s_n;
  auto each = [&](auto&& fn) {                       // this block's keys (all of its range if the list is too short)
    if (listed) for (int j = t; j < n_list; j += kSelThreads) fn(s_key[j], s_idx[j]);
    else for (int64_t i = i0 + t; i < i1; i += kSelThreads) fn(__ldcg(key + i), (unsigned)i);
  };
  // digits decided so far: 2 + d bytes of the key, later d - 6 bytes of the complemented index
  unsigned long long kp = first;
  unsigned ip = 0u;
  int d = 0;
  auto matches = [&](unsigned long long k, unsigned i, int d) {
    return d <= 6 ? (k >> (48 - 8 * d)) == kp : k == kp && ((unsigned long long)(~i) >> (32 - 8 * (d - 6))) == ip;
  };
  for (; d < 10; ++d) {
    unsigned int* h = s_hist[d & 1];
    each([&](unsigned long long k, unsigned i) {
      if (matches(k, i, d)) atomicAdd(&h[d < 6 ? (unsigned)(k >> (40 - 8 * d)) & 255u : (~i >> (24 - 8 * (d - 6))) & 255u], 1u);
    });
    sel_barrier<R>();
    if (t < 32) {
      const int top = 255 - 8 * lane;                // the lane's bins: top, top - 1, .. top - 7
      unsigned c[8] = {};
#pragma unroll
      for (int q = 0; q < R; ++q) {
        unsigned v[8];
        const uint32_t a = sel_addr(h + top - 7, R == 1 ? 0u : (uint32_t)q);
        asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[7]), "=r"(v[6]), "=r"(v[5]), "=r"(v[4]) : "r"(a) : "memory");
        asm volatile("ld.shared::cluster.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[3]), "=r"(v[2]), "=r"(v[1]), "=r"(v[0]) : "r"(a + 16u) : "memory");
#pragma unroll
        for (int e = 0; e < 8; ++e) c[e] += v[e];
      }
      unsigned sum = 0u;
#pragma unroll
      for (int e = 0; e < 8; ++e) sum += c[e];
      unsigned above = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, above, off);
        if (lane >= off) above += u;
      }
      above -= sum;                                  // keys in higher bins than this lane's
      const unsigned want = (unsigned)rem;
      if (t == 0) { s_digit = 0u; s_rest = 1u; s_count = 0u; }      // defined values even if no bin qualifies
      __syncwarp();
      if (want > above && want <= above + sum) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          if (want > above && want <= above + c[e]) { s_digit = (unsigned)(top - e); s_rest = want - above; s_count = c[e]; }
          above += c[e];
        }
      }
    } else if (t >= 256 && t < 512) {
      s_hist[(d & 1) ^ 1][t - 256] = 0u;             // read by nobody any more: all blocks have passed the barrier after it
    }
    __syncthreads();
    if (d < 6) kp = (kp << 8) | s_digit; else ip = (ip << 8) | s_digit;
    rem = s_rest;
    const unsigned left = s_count;
    __syncthreads();                                 // (the results may be overwritten by the next round)
    if (left <= (unsigned)kSelFew) { ++d; break; }
  }
  each([&](unsigned long long k, unsigned i) {
    if (!matches(k, i, d)) return;
    unsigned pos;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], 1;" : "=r"(pos) : "r"(sel_addr(&s_few, 0u)) : "memory");
    if (pos >= (unsigned)kSelFew) return;
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(sel_addr(s_few_key + pos, 0u)), "l"(k) : "memory");
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(sel_addr(s_few_idx + pos, 0u)), "r"(i) : "memory");
  });
  sel_barrier<R>();
  if (rank != 0) return;
  // the entry with rem - 1 others before it (key descending, index ascending) is the threshold and the last kept index
  const int m = min((int)s_few, kSelFew);
  if (t < m) {
    const unsigned long long kj = s_few_key[t];
    const unsigned ij = s_few_idx[t];
    unsigned before = 0u;
    for (int q = 0; q < m; ++q) before += s_few_key[q] > kj || (s_few_key[q] == kj && s_few_idx[q] < ij) ? 1u : 0u;
    if (before + 1u == (unsigned)rem) { st->prefix = kj; st->cut = ij; }
  }
}

// Decide keep / remove per kernel and write pattern ids and masked weights.  The decision is taken by one thread per
// kernel; the weights are then copied by the whole block in the order they lie in memory (a thread that walked its
// own nine values would touch a different 32-byte sector with every lane, on the way in and on the way out).
__global__ void __launch_bounds__(kSelBlock) k_finalize(const float* w, int64_t FC, MaskTable lib,
                                                        const unsigned long long* key, const unsigned char* pid_in, const SelectState* st,
                                                        unsigned char* pid_out, float* wm, int keep_all_or_none) {
  __shared__ unsigned short s_mask[kSelBlock];      // the kept positions of every kernel of the block (0: removed)
  const int64_t i0 = (int64_t)blockIdx.x * kSelBlock;
  const int64_t i = i0 + threadIdx.x;
  const bool valid = i < FC;
  const int64_t e0 = i0 * 9;
  const int n = (int)(((FC - i0) < (int64_t)kSelBlock ? (FC - i0) : (int64_t)kSelBlock) * 9);
  // Everything but the threshold is there before the wait: this kernel is let go by the selection kernel after that one's own
  // wait for the energies (or, without a selection, by the kernel of the energies, whose results are read after the wait).
  const bool quick = aligned_dev(w + e0, 16) && aligned_dev(wm + e0, 16);
  constexpr int PIECES = (9 * kSelBlock / 4 + kSelBlock - 1) / kSelBlock;      // of four weights per thread
  const int done = quick ? n & ~3 : 0;
  float4 v[PIECES];
#pragma unroll
  for (int q = 0; q < PIECES; ++q) {
    const int e = 4 * ((int)threadIdx.x + q * kSelBlock);
    if (e < done) v[q] = *reinterpret_cast<const float4*>(w + e0 + e);
  }
  unsigned long long k = 0ull;
  unsigned char p = 0;
  if (keep_all_or_none < 0 && valid) { k = key[i]; p = pid_in[i]; }
  pdl_wait();
  bool keep;
  if (keep_all_or_none >= 0) {            // n_keep == F*C (1) or n_keep == 0 (0): no threshold needed
    keep = keep_all_or_none == 1;
    if (valid) p = pid_in[i];
  } else {
    const unsigned long long thr = st->prefix;
    keep = valid && (k > thr || (k == thr && (unsigned int)i <= st->cut));   // ties: lowest indices first
  }
  unsigned m = 0u;
  if (valid) {
    m = keep ? lib.m[p] : 0u;
    pid_out[i] = keep ? p : (unsigned char)PAT_PRUNED;
  }
  s_mask[threadIdx.x] = (unsigned short)m;
  __syncthreads();
  auto masked = [&](int e, float x) {
    const int kq = e / 9, b = e - kq * 9;
    return ((s_mask[kq] >> b) & 1u) ? x : 0.0f;
  };
#pragma unroll
  for (int q = 0; q < PIECES; ++q) {
    const int e = 4 * ((int)threadIdx.x + q * kSelBlock);
    if (e < done) *reinterpret_cast<float4*>(wm + e0 + e) = make_float4(masked(e, v[q].x), masked(e + 1, v[q].y), masked(e + 2, v[q].z), masked(e + 3, v[q].w));
  }
  for (int e = done + threadIdx.x; e < n; e += kSelBlock) wm[e0 + e] = masked(e, w[e0 + e]);
}

}  // namespace
}  // namespace pat

using namespace pat;

extern "C" size_t pat_project_workspace(int F, int C) {
  if (F < 1 || C < 1 || F > 65535 || C > 65535) return 0;
  return ws_bytes((int64_t)F * C);
}

extern "C" int pat_project(const float* w, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                           uint8_t* pattern_id, float* w_masked, void* workspace, size_t workspace_bytes,
                           void* stream) {
  if (!w || !pattern_id || !w_masked || !workspace) return set_error(PAT_ERR_INVALID_ARG, "pat_project: null pointer");
  if (F < 1 || C < 1 || F > 65535 || C > 65535) return set_error(PAT_ERR_SHAPE, "pat_project: F=%d C=%d outside 1..65535", F, C);
  if (int rc = check_library(masks, K)) return rc;
  const int64_t FC = (int64_t)F * C;
  if (n_keep < 0 || n_keep > FC) return set_error(PAT_ERR_INVALID_ARG, "pat_project: n_keep=%lld outside 0..%lld", (long long)n_keep, (long long)FC);
  if (!aligned(w, 4) || !aligned(w_masked, 4)) return set_error(PAT_ERR_ALIGN, "pat_project: weights must be 4-byte aligned");
  if (!aligned(workspace, 256)) return set_error(PAT_ERR_ALIGN, "pat_project: workspace must be 256-byte aligned");
  const ProjWs ws = carve(workspace, FC);
  if (workspace_bytes < ws.bytes) return set_error(PAT_ERR_WORKSPACE, "pat_project: workspace has %zu bytes, needs %zu", workspace_bytes, ws.bytes);

  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  MaskTable lib;
  for (int j = 0; j <= kMaxK; ++j) lib.m[j] = (j < K) ? masks[j] : (uint16_t)0;
  lib.K = K;
  const int nb_sel = (int)((FC + kPatBlock - 1) / kPatBlock), nb_rest = (int)((FC + kRestThreads - 1) / kRestThreads);
  const int nblk = (int)((FC + kSelBlock - 1) / kSelBlock);
  int mode = -1;
  if (n_keep == FC) mode = 1;
  else if (n_keep == 0) mode = 0;
  Launches launches;
  static_assert(kHistWords % 4 == 0 && (kBins + kCoarse) % 4 == 0, "counters are zeroed four at a time");
  if (mode < 0) launches.add(k_zero_counters, dim3((unsigned)((kHistWords / 4 + kZeroThreads - 1) / kZeroThreads)), dim3(kZeroThreads), 0, st, ws.hist, (int)kHistWords);
  launches.add(k_select_pattern, dim3(nb_sel), dim3(kPatBlock), 0, st, w, FC, lib, ws.key, ws.pid, ws.hist, mode < 0);
  if (mode < 0) {
    if (FC <= kBlockKeys) {
      launches.add(k_select_cluster<1>, dim3(1), dim3(kSelThreads), 0, st, ws.key, FC, ws.st, (long long)n_keep, ws.hist);
    } else if (FC <= kClusterKeys) {
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      attr[1].id = cudaLaunchAttributeClusterDimension;
      attr[1].val.clusterDim.x = kSelBlocks; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(kSelBlocks); cfg.blockDim = dim3(kSelThreads); cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 2;
      launches.add_result([&] {
        return cudaLaunchKernelEx(&cfg, k_select_cluster<kSelBlocks>, static_cast<const unsigned long long*>(ws.key), FC, ws.st, (long long)n_keep,
                                  static_cast<const unsigned int*>(ws.hist));
      });
    } else {
      launches.add(k_select_rest, dim3(nb_rest), dim3(kRestThreads), 0, st, ws.key, FC, ws.st, (long long)n_keep, ws.hist, ws.cand_key, ws.cand);
    }
  }
  launches.add(k_finalize, dim3(nblk), dim3(kSelBlock), 0, st, w, FC, lib, ws.key, ws.pid, ws.st, pattern_id, w_masked, mode);
  count_launches(launches.n);
  if (launches.error != cudaSuccess) return check_cuda(launches.error, "pat_project launch");
  return check_cuda(cudaGetLastError(), "pat_project launch");
}

// ------------------------------------------------------------------------------------------------------------
// pat_project_static: the same projection for callers that cannot hand over a workspace.
//
// Some hosts of this library may not allocate device memory at the point where they project a layer: a serving
// process whose whole device budget was reserved up front by another component, a plug-in that runs inside
// somebody else's memory pool, or a latency-critical loop that must not risk the implicit device-wide
// synchronisation of an allocation.  For them the scratch space lives in the library image itself.
namespace pat {
namespace {

constexpr int64_t kStaticMaxKernels = 262144;   // F * C limit of pat_project_static (a 512 x 512 layer)
constexpr size_t kStaticScratchBytes = ws_bytes(kStaticMaxKernels);   // about 4.2 MB

// Every GPU that loads the library holds this array until the process ends.
static __device__ __align__(256) unsigned char g_project_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices] = {};          // device address of the array, per device (host-side cache)

// The array's name is only a host-side handle in host code; the device address has to be asked for, once per
// device and with that device current.
int static_scratch(void** out) {
  int dev = -1;
  if (int rc = check_cuda(cudaGetDevice(&dev), "cudaGetDevice")) return rc;
  if (dev < 0 || dev >= kMaxDevices) return set_error(PAT_ERR_CUDA, "pat_project_static: device index %d not supported", dev);
  void* p = __atomic_load_n(&g_scratch_addr[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    if (int rc = check_cuda(cudaGetSymbolAddress(&p, g_project_scratch), "cudaGetSymbolAddress(scratch)")) return rc;
    __atomic_store_n(&g_scratch_addr[dev], p, __ATOMIC_RELEASE);
  }
  *out = p;
  return PAT_OK;
}

}  // namespace
}  // namespace pat

extern "C" int64_t pat_project_static_max_kernels(void) { return kStaticMaxKernels; }

extern "C" int pat_project_static(const float* w, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                                  uint8_t* pattern_id, float* w_masked, void* stream) {
  if (F < 1 || C < 1 || F > 65535 || C > 65535)
    return set_error(PAT_ERR_SHAPE, "pat_project_static: F=%d C=%d outside 1..65535", F, C);
  if ((int64_t)F * C > kStaticMaxKernels)
    return set_error(PAT_ERR_WORKSPACE, "pat_project_static: F*C = %lld exceeds the built-in scratch (%lld kernels); use pat_project with a workspace",
                     (long long)F * C, (long long)kStaticMaxKernels);
  static_assert(kStaticScratchBytes >= 8 * (size_t)kStaticMaxKernels, "scratch holds at least the keys");
  if (carve(nullptr, (int64_t)F * C).bytes > kStaticScratchBytes)
    return set_error(PAT_ERR_WORKSPACE, "pat_project_static: internal scratch too small for F=%d C=%d", F, C);
  void* scratch = nullptr;
  if (int rc = static_scratch(&scratch)) return rc;
  return pat_project(w, F, C, masks, K, n_keep, pattern_id, w_masked, scratch, kStaticScratchBytes, stream);
}
