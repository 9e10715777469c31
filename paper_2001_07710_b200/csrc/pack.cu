// pat_pack / pat_unpack: compressed, re-ordered weight storage.
//
// Section 6.2 re-orders filters so that filters with similar kernels sit together (balanced work per thread
// group) and groups, inside each filter, the kernels that share a pattern (one code path per group, no
// branches inside it).  The blob holds a canonical section in exactly that order and an execution section in
// which each filter's kernels are re-sorted by blocks of 16 input channels (the unit in which the convolution
// kernels stage activations), then pattern, then channel.  The execution section has its own filter order:
// filters stay inside their aligned group of 32 original filters (so that a thread block that owns a group
// writes 32 adjacent output channels) and are sorted inside the group by kept-kernel count, descending, so
// that pairing position i with position 31 - i gives every warp the same amount of work.
#include <cuda_bf16.h>
#include "common.cuh"

namespace pat {
namespace {

struct BlobPtrs {
  BlobHeader* hdr;
  int32_t *perm, *fptr, *pptr;
  uint16_t* chan;
  void* w4;
  int32_t* xfilt;      // execution position -> original filter
  int32_t* tptr;
  uint32_t* tmeta;
  void* tw4;
  uint32_t* dboff;     // descriptor block -> offset inside dblk, in 16-byte units (nblk + 1 entries)
  char* dblk;
  unsigned short* dense;   // the masked weights in dense form (nullptr: the blob holds none), see mma_weights
  int32_t *hist, *cnt, *inv, *xinv, *xbase;
  uint32_t* stages;    // [F][2][words of 32 tiles]: a filter (execution order) has kernels in the lower / upper half of a tile
};

__host__ __device__ inline BlobPtrs blob_ptrs(void* blob, const BlobLayout& L, int F, int K) {
  char* b = static_cast<char*>(blob);
  BlobPtrs p;
  p.hdr = reinterpret_cast<BlobHeader*>(b);
  p.perm = reinterpret_cast<int32_t*>(b + L.perm);
  p.fptr = reinterpret_cast<int32_t*>(b + L.fptr);
  p.pptr = reinterpret_cast<int32_t*>(b + L.pptr);
  p.chan = reinterpret_cast<uint16_t*>(b + L.chan);
  p.w4 = b + L.w4;
  p.xfilt = reinterpret_cast<int32_t*>(b + L.xfilt);
  p.tptr = reinterpret_cast<int32_t*>(b + L.tptr);
  p.tmeta = reinterpret_cast<uint32_t*>(b + L.tmeta);
  p.tw4 = b + L.tw4;
  p.dboff = reinterpret_cast<uint32_t*>(b + L.dboff);
  p.dblk = b + L.dblk;
  p.dense = L.dense ? reinterpret_cast<unsigned short*>(b + L.dense) : nullptr;
  p.hist = reinterpret_cast<int32_t*>(b + L.scratch);
  p.cnt = p.hist + (size_t)F * K;
  p.inv = reinterpret_cast<int32_t*>(b + inv_offset(L, F, K));
  p.xinv = p.inv + F;
  p.xbase = p.xinv + F;
  p.stages = reinterpret_cast<uint32_t*>(p.xbase + F);
  return p;
}

// One block per original filter: per-pattern counts and kept count.
__global__ void __launch_bounds__(256) k_pack_count(const uint8_t* pid, int C, int K, BlobPtrs bp, int* status) {
  pdl_wait();
  extern __shared__ int sh[];   // K counters
  const int f = blockIdx.x;
  for (int j = threadIdx.x; j < K; j += blockDim.x) sh[j] = 0;
  __syncthreads();
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    const int p = pid[(size_t)f * C + c];
    if (p == PAT_PRUNED) continue;
    if (p >= K) { atomicExch(status, PAT_ERR_BLOB); continue; }
    atomicAdd(&sh[p], 1);
  }
  __syncthreads();
  int tot = 0;
  for (int j = threadIdx.x; j < K; j += blockDim.x) bp.hist[(size_t)f * K + j] = sh[j];
  if (threadIdx.x == 0) {
    for (int j = 0; j < K; ++j) tot += sh[j];
    bp.cnt[f] = tot;
  }
}

// Adds v over the threads of a warp.
__device__ inline int warp_sum(int v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

// One block per filter: position = number of filters that come before it in the ordering
// (kept count descending, per-pattern counts lexicographically descending, original index ascending);
// the threads of the block share the comparisons.  The kept kernels of the filters before it, added up in the same pass,
// are where its own begin (no scan over the filters, which was a launch of one block); block 0 writes the header.
constexpr int kRankThreads = 128;
__global__ void __launch_bounds__(kRankThreads) k_pack_rank(int F, int C, int K, long long n_keep, int dtype, MaskTable lib,
                                                            unsigned long long total_bytes, BlobPtrs bp, int* status) {
  pdl_wait();
  __shared__ int s_sum[5];                 // rank, kernels before; rank and kernels before in execution order; all kernels
  __shared__ int s_hist[kMaxK + 1];
  const int f = blockIdx.x;
  if (threadIdx.x < 5) s_sum[threadIdx.x] = 0;
  for (int j = threadIdx.x; j < K; j += kRankThreads) s_hist[j] = bp.hist[(size_t)f * K + j];
  __syncthreads();
  const int nf = bp.cnt[f];
  const int g0 = (f / kExecGroup) * kExecGroup, g1 = min(F, g0 + kExecGroup);
  int sum[5] = {0, 0, 0, 0, 0};
  // four filters at a time, their counts and first two pattern counts (which decide nearly always) read together
  constexpr int AT_ONCE = 4;
  for (int gb = threadIdx.x; gb < F; gb += AT_ONCE * kRankThreads) {
    int ns[AT_ONCE], h0[AT_ONCE], h1[AT_ONCE];
#pragma unroll
    for (int i = 0; i < AT_ONCE; ++i) {
      const int g = min(gb + i * kRankThreads, F - 1);
      ns[i] = bp.cnt[g];
      h0[i] = bp.hist[(size_t)g * K];
      h1[i] = bp.hist[(size_t)g * K + (K > 1 ? 1 : 0)];
    }
#pragma unroll
    for (int i = 0; i < AT_ONCE; ++i) {
      const int g = gb + i * kRankThreads, ng = ns[i];
      if (g >= F) break;
      sum[4] += ng;
      if (g == f) continue;
      bool before;
      if (ng != nf) before = ng > nf;
      else if (h0[i] != s_hist[0]) before = h0[i] > s_hist[0];
      else if (K > 1 && h1[i] != s_hist[1]) before = h1[i] > s_hist[1];
      else {
        const int32_t* hg = bp.hist + (size_t)g * K;
        int j = 0;
        while (j < K && hg[j] == s_hist[j]) ++j;
        before = (j < K) ? (hg[j] > s_hist[j]) : (g < f);
      }
      if (before) { sum[0] += 1; sum[1] += ng; }
      // execution order: inside the aligned group of 32 original filters, by kept count (descending), then index
      const bool in_group = g >= g0 && g < g1;
      if (in_group && (ng > nf || (ng == nf && g < f))) { sum[2] += 1; sum[3] += ng; }
      if (g < g0) sum[3] += ng;
    }
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const int v = warp_sum(sum[q]);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum[q], v);
  }
  __syncthreads();
  const int q = s_sum[0], start = s_sum[1], x = g0 + s_sum[2], total = s_sum[4];
  if (threadIdx.x == 0) {
    bp.perm[q] = f;
    bp.inv[f] = q;
    bp.fptr[q] = start;
    bp.xfilt[x] = f;
    bp.xinv[f] = x;
    bp.xbase[x] = s_sum[3];
  }
  for (int j = threadIdx.x; j <= K; j += kRankThreads) {
    int pos = start;
    for (int i = 0; i < j; ++i) pos += s_hist[i];
    bp.pptr[(size_t)q * (K + 1) + j] = pos;
  }
  if (f == 0) {
    BlobHeader* h = bp.hdr;
    for (int j = threadIdx.x; j <= kMaxK; j += kRankThreads) h->masks[j] = lib.m[j];
    if (threadIdx.x == 0) {
      bp.fptr[F] = total;
      const bool ok = (long long)total == n_keep;
      if (!ok) atomicExch(status, PAT_ERR_BLOB);
      h->magic = ok ? kBlobMagic : 0u;
      h->version = kBlobVersion;
      h->F = F; h->C = C; h->K = K; h->dtype = dtype;
      h->n_keep = n_keep;
      h->total_bytes = total_bytes;
      h->max_block_entries = 0;   // raised by k_pack_blocks
    }
  }
}

template <typename T> __device__ inline T cvt_weight(float v);
template <> __device__ inline float cvt_weight<float>(float v) { return v; }
template <> __device__ inline __half cvt_weight<__half>(float v) { return __float2half_rn(v); }

// The bf16 number next to v; a finite one that would round to infinity is cut off instead (its rest is a bf16 number too).
__device__ inline __nv_bfloat16 finite_bf16(float v) {
  const uint32_t b = __float_as_uint(v), r = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v));
  return __ushort_as_bfloat16((unsigned short)((r & 0x7FFFu) == 0x7F80u ? b >> 16 : r));
}

// Two neighbouring values of the dense form: fp16, or fp32 as a sum of three bf16 numbers, each the rounded rest of those
// before it.
template <typename T> __device__ inline void dense_store(uint32_t* dst, size_t term, float v0, float v1);
template <> __device__ inline void dense_store<__half>(uint32_t* dst, size_t, float v0, float v1) {
  *dst = (uint32_t)__half_as_ushort(__float2half_rn(v0)) | ((uint32_t)__half_as_ushort(__float2half_rn(v1)) << 16);
}
template <> __device__ inline void dense_store<float>(uint32_t* dst, size_t term, float v0, float v1) {
#pragma unroll
  for (int t = 0; t < kMmaTermsF32; ++t) {
    const __nv_bfloat16 h0 = finite_bf16(v0), h1 = finite_bf16(v1);
    dst[t * term] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
    v0 -= __bfloat162float(h0);            // exact: the rest has fewer significant bits
    v1 -= __bfloat162float(h1);
  }
}

// One block per original filter: its first four warps place every kept kernel in the canonical and in the execution
// order, the other four write its rows of the dense form (zeros included) meanwhile.
// Positions are counted, never searched: per (16-channel tile, pattern) counts in shared memory give, after
// prefix sums over the tiles, the start of every (pattern) run in the canonical order and of every tile in the
// execution order; the rank of a kernel inside its tile needs a look at the 16 channels of that tile only.
// TABLE = false (tile x pattern table too large for shared memory): the counts are taken by direct loops.
// Five blocks per SM (48 registers; the addresses of 27 planes are what spills in fp32) keep all filters of a 512-filter layer
// in flight: without the bound 178 registers, 43 instead of 28 us a call.  The work before the wait took the call from 10.3 to
// 8.0 us at 64 x 64, 16.9 to 14.0 at 512 x 512 (fp16).
constexpr int kScatterThreads = 256, kListThreads = 128;
constexpr size_t kScatterStatic = 1024;    // static shared memory
template <typename T, bool TABLE>
__global__ void __launch_bounds__(kScatterThreads, 5) k_pack_scatter(const float* __restrict__ wm, const uint8_t* __restrict__ pid,
                                                                  int C, int K, int nct, bool blocks, MaskTable lib, BlobPtrs bp) {
  extern __shared__ __align__(16) uint8_t sm_raw[];
  int* tile_pat = reinterpret_cast<int*>(sm_raw);                          // [nct][K] (TABLE only)
  int* tile_start = tile_pat + (TABLE ? nct * K : 0);                      // [nct + 1] kept kernels before tile t
  uint32_t* stage_bits = reinterpret_cast<uint32_t*>(tile_start + nct + 1);   // [2][words] (blocks only)
  const int words = (nct + 31) / 32;
  uint8_t* spid = reinterpret_cast<uint8_t*>(stage_bits + (blocks ? 2 * words : 0));        // C pattern ids of this filter
  __shared__ int s_pptr[kMaxK];
  static_assert(sizeof(s_pptr) <= kScatterStatic, "what pat_pack counts with");
  const int f = blockIdx.x, tid = threadIdx.x;
  for (int c = tid; c < C; c += kScatterThreads) spid[c] = pid[(size_t)f * C + c];
  if (TABLE)
    for (int i = tid; i < nct * K; i += kScatterThreads) tile_pat[i] = 0;
  __syncthreads();
  // What stands in pattern_id and w_masked is complete before this kernel starts (k_pack_count has waited for it, and
  // k_pack_rank, which lets this one go, for k_pack_count): the counting and the first weights of the dense form come before the wait.
  // Refused by k_pack_rank (pattern_id keeps another number of kernels than n_keep: the positions computed below would leave the
  // sections sized by n_keep): nothing is written.
  if (tid >= kListThreads) {
    const int pitch = mma_pitch(C);                     // a multiple of eight
    const size_t plane = (size_t)gridDim.x * pitch;
    float v[2][9];
    auto fetch = [&](int c) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = c + h < C ? spid[c + h] : PAT_PRUNED;
        const unsigned m = (j == PAT_PRUNED || j >= K) ? 0u : lib.m[j];
        const float* src = wm + ((size_t)f * C + c + h) * 9;
#pragma unroll
        for (int b = 0; b < 9; ++b) v[h][b] = (m >> b) & 1u ? __ldg(src + b) : 0.0f;
      }
    };
    int c = 2 * (tid - kListThreads);
    if (bp.dense && c < pitch) fetch(c);
    pdl_wait();
    if (!bp.dense || bp.hdr->magic != kBlobMagic) return;
    while (c < pitch) {
      uint32_t* dst = reinterpret_cast<uint32_t*>(bp.dense + (size_t)f * pitch + c);
#pragma unroll
      for (int b = 0; b < 9; ++b) dense_store<T>(dst + b * (plane / 2), 9 * (plane / 2), v[0][b], v[1][b]);
      c += 2 * (kScatterThreads - kListThreads);
      if (c < pitch) fetch(c);
    }
    return;
  }
  auto list_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kListThreads) : "memory"); };
  // kept kernels per tile (and per tile and pattern)
  for (int t = tid; t < (nct + 31) / 32 * 32; t += kListThreads) {
    int n = 0, lower = 0;
    const int c0 = t * kChanTile, c1 = min(c0 + kChanTile, C);
    for (int c = c0; c < c1; ++c) {
      const int j = spid[c];
      if (j == PAT_PRUNED || j >= K) continue;
      ++n;
      lower += c - c0 < kChanTile / 2 ? 1 : 0;
      if (TABLE) tile_pat[t * K + j] += 1;        // one thread per tile: no race
    }
    if (t < nct) tile_start[t + 1] = n;
    const unsigned lo = __ballot_sync(0xFFFFFFFFu, lower > 0), hi = __ballot_sync(0xFFFFFFFFu, n > lower);
    if ((t & 31) == 0 && blocks) {                // for k_pack_blocks
      stage_bits[t >> 5] = lo;
      stage_bits[words + (t >> 5)] = hi;
    }
  }
  list_sync();
  // exclusive prefix sums over the tiles: a warp per pattern column, one more column for the tile totals
  {
    const int lane = tid & 31;
    for (int j = tid >> 5; j <= (TABLE ? K : 0); j += kListThreads >> 5) {
      const bool totals = j == (TABLE ? K : 0);
      int run = 0;
      for (int t0 = 0; t0 < nct; t0 += 32) {
        const int t = t0 + lane;
        const int v = t < nct ? (totals ? tile_start[t + 1] : tile_pat[t * K + j]) : 0;
        int incl = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int u = __shfl_up_sync(0xFFFFFFFFu, incl, off);
          if (lane >= off) incl += u;
        }
        if (t < nct) {
          if (totals) tile_start[t + 1] = run + incl;
          else tile_pat[t * K + j] = run + incl - v;
        }
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
      }
      if (totals && lane == 0) tile_start[0] = 0;
    }
  }
  list_sync();
  pdl_wait();
  if (bp.hdr->magic != kBlobMagic) return;
  const int q = bp.inv[f], xe = bp.xinv[f];
  const int f0 = bp.xbase[xe];
  for (int j = tid; j < K; j += kListThreads) s_pptr[j] = bp.pptr[(size_t)q * (K + 1) + j];
  list_sync();
  for (int t = tid; t <= nct; t += kListThreads) bp.tptr[(size_t)xe * (nct + 1) + t] = f0 + tile_start[t];
  if (blocks)
    for (int i = tid; i < 2 * words; i += kListThreads) bp.stages[(size_t)xe * 2 * words + i] = stage_bits[i];
  T* w4 = static_cast<T*>(bp.w4);
  T* tw4 = static_cast<T*>(bp.tw4);
  for (int c = tid; c < C; c += kListThreads) {
    const int j = spid[c];
    if (j == PAT_PRUNED || j >= K) continue;
    unsigned m = lib.m[j];
    float v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {                 // ascending bit order
      v[t] = __ldg(wm + ((size_t)f * C + c) * 9 + (__ffs(m) - 1));
      m &= m - 1u;
    }
    const int tile = c / kChanTile;
    const int c0 = tile * kChanTile, c1 = min(c0 + kChanTile, C);
    int same_in_tile = 0;     // kernels of the same pattern on lower channels of this tile
    int exec_in_tile = 0;     // kernels of this tile ordered before (pattern, channel)
    for (int d = c0; d < c1; ++d) {
      const int pd = spid[d];
      if (pd == PAT_PRUNED || pd >= K) continue;
      same_in_tile += (pd == j && d < c) ? 1 : 0;
      exec_in_tile += (pd < j || (pd == j && d < c)) ? 1 : 0;
    }
    int same_before;          // kernels of the same pattern on lower channels (canonical order)
    if (TABLE) same_before = tile_pat[tile * K + j] + same_in_tile;
    else {
      same_before = same_in_tile;
      for (int d = 0; d < c0; ++d) same_before += (spid[d] == j) ? 1 : 0;
    }
    const int pos = s_pptr[j] + same_before;
    const int tpos = f0 + tile_start[tile] + exec_in_tile;
    bp.chan[pos] = (uint16_t)c;
    bp.tmeta[tpos] = (uint32_t)c | ((uint32_t)j << 16);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      w4[(size_t)pos * 4 + t] = cvt_weight<T>(v[t]);
      tw4[(size_t)tpos * 4 + t] = cvt_weight<T>(v[t]);
    }
  }
}

// Descriptor blocks of the multiply-add kernel that copies its work lists with one bulk copy per pipeline
// stage (8 channels).  One block per (group of 32 filters in execution order, stage), groups major.  A block is the
// work of the kernel's 16 consumer warps in that stage; warp w owns filter slots w ("A") and 31 - w ("B") of the
// group and keeps one accumulator tile in registers, the other parked.  The order of a warp's operations is fixed
// here, at pack time: starting from the tile it holds when the stage begins (A at the first stage; afterwards
// whatever the previous stage left), first the kernels of that filter, then - only if the other filter has kernels
// in this stage - a swap and the other filter's kernels.
//   header   32 words; word w < 16: first operation of warp w (bits 0-15) | filter whose tile is in registers when
//            the stage begins (bit 31).
//   lists    32 bytes per operation, warp after warp, every list one slot longer than the warp's kernels:
//            {channel inside the stage | pattern_word(mask) | flags, byte offset of the window in an fp32 stage image
//             (channel plane + window row shift), taps 0-1}, {taps 2-3, 0, 0}
//            flags: kOpSwap on the first kernel after the swap, kOpEnd on the warp's last operation, together with
//            the start of the warp's list in the next stage's block (bits 21-31).  A warp without kernels in the
//            stage gets one operation with the flag kOpNop; otherwise the spare slot stays unused.
// A tile of 16 channels of the execution section gives two stages: its kernels with channel 0-7 and 8-15, each in
// (pattern, channel) order.  Offsets (header words, "next list", dboff) count 16-byte units, so an operation is two units.
// Launched with one warp per block (lane = consumer warp, lanes 16-31 idle apart from the walk and the shuffles).  Which
// stages a filter has kernels in comes as bits from k_pack_scatter: counting all earlier stages' kernels here was quadratic
// in the channels (512 x 512, keep 1/8: the packing 77 -> 27 us; 256 x 256: 39 -> 19).
__global__ void __launch_bounds__(32) k_pack_blocks(int nct, int nblk, MaskTable lib, BlobPtrs bp) {
  pdl_wait();
  if (bp.hdr->magic != kBlobMagic) return;   // refused by k_pack_rank, see k_pack_scatter
  const int blk = blockIdx.x, lane = threadIdx.x;
  const int nst = 2 * nct;                                   // stages of 8 channels
  const int g = blk / nst, st8 = blk % nst;
  const bool active = lane < kBlockWarps;
  const int w = active ? lane : 0;
  const int32_t* rowA = bp.tptr + (size_t)(g * kExecGroup + w) * (nct + 1);
  const int32_t* rowB = bp.tptr + (size_t)(g * kExecGroup + kExecGroup - 1 - w) * (nct + 1);
  // Kernels of the lane's own filter slot in this stage and in the next one, and in earlier stages: one walk over the tile
  // of this stage (and over the next tile, if the next stage is its lower half); slots A and B of a warp are lanes w and 31 - w.
  const int t16 = st8 >> 1, half = st8 & 1;
  const int32_t* row = bp.tptr + (size_t)(g * kExecGroup + lane) * (nct + 1);
  const int k0 = row[t16], k1 = row[t16 + 1], k2 = half && t16 + 1 < nct ? row[t16 + 2] : k1;
  int lower = 0, next_lower = 0;
  for (int k = k0; k < k2; ++k) {
    const int low = (bp.tmeta[k] & 8u) == 0u ? 1 : 0;        // channel below 8 inside its tile
    if (k < k1) lower += low; else next_lower += low;
  }
  const int n_own = half ? k1 - k0 - lower : lower, n_own_next = half ? next_lower : k1 - k0 - lower;
  int before = k0 - row[0] + (half ? lower : 0);
  // which tile the warp holds when this stage begins: it swaps in every stage in which the other filter has kernels
  int cur = 0;
  const int words = (nct + 31) / 32;
  const uint32_t* stA = bp.stages + (size_t)(g * kExecGroup + w) * 2 * words;
  const uint32_t* stB = bp.stages + (size_t)(g * kExecGroup + kExecGroup - 1 - w) * 2 * words;
  for (int t = 0; t < st8; t += 64) {                        // 32 tiles, two stages each
    const uint32_t a0 = stA[t >> 6], a1 = stA[words + (t >> 6)], b0 = stB[t >> 6], b1 = stB[words + (t >> 6)];
    for (int s = t; s < min(st8, t + 64); ++s)
      cur ^= (int)(((cur ? (s & 1 ? a1 : a0) : (s & 1 ? b1 : b0)) >> ((s >> 1) & 31)) & 1u);
  }
  const int nA = n_own, nB = __shfl_sync(0xFFFFFFFFu, n_own, 31 - lane), n_next = n_own_next + __shfl_sync(0xFFFFFFFFu, n_own_next, 31 - lane);
  const int cap = active ? nA + nB + 1 : 0;
  const int cap_next = (active && st8 + 1 < nst) ? n_next + 1 : 0;
  int incl = cap, incl_next = cap_next;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, incl, off), vn = __shfl_up_sync(0xFFFFFFFFu, incl_next, off);
    if (lane >= off) { incl += v; incl_next += vn; }
  }
  const int start = incl - cap, start_next = incl_next - cap_next;
  const int tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
  // kernels of this group in earlier stages (all 32 filter slots)
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, off);
  const uint32_t group_first = (uint32_t)bp.tptr[(size_t)(g * kExecGroup) * (nct + 1)];
  const uint32_t off16 = (uint32_t)blk * (uint32_t)(kBlockHeaderBytes / 16 + 2 * kBlockWarps) + 2u * (group_first + (uint32_t)before);
  if (lane == 0) {
    bp.dboff[blk] = off16;
    if (blk == nblk - 1) bp.dboff[nblk] = off16 + kBlockHeaderBytes / 16 + 2u * (uint32_t)tot;
    atomicMax(&bp.hdr->max_block_entries, tot);
  }
  char* base = bp.dblk + (size_t)off16 * 16;
  reinterpret_cast<uint32_t*>(base)[lane] = active ? ((uint32_t)(2 * start) | ((uint32_t)cur << 31)) : 0u;
  if (!active) return;
  uint4* ent = reinterpret_cast<uint4*>(base + kBlockHeaderBytes) + 2 * start;
  const uint4* tw4 = static_cast<const uint4*>(bp.tw4);       // four fp32 taps per kernel
  const int n_first = cur ? nB : nA, n_second = cur ? nA : nB;
  const int n_ops = n_first + n_second;
  const uint32_t end_flags = kOpEnd | ((uint32_t)(2 * start_next) << kOpNextShift);
  if (n_ops == 0) {
    ent[0] = make_uint4(kOpNop | end_flags, 0u, 0u, 0u);
    ent[1] = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  int k_out = 0;
  for (int pass = 0; pass < 2; ++pass) {
    const int32_t* r = (pass == 0) == (cur == 0) ? rowA : rowB;   // first the filter whose tile is held
    for (int k = r[t16]; k < r[t16 + 1]; ++k) {
      const uint32_t mt = bp.tmeta[k];
      const uint32_t ch16 = (mt & 0xFFFFu) - (uint32_t)(t16 * kChanTile);
      if ((int)(ch16 >> 3) != half) continue;
      const uint32_t ch = ch16 & 7u;
      const uint32_t pw = pattern_word(lib.m[mt >> 16]);
      uint32_t flags = 0u;
      if (k_out == n_first) flags |= kOpSwap;
      if (k_out == n_ops - 1) flags |= end_flags;
      const uint4 wv = tw4[k];
      ent[2 * k_out] = make_uint4(ch | pw | flags, ch * (uint32_t)kImgPlaneBytesF32 + ((pw >> 17) & 1u) * (uint32_t)kImgRowBytesF32, wv.x, wv.y);
      ent[2 * k_out + 1] = make_uint4(wv.z, wv.w, 0u, 0u);
      ++k_out;
    }
  }
}

__device__ inline bool header_matches(const BlobHeader* h, int F, int C, int K, long long n_keep, int dtype, const MaskTable& lib) {
  if (h->magic != kBlobMagic || h->version != kBlobVersion) return false;
  if (h->F != F || h->C != C || h->K != K || h->dtype != dtype || h->n_keep != n_keep) return false;
  for (int j = 0; j < K; ++j) if (h->masks[j] != lib.m[j]) return false;
  return true;
}

// One block per re-ordered filter: its kept entries are put into a row of zeros in shared memory, which leaves in one
// piece (a memset before the kernel costs another launch and another pass over the output).
// ROW = false (C too large for that): into the output, zeroed by a memset before.
constexpr int kUnpackThreads = 256;
template <typename T, bool ROW>
__global__ void __launch_bounds__(kUnpackThreads) k_unpack(BlobPtrs bp, int F, int C, int K, long long n_keep, int dtype, MaskTable lib,
                                                           float* __restrict__ out, int* status) {
  extern __shared__ __align__(16) float s_row[];           // [C][9] (ROW only)
  const int n = 9 * C;
  if (ROW)
    for (int e = threadIdx.x; e < n; e += kUnpackThreads) s_row[e] = 0.0f;
  pdl_wait();
  if (!header_matches(bp.hdr, F, C, K, n_keep, dtype, lib)) {
    // the output of a refused blob is all zeros, as it was with the memset
    if (ROW)
      for (int e = threadIdx.x; e < n; e += kUnpackThreads) out[(size_t)blockIdx.x * n + e] = 0.0f;
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicExch(status, PAT_ERR_BLOB);
    return;
  }
  const int q = blockIdx.x;
  const int f = bp.perm[q];
  const T* w4 = static_cast<const T*>(bp.w4);
  float* row = ROW ? s_row : out + (size_t)f * n;
  if (ROW) __syncthreads();
  const int32_t* pp = bp.pptr + (size_t)q * (K + 1);
  const int a = bp.fptr[q], b = bp.fptr[q + 1];
  for (int k = a + threadIdx.x; k < b; k += kUnpackThreads) {
    int lo = 0, hi = K - 1;                  // the pattern segment that holds kernel k: the last one that starts at or before it
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (pp[mid] <= k) lo = mid; else hi = mid - 1;
    }
    unsigned m = lib.m[lo];
    float* dst = row + 9 * (int)bp.chan[k];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      dst[__ffs(m) - 1] = (float)w4[(size_t)k * 4 + t];
      m &= m - 1u;
    }
  }
  if (!ROW) return;
  __syncthreads();
  float* o = out + (size_t)f * n;
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(o) & 15) == 0) {
    done = n & ~3;
    for (int e = 4 * threadIdx.x; e < done; e += 4 * kUnpackThreads) *reinterpret_cast<float4*>(o + e) = *reinterpret_cast<const float4*>(s_row + e);
  }
  for (int e = done + threadIdx.x; e < n; e += kUnpackThreads) o[e] = s_row[e];
}

int common_checks(const char* who, int F, int C, const uint16_t* masks, int K, int64_t n_keep, int dtype) {
  if (F < 1 || C < 1 || F > 65535 || C > 65535) return set_error(PAT_ERR_SHAPE, "%s: F=%d C=%d outside 1..65535", who, F, C);
  if (int rc = check_library(masks, K)) return rc;
  if (dtype != PAT_F32 && dtype != PAT_F16) return set_error(PAT_ERR_DTYPE, "%s: dtype %d", who, dtype);
  if (n_keep < 0 || n_keep > (int64_t)F * C) return set_error(PAT_ERR_INVALID_ARG, "%s: n_keep=%lld outside 0..F*C", who, (long long)n_keep);
  return PAT_OK;
}

MaskTable make_table(const uint16_t* masks, int K) {
  MaskTable lib;
  for (int j = 0; j <= kMaxK; ++j) lib.m[j] = (j < K) ? masks[j] : (uint16_t)0;
  lib.K = K;
  return lib;
}

}  // namespace
}  // namespace pat

using namespace pat;

extern "C" int pat_pack(const float* w_masked, const uint8_t* pattern_id, int F, int C,
                        const uint16_t* masks, int K, int64_t n_keep, int dtype,
                        void* blob, size_t blob_bytes, void* stream) {
  if (!w_masked || !pattern_id || !blob) return set_error(PAT_ERR_INVALID_ARG, "pat_pack: null pointer");
  if (int rc = common_checks("pat_pack", F, C, masks, K, n_keep, dtype)) return rc;
  if (!aligned(blob, 256)) return set_error(PAT_ERR_ALIGN, "pat_pack: blob must be 256-byte aligned");
  BlobLayout L = blob_layout(F, C, K, n_keep, dtype);
  // a buffer sized when such layers had no dense form, which stands behind everything else: the blob goes without
  if (dense_form_end(L, C) && blob_bytes < L.total && blob_bytes >= L.dense) { L.total = L.dense; L.dense = 0; }
  if (blob_bytes < L.total) return set_error(PAT_ERR_WORKSPACE, "pat_pack: blob has %zu bytes, needs %zu", blob_bytes, L.total);
  int* status = status_word();
  if (!status) return set_error(PAT_ERR_CUDA, "pat_pack: cannot resolve the status word");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const MaskTable lib = make_table(masks, K);
  const BlobPtrs bp = blob_ptrs(blob, L, F, K);
  // every check that can refuse the call comes before the first launch
  const size_t table = sizeof(int) * (size_t)L.nct * K;
  const bool use_table = table <= 24 * 1024;
  const size_t lists = (use_table ? table : 0) + sizeof(int) * ((size_t)L.nct + 1) + (size_t)C;
  if (lists > 48 * 1024) return set_error(PAT_ERR_SHAPE, "pat_pack: C=%d too large for the packing kernel", C);
  const size_t smem = lists + sizeof(int) * (L.nblk ? 2 * (((size_t)L.nct + 31) / 32) : 0);
  const auto scatter = dtype == PAT_F16 ? (use_table ? k_pack_scatter<__half, true> : k_pack_scatter<__half, false>)
                                        : (use_table ? k_pack_scatter<float, true> : k_pack_scatter<float, false>);
  // with the kernel's static arrays the last of these sizes are above what a launch gets without asking (always the same value:
  // another thread may be packing another size)
  constexpr int kScatterMost = 49 * 1024;    // lists of 48 KB leave room for 616 bytes of stage bits at most
  if (smem + kScatterStatic > 48 * 1024)
    if (int rc = check_cuda(cudaFuncSetAttribute(scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, kScatterMost), "set shared memory size")) return rc;
  Launches launches;
  launches.add(k_pack_count, dim3(F), dim3(256), K * sizeof(int), st, pattern_id, C, K, bp, status);
  launches.add(k_pack_rank, dim3(F), dim3(kRankThreads), 0, st, F, C, K, (long long)n_keep, dtype, lib, (unsigned long long)L.total, bp, status);
  launches.add(scatter, dim3(F), dim3(kScatterThreads), smem, st, w_masked, pattern_id, C, K, L.nct, L.nblk > 0, lib, bp);
  if (L.nblk > 0) launches.add(k_pack_blocks, dim3(L.nblk), dim3(32), 0, st, L.nct, L.nblk, lib, bp);
  count_launches(launches.n);
  if (launches.error != cudaSuccess) return check_cuda(launches.error, "pat_pack launch");
  return check_cuda(cudaGetLastError(), "pat_pack launch");
}

extern "C" int pat_unpack(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                          int dtype, float* w_dense_out, void* stream) {
  if (!blob || !w_dense_out) return set_error(PAT_ERR_INVALID_ARG, "pat_unpack: null pointer");
  if (int rc = common_checks("pat_unpack", F, C, masks, K, n_keep, dtype)) return rc;
  if (!aligned(blob, 256)) return set_error(PAT_ERR_ALIGN, "pat_unpack: blob must be 256-byte aligned");
  int* status = status_word();
  if (!status) return set_error(PAT_ERR_CUDA, "pat_unpack: cannot resolve the status word");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const BlobLayout L = blob_layout(F, C, K, n_keep, dtype);
  const BlobPtrs bp = blob_ptrs(const_cast<void*>(blob), L, F, K);
  const MaskTable lib = make_table(masks, K);
  const size_t row = sizeof(float) * 9 * (size_t)C;
  cudaError_t le;
  if (row <= 48 * 1024) {
    le = launch_dependent(dtype == PAT_F16 ? k_unpack<__half, true> : k_unpack<float, true>, dim3(F), dim3(kUnpackThreads), row, st,
                          bp, F, C, K, (long long)n_keep, dtype, lib, w_dense_out, status);
  } else {
    if (int rc = check_cuda(cudaMemsetAsync(w_dense_out, 0, sizeof(float) * 9 * (size_t)F * C, st), "pat_unpack memset")) return rc;
    le = launch_dependent(dtype == PAT_F16 ? k_unpack<__half, false> : k_unpack<float, false>, dim3(F), dim3(kUnpackThreads), 0, st,
                          bp, F, C, K, (long long)n_keep, dtype, lib, w_dense_out, status);
  }
  if (le != cudaSuccess) return check_cuda(le, "pat_unpack launch");
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pat_unpack launch");
}
