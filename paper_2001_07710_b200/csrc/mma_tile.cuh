// Pieces shared by the tensor-core convolution kernels: PTX wrappers (tcgen05, TMA,
// clusters), the numbering of positions that turns a 3x3 convolution into nine shifted matrix products over the same
// shared-memory rows, and the epilogue that writes NHWC results.
//
// Positions.  An image (or a column strip of a wide one) is seen as rows of P positions: the output columns plus one
// column of padding (the right neighbour of a row's last column is the left padding of the next row), or plus two real
// halo columns when the image is cut into strips.  Rows of all images are stacked, one zero row (two when pooling)
// between images.  In this numbering the output at position m needs, for kernel tap (r, s), the input at position
// m + r P + s of the same numbering moved up by one row and left by one column: the A operand of a tap is the same
// shared-memory buffer, started r P + s rows further on.  What is lost is the padding
// positions: about 1 / (W + 1) + 1 / (H + 1) of the multiply-adds.
// Stride 2: the input is taken as four planes (even / odd rows x even / odd columns), each with the one, two or four
// taps that read it, again by constant shifts.
#pragma once
#include <algorithm>
#include <type_traits>
#include <cuda.h>
#include "conv_tile.cuh"
#include "plain_tile.cuh"

namespace pat {
namespace tmma {
using tile::smem_u32;
using tile::mbar_init;
using tile::mbar_arrive;
using tile::mbar_arrive_expect_tx;
using tile::mbar_try_wait;
using tile::mbar_wait;
using tile::global_ns;
using tile::kSpinLimit;

constexpr int SUB = 128;                   // rows of one accumulator
constexpr int MAX_P = 62;                  // positions per row
constexpr int EPI_WARPS = 8;
constexpr uint32_t TMEM_COLS = 512;
constexpr int RING_AT = 1024, RING_TO = 232448;      // shared memory behind the barriers

// What the kernels' parameter blocks have in common.
struct Geometry {
  const void* x;
  void* y;
  const BlobHeader* hdr;
  const int32_t *inv, *pptr; // the packed kernels in canonical order, see kept_taps
  const uint16_t* chan;
  const void* w4;
  int* status;
  int N, H, W, F, C, K, dtype;
  long long n_keep;
  unsigned long long dense_end;  // dense_form_end of the layer
  int Ho, Wo;                // output size before pooling
  int P, HP, Ws, strips;     // positions per row, rows per image (with its zero rows), columns and number of strips
  int tile_size, mstep;      // positions of a tile, positions from one tile to the next (whole row pairs when pooling)
  int ext;                   // last input position a tile needs, counted from its first
  int tiles;
  int BN, groups;            // filters per group (multiple of 16), groups
  int items;                 // work items: (tile or pair of tiles) x group, groups fastest
  int ncb, ks_last;          // channel blocks, 16-channel steps of the last one
  int stride, planes;        // input planes (1, or 4 for stride 2)
  int parts, lparts;         // CTAs of a cluster that share an item's channel blocks (a power of two), its logarithm
  uint32_t recv;             // parts > 1: where the other CTAs' partial sums arrive, from the start of shared memory
  int share;                 // columns that one part adds up, at most
  int handshake;             // that place overlaps the rings: its owner says when they are free
  int act;                   // 0, 1: rectifier, 2: rectifier and 2 x 2 max pooling
  int wide;                  // rows of results start at multiples of 32 bytes
  int b_slots;               // ring slots of weights
  uint32_t b_bytes;          // bytes of one
  uint32_t idesc;
  unsigned long long wait_ns;   // limit of every wait
  int test_skip;             // test hook: the weights of this stage number are never copied (-1: none)
  FastDiv d_P, d_HP, d_strips, d_groups, d_chunks;
  uint16_t masks[256];
};

// ------------------------------------------------------------------------------------------ PTX
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Instructions marked .aligned are undefined in a warp whose lanes have parted, and only __syncwarp() promises that they have met
// again behind a branch that they did not all take.  The ones that run a few times a launch begin with it; for those on tensor
// memory, store_piece and send_part, whose branches precede them, end with it.

// The two halves of a barrier of the whole cluster (threads that have exited count as arrived).
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// The same for a slot that has been read: nothing that this thread has written is passed on with it, so it need not wait until that is
// seen by the cluster.
__device__ __forceinline__ void arrive_remote_read(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Sixteen bytes into another CTA's shared memory; they are counted on its barrier when they have arrived.
__device__ __forceinline__ void store_async(uint32_t addr, const float4& v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];"
               ::"r"(addr), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar) : "memory");
}
// What the other CTAs stored before a completed phase of the barrier is seen from here on.
__device__ __forceinline__ void acquire_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
}
// Copies of a CTA pair report to the barrier of the pair's even CTA (bit 24 of a shared::cluster address is the CTA).
template <int CG>
__device__ __forceinline__ void load_4d(uint32_t dst, const CUtensorMap* m, int c, int x, int y, int n, uint32_t bar) {
  if constexpr (CG == 2)
    asm volatile("cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(x), "r"(y), "r"(n), "r"(bar & 0xFEFFFFFFu) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(x), "r"(y), "r"(n), "r"(bar) : "memory");
}
template <int CG>
__device__ __forceinline__ void load_3d(uint32_t dst, const CUtensorMap* m, int c, int f, int t, uint32_t bar) {
  if constexpr (CG == 2)
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(f), "r"(t), "r"(bar & 0xFEFFFFFFu) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(f), "r"(t), "r"(bar) : "memory");
}
__device__ __forceinline__ void prefetch_4d(const CUtensorMap* m, int c, int x, int y, int n) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global [%0, {%1, %2, %3, %4}];" ::"l"(m), "r"(c), "r"(x), "r"(y), "r"(n) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}
// Descriptor of a K-major operand: rows of ROW = 128 or 64 bytes with the swizzle of that span (taken on address bits, so
// a matrix may start at any row), eight rows from one group to the next.
template <int ROW> constexpr uint32_t kOperandHi = (ROW * 8u >> 4) | (1u << 14) | ((ROW == 128 ? 2u : 4u) << 29);
__device__ __forceinline__ uint32_t operand_lo(uint32_t addr) { return ((addr & 0x3FFFFu) >> 4) | (1u << 16); }
// D (tensor memory) = A B, plus D when `accumulate` is set; a, b: low words of the operands' descriptors.
template <int CG, int ROW>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t accumulate) {
#define PAT_MMA(G)                                                                                                       \
  asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b64 x, {%1, %5};\n\tmov.b64 y, {%2, %5};\n\t" \
               "tcgen05.mma.cta_group::" G ".kind::f16 [%0], x, y, %3, p;\n\t}"                                        \
               ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"(accumulate), "n"(kOperandHi<ROW>) : "memory")
  if constexpr (CG == 2) PAT_MMA("2"); else PAT_MMA("1");
#undef PAT_MMA
}
// The multiply-adds issued so far by this thread arrive on the barrier (of both CTAs of a pair) when they are done.
// `pair`: cluster rank of the pair's even CTA.
template <int CG>
__device__ __forceinline__ void commit(uint32_t bar, uint32_t pair) {
  if constexpr (CG == 2)
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((unsigned short)(3u << pair)) : "memory");
  else
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
template <int CG>
__device__ __forceinline__ void alloc_columns(uint32_t smem_dst) {
  __syncwarp();
  if constexpr (CG == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "n"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  } else {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "n"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
}
template <int CG>
__device__ __forceinline__ void free_columns(uint32_t taddr) {
  __syncwarp();
  if constexpr (CG == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(TMEM_COLS) : "memory");
  else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(TMEM_COLS) : "memory");
}
__device__ __forceinline__ void tmem_load16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                 "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_store16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
                 "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
// v += the sums of 16 columns in tensor memory, rounded to nearest.
__device__ __forceinline__ void tmem_add16(uint32_t taddr, uint32_t (&v)[16]) {
  uint32_t s[16];
  tmem_load16(taddr, s);
  tile::tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(s[i]));
}
__device__ __forceinline__ bool all_epilogue_warps(bool v) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\tbarrier.cta.red.and.pred b, 2, %2, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
               : "=r"(r) : "r"((uint32_t)v), "n"(EPI_WARPS * 32) : "memory");
  return r != 0;
}
// Has the phase completed?  Never suspends the thread: for a look ahead of the wait itself.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// mbar_wait by a whole warp with a warp-uniform answer.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns) {
  if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
  return __all_sync(0xFFFFFFFFu, mbar_wait<0>(bar, parity, abort_flag, limit_ns)) != 0;
}
__device__ __forceinline__ uint32_t pack_f16(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ------------------------------------------------------------------------------------------ positions
// The taps that read an input plane (stride 2; stride 1 has one plane with all nine), along one axis: how many, and for
// the k-th of them its kernel row / column and its shift in rows / columns of positions.
__device__ __forceinline__ int axis_taps(int stride, int odd) { return stride == 1 ? 3 : (odd ? 2 : 1); }
__device__ __forceinline__ int axis_tap(int stride, int odd, int k) { return stride == 1 ? k : (odd ? 2 * k : 1); }
__device__ __forceinline__ int axis_shift(int stride, int odd, int k) { return stride == 1 ? k : (odd ? k : 1); }

// The blob was packed with the parameters of this call (one warp; the same answer in every lane).  A word of the header and masks
// per lane, read side by side: the first weights wait for this.
__device__ __forceinline__ bool blob_matches_warp(const Geometry& p) {
  const int lane = threadIdx.x & 31;
  const BlobHeader* bh = p.hdr;
  static_assert(offsetof(BlobHeader, version) == 4 && offsetof(BlobHeader, F) == 8 && offsetof(BlobHeader, C) == 12 && offsetof(BlobHeader, K) == 16 &&
                offsetof(BlobHeader, dtype) == 20 && offsetof(BlobHeader, n_keep) == 24, "the header's first eight words");
  uint32_t word = 0u, want = 0u, mask = 0u, want_mask = 0u;
  if (lane < 8) word = reinterpret_cast<const uint32_t*>(bh)[lane];
  if (lane < p.K) mask = bh->masks[lane];
  if (lane == 0) want = kBlobMagic;
  if (lane == 1) want = kBlobVersion;
  if (lane == 2) want = (uint32_t)p.F;
  if (lane == 3) want = (uint32_t)p.C;
  if (lane == 4) want = (uint32_t)p.K;
  if (lane == 5) want = (uint32_t)p.dtype;
  if (lane == 6) want = (uint32_t)p.n_keep;
  if (lane == 7) want = (uint32_t)((unsigned long long)p.n_keep >> 32);
  if (lane < p.K) want_mask = p.masks[lane];
  bool ok = word == want && mask == want_mask;
  for (int j = lane + 32; j < p.K; j += 32) ok = ok && bh->masks[j] == p.masks[j];
  return __all_sync(0xFFFFFFFFu, ok) != 0;
}

// The blob holds no dense form, see dense_form_end: the results are formed from the packed kept taps alone (plain_results).  Every
// role finds that out for itself, while it waits for its first data: a wait that is given up takes 130 us to notice it.
__device__ __forceinline__ bool no_dense_form(const Geometry& p) { return p.dense_end != 0 && p.hdr->total_bytes < p.dense_end; }

// Output pixel of position m: index (n Ho + y) Wo + x, or -1 for padding positions.
__device__ __forceinline__ int pixel_of(const Geometry& p, int m, int& y, int& x, int& n) {
  const int v = p.d_P.div(m), i = m - v * p.P;
  const int vi = p.d_HP.div(v);
  y = v - vi * p.HP;
  n = p.d_strips.div(vi);
  const int strip = vi - n * p.strips;
  x = strip * p.Ws + i;
  if (i >= p.Ws || y >= p.Ho || x >= p.Wo || n >= p.N) return -1;
  return (n * p.Ho + y) * p.Wo + x;
}

// ------------------------------------------------------------------------------------------ results
// The larger one, NaN if one of them is.  (fmaxf and __hmax2 give the other one.)
__device__ __forceinline__ float max_nan(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}
template <bool F32>
__device__ __forceinline__ uint32_t max1(uint32_t a, uint32_t b) {
  if constexpr (F32) return __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b)));
  const __half2 m = __hmax2(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
  return *reinterpret_cast<const uint32_t*>(&m);
}
template <bool F32>
__device__ __forceinline__ uint4 max4(const uint4& a, const uint4& b) {
  return make_uint4(max1<F32>(a.x, b.x), max1<F32>(a.y, b.y), max1<F32>(a.z, b.z), max1<F32>(a.w, b.w));
}

// Infinities and NaN.  The dense form multiplies an input by the zeros of removed taps and kernels too, and zero times
// infinity is no number; of an infinity the fp32 kernel's three parts are infinity, NaN and NaN.  So a sum that is not a number
// may only say that something in its neighbourhood is not finite, and is formed again from the kept taps alone.  (A sum that
// is a number needs nothing: an infinity that it read met a kept weight.)  The epilogue stores such a sum as NaN, with a
// rectifier too, and takes a note; a block that has taken one goes over its results again at the end, when nothing waits
// for it.  With pooling the numbers of a window are stored, and which of its sums were none is told by the inputs and weights
// that they read.  (Forming them in the epilogue itself, out of line, took 0.6 us of an 8.7 us launch in fp16 and 2 of 10 in
// fp32: a call inside its loops costs registers whether it is taken or not.)
struct Note {                              // zero as long as all values seen were finite, then NaN
  float2 t = {0.0f, 0.0f};
  template <bool F32>
  __device__ __forceinline__ void see(const uint4& v) {
    if constexpr (F32) {
      t.x = fmaf(__uint_as_float(v.x), 0.0f, t.x);
      t.y = fmaf(__uint_as_float(v.y), 0.0f, t.y);
      t.x = fmaf(__uint_as_float(v.z), 0.0f, t.x);
      t.y = fmaf(__uint_as_float(v.w), 0.0f, t.y);
    } else {
      const __half2 z = __float2half2_rn(0.0f);
      const __half2* h = reinterpret_cast<const __half2*>(&v);
      __half2 s0 = *reinterpret_cast<__half2*>(&t.x), s1 = *reinterpret_cast<__half2*>(&t.y);     // (two chains)
      s0 = __hfma2(h[2], z, __hfma2(h[0], z, s0));
      s1 = __hfma2(h[3], z, __hfma2(h[1], z, s1));
      t.x = *reinterpret_cast<float*>(&s0);
      t.y = *reinterpret_cast<float*>(&s1);
    }
  }
  // (floats or pairs of halves, each of either sign's zero or NaN)
  __device__ __forceinline__ bool taken() const { return ((__float_as_uint(t.x) | __float_as_uint(t.y)) & 0x7FFF7FFFu) != 0u; }
};
template <bool F32>
__device__ __forceinline__ float stored(const void* a, size_t i) {
  if constexpr (F32) return static_cast<const float*>(a)[i];
  else return __half2float(static_cast<const __half*>(a)[i]);
}
// The sum over the kept taps of filter f for output (n, y, x), in fp32: what the packed weights say.
template <bool F32>
__device__ __noinline__ float kept_taps(const Geometry& p, int f, int n, int y, int x) {
  const int32_t* pp = p.pptr + (size_t)p.inv[f] * (p.K + 1);
  const int y0 = y * p.stride - 1, x0 = x * p.stride - 1;
  float sum = 0.0f;
  for (int j = 0; j < p.K; ++j)
    for (int k = pp[j]; k < pp[j + 1]; ++k) {
      const int c = p.chan[k];
      unsigned m = p.masks[j];
#pragma unroll
      for (int t = 0; t < 4; ++t) {                    // ascending bit order
        const int b = __ffs(m) - 1, yy = y0 + b / 3, xx = x0 + b % 3;
        m &= m - 1u;
        if (yy >= 0 && yy < p.H && xx >= 0 && xx < p.W)
          sum = fmaf(stored<F32>(p.x, (((size_t)n * p.H + yy) * p.W + xx) * p.C + c), stored<F32>(p.w4, (size_t)k * 4 + t), sum);
      }
    }
  return sum;
}
template <bool F32>
__device__ __forceinline__ void store_one(const Geometry& p, size_t at, float v) {
  if constexpr (F32) static_cast<float*>(p.y)[at] = v;
  else static_cast<__half*>(p.y)[at] = __float2half_rn(v);
}
// All results of a layer whose blob holds no dense form, by all threads of all blocks: the tiles of the generic kernel (see
// conv_generic.cu: 8 x 32 outputs, four filters a warp, 16 channels staged at a time) by teams of warps, so that some stage while
// others multiply.  The sums are those of that kernel, in its order.  Bound by staging and by reads of shared memory; a team has as
// many warps as the layer has fours of filters, up to half of the block: what a stage brings then feeds most.  14 or 18 warps a block
// instead of 24 a multiprocessor: 0.5 - 1.4 of the generic kernel's times (28x28x260 -> 256, batch 32, keep 1/4, fp16 725 us, 650
// there, fp32 744, 654; 224x224x36 -> 64, batch 4, fp32 231, 167; 112x112x28 -> 8, batch 16, fp16 39, 73).  A lane per result that
// gathers its own taps, as renew_results does it, took 36900 us for the first one.  Every role looks for the dense form itself, while it
// waits for its first data: a wait that is given up takes 130 us to notice it.
__device__ __forceinline__ void four_floats(const float4& a, float (&v)[4]) { v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; }
__device__ __forceinline__ void four_floats(const uint2& a, float (&v)[4]) {
  const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&a.x)), hi = __half22float2(*reinterpret_cast<const __half2*>(&a.y));
  v[0] = lo.x; v[1] = lo.y; v[2] = hi.x; v[3] = hi.y;
}
constexpr int MAX_TEAMS = 9, TEAM_BARRIER = 3;           // first of the teams' named barriers
template <bool F32, int STRIDE>
__device__ __forceinline__ void plain_results(const Geometry& p, unsigned char* smem, int bytes) {
  using T = typename std::conditional<F32, float, __half>::type;
  using Four = typename std::conditional<F32, float4, uint2>::type;
  using G = plain::Geo<STRIDE>;
  using plain::TH; using plain::TW; using plain::RF; using plain::CB;
  constexpr int STAGE = CB * G::PLANE;
  const int warps = (int)blockDim.x >> 5, quads = (p.F + RF - 1) / RF;
  int4* tapoff = reinterpret_cast<int4*>(smem);          // [K] offsets of the stored taps inside a plane
  float* stages = reinterpret_cast<float*>(smem + 16 * 256);
  const int room = min(MAX_TEAMS, (bytes - 16 * 256) / (STAGE * 4));
  const int teams = min(room, max(2, warps / min(quads, warps / 2))), team = warps / teams, id = ((int)threadIdx.x >> 5) / team;
  const BlobLayout L = blob_layout(p.F, p.C, p.K, p.n_keep, F32 ? PAT_F32 : PAT_F16);
  const char* blob = reinterpret_cast<const char*>(p.hdr);
  const int32_t* perm = reinterpret_cast<const int32_t*>(blob + L.xfilt);
  const int32_t* tptr = reinterpret_cast<const int32_t*>(blob + L.tptr);
  const uint32_t* tmeta = reinterpret_cast<const uint32_t*>(blob + L.tmeta);
  const Four* tw4 = reinterpret_cast<const Four*>(blob + L.tw4);
  const T* x = static_cast<const T*>(p.x);
  for (int i = (int)threadIdx.x; i < p.K; i += (int)blockDim.x) {
    unsigned m = p.masks[i];
    int at[4];
#pragma unroll
    for (int tp = 0; tp < 4; ++tp, m &= m - 1u) {        // ascending bit order
      const int b = __ffs(m) - 1;
      at[tp] = (b / 3) * G::IWP + (b % 3);
    }
    tapoff[i] = make_int4(at[0], at[1], at[2], at[3]);
  }
  __syncthreads();
  if (id >= teams) return;
  const int lane = (int)threadIdx.x & 31, t = (int)threadIdx.x - id * team * 32, warp = t >> 5, threads = team * 32;
  auto meet = [&] { asm volatile("barrier.sync %0, %1;" ::"r"(TEAM_BARRIER + id), "r"(threads) : "memory"); };
  float* tile = stages + id * STAGE;
  const int tiles_x = (p.Wo + TW - 1) / TW, tiles_y = (p.Ho + TH - 1) / TH, passes = (quads + team - 1) / team;
  const long long n_units = (long long)p.N * tiles_y * tiles_x * passes;
  for (long long unit = (long long)blockIdx.x * teams + id; unit < n_units; unit += (long long)gridDim.x * teams) {
    const long long tl = unit / passes, ny = tl / tiles_x;
    const int q0 = ((int)(unit - tl * passes) * team + warp) * RF;
    const int n = (int)(ny / tiles_y), oy0 = (int)(ny - (long long)n * tiles_y) * TH, ox0 = (int)(tl - ny * tiles_x) * TW;
    const int iy0 = oy0 * STRIDE - 1, ix0 = ox0 * STRIDE - 1;
    float acc[RF][TH];
#pragma unroll
    for (int r = 0; r < RF; ++r)
#pragma unroll
      for (int k = 0; k < TH; ++k) acc[r][k] = 0.0f;
    for (int cb = 0; cb < L.nct; ++cb) {
      meet();                                            // the stage before has been read
      for (int i = t; i < G::IH * G::IW; i += threads) {       // a position's 16 channels, in pieces of four (C is a multiple of that)
        const int ty = i / G::IW, tx = i - ty * G::IW, yi = iy0 + ty, xi = ix0 + tx;
        const bool in = yi >= 0 && yi < p.H && xi >= 0 && xi < p.W;
        const T* src = x + (in ? (size_t)((n * p.H + yi) * p.W + xi) * p.C : 0) + cb * CB;
        float* dst = tile + ty * G::IWP + tx;
        constexpr int AT_ONCE = F32 ? 2 : 4;                   // loads of a thread in flight (more in fp32 takes registers from the kernel's own loops)
#pragma unroll 1
        for (int c0 = 0; c0 < CB / 4; c0 += AT_ONCE) {
          Four piece[AT_ONCE];
#pragma unroll
          for (int u = 0; u < AT_ONCE; ++u) {
            piece[u] = {};
            if (in && cb * CB + 4 * (c0 + u) < p.C) piece[u] = *reinterpret_cast<const Four*>(src + 4 * (c0 + u));
          }
#pragma unroll
          for (int u = 0; u < AT_ONCE; ++u) {
            float v[4];
            four_floats(piece[u], v);
#pragma unroll
            for (int k = 0; k < 4; ++k) dst[(4 * (c0 + u) + k) * G::PLANE] = v[k];
          }
        }
      }
      meet();
#pragma unroll
      for (int r = 0; r < RF; ++r) {
        const int q = q0 + r;
        if (q >= p.F) continue;
        const int kb = tptr[(size_t)q * (L.nct + 1) + cb], ke = tptr[(size_t)q * (L.nct + 1) + cb + 1];
        // fp16: the next kernel's word and weights are read ahead
        constexpr bool AHEAD = !F32;
        uint32_t meta = 0u;
        Four next = {};
        if (AHEAD && kb < ke) { meta = tmeta[kb]; next = tw4[kb]; }
        for (int k = kb; k < ke; ++k) {
          if (!AHEAD) { meta = tmeta[k]; next = tw4[k]; }
          const float* plane = tile + ((int)(meta & 0xFFFFu) - cb * CB) * G::PLANE + lane * STRIDE;
          const int4 taps = tapoff[meta >> 16];
          float w[4];
          four_floats(next, w);
          if (AHEAD && k + 1 < ke) { meta = tmeta[k + 1]; next = tw4[k + 1]; }
          const int at[4] = {taps.x, taps.y, taps.z, taps.w};
#pragma unroll
          for (int tp = 0; tp < 4; ++tp) {
            const float* src = plane + at[tp];
#pragma unroll
            for (int j = 0; j < TH; ++j) acc[r][j] = fmaf(w[tp], src[j * STRIDE * G::IWP], acc[r][j]);
          }
        }
      }
    }
    const int ox = ox0 + lane;
    if (ox < p.Wo) {
#pragma unroll
      for (int r = 0; r < RF; ++r) {
        if (q0 + r >= p.F) continue;
        const int f = perm[q0 + r];
#pragma unroll
        for (int k = 0; k < TH; ++k)
          if (oy0 + k < p.Ho) store_one<F32>(p, (((size_t)n * p.Ho + oy0 + k) * p.Wo + ox) * p.F + f, p.act ? fmaxf(acc[r][k], 0.0f) : acc[r][k]);
      }
    }
    __syncwarp();
  }
}

// The results that this block has stored - columns c_begin to c_end of its items - gone over by all its warps.  `all`: none has
// been stored, there is no dense form.
template <bool F32, int CG>
__device__ __noinline__ void renew_results(const Geometry& p, int unit, int n_units, int side, int c_begin, int c_end, bool all) {
  if (all) {
    extern __shared__ __align__(1024) unsigned char smem[];
    if (p.stride == 1) plain_results<F32, 1>(p, smem + RING_AT, RING_TO - RING_AT);
    else plain_results<F32, 2>(p, smem + RING_AT, RING_TO - RING_AT);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = (int)blockDim.x >> 5;
  const int hw = p.Ws >> 1, n_out = p.act == 2 ? (p.d_P.div(p.mstep) >> 1) * hw : p.mstep;
  for (int item = unit; item < p.items; item += n_units) {
    const int tg = p.d_groups.div(item), g = item - tg * p.groups, m0 = (CG * tg + side) * p.mstep;
    const int f0 = g * p.BN + c_begin, f1 = min(g * p.BN + c_end, p.F);
    unsigned odd_filter = 0u;                          // bit j: filter f0 + lane + 32 j has a weight that is not finite
    if (p.act == 2)
      for (int f = f0 + lane, j = 0; f < f1; f += 32, ++j) {
        const int32_t* pp = p.pptr + (size_t)p.inv[f] * (p.K + 1);
        for (size_t i = (size_t)pp[0] * 4; i < (size_t)pp[p.K] * 4; ++i)
          if (!isfinite(stored<F32>(p.w4, i))) odd_filter |= 1u << j;
      }
    for (int t = warp; t < n_out; t += warps) {        // a warp per output pixel
      int yy, xx, nn;
      if (p.act != 2) {
        const int pixel = pixel_of(p, m0 + t, yy, xx, nn);
        if (pixel < 0) continue;
        for (int f = f0 + lane; f < f1; f += 32) {
          const size_t at = (size_t)pixel * p.F + f;
          const float old = stored<F32>(p.y, at);
          if (old == old) continue;
          const float v = kept_taps<F32>(p, f, nn, yy, xx);
          store_one<F32>(p, at, p.act ? fmaxf(v, 0.0f) : v);       // (what pat_relu_maxpool makes of a NaN)
        }
        continue;
      }
      const int jj = t / hw;
      if (pixel_of(p, m0 + 2 * jj * p.P + 2 * (t - jj * hw), yy, xx, nn) < 0) continue;
      unsigned odd = 0u;                               // bit k: the window's k-th sum has read an input that is not finite
      for (int k = 0; k < 4; ++k) {
        bool any = false;
        for (int b = 0; b < 9; ++b) {
          const int y = yy + (k >> 1) + b / 3 - 1, x = xx + (k & 1) + b % 3 - 1;
          if (y < 0 || y >= p.H || x < 0 || x >= p.W) continue;
          for (int c = lane; c < p.C; c += 32) any = any || !isfinite(stored<F32>(p.x, (((size_t)nn * p.H + y) * p.W + x) * p.C + c));
        }
        if (__any_sync(0xFFFFFFFFu, any)) odd |= 1u << k;
      }
      for (int f = f0 + lane, j = 0; f < f1; f += 32, ++j) {
        const unsigned again = (odd_filter >> j) & 1u ? 15u : odd;
        if (!again) continue;
        const size_t at = (((size_t)nn * (p.Ho >> 1) + (yy >> 1)) * (p.Wo >> 1) + (xx >> 1)) * p.F + f;
        float v = fmaxf(stored<F32>(p.y, at), 0.0f);
        for (int k = 0; k < 4; ++k)
          if ((again >> k) & 1u) v = fmaxf(v, kept_taps<F32>(p, f, nn, yy + (k >> 1), xx + (k & 1)));
        store_one<F32>(p, at, v);
      }
    }
  }
}

// One pass of the epilogue with pooling: the results of up to 64 fp16 / 32 fp32 columns lie in the staging, 128 bytes per
// position (16-byte chunks swizzled by the position's low bits), and leave as runs of 128 bytes of NHWC output.  HALVES = 2:
// warps 4-7 hold other columns of the same 128 positions (in staging rows 128-255) instead of 128 more positions.
template <bool F32, int HALVES>
__device__ __forceinline__ void pool_results(const Geometry& p, uint32_t st, int g, int c0, int nc, int m0, int warp, int lane, Note& note) {
  constexpr int PER = F32 ? 4 : 8;                     // values per 16-byte chunk
  const int q = lane & 7, f = g * p.BN + c0 + q * PER;
  const bool mine = q * PER < nc && f < p.F;
  char* y = static_cast<char*>(p.y);
  // 2 x 2 max pooling: a tile is whole pairs of rows, so the four positions of a window lie in the staging
  asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
  const int hw = p.Ws >> 1, n_out = (p.d_P.div(p.mstep) >> 1) * hw, v0 = p.d_P.div(m0);
  const int rbase = HALVES == 2 ? (warp >> 2) * SUB : 0;
  for (int t = ((HALVES == 2 ? warp & 3 : warp) * 32 + lane) >> 3; t < n_out; t += EPI_WARPS / HALVES * 4) {
    const int jj = t / hw, ii = t - jj * hw;
    const int v = v0 + 2 * jj, vi = p.d_HP.div(v), yy = v - vi * p.HP, n = p.d_strips.div(vi);
    const int xx = (vi - n * p.strips) * p.Ws + 2 * ii;
    const bool keep = mine && yy < p.Ho && xx < p.Wo && n < p.N;
    const int r0 = rbase + 2 * jj * p.P + 2 * ii;
    uint4 w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int r = r0 + (k >> 1) * p.P + (k & 1);
      tile::lds128(st + (uint32_t)r * 128u + (uint32_t)((q ^ (r & 7)) << 4), w[k].x, w[k].y, w[k].z, w[k].w);
    }
    const uint4 m = max4<F32>(max4<F32>(w[0], w[1]), max4<F32>(w[2], w[3]));
    if (keep)
#pragma unroll
      for (int k = 0; k < 4; ++k) note.see<F32>(w[k]);
    if (keep) *reinterpret_cast<uint4*>(y + ((((size_t)n * (p.Ho >> 1) + (yy >> 1)) * (p.Wo >> 1) + (xx >> 1)) * p.F + f) * (F32 ? 4 : 2)) = m;
  }
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
}

// One 16-column piece of this lane's position, straight from registers in 32-byte sectors (where rows start at multiples of them).
// What a tile's end costs is the latency of its instructions, and through shared memory there were three times as many:
// 188x188x32 -> 96, fp16, batch 5 22.4 -> 17.9 us, 28x28x128, batch 8 9.8 -> 9.2; fp32 84x88x16 -> 192, batch 36 138 -> 121.
template <bool F32>
__device__ __forceinline__ void store_piece(const Geometry& p, int f, int pixel, const float (&v)[16], Note& note) {
  constexpr int WORDS = F32 ? 16 : 8, PER = F32 ? 4 : 8;
  uint32_t w[WORDS];
  if constexpr (F32) {
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = __float_as_uint(v[i]);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_f16(v[2 * i], v[2 * i + 1]);
  }
  if (pixel >= 0 && f < p.F) {
    char* y = static_cast<char*>(p.y) + ((size_t)pixel * p.F + f) * (F32 ? 4 : 2);
    const int left = p.F - f;                            // a multiple of eight
#pragma unroll
    for (int i = 0; i < WORDS; i += 8) {
      if (F32 && i / 8 * 8 >= left) break;
      note.see<F32>(make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]));
      note.see<F32>(make_uint4(w[i + 4], w[i + 5], w[i + 6], w[i + 7]));
      if (p.wide && (F32 || left >= 16)) {
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(y + 4 * i), "r"(w[i]), "r"(w[i + 1]), "r"(w[i + 2]), "r"(w[i + 3]),
                     "r"(w[i + 4]), "r"(w[i + 5]), "r"(w[i + 6]), "r"(w[i + 7]) : "memory");
      } else {
        *reinterpret_cast<uint4*>(y + 4 * i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
        if ((i + 4) * PER / 4 < left) *reinterpret_cast<uint4*>(y + 4 * i + 16) = make_uint4(w[i + 4], w[i + 5], w[i + 6], w[i + 7]);
      }
    }
  }
  __syncwarp();                                        // positions of padding store nothing
}

// One 16-column piece of a position's results into the staging (see pool_results).
template <bool F32>
__device__ __forceinline__ void stage_results(uint32_t row, uint32_t sw, int q, const float (&f)[16]) {
  if constexpr (F32) {
#pragma unroll
    for (int h = 0; h < 4; ++h)
      tile::sts128(row + (((uint32_t)(4 * q + h) ^ sw) << 4), __float_as_uint(f[4 * h]), __float_as_uint(f[4 * h + 1]),
                     __float_as_uint(f[4 * h + 2]), __float_as_uint(f[4 * h + 3]));
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      tile::sts128(row + (((uint32_t)(2 * q + h) ^ sw) << 4), pack_f16(f[8 * h], f[8 * h + 1]), pack_f16(f[8 * h + 2], f[8 * h + 3]),
                     pack_f16(f[8 * h + 4], f[8 * h + 5]), pack_f16(f[8 * h + 6], f[8 * h + 7]));
  }
}

// parts > 1: CTA q * CG + side of the cluster has the sums of channel piece q, and each part adds up its share of the columns
// (chunks of PER of them: 16 bytes of results).  A CTA sends its sums where they are added up, [part][four columns][T
// positions][4] fp32, straight from its registers: stores into another CTA's shared memory move 17 bytes per clock and SM
// and need nobody to wait for them, loads from it 7 (64 KB in a cluster of four: 3000 against 6800 clocks), and a barrier
// that counts the bytes replaces two cluster-wide ones.  Positions that are not in the output are not sent.
constexpr int MAX_PARTS_MMA = 8;
template <bool F32> constexpr int kPer = F32 ? 4 : 8;
template <bool F32>
__device__ __forceinline__ int first_column(const Geometry& p, int part) { return (part * (p.BN / kPer<F32>) >> p.lparts) * kPer<F32>; }
// The bytes that the other parts send for `positions` positions.
template <bool F32>
__device__ __forceinline__ uint32_t expected_bytes(const Geometry& p, int part, int positions) {
  return (uint32_t)((p.parts - 1) * positions * (first_column<F32>(p, part + 1) - first_column<F32>(p, part))) * 4u;
}
// 16 columns, from c on, of position px.
template <bool F32, int T, int CG>
__device__ __forceinline__ void send_part(const Geometry& p, uint32_t sbase, uint32_t bar, uint32_t rank, int c, int px, bool valid, const float (&v)[16]) {
  const int side = (int)rank % CG, part = (int)rank / CG;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int col = c + 4 * i, owner = p.d_chunks.div((col / kPer<F32> + 1) * p.parts - 1);
    const uint32_t at = sbase + p.recv + (uint32_t)((part * p.share + col - first_column<F32>(p, owner)) * T + px * 4) * 4u;
    const float4 w = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    if (owner == part) {
      tile::sts128(at, __float_as_uint(w.x), __float_as_uint(w.y), __float_as_uint(w.z), __float_as_uint(w.w));
    } else if (valid) {
      const uint32_t to = (uint32_t)(owner * CG + side);
      store_async(map_to_rank(at, to), w, map_to_rank(bar, to));
    }
  }
  __syncwarp();                                        // positions of padding send nothing
}
// This CTA's share, by the epilogue's warps, in the order of the channels.
template <bool F32, int T, int CG>
__device__ __forceinline__ void add_parts(const Geometry& p, uint32_t sbase, int item, uint32_t rank, Note& note) {
  constexpr int PER = kPer<F32>, Q = PER / 4, THREADS = EPI_WARPS * 32;
  const int side = (int)rank % CG, part = (int)rank / CG;
  const int tg = p.d_groups.div(item), g = item - tg * p.groups, m0 = (CG * tg + side) * p.mstep;
  const int c_begin = first_column<F32>(p, part), c_end = first_column<F32>(p, part + 1);
  const bool pool = p.act == 2;
  const int px = (int)threadIdx.x & ((pool ? T / 4 : T) - 1);
  int yy, xx, nn, pos = px, pixel;
  size_t out;
  if (pool) {
    const int hw = p.Ws >> 1, jj = px / hw;
    pos = 2 * jj * p.P + 2 * (px - jj * hw);
    pixel = px < (p.d_P.div(p.mstep) >> 1) * hw ? pixel_of(p, m0 + pos, yy, xx, nn) : -1;
    if (pixel < 0) return;
    out = ((size_t)nn * (p.Ho >> 1) + (yy >> 1)) * (p.Wo >> 1) + (xx >> 1);
  } else {
    pixel = px < p.mstep ? pixel_of(p, m0 + px, yy, xx, nn) : -1;
    if (pixel < 0) return;
    out = (size_t)pixel;
  }
  char* y = static_cast<char*>(p.y);
  const uint32_t part_bytes = (uint32_t)(p.share * T) * 4u;
  for (int c = c_begin + (pool ? (int)threadIdx.x / (T / 4) : (int)threadIdx.x / T) * PER; c < c_end; c += (pool ? THREADS / (T / 4) : THREADS / T) * PER) {
    const int f = g * p.BN + c;
    if (f >= p.F) break;
    float s[PER];
#pragma unroll 1
    for (int k = 0; k < (pool ? 4 : 1); ++k) {
      const uint32_t at = sbase + p.recv + (uint32_t)((c - c_begin) * T + (pos + (k >> 1) * p.P + (k & 1)) * 4) * 4u;
      float v[PER];
#pragma unroll
      for (int j = 0; j < Q; ++j) {
        uint32_t w[MAX_PARTS_MMA][4];
#pragma unroll
        for (int q = 0; q < MAX_PARTS_MMA; ++q) {
          if (q >= p.parts) break;
          tile::lds128(at + (uint32_t)q * part_bytes + (uint32_t)(j * T * 16), w[q][0], w[q][1], w[q][2], w[q][3]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) v[4 * j + i] = 0.0f;
#pragma unroll
        for (int q = 0; q < MAX_PARTS_MMA; ++q) {
          if (q >= p.parts) break;
#pragma unroll
          for (int i = 0; i < 4; ++i) v[4 * j + i] += __uint_as_float(w[q][i]);
        }
      }
      if (pool)
#pragma unroll
        for (int j = 0; j < PER; j += 4)
          note.see<true>(make_uint4(__float_as_uint(v[j]), __float_as_uint(v[j + 1]), __float_as_uint(v[j + 2]), __float_as_uint(v[j + 3])));
#pragma unroll
      for (int j = 0; j < PER; ++j) s[j] = k == 0 ? v[j] : fmaxf(s[j], v[j]);
    }
    if (p.act)
#pragma unroll
      for (int j = 0; j < PER; ++j) s[j] = pool ? fmaxf(s[j], 0.0f) : max_nan(s[j], 0.0f);
    uint4 r;
    if constexpr (F32) r = make_uint4(__float_as_uint(s[0]), __float_as_uint(s[1]), __float_as_uint(s[2]), __float_as_uint(s[3]));
    else r = make_uint4(pack_f16(s[0], s[1]), pack_f16(s[2], s[3]), pack_f16(s[4], s[5]), pack_f16(s[6], s[7]));
    if (!pool) note.see<true>(make_uint4(__float_as_uint(s[0]), __float_as_uint(s[1]), __float_as_uint(s[2]), __float_as_uint(s[3])));
    if (!pool && PER == 8) note.see<true>(make_uint4(__float_as_uint(s[PER - 4]), __float_as_uint(s[PER - 3]), __float_as_uint(s[PER - 2]), __float_as_uint(s[PER - 1])));
    *reinterpret_cast<uint4*>(y + (out * p.F + f) * (F32 ? 4 : 2)) = r;
  }
}
// Before the sums are sent: the barrier is told how many bytes come, and the place they go to is free in every CTA.
template <bool F32, int CG>
__device__ __forceinline__ bool open_exchange(const Geometry& p, uint32_t received, uint32_t go, uint32_t rank, int warp, int lane, bool valid,
                                              volatile int* abort_flag) {
  const unsigned there = __ballot_sync(0xFFFFFFFFu, valid);
  if (lane == 0 && (!F32 || warp < 4)) mbar_arrive_expect_tx(received, expected_bytes<F32>(p, (int)rank / CG, __popc(there)));
  if (!p.handshake) return true;
  if (warp == 0 && lane < p.parts) arrive_remote(map_to_rank(go, (uint32_t)(lane * CG) + rank % CG));
  return mbar_wait<0>(go, 0u, abort_flag, p.wait_ns);
}
// The sums of all parts have arrived (for all of the epilogue's warps or for none).
__device__ __forceinline__ bool close_exchange(const Geometry& p, uint32_t received, bool alive, volatile int* abort_flag) {
  alive = alive && mbar_wait<0>(received, 0u, abort_flag, p.wait_ns);
  if (alive) acquire_cluster(received, 0u);
  return all_epilogue_warps(alive);
}

// ------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
// Clusters of `size` CTAs of a kernel that run at the same time (whole SMs each; a cluster stays inside one group of SMs, so
// that e.g. sixteen clusters of eight do not fit 148 SMs).
template <typename Kernel>
int clusters_at_once(Kernel fn, int size, int threads, int smem) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)size; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)size); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = (size_t)smem;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess || n < 1) { (void)cudaGetLastError(); n = 1; }
  return n;
}
inline EncodeFn encode_fn() {
  static const EncodeFn fn = [] {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess;
    return reinterpret_cast<EncodeFn>(ok ? sym : nullptr);
  }();
  return fn;
}

// Where partial sums are exchanged, at the end of shared memory: beside the rings when `ring_needs` bytes are left for
// them.  Returns the rings' bytes.
inline int set_exchange(Geometry& p, int per, int smem_bytes, int ring_at, int ring_bytes, int ring_needs) {
  p.lparts = 0;
  while ((1 << p.lparts) < p.parts) ++p.lparts;
  const int chunks = p.BN / per;
  p.d_chunks.set(chunks);
  p.share = (chunks + p.parts - 1) / p.parts * per;
  const int bytes = p.parts * p.share * p.tile_size * 4;
  p.recv = (uint32_t)(smem_bytes - bytes);
  p.handshake = 0;
  if (p.parts == 1) return ring_bytes;
  if ((int)p.recv - ring_at >= ring_needs) return std::min(ring_bytes, (int)p.recv - ring_at);
  p.handshake = 1;
  return ring_bytes;
}

// Where the packed kernels are (see kept_taps).
inline void set_packed(Geometry& p, const void* x, const void* blob, const BlobLayout& L, int F, int C, int K) {
  p.dense_end = dense_form_end(L, C);
  const char* b = static_cast<const char*>(blob);
  p.x = x;
  p.hdr = reinterpret_cast<const BlobHeader*>(b);
  p.inv = reinterpret_cast<const int32_t*>(b + inv_offset(L, F, K));
  p.pptr = reinterpret_cast<const int32_t*>(b + L.pptr);
  p.chan = reinterpret_cast<const uint16_t*>(b + L.chan);
  p.w4 = b + L.w4;
}

// Positions, tiles and their input rows (see the head of the file).  False: more than an int counts.
inline bool set_geometry(Geometry& p, int tile_size, int N, int H, int W, int stride, int act) {
  p.tile_size = tile_size;
  p.N = N; p.H = H; p.W = W; p.stride = stride; p.act = act;
  p.Ho = (H - 1) / stride + 1; p.Wo = (W - 1) / stride + 1;
  p.strips = p.Wo + 1 <= MAX_P ? 1 : (p.Wo + MAX_P - 3) / (MAX_P - 2);
  p.Ws = (p.Wo + p.strips - 1) / p.strips;
  if (act == 2) p.Ws += p.Ws & 1;                      // pooling windows stay inside a strip
  p.P = p.Ws + (p.strips == 1 ? 1 : 2);
  p.HP = p.Ho + (act == 2 ? 2 : 1);                    // pooling: row pairs start at even rows in every image
  p.planes = stride == 2 ? 4 : 1;
  const int tail = stride == 2 ? p.P + 1 : 2 * p.P + 2;        // how far the last tap reaches
  p.mstep = tile_size;
  int used = tile_size;
  if (act == 2) { p.mstep = tile_size / (2 * p.P) * 2 * p.P; used = p.mstep - (p.P - p.Ws); }
  p.ext = used - 1 + tail;
  const long long total = (long long)N * p.strips * p.HP * p.P, tiles = (total + p.mstep - 1) / p.mstep;
  if (total > 0x7FFFFFFFll - 8 * tile_size || (long long)N * H * W > 0x7FFFFFFFll) return false;
  p.tiles = (int)tiles;
  p.d_P.set(p.P); p.d_HP.set(p.HP); p.d_strips.set(p.strips);
  return true;
}

}  // namespace tmma
}  // namespace pat
