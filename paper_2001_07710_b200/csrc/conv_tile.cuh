// Pieces shared by the convolution kernels (sm_100a): PTX wrappers (mbarrier, shared memory, tensor memory), bounded waits
// and the thread-tile geometry of the multiply-add kernel (conv_f32_img.cu).
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace pat {
namespace tile {

constexpr int TR4 = 4, TC = 14;         // pixel tile of a thread
constexpr int LX = 4, LY = 8;           // tiles of a warp: 4 column slots x 8 tile rows
constexpr int RF = 2;                   // filters per consumer warp
constexpr int NCW = 16;                // consumer warps of a block
constexpr int FG = NCW * RF;            // filters per work item (32)
static_assert(FG == kExecGroup, "a work item is one execution group of the blob");
constexpr int LAUNCH_REGS = 96;         // registers per thread at launch (the pool that setmaxnreg redistributes)
constexpr uint32_t kSpinLimit = 1u << 22;
constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s: far beyond any healthy wait
constexpr int kFillSleepNs = 200;                       // pause between polls of a waiting producer warp

// ------------------------------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after limit_ns of wall time (or kSpinLimit polls), raises the block-wide abort flag
// and returns false; also returns false as soon as another thread of the block has given up.
// SLEEP_NS > 0: sleep between polls.  Warps with slack wait that way (producers, epilogues): a polling warp takes issue
// slots from the others of its SM partition.  Warps that must restart at once poll without sleeping.
template <int SLEEP_NS>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns = kWaitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
    if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 31u) == 31u) {
      if (*abort_flag) return false;
      if (global_ns() - t0 > limit_ns) break;
    }
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void lds128(uint32_t addr, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(addr));
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t a) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}
// ---- tensor memory (256 KB per SM, 128 lanes x 512 columns of 32 bits) as the multiply-add kernel uses it: it only parks the accumulators of the filter a warp is not working on, so that the per-pattern
// code exists once (for one set of accumulator registers) and stays inside the instruction cache.  A warp may
// touch the 32 lanes of its own quarter (warp index % 4); thread i of the warp reads / writes lane i.
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {      // whole warp; ncols: power of two >= 32
  __syncwarp();
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {         // whole warp
  __syncwarp();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
template <int REGS>
__device__ __forceinline__ void set_warp_registers() {
  if constexpr (REGS > LAUNCH_REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS));
  else if constexpr (REGS < LAUNCH_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS));
}

// ---- 4 x 14 pixel tiles (56 accumulators)
__host__ __device__ constexpr int last_tap_row(uint32_t mask) { return (mask >> 6) ? 2 : ((mask >> 3) ? 1 : 0); }

// A tile in tensor memory: 56 consecutive columns of the thread's lane, value (y, x) at column 14 y + x, moved by
// three transfers of 32, 16 and 8 columns whose register lists are the tile in that order (no padding values, so
// the accumulators can stay where they are).  tmem_store_tile / tmem_load_tile only issue the transfers;
// tmem_wait_st / tmem_wait_ld complete them.
#define PAT_F(i) "f"(a[(i) / TC][(i) % TC])
#define PAT_O(i) "=f"(a[(i) / TC][(i) % TC])
__device__ __forceinline__ void tmem_store_tile(uint32_t taddr, const float (&a)[TR4][TC]) {
  static_assert(TR4 * TC == 56, "32 + 16 + 8 columns");
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), PAT_F(0), PAT_F(1), PAT_F(2), PAT_F(3), PAT_F(4), PAT_F(5), PAT_F(6), PAT_F(7), PAT_F(8), PAT_F(9), PAT_F(10),
        PAT_F(11), PAT_F(12), PAT_F(13), PAT_F(14), PAT_F(15), PAT_F(16), PAT_F(17), PAT_F(18), PAT_F(19), PAT_F(20), PAT_F(21),
        PAT_F(22), PAT_F(23), PAT_F(24), PAT_F(25), PAT_F(26), PAT_F(27), PAT_F(28), PAT_F(29), PAT_F(30), PAT_F(31)
      : "memory");
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr + 32u), PAT_F(32), PAT_F(33), PAT_F(34), PAT_F(35), PAT_F(36), PAT_F(37), PAT_F(38), PAT_F(39), PAT_F(40),
        PAT_F(41), PAT_F(42), PAT_F(43), PAT_F(44), PAT_F(45), PAT_F(46), PAT_F(47)
      : "memory");
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
      ::"r"(taddr + 48u), PAT_F(48), PAT_F(49), PAT_F(50), PAT_F(51), PAT_F(52), PAT_F(53), PAT_F(54), PAT_F(55)
      : "memory");
}
__device__ __forceinline__ void tmem_load_tile(uint32_t taddr, float (&a)[TR4][TC]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : PAT_O(0), PAT_O(1), PAT_O(2), PAT_O(3), PAT_O(4), PAT_O(5), PAT_O(6), PAT_O(7), PAT_O(8), PAT_O(9), PAT_O(10),
        PAT_O(11), PAT_O(12), PAT_O(13), PAT_O(14), PAT_O(15), PAT_O(16), PAT_O(17), PAT_O(18), PAT_O(19), PAT_O(20), PAT_O(21),
        PAT_O(22), PAT_O(23), PAT_O(24), PAT_O(25), PAT_O(26), PAT_O(27), PAT_O(28), PAT_O(29), PAT_O(30), PAT_O(31)
      : "r"(taddr) : "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : PAT_O(32), PAT_O(33), PAT_O(34), PAT_O(35), PAT_O(36), PAT_O(37), PAT_O(38), PAT_O(39), PAT_O(40),
        PAT_O(41), PAT_O(42), PAT_O(43), PAT_O(44), PAT_O(45), PAT_O(46), PAT_O(47)
      : "r"(taddr + 32u) : "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : PAT_O(48), PAT_O(49), PAT_O(50), PAT_O(51), PAT_O(52), PAT_O(53), PAT_O(54), PAT_O(55)
      : "r"(taddr + 48u) : "memory");
}
#undef PAT_F
#undef PAT_O

}  // namespace tile
}  // namespace pat
