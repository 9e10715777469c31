// Sparse 3x3 convolution on the tensor cores (sm_100a, tcgen05), fp16 storage / fp32 accumulation: an implicit GEMM
// over the masked weights in dense form.
//
// Why dense.  At keep 12.5 % a layer's weights are 5.6 % dense as a GEMM operand, and 1 / 0.056 = 18 times the useful
// multiply-adds have to be executed - but dense fp16 tensor throughput is 22 times the fp32 multiply-add rate, and a
// multiply-add kernel over the kept taps reached 30 - 52 % of that one: it needs the activations re-arranged in a pass of
// its own and is bound by instruction issue.  This kernel reads NHWC activations directly, so the pass is gone too; it was
// the faster one at every density down to 1 % (28x28x512 -> 512, batch 32: 67 against 70 us there, 133 at keep 1/16).
// Measured, VGG-16 at batch 64, keep 12.5 %: 56x56x256 -> 256 390 -> 122 us (1.95 PFLOP/s dense: what the tensor cores
// give at the clock they hold), 224x224x64 -> 64 600 -> 208 us (bound by reading the operands of 256 x 64 products from shared
// memory: 44 clocks for 32 of arithmetic; its bytes take 126).
//
// The positions and shifts that make nine matrix products of a convolution are described in mma_tile.cuh.  A tile of 256
// consecutive positions loads its input rows once and serves all nine taps from them (a TMA copy takes four rows of an image, one
// where fewer are left; out-of-bounds rows and columns arrive as zeros); nine separate tap loads would need 64 B per clock and SM where
// L2 delivers 36.  Stride 2: the tensor map's element strides pick the four planes.
//
// Work split.  CG = 2: a pair of CTAs (cta_group::2) shares a group of up to 256 filters: each CTA holds 256 positions (two
// 128-row accumulators in its tensor memory) and half of the weights, so that a weight tile read from L2 serves 512
// positions.  CG = 1 (small problems): one CTA per 256 positions and up to 128 filters, the input channels cut into
// `parts` pieces that run on the CTAs of a cluster and are added up through distributed shared memory in a fixed order.
//
// Accuracy.  Products are exact in the tensor core's fp32 sums, but those drop what does not fit their last bit, about 2^-24.5
// of the running sum a step, so long sums drift towards zero.  They are no longer than CHUNK channels (288 steps; positive
// data: 1.2e-5 low, against 2^-11 of rounding the result); further chunks are added up, rounded to nearest, in columns of
// tensor memory of their own, which halves the filters that a pair takes.
//
// Channels an odd multiple of four (ROWS8): activation rows start at multiples of 8 bytes only, which TMA does not take; four
// warps then fill the same buffers with 8-byte cp.async (four: eight are no faster, the epilogue spills; 56x56x68 -> 200, batch 16:
// 44 us, 72 channels through TMA 26: bound by the copies' issue and, in pairs, by an arrival across the cluster that every
// loading warp makes a stage).  These layers ran the generic multiply-add kernel before (keep 1/4):
// 28x28x260 -> 256, batch 32 650 -> 47 us, 9x10x212 -> 152, batch 8 118 -> 12, 80x81x20 -> 24, stride 2, batch 2 47 -> 14.
//
// Roles: warps 0-7 epilogue (tensor memory -> fp32 -> rectifier -> fp16 -> whole sectors of the output; pooled through shared memory), warp 8
// copies activations, warp 9 weights, warp 10 issues the multiply-adds (in the even CTA of a pair).  Every wait is
// bounded; tensor memory is released on every path.
#include "mma_tile.cuh"

namespace pat {
namespace tmma {
namespace {

constexpr int TILE = 256;                   // positions per CTA
constexpr int KB = 64;                      // channels per stage (128 bytes)
constexpr int W_A = 8, W_B = 9, W_MMA = 10, NWARPS = 12;
constexpr int ROW_WARPS = 4;                // ROWS8: warps that copy activations (W_A and those behind W_MMA)
constexpr int threads_of(bool rows8) { return (rows8 ? W_MMA + ROW_WARPS : NWARPS) * 32; }
constexpr int MAX_A = 4, MAX_B = 8;             // ring slots
constexpr int CHUNK = 8;                        // channel blocks in one sum of the tensor core
constexpr int ST_BYTES = TILE * 128;            // epilogue staging: 128 bytes per position
constexpr int OFF_RING = 1024, RING_BYTES = 198656, OFF_ST = OFF_RING + RING_BYTES, SMEM_BYTES = OFF_ST + ST_BYTES;
static_assert(SMEM_BYTES <= 232448 && OFF_ST % 1024 == 0 && OFF_RING == RING_AT && SMEM_BYTES == RING_TO, "shared memory budget of one SM");
static_assert(SMEM_BYTES - OFF_RING >= (128 + MAX_PARTS_MMA * kPer<false>) * TILE * 4, "the partial sums of 128 filters fit");

struct alignas(64) Maps { CUtensorMap a, rows, b; };     // rows: ROWS image rows at a time
// A tile is 7 (56 columns) to 35 (7 columns) image rows; one thread issues their copies, 50 clocks each, and with four rows in one
// the first stage of 14x14 arrives 700 clocks sooner.  (Whole images at a time would not fit what is left of a slot.)
constexpr int ROWS = 4;

struct Params : Geometry {
  int a_slots;               // ring slots of activations
  uint32_t a_bytes;          // bytes of one
  int resident;              // the weights of the only group stay in shared memory
};

// LONG: more than CHUNK channel blocks.  (A variant of its own: in the common one the branches took 1 % of VGG-16.)
template <int CG, bool LONG, bool ROWS8>
__global__ void __launch_bounds__(threads_of(ROWS8), 1) k_conv_mma_f16(const __grid_constant__ Maps maps, const __grid_constant__ Params p) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sbase = smem_u32(smem);
  auto full_a = [&](int s) { return sbase + 8u * s; };
  auto empty_a = [&](int s) { return sbase + 8u * (MAX_A + s); };
  auto full_b = [&](int s) { return sbase + 8u * (2 * MAX_A + s); };
  auto empty_b = [&](int s) { return sbase + 8u * (2 * MAX_A + MAX_B + s); };
  auto acc_full = [&](int s) { return sbase + 8u * (2 * MAX_A + 2 * MAX_B + s); };
  auto acc_empty = [&](int s) { return sbase + 8u * (2 * MAX_A + 2 * MAX_B + 2 + s); };
  constexpr int BARS = 2 * MAX_A + 2 * MAX_B + 7;
  const uint32_t received = sbase + 8u * (BARS - 3), go = sbase + 8u * (BARS - 2), drain = sbase + 8u * (BARS - 1);
  int& s_abort = *reinterpret_cast<int*>(smem + 8 * BARS);           // a wait has given up, or the blob was refused
  int& s_refused = *reinterpret_cast<int*>(smem + 8 * BARS + 4);
  int& s_note = *reinterpret_cast<int*>(smem + 8 * BARS + 12);       // a result is not finite, see Note
  uint32_t& s_tmem = *reinterpret_cast<uint32_t*>(smem + 8 * BARS + 8);
  int& s_plain = *reinterpret_cast<int*>(smem + 8 * BARS + 16);      // the blob holds no dense form
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = CG == 1 || rank == 0;

  if (threadIdx.x == 0) {
    s_abort = 0;
    s_refused = 0;
    s_note = 0;
    if (ROWS8) s_plain = 0;
  }
  if (!ROWS8 && threadIdx.x == W_A * 32) { prefetch_map(&maps.a); prefetch_map(&maps.rows); }
  if (threadIdx.x == W_B * 32) prefetch_map(&maps.b);
  if (threadIdx.x < BARS) {                // a barrier each: 30 of them in a row by one thread showed in the launch
    const int t = (int)threadIdx.x, acc = t - (2 * MAX_A + 2 * MAX_B + 2);
    const int count = ROWS8 && t < MAX_A ? CG * ROW_WARPS : acc == 0 || acc == 1 ? CG * EPI_WARPS : t == BARS - 3 ? EPI_WARPS : t == BARS - 2 ? p.parts : 1;
    mbar_init(sbase + 8u * (uint32_t)t, (uint32_t)count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W_MMA) alloc_columns<CG>(smem_u32(&s_tmem));
  const int unit = CG == 2 ? (int)(blockIdx.x >> 1) : (int)blockIdx.x / p.parts;
  // Where an item's input rows are.  The tile's first position goes to row P of the slot, wherever it lies in its image row: both CTAs
  // of a pair are addressed by the same descriptors.
  struct Rows { int off, n_rows, y, strip, n; uint32_t bytes; };
  auto find_rows = [&](int item) {
    Rows r;
    const int tg = p.d_groups.div(item);
    const int m0 = (CG == 2 ? 2 * tg + (int)rank : tg) * p.mstep;
    const int v1 = p.d_P.div(m0);
    r.off = m0 - v1 * p.P;
    r.n_rows = p.d_P.div(r.off + p.ext) + 1;
    r.bytes = (uint32_t)(r.n_rows * p.P) * 128u;
    if (CG == 2) {                           // and the other CTA's copies, which report here too (rank 0 arms the barrier)
      const int m1 = m0 + p.mstep;
      r.bytes += (uint32_t)((p.d_P.div(m1 - p.d_P.div(m1) * p.P + p.ext) + 1) * p.P) * 128u;
    }
    const int v0 = v1 - 1, vi = v0 < 0 ? 0 : p.d_HP.div(v0);
    r.y = v0 - vi * p.HP;                    // -1 above the first image
    r.n = p.d_strips.div(vi);
    r.strip = vi - r.n * p.strips;
    return r;
  };
  // The other CTAs' barriers exist: a pair waits for that before its first copy, the parts of a layer before they send sums.
  // Blocks take a whole SM each, so most of a launch's blocks start when the kernel before it ends: what they do until
  // here is not hidden.
  const bool clustered = CG == 2 || p.parts > 1;
  if (clustered) cluster_arrive();
  bool met = !clustered, left = false;     // has waited for the first, has arrived at the last barrier of the cluster
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  Rows at = {};
  if (!ROWS8 && warp == W_A) at = find_rows(unit);     // while the kernel before this one still runs
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (CG == 2) { cluster_wait(); met = true; }
  volatile int* abort_flag = &s_abort;
  const uint32_t tmem = s_tmem;
  const uint32_t ring_b = sbase + OFF_RING + (uint32_t)p.a_slots * p.a_bytes;

  // accumulator sets, beside the columns of the sums over several chunks
  const int sum_cols = LONG ? 2 * p.BN : 0, n_acc = 2 * 2 * p.BN + sum_cols <= (int)TMEM_COLS ? 2 : 1;
  // CG = 2: a pair walks over the items; CG = 1: a cluster of `parts` CTAs has one item, or single CTAs walk
  const int n_units = CG == 2 ? (int)(gridDim.x >> 1) : (int)gridDim.x / p.parts;
  const int cb0 = CG == 2 ? 0 : (int)rank * p.ncb / p.parts;
  const int cb1 = CG == 2 ? p.ncb : ((int)rank + 1) * p.ncb / p.parts;
  const int rows_b = p.BN / CG;
  bool alive = true;
  // After a failed wait the copies that a thread has armed still write this block's shared memory: (bounded) time to land.
  auto let_land = [&](uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = global_ns();
    for (uint32_t spin = 0; spin < kSpinLimit && !mbar_try_wait(bar, parity) && global_ns() - t0 <= p.wait_ns; ++spin) {}
  };

  if (ROWS8 && (warp == W_A || warp > W_MMA)) {
    // =========================================================================== activations, in pieces of four channels
    // The rows, their order and places are those of the TMA copies below; a warp takes every fourth row, 2, 4 or 8 positions at
    // a time (as many pieces of each as the stage's channel steps read).  A stage is reported when the next one's copies have
    // been issued, or when its slot is not free yet.  (What this costs is the latency of the address arithmetic: four copies
    // are computed side by side.)
    const int lw = warp == W_A ? 0 : warp - W_MMA;
    const __half* x = static_cast<const __half*>(p.x);
    const uint64_t blob_bytes = p.hdr->total_bytes;     // looked at when the first copies have been issued
    int slot = 0, pending = -1;
    uint32_t par = 1u;
    auto report = [&](int s) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // before the tensor core reads them
      __syncwarp();
      if (lane == 0) {
        if (CG == 2) arrive_remote(map_to_rank(full_a(s), 0u));
        else mbar_arrive(full_a(s));
      }
    };
    for (int item = unit; item < p.items && alive; item += n_units) {
      const int tg = p.d_groups.div(item);
      const int m0 = (CG == 2 ? 2 * tg + (int)rank : tg) * p.mstep;
      const int v1 = p.d_P.div(m0), off = m0 - v1 * p.P, rows = p.d_P.div(off + p.ext) + 1;
      for (int cb = cb0; cb < cb1 && alive; ++cb) {
        const int ks = cb + 1 == p.ncb ? p.ks_last : KB / 16, lp = ks == 1 ? 2 : ks == 2 ? 3 : 4;     // 2^lp pieces of a position
        const int piece = lane & ((1 << lp) - 1), i0 = lane >> lp, di = 32 >> lp, c = cb * KB + piece * 4;
        for (int pl = 0; pl < p.planes; ++pl) {
          const int dy = pl >> 1, dx = (pl & 1) - p.stride;
          if (!__all_sync(0xFFFFFFFFu, mbar_try_wait(empty_a(slot), par))) {
            if (pending >= 0) {
              asm volatile("cp.async.wait_all;" ::: "memory");
              report(pending);
              pending = -1;
            }
            if (!__all_sync(0xFFFFFFFFu, mbar_wait<20>(empty_a(slot), par, abort_flag, p.wait_ns))) { alive = false; break; }
          }
          const uint32_t row0 = sbase + OFF_RING + (uint32_t)slot * p.a_bytes;
          // Narrow images: what counts is the number of rows that a warp goes through, one after the other, most of its lanes idle.
          // There the lanes take positions of any row, which costs three divisions a piece (400 7x7x36, stride 2, 64 filters 19 -> 23
          // us: so only below).  4 -> 64, us, rows and positions: 1x1 16.5, 6.2, stride 2 50.6, 9.5; 7x7 8.3, 6.4; 28x28 6.5, 6.9.
          if (2 * p.P <= 5 * di) {
            const int total = rows * p.P;
            for (int e0 = 4 * di * lw + i0; e0 < total; e0 += ROW_WARPS * 4 * di)
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                const int e = e0 + u * di, j = p.d_P.div(e), i = e - j * p.P;
                const int v = v1 - 1 + j, vi = v < 0 ? 0 : p.d_HP.div(v), yr = v - vi * p.HP, n = p.d_strips.div(vi);
                const int y = yr * p.stride + dy, xx = ((vi - n * p.strips) * p.Ws + i) * p.stride + dx;
                const bool in = yr >= 0 && y < p.H && n < p.N && c < p.C && (unsigned)xx < (unsigned)p.W;
                const uint32_t t = (uint32_t)(p.P - off + e), dst = row0 + t * 128u + ((((uint32_t)piece >> 1) ^ (t & 7u)) << 4) + ((uint32_t)piece & 1u) * 8u;
                if (e < total)
                  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;"
                               ::"r"(dst), "l"(x + (in ? (size_t)((n * p.H + y) * p.W + xx) * p.C + c : 0)), "r"(in ? 8 : 0) : "memory");
              }
          } else {
            for (int j = lw; j < rows; j += ROW_WARPS) {
              const int v = v1 - 1 + j, vi = v < 0 ? 0 : p.d_HP.div(v), yr = v - vi * p.HP, n = p.d_strips.div(vi);
              const int y = yr * p.stride + dy, x0 = (vi - n * p.strips) * p.Ws * p.stride + dx;
              const bool row_in = yr >= 0 && y < p.H && n < p.N && c < p.C;
              const __half* src = x + (((size_t)(row_in ? n : 0) * p.H + (row_in ? y : 0)) * p.W) * p.C + (row_in ? c : 0);
              const uint32_t t0 = (uint32_t)(p.P - off + j * p.P), sub = ((uint32_t)piece & 1u) * 8u, chunk = (uint32_t)piece >> 1;
              const int w = row_in ? p.W : 0;
              for (int i = i0; i < p.P; i += 4 * di)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const int iu = i + u * di, xx = x0 + iu * p.stride;
                  const bool in = (unsigned)xx < (unsigned)w;
                  const uint32_t t = t0 + (uint32_t)iu, dst = row0 + t * 128u + ((chunk ^ (t & 7u)) << 4) + sub;
                  if (iu < p.P)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src + (in ? (ptrdiff_t)xx * p.C : 0)), "r"(in ? 8 : 0) : "memory");
                }
            }
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
          if (pending >= 0) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            report(pending);
          }
          pending = slot;
          if (++slot == p.a_slots) { slot = 0; par ^= 1u; }
          if (blob_bytes < p.dense_end) { alive = false; break; }
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (alive && pending >= 0) report(pending);
  } else if (warp == W_A) {
    // =========================================================================== activations
    if (!ROWS8 && elect_one()) {
      int slot = 0;
      uint32_t par = 1u, armed = 0u, armed_par = 0u;
      const uint32_t row_bytes = (uint32_t)p.P * 128u;
      for (int item = unit; item < p.items && alive; item += n_units) {
        if (item != unit) at = find_rows(item);
        for (int cb = cb0; cb < cb1 && alive; ++cb)
          for (int pl = 0; pl < p.planes; ++pl) {
            const int dy = p.stride == 2 ? (pl >> 1) : 0, dx = (p.stride == 2 ? (pl & 1) : 0) - p.stride;
            // fn(several, x, y, n): the rows from y on, as many of an image as there are at a time
            auto each = [&](auto&& fn) {
              int y = at.y, strip = at.strip, n = at.n;
              for (int left = at.n_rows; left > 0;) {
                const bool several = min(left, p.HP - y) >= ROWS;
                fn(several, strip * p.Ws * p.stride + dx, y * p.stride + dy, n);
                const int step = several ? ROWS : 1;
                left -= step;
                y += step;
                if (y == p.HP) { y = 0; if (++strip == p.strips) { strip = 0; ++n; } }
              }
            };
            if (!mbar_try_wait(empty_a(slot), par)) {
              // the slot is still in use: bring the rows into L2 meanwhile (several from the row above the first image on: some are real)
              each([&](bool several, int x, int y, int n) {
                if ((y >= 0 || several) && y < p.H && n < p.N) prefetch_4d(several ? &maps.rows : &maps.a, cb * KB, x, y, n);
              });
              if (!mbar_wait<20>(empty_a(slot), par, abort_flag, p.wait_ns)) { alive = false; break; }
            }
            if (leader) mbar_arrive_expect_tx(full_a(slot), at.bytes);
            uint32_t dst = sbase + OFF_RING + (uint32_t)slot * p.a_bytes + (uint32_t)(p.P - at.off) * 128u;
            each([&](bool several, int x, int y, int n) {
              load_4d<CG>(dst, several ? &maps.rows : &maps.a, cb * KB, x, y, n, full_a(slot));
              dst += several ? ROWS * row_bytes : row_bytes;
            });
            armed |= 1u << slot;
            armed_par = (armed_par & ~(1u << slot)) | ((par ^ 1u) << slot);
            if (++slot == p.a_slots) { slot = 0; par ^= 1u; }
          }
      }
      if (!alive && leader)
        for (int s = 0; s < p.a_slots; ++s)
          if ((armed >> s) & 1u) let_land(full_a(s), (armed_par >> s) & 1u);
    }
  } else if (warp == W_B) {
    // =========================================================================== weights
    // nothing of the blob but its header is read before the header has been checked (the same answer in every CTA)
    if (!blob_matches_warp(p)) {
      alive = false;
      if (lane == 0) { s_refused = 1; s_abort = 1; atomicExch(p.status, PAT_ERR_BLOB); }
    } else if (ROWS8 && no_dense_form(p)) {
      alive = false;
      if (lane == 0) { s_refused = 1; s_plain = 1; s_abort = 1; }
    } else if (elect_one()) {
      int slot = 0, stage_no = 0;
      uint32_t par = 1u, armed = 0u, armed_par = 0u;
      const uint32_t tile_bytes = (uint32_t)rows_b * 128u;
      bool loaded = false;
      for (int item = unit; item < p.items && alive && !loaded; item += n_units) {
        const int g = item - p.d_groups.div(item) * p.groups;
        const int f0 = g * p.BN + (CG == 2 ? (int)rank * rows_b : 0);
        uint32_t dst_res = ring_b;
        if (p.resident && leader)            // a barrier for each of the first tiles, the last one for all others
          for (int s = 0; s < MAX_B; ++s)
            mbar_arrive_expect_tx(full_b(s), (uint32_t)(CG * (s < MAX_B - 1 ? 1 : 9 * (cb1 - cb0) - (MAX_B - 1))) * tile_bytes);
        for (int cb = cb0; cb < cb1 && alive; ++cb)
          for (int pl = 0; pl < p.planes && alive; ++pl) {
            const int py = pl >> 1, px = pl & 1, nr = axis_taps(p.stride, py), nc = axis_taps(p.stride, px);
            for (int tr = 0; tr < nr && alive; ++tr)
              for (int tc = 0; tc < nc; ++tc, ++stage_no) {
                const int tap = 3 * axis_tap(p.stride, py, tr) + axis_tap(p.stride, px, tc);
                if (p.resident) {
                  if (stage_no != p.test_skip) load_3d<CG>(dst_res, &maps.b, cb * KB, f0, tap, full_b(min(stage_no, MAX_B - 1)));
                  dst_res += tile_bytes;
                  armed = (1u << MAX_B) - 1u;
                  continue;
                }
                if (!mbar_wait<20>(empty_b(slot), par, abort_flag, p.wait_ns)) { alive = false; break; }
                if (leader) mbar_arrive_expect_tx(full_b(slot), (uint32_t)CG * tile_bytes);
                if (stage_no != p.test_skip) load_3d<CG>(ring_b + (uint32_t)slot * p.b_bytes, &maps.b, cb * KB, f0, tap, full_b(slot));
                armed |= 1u << slot;
                armed_par = (armed_par & ~(1u << slot)) | ((par ^ 1u) << slot);
                if (++slot == p.b_slots) { slot = 0; par ^= 1u; }
              }
          }
        loaded = p.resident != 0;
      }
      if (!alive && leader)
        for (int s = 0; s < MAX_B; ++s)
          if ((armed >> s) & 1u) let_land(full_b(s), (armed_par >> s) & 1u);
    }
  } else if (warp == W_MMA) {
    // =========================================================================== multiply-adds (even CTA of a pair)
    // The whole warp runs the loop with warp-uniform values and control flow (so that the operands' descriptors stay in
    // uniform registers) and one elected lane issues.  What the loop costs beside the multiply-adds shows: the tensor core
    // takes a tap's eight of them in 360 clocks at 64 filters; as one thread's loop they were issued in 640.
    if (ROWS8) alive = __all_sync(0xFFFFFFFFu, !no_dense_form(p)) != 0;
    if (leader) {
      const bool el = elect_one();
      int sa = 0, sb = 0, buf = 0;
      uint32_t pa = 0u, pb = 0u, pe = 1u;
      bool res_wait = p.resident != 0;       // the resident weights are still arriving, barrier sb comes next
      // The weights of the next tap are looked at before this tap's products are issued: a wait between two taps, even one
      // that ends at once, lets the tensor core's queue run empty (128 x 64: 49 -> 70 clocks a product).
      bool b_seen = false;
      const uint32_t idesc = p.idesc, row8 = (uint32_t)p.P * 8u;      // descriptors count 16-byte units
      const uint32_t utmem = __reduce_or_sync(0xFFFFFFFFu, tmem), ring_lo = operand_lo(sbase + OFF_RING), ringb_lo = operand_lo(ring_b);
      const uint32_t a_step = p.a_bytes >> 4, b_step = p.b_bytes >> 4;
      for (int item = unit; item < p.items && alive; item += n_units) {
        if (!wait_warp(acc_empty(buf), pe, abort_flag, p.wait_ns)) { alive = false; break; }
        uint32_t d0 = utmem + (uint32_t)(buf * 2 * p.BN), d1 = d0 + (uint32_t)p.BN;
        uint32_t acc = 0u;
        uint32_t b_res = ringb_lo;
        for (int cb = cb0, chunk_end = cb0 + CHUNK; cb < cb1 && alive; ++cb) {
          if (LONG && cb == chunk_end) {       // on with the next set
            chunk_end += CHUNK;
            if (el) commit<CG>(acc_full(buf), 0u);
            __syncwarp();
            if (++buf == n_acc) { buf = 0; pe ^= 1u; }
            if (!wait_warp(acc_empty(buf), pe, abort_flag, p.wait_ns)) { alive = false; break; }
            d0 = utmem + (uint32_t)(buf * 2 * p.BN);
            d1 = d0 + (uint32_t)p.BN;
            acc = 0u;
          }
          const int ks = cb + 1 == p.ncb ? p.ks_last : KB / 16;
          for (int pl = 0; pl < p.planes && alive; ++pl) {
            const int py = pl >> 1, px = pl & 1, nr = axis_taps(p.stride, py), nc = axis_taps(p.stride, px);
            if (!wait_warp(full_a(sa), pa, abort_flag, p.wait_ns)) { alive = false; break; }
            uint32_t a_row = ring_lo + (uint32_t)sa * a_step + row8 +
                             (uint32_t)axis_shift(p.stride, py, 0) * row8 + (uint32_t)axis_shift(p.stride, px, 0) * 8u;
            for (int tr = 0; tr < nr && alive; ++tr, a_row += row8) {
              uint32_t a_tap = a_row;
              for (int tc = 0; tc < nc; ++tc, a_tap += 8u) {
                uint32_t b_tap = ringb_lo + (uint32_t)sb * b_step;
                if (p.resident) {
                  if (res_wait) {
                    if (!__all_sync(0xFFFFFFFFu, b_seen) && !wait_warp(full_b(sb), 0u, abort_flag, p.wait_ns)) { alive = false; break; }
                    if (sb < MAX_B - 1) ++sb;
                    b_seen = mbar_test(full_b(sb), 0u);
                  }
                  b_tap = b_res;
                  b_res += (uint32_t)rows_b * 8u;
                } else if (!__all_sync(0xFFFFFFFFu, b_seen) && !wait_warp(full_b(sb), pb, abort_flag, p.wait_ns)) { alive = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int this_b = sb;
                if (!p.resident) {
                  if (++sb == p.b_slots) { sb = 0; pb ^= 1u; }
                  b_seen = mbar_test(full_b(sb), pb);
                }
                if (el) {
                  mma<CG, 128>(d0, a_tap, b_tap, idesc, acc);
                  mma<CG, 128>(d1, a_tap + SUB * 8u, b_tap, idesc, acc);
                  // (a loop over the steps takes 400 clocks a tap whatever it issues)
#pragma unroll
                  for (int k = 1; k < KB / 16; ++k)
                    if (k < ks) {
                      mma<CG, 128>(d0, a_tap + 2u * k, b_tap + 2u * k, idesc, 1u);
                      mma<CG, 128>(d1, a_tap + SUB * 8u + 2u * k, b_tap + 2u * k, idesc, 1u);
                    }
                  if (!p.resident) commit<CG>(empty_b(this_b), 0u);
                }
                __syncwarp();
                acc = 1u;
              }
            }
            if (!alive) break;
            if (el) commit<CG>(empty_a(sa), 0u);
            __syncwarp();
            if (++sa == p.a_slots) { sa = 0; pa ^= 1u; }
          }
        }
        if (!alive) break;
        res_wait = false;
        if (el) commit<CG>(acc_full(buf), 0u);
        __syncwarp();
        if (++buf == n_acc) { buf = 0; pe ^= 1u; }
      }
      if (!alive && el) {                    // multiply-adds already issued still read shared memory
        if (CG == 2) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain) : "memory");
        else commit<1>(drain, 0u);
        let_land(drain, 0u);
      }
    }
  } else if (warp < EPI_WARPS) {
    // =========================================================================== results
    constexpr int CCOLS = 64;                          // columns per pass: 128 bytes of results per position
    int buf = 0;
    uint32_t pf = 0u;
    const uint32_t st = sbase + OFF_ST;
    const int px = warp * 32 + lane;                   // position inside the tile
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    Note note;
    const float floor_at = p.act != 0 ? 0.0f : -INFINITY;       // the rectifier
    if (ROWS8) alive = __all_sync(0xFFFFFFFFu, !no_dense_form(p)) != 0;
    for (int item = unit; item < p.items && alive; item += n_units) {
      const int tg = p.d_groups.div(item), g = item - tg * p.groups;
      const int m0 = (CG == 2 ? 2 * tg + (int)rank : tg) * p.mstep;
      int yy, xx, nn;
      const int pixel = pixel_of(p, m0 + px, yy, xx, nn);
      // the chunks but the last
      const uint32_t scol = lane_base + (uint32_t)(n_acc * 2 * p.BN + (warp >> 2) * p.BN);
      bool summed = false;
      for (int cb = cb0 + CHUNK; LONG && cb < cb1; cb += CHUNK) {
        alive = __all_sync(0xFFFFFFFFu, mbar_wait<20>(acc_full(buf), pf, abort_flag, p.wait_ns)) != 0;
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t tcol = lane_base + (uint32_t)(buf * 2 * p.BN + (warp >> 2) * p.BN);
        for (int c = 0; c < p.BN; c += 16) {
          uint32_t v[16];
          tmem_load16(tcol + (uint32_t)c, v);
          tile::tmem_wait_ld();
          if (summed) tmem_add16(scol + (uint32_t)c, v);
          tmem_store16(scol + (uint32_t)c, v);
        }
        tile::tmem_wait_st();
        summed = true;
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          if (CG == 2) arrive_remote_read(map_to_rank(acc_empty(buf), 0));
          else mbar_arrive(acc_empty(buf));
        }
        if (++buf == n_acc) { buf = 0; pf ^= 1u; }
      }
      alive = alive && mbar_wait<20>(acc_full(buf), pf, abort_flag, p.wait_ns);
      if (p.act == 2 || p.parts > 1) alive = all_epilogue_warps(alive);       // they meet at barriers below: all go on or none
      if (!__all_sync(0xFFFFFFFFu, alive)) { alive = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tcol = lane_base + (uint32_t)(buf * 2 * p.BN + (warp >> 2) * p.BN);
      if (CG == 1 && p.parts > 1) {
        // partial sums to the CTAs that add them up, the next one's first so that not all send to the same
        const bool sent = px < p.mstep && pixel >= 0;
        cluster_wait();
        met = true;
        alive = __all_sync(0xFFFFFFFFu, open_exchange<false, 1>(p, received, go, rank, warp, lane, sent, abort_flag)) != 0;
        if (alive) {
          int c = first_column<false>(p, ((int)rank + 1) & (p.parts - 1)) & ~15;
          for (int n = p.BN; n > 0; n -= 16) {
            uint32_t v[16];
            tmem_load16(tcol + (uint32_t)c, v);
            tile::tmem_wait_ld();
            if (LONG && summed) tmem_add16(scol + (uint32_t)c, v);
            float f[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(v[i]);
            send_part<false, TILE, 1>(p, sbase, received, rank, c, px, sent, f);
            c += 16;
            if (c == p.BN) c = 0;
          }
        }
        alive = close_exchange(p, received, alive, abort_flag);
        if (alive) add_parts<false, TILE, 1>(p, sbase, item, rank, note);
        break;
      }
      for (int c0 = 0; c0 < p.BN; c0 += CCOLS) {
        const int nc = min(CCOLS, p.BN - c0);
        uint32_t v[CCOLS / 16][16];
#pragma unroll
        for (int q = 0; q < CCOLS / 16; ++q)
          if (q * 16 < nc) tmem_load16(tcol + (uint32_t)(c0 + q * 16), v[q]);
        tile::tmem_wait_ld();
        if (c0 + CCOLS >= p.BN) {                      // the accumulators have been read
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (CG == 2) arrive_remote_read(map_to_rank(acc_empty(buf), 0));
            else mbar_arrive(acc_empty(buf));
          }
          if (CG == 2 && item + n_units >= p.items) { cluster_arrive(); left = true; }
        }
        const uint32_t row = st + (uint32_t)px * 128u, sw = (uint32_t)(px & 7);
#pragma unroll
        for (int q = 0; q < CCOLS / 16; ++q) {
          if (q * 16 >= nc) break;
          if (LONG && summed) tmem_add16(scol + (uint32_t)(c0 + q * 16), v[q]);
          float f[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) f[i] = max_nan(__uint_as_float(v[q][i]), floor_at);
          if (p.act != 2) store_piece<false>(p, g * p.BN + c0 + q * 16, px < p.mstep ? pixel : -1, f, note);
          else stage_results<false>(row, sw, q, f);
        }
        if (p.act == 2) pool_results<false, 1>(p, st, g, c0, nc, m0, warp, lane, note);
      }
      if (++buf == n_acc) { buf = 0; pf ^= 1u; }
    }
    if (note.taken()) s_note = 1;
  }
  // every warp comes here, also after a failed wait: tensor memory is given back, and no CTA of a pair leaves while the other
  // may still signal its barriers.  A CTA that has received all partial sums is sent nothing more.
  if (!met) cluster_wait();
  if (CG == 2 && !left) cluster_arrive();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (!alive && !s_refused) atomicExch(p.status, PAT_ERR_TIMEOUT);
  auto give_time = [] {                                // 20 us: more than a copy or a store in flight takes
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < 20000ull) {}
  };
  const bool failed = s_abort != 0 && !(ROWS8 && s_plain);  // (without the dense form nothing has been copied that could still arrive)
  if (failed) give_time();                             // copies that the other CTA of a pair did not arm
  if (CG == 2) {
    cluster_wait();
  } else if (s_abort != 0 && clustered) {
    cluster_arrive();
    cluster_wait();
  }
  if (failed && p.parts > 1) give_time();              // what the others had sent by then
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == W_MMA) free_columns<CG>(tmem);
  if ((s_note && s_abort == 0) || (ROWS8 && s_plain)) {
    const bool whole = CG == 2 || p.parts == 1;
    renew_results<false, CG>(p, unit, n_units, CG == 2 ? (int)rank : 0, whole ? 0 : first_column<false>(p, (int)rank),
                             whole ? p.BN : first_column<false>(p, (int)rank + 1), ROWS8 && s_plain != 0);
  }
}

// How the work is cut: pairs of CTAs over large problems; single CTAs, the channels cut among the CTAs of a cluster, over
// small ones.  The choice with the smallest estimated time.
struct Split { int cg, BN, groups, parts; };
// at_once[log2(cluster size)]: clusters that run at the same time.
Split choose_split(const Geometry& g, int F, int C, const int (&at_once)[4]) {
  const int ks = (C + 15) / 16, ncb = (C + KB - 1) / KB;
  Split best{2, 0, 0, 1};
  double best_t = 1e30;
  auto consider = [&](int cg, int groups, int parts) {
    const int unit = cg == 2 ? 32 : 16;
    const int BN = ((F + groups - 1) / groups + unit - 1) / unit * unit;
    const long long items = (long long)((g.tiles + cg - 1) / cg) * groups;
    const int size = cg * parts;
    const long long slots = at_once[size == 1 ? 0 : size == 2 ? 1 : size == 4 ? 2 : 3], rounds = (items + slots - 1) / slots;
    if (parts > 1 && rounds > 1) return;
    const double steps = 2.0 * 9.0 * ks;
    // clocks of a 16-channel step: the products, or fetching their operands from shared memory (measured: 128 x 64 and
    // 128 x 32 take 49 and 41, 256 x 64 by a pair 45)
    const double step = std::max(BN / 2.0, cg == 2 ? 36.0 + BN / 8.0 : 36.0 + BN / 4.0);
    const double fill = 3000.0, tail = (4 * BN > 512 || rounds == 1) ? 8.0 * BN : 0.0;
    // sums of several chunks: adding one up holds the tensor core up unless there is a second accumulator set
    const int chunks = (ncb / parts + CHUNK - 1) / CHUNK;
    const double adding = chunks > 1 && 6 * BN > 512 ? 16.0 * BN * (chunks - 1) : 0.0;
    const double t = fill + rounds * (steps * step / parts + tail + adding) + (parts > 1 ? 2500.0 + 4.0 * BN : 0.0);
    if (t < best_t) { best_t = t; best = Split{cg, BN, groups, parts}; }
  };
  const int most = ncb > CHUNK ? 128 : 256;
  for (int groups = (F + most - 1) / most; groups <= (F + 31) / 32; groups *= 2) consider(2, groups, 1);
  for (int groups = (F + 127) / 128; groups <= (F + 15) / 16; groups *= 2)
    for (int parts = 1; parts <= MAX_PARTS_MMA && parts <= ncb; parts *= 2) consider(1, groups, parts);
  return best;
}

}  // namespace
}  // namespace tmma

// True when the tensor-core kernel can run this layer.
bool conv_mma_f16_supported(int F, int C, int dtype, int N, int H, int W, int stride) {
  using namespace tmma;
  if (dtype != PAT_F16 || !mma_weights(F, C) || !encode_fn()) return false;
  Geometry p;
  return set_geometry(p, TILE, N, H, W, stride, 0) && set_geometry(p, TILE, N, H, W, stride, 2);
}

int conv_mma_f16(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, const void* x, void* y,
                 int N, int H, int W, int stride, int act, unsigned long long wait_ns, int test_skip, cudaStream_t st) {
  using namespace tmma;
  const BlobLayout L = blob_layout(F, C, K, n_keep, PAT_F16);
  const char* b = static_cast<const char*>(blob);
  static thread_local DeviceSlot slots[kMaxDevices];
  DeviceSlot* dv = device_slot(slots);
  if (!dv) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cannot query the current device");
  Params p;
  using KernelFn = void (*)(const Maps, const Params);
  static const KernelFn kernels[8] = {k_conv_mma_f16<1, false, false>, k_conv_mma_f16<2, false, false>, k_conv_mma_f16<1, true, false>, k_conv_mma_f16<2, true, false>,
                                      k_conv_mma_f16<1, false, true>, k_conv_mma_f16<2, false, true>, k_conv_mma_f16<1, true, true>, k_conv_mma_f16<2, true, true>};
  const bool rows8 = C % 8 != 0;
  static thread_local int at_once[kMaxDevices][4];
  const int di = (int)(dv - slots);
  if (!dv->ready) {
    for (KernelFn fn : kernels)
      if (int rc = check_cuda(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES), "set shared memory size")) return rc;
    for (int i = 0; i < 4; ++i) at_once[di][i] = clusters_at_once(kernels[i == 1], 1 << i, threads_of(false), SMEM_BYTES);
    dv->ready = true;
  }
  if (!set_geometry(p, TILE, N, H, W, stride, 0)) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: too many tiles");
  Split sp = choose_split(p, F, C, at_once[di]);           // the same for every `act`: the same sums
  if (act == 2 && !set_geometry(p, TILE, N, H, W, stride, 2)) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: too many tiles");
  p.act = act;
  p.y = y;
  p.wide = aligned(y, 32) && F * 2 % 32 == 0;
  set_packed(p, x, blob, L, F, C, K);
  p.status = status_word();
  if (!p.status) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cannot resolve the status word");
  p.F = F; p.C = C; p.K = K; p.dtype = PAT_F16; p.n_keep = n_keep;
  p.BN = sp.BN; p.groups = sp.groups; p.parts = sp.parts;
  p.items = (p.tiles + sp.cg - 1) / sp.cg * p.groups;
  p.ncb = (C + KB - 1) / KB;
  p.ks_last = (C - (p.ncb - 1) * KB + 15) / 16;
  // rings: whole rows from the one that holds the tile's first position on, which starts up to P rows into the slot
  p.a_bytes = (uint32_t)((2 * p.P + p.ext + 1) * 128 + 1023) / 1024 * 1024;
  p.b_bytes = (uint32_t)(p.BN / sp.cg) * 128u;
  const long long all_b = 9ll * p.ncb * p.b_bytes;
  const int ring = set_exchange(p, kPer<false>, SMEM_BYTES, OFF_RING, RING_BYTES, (int)(2 * p.a_bytes + 4 * p.b_bytes));
  p.resident = p.groups == 1 && p.parts == 1 && all_b + 2ll * p.a_bytes <= ring;
  if (p.resident) {
    p.a_slots = std::min(MAX_A, (int)((ring - all_b) / p.a_bytes));
    p.b_slots = 1;
  } else {
    p.a_slots = std::max(2, std::min(MAX_A, (int)((ring - 4 * (int)p.b_bytes) / (int)p.a_bytes)));
    p.b_slots = std::min(MAX_B, (int)((ring - p.a_slots * (int)p.a_bytes) / (int)p.b_bytes));
  }
  p.idesc = (1u << 4) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)((sp.cg * SUB) >> 4) << 24);
  p.wait_ns = wait_ns; p.test_skip = test_skip;
  p.d_groups.set(p.groups);
  for (int j = 0; j < 256; ++j) p.masks[j] = (j < K) ? masks[j] : (uint16_t)0;

  Maps maps;
  const cuuint32_t one[4] = {1, 1, 1, 1};
  if (!rows8) {
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
    const cuuint64_t pitch[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
    const cuuint32_t step[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
    for (int rows : {1, ROWS}) {
      const cuuint32_t box[4] = {KB, (cuuint32_t)(stride * (p.P - 1) + 1), (cuuint32_t)(stride * (rows - 1) + 1), 1};
      const CUresult r = encode_fn()(rows == 1 ? &maps.a : &maps.rows, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(x), dims, pitch, box, step,
                                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cuTensorMapEncodeTiled failed (%d)", (int)r);
    }
  }
  {
    const cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)F, 9};
    const cuuint64_t pitch[2] = {(cuuint64_t)mma_pitch(C) * 2, (cuuint64_t)F * mma_pitch(C) * 2};
    const cuuint32_t box[3] = {KB, (cuuint32_t)(p.BN / sp.cg), 1};
    const CUresult r = encode_fn()(&maps.b, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<char*>(b) + L.dense, dims, pitch, box, one,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cuTensorMapEncodeTiled failed (%d)", (int)r);
  }

  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = sp.cg == 2 ? 2 : sp.parts; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 2;
  cfg.blockDim = dim3((unsigned)threads_of(rows8)); cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.gridDim = dim3((unsigned)(sp.parts > 1 ? p.items * sp.parts : sp.cg * std::min(p.items, at_once[di][sp.cg - 1])));
  if (int rc = check_cuda(cudaLaunchKernelEx(&cfg, kernels[sp.cg - 1 + (p.ncb > CHUNK ? 2 : 0) + (rows8 ? 4 : 0)], maps, p), "pat_conv3x3 launch")) return rc;
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pat_conv3x3 launch");
}

}  // namespace pat
