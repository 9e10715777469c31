// Sparse 3x3 convolution on the tensor cores (sm_100a, tcgen05), fp32 storage: the implicit GEMM of conv_mma_f16.cu with
// every fp32 number taken as the sum of three bf16 numbers (8 + 8 + 8 significant bits: nothing of the operand is lost).
// Of the nine products of two such sums the six largest are formed; the three left out are below 2^-25 of the whole.
//
// Accuracy.  The products are exact in the tensor core's fp32 sums, but those sums drop what does not fit their last bit
// instead of rounding it, so long ones drift towards zero.  Therefore they are kept short: the main products (first
// parts) and the five small ones have accumulators of their own, and both are added up, rounded to nearest, in registers
// of the epilogue warps after every 32 channels (eighteen steps of main products).  Measured against 64-bit sums (norm):
// 4e-8 (64 channels) to 1e-7 (256 channels, nothing pruned), where fp32 multiply-adds were 7e-8 to 4e-7 off; adding up
// after every kernel row costs 35 % on 56x56x64 (the epilogue warps hold the tensor core up) and is no closer.
//
// Why this is faster.  Six times the 9 F C multiply-adds per position in place of the 4 n_keep useful ones, at 22 times
// the fp32 multiply-add rate, of which the multiply-add kernel (conv_f32_img.cu) reached 4 - 38 %: it needs a re-arranged
// copy of the activations, and cuts small problems badly.  28x28x256 -> 256, batch 32: 479 (keep 1) and 212 us (keep 1/8)
// -> 104 us = 1.7 PFLOP/s of bf16 products; the 3x3 layers of ResNet-50 at batch 32: 1.85 -> 0.74 ms.  With 64 filters or fewer
// shared memory bounds it (the operands of a 256 x 64 product take 44 clocks to read, the product 32), with stride 2 the
// splitting of the activations (four planes for nine taps).
//
// Any multiple of four channels: activations are read 16 bytes at a time (28x28x260 -> 256, batch 32, keep 1/4 654 us with the generic
// kernel, 113 here; 56x56x68 -> 200, batch 16 286 and 80).
//
// Positions, taps and shifts: mma_tile.cuh.  A tile is 128 positions.  CG = 2: a pair of CTAs shares a group of up to 128
// filters (half of the weights in each); CG = 1: one CTA per tile and group.  `parts`: the input channels are cut among
// that many CTAs or pairs of a cluster and added up through distributed shared memory in a fixed order.
//
// Roles: warps 0-7 add up and write the results (warps 4-7 the upper half of the columns); warps 8-15 read the NHWC
// activations, split them and write the three parts to shared memory (rows of 32 channels = 64 bytes, in the 64-byte swizzle
// that the tensor core expects), one stage ahead; warp 16 copies weights (TMA); warp 17 issues the multiply-adds (in
// the odd CTA of a pair it reports that CTA's stages to the even one).
#include "mma_tile.cuh"

namespace pat {
namespace tmma {
namespace {

constexpr int TILE = 128, KB = 32, TERMS = kMmaTermsF32, PRODUCTS = 6;
constexpr int LOAD_WARPS = 8, W_LOAD = EPI_WARPS, W_B = W_LOAD + LOAD_WARPS, W_MMA = W_B + 1, NTHREADS = (W_MMA + 1) * 32;
constexpr int MAX_A = 4, MAX_B = 8;         // ring slots
constexpr int A_ROWS = 256;                // most rows of a stage
constexpr int UNITS = A_ROWS * 4 / (LOAD_WARPS * 32);      // (position, 8 channels) pieces per loading thread
static_assert(TILE + 2 * MAX_P + 2 <= A_ROWS, "a tile's rows fit a stage");
constexpr int ST_BYTES = 256 * 128;
constexpr int OFF_RING = 1024, RING_BYTES = 198656, OFF_ST = OFF_RING + RING_BYTES, SMEM_BYTES = OFF_ST + ST_BYTES;
static_assert(SMEM_BYTES <= 232448 && OFF_ST % 1024 == 0 && OFF_RING == RING_AT && SMEM_BYTES == RING_TO, "shared memory budget of one SM");
static_assert(SMEM_BYTES - OFF_RING >= (128 + MAX_PARTS_MMA * kPer<true>) * TILE * 4, "the partial sums of 128 filters fit");
constexpr int BUF_COLS = 256;              // tensor memory: two buffers of 128 columns of main and 128 of small products

struct alignas(64) Maps { CUtensorMap b; };
struct Params : Geometry {
  int a_rows, a_slots;       // activations: rows of a part of a stage, ring slots
  uint32_t a_bytes;          // bytes of a slot (three parts)
  int step_v, step_i;        // rows and columns from a position to the one A_ROWS / UNITS further on
};

__device__ __forceinline__ void load_b(int cg, uint32_t dst, const CUtensorMap* m, int c, int f, int t, uint32_t bar) {
  if (cg == 2)
    asm volatile("cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(f), "r"(t), "r"(0), "r"(bar & 0xFEFFFFFFu) : "memory");
  else
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(m), "r"(c), "r"(f), "r"(t), "r"(0), "r"(bar) : "memory");
}

// The bf16 numbers next to two values, lo in the lower half.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}
// The same, but a finite value that would round to infinity is cut off instead.
__device__ __forceinline__ uint32_t pack_bf16_finite(float lo, float hi) {
  auto part = [](float v) {
    const uint32_t b = __float_as_uint(v), r = b + 0x8000u;
    return ((r & 0x7FFFFFFFu) >= 0x7F800000u ? b : r) >> 16;
  };
  return part(lo) | (part(hi) << 16);
}

// FOURS: the channels are an odd multiple of four.  (A variant of its own: the check alone took 0.3 us of a 10.5 us launch.)
template <int CG, bool FOURS>
__global__ void __launch_bounds__(NTHREADS, 1) k_conv_mma_f32(const __grid_constant__ Maps maps, const __grid_constant__ Params p) {
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
  const uint32_t rank = cluster_rank(), side = rank % CG, pair = rank - side, part = rank / CG;
  const bool leader = side == 0;

  const int unit = (int)blockIdx.x / (CG * p.parts), n_units = (int)gridDim.x / (CG * p.parts);
  // Loading warps: four lanes take a position's 32 channels, eight each.
  const int tid = (int)threadIdx.x - W_LOAD * 32, chunk = tid & 3, t0 = tid >> 2;
  const int rows = SUB + (p.stride == 2 ? p.P + 1 : 2 * p.P + 2);      // positions the taps reach
  int base[UNITS] = {};                    // pixel index of the position in plane 0
  uint32_t valid = 0u;                     // bit 4 j + plane: inside the image
  auto locate = [&](int item) {
    const int m0 = (CG * p.d_groups.div(item) + (int)side) * p.mstep;
    valid = 0u;
    // the first piece's position by divisions, the others by steps of 64 positions from it
    const int q = m0 + t0, v1 = p.d_P.div(q), vi = v1 == 0 ? 0 : p.d_HP.div(v1 - 1);
    int i = q - v1 * p.P, yr = v1 - 1 - vi * p.HP, n = p.d_strips.div(vi), strip = vi - n * p.strips;
#pragma unroll
    for (int j = 0; j < UNITS; ++j) {
      const int y = yr * p.stride, x = (strip * p.Ws + i - 1) * p.stride;
      base[j] = (n * p.H + y) * p.W + x;
      if (t0 + j * (A_ROWS / UNITS) < rows && n < p.N && yr >= 0) {
        const uint32_t in_y = (y < p.H ? 3u : 0u) | (y + 1 < p.H ? 12u : 0u), x1 = x + 1;
        valid |= (in_y & ((x >= 0 && x < p.W ? 5u : 0u) | ((int)x1 >= 0 && (int)x1 < p.W ? 10u : 0u))) << (4 * j);
      }
      i += p.step_i;
      yr += p.step_v;
      if (i >= p.P) { i -= p.P; ++yr; }
      while (yr >= p.HP) {
        yr -= p.HP;
        if (++strip == p.strips) { strip = 0; ++n; }
      }
    }
  };
  if (warp >= W_LOAD && warp < W_LOAD + LOAD_WARPS) locate(unit);      // while the kernel before this one still runs

  if (threadIdx.x == 0) {
    s_abort = 0;
    s_refused = 0;
    s_note = 0;
    if (FOURS) s_plain = 0;
  }
  if (threadIdx.x == W_B * 32) prefetch_map(&maps.b);
  if (threadIdx.x < BARS) {                // a barrier each: 30 of them in a row by one thread showed in the launch
    const int t = (int)threadIdx.x, acc = t - (2 * MAX_A + 2 * MAX_B + 2);
    const int count = t < MAX_A ? LOAD_WARPS + (CG == 2 && leader ? 1 : 0) : acc == 0 || acc == 1 ? CG * EPI_WARPS : t == BARS - 3 ? EPI_WARPS / 2 : t == BARS - 2 ? p.parts : 1;
    mbar_init(sbase + 8u * (uint32_t)t, (uint32_t)count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == W_MMA) alloc_columns<CG>(smem_u32(&s_tmem));
  // The other CTAs' barriers exist: a pair waits for that before its first copy, the parts of a layer before they send sums.
  // Blocks take a whole SM each, so most of a launch's blocks start when the kernel before it ends: what they do until
  // here is not hidden.
  const bool clustered = CG == 2 || p.parts > 1;
  if (clustered) cluster_arrive();
  bool met = !clustered, left = false;     // has waited for the first, has arrived at the last barrier of the cluster
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (CG == 2) { cluster_wait(); met = true; }
  volatile int* abort_flag = &s_abort;
  const uint32_t tmem = s_tmem;
  const uint32_t ring_b = sbase + OFF_RING + (uint32_t)p.a_slots * p.a_bytes;

  const int cb0 = (int)part * p.ncb / p.parts, cb1 = ((int)part + 1) * p.ncb / p.parts;
  const int rows_b = p.BN / CG;
  bool alive = true;
  // After a failed wait the copies that a thread has armed still write this block's shared memory: (bounded) time to land.
  auto let_land = [&](uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = global_ns();
    for (uint32_t spin = 0; spin < kSpinLimit && !mbar_try_wait(bar, parity) && global_ns() - t0 <= p.wait_ns; ++spin) {}
  };

  if (warp >= W_LOAD && warp < W_LOAD + LOAD_WARPS) {
    // =========================================================================== activations
    // the values of the next stage are in registers before its buffer is free
    int slot = 0;
    uint32_t par = 1u;
    for (int item = unit; item < p.items && alive; item += n_units) {
      if (item != unit) locate(item);
      for (int cb = cb0; cb < cb1 && alive; ++cb)
        for (int pl = 0; pl < p.planes; ++pl) {
          const int c = cb * KB + chunk * 8, shift = (pl >> 1) * p.W + (pl & 1);
          float4 v[UNITS][2];
#pragma unroll
          for (int j = 0; j < UNITS; ++j) {
            v[j][0] = make_float4(0.f, 0.f, 0.f, 0.f);
            v[j][1] = v[j][0];
            if (((valid >> (4 * j + pl)) & 1u) && c < p.C) {
              // not through the read-only path: the kernel that writes x may still run when this block starts
              const float4* src = reinterpret_cast<const float4*>(static_cast<const float*>(p.x) + (size_t)(base[j] + shift) * p.C + c);
              v[j][0] = src[0];
              if (!FOURS || c + 4 < p.C) v[j][1] = src[1];
            }
          }
          if ((FOURS && pl == 0 && cb == cb0 && no_dense_form(p)) || !mbar_wait<20>(empty_a(slot), par, abort_flag, p.wait_ns)) alive = false;
          if (!__all_sync(0xFFFFFFFFu, alive)) { alive = false; break; }
          const uint32_t st = sbase + OFF_RING + (uint32_t)slot * p.a_bytes;
#pragma unroll
          for (int j = 0; j < UNITS; ++j) {
            if (j * (A_ROWS / UNITS) >= rows) break;
            const int t = t0 + j * (A_ROWS / UNITS);
            if (t >= p.a_rows) break;
            const uint32_t dst = st + (uint32_t)t * 64u + (uint32_t)((chunk ^ ((t >> 1) & 3)) << 4);
            float r[8] = {v[j][0].x, v[j][0].y, v[j][0].z, v[j][0].w, v[j][1].x, v[j][1].y, v[j][1].z, v[j][1].w};
#pragma unroll
            for (int term = 0; term < TERMS; ++term) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) w[e] = pack_bf16(r[2 * e], r[2 * e + 1]);
              if (term == 0) {
                // an exponent of all ones: infinite, not a number, or rounded up past the largest bf16 number
                const uint32_t m = 0x7F807F80u, one = 0x00800080u;
                if ((((w[0] & m) + one) | ((w[1] & m) + one) | ((w[2] & m) + one) | ((w[3] & m) + one)) & 0x80008000u)
#pragma unroll
                  for (int e = 0; e < 4; ++e) w[e] = pack_bf16_finite(r[2 * e], r[2 * e + 1]);
              }
              if (term + 1 < TERMS)
#pragma unroll
                for (int e = 0; e < 4; ++e) {              // exact
                  r[2 * e] -= __uint_as_float(w[e] << 16);
                  r[2 * e + 1] -= __uint_as_float(w[e] & 0xFFFF0000u);
                }
              tile::sts128(dst + (uint32_t)(term * p.a_rows) * 64u, w[0], w[1], w[2], w[3]);
            }
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");     // before the tensor core reads them
          __syncwarp();
          if (lane == 0) mbar_arrive(full_a(slot));
          if (++slot == p.a_slots) { slot = 0; par ^= 1u; }
        }
    }
  } else if (warp == W_B) {
    // =========================================================================== weights
    // nothing of the blob but its header is read before the header has been checked (the same answer in every CTA)
    if (!blob_matches_warp(p)) {
      alive = false;
      if (lane == 0) { s_refused = 1; s_abort = 1; atomicExch(p.status, PAT_ERR_BLOB); }
    } else if (FOURS && no_dense_form(p)) {
      alive = false;
      if (lane == 0) { s_refused = 1; s_plain = 1; s_abort = 1; }
    } else if (elect_one()) {
      int slot = 0, stage_no = 0;
      uint32_t par = 1u, armed = 0u, armed_par = 0u;
      for (int item = unit; item < p.items && alive; item += n_units) {
        const int g = item - p.d_groups.div(item) * p.groups;
        const int f0 = g * p.BN + (int)side * rows_b;
        for (int cb = cb0; cb < cb1 && alive; ++cb)
          for (int pl = 0; pl < p.planes && alive; ++pl) {
            const int py = pl >> 1, px = pl & 1, nr = axis_taps(p.stride, py), nc = axis_taps(p.stride, px);
            for (int tr = 0; tr < nr && alive; ++tr)
              for (int tc = 0; tc < nc; ++tc, ++stage_no) {
                const int tap = 3 * axis_tap(p.stride, py, tr) + axis_tap(p.stride, px, tc);
                if (!mbar_wait<20>(empty_b(slot), par, abort_flag, p.wait_ns)) { alive = false; break; }
                if (leader) mbar_arrive_expect_tx(full_b(slot), CG * p.b_bytes);
                if (stage_no != p.test_skip) load_b(CG, ring_b + (uint32_t)slot * p.b_bytes, &maps.b, cb * KB, f0, tap, full_b(slot));
                armed |= 1u << slot;
                armed_par = (armed_par & ~(1u << slot)) | ((par ^ 1u) << slot);
                if (++slot == p.b_slots) { slot = 0; par ^= 1u; }
              }
          }
      }
      if (!alive && leader)
        for (int s = 0; s < p.b_slots; ++s)
          if ((armed >> s) & 1u) let_land(full_b(s), (armed_par >> s) & 1u);
    }
  } else if (warp == W_MMA) {
    // =========================================================================== multiply-adds (even CTA of a pair)
    // warp-uniform values and control flow, one elected lane issues (see conv_mma_f16.cu)
    if (FOURS) alive = __all_sync(0xFFFFFFFFu, !no_dense_form(p)) != 0;
    if (leader) {
      const bool el = elect_one();
      int sa = 0, sb = 0, buf = 0;
      uint32_t pa = 0u, pb = 0u, pe = 1u;
      // The weights of the next tap and the next accumulators are looked at before this tap's products are issued: a wait
      // between two taps, even one that ends at once, lets the tensor core's queue run empty (49 -> 70 clocks a product of
      // 128 x 64 when there is one after every eight).
      bool b_seen = false;
      const uint32_t idesc = p.idesc, row4 = (uint32_t)p.P * 4u;      // descriptors count 16-byte units
      const uint32_t utmem = __reduce_or_sync(0xFFFFFFFFu, tmem), a_lo = operand_lo(sbase + OFF_RING), b_lo = operand_lo(ring_b);
      const uint32_t b_step = p.b_bytes >> 4, b_term = b_step / TERMS, T = (uint32_t)p.a_rows * 4u;
      for (int item = unit; item < p.items && alive; item += n_units)
        for (int cb = cb0; cb < cb1 && alive; ++cb) {
          const int ks = cb + 1 == p.ncb ? p.ks_last : KB / 16;
          if (!wait_warp(acc_empty(buf), pe, abort_flag, p.wait_ns)) { alive = false; break; }
          const uint32_t dm = utmem + (uint32_t)(buf * BUF_COLS), ds = dm + BUF_COLS / 2;
          uint32_t acc = 0u;
          for (int pl = 0; pl < p.planes && alive; ++pl) {
            const int py = pl >> 1, px = pl & 1, nr = axis_taps(p.stride, py), nc = axis_taps(p.stride, px);
            if (!wait_warp(full_a(sa), pa, abort_flag, p.wait_ns)) { alive = false; break; }
            uint32_t a_row = a_lo + (uint32_t)sa * (p.a_bytes >> 4) +
                             (uint32_t)axis_shift(p.stride, py, 0) * row4 + (uint32_t)axis_shift(p.stride, px, 0) * 4u;
            for (int tr = 0; tr < nr && alive; ++tr, a_row += row4) {
              uint32_t a_tap = a_row;
              for (int tc = 0; tc < nc; ++tc, a_tap += 4u) {
                if (!__all_sync(0xFFFFFFFFu, b_seen) && !wait_warp(full_b(sb), pb, abort_flag, p.wait_ns)) { alive = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t b_tap = b_lo + (uint32_t)sb * b_step;
                const int this_b = sb;
                if (++sb == p.b_slots) { sb = 0; pb ^= 1u; }
                b_seen = mbar_test(full_b(sb), pb);
                if (el) {
                  
                  mma<CG, 64>(ds, a_tap + 2u * T, b_tap, idesc, acc);
                  mma<CG, 64>(ds, a_tap + T, b_tap + b_term, idesc, 1u);
                  mma<CG, 64>(ds, a_tap, b_tap + 2u * b_term, idesc, 1u);
                  mma<CG, 64>(ds, a_tap + T, b_tap, idesc, 1u);
                  mma<CG, 64>(ds, a_tap, b_tap + b_term, idesc, 1u);
                  mma<CG, 64>(dm, a_tap, b_tap, idesc, acc);
                  if (ks == KB / 16) {
                    mma<CG, 64>(ds, a_tap + 2u * T + 2u, b_tap + 2u, idesc, 1u);
                    mma<CG, 64>(ds, a_tap + T + 2u, b_tap + b_term + 2u, idesc, 1u);
                    mma<CG, 64>(ds, a_tap + 2u, b_tap + 2u * b_term + 2u, idesc, 1u);
                    mma<CG, 64>(ds, a_tap + T + 2u, b_tap + 2u, idesc, 1u);
                    mma<CG, 64>(ds, a_tap + 2u, b_tap + b_term + 2u, idesc, 1u);
                    mma<CG, 64>(dm, a_tap + 2u, b_tap + 2u, idesc, 1u);
                  }
                  commit<CG>(empty_b(this_b), pair);
                }
                __syncwarp();
                acc = 1u;
              }
            }
            if (!alive) break;
            if (el) commit<CG>(empty_a(sa), pair);
            __syncwarp();
            if (++sa == p.a_slots) { sa = 0; pa ^= 1u; }
          }
          if (!alive) break;
          if (el) commit<CG>(acc_full(buf), pair);
          __syncwarp();
          if (++buf == 2) { buf = 0; pe ^= 1u; }
        }
      if (!alive && el) {                    // multiply-adds already issued still read shared memory
        if (CG == 2) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain) : "memory");
        else commit<1>(drain, 0u);
        let_land(drain, 0u);
      }
    } else if (CG == 2) {
      // The odd CTA's stages are reported to the even one by this warp, once each: an arrival on another CTA's barrier that
      // passes on what was written before it waits for all of the thread's own accesses, which held the loading warps up (eight
      // such arrivals a stage: 56x56x128 -> 128, stride 2, batch 32 61 us, 41 like this).
      int sa = 0;
      uint32_t pa = 0u;
      for (int item = unit; item < p.items && alive; item += n_units)
        for (int stage = (cb1 - cb0) * p.planes; stage > 0; --stage) {
          if (!wait_warp(full_a(sa), pa, abort_flag, p.wait_ns)) { alive = false; break; }
          if (lane == 0) arrive_remote(map_to_rank(full_a(sa), pair));
          __syncwarp();
          if (++sa == p.a_slots) { sa = 0; pa ^= 1u; }
        }
    }
  } else if (warp < EPI_WARPS) {
    // =========================================================================== sums and results
    const int half = p.BN / 2, col0 = (warp >> 2) * half;      // this warp's columns
    const int px = (warp & 3) * 32 + lane;                     // position inside the tile
    const uint32_t st = sbase + OFF_ST;
    const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col0;
    Note note;
    const float floor_at = p.act != 0 ? 0.0f : -INFINITY;       // the rectifier
    const int n_chunks = FOURS && no_dense_form(p) ? 0 : cb1 - cb0;
    int buf = 0;
    uint32_t pf = 0u;
    for (int item = unit; item < p.items && alive; item += n_units) {
      if (FOURS && n_chunks == 0) break;
      const int tg = p.d_groups.div(item), g = item - tg * p.groups;
      const int m0 = (CG * tg + (int)side) * p.mstep;
      float acc[4][16];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[q][i] = 0.0f;
      for (int c = 0; c < n_chunks; ++c) {
        alive = mbar_wait<20>(acc_full(buf), pf, abort_flag, p.wait_ns);
        if (!__all_sync(0xFFFFFFFFu, alive)) { alive = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t tc = lane_base + (uint32_t)(buf * BUF_COLS);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q * 16 < half) {
            uint32_t v[16], w[16];
            tmem_load16(tc + (uint32_t)(BUF_COLS / 2 + q * 16), v);
            tmem_load16(tc + (uint32_t)(q * 16), w);
            tile::tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[q][i] = (acc[q][i] + __uint_as_float(v[i])) + __uint_as_float(w[i]);
          }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          if (CG == 2) arrive_remote_read(map_to_rank(acc_empty(buf), pair));
          else mbar_arrive(acc_empty(buf));
        }
        if (CG == 2 && c + 1 == n_chunks && item + n_units >= p.items) { cluster_arrive(); left = true; }
        if (++buf == 2) { buf = 0; pf ^= 1u; }
      }
      if (p.act == 2 || p.parts > 1) alive = all_epilogue_warps(alive);         // they meet at barriers below: all go on or none
      if (!alive) break;
      int yy, xx, nn;
      const int pixel = px < p.mstep ? pixel_of(p, m0 + px, yy, xx, nn) : -1;
      if (p.parts > 1) {                       // partial sums to the CTAs that add them up
        if (!met) { cluster_wait(); met = true; }
        alive = open_exchange<true, CG>(p, received, go, rank, warp, lane, pixel >= 0, abort_flag);
        alive = __all_sync(0xFFFFFFFFu, alive) != 0;
        if (alive)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q * 16 < half) send_part<true, TILE, CG>(p, sbase, received, rank, col0 + q * 16, px, pixel >= 0, acc[q]);
        alive = close_exchange(p, received, alive, abort_flag);
        if (alive) add_parts<true, TILE, CG>(p, sbase, item, rank, note);
        break;
      }
      if (p.act != 2) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q * 16 < half) {
            float f[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) f[i] = max_nan(acc[q][i], floor_at);
            store_piece<true>(p, g * p.BN + col0 + q * 16, pixel, f, note);
          }
        continue;
      }
      const uint32_t row = st + (uint32_t)(warp * 32 + lane) * 128u, sw = (uint32_t)(lane & 7);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (h * 32 < half) {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if ((2 * h + q) * 16 < half) {
              float f[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) f[i] = max_nan(acc[2 * h + q][i], floor_at);
              stage_results<true>(row, sw, q, f);
            }
          pool_results<true, 2>(p, st, g, col0 + h * 32, min(32, half - h * 32), m0, warp, lane, note);
        }
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
  const bool failed = s_abort != 0 && !(FOURS && s_plain);  // (without the dense form nothing has been copied that could still arrive)
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
  if ((s_note && s_abort == 0) || (FOURS && s_plain)) {
    const bool whole = p.parts == 1;
    renew_results<true, CG>(p, unit, n_units, (int)side, whole ? 0 : first_column<true>(p, (int)part),
                             whole ? p.BN : first_column<true>(p, (int)part + 1), FOURS && s_plain != 0);
  }
}

// How the work is cut (pairs or single CTAs, filters per group, channel pieces): the choice with the smallest estimated time.
struct Split { int cg, BN, groups, parts; };
// at_once[log2(cluster size)]: clusters that run at the same time.
double split_clocks(const Split& s, int tiles, int C, const int (&at_once)[4], long long* rounds_out = nullptr) {
  const int ks = (C + 15) / 16, size = s.cg * s.parts;
  const long long items = (long long)((tiles + s.cg - 1) / s.cg) * s.groups;
  const long long slots = at_once[size == 1 ? 0 : size == 2 ? 1 : size == 4 ? 2 : 3], rounds = (items + slots - 1) / slots;
  if (rounds_out) *rounds_out = rounds;
  const double steps = 9.0 * PRODUCTS * ((ks + s.parts - 1) / s.parts);
  // clocks of a 16-channel step: the products, or fetching their operands from shared memory (see conv_mma_f16.cu)
  const double step = std::max(s.BN / 2.0, s.cg == 2 ? 36.0 + s.BN / 8.0 : 33.0 + s.BN / 4.0);
  return 4000.0 + rounds * (steps * step + 4.0 * s.BN) + (s.parts > 1 ? 2000.0 + 8.0 * s.BN : 0.0);
}
Split choose_split(int tiles, int F, int C, const int (&at_once)[4]) {
  const int ncb = (C + KB - 1) / KB;
  Split best{2, 0, 0, 1};
  double best_t = 1e30;
  for (int cg = 1; cg <= 2; ++cg)
    for (int groups = (F + 127) / 128; groups <= (F + 31) / 32; groups *= 2)
      for (int parts = 1; parts * cg <= MAX_PARTS_MMA && parts <= ncb; parts *= 2) {
        const Split s{cg, ((F + groups - 1) / groups + 31) / 32 * 32, groups, parts};
        long long rounds;
        const double t = split_clocks(s, tiles, C, at_once, &rounds);
        if ((parts == 1 || rounds == 1) && t < best_t) { best_t = t; best = s; }
      }
  return best;
}

// The kernels' attributes are set and the clusters that fit at once counted, once per thread and device.
using KernelFn = void (*)(const Maps, const Params);
constexpr KernelFn kKernels[4] = {k_conv_mma_f32<1, false>, k_conv_mma_f32<2, false>, k_conv_mma_f32<1, true>, k_conv_mma_f32<2, true>};
struct Device { const int (*at_once)[4]; int rc; };
Device device() {
  static thread_local DeviceSlot slots[kMaxDevices];
  static thread_local int at_once[kMaxDevices][4];
  DeviceSlot* dv = device_slot(slots);
  if (!dv) return {nullptr, set_error(PAT_ERR_CUDA, "pat_conv3x3: cannot query the current device")};
  int (&a)[4] = at_once[dv - slots];
  if (!dv->ready) {
    for (KernelFn fn : kKernels)
      if (int rc = check_cuda(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES), "set shared memory size")) return {nullptr, rc};
    for (int i = 0; i < 4; ++i) a[i] = clusters_at_once(kKernels[i > 0], 1 << i, NTHREADS, SMEM_BYTES);
    dv->ready = true;
  }
  return {&a, PAT_OK};
}

}  // namespace
}  // namespace tmma

// True when the tensor-core kernel can run this layer.
bool conv_mma_f32_supported(int F, int C, int dtype, int N, int H, int W, int stride) {
  using namespace tmma;
  if (dtype != PAT_F32 || !mma_weights(F, C) || !encode_fn()) return false;
  Geometry p;
  return set_geometry(p, TILE, N, H, W, stride, 0) && set_geometry(p, TILE, N, H, W, stride, 2);
}

// Estimated clocks of a call (13 % above the sum of its parts, as measured from 28x28 to 224x224 at batch 8 and 32).
double conv_mma_f32_clocks(int F, int C, int N, int H, int W, int stride) {
  using namespace tmma;
  const Device d = device();
  Geometry p;
  if (d.rc || !set_geometry(p, TILE, N, H, W, stride, 0)) return 1e30;
  const Split sp = choose_split(p.tiles, F, C, *d.at_once);
  return 1.13 * split_clocks(sp, p.tiles, C, *d.at_once);
}

int conv_mma_f32(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, const void* x, void* y,
                 int N, int H, int W, int stride, int act, unsigned long long wait_ns, int test_skip, cudaStream_t st) {
  using namespace tmma;
  const BlobLayout L = blob_layout(F, C, K, n_keep, PAT_F32);
  const char* b = static_cast<const char*>(blob);
  const Device d = device();
  if (d.rc) return d.rc;
  Params p;
  if (!set_geometry(p, TILE, N, H, W, stride, 0)) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: too many tiles");
  Split sp = choose_split(p.tiles, F, C, *d.at_once);           // the same for every `act`: the same sums
  if (act == 2 && !set_geometry(p, TILE, N, H, W, stride, 2)) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: too many tiles");
  p.act = act;
  p.y = y;
  p.wide = aligned(y, 32) && F * 4 % 32 == 0;
  set_packed(p, x, blob, L, F, C, K);
  p.status = status_word();
  if (!p.status) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cannot resolve the status word");
  p.F = F; p.C = C; p.K = K; p.dtype = PAT_F32; p.n_keep = n_keep;
  p.BN = sp.BN; p.groups = sp.groups; p.parts = sp.parts;
  p.items = (p.tiles + sp.cg - 1) / sp.cg * p.groups;
  p.ncb = (C + KB - 1) / KB;
  p.ks_last = (C - (p.ncb - 1) * KB + 15) / 16;
  p.b_bytes = (uint32_t)(TERMS * (p.BN / sp.cg)) * 64u;
  // stages of activations as long as four taps of weights fit beside them (stride 2 has short stages: more of them)
  p.a_rows = (SUB + (stride == 2 ? p.P + 1 : 2 * p.P + 2) + 7) / 8 * 8;
  p.a_bytes = (uint32_t)(TERMS * p.a_rows) * 64u;
  p.a_bytes = (p.a_bytes + 1023) / 1024 * 1024;
  p.step_v = A_ROWS / UNITS / p.P;
  p.step_i = A_ROWS / UNITS % p.P;
  const int ring = set_exchange(p, kPer<true>, SMEM_BYTES, OFF_RING, RING_BYTES, (int)(2 * p.a_bytes + 3 * p.b_bytes));
  p.a_slots = std::max(2, std::min(MAX_A, (ring - 4 * (int)p.b_bytes) / (int)p.a_bytes));
  p.b_slots = std::min(MAX_B, (ring - p.a_slots * (int)p.a_bytes) / (int)p.b_bytes);
  p.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)((sp.cg * SUB) >> 4) << 24);   // bf16 x bf16
  p.wait_ns = wait_ns; p.test_skip = test_skip;
  p.d_groups.set(p.groups);
  for (int j = 0; j < 256; ++j) p.masks[j] = (j < K) ? masks[j] : (uint16_t)0;

  Maps maps;
  {
    const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)F, 9, TERMS};
    const cuuint64_t fpitch = (cuuint64_t)mma_pitch(C) * 2, pitch[3] = {fpitch, F * fpitch, 9 * F * fpitch};
    const cuuint32_t box[4] = {KB, (cuuint32_t)(p.BN / sp.cg), 1, TERMS}, one[4] = {1, 1, 1, 1};
    const CUresult r = encode_fn()(&maps.b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<char*>(b) + L.dense, dims, pitch, box, one,
                                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(PAT_ERR_CUDA, "pat_conv3x3: cuTensorMapEncodeTiled failed (%d)", (int)r);
  }

  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = sp.cg * sp.parts; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 2;
  cfg.blockDim = dim3(NTHREADS); cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.gridDim = dim3((unsigned)(sp.parts > 1 ? p.items * sp.cg * sp.parts : sp.cg * std::min(p.items, (*d.at_once)[sp.cg - 1])));
  if (int rc = check_cuda(cudaLaunchKernelEx(&cfg, kKernels[sp.cg - 1 + (C % 8 ? 2 : 0)], maps, p), "pat_conv3x3 launch")) return rc;
  count_launches(1);
  return check_cuda(cudaGetLastError(), "pat_conv3x3 launch");
}

}  // namespace pat
