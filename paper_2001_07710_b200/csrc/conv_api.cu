// pat_conv3x3: argument validation and choice of the kernel for a layer shape.
#include "common.cuh"

namespace pat {
int conv_generic(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, int dtype,
                 const void* x, void* y, int N, int H, int W, int stride, cudaStream_t st);
bool conv_mma_f16_supported(int F, int C, int dtype, int N, int H, int W, int stride);
int conv_mma_f16(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, const void* x, void* y,
                 int N, int H, int W, int stride, int act, unsigned long long wait_ns, int test_skip, cudaStream_t st);
bool conv_mma_f32_supported(int F, int C, int dtype, int N, int H, int W, int stride);
double conv_mma_f32_clocks(int F, int C, int N, int H, int W, int stride);
int conv_mma_f32(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, const void* x, void* y,
                 int N, int H, int W, int stride, int act, unsigned long long wait_ns, int test_skip, cudaStream_t st);
size_t conv_img_workspace(int F, int C, int dtype, int N, int H, int W, int stride);
double conv_f32_img_clocks(int F, int C, const uint16_t* masks, int K, int64_t n_keep, int N, int H, int W, int sms);
int conv_f32_img(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                 const void* x, void* y, int N, int H, int W, int relu, void* workspace, cudaStream_t st);
}

using namespace pat;

// test hooks of the bounded waits (see pat_debug_set)
static constexpr unsigned long long kDefaultWaitNs = 2000000000ull;   // 2 s: far beyond any healthy wait
static unsigned long long g_wait_ns = kDefaultWaitNs;
static int g_test_skip = -1;
extern "C" int pat_debug_set(int what, long long value) {
  if (what == 0) g_wait_ns = value > 0 ? (unsigned long long)value : kDefaultWaitNs;
  else if (what == 1) g_test_skip = value < 0 ? -1 : (int)value;
  else return set_error(PAT_ERR_INVALID_ARG, "pat_debug_set: unknown switch %d", what);
  return PAT_OK;
}

static int check_conv_args(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, int dtype,
                           const void* x, const void* y, int N, int H, int W, int stride) {
  if (!blob || !x || !y) return set_error(PAT_ERR_INVALID_ARG, "pat_conv3x3: null pointer");
  if (F < 1 || C < 1 || F > 65535 || C > 65535) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: F=%d C=%d outside 1..65535", F, C);
  if (int rc = check_library(masks, K)) return rc;
  if (dtype != PAT_F32 && dtype != PAT_F16) return set_error(PAT_ERR_DTYPE, "pat_conv3x3: dtype %d", dtype);
  if (n_keep < 0 || n_keep > (int64_t)F * C) return set_error(PAT_ERR_INVALID_ARG, "pat_conv3x3: n_keep outside 0..F*C");
  if (N < 1 || H < 1 || W < 1) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: N, H, W must be positive");
  if (stride != 1 && stride != 2) return set_error(PAT_ERR_INVALID_ARG, "pat_conv3x3: stride %d (1 or 2)", stride);
  if (!aligned(blob, 256)) return set_error(PAT_ERR_ALIGN, "pat_conv3x3: blob must be 256-byte aligned");
  if (!aligned(x, 16) || !aligned(y, 16)) return set_error(PAT_ERR_ALIGN, "pat_conv3x3: x and y must be 16-byte aligned");
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  if ((size_t)N * ((Ho + 7) / 8) * ((Wo + 31) / 32) > 0x7FFFFFFFull) return set_error(PAT_ERR_SHAPE, "pat_conv3x3: too many tiles");
  return PAT_OK;
}

// Odd multiples of four channels so few that a stage of the tensor-core kernels is mostly empty, with few filters: large images are
// faster in the generic kernel, which pays by the kept kernel.  In fp32 its rows of 8 - 40 bytes of weights, read by all SMs at once,
// lie in a few lines of L2 on top of that.  fp32, four patterns, generic and tensor cores, us:
//   8 x 256x256, 4 -> 8 keep 1 67, 175, 4 -> 32 keep 0.3 115, 167 (keep 1 133, 160), 4 -> 40 keep 0.1 149, 202 (keep 1 186, 168), 4 -> 64 205, 137
//   12 -> 8 keep 0.3 65, 78, 12 -> 16 keep 0.1 67, 97 (0.3 84, 79), 12 -> 24 keep 0.1 87, 79, 20 -> 8 keep 0.1 82, 110 (0.3 103, 103)
//   2 x 256x256, 4 -> 16 keep 0.3 29, 29, 4 -> 24 34, 33, 4 -> 32 43, 46; 8 x 112x112, 4 -> 8 20, 26, 4 -> 16 23, 23, 4 -> 40 36, 44, one image 4 -> 8 10, 9; stride 2, 24 x 224x224, 4 -> 8 keep 0.3 68, 81, 4 -> 16
//   keep 0.1 70, 78 (0.3 75, 74), 8 x 112x112 18, 13
// (a rectifier behind the generic kernel, a pass of its own, adds 2 - 20 us)
// fp16: 24 x 224x224, 12 -> 8 keep 0.02 100, 116, 0.3 no difference.
static bool few_channels(int F, int C, int64_t n_keep, int dtype, int N, int H, int W, int stride) {
  if (C % 8 == 0 || C > 20) return false;
  const long long positions = (long long)N * ((H - 1) / stride + 1) * ((W - 1) / stride + 1);
  const bool sparse = 8 * n_keep <= (int64_t)F * C;
  if (dtype == PAT_F16) return stride == 1 && C <= 12 && F == 8 && sparse && positions >= 500000;
  const bool large = positions >= 250000, third = 3 * n_keep <= (int64_t)F * C;
  if (stride == 2) return positions >= 130000 && C <= 12 && (F == 8 ? C == 4 || sparse : C == 4 && F <= 16 && sparse);
  if (C == 4) return F == 8 ? positions >= 20000 : (F <= 32 && large) || (F > 24 && F <= 40 && third && positions >= 90000);
  return positions >= 130000 && ((sparse && F <= (C == 12 ? 16 : 8)) || (C == 12 && F == 8 && large && third));
}

static bool on_tensor_cores(int F, int C, int64_t n_keep, int dtype, int N, int H, int W, int stride) {
  if (few_channels(F, C, n_keep, dtype, N, H, W, stride)) return false;
  return dtype == PAT_F16 ? conv_mma_f16_supported(F, C, dtype, N, H, W, stride) : conv_mma_f32_supported(F, C, dtype, N, H, W, stride);
}
static int conv_mma(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep, int dtype, const void* x, void* y,
                    int N, int H, int W, int stride, int act, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  return dtype == PAT_F16 ? conv_mma_f16(blob, F, C, masks, K, n_keep, x, y, N, H, W, stride, act, g_wait_ns, g_test_skip, st)
                          : conv_mma_f32(blob, F, C, masks, K, n_keep, x, y, N, H, W, stride, act, g_wait_ns, g_test_skip, st);
}

// Which kernels run an fp32 call with a workspace whose blob serves both: the ones with the smaller estimate.  Both sides
// measured: 56x56x256 -> 256, batch 32, keep 1/8, eight patterns: multiply-adds 313 us, tensor cores 347 (six products
// for 18 times the useful work); batch 1: 36 and 27 us (the multiply-add kernels' items do not fill the chip);
// 28x28x256, batch 32, twelve patterns: 213 and 104 us.  The estimates are those of the plain convolution whatever follows it,
// so that fused pooling has the sums of the two passes that it replaces (the two kernels' sums differ in their last bits).
static bool prefer_img(int F, int C, const uint16_t* masks, int K, int64_t n_keep, int dtype, int N, int H, int W, int stride) {
  if (stride != 1 || !img_blocks(F, C, n_keep, dtype)) return false;     // stride 2 has a quarter of the positions there
  static thread_local DeviceSlot slots[kMaxDevices];
  DeviceSlot* dv = device_slot(slots);
  return conv_f32_img_clocks(F, C, masks, K, n_keep, N, H, W, dv ? dv->sms : 148) < conv_mma_f32_clocks(F, C, N, H, W, stride);
}

extern "C" int pat_conv3x3(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                           int dtype, const void* x, void* y, int N, int H, int W, int stride, void* stream) {
  if (int rc = check_conv_args(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride)) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (on_tensor_cores(F, C, n_keep, dtype, N, H, W, stride)) return conv_mma(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride, 0, stream);
  return conv_generic(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride, st);
}

extern "C" size_t pat_conv3x3_workspace(int F, int C, int dtype, int N, int H, int W, int stride) {
  if (F < 1 || C < 1 || N < 1 || H < 1 || W < 1) return 0;
  return conv_img_workspace(F, C, dtype, N, H, W, stride);
}

extern "C" int pat_relu_maxpool(const void* x, int dtype, int N, int H, int W, int C, int pool, void* y, void* stream);

extern "C" int pat_conv3x3_ws_act(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                                  int dtype, const void* x, void* y, int N, int H, int W, int stride, int act,
                                  void* workspace, size_t workspace_bytes, void* stream) {
  if (act < 0 || act > 2) return set_error(PAT_ERR_INVALID_ARG, "pat_conv3x3_ws_act: act %d (0: none, 1: rectifier, 2: rectifier and 2 x 2 max pooling)", act);
  if (int rc = check_conv_args(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride)) return rc;
  const size_t need = pat_conv3x3_workspace(F, C, dtype, N, H, W, stride);
  // pooling happens inside a tile of the kernels: no other kernel writes a pooled image (y is too
  // small for the full-size result, so there is no two-pass substitute without memory of the library's own)
  if (act == 2 && (need == 0 || stride != 1 || (H & 1) || (W & 1)))
    return set_error(PAT_ERR_SHAPE, "pat_conv3x3_ws_act: act 2 needs a layer the workspace kernels cover, stride 1, even H and W "
                                    "(otherwise: act 1, then pat_relu_maxpool)");
  if (need > 0) {
    if (!workspace || workspace_bytes < need)
      return set_error(PAT_ERR_WORKSPACE, "pat_conv3x3_ws: workspace has %zu bytes, needs %zu", workspace_bytes, need);
    if (!aligned(workspace, 256)) return set_error(PAT_ERR_ALIGN, "pat_conv3x3_ws: workspace must be 256-byte aligned");
    if (prefer_img(F, C, masks, K, n_keep, dtype, N, H, W, stride))
      return conv_f32_img(blob, F, C, masks, K, n_keep, x, y, N, H, W, act, workspace, reinterpret_cast<cudaStream_t>(stream));
  }
  if (on_tensor_cores(F, C, n_keep, dtype, N, H, W, stride)) return conv_mma(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride, act, stream);
  if (act == 2) return set_error(PAT_ERR_SHAPE, "pat_conv3x3_ws_act: image too large");
  // the plain convolution, then the rectifier in place
  if (int rc = pat_conv3x3(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride, stream)) return rc;
  if (!act) return PAT_OK;
  return pat_relu_maxpool(y, dtype, N, (H - 1) / stride + 1, (W - 1) / stride + 1, F, 0, y, stream);
}

extern "C" int pat_conv3x3_ws(const void* blob, int F, int C, const uint16_t* masks, int K, int64_t n_keep,
                              int dtype, const void* x, void* y, int N, int H, int W, int stride,
                              void* workspace, size_t workspace_bytes, void* stream) {
  return pat_conv3x3_ws_act(blob, F, C, masks, K, n_keep, dtype, x, y, N, H, W, stride, 0, workspace, workspace_bytes, stream);
}
