// Tiles of the multiply-add convolution over the packed kept taps: what conv_generic.cu and, for blobs without the dense form, the
// tensor-core kernels share.
#pragma once
#include "common.cuh"

namespace pat {
namespace plain {

constexpr int TH = 8, TW = 32, RF = 4, CB = kChanTile;      // a tile's output rows and columns, filters of a warp, channels of a stage

template <typename T> __device__ inline float to_f32(T v);
template <> __device__ inline float to_f32<float>(float v) { return v; }
template <> __device__ inline float to_f32<__half>(__half v) { return __half2float(v); }
template <typename T> __device__ inline T from_f32(float v);
template <> __device__ inline float from_f32<float>(float v) { return v; }
template <> __device__ inline __half from_f32<__half>(float v) { return __float2half_rn(v); }

template <int STRIDE> struct Geo {
  static constexpr int IH = (TH - 1) * STRIDE + 3;
  static constexpr int IW = (TW - 1) * STRIDE + 3;
  static constexpr int IWP = IW | 1;                 // odd row pitch
  static constexpr int PLANE = IH * IWP + ((IH * IWP) % 2 == 0 ? 1 : 0);   // odd plane pitch
};

}  // namespace plain
}  // namespace pat
