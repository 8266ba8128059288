// Weights in the operand layout of the shifted-window convolution
// (nm_conv_tile.cu), for a network that lays out all its layers' in one launch.
#pragma once
#include "nm_internal.cuh"

namespace nm {

// The weights of a convolution of cin inputs and cout outputs as an image of
// tile_image_elems BF16 values (out, 16-byte aligned), from w[cout][kpad(cin)]
// or, of a layer's input gradient (cin = the layer's outputs, cout = its
// inputs), from the layer's own weights with the taps reversed (flip).
struct TileImage {
  const uint16_t* w;
  uint16_t* out;
  int cin, cout, flip;
  int kpad;                                          // set by launch_tile_images
};
constexpr int kMaxImages = 32;                       // of one launch
long long tile_image_elems(int cin, int cout);
cudaError_t launch_tile_images(const TileImage* images, int count, cudaStream_t s);

// Whether conv3d_fwd would take the shifted-window kernel (the description's
// form, NM_CONV_GATHER); then the same convolution from an image.
bool conv_image_ok(const nm_conv3d_desc& d);
cudaError_t conv3d_fwd_image(const nm_conv3d_desc& d, const void* x, const void* image, const float* bias, void* y,
                             int relu, uint32_t* status, cudaStream_t s);
// With the denoiser's 1x1x1 head fused into the epilogue (16 outputs, ReLU):
// yh[v] = head_w[16] + xin[v][0] + sum_c head_w[c] act[v][c].
cudaError_t conv3d_fwd_image_head(const nm_conv3d_desc& d, const void* x, const void* image, const float* bias,
                                  const float* head_w, const void* xin, int cx, float* yh, uint32_t* status,
                                  cudaStream_t s);

}  // namespace nm
