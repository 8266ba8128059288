// Weight gradients from halo tiles: the row kernel for single layers
// (nm_wgrad_rows.cu), and the bias gradient it shares with nm_wgrad_tile.cu.
#pragma once
#include "nm_internal.cuh"

namespace nm {

// db[co] = the sum of dY over all voxels, in a fixed order; bpart:
// kBiasBlocks x cout floats.  16, 32, 64 or 128 outputs.
constexpr int kBiasBlocks = 256;
void bias_grad(const nm_conv3d_desc& d, const void* dy, float* bpart, float* db, cudaStream_t s);

// Single-source layers whose input is 8 channels or whole chunks of 16, where
// the row kernel is the faster one.  dw (16-byte aligned) and db as of
// conv3d_wgrad; db may be null.  A dw that is not finite sets kWgradNonFinite
// in the status word: the kernel also multiplies X by dY's zeroed halo, which
// turns an infinity into NaN, so such a gradient is to be taken again with
// conv3d_wgrad.
constexpr uint32_t kWgradNonFinite = 1u << 30;
bool conv_wgrad_rows_ok(const nm_conv3d_desc& d);
size_t conv_wgrad_rows_workspace(const nm_conv3d_desc& d);
cudaError_t conv3d_wgrad_rows(const nm_conv3d_desc& d, const void* x, const void* dy, float* dw, float* db,
                              void* workspace, uint32_t* status, cudaStream_t s);

}  // namespace nm
