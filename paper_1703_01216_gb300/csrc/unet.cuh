// Internal interface of the U-Net post-corrector's kernels (unet_conv.cu, unet.cu).
#pragma once

#include <stdint.h>

namespace fr3d {

constexpr float kLeaky = 0.01f;   // slope of leaky ReLU for negative inputs

enum ConvMode { kConvFwd = 0, kConvDgradMask = 1, kConvDgradPlain = 2, kConvHead = 3 };

// One 3 x 3 x 3 convolution (or its input gradient) over CP tensors (see unet_conv.cu).  Tensors are
// byte pointers to [B][chunks][Vs][8] BF16; x_off / y_off / mask_off select a channel-chunk range of a
// larger tensor (the concatenations of the decoder).
struct ConvArgs {
  const unsigned char* x;
  int x_chunks, x_off, Cin;
  // [N / Ng groups][3 (e)][Cin / 16][3 (f)][3 (a = 2, 1, 0)][Ng / 8][2 chunks][8][8] BF16, K-major core matrices
  const unsigned char* wimg;
  int N, Ng;                   // output channels, and those of one CTA (conv_group)
  unsigned char* y;            // kConvHead: may be null (the output is not kept)
  int y_chunks, y_off;
  const float* bias;           // kConvFwd, kConvHead: [N] (may be null)
  const unsigned char* mask;   // kConvDgradMask: the tensor whose leaky derivative multiplies the result
  int mask_chunks, mask_off;
  // kConvHead (N = Ng = 16): the network's 1 x 1 x 1 head on the 16 outputs of a voxel: ys = bf16(s x) + w h + b
  // (any of ys and out = ys / s may be null), x, ys and out [B][D][H][W]
  const float *hx, *hw;        // input, head weights and bias [17]
  float *hys, *hout;
  float hs;
  int mode;
  int B, D, H, W, Wp;
  long HW, Vs;                 // voxels of a padded (h, w) plane, and of a padded volume with its guard
  int q_first;                 // first interior position of a plane
  int ntiles;                  // 128-position tiles of a plane (conv_tiles)
  int* err;                    // FR3D_INFO_TIMEOUT on a bounded wait that gave up (may be null)
  int ngroups, nd, nchunks, stages, slog;   // set by conv3_launch (slog: log2 of the accumulator slots)
};

constexpr int kWgVox = 128;    // voxels (K) of a weight-gradient stage
constexpr int kWgChain = 4096; // voxels at most that one FP32 accumulator of the weight gradient adds up
constexpr int kWgCg = 16;      // input channels of a weight-gradient CTA

// Weight gradient: partial sums per unit (sample, span of in-plane positions, depth chunk) and pair of
// channel groups, then their ordered sum.
struct WgradArgs {
  const unsigned char* g;      // output gradient (pre-activation), Cout channels
  int g_chunks, g_off, Cout;
  const unsigned char* x;      // layer input, Cin channels
  int x_chunks, x_off, Cin;
  int B, D, Wp;
  long HW, Vs, zero_pos;       // zero_pos: first voxel of the planes' zero guard
  int q_first, q_last;         // interior positions of a plane (with the halo between them)
  float* partials;             // [units][pairs][3 Og][9 kWgCg], then the bias sums [units][Cout]
  int* err;
  int Og, n_og, n_cg, span, nspans, nd, nchunks, slots, gslots;   // wgrad_plan
  float* bias_partials;        // set by wgrad3_launch
};

int conv_tiles(int q_first, int q_last);
int conv_group(int Cin, int N, int D, int ntiles, int B);
int conv3_launch(const ConvArgs& a, cudaStream_t st);
int wgrad_plan(WgradArgs* a, int B);
size_t wgrad_partial_floats(const WgradArgs& a, int B);
// dW [Cout][ci][27] and db [Cout]; ci: the layer's unpadded input channels
int wgrad3_launch(const WgradArgs& a, int ci, float* dW, float* db, cudaStream_t st);

}  // namespace fr3d
