// The learned post-corrector (fr3d_unet_*): a 4-level 3D U-Net of base width 16 that maps the Tikhonov
// reconstruction of Algorithm 1 to a corrected xi, trained and run on the GPU.  The paper has no network;
// the learned part of the benchmark suite asks for one to put back what the normal solution leaves out
// (with one observation plane, M' - 1 depth directions per frequency, Assumption U of Sec. 4).
//
// Network (the FP64 oracle restates it): level 0 conv(1 -> 16), conv(16 -> 16); levels 1, 2: average
// pooling by 2, conv(w_{l-1} -> w_l), conv(w_l -> w_l); level 3 (bottom): pooling, three conv to 128
// channels; going up, nearest upsampling by 2 concatenated with the encoder output of the level,
// conv(w_{l+1} + w_l -> w_l), conv(w_l -> w_l); every conv 3 x 3 x 3 with bias and leaky ReLU (slope 0.01);
// a 1 x 1 x 1 head 16 -> 1 added to the input.  Inputs are scaled by in_scale inside (x_s = in_scale x),
// the prediction is returned in the caller's units; the loss is the batch mean of ||y - t||^2 / ||t||^2.
//
// Storage: FP32 master parameters, gradients and Adam moments; BF16 weight images (forward and input
// gradient, see unet_conv.cu) rebuilt after every update; BF16 activations and activation gradients in
// the padded channel-chunked layout of unet_conv.cu (zero halos and guards, allocated once per network
// for its maximum batch).  Convolutions and their gradients run on the tensor cores (unet_conv.cu; the last
// convolution applies the head); pooling, upsampling, the head's gradient, loss, reductions and Adam are the CUDA-core
// kernels below.  Every reduction
// has a fixed order (block partials, then one ordered pass), so results do not depend on the run, nor on the largest batch
// a network was made for.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "ops.cuh"
#include "tc.cuh"
#include "unet.cuh"

namespace fr3d {

namespace {

constexpr int kL = 4;
constexpr int kWidth[kL] = {16, 32, 64, 128};
constexpr int kGuard = 128;
constexpr int kNumConv = 15;

struct Level {
  int D, H, W, Hp, Wp;
  long HW, Vp, Vs;
  int q_first, q_last;   // interior positions of an (h, w) plane (with the halo between its rows)
};

Level make_level(int D, int H, int W) {
  Level l;
  l.D = D;
  l.H = H;
  l.W = W;
  l.Hp = H + 2;
  l.Wp = W + 2;
  l.Vp = (long)(D + 2) * l.Hp * l.Wp;
  l.Vs = l.Vp + kGuard;
  l.HW = (long)l.Hp * l.Wp;
  l.q_first = l.Wp + 1;
  l.q_last = (int)l.HW - 2 - l.Wp;
  return l;
}

// tensor ids
enum {
  T_X = 0,
  T_E1 = 1,     // + l (0..2): encoder conv 1 output
  T_CAT = 4,    // + l (0..2): [upsampled w_{l+1} | encoder output w_l]
  T_P = 7,      // + l - 1 (l = 1..3): pooled input of level l
  T_B = 10,     // + 0..2: bottom conv outputs
  T_D1 = 13,    // + l: decoder conv 1 output
  T_D2 = 16,    // + l: decoder conv 2 output
  T_N = 19
};

struct TensorDesc {
  int C = 0, lvl = 0;
};

struct Layer {
  int ci = 0, ci_pad = 0, co = 0, lvl = 0;
  long woff = 0;                  // w [co][ci][27] at woff, b [co] at woff + co ci 27 (flat parameters)
  int in_t = 0, in_off = 0;       // input tensor and channel offset
  int out_t = 0, out_off = 0;
  int dgrad = 0;                  // 0 none, 1 with the leaky derivative of the input, 2 plain
  size_t img_f = 0, img_b = 0;    // byte offsets of the weight images
  int ng_f = 0, ng_b = 0;         // output channels per CTA of the convolution and of its input gradient
  WgradArgs wg{};                 // weight-gradient plan of Unet::wg_batch (the tensors are filled in per call)
};

}  // namespace

struct Unet {
  int dev = 0;
  int D = 0, H = 0, W = 0, Bmax = 0;
  float in_scale = 1.f;
  Level lv[kL];
  TensorDesc td[T_N];
  unsigned char* t[T_N] = {};     // activations
  unsigned char* g[T_N] = {};     // activation gradients
  size_t tbytes[T_N] = {};
  Layer layer[kNumConv];
  long n_params = 0;
  long head_off = 0;
  float* params = nullptr;        // FP32 master
  float* grads = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  int adam_t = 0;
  unsigned char* imgs = nullptr;  // BF16 weight images
  size_t img_bytes = 0;
  float* y = nullptr;             // scaled prediction [Bmax][D][H][W]
  float* partials = nullptr;      // weight-gradient partials
  size_t partial_floats = 0;      // for every batch up to Bmax
  int wg_batch = 0;               // the batch size that the layers' weight-gradient plans are for
  float* red = nullptr;           // small reduction buffers
  size_t red_floats = 0;
  double* lossbuf = nullptr;      // [Bmax][2] sums, [1] loss
  int* err = nullptr;
};

namespace {

__device__ __forceinline__ float bfv(uint32_t u, int hi) { return __uint_as_float(hi ? (u & 0xFFFF0000u) : (u << 16)); }
__device__ __forceinline__ uint32_t pk(float a, float b) {
  return (uint32_t)tc::bf16_rn(a) | ((uint32_t)tc::bf16_rn(b) << 16);
}
__device__ __forceinline__ void unpack8(const uint4& q, float* f) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    f[2 * k] = bfv(w[k], 0);
    f[2 * k + 1] = bfv(w[k], 1);
  }
}
__device__ __forceinline__ uint4 pack8(const float* f) {
  return make_uint4(pk(f[0], f[1]), pk(f[2], f[3]), pk(f[4], f[5]), pk(f[6], f[7]));
}
__device__ __forceinline__ float bf16r(float x) { return tc::bf16_val(tc::bf16_rn(x)); }

struct LevelArg {
  int D, H, W, Hp, Wp;
  long Vs;
};
LevelArg larg(const Level& l) { return LevelArg{l.D, l.H, l.W, l.Hp, l.Wp, l.Vs}; }

__device__ __forceinline__ long ppos(const LevelArg& L, int d, int h, int w) {
  return ((long)(d + 1) * L.Hp + (h + 1)) * L.Wp + (w + 1);
}

// Pooling, upsampling, their adjoints, the convolutions and the weight gradients are launched programmatically: their
// set-up (barriers, tensor memory) and their launch run while the kernel before them leaves the SMs (24 and 62 launches:
// 1024 -> 973 us forward and 3462 -> 3305 us gradient at 128^2 x 32, batch 8; 177 -> 117 and 600 -> 412 us at 24^2 x 8,
// batch 1).  Each waits for that kernel before its first access to global memory; the others are launched as usual.
// What that kernel writes is read with coherent loads (__ldca: neighbouring lanes share sectors, and the second half of a
// sector comes from L1): the read-only path asks for data that no one writes while the reader runs, and a reader
// launched programmatically runs before its predecessor has ended.  Tensors that were complete before the predecessor
// began (the forward activations in the backward pass) keep __ldg.
//
// The elementwise kernels below run one (chunk, depth, row) per blockDim.y lane group and consecutive w per
// thread, so that the index divisions are per row and in 32 bits (per voxel and in 64 bits they cost more than
// the memory traffic: the level-0 upsampling took 117 us for 310 MB).
struct Row {
  int b, j, d, h;
  bool ok;
};
__device__ __forceinline__ Row row_of(int B, int nc, int D, int H) {
  const unsigned r = blockIdx.x * blockDim.y + threadIdx.y;
  Row q;
  q.ok = r < (unsigned)(B * nc * D * H);
  q.h = (int)(r % H);
  unsigned t = r / H;
  q.d = (int)(t % D);
  t /= D;
  q.j = (int)(t % nc);
  q.b = (int)(t / nc);
  return q;
}
// lanes along w: the power of two covering the row, at most 128; 256 threads per block
dim3 row_block(int W) {
  int tx = 8;
  while (tx < W && tx < 128) tx <<= 1;
  return dim3(tx, 256 / tx);
}
int row_grid(int B, int nc, int D, int H, dim3 blk) { return (B * nc * D * H + blk.y - 1) / blk.y; }

__device__ __forceinline__ const uint4* vox(const unsigned char* t, int b, int chunks, int j, const LevelArg& L, long p) {
  return reinterpret_cast<const uint4*>(t + (((long)b * chunks + j) * L.Vs + p) * 16);
}
__device__ __forceinline__ uint4* vox(unsigned char* t, int b, int chunks, int j, const LevelArg& L, long p) {
  return reinterpret_cast<uint4*>(t + (((long)b * chunks + j) * L.Vs + p) * 16);
}

// x_s = in_scale x into channel 0 of the input tensor (16 channels, the other 15 stay zero)
__global__ void k_pack_input(const float* __restrict__ x, int B, LevelArg L, float s, unsigned char* __restrict__ X) {
  const Row q = row_of(B, 1, L.D, L.H);
  if (!q.ok) return;
  const float* src = x + (((long)q.b * L.D + q.d) * L.H + q.h) * L.W;
  uint4* dst = vox(X, q.b, 2, 0, L, ppos(L, q.d, q.h, 0));
  for (int w = threadIdx.x; w < L.W; w += blockDim.x) dst[w] = make_uint4(tc::bf16_rn(s * src[w]), 0, 0, 0);
}

// average pooling by 2: dst (level l+1, chunks [0, nc)) from src (level l, chunks [soff, soff + nc))
__global__ void k_pool(const unsigned char* __restrict__ src, int s_chunks, int soff, LevelArg Ls,
                       unsigned char* __restrict__ dst, int d_chunks, LevelArg Ld, int nc, int B) {
  pdl_wait();
  pdl_release();
  const Row q = row_of(B, nc, Ld.D, Ld.H);
  if (!q.ok) return;
  for (int w = threadIdx.x; w < Ld.W; w += blockDim.x) {
    uint4 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      v[c] = __ldca(vox(src, q.b, s_chunks, soff + q.j, Ls,
                       ppos(Ls, 2 * q.d + (c >> 2), 2 * q.h + ((c >> 1) & 1), 2 * w + (c & 1))));
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float f[8];
      unpack8(v[c], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] += f[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] *= 0.125f;
    *vox(dst, q.b, d_chunks, q.j, Ld, ppos(Ld, q.d, q.h, w)) = pack8(acc);
  }
}

// nearest upsampling by 2: dst (level l, chunks [0, nc)) from src (level l+1, chunks [0, nc)); lane w
// reads the parent of the row's voxel w and writes it to the four child rows, 512 contiguous bytes per warp
// (a parent per lane left 16 of every 32 bytes to a second store: 74 us to level 0 at 128^2 x 32, batch 8, now 51)
__global__ void k_up(const unsigned char* __restrict__ src, int s_chunks, LevelArg Ls, unsigned char* __restrict__ dst,
                     int d_chunks, LevelArg Ld, int nc, int B) {
  pdl_wait();
  pdl_release();
  const Row q = row_of(B, nc, Ls.D, Ls.H);
  if (!q.ok) return;
  for (int w = threadIdx.x; w < Ld.W; w += blockDim.x) {
    const uint4 v = __ldca(vox(src, q.b, s_chunks, q.j, Ls, ppos(Ls, q.d, q.h, w >> 1)));
#pragma unroll
    for (int c = 0; c < 4; ++c) *vox(dst, q.b, d_chunks, q.j, Ld, ppos(Ld, 2 * q.d + (c >> 1), 2 * q.h + (c & 1), w)) = v;
  }
}

// gradient of the upsampling, times the leaky derivative of the upsampled tensor (its only consumer):
// gs[parent] = bf16(leaky'(s[parent]) * bf16(sum over the 8 children of gd))
__global__ void k_up_backward(const unsigned char* __restrict__ gd, int d_chunks, LevelArg Ld,
                              const unsigned char* __restrict__ s, unsigned char* __restrict__ gs, int s_chunks,
                              LevelArg Ls, int nc, int B) {
  pdl_wait();
  pdl_release();
  const Row q = row_of(B, nc, Ls.D, Ls.H);
  if (!q.ok) return;
  for (int w = threadIdx.x; w < Ls.W; w += blockDim.x) {
    uint4 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      v[c] = __ldca(vox(gd, q.b, d_chunks, q.j, Ld,
                       ppos(Ld, 2 * q.d + (c >> 2), 2 * q.h + ((c >> 1) & 1), 2 * w + (c & 1))));
    const long o = ppos(Ls, q.d, q.h, w);
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0}, m[8];
    unpack8(__ldg(vox(s, q.b, s_chunks, q.j, Ls, o)), m);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float f[8];
      unpack8(v[c], f);
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] += f[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = bf16r(acc[k]) * (m[k] > 0.f ? 1.f : kLeaky);
    *vox(gs, q.b, s_chunks, q.j, Ls, o) = pack8(acc);
  }
}

// gradient of an encoder output (consumed by the pooling and the skip connection), in place in the skip
// gradient: g = bf16(leaky'(s) * (bf16(gp[parent] / 8) + g))
__global__ void k_pool_backward(const unsigned char* __restrict__ gp, int p_chunks, LevelArg Lp,
                                const unsigned char* __restrict__ s, unsigned char* __restrict__ g, int c_chunks,
                                int coff, LevelArg Lc, int nc, int B) {
  pdl_wait();
  pdl_release();
  const Row q = row_of(B, nc, Lc.D, Lc.H);
  if (!q.ok) return;
  for (int w = threadIdx.x; w < Lc.W; w += blockDim.x) {
    const long o = ppos(Lc, q.d, q.h, w);
    uint4* gq = vox(g, q.b, c_chunks, coff + q.j, Lc, o);
    float up[8], sk[8], m[8];
    unpack8(__ldca(vox(gp, q.b, p_chunks, q.j, Lp, ppos(Lp, q.d / 2, q.h / 2, w / 2))), up);
    unpack8(*gq, sk);
    unpack8(__ldg(vox(s, q.b, c_chunks, coff + q.j, Lc, o)), m);
#pragma unroll
    for (int k = 0; k < 8; ++k) sk[k] = (bf16r(up[k] * 0.125f) + sk[k]) * (m[k] > 0.f ? 1.f : kLeaky);
    *gq = pack8(sk);
  }
}

// per-block partial sums of (y_s - t_s)^2 and t_s^2 for each sample.  The predictions come from the last
// convolution, which applies the head to its outputs while it holds them
// (a pass of its own read the 134 MB back: 61 us at 128^2 x 32, batch 8; now 6 us of that convolution and 13 us here).
constexpr int kHeadThreads = 256;
__global__ void __launch_bounds__(kHeadThreads) k_loss_partial(const float* __restrict__ ys, const float* __restrict__ t,
                                                               unsigned nvox, float s, float* __restrict__ part) {
  __shared__ float red[2][kHeadThreads];
  const int b = blockIdx.y;
  float e2 = 0.f, t2 = 0.f;
#pragma unroll 4
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += gridDim.x * blockDim.x) {
    const long gi = (long)b * nvox + i;
    const float tv = s * t[gi], e = ys[gi] - tv;
    e2 += e * e;
    t2 += tv * tv;
  }
  red[0][threadIdx.x] = e2;
  red[1][threadIdx.x] = t2;
  __syncthreads();
  for (int k = kHeadThreads / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) {
      red[0][threadIdx.x] += red[0][threadIdx.x + k];
      red[1][threadIdx.x] += red[1][threadIdx.x + k];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[((long)b * gridDim.x + blockIdx.x) * 2] = red[0][0];
    part[((long)b * gridDim.x + blockIdx.x) * 2 + 1] = red[1][0];
  }
}

// loss = mean_b e2_b / t2_b (FP64 over the block partials, one warp per sample, then the samples in order);
// keeps t2_b for the gradient
constexpr int kLossThreads = 256;
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}
__global__ void __launch_bounds__(kLossThreads) k_loss(const float* __restrict__ part, int nblk, int B,
                                                       double* __restrict__ sums, float* __restrict__ loss) {
  const int lane = threadIdx.x & 31;
  for (int b = threadIdx.x >> 5; b < B; b += kLossThreads / 32) {
    double e2 = 0.0, t2 = 0.0;
    for (int k = lane; k < nblk; k += 32) {
      const float2 v = reinterpret_cast<const float2*>(part)[(long)b * nblk + k];
      e2 += v.x;
      t2 += v.y;
    }
    e2 = warp_sum(e2);
    t2 = warp_sum(t2);
    if (lane == 0) {
      sums[2 * b] = e2;
      sums[2 * b + 1] = t2;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && loss) {
    double l = 0.0;
    for (int b = 0; b < B; ++b) l += sums[2 * b] / sums[2 * b + 1];
    *loss = (float)(l / B);
  }
}

// head backward (82 -> 74 us at 128^2 x 32, batch 8, with the loads of two voxels in flight): dy = 2 (y_s - t_s) / (B t2_b); gradient of the head input h (bf16(leaky'(h) bf16(w dy)))
// and per-block partials of the head's weight and bias gradients sum dy h_c, sum dy
__global__ void __launch_bounds__(kHeadThreads) k_head_backward(const unsigned char* __restrict__ Hd, LevelArg L,
                                                                const float* __restrict__ ys, const float* __restrict__ t,
                                                                const float* __restrict__ wb, float s, int B,
                                                                const double* __restrict__ sums,
                                                                unsigned char* __restrict__ G, float* __restrict__ part) {
  __shared__ float red[kHeadThreads];
  const unsigned nvox = (unsigned)(L.D * L.H * L.W);
  const int b = blockIdx.y;
  float w[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) w[c] = bf16r(wb[c]);
  const float scale = (float)(2.0 / ((double)B * sums[2 * b + 1]));
  float acc[17];
#pragma unroll
  for (int c = 0; c < 17; ++c) acc[c] = 0.f;
#pragma unroll 2
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += gridDim.x * blockDim.x) {
    const unsigned r = i / L.W;
    const int ww = (int)(i - r * L.W), h = (int)(r % L.H), d = (int)(r / L.H);
    const long p = ppos(L, d, h, ww);
    const long gi = (long)b * nvox + i;
    const float dy = scale * (ys[gi] - s * t[gi]);
    uint4 hv[2];
#pragma unroll
    for (int half = 0; half < 2; ++half) hv[half] = __ldg(reinterpret_cast<const uint4*>(Hd + (((long)b * 2 + half) * L.Vs + p) * 16));
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const long o = (((long)b * 2 + half) * L.Vs + p) * 16;
      float a[8], gg[8];
      unpack8(hv[half], a);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        acc[8 * half + k] = fmaf(dy, a[k], acc[8 * half + k]);
        gg[k] = bf16r(w[8 * half + k] * dy) * (a[k] > 0.f ? 1.f : kLeaky);
      }
      *reinterpret_cast<uint4*>(G + o) = pack8(gg);
    }
    acc[16] += dy;
  }
  for (int c = 0; c < 17; ++c) {
    red[threadIdx.x] = acc[c];
    __syncthreads();
    for (int k = kHeadThreads / 2; k > 0; k >>= 1) {
      if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
      __syncthreads();
    }
    if (threadIdx.x == 0) part[((long)b * gridDim.x + blockIdx.x) * 17 + c] = red[0];
    __syncthreads();
  }
}

// one block per head parameter: the block partials in FP64, a fixed tree
__global__ void __launch_bounds__(kLossThreads) k_head_grad_reduce(const float* __restrict__ part, int n, float* __restrict__ g) {
  __shared__ double red[kLossThreads / 32];
  const int c = blockIdx.x;
  double s = 0.0;
  for (int k = threadIdx.x; k < n; k += kLossThreads) s += part[(long)k * 17 + c];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kLossThreads / 32; ++w) s += red[w];
    g[c] = (float)s;
  }
}

// Weight images from the FP32 master (see unet_conv.cu): forward [group][e][c pair][f][a = 2, 1, 0][o of the
// group][16 c] and input gradient [group][e][o pair][f][a = 2, 1, 0][c of the group][16 o] holding
// W[o][c][2 - a][2 - e][2 - f], both as K-major core matrices [o / 8][2][8][8].
__global__ void k_images(const float* __restrict__ w, int co, int ci, int ci_pad, int ngf, int ngb,
                         uint16_t* __restrict__ fwd, uint16_t* __restrict__ bwd) {
  const int total = 27 * co * ci_pad;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int cc = i & 7, r = (i >> 3) & 7, h = (i >> 6) & 1;
#pragma unroll
    for (int dir = 0; dir < 2; ++dir) {
      const int ng = dir ? ngb : ngf, pairs = (dir ? co : ci_pad) / 16;
      int rest = i >> 7;
      const int g8 = rest % (ng / 8);
      rest /= ng / 8;
      const int a = 2 - rest % 3;
      rest /= 3;
      const int f = rest % 3;
      rest /= 3;
      const int kp = rest % pairs;
      rest /= pairs;
      const int e = rest % 3, grp = rest / 3;
      const int row = grp * ng + 8 * g8 + r, col = kp * 16 + h * 8 + cc;
      if (dir == 0) {
        fwd[i] = tc::bf16_rn(col < ci ? w[((long)row * ci + col) * 27 + a * 9 + e * 3 + f] : 0.f);
      } else {
        bwd[i] = tc::bf16_rn(row < ci ? w[((long)col * ci + row) * 27 + (2 - a) * 9 + (2 - e) * 3 + (2 - f)] : 0.f);
      }
    }
  }
}

__global__ void k_adam_unet(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, long n, float lr, float c1, float c2) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
  }
}

int grid_for(long n, int threads = 256) { return (int)std::max<long>(1, std::min<long>((n + threads - 1) / threads, 152L * 8)); }

// ---------------------------------------------------------------------------------------- host side
int build_images(Unet* U, cudaStream_t st) {
  for (int k = 0; k < kNumConv; ++k) {
    const Layer& Ly = U->layer[k];
    k_images<<<grid_for(27L * Ly.co * Ly.ci_pad), 256, 0, st>>>(U->params + Ly.woff, Ly.co, Ly.ci, Ly.ci_pad, Ly.ng_f, Ly.ng_b,
                                                                 reinterpret_cast<uint16_t*>(U->imgs + Ly.img_f),
                                                                 reinterpret_cast<uint16_t*>(U->imgs + Ly.img_b));
  }
  FR3D_CUDA_TRY(cudaGetLastError());
  return FR3D_OK;
}

ConvArgs conv_args(const Unet* U, int lvl, int B) {
  ConvArgs a{};
  const Level& L = U->lv[lvl];
  a.B = B;
  a.D = L.D;
  a.H = L.H;
  a.W = L.W;
  a.Wp = L.Wp;
  a.HW = L.HW;
  a.Vs = L.Vs;
  a.q_first = L.q_first;
  a.ntiles = conv_tiles(L.q_first, L.q_last);
  a.err = U->err;
  return a;
}

ConvArgs conv_forward_args(const Unet* U, int k, int B) {
  const Layer& Ly = U->layer[k];
  ConvArgs a = conv_args(U, Ly.lvl, B);
  a.x = U->t[Ly.in_t];
  a.x_chunks = U->td[Ly.in_t].C / 8;
  a.x_off = Ly.in_off / 8;
  a.Cin = Ly.ci_pad;
  a.wimg = U->imgs + Ly.img_f;
  a.N = Ly.co;
  a.Ng = Ly.ng_f;
  a.y = U->t[Ly.out_t];
  a.y_chunks = U->td[Ly.out_t].C / 8;
  a.y_off = Ly.out_off / 8;
  a.bias = U->params + Ly.woff + (long)Ly.co * Ly.ci * 27;
  a.mode = kConvFwd;
  return a;
}
int conv_forward(const Unet* U, int k, int B, cudaStream_t st) { return conv3_launch(conv_forward_args(U, k, B), st); }

// The weight gradients' plans for batches of B: by the batch that is run, not the network's largest, so that the order of a
// batch's sums does not depend on the network it runs in.
int plan_wgrads(Unet* U, int B) {
  if (U->wg_batch == B) return FR3D_OK;
  U->wg_batch = 0;
  for (Layer& Ly : U->layer) FR3D_TRY(wgrad_plan(&Ly.wg, B));
  U->wg_batch = B;
  return FR3D_OK;
}

int conv_backward(Unet* U, int k, int B, cudaStream_t st) {
  const Layer& Ly = U->layer[k];
  // weight and bias gradient: partial sums, then their ordered sum
  WgradArgs w = Ly.wg;
  w.g = U->g[Ly.out_t];
  w.x = U->t[Ly.in_t];
  w.B = B;
  w.partials = U->partials;
  w.err = U->err;
  FR3D_TRY(wgrad3_launch(w, Ly.ci, U->grads + Ly.woff, U->grads + Ly.woff + (long)Ly.co * Ly.ci * 27, st));
  // input gradient
  if (Ly.dgrad) {
    ConvArgs a = conv_args(U, Ly.lvl, B);
    a.x = U->g[Ly.out_t];
    a.x_chunks = U->td[Ly.out_t].C / 8;
    a.x_off = Ly.out_off / 8;
    a.Cin = Ly.co;
    a.wimg = U->imgs + Ly.img_b;
    a.N = Ly.ci_pad;
    a.Ng = Ly.ng_b;
    a.y = U->g[Ly.in_t];
    a.y_chunks = U->td[Ly.in_t].C / 8;
    a.y_off = Ly.in_off / 8;
    a.mode = Ly.dgrad == 1 ? kConvDgradMask : kConvDgradPlain;
    a.mask = U->t[Ly.in_t];
    a.mask_chunks = U->td[Ly.in_t].C / 8;
    a.mask_off = Ly.in_off / 8;
    FR3D_TRY(conv3_launch(a, st));
  }
  return FR3D_OK;
}

constexpr int kLossBlocks = 128;   // per sample

int forward(Unet* U, const float* x, int B, const float* t, float* out, cudaStream_t st) {
  const Level& L0 = U->lv[0];
  dim3 blk = row_block(L0.W);
  k_pack_input<<<row_grid(B, 1, L0.D, L0.H, blk), blk, 0, st>>>(x, B, larg(L0), U->in_scale, U->t[T_X]);
  FR3D_CUDA_TRY(cudaGetLastError());
  FR3D_TRY(conv_forward(U, 0, B, st));
  FR3D_TRY(conv_forward(U, 1, B, st));
  for (int l = 1; l < kL; ++l) {
    const int src = T_CAT + l - 1;
    const int nc = kWidth[l - 1] / 8;
    blk = row_block(U->lv[l].W);
    FR3D_TRY(launch_on(true, k_pool, row_grid(B, nc, U->lv[l].D, U->lv[l].H, blk), blk, 0, st,
                       U->t[src], U->td[src].C / 8, kWidth[l] / 8, larg(U->lv[l - 1]), U->t[T_P + l - 1], nc, larg(U->lv[l]), nc, B));
    FR3D_TRY(conv_forward(U, 2 * l, B, st));
    FR3D_TRY(conv_forward(U, 2 * l + 1, B, st));
    if (l == kL - 1) FR3D_TRY(conv_forward(U, 8, B, st));
  }
  for (int l = kL - 2; l >= 0; --l) {
    const int src = l == kL - 2 ? T_B + 2 : T_D2 + l + 1;
    const int nc = kWidth[l + 1] / 8;
    blk = row_block(U->lv[l].W);
    FR3D_TRY(launch_on(true, k_up, row_grid(B, nc, U->lv[l + 1].D, U->lv[l + 1].H, blk), blk, 0, st,
                       U->t[src], U->td[src].C / 8, larg(U->lv[l + 1]), U->t[T_CAT + l], U->td[T_CAT + l].C / 8, larg(U->lv[l]), nc, B));
    const int k = 9 + 2 * (kL - 2 - l);
    FR3D_TRY(conv_forward(U, k, B, st));
    if (l > 0) FR3D_TRY(conv_forward(U, k + 1, B, st));
  }
  // the last convolution with the head; its own output is kept for the gradient only
  ConvArgs a = conv_forward_args(U, kNumConv - 1, B);
  a.mode = kConvHead;
  a.hx = x;
  a.hw = U->params + U->head_off;
  a.hs = U->in_scale;
  a.hout = out;
  if (t) a.hys = U->y;
  else a.y = nullptr;
  FR3D_TRY(conv3_launch(a, st));
  if (t)
    k_loss_partial<<<dim3(kLossBlocks, B), kHeadThreads, 0, st>>>(U->y, t, (unsigned)(L0.D * L0.H * L0.W), U->in_scale, U->red);
  FR3D_CUDA_TRY(cudaGetLastError());
  return FR3D_OK;
}

int backward(Unet* U, const float* t, int B, float* loss, cudaStream_t st) {
  const Level& L0 = U->lv[0];
  const int nblk = kLossBlocks;
  FR3D_TRY(plan_wgrads(U, B));
  k_loss<<<1, kLossThreads, 0, st>>>(U->red, nblk, B, U->lossbuf, loss);
  k_head_backward<<<dim3(nblk, B), kHeadThreads, 0, st>>>(U->t[T_D2], larg(L0), U->y, t, U->params + U->head_off,
                                                          U->in_scale, B, U->lossbuf, U->g[T_D2], U->red);
  k_head_grad_reduce<<<17, kLossThreads, 0, st>>>(U->red, nblk * B, U->grads + U->head_off);
  FR3D_CUDA_TRY(cudaGetLastError());
  for (int l = 0; l <= kL - 2; ++l) {
    const int k = 9 + 2 * (kL - 2 - l);
    FR3D_TRY(conv_backward(U, k + 1, B, st));
    FR3D_TRY(conv_backward(U, k, B, st));
    const int dst = l == kL - 2 ? T_B + 2 : T_D2 + l + 1;
    const int nc = kWidth[l + 1] / 8;
    const dim3 blk = row_block(U->lv[l + 1].W);
    FR3D_TRY(launch_on(true, k_up_backward, row_grid(B, nc, U->lv[l + 1].D, U->lv[l + 1].H, blk), blk, 0, st,
                       U->g[T_CAT + l], U->td[T_CAT + l].C / 8, larg(U->lv[l]), U->t[dst], U->g[dst], U->td[dst].C / 8, larg(U->lv[l + 1]), nc, B));
  }
  FR3D_TRY(conv_backward(U, 8, B, st));
  FR3D_TRY(conv_backward(U, 7, B, st));
  FR3D_TRY(conv_backward(U, 6, B, st));
  for (int l = kL - 2; l >= 0; --l) {
    const int nc = kWidth[l] / 8;
    const dim3 blk = row_block(U->lv[l].W);
    FR3D_TRY(launch_on(true, k_pool_backward, row_grid(B, nc, U->lv[l].D, U->lv[l].H, blk), blk, 0, st,
                       U->g[T_P + l], nc, larg(U->lv[l + 1]), U->t[T_CAT + l] + 0, U->g[T_CAT + l], U->td[T_CAT + l].C / 8, kWidth[l + 1] / 8, larg(U->lv[l]), nc, B));
    FR3D_TRY(conv_backward(U, 2 * l + 1, B, st));
    FR3D_TRY(conv_backward(U, 2 * l, B, st));
  }
  return FR3D_OK;
}

int check_input(const Unet* U, const void* x, int B) {
  if (!x || B < 1 || B > U->Bmax) return FR3D_ERR_INVALID_ARG;
  int dev = -1;
  FR3D_CUDA_TRY(cudaGetDevice(&dev));
  return dev == U->dev ? FR3D_OK : FR3D_ERR_INVALID_ARG;
}

uint64_t splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

}  // namespace fr3d

struct fr3d_unet {
  fr3d::Unet u;
};

using fr3d::Unet;

static void unet_free(Unet* U) {
  for (int i = 0; i < fr3d::T_N; ++i) {
    if (U->t[i]) cudaFree(U->t[i]);
    if (U->g[i]) cudaFree(U->g[i]);
  }
  void* ps[] = {U->params, U->grads, U->m, U->v, U->imgs, U->y, U->partials, U->red, U->lossbuf, U->err};
  for (void* p : ps)
    if (p) cudaFree(p);
}

extern "C" int fr3d_unet_create(int depth, int height, int width, int max_batch, float in_scale,
                                unsigned long long seed, fr3d_unet** out) {
  using namespace fr3d;
  if (!out || max_batch < 1 || !(in_scale > 0.f) || !isfinite(in_scale)) return FR3D_ERR_INVALID_ARG;
  if (depth < 8 || height < 8 || width < 8 || depth % 8 || height % 8 || width % 8 || depth > 256 || height > 512 ||
      width > 512)
    return FR3D_ERR_UNSUPPORTED_SIZE;
  fr3d_unet* h = new (std::nothrow) fr3d_unet();
  if (!h) return FR3D_ERR_OOM;
  Unet* U = &h->u;
  int rc = FR3D_OK;
  do {
    if (cudaGetDevice(&U->dev) != cudaSuccess) {
      rc = FR3D_ERR_CUDA;
      break;
    }
    U->D = depth;
    U->H = height;
    U->W = width;
    U->Bmax = max_batch;
    U->in_scale = in_scale;
    for (int l = 0; l < kL; ++l) U->lv[l] = make_level(depth >> l, height >> l, width >> l);
    // tensors
    U->td[T_X] = {16, 0};
    for (int l = 0; l < kL - 1; ++l) {
      U->td[T_E1 + l] = {kWidth[l], l};
      U->td[T_CAT + l] = {kWidth[l + 1] + kWidth[l], l};
      U->td[T_D1 + l] = {kWidth[l], l};
      U->td[T_D2 + l] = {kWidth[l], l};
    }
    for (int l = 1; l < kL; ++l) U->td[T_P + l - 1] = {kWidth[l - 1], l};
    for (int k = 0; k < 3; ++k) U->td[T_B + k] = {kWidth[kL - 1], kL - 1};
    for (int i = 0; i < T_N && rc == FR3D_OK; ++i) {
      const size_t b = (size_t)max_batch * (U->td[i].C / 8) * U->lv[U->td[i].lvl].Vs * 16;
      U->tbytes[i] = b;
      if (cudaMalloc(&U->t[i], b) != cudaSuccess || cudaMalloc(&U->g[i], b) != cudaSuccess ||
          cudaMemset(U->t[i], 0, b) != cudaSuccess || cudaMemset(U->g[i], 0, b) != cudaSuccess)
        rc = FR3D_ERR_OOM;
    }
    if (rc) break;
    // layers in the oracle's order
    struct Spec {
      int ci, co, lvl, in_t, in_off, out_t, out_off, dgrad;
    };
    const Spec sp[kNumConv] = {
        {1, 16, 0, T_X, 0, T_E1 + 0, 0, 0},
        {16, 16, 0, T_E1 + 0, 0, T_CAT + 0, 32, 1},
        {16, 32, 1, T_P + 0, 0, T_E1 + 1, 0, 2},
        {32, 32, 1, T_E1 + 1, 0, T_CAT + 1, 64, 1},
        {32, 64, 2, T_P + 1, 0, T_E1 + 2, 0, 2},
        {64, 64, 2, T_E1 + 2, 0, T_CAT + 2, 128, 1},
        {64, 128, 3, T_P + 2, 0, T_B + 0, 0, 2},
        {128, 128, 3, T_B + 0, 0, T_B + 1, 0, 1},
        {128, 128, 3, T_B + 1, 0, T_B + 2, 0, 1},
        {192, 64, 2, T_CAT + 2, 0, T_D1 + 2, 0, 2},
        {64, 64, 2, T_D1 + 2, 0, T_D2 + 2, 0, 1},
        {96, 32, 1, T_CAT + 1, 0, T_D1 + 1, 0, 2},
        {32, 32, 1, T_D1 + 1, 0, T_D2 + 1, 0, 1},
        {48, 16, 0, T_CAT + 0, 0, T_D1 + 0, 0, 2},
        {16, 16, 0, T_D1 + 0, 0, T_D2 + 0, 0, 1},
    };
    long off = 0;
    size_t ioff = 0, pmax = 0;
    for (int k = 0; k < kNumConv; ++k) {
      Layer& Ly = U->layer[k];
      Ly.ci = sp[k].ci;
      Ly.ci_pad = std::max(16, sp[k].ci);
      Ly.co = sp[k].co;
      Ly.lvl = sp[k].lvl;
      Ly.in_t = sp[k].in_t;
      Ly.in_off = sp[k].in_off;
      Ly.out_t = sp[k].out_t;
      Ly.out_off = sp[k].out_off;
      Ly.dgrad = sp[k].dgrad;
      Ly.woff = off;
      off += (long)Ly.co * Ly.ci * 27 + Ly.co;
      const size_t ib = 27 * (size_t)Ly.co * Ly.ci_pad * 2;
      Ly.img_f = ioff;
      ioff += (ib + 255) & ~(size_t)255;
      Ly.img_b = ioff;
      ioff += (ib + 255) & ~(size_t)255;
      const Level& L = U->lv[Ly.lvl];
      const int nt = conv_tiles(L.q_first, L.q_last);
      Ly.ng_f = conv_group(Ly.ci_pad, Ly.co, L.D, nt, max_batch);
      Ly.ng_b = conv_group(Ly.co, Ly.ci_pad, L.D, nt, max_batch);
      WgradArgs& w = Ly.wg;
      w.g_chunks = U->td[Ly.out_t].C / 8;
      w.g_off = Ly.out_off / 8;
      w.Cout = Ly.co;
      w.x_chunks = U->td[Ly.in_t].C / 8;
      w.x_off = Ly.in_off / 8;
      w.Cin = Ly.ci_pad;
      w.D = L.D;
      w.Wp = L.Wp;
      w.HW = L.HW;
      w.Vs = L.Vs;
      w.zero_pos = L.Vp;
      w.q_first = L.q_first;
      w.q_last = L.q_last;
      // (the largest batch is planned last: its plan is the one that stays)
      for (int b = 1; b <= max_batch; ++b) {
        if (!Ly.ng_f || !Ly.ng_b || wgrad_plan(&w, b) != FR3D_OK) rc = FR3D_ERR_UNSUPPORTED_SIZE;
        if (rc) break;
        pmax = std::max(pmax, wgrad_partial_floats(w, b));
      }
    }
    if (rc) break;
    U->head_off = off;
    U->n_params = off + kWidth[0] + 1;
    U->img_bytes = ioff;
    U->partial_floats = pmax;
    U->wg_batch = max_batch;
    U->red_floats = (size_t)128 * 17 * max_batch;
    const size_t np = (size_t)U->n_params;
    if (cudaMalloc(&U->params, np * 4) != cudaSuccess || cudaMalloc(&U->grads, np * 4) != cudaSuccess ||
        cudaMalloc(&U->m, np * 4) != cudaSuccess || cudaMalloc(&U->v, np * 4) != cudaSuccess ||
        cudaMalloc(&U->imgs, ioff) != cudaSuccess ||
        cudaMalloc(&U->y, (size_t)max_batch * depth * height * width * 4) != cudaSuccess ||
        cudaMalloc(&U->partials, pmax * 4) != cudaSuccess || cudaMalloc(&U->red, U->red_floats * 4) != cudaSuccess ||
        cudaMalloc(&U->lossbuf, sizeof(double) * 2 * (max_batch + 1)) != cudaSuccess ||
        cudaMalloc(&U->err, sizeof(int)) != cudaSuccess) {
      rc = FR3D_ERR_OOM;
      break;
    }
    // He-normal weights (std sqrt(2 / (27 ci))) from SplitMix64 + Box-Muller, zero biases, zero head
    std::vector<float> p(np, 0.f);
    uint64_t s = seed;
    for (int k = 0; k < kNumConv; ++k) {
      const Layer& Ly = U->layer[k];
      const double sd = sqrt(2.0 / (27.0 * Ly.ci));
      for (long i = 0; i < (long)Ly.co * Ly.ci * 27; ++i) {
        const double u1 = ((splitmix(s) >> 11) + 1.0) * (1.0 / 9007199254740993.0);
        const double u2 = (splitmix(s) >> 11) * (1.0 / 9007199254740992.0);
        p[Ly.woff + i] = (float)(sd * sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2));
      }
    }
    if (cudaMemcpy(U->params, p.data(), np * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(U->m, 0, np * 4) != cudaSuccess || cudaMemset(U->v, 0, np * 4) != cudaSuccess ||
        cudaMemset(U->grads, 0, np * 4) != cudaSuccess || cudaMemset(U->err, 0, sizeof(int)) != cudaSuccess) {
      rc = FR3D_ERR_CUDA;
      break;
    }
    rc = build_images(U, 0);
    if (rc == FR3D_OK && cudaDeviceSynchronize() != cudaSuccess) rc = FR3D_ERR_CUDA;
  } while (0);
  if (rc != FR3D_OK) {
    unet_free(U);
    delete h;
    return rc;
  }
  *out = h;
  return FR3D_OK;
}

extern "C" void fr3d_unet_destroy(fr3d_unet* net) {
  if (!net) return;
  unet_free(&net->u);
  delete net;
}

extern "C" int fr3d_unet_query(const fr3d_unet* net, int* n_params) {
  if (!net) return FR3D_ERR_INVALID_ARG;
  if (n_params) *n_params = (int)net->u.n_params;
  return FR3D_OK;
}

extern "C" int fr3d_unet_get_params(fr3d_unet* net, float* params) {
  if (!net || !params) return FR3D_ERR_INVALID_ARG;
  FR3D_CUDA_TRY(cudaDeviceSynchronize());
  FR3D_CUDA_TRY(cudaMemcpy(params, net->u.params, sizeof(float) * net->u.n_params, cudaMemcpyDeviceToHost));
  return FR3D_OK;
}

extern "C" int fr3d_unet_set_params(fr3d_unet* net, const float* params) {
  if (!net || !params) return FR3D_ERR_INVALID_ARG;
  Unet* U = &net->u;
  const size_t b = sizeof(float) * U->n_params;
  FR3D_CUDA_TRY(cudaDeviceSynchronize());
  FR3D_CUDA_TRY(cudaMemcpy(U->params, params, b, cudaMemcpyHostToDevice));
  FR3D_CUDA_TRY(cudaMemset(U->m, 0, b));
  FR3D_CUDA_TRY(cudaMemset(U->v, 0, b));
  U->adam_t = 0;
  FR3D_TRY(fr3d::build_images(U, 0));
  FR3D_CUDA_TRY(cudaDeviceSynchronize());
  return FR3D_OK;
}

extern "C" int fr3d_unet_forward(fr3d_unet* net, const float* x, int B, float* y, void* stream) {
  if (!net || !y) return FR3D_ERR_INVALID_ARG;
  FR3D_TRY(fr3d::check_input(&net->u, x, B));
  return fr3d::forward(&net->u, x, B, nullptr, y, (cudaStream_t)stream);
}

extern "C" int fr3d_unet_gradient(fr3d_unet* net, const float* x, const float* t, int B, float* grad, float* loss,
                                  void* stream) {
  if (!net || !t) return FR3D_ERR_INVALID_ARG;
  FR3D_TRY(fr3d::check_input(&net->u, x, B));
  Unet* U = &net->u;
  cudaStream_t st = (cudaStream_t)stream;
  FR3D_TRY(fr3d::forward(U, x, B, t, nullptr, st));
  FR3D_TRY(fr3d::backward(U, t, B, loss, st));
  if (grad) FR3D_CUDA_TRY(cudaMemcpyAsync(grad, U->grads, sizeof(float) * U->n_params, cudaMemcpyDeviceToDevice, st));
  return FR3D_OK;
}

extern "C" int fr3d_unet_train_step(fr3d_unet* net, const float* x, const float* t, int B, float lr, float* loss,
                                    void* stream) {
  if (!net || !t || !(lr > 0.f) || !isfinite(lr)) return FR3D_ERR_INVALID_ARG;
  FR3D_TRY(fr3d::check_input(&net->u, x, B));
  Unet* U = &net->u;
  cudaStream_t st = (cudaStream_t)stream;
  FR3D_TRY(fr3d::forward(U, x, B, t, nullptr, st));
  FR3D_TRY(fr3d::backward(U, t, B, loss, st));
  ++U->adam_t;
  const float c1 = 1.f - powf(0.9f, (float)U->adam_t), c2 = 1.f - powf(0.999f, (float)U->adam_t);
  fr3d::k_adam_unet<<<fr3d::grid_for(U->n_params), 256, 0, st>>>(U->params, U->m, U->v, U->grads, U->n_params, lr, c1,
                                                                   c2);
  FR3D_CUDA_TRY(cudaGetLastError());
  return fr3d::build_images(U, st);
}

extern "C" int fr3d_test_unet_wgrad_plan(fr3d_unet* net, int layer, int B, int* units, int* span) {
  if (!net || layer < 0 || layer >= fr3d::kNumConv || B < 1 || B > net->u.Bmax) return FR3D_ERR_INVALID_ARG;
  fr3d::WgradArgs w = net->u.layer[layer].wg;
  FR3D_TRY(fr3d::wgrad_plan(&w, B));
  if (units) *units = B * w.nspans * w.nchunks;
  if (span) *span = w.span;
  return FR3D_OK;
}

extern "C" int fr3d_unet_error_flags(fr3d_unet* net, int* flags) {
  if (!net || !flags) return FR3D_ERR_INVALID_ARG;
  FR3D_CUDA_TRY(cudaDeviceSynchronize());
  FR3D_CUDA_TRY(cudaMemcpy(flags, net->u.err, sizeof(int), cudaMemcpyDeviceToHost));
  return FR3D_OK;
}
