// FP32 instantiation of the transform, solve and combination kernels, and its combination table.  Scalar complex adds here: with
// packed FP32x2 adds the row pass with the combination (k_row_c2r, xi output) needs more registers and
// runs 17 % slower at n = 512 (measured at the paper geometry: 0.154 against 0.131 ms).
#define FR3D_SCALAR_COMPLEX_ADDS
#include "ops_impl.cuh"
template struct fr3d::Ops<float>;

namespace fr3d {

// V0_q at the voxels 2m and 2m + 1 of rows y and y + 1, with the roundings of v0_at
__device__ __forceinline__ void v0_quad(const Src32& s, const RowGeom& g, int q, int y, int m, float z, float2* v) {
  const float hh = (float)g.h, xa = (float)g.x0 + ((float)(2 * m) + 0.5f) * hh, xb = xa + hh;
  const float ya = (float)g.y0 + ((float)y + 0.5f) * hh, yb = (float)g.y0 + ((float)(y + 1) + 0.5f) * hh;
  const float4* p = s.pts + q * s.L;
  v[0] = v[1] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int l = 0; l < s.L; ++l) {
    const float4 a = __ldg(p + l);
    const float dxa = xa - a.x, dxb = xb - a.x, dya = ya - a.y, dyb = yb - a.y, dz = z - a.z, zz = dz * dz;
    const float ra = fmaf(dya, dya, zz), rb = fmaf(dyb, dyb, zz);
    v[0].x += rsqrtf(fmaf(dxa, dxa, ra));
    v[0].y += rsqrtf(fmaf(dxb, dxb, ra));
    v[1].x += rsqrtf(fmaf(dxa, dxa, rb));
    v[1].y += rsqrtf(fmaf(dxb, dxb, rb));
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) v[r] = make_float2(s.coef * v[r].x, s.coef * v[r].y);
}

// W_q = V0_q / sum_q' V0_q'^2 on the R grid for the unfused row pass (n = 512), [Q][M'][n][n], from the row pass's own
// FP32 evaluation of V0.  Bound by the FP32 pipe, about nine instructions per voxel, source and point, so that a program
// that moves its sources on every call pays what the evaluation in the row pass cost.  Through k_wtab (FP64 differences
// and scaling) the table took 2.2 ms at 512^2 x 32, four sources of five points, now 80 us; and xi was up to
// 5 % further from FP64 than with the row pass's evaluation, now less than 1 %.
// A thread takes two voxels of two rows at a time: four reciprocal square roots in flight per point.
__global__ void __launch_bounds__(256) k_wtab_row(float* __restrict__ W, int Q, int Mp, int n, Src32 src, RowGeom g,
                                                  const float* __restrict__ zr) {
  constexpr int kKeep = 8;   // sources whose V0 stays in registers; the rest are evaluated again
  const int L = n / 2, m = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.z;
  if (m >= L) return;
  const float z = zr[j];
  const long qs = (long)Mp * n * L;
  for (int y = 2 * blockIdx.y; y < n; y += 2 * gridDim.y) {
    float2* w = reinterpret_cast<float2*>(W) + ((long)j * n + y) * L + m;
    float2 keep[kKeep][2], s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    auto squares = [&](const float2* v) {
#pragma unroll
      for (int r = 0; r < 2; ++r) s[r] = make_float2(fmaf(v[r].x, v[r].x, s[r].x), fmaf(v[r].y, v[r].y, s[r].y));
    };
    auto put = [&](int q, const float2* v) {
#pragma unroll
      for (int r = 0; r < 2; ++r) w[q * qs + r * L] = make_float2(v[r].x / s[r].x, v[r].y / s[r].y);
    };
#pragma unroll
    for (int q = 0; q < kKeep; ++q)
      if (q < Q) {
        v0_quad(src, g, q, y, m, z, keep[q]);
        squares(keep[q]);
      }
    for (int q = kKeep; q < Q; ++q) {
      float2 v[2];
      v0_quad(src, g, q, y, m, z, v);
      squares(v);
    }
#pragma unroll
    for (int q = 0; q < kKeep; ++q)
      if (q < Q) put(q, keep[q]);
    for (int q = kKeep; q < Q; ++q) {
      float2 v[2];
      v0_quad(src, g, q, y, m, z, v);
      put(q, v);
    }
  }
}

int build_wtab_row(const Handle* H, float* W, int Q, int L, double coef, cudaStream_t st) {
  const Src32 s{H->pts32, L, (float)coef};
  const RowGeom g{H->x0, H->y0, H->h};
  const int half = H->n / 2, rows = std::max(1, std::min(half, 152 * 32 / H->Mp));
  k_wtab_row<<<dim3((half + 255) / 256, rows, H->Mp), std::min(half, 256), 0, st>>>(W, Q, H->Mp, H->n, s, g, H->zr32);
  return cudaGetLastError() == cudaSuccess ? FR3D_OK : FR3D_ERR_CUDA;
}

}  // namespace fr3d
