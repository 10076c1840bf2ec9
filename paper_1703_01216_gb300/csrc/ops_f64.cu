// FP64 instantiation of the transform, solve and combination kernels, and the FP64 combination table.
#include "ops_impl.cuh"
template struct fr3d::Ops<double>;

namespace fr3d {

// W_q = V0_q / sum_q' V0_q'^2 on the R grid in FP64 (Algorithm 1 step 4 for several source parameters).
// Built once per geometry and source set; bound by the FP64 pipe (one reciprocal square root per voxel,
// source and point).
__global__ void k_wtab64(double* __restrict__ W, int Q, int Mp, int n, Src64 src, double x0, double y0, double h,
                         const double* __restrict__ zr) {
  const long plane = (long)n * n, total = (long)Mp * plane;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int j = (int)(idx / plane);
    const long pix = idx % plane;
    const double x = x0 + ((double)(pix % n) + 0.5) * h, y = y0 + ((double)(pix / n) + 0.5) * h;
    double s = 0.0;
    for (int q = 0; q < Q; ++q) {
      const double v = v0_at(src, q, x, y, zr[j]);
      W[(long)q * total + idx] = v;
      s = fma(v, v, s);
    }
    const double r = 1.0 / s;
    for (int q = 0; q < Q; ++q) W[(long)q * total + idx] *= r;
  }
}

int build_wtab64(const Handle* H, double* W, int Q, const double* pts64, int L, double coef, cudaStream_t st) {
  const Src64 s{pts64, L, coef};
  const long total = (long)H->Mp * H->n * H->n;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 16);
  k_wtab64<<<blocks, 256, 0, st>>>(W, Q, H->Mp, H->n, s, H->x0, H->y0, H->h, H->zr64);
  return cudaGetLastError() == cudaSuccess ? FR3D_OK : FR3D_ERR_CUDA;
}

}  // namespace fr3d
