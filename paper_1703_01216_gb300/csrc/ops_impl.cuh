// Per-precision kernel launchers (included once per precision by ops_f32.cu / ops_f64.cu).
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "fft2d.cuh"
#include "ops.cuh"

namespace fr3d {

#define FR3D_FOR_EACH_N(X) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512)

template <typename K> static int set_smem(K kernel, size_t bytes) {
  return smem_optin(reinterpret_cast<const void*>(kernel), bytes);
}

template <typename T> static const typename cpx<T>::t* tw_of(const Handle* H, int L) {
  const int off = twiddle_offset(H, L);
  if constexpr (sizeof(T) == 4) return H->tw32 + off;
  else return H->tw64 + off;
}

constexpr int kSmallGrid = 2 * 152;  // below this many CTAs with the large tile, use the small one

template <typename T, int N, int TY, class PM = StridedPlanes<T>>
static int row_r2c_t(const Handle* H, const PM& pm, int nplanes, cudaStream_t st) {
  constexpr size_t sm = row_r2c_smem<T, N, TY>();
  auto kern = k_row_r2c<T, N, TY, PM>;
  FR3D_TRY(set_smem(kern, sm));
  dim3 grid(N / TY, nplanes);
  return launch_on(true, kern, grid, kThreads, sm, st, pm, tw_of<T>(H, N));
}

template <typename T, int N>
static int row_r2c_n(const Handle* H, const T* in, long in_ps, typename cpx<T>::t* out, int nplanes, cudaStream_t st) {
  constexpr int TY = RowTile<T, N>::v;
  const StridedPlanes<T> pm{in, in_ps, out, (long)(N / 2 + 1) * N};
  if ((long)nplanes * (N / TY) < kSmallGrid && SmallTile<N>::row < TY)
    return row_r2c_t<T, N, SmallTile<N>::row>(H, pm, nplanes, st);
  return row_r2c_t<T, N, TY>(H, pm, nplanes, st);
}

template <typename T, int N, bool INV, class Op, int TC>
static int col_t(const Handle* H, const Op& op, int nplanes, cudaStream_t st) {
  constexpr size_t sm = col_smem<T, N, TC>();
  auto kern = k_col_fft<T, N, INV, Op, TC>;
  FR3D_TRY(set_smem(kern, sm));
  dim3 grid((N / 2 + 1 + TC - 1) / TC, nplanes);
  return launch_on(true, kern, grid, kThreads, sm, st, op, tw_of<T>(H, N));
}

template <typename T, int N, bool INV, class Op>
static int col_n(const Handle* H, const Op& op, int nplanes, cudaStream_t st) {
  constexpr int TC = ColTile<T, N>::v;
  if ((long)nplanes * ((N / 2 + TC) / TC) < kSmallGrid && SmallTile<N>::col < TC)
    return col_t<T, N, INV, Op, SmallTile<N>::col>(H, op, nplanes, st);
  return col_t<T, N, INV, Op, TC>(H, op, nplanes, st);
}

template <typename T, int N, int MODE, int TY>
static int row_c2r_t(const Handle* H, const typename cpx<T>::t* in, T* out, int nplanes, int Q, int j0,
                     int out_stride, const SrcHost& src, const T* W, cudaStream_t st) {
  constexpr size_t sm = row_c2r_smem<T, N, TY>();
  auto kern = k_row_c2r<T, N, MODE, TY>;
  FR3D_TRY(set_smem(kern, sm));
  typename SrcOf<T>::t s;
  s.pts = reinterpret_cast<decltype(s.pts)>(src.pts);
  s.L = src.L;
  s.coef = (T)src.coef;
  RowGeom g{H->x0, H->y0, H->h};
  const T* zr;
  if constexpr (sizeof(T) == 4) zr = H->zr32;
  else zr = H->zr64;
  dim3 grid(N / TY, nplanes);
  return launch_on(true, kern, grid, kThreads, sm, st, in, out, Q, j0, out_stride, s, g, zr, W, (long)H->Mp * N * N,
                   tw_of<T>(H, N));
}

template <typename T, int N, int MODE>
static int row_c2r_n(const Handle* H, const typename cpx<T>::t* in, T* out, int nplanes, int Q, int j0,
                     int out_stride, const SrcHost& src, const T* W, cudaStream_t st) {
  constexpr int TY = row_c2r_tile<T, N, MODE>();
  // few planes: small tiles put more CTAs in flight (the forward operator's eight planes of 256^2: 64 CTAs of 32
  // rows take 12.6 us, 256 of 8 rows 5)
  if constexpr (MODE == 0 && SmallTile<N>::row < TY)
    if ((long)nplanes * (N / TY) < kSmallGrid)
      return row_c2r_t<T, N, MODE, SmallTile<N>::row>(H, in, out, nplanes, Q, j0, out_stride, src, W, st);
  return row_c2r_t<T, N, MODE, TY>(H, in, out, nplanes, Q, j0, out_stride, src, W, st);
}

template <typename T>
int Ops<T>::row_r2c(const Handle* H, const T* in, long in_ps, C* out, int nplanes, cudaStream_t st) {
  switch (H->n) {
#define X(N) \
  case N: return row_r2c_n<T, N>(H, in, in_ps, out, nplanes, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

template <typename T>
int Ops<T>::col_plain(const Handle* H, const C* in, C* out, int nplanes, bool inverse, cudaStream_t st) {
  ColPlain<T> op{in, out, (long)(H->n / 2 + 1) * H->n};
  switch (H->n) {
#define X(N)                                                         \
  case N:                                                            \
    return inverse ? col_n<T, N, true>(H, op, nplanes, st) : col_n<T, N, false>(H, op, nplanes, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

// the sizes of bin-ordered spectra (multi.cu)
template <typename T, bool INV>
static int col_bins(const Handle* H, const typename cpx<T>::t* in, typename cpx<T>::t* out, int nplanes, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    switch (H->n) {
#define X(N)                                                                                                       \
  case N: {                                                                                                        \
    constexpr int PB = ColTile<float, N>::v;                                                                       \
    constexpr size_t sm = col_smem<float, N, PB>();                                                                \
    auto kern = k_col_bins<N, INV, PB>;                                                                            \
    FR3D_TRY(set_smem(kern, sm));                                                                                  \
    return launch_on(true, kern, dim3(N / 2 + 1, (nplanes + PB - 1) / PB), kThreads, sm, st, in, out, nplanes,     \
                     tw_of<float>(H, N));                                                                          \
  }
      X(192) X(256) X(384) X(512)
#undef X
    }
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}
template <typename T>
int Ops<T>::col_to_bins(const Handle* H, const C* planes, C* bins, int nplanes, cudaStream_t st) {
  return col_bins<T, false>(H, planes, bins, nplanes, st);
}
template <typename T>
int Ops<T>::col_from_bins(const Handle* H, const C* bins, C* planes, int nplanes, cudaStream_t st) {
  return col_bins<T, true>(H, bins, planes, nplanes, st);
}

template <typename T>
int Ops<T>::col_solve1(const Handle* H, const C* Uh, C* out, const T* A, const T* D, const int* aidx, int nb, int Q,
                       int j0, int nj, cudaStream_t st) {
  ColSolve1<T> op;
  op.cband = H->cband;
  op.nb = nb;
  op.Uh = Uh;
  op.out = out;
  op.A = A;
  op.D = D;
  op.aidx = aidx;
  op.ps = (long)(H->n / 2 + 1) * H->n;
  op.Q = Q;
  op.j0 = j0;
  op.n = H->n;
  op.Cn = H->C;
  op.drow = nullptr;
  switch (H->n) {
#define X(N) \
  case N: return col_n<T, N, true>(H, op, nj * Q, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

template <typename T>
int Ops<T>::row_c2r_plain(const Handle* H, const C* in, T* out, int nplanes, int Q, int j0, int out_stride,
                          cudaStream_t st) {
  SrcHost none{nullptr, 0, 0.0};
  switch (H->n) {
#define X(N) \
  case N: return row_c2r_n<T, N, 0>(H, in, out, nplanes, Q, j0, out_stride, none, nullptr, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

template <typename T>
int Ops<T>::row_c2r_xi(const Handle* H, const C* in, T* out, int nj, int Q, int j0, const SrcHost& src, const T* W,
                       cudaStream_t st) {
  switch (H->n) {
#define X(N)                                                                                      \
  case N:                                                                                         \
    return W ? row_c2r_n<T, N, 2>(H, in, out, nj, Q, j0, 0, src, W, st)                             \
             : row_c2r_n<T, N, 1>(H, in, out, nj, Q, j0, 0, src, nullptr, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

// ---------------------------------------------------------------- forward contraction (Eq. (5)-(6))
template <typename T, typename C>
__global__ void k_contract_fwd(const C* __restrict__ Zh, C* __restrict__ Uh, const T* __restrict__ A, int Q, int M,
                               int Mp, long ps, T inv_n2) {
  const long total = (long)Q * M * ps;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const long bin = idx % ps;
    const int qi = (int)(idx / ps);
    const int q = qi / M, i = qi - q * M;
    const C* z = Zh + (long)q * Mp * ps + bin;
    const T* a = A + (long)i * Mp * ps + bin;
    T re = 0, im = 0;
    for (int j = 0; j < Mp; ++j) {
      const T w = a[(long)j * ps];
      const C v = z[(long)j * ps];
      re += w * v.x;
      im += w * v.y;
    }
    C r;
    r.x = re * inv_n2;
    r.y = im * inv_n2;
    Uh[idx] = r;
  }
}

template <typename T>
int Ops<T>::contract_fwd(const Handle* H, const C* Zh, C* Uh, const T* A, int Q, cudaStream_t st) {
  const long ps = (long)(H->n / 2 + 1) * H->n;
  const long total = (long)Q * H->M * ps;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 16);
  k_contract_fwd<T, C><<<blocks, 256, 0, st>>>(Zh, Uh, A, Q, H->M, H->Mp, ps, (T)(1.0 / ((double)H->n * H->n)));
  return cudaGetLastError() == cudaSuccess ? FR3D_OK : FR3D_ERR_CUDA;
}

template <typename T, int N>
static int col_contract_n(const Handle* H, const typename cpx<T>::t* Zh, typename cpx<T>::t* part, long part_cs,
                          const T* A, int Q, int chunks, cudaStream_t st) {
  constexpr int TC = ContractTile<T, N>::v;
  constexpr size_t sm = col_smem<T, N, TC>();
  auto kern = k_col_contract<T, N, TC>;
  FR3D_TRY(set_smem(kern, sm));
  const dim3 grid((N / 2 + TC) / TC, Q, chunks);
  return launch_on(true, kern, grid, kContractThreads, sm, st, Zh, part, A, H->Mp, (H->Mp + chunks - 1) / chunks, part_cs,
                   tw_of<T>(H, N));
}

// Depth chunks of the contraction: enough CTAs to fill the SMs (five each at n = 256), at least four depths each (FP64: one;
// a depth in FP64 takes as long as four; 192^2 x 8: 95 -> 65 us), no
// empty chunk; more partials than kMaxChunks cost the sum more than the extra CTAs give (16 chunks: 17 us).
template <typename T>
int Ops<T>::contract_chunks(const Handle* H, int Q) {
  int tc = (sizeof(T) == 4 ? 2048 : 1024) / H->n;
  tc = std::max(1, std::min(tc, H->n / 2 + 1));
  const int ctas = ((H->n / 2 + tc) / tc) * Q;
  const int want = std::max(1, std::min({(5 * 152 + ctas - 1) / ctas, sizeof(T) == 8 ? H->Mp : H->Mp / 4, kMaxChunks}));
  const int per = (H->Mp + want - 1) / want;
  return (H->Mp + per - 1) / per;
}

template <typename T>
int Ops<T>::col_contract(const Handle* H, const C* Zh, C* part, long part_cs, const T* A, int Q, int chunks,
                         cudaStream_t st) {
  switch (H->n) {
#define X(N) \
  case N: return col_contract_n<T, N>(H, Zh, part, part_cs, A, Q, chunks, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

template <typename T>
int Ops<T>::col_sum(const Handle* H, const C* part, long part_cs, C* Uh, int Q, int chunks, cudaStream_t st) {
  const ColSum<T> op{part, Uh, (long)(H->n / 2 + 1) * H->n, part_cs, chunks, H->n, (T)(1.0 / ((double)H->n * H->n))};
  switch (H->n) {
#define X(N) \
  case N: return col_n<T, N, true>(H, op, Q, st);
    FR3D_FOR_EACH_N(X)
#undef X
  }
  return FR3D_ERR_UNSUPPORTED_SIZE;
}

// ---------------------------------------------------------------- zeta = xi V0 (Sec. 2)
template <typename T, typename S>
__global__ void k_zeta_from_xi(const T* __restrict__ xi, T* __restrict__ zeta, int Q, int Mp, int n, S src,
                               RowGeom g, const T* __restrict__ zr) {
  const long plane = (long)n * n;
  const long total = (long)Q * Mp * plane;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const long pix = idx % plane;
    const int qj = (int)(idx / plane);
    const int q = qj / Mp, j = qj - q * Mp;
    const int a = (int)(pix % n), b = (int)(pix / n);
    const T x = (T)g.x0 + ((T)a + (T)0.5) * (T)g.h, y = (T)g.y0 + ((T)b + (T)0.5) * (T)g.h;
    zeta[idx] = xi[(long)j * plane + pix] * v0_at(src, q, x, y, zr[j]);
  }
}

template <typename T>
int Ops<T>::zeta_from_xi(const Handle* H, const T* xi, T* zeta, int Q, const SrcHost& src, cudaStream_t st) {
  typename SrcOf<T>::t s;
  s.pts = reinterpret_cast<decltype(s.pts)>(src.pts);
  s.L = src.L;
  s.coef = (T)src.coef;
  RowGeom g{H->x0, H->y0, H->h};
  const T* zr;
  if constexpr (sizeof(T) == 4) zr = H->zr32;
  else zr = H->zr64;
  const long total = (long)Q * H->Mp * H->n * H->n;
  const int blocks = (int)std::min<long>((total + 255) / 256, 152L * 16);
  k_zeta_from_xi<T><<<blocks, 256, 0, st>>>(xi, zeta, Q, H->Mp, H->n, s, g, zr);
  return cudaGetLastError() == cudaSuccess ? FR3D_OK : FR3D_ERR_CUDA;
}

// ---------------------------------------------------------------- discrepancy principle (Sec. 4)
// (p, q) of class c = p (p + 1) / 2 + q, q <= p (exact integer correction of a float estimate)
__device__ __forceinline__ void class_pq(int c, int& p, int& q) {
  p = (int)((sqrtf(8.f * (float)c + 1.f) - 1.f) * 0.5f);
  while ((p + 1) * (p + 2) / 2 <= c) ++p;
  while (p * (p + 1) / 2 > c) --p;
  q = c - p * (p + 1) / 2;
}

constexpr int kAlphaThreads = 256;
constexpr int kAlphaCPB = 64;      // classes per block at most
constexpr int kAlphaFill = 160;    // blocks that fill the chip (about one per SM)

// Per band b of frequency classes (one band: the whole spectrum),
//   r_b^2(alpha_k) = n^-2 sum_{c in b} Ft[c][k] P[c]  (Parseval; M = 1 closed form of the residual),
// with P[c] the data power of class c: every stored half-spectrum bin of the class, weighted 1 on
// the kx = 0 and kx = n/2 columns and 2 elsewhere (their mirror bins are not stored), summed over
// planes.  The discrepancy rule picks, per band, the largest alpha_k with r_b^2 <= thr2.t[b].
// The kernel is a chain of dependent steps (6 MB at 256^2, 8 sources, 64 candidates, about 1 us of HBM time), so the
// steps are kept short: the classes per block weigh the FP64 products of a block (64 classes and 64 candidates take
// 1 us) against the sums of more blocks (alpha_cpb), a block's filter slab is fetched by asynchronous copies before the data
// transform has finished (programmatic launch; the slab depends on the handle only), and the
// block sums are reduced in one or two levels of tickets (alpha_group).
// Deterministic: fixed-order sums of a block's classes; block sums in a fixed interleaved order.
// FP64 runs at a small fraction of the FP32 rate on this GPU, so the serial parts avoid FP64 chains:
// the choice is a warp ballot per band rather than a loop over candidates.
struct BandThr {
  double t[FR3D_MAX_BANDS];
};

inline int alpha_blocks(int Cn, int cpb) { return (Cn + cpb - 1) / cpb; }
// Blocks per group of the reduction's first level.  One SM adds two FP64 numbers per cycle: up to 2048 numbers the last
// block adds them all (a second level costs about 2600 cycles of fences and tickets), above that about sqrt(blocks)
// groups share the work (132 blocks of 64 sums in one level: 4200 cycles; in 11 groups of 12: 384 + 352).
inline int alpha_group(int nblk, int O) {
  if (nblk * O <= 2048) return nblk;
  int g = 8;
  while (g * g < nblk) ++g;
  return g;
}
// Classes per block for a single call (a multiple of 8 up to 64, at most kAlphaFill blocks unless 64 classes need
// more): the fewest FP64 cycles of the products of a block and of the reduction of the blocks' sums.
inline int alpha_cpb(int Cn, int na, int nb) {
  const int O = na * nb;
  int best = kAlphaCPB;
  long bc = -1;
  for (int c = kAlphaCPB; c >= 8; c -= 8) {
    const int nblk = alpha_blocks(Cn, c), g = alpha_group(nblk, O), ngr = (nblk + g - 1) / g;
    if (nblk > kAlphaFill && c < kAlphaCPB) break;
    const long cost = (long)c * na / 2 + (ngr == 1 ? (long)nblk * O / 2 : 2600 + (long)(g + ngr) * O / 2);
    if (bc < 0 || cost < bc) {
      bc = cost;
      best = c;
    }
  }
  return best;
}
// the group tickets of the alpha rule in the handle's partial-sum buffer (tables.cu)
unsigned* alpha_tickets(const Handle* H);

__device__ __forceinline__ void cp_async(void* dst, const void* src, bool wide) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if (wide) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// Sum of cnt vectors of O values, O apart: thread (t, o) adds every TPO-th vector (B loads in flight), the TPO sums of
// an o are added in order and handed to emit(o, sum).  red: kAlphaThreads doubles.
template <int B, class Em>
__device__ __forceinline__ void alpha_reduce(const double* __restrict__ src, int cnt, int O, double* red, Em emit, int tid) {
  const int Ow = min(O, kAlphaThreads), TPO = kAlphaThreads / Ow;
  const int ol = tid % Ow, t = tid / Ow;
  for (int o0 = 0; o0 < O; o0 += Ow) {
    const int o = o0 + ol;
    double s = 0.0;
    if (o < O && t < TPO) {
      for (int q0 = t; q0 < cnt; q0 += B * TPO) {
        double v[B];
#pragma unroll
        for (int i = 0; i < B; ++i) v[i] = __ldcg(src + (long)min(q0 + i * TPO, cnt - 1) * O + o);
#pragma unroll
        for (int i = 0; i < B; ++i)
          if (q0 + i * TPO < cnt) s += v[i];   // (adding the zeros would cost the FP64 pipe as much)
      }
    }
    red[tid] = s;
    __syncthreads();
    if (t == 0 && o < O) {
      for (int k = 1; k < TPO; ++k) s += red[k * Ow + ol];
      emit(o, s);
    }
    __syncthreads();
  }
}

template <int B, typename C>
__device__ __forceinline__ void alpha_choose_body(const C* __restrict__ Uh, long ps, int nplanes, int n, int Cn,
                                                  const double* __restrict__ Ft, int na, const BandThr& thr2,
                                                  const unsigned char* __restrict__ cband, int nb, double inv_n2,
                                                  double* __restrict__ partials, unsigned* __restrict__ counter,
                                                  int* __restrict__ aidx, double* __restrict__ res_out,
                                                  int* __restrict__ info, unsigned* __restrict__ gticket, int blk,
                                                  int nblk, int cpb, int gsize) {
  // partials: [nblk][O] block sums, then [groups][O] group sums; gticket: one ticket per group
  // (alpha_tickets); counter: the ticket over the groups.  Every ticket is zero between launches.
  // Accumulation types: the class power P[c] is summed in the data's precision (at most 4 nplanes
  // positive terms); the residual sums F[c][k] P[c] over classes and blocks are FP64.
  using A = typename std::conditional<std::is_same<C, float2>::value, float, double>::type;
  __shared__ double sP[kAlphaCPB];
  __shared__ unsigned char sB[kAlphaCPB];
  __shared__ unsigned present;
  __shared__ double red[kAlphaThreads];
  __shared__ double sPart[FR3D_MAX_BANDS * FR3D_MAX_ALPHAS];   // this block's sums; later the r^2 curves
  __shared__ int flg[FR3D_MAX_BANDS];
  __shared__ bool last;
  extern __shared__ __align__(16) double sF[];   // [cpb][na] slab of Ft for this block's classes
  const int tid = threadIdx.x;
  const int c0 = blk * cpb, ncl = min(cpb, Cn - c0), O = nb * na;
  {
    const double* slab = Ft + (long)c0 * na;   // 16-byte aligned: c0 is a multiple of 8
    const int nF = ncl * na;
    for (int e = 2 * tid; e < nF; e += 2 * kAlphaThreads) cp_async(sF + e, slab + e, e + 1 < nF);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (tid == 0) present = 0;
  for (int o = tid; o < O; o += kAlphaThreads) sPart[o] = 0.0;
  // class powers: `split` adjacent lanes per class share its (member, plane) items; member m of class (p, q):
  // (p, q), (p, n - q), (q, p), (q, n - p), where they are distinct stored bins
  const int split = 1 << (31 - __clz(kAlphaThreads / cpb)), cl = tid / split, sub = tid % split, c = c0 + cl;
  int p = 0, q = 0;
  if (cl < ncl) class_pq(c, p, q);
  const bool mirq = q != 0 && 2 * q != n, mirp = p != 0 && 2 * p != n;
  const A wp = (p == 0 || 2 * p == n) ? A(1) : A(2), wq = (q == 0 || 2 * q == n) ? A(1) : A(2);
  pdl_wait();   // the data spectra
  A acc = 0;
  if (cl < ncl)
    for (int i0 = sub; i0 < 4 * nplanes; i0 += 8 * split) {
      C v[8];
      A w[8];   // 0: no such item (it reads the class's first bin instead: no branch between the loads)
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * split, m = i & 3, pl = i >> 2;
        const bool has = pl < nplanes && (m == 0 || (m == 1 && mirq) || (m == 2 && p != q) || (m == 3 && p != q && mirp));
        const int kx = m < 2 ? p : q, ky = m == 0 ? q : (m == 1 ? n - q : (m == 2 ? p : n - p));
        v[u] = __ldcg(Uh + (has ? pl * ps + (long)kx * n + ky : (long)p * n + q));
        w[u] = has ? (m < 2 ? wp : wq) : A(0);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (w[u] != A(0)) acc += w[u] * (v[u].x * v[u].x + v[u].y * v[u].y);
    }
  for (int m = 1; m < split; m <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);   // fixed order
  __syncthreads();   // present and the zeros
  if (sub == 0 && cl < ncl) {
    sP[cl] = (double)acc;
    const int b = nb > 1 ? (int)cband[c] : 0;
    sB[cl] = (unsigned char)b;
    if (nb > 1) atomicOr(&present, 1u << b);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // per band of this block: the sums of F[c][k] P[c] (S threads per candidate, fixed order)
  const int S = kAlphaThreads / na, kc = tid % na, sb = tid / na;
  for (unsigned bands = nb > 1 ? present : 1u; bands; bands &= bands - 1) {
    const int b = __ffs(bands) - 1;
    double a2 = 0.0;
    if (sb < S) {
#pragma unroll 4
      for (int cc = sb; cc < ncl; cc += S)
        if (nb == 1 || sB[cc] == b) a2 = fma(sF[cc * na + kc], sP[cc], a2);
    }
    red[tid] = a2;
    __syncthreads();
    if (tid < na) {
      for (int k = 1; k < S; ++k) a2 += red[k * na + tid];
      sPart[b * na + tid] = a2;
    }
    __syncthreads();
  }
  for (int o = tid; o < O; o += kAlphaThreads) partials[(long)blk * O + o] = sPart[o];
  // level 1: a ticket of the block's group; the group's last block adds the group's block sums
  const int ngr = (nblk + gsize - 1) / gsize, g = blk / gsize, gsz = min(gsize, nblk - g * gsize);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(gticket + g, 1u) == (unsigned)(gsz - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) gticket[g] = 0u;
  auto final_sum = [&](int o, double s) {
    s *= inv_n2;
    sPart[o] = s;
    if (res_out) res_out[o] = s;
  };
  const double* mine = partials + (long)g * gsize * O;
  if (ngr == 1) {
    pdl_release();   // every other block has finished: a programmatic successor may start its set-up
    alpha_reduce<B>(mine, gsz, O, red, final_sum, tid);
  } else {
    // level 2: a ticket over the groups; the last group adds the group sums
    double* gpart = partials + (long)nblk * O;
    alpha_reduce<B>(mine, gsz, O, red, [&](int o, double s) { gpart[(long)g * O + o] = s; }, tid);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(counter, 1u) == (unsigned)(ngr - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    pdl_release();
    alpha_reduce<B>(gpart, ngr, O, red, final_sum, tid);
    if (tid == 0) *counter = 0u;
  }
  __syncthreads();
  // choice per band, one warp per band: ballots of r^2 <= thr over the candidates, largest index wins
  const int warp = tid >> 5, lane = tid & 31;
  for (int b = warp; b < nb; b += 8) {
    int best = -1, ok = 0, flags = 0;
    for (int k0 = 0; k0 < na; k0 += 32) {
      const int k = k0 + lane;
      bool good = false, bad = false;
      if (k < na) {
        const double v = sPart[b * na + k];
        const long long bits = __double_as_longlong(v);
        bad = ((bits >> 52) & 0x7ff) == 0x7ff;      // Inf or NaN
        good = v <= thr2.t[b];
      }
      const unsigned bg = __ballot_sync(0xffffffffu, good);
      if (__ballot_sync(0xffffffffu, bad)) flags |= FR3D_INFO_NONFINITE;
      if (bg) best = k0 + 31 - __clz(bg);
      ok += __popc(bg);
    }
    if (best < 0) {
      best = 0;
      flags |= FR3D_INFO_ALPHA_NONE_SATISFIES;
    } else if (ok == na) {
      flags |= FR3D_INFO_ALPHA_ALL_SATISFY;
    }
    if (lane == 0) {
      aidx[b] = best;
      flg[b] = flags;
    }
  }
  __syncthreads();
  if (tid == 0) {
    int flags = 0;
    for (int b = 0; b < nb; ++b) flags |= flg[b];
    if (info) *info = flags;
  }
}

template <typename C>
__global__ void __launch_bounds__(kAlphaThreads) k_alpha_choose(
    const C* __restrict__ Uh, long ps, int nplanes, int n, int Cn, const double* __restrict__ Ft, int na, BandThr thr2,
    const unsigned char* __restrict__ cband, int nb, double inv_n2, double* __restrict__ partials,
    unsigned* __restrict__ counter, int* __restrict__ aidx, double* __restrict__ res_out, int* __restrict__ info,
    unsigned* __restrict__ gticket, int cpb, int gsize) {
  alpha_choose_body<16>(Uh, ps, nplanes, n, Cn, Ft, na, thr2, cband, nb, inv_n2, partials, counter, aidx, res_out, info,
                        gticket, (int)blockIdx.x, (int)gridDim.x, cpb, gsize);
}

template <typename T>
int Ops<T>::alpha_choose(Handle* H, const C* Uh, int nplanes, int n_alpha, const double* thr2, int nb, int* aidx,
                         double* residuals, int* info, cudaStream_t st) {
  const int cpb = alpha_cpb(H->C, n_alpha, nb), blocks = alpha_blocks(H->C, cpb);
  FR3D_TRY(ensure_partials(H));
  const long ps = (long)(H->n / 2 + 1) * H->n;
  const size_t sm = sizeof(double) * cpb * n_alpha;
  FR3D_TRY(set_smem(k_alpha_choose<C>, sm));
  BandThr t;
  for (int b = 0; b < nb; ++b) t.t[b] = thr2[b];
  return launch_on(true, k_alpha_choose<C>, dim3(blocks), kAlphaThreads, sm, st, Uh, ps, nplanes, H->n, H->C, H->Ft, n_alpha,
                    t, H->cband, nb, 1.0 / ((double)H->n * H->n), H->partials, H->counter, aidx, residuals, info,
                    alpha_tickets(H), cpb, alpha_group(blocks, nb * n_alpha));
}

}  // namespace fr3d
