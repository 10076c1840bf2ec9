// The U-Net post-corrector's 3 x 3 x 3 convolutions on the tensor cores (tcgen05, BF16 operands, FP32
// accumulation in TMEM), as implicit GEMMs over a padded, channel-chunked activation layout.
//
// Activation layout ("CP"): per sample and per chunk of 8 channels, one plane of Vs voxels of 16 bytes
// (8 BF16 channels), Vs = (D + 2)(H + 2)(W + 2) + 128: the volume with a one-voxel zero halo on every
// side, linearised (w fastest), plus 128 zero guard voxels.  A tap (a, e, f) of the 3 x 3 x 3 stencil is
// then a constant shift s(a, e, f) = (a - 1) Hp Wp + (e - 1) Wp + (f - 1) of the linear position, with
// the zero padding supplied by the halo; outputs are computed for 128 consecutive positions at a time
// (an MMA tile of M = 128 rows) and only the interior ones are stored.
//
// Forward and input-gradient kernel (k_conv3): D[p][n] = sum over taps and input channels of
// X[p + s(tap)][c] * Wimg[tap][n][c], by plane sweeps.  A CTA keeps the weights of Ng output channels in
// shared memory for its whole life and walks the depth of a 128-position tile of the (h, w) plane: every
// input plane is loaded once per (e, 16 input channels) (a slab of 130 positions of two channel chunks; the
// three f taps are the same slab with the operand's start moved by 16 bytes) and multiplied with the taps of
// all three a at once, N = 3 Ng columns: they belong to the outputs of the three neighbouring planes, whose
// accumulators ("slots" of Ng TMEM columns, zeroed when they are handed back) lie side by side in a ring.  One
// CTA per SM runs up to four independent pipes (tiles), each with a producer warp, an MMA warp and four epilogue
// warps that drain a plane's slot while the next planes run.
//   Before, every (a, e) re-read the slab and the weights for each tile, with N = Ng columns per MMA: 188 us for
//   16 -> 16 channels at 128^2 x 32, batch 8, now 78 us (tensors in and out of HBM: 41 us).  A single pipe takes
//   197 us, two 115: an MMA of 48 columns needs 46 cycles of issue and operand reads, and what a pipe waits and
//   issues between its stages is only hidden behind the other pipes' MMAs.
//   The products of an output are accumulated in the order (a, e, channel pair, f) whatever Ng, depth chunk
//   and grid, so the results do not depend on them, bit for bit.
// Weight-gradient kernel (k_wgrad3): dW[tap][o][c] = sum_p G[p][o] X[p + s(tap)][c], a GEMM whose K is the
// voxels: both operands come straight from CP planes, which hold 8 channels per 16 bytes, i.e. they are
// MN-major operands (the instruction descriptor's transpose bits).  The rows stack the three f taps (the
// output gradient shifted by one voxel) of Og <= 32 output channels, the columns the three a and three e taps of
// 16 input channels; the a taps are the input planes d - 1, d, d + 1 of a ring, so a plane sweep loads every
// input window once instead of once per a, and one CTA covers all 27 taps with one MMA per 16 voxels.
#include <math.h>

#include <algorithm>
#include <mutex>

#include "ops.cuh"
#include "tc.cuh"
#include "unet.cuh"
#include "wide_sum.cuh"

namespace fr3d {

namespace {

constexpr long kPolls = 1L << 22;
constexpr uint32_t kSleepNs = 1000;   // suspend-time hint of the waits: a waiting thread parks (bound: kPolls * 1 us)
constexpr int kSlabPos = 130;                   // positions of one e slab: 128 + the two f neighbours
constexpr int kSlabBytes = kSlabPos * 16;       // one channel chunk of a slab
constexpr int kItemBytes = 2 * kSlabBytes;      // one (e, 16 channels) item: two chunks
constexpr int kConvStageBytes = 3 * kItemBytes; // a stage: three consecutive items (3 Cin / 16 items per plane)
constexpr int kConvMaxStages = 8;               // per pipe
constexpr int kConvPipes = 4;                   // pipes of a CTA at most
constexpr int kPipeThreads = 192;               // per pipe: four epilogue warps, a producer and an MMA warp
constexpr int kTmemCols = 512;
constexpr int kMaxSlots = kTmemCols / 16;
constexpr size_t kMaxSmem = 227 * 1024;
// MN-major shared-memory descriptor: byte strides between core matrices along MN (channel chunks) and
// along K (groups of 8 voxels); the MN stride goes in the SBO field, the K stride in LBO (measured)
__device__ __forceinline__ uint64_t desc_mn(uint32_t saddr, uint32_t mn_stride, uint32_t k_stride) {
  return tc::desc_kmajor(saddr, k_stride, mn_stride);
}
__host__ __device__ constexpr uint32_t idesc_mn(int M, int N) {
  return tc::idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  return (uint32_t)tc::bf16_rn(a) | ((uint32_t)tc::bf16_rn(b) << 16);
}
__device__ __forceinline__ float lo16(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float hi16(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

__device__ __forceinline__ int flag(const int* f) { return *reinterpret_cast<const volatile int*>(f); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}

// ------------------------------------------------------------------------------------------ k_conv3
// a unit of work: the depth chunk o0 .. o0 + cnt - 1 (padded plane indices) of the tile at q0 of sample b
struct ConvUnit {
  int b, q0, o0, cnt;
  int kmin, kmax;   // input planes o0 - 1 + k, k in [kmin, kmax]: the zero halo planes at both ends are skipped
};
__device__ __forceinline__ ConvUnit conv_unit(const ConvArgs& a, int u) {
  ConvUnit c;
  const int ch = u % a.nchunks, r = u / a.nchunks;
  c.b = r / a.ntiles;
  c.q0 = a.q_first + (r - c.b * a.ntiles) * 128;
  c.o0 = 1 + ch * a.nd;
  c.cnt = min(a.nd, a.D + 1 - c.o0);
  c.kmin = c.o0 == 1 ? 1 : 0;
  c.kmax = c.o0 + c.cnt - 1 == a.D ? c.cnt : c.cnt + 1;
  return c;
}

struct ConvPipe {
  uint64_t full[kConvMaxStages], empty[kConvMaxStages], sdone[kMaxSlots], sfree[kMaxSlots], zeroed, drain;
  int issued;
};

// HEAD: mode kConvHead, an instance of its own (as a branch of the others' epilogue it slowed the input gradients by 7 %)
template <int PIPES, bool HEAD>
__global__ void __launch_bounds__(PIPES* kPipeThreads, 1) k_conv3(ConvArgs a) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) ConvPipe pipes[PIPES];
  __shared__ __align__(8) uint64_t wfull;
  __shared__ uint32_t tbase;
  __shared__ int sabort;
  __shared__ float sbias[64], shead[17];
  // warps [0, 4 PIPES): epilogue (pipe = warp / 4; warp % 4 picks the 32 TMEM lanes it may read), then the
  // producers, then the MMA warps
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int role = warp < 4 * PIPES ? 0 : (warp < 5 * PIPES ? 1 : 2);
  const int pipe = role == 0 ? warp >> 2 : (role == 1 ? warp - 4 * PIPES : warp - 5 * PIPES);
  ConvPipe& P = pipes[pipe];
  uint64_t *full = P.full, *empty = P.empty, *sdone = P.sdone, *sfree = P.sfree;
  const int Ng = a.Ng, cpairs = a.Cin / 16, S = a.stages, slog = a.slog, nslots = 1 << slog, smask = nslots - 1;
  const int grp = blockIdx.x % a.ngroups;
  // units go round the CTAs first and round their pipes next, so that the CTAs' shares differ by one unit at most
  const int ctas = gridDim.x / a.ngroups, w0 = blockIdx.x / a.ngroups + pipe * ctas, wstep = ctas * PIPES;
  const int nunits = a.B * a.ntiles * a.nchunks;
  const uint32_t wbytes = (uint32_t)(27 * a.Cin * Ng * 2);
  unsigned char* stages = sm + ((wbytes + 127) & ~127u) + (size_t)pipe * S * kConvStageBytes;
  if (tid < PIPES) {
    ConvPipe& Q = pipes[tid];
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&Q.full[s], 1);
      tc::mbar_init(&Q.empty[s], 1);
    }
    for (int s = 0; s < nslots; ++s) {
      tc::mbar_init(&Q.sdone[s], 1);
      tc::mbar_init(&Q.sfree[s], 4);
    }
    tc::mbar_init(&Q.zeroed, 4);
    tc::mbar_init(&Q.drain, 1);
    Q.issued = 0;
    if (tid == 0) {
      tc::mbar_init(&wfull, 1);
      sabort = 0;
    }
    tc::mbar_fence_init();
  }
  if (warp == 0) tc::tmem_alloc(&tbase, kTmemCols);
  pdl_wait();
  if (tid < Ng) sbias[tid] = a.bias ? a.bias[grp * Ng + tid] : 0.f;
  if (HEAD && tid < 17) shead[tid] = tid < 16 ? tc::bf16_val(tc::bf16_rn(a.hw[tid])) : a.hw[16];
  tc::fence_before_sync();
  __syncthreads();
  pdl_release();   // the CTA holds its tensor memory: a successor's CTA on this SM cannot take it while it waits for this one
  tc::fence_after_sync();
  const uint32_t tmem = tbase + pipe * (kTmemCols / PIPES);
  if (role == 1) {
    // producer: the group's weights once, then the slabs of every plane of every unit
    if (pipe == 0) {
      if (lane == 0) tc::mbar_arrive_expect_tx(&wfull, wbytes);
      __syncwarp();
      const unsigned char* wsrc = a.wimg + (size_t)grp * wbytes;
      for (uint32_t o = lane * 8192u; o < wbytes; o += 32u * 8192u)
        tc::bulk_g2s(sm + o, wsrc + o, min(8192u, wbytes - o), &wfull);
    }
    // Every value is the same in all lanes and one elected lane issues, as in the MMA warp: a copy per lane is
    // issued lane by lane.  192 -> 64 channels at 32^2 x 8, batch 8, on one pipe: 103 -> 89 us.
    int s = 0, use = 0;
    bool ok = true;
    for (int u = w0; u < nunits && ok; u += wstep) {
      const ConvUnit c = conv_unit(a, u);
      const unsigned char* src = a.x + (((long)c.b * a.x_chunks + a.x_off) * a.Vs + (long)(c.o0 - 1) * a.HW + c.q0 - 1) * 16;
      for (int k = c.kmin; k <= c.kmax && ok; ++k) {
        int e = -1, cp = 0;   // item: e row shift, channel pair
        for (int st = 0; st < cpairs; ++st) {
          ok = !flag(&sabort);
          if (ok && use > 0) ok = tc::mbar_wait_sleep(&empty[s], (uint32_t)((use - 1) & 1), kPolls, kSleepNs);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          const bool one = tc::elect_one();
          if (one) {
            tc::mbar_arrive_expect_tx(&full[s], kConvStageBytes);
            ++P.issued;
          }
          unsigned char* dst = stages + s * kConvStageBytes;
#pragma unroll
          for (int it = 0; it < 3; ++it) {
            if (one) {
              const unsigned char* from = src + (2L * cp * a.Vs + (long)k * a.HW + e * a.Wp) * 16;
              tc::bulk_g2s(dst + it * kItemBytes, from, kSlabBytes, &full[s]);
              tc::bulk_g2s(dst + it * kItemBytes + kSlabBytes, from + a.Vs * 16, kSlabBytes, &full[s]);
            }
            if (++cp == cpairs) {
              cp = 0;
              ++e;
            }
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ++use;
          }
        }
      }
    }
    if (!ok) sabort = 1;
  } else if (role == 2) {
    // MMA warp: every value is the same in all its lanes (the tensor instructions take their descriptors from
    // uniform registers; a single-lane branch cost 165 cycles per MMA), one elected lane issues
    bool ok = tc::mbar_wait_sleep(&wfull, 0u, kPolls, kSleepNs) && tc::mbar_wait_sleep(&P.zeroed, 0u, kPolls, kSleepNs);
    int s = 0, ph = 0, n0 = 0;
    const uint32_t da0 = tc::smem_addr(stages) >> 4, db0 = tc::smem_addr(sm) >> 4;
    const uint64_t dah = tc::desc_kmajor(0, kSlabBytes, 128), dbh = tc::desc_kmajor(0, 128, 256);
    const uint32_t id1 = tc::idesc_bf16(128, Ng), dn = (uint32_t)(Ng >> 3) << 17;   // one more block of Ng columns
    for (int u = w0; u < nunits && ok; u += wstep) {
      const ConvUnit c = conv_unit(a, u);
      for (int k = c.kmin; k <= c.kmax && ok; ++k) {
        // the outputs this input plane feeds: r = k - 2 .. k (taps a = 2, 1, 0; weight blocks 0, 1, 2): one run of
        // adjacent slots, or two where the ring wraps
        const int r0 = max(0, k - 2), r1 = min(c.cnt - 1, k);
        const int s0 = (n0 + r0) & smask;
        if (k < c.cnt || k == c.kmin)   // slots touched for the first time: wait until they have been drained
          for (int r = k == c.kmin ? r0 : k; r <= r1 && ok; ++r) {
            const int n = n0 + r;
            if (n > smask) ok = tc::mbar_wait_sleep(&sfree[n & smask], (uint32_t)(((n >> slog) - 1) & 1), kPolls, kSleepNs);
          }
        const int m0 = min(r1 - r0 + 1, nslots - s0), m1 = r1 - r0 + 1 - m0;
        const uint32_t c0 = tmem + s0 * Ng, i0 = id1 + (m0 - 1) * dn, i1 = id1 + (m1 - 1) * dn;
        const uint32_t b0 = (uint32_t)((r0 - (k - 2)) * 2 * Ng), b1 = b0 + m0 * 2 * Ng;
        tc::fence_after_sync();
        for (int st = 0; st < cpairs && ok; ++st) {
          ok = tc::mbar_wait_sleep(&full[s], (uint32_t)ph, kPolls, kSleepNs);
          if (!ok) break;
          tc::fence_after_sync();
          const uint32_t da = da0 + s * (kConvStageBytes / 16), db = db0 + st * 54 * Ng;
          if (tc::elect_one()) {
#pragma unroll
            for (int x = 0; x < 9; ++x) {   // items x / 3, taps f = x % 3
              const uint64_t dax = dah | (da + (x / 3) * (kItemBytes / 16) + x % 3);
              tc::mma_bf16(c0, dax, dbh | (db + x * 6 * Ng + b0), i0, true);
              if (m1 > 0) tc::mma_bf16(tmem, dax, dbh | (db + x * 6 * Ng + b1), i1, true);
            }
            tc::mma_commit(&empty[s]);
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1;
          }
        }
        // outputs complete with this plane
        if (ok && k >= 2 && tc::elect_one())
          for (int r = k - 2; r < c.cnt && (r == k - 2 || k == c.kmax); ++r) tc::mma_commit(&sdone[(n0 + r) & smask]);
        if (ok && k < 2 && k == c.kmax && tc::elect_one())
          for (int r = 0; r < c.cnt; ++r) tc::mma_commit(&sdone[(n0 + r) & smask]);
        __syncwarp();
      }
      n0 += c.cnt;
      if (flag(&sabort)) ok = false;
    }
    if (!ok) sabort = 1;
    if (tc::elect_one()) tc::mma_commit(&P.drain);
    __syncwarp();
  } else {
    // epilogue: row = position q0 + row of the tile
    const int row = tid & 127;
    int n0 = 0;
    bool ok = true;
    const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    // every slot starts at zero, and is handed back as zeros
    for (int j = 0; j < nslots * Ng; j += 16) tc::tmem_st16_zero(tw + j);
    tc::tmem_st_wait();
    tc::fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(&P.zeroed);
    for (int u = w0; u < nunits && ok; u += wstep) {
      const ConvUnit c = conv_unit(a, u);
      const int q = c.q0 + row, hh = q / a.Wp, ww = q - hh * a.Wp;
      const bool valid = hh >= 1 && hh <= a.H && ww >= 1 && ww <= a.W;
      for (int r = 0; r < c.cnt; ++r) {
        const int n = n0 + r, use = n >> slog, slot = n & smask;
        const bool got = !flag(&sabort) && tc::mbar_wait_sleep(&sdone[slot], (uint32_t)(use & 1), kPolls, kSleepNs);
        ok = __all_sync(0xffffffffu, got);
        if (!ok) {
          sabort = 1;
          break;
        }
        tc::fence_after_sync();
        const long p = (long)(c.o0 + r) * a.HW + q;
        for (int j = 0; j < Ng / 8; j += 2) {
          float v[16];
          tc::tmem_ld16(tw + slot * Ng + 8 * j, v);
          tc::tmem_st16_zero(tw + slot * Ng + 8 * j);
          if (j + 2 >= Ng / 8) {   // the slot's last read: hand it back
            tc::tmem_st_wait();
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sfree[slot]);
          }
          if (valid) {
            const long jc = (long)grp * (Ng / 8) + j;
            if (HEAD || a.mode == kConvFwd) {
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const float z = v[k] + sbias[8 * j + k];
                v[k] = z > 0.f ? z : kLeaky * z;
              }
            } else if (a.mode == kConvDgradMask) {
              // the gradient is stored (rounded) first, then scaled by the leaky derivative and rounded again,
              // as the two steps of the chain rule store it
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const uint4 m = __ldg(reinterpret_cast<const uint4*>(
                    a.mask + (((long)c.b * a.mask_chunks + a.mask_off + jc + h) * a.Vs + p) * 16));
                const uint32_t mw[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  float& lo = v[8 * h + 2 * k];
                  float& hi = v[8 * h + 2 * k + 1];
                  const uint32_t st = pack2(lo, hi);
                  lo = lo16(st);
                  hi = hi16(st);
                  if (!(lo16(mw[k]) > 0.f)) lo *= kLeaky;
                  if (!(hi16(mw[k]) > 0.f)) hi *= kLeaky;
                }
              }
            }
            if constexpr (HEAD) {
              // the head multiplies the stored (rounded) outputs, in the order of channel pairs (k, 8 + k)
              const long gi = (((long)c.b * a.D + c.o0 + r - 1) * a.H + hh - 1) * a.W + ww - 1;
              float h = shead[16];
#pragma unroll
              for (int k = 0; k < 8; ++k)
                h = fmaf(shead[k], tc::bf16_val(tc::bf16_rn(v[k])), fmaf(shead[8 + k], tc::bf16_val(tc::bf16_rn(v[8 + k])), h));
              const float y = tc::bf16_val(tc::bf16_rn(a.hs * __ldg(a.hx + gi))) + h;
              if (a.hys) a.hys[gi] = y;
              if (a.hout) a.hout[gi] = y / a.hs;
            }
#pragma unroll
            for (int h = 0; h < 2 && (!HEAD || a.y); ++h) {
              uint4 o;
              o.x = pack2(v[8 * h], v[8 * h + 1]);
              o.y = pack2(v[8 * h + 2], v[8 * h + 3]);
              o.z = pack2(v[8 * h + 4], v[8 * h + 5]);
              o.w = pack2(v[8 * h + 6], v[8 * h + 7]);
              *reinterpret_cast<uint4*>(a.y + (((long)c.b * a.y_chunks + a.y_off + jc + h) * a.Vs + p) * 16) = o;
            }
          }
          __syncwarp();
        }
      }
      n0 += c.cnt;
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (sabort && tid < PIPES) {
    // a bounded wait gave up: report it, and let the copies and MMAs in flight finish (bounded) before leaving
    ConvPipe& Q = pipes[tid];
    if (a.err) atomicOr(a.err, FR3D_INFO_TIMEOUT);
    tc::mbar_wait(&wfull, 0u, kPolls);
    for (int i = max(0, Q.issued - S); i < Q.issued; ++i) tc::mbar_wait(&Q.full[i % S], (uint32_t)((i / S) & 1), kPolls);
    tc::mbar_wait(&Q.drain, 0u, kPolls);
  }
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tbase, kTmemCols);
}

// ------------------------------------------------------------------------------------------ k_wgrad3
constexpr int kWgMaxSlots = 16;                 // ring slots at most
constexpr int kWgThreads = 192;                 // warps 0-3 bias sums and epilogue, 4 producer, 5 MMA
constexpr int kWgPlane = kWgVox * 16;           // bytes of one window: kWgVox voxels of one channel chunk
constexpr int kWgX = 3 * kWgCg / 8;             // input windows of a plane: [e][two chunks]
static_assert(kWgCg == 16, "an input group is two chunks");
constexpr int kWgCols = 9 * kWgCg;              // accumulator columns: [a][e][c]
constexpr uint32_t kWgTmem = 256;

// One CTA: the partial sums of one unit (sample, span of in-plane positions, depth chunk) for one pair of
// channel groups.  A span is walked in sub-ranges of kWgVox positions, each swept through the depth.  Step k
// of a sweep loads the input plane g0 - 1 + k (three e windows per chunk) and, from k = 2 on, the gradient plane
// g0 - 2 + k (three f windows per chunk) and multiplies that gradient plane with the input planes of steps
// k - 2, k - 1 and k: the taps a = 0, 1, 2.  The input planes lie in a ring of their own, so the three are
// adjacent and one MMA of N = 144 columns takes them all (two where the ring wraps: 2 steps in 9 or 14).  The
// idle epilogue warps add the bias gradient from the gradient windows meanwhile.  48 gradient rows (Og = 16) run
// with M = 64, which reads half of the A operand; with M = 128 the rows past 3 Og are whatever lies behind them
// in shared memory (the input ring follows) and their accumulators are never read.
// Bound (16 -> 16 channels at 128^2 x 32, batch 8): the window copies, 57 cycles per KB and 83 per 2 KB and SM, hence
// windows of 128 voxels (64: 173 us, 128: 122), then issue and operand reads of the MMAs, 2 KB + 4.5 KB per 16 voxels.
// With windows of 64 voxels copied by a lane each and one MMA per a, of 48 to 160 columns: 225 us, and 568 us for
// 48 -> 16 channels, now 322.
__global__ void __launch_bounds__(kWgThreads, 2) k_wgrad3(WgradArgs a) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t full[kWgMaxSlots], xempty[kWgMaxSlots], gempty[kWgMaxSlots], done;
  __shared__ uint32_t tbase;
  __shared__ int sabort, issued;
  __shared__ float sb[4][32];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int S = a.slots, SG = a.gslots;
  const int gc = a.Og / 8, nG = 3 * gc;
  const int gbytes = nG * kWgPlane;
  unsigned char* xring = sm + SG * gbytes;
  const int npairs = a.n_og * a.n_cg;
  const int pair = blockIdx.x % npairs, unit = blockIdx.x / npairs;
  const int og = pair / a.n_cg, cg = pair - og * a.n_cg;
  const int ch = unit % a.nchunks, rest = unit / a.nchunks;
  const int b = rest / a.nspans, sp = rest - b * a.nspans;
  const int g0 = 1 + ch * a.nd, cnt = min(a.nd, a.D + 1 - g0);
  const int v0 = a.q_first + sp * a.span, v1 = min(v0 + a.span, a.q_last + 1);   // in-plane positions [v0, v1)
  const bool bias = cg == 0;
  if (tid == 0) {
    const uint32_t readers = bias ? 5 : 1;   // the MMA warp's commit, and the four bias warps
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&xempty[s], readers);
    }
    for (int s = 0; s < SG; ++s) tc::mbar_init(&gempty[s], readers);
    tc::mbar_init(&done, 1);
    tc::mbar_fence_init();
    sabort = 0;
    issued = 0;
  }
  if (warp == 0) tc::tmem_alloc(&tbase, kWgTmem);
  pdl_wait();
  tc::fence_before_sync();
  __syncthreads();
  pdl_release();   // after the allocation, as in k_conv3
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  if (warp == 4) {
    // Producer warp.  Like the MMA warp it keeps every value the same in all lanes and lets one elected lane issue: the
    // copy takes its operands from uniform registers, and a copy per lane is issued lane by lane (1 KB a lane: 77
    // cycles per copy and SM; 16 -> 16 channels with the 2 KB windows: 135 instead of 122 us).
    const unsigned char* gsrc = a.g + ((long)b * a.g_chunks + a.g_off + og * gc) * a.Vs * 16;
    const unsigned char* xsrc = a.x + ((long)b * a.x_chunks + a.x_off + cg * (kWgCg / 8)) * a.Vs * 16;
    int s = 0, use = 0, sg = 0, guse = 0;
    bool ok = true;
    for (int v = v0; v < v1 && ok; v += kWgVox) {
      const int rem = min(kWgVox, v1 - v), kv = (rem + 15) & ~15;
      for (int k = 0; k < cnt + 2; ++k) {
        ok = !flag(&sabort);
        if (ok && use > 0) ok = tc::mbar_wait_sleep(&xempty[s], (uint32_t)((use - 1) & 1), kPolls, kSleepNs);
        if (ok && k >= 2 && guse > 0) ok = tc::mbar_wait_sleep(&gempty[sg], (uint32_t)((guse - 1) & 1), kPolls, kSleepNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (tc::elect_one()) {
          tc::mbar_arrive_expect_tx(&full[s], (uint32_t)((kWgX + (k >= 2 ? nG : 0)) * kv * 16));
          ++issued;
          const unsigned char* xs = xsrc + ((long)(g0 - 1 + k) * a.HW + v) * 16;
          unsigned char* xd = xring + s * (kWgX * kWgPlane);
#pragma unroll
          for (int j = 0; j < kWgX; ++j)
            tc::bulk_g2s(xd + j * kWgPlane, xs + ((j & 1) * a.Vs + ((j >> 1) - 1) * a.Wp) * 16, (uint32_t)(kv * 16), &full[s]);
          if (k >= 2) {
            // (the last K step of a span may end past it: the gradient's tail comes from the plane's zero guard)
            const unsigned char* gs = gsrc + ((long)(g0 - 2 + k) * a.HW + v) * 16;
            unsigned char* gd = sm + sg * gbytes;
            for (int c = 0; c < gc; ++c) {
#pragma unroll
              for (int f = 0; f < 3; ++f) {
                unsigned char* dst = gd + (f * gc + c) * kWgPlane;
                tc::bulk_g2s(dst, gs + (c * a.Vs - (f - 1)) * 16, (uint32_t)(rem * 16), &full[s]);
                if (kv > rem) tc::bulk_g2s(dst + rem * 16, gsrc + a.zero_pos * 16, (uint32_t)((kv - rem) * 16), &full[s]);
              }
            }
          }
        }
        __syncwarp();
        if (k >= 2 && ++sg == SG) {
          sg = 0;
          ++guse;
        }
        if (++s == S) {
          s = 0;
          ++use;
        }
      }
    }
    if (!ok) sabort = 1;
  } else if (warp == 5) {
    // MMA warp: uniform values, one elected lane issues (as in k_conv3)
    const int M = nG * 8 <= 64 ? 64 : 128;
    const uint64_t dh = desc_mn(0, kWgPlane, 128);
    const uint32_t dg0 = tc::smem_addr(sm) >> 4, dx0 = tc::smem_addr(xring) >> 4;
    int s = 0, ph = 0, sg = 0;
    bool ok = true, acc = false;
    for (int v = v0; v < v1 && ok; v += kWgVox) {
      const int ks = (min(kWgVox, v1 - v) + 15) / 16;
      for (int k = 0; k < cnt + 2; ++k) {
        ok = tc::mbar_wait_sleep(&full[s], (uint32_t)ph, kPolls, kSleepNs);
        if (!ok) break;
        if (k >= 2) {
          tc::fence_after_sync();
          const int s1 = s >= 1 ? s - 1 : s - 1 + S, s2 = s >= 2 ? s - 2 : s - 2 + S;
          const int m0 = min(3, S - s2);   // planes of the first run; the rest start over at slot 0
          const uint32_t da = dg0 + sg * (gbytes / 16), db0 = dx0 + s2 * (kWgX * kWgPlane / 16);
          const uint32_t i0 = idesc_mn(M, m0 * 3 * kWgCg), i1 = idesc_mn(M, (3 - m0) * 3 * kWgCg);
          const uint32_t c1 = tmem + m0 * 3 * kWgCg;
          if (tc::elect_one()) {
#pragma unroll
            for (int kk = 0; kk < kWgVox / 16; ++kk)
              if (kk < ks) {
                tc::mma_bf16(tmem, dh | (da + 16 * kk), dh | (db0 + 16 * kk), i0, acc || kk > 0);
                if (m0 < 3) tc::mma_bf16(c1, dh | (da + 16 * kk), dh | (dx0 + 16 * kk), i1, acc || kk > 0);
              }
            tc::mma_commit(&gempty[sg]);
            tc::mma_commit(&xempty[s2]);
            if (k == cnt + 1) {
              tc::mma_commit(&xempty[s1]);
              tc::mma_commit(&xempty[s]);
            }
          }
          acc = true;
          __syncwarp();
          if (++sg == SG) sg = 0;
        }
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok) sabort = 1;
    if (tc::elect_one()) tc::mma_commit(&done);
    __syncwarp();
  } else {
    if (bias) {
      // bias gradient: every thread adds its voxels of the unshifted (f = 1) windows
      float acc[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) acc[k] = 0.f;
      int s = 0, ph = 0, sg = 0;
      bool ok = true;
      for (int v = v0; v < v1 && ok; v += kWgVox) {
        const int rem = min(kWgVox, v1 - v);
        for (int k = 0; k < cnt + 2; ++k) {
          ok = __all_sync(0xffffffffu, tc::mbar_wait_sleep(&full[s], (uint32_t)ph, kPolls, kSleepNs));
          if (!ok) break;
          if (k >= 2) {
            for (int vx = tid; vx < rem; vx += 128) {
              const unsigned char* w = sm + sg * gbytes + gc * kWgPlane + vx * 16;
#pragma unroll
              for (int h = 0; h < 4; ++h)
                if (h < gc) {
                  const uint4 q = *reinterpret_cast<const uint4*>(w + h * kWgPlane);
                  const uint32_t qw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    acc[8 * h + 2 * i] += lo16(qw[i]);
                    acc[8 * h + 2 * i + 1] += hi16(qw[i]);
                  }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&gempty[sg]);
            if (++sg == SG) sg = 0;
          }
          if (lane == 0) mbar_arrive(&xempty[s]);
          if (++s == S) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) sabort = 1;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], m);
        if (lane == i) sb[warp][i] = acc[i];
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (tid < a.Og)
        a.bias_partials[(long)unit * a.Cout + og * a.Og + tid] = (sb[0][tid] + sb[1][tid]) + (sb[2][tid] + sb[3][tid]);
    }
    // epilogue: accumulator row (f, o) is lane tid, with M = 64 the first 16 lanes of each warp
    const bool got = tc::mbar_wait_sleep(&done, 0u, kPolls, kSleepNs);
    if (!__all_sync(0xffffffffu, got)) sabort = 1;
    tc::fence_after_sync();
    const uint32_t tw = tmem + ((uint32_t)(warp * 32) << 16);
    const bool half = nG * 8 <= 64;
    const int row = half ? (lane < 16 ? warp * 16 + lane : nG * 8) : tid;
    float* dst = a.partials + ((long)blockIdx.x * nG * 8 + row) * kWgCols;
    for (int n = 0; n < kWgCols; n += 16) {
      float v[16];
      tc::tmem_ld16(tw + n, v);
      if (row < nG * 8)
#pragma unroll
        for (int k = 0; k < 16; k += 4)
          *reinterpret_cast<float4*>(dst + n + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (sabort && tid == 0) {
    if (a.err) atomicOr(a.err, FR3D_INFO_TIMEOUT);
    for (int i = max(0, issued - S); i < issued; ++i) tc::mbar_wait(&full[i % S], (uint32_t)((i / S) & 1), kPolls);
    tc::mbar_wait(&done, 0u, kPolls);
  }
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, kWgTmem);
}

// dW[o][c][tap] (c < ci) and db[o]: the units' partial sums added in a fixed order (blockDim.y threads per element
// take every blockDim.y-th unit, then their sums in order).  A thread adds in three FP32 words, which lose less than FP64
// additions (wide_sum.cuh): those and the conversions were the bound.
// 29 MB of partials: 42 -> 22 us, 86 MB: 98 -> 58 us, with four times the loads in flight; the loads of eight units are
// requested before the first is added (the gradient at 128^2 x 32, batch 8: 3329 -> 3253 us).  Sums that are not finite
// are added again in FP64, as a chain that leaves FP32's range on the way has to be.  The partials are read with coherent
// loads: k_wgrad3 may still be writing them when this kernel starts.
constexpr int kWgRedThreads = 512;
__global__ void __launch_bounds__(kWgRedThreads) k_wgrad_reduce(WgradArgs a, int nunits, int ci, float* __restrict__ dW,
                                                               float* __restrict__ db) {
  __shared__ double red[kWgRedThreads];
  pdl_wait();
  pdl_release();
  const int per = 3 * a.Og * kWgCols, npairs = a.n_og * a.n_cg, nw = per * npairs;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool ok = i < nw + a.Cout;
  double s = 0.0;
  if (ok) {
    const float* p = i < nw ? a.partials + i : a.bias_partials + (i - nw);
    const long ustep = i < nw ? nw : a.Cout;
    WideSum sum;
    constexpr int kFlight = 8;   // loads requested before the first addition
    const int step = blockDim.y;
    int u = threadIdx.y;
    for (; u + (kFlight - 1) * step < nunits; u += kFlight * step) {
      float x[kFlight];
#pragma unroll
      for (int k = 0; k < kFlight; ++k) x[k] = __ldcg(p + (u + k * step) * ustep);
#pragma unroll
      for (int k = 0; k < kFlight; ++k) sum.add(x[k]);
    }
    for (; u < nunits; u += step) sum.add(__ldcg(p + u * ustep));
    s = sum.value();
    if (!sum.finite()) {
      s = 0.0;
      for (int u = threadIdx.y; u < nunits; u += blockDim.y) s += (double)__ldcg(p + u * ustep);
    }
  }
  if (blockDim.y > 1) {
    red[threadIdx.y * blockDim.x + threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y != 0) return;
    for (unsigned y = 1; y < blockDim.y; ++y) s += red[y * blockDim.x + threadIdx.x];
  }
  if (!ok) return;
  if (i >= nw) {
    db[i - nw] = (float)s;
    return;
  }
  const int pair = i / per, m = (i - pair * per) / kWgCols, n = i % kWgCols;
  const int og = pair / a.n_cg, cg = pair - og * a.n_cg;
  const int f = m / a.Og, o = og * a.Og + m % a.Og;
  const int ta = n / (3 * kWgCg), e = n / kWgCg - 3 * ta, c = cg * kWgCg + n % kWgCg;
  if (c < ci) dW[((long)o * ci + c) * 27 + ta * 9 + e * 3 + f] = (float)s;
}

int sm_count(int* sms) {
  int dev = 0;
  FR3D_CUDA_TRY(cudaGetDevice(&dev));
  FR3D_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return FR3D_OK;
}

// input planes a depth chunk of nd outputs reads (the zero halo planes at the ends of the depth are skipped)
int conv_planes(int D, int nd) { return nd >= D ? D : (2 * nd >= D ? nd + 1 : nd + 2); }

// A way to run a convolution: output channels per CTA, pipes per CTA, stages per pipe, planes per depth chunk.
struct ConvPlan {
  int Ng = 0, pipes = 0, stages = 0, nd = 0;
  double cost = 0;
};
size_t conv_weight_bytes(int Cin, int Ng) { return ((size_t)27 * Cin * Ng * 2 + 127) & ~(size_t)127; }
constexpr size_t kSmemSlack = 3 * 1024;   // static shared memory and alignment kept out of the dynamic allocation

// Cycles per MMA of N columns with c pipes of a CTA at work, fitted to measurements (N = 48, 96, 144): alone, the
// waits and the issue of a pipe's stages are exposed; with four pipes the operand reads and the slabs' writes to
// shared memory are what is left.  (16 -> 16 channels at 128^2 x 32, batch 8: 197 us with one pipe, 115 with two,
// 78 with four.)
double conv_mma_cycles(int N, int c) { return c == 1 ? 49 + 0.75 * N : (c == 2 ? 60 + 0.35 * N : 45 + 0.38 * N); }

// The plan whose largest share takes the fewest cycles: units of a CTA x planes x MMAs x cycles per MMA.  Larger
// groups read the slabs less often, smaller ones and shorter depth chunks spread a small volume over more SMs.
// ng: only this group size (0: any).
ConvPlan conv_plan(int Cin, int N, int D, int ntiles, int B, int ng, int sms) {
  ConvPlan best;
  const int cand[] = {64, 48, 32, 16};
  for (int Ng : cand) {
    if (N % Ng || (ng && Ng != ng)) continue;
    const size_t wb = conv_weight_bytes(Cin, Ng);
    if (wb > kMaxSmem - kSmemSlack) continue;
    for (int pipes = kConvPipes; pipes >= 1; pipes >>= 1) {
      if (4 * Ng > kTmemCols / pipes) continue;   // four slots: three live, one being drained
      const int stages = (int)std::min<size_t>(kConvMaxStages, (kMaxSmem - kSmemSlack - wb) / (pipes * (size_t)kConvStageBytes));
      if (stages < (pipes == 1 ? 4 : 3)) continue;
      const int workers = std::max(1, sms / (N / Ng));
      for (int nch = 1; nch <= std::min(D, 16); ++nch) {
        const int nd = (D + nch - 1) / nch;
        const long units = (long)B * ntiles * ((D + nd - 1) / nd);
        const long share = (units + workers - 1) / workers;
        const double mma = conv_mma_cycles(3 * Ng, (int)std::min<long>(pipes, share));
        const double c = share * (conv_planes(D, nd) * (Cin / 16) * 9 * mma + 300);
        if (!best.Ng || c < best.cost) best = ConvPlan{Ng, pipes, stages, nd, c};
      }
    }
  }
  return best;
}

template <int PIPES, bool HEAD> int conv3_launch_t(const ConvArgs& a, int ctas, cudaStream_t st) {
  // all of the SM's tensor memory is one CTA's: ask for more than half of its shared memory
  const size_t smem = std::max(conv_weight_bytes(a.Cin, a.Ng) + (size_t)PIPES * a.stages * kConvStageBytes, (size_t)120 * 1024);
  FR3D_TRY(smem_optin(reinterpret_cast<const void*>(k_conv3<PIPES, HEAD>), smem));
  return launch_on(true, k_conv3<PIPES, HEAD>, ctas, PIPES * kPipeThreads, smem, st, a);
}

}  // namespace

int conv_tiles(int q_first, int q_last) { return (q_last - q_first + 128) / 128; }

int conv_group(int Cin, int N, int D, int ntiles, int B) {
  int sms = 0;
  if (sm_count(&sms) != FR3D_OK) return 0;
  return conv_plan(Cin, N, D, ntiles, B, 0, sms).Ng;
}

int conv3_launch(const ConvArgs& args, cudaStream_t st) {
  ConvArgs a = args;
  if (a.Cin % 16 || a.Ng % 16 || a.Ng < 16 || a.Ng > 64 || a.N % a.Ng) return FR3D_ERR_UNSUPPORTED_SIZE;
  if (a.mode == kConvHead && (a.N != 16 || !a.hx || !a.hw)) return FR3D_ERR_UNSUPPORTED_SIZE;
  int sms = 0;
  FR3D_TRY(sm_count(&sms));
  const ConvPlan p = conv_plan(a.Cin, a.N, a.D, a.ntiles, a.B, a.Ng, sms);
  if (!p.Ng) return FR3D_ERR_UNSUPPORTED_SIZE;
  a.ngroups = a.N / a.Ng;
  a.nd = p.nd;
  a.nchunks = (a.D + a.nd - 1) / a.nd;
  a.stages = p.stages;
  a.slog = 0;
  while ((2 << a.slog) * a.Ng <= kTmemCols / p.pipes) ++a.slog;   // slots of a pipe's ring: a power of two
  const long units = (long)a.B * a.ntiles * a.nchunks;
  const long ctas = std::max<long>(1, std::min<long>(units, sms / a.ngroups));
  const int nc = (int)ctas * a.ngroups;
  const bool head = a.mode == kConvHead;
  switch (p.pipes) {
    case 4: return head ? conv3_launch_t<4, true>(a, nc, st) : conv3_launch_t<4, false>(a, nc, st);
    case 2: return head ? conv3_launch_t<2, true>(a, nc, st) : conv3_launch_t<2, false>(a, nc, st);
    default: return head ? conv3_launch_t<1, true>(a, nc, st) : conv3_launch_t<1, false>(a, nc, st);
  }
}

// Channel groups and units of a layer's weight gradient for batches up to B (fills Og .. nchunks, slots).
// A unit's accumulators see at most kWgChain voxels, as many as one FP32 chain of the partial sums may have.
int wgrad_plan(WgradArgs* a, int B) {
  if (a->Cin % kWgCg || a->Cout % 16) return FR3D_ERR_UNSUPPORTED_SIZE;
  a->Og = a->Cout % 32 == 0 ? 32 : 16;
  a->n_og = a->Cout / a->Og;
  a->n_cg = a->Cin / kWgCg;
  a->nd = std::min(a->D, kWgChain / kWgVox);
  a->nchunks = (a->D + a->nd - 1) / a->nd;
  a->nd = (a->D + a->nchunks - 1) / a->nchunks;
  const size_t room = 112 * 1024 - kSmemSlack;   // two CTAs per SM, which also share the tensor memory
  // about half of the room for each ring: the input ring holds two more planes than the steps in flight
  const int gplane = 3 * a->Og / 8 * kWgPlane, xplane = kWgX * kWgPlane;
  a->gslots = std::min<int>(kWgMaxSlots - 3, (int)((room - 3 * xplane) / (gplane + xplane)));
  a->slots = std::min<int>(kWgMaxSlots, (int)((room - (size_t)a->gslots * gplane) / xplane));
  int sms = 0;
  FR3D_TRY(sm_count(&sms));
  const int slots = 2 * sms;
  const int len = a->q_last - a->q_first + 1, npairs = a->n_og * a->n_cg;
  double bc = 0;
  a->span = 0;
  for (int span = kWgVox; span * a->nd <= std::max(kWgChain, kWgVox * a->nd) && span < len + kWgVox; span += kWgVox) {
    const long units = (long)B * a->nchunks * ((len + span - 1) / span);
    const long rounds = (units * npairs + slots - 1) / slots;
    // steps of a unit (two CTAs share an SM) against the bytes of the partials (written and read once), in cycles
    const double c = (double)rounds * ((span / kWgVox) * (a->nd + 2) * 12.5 * kWgVox + 4000) +
                     (double)units * npairs * 3 * a->Og * kWgCols * 8 / 2500.0;
    if (!a->span || c < bc) {
      a->span = span;
      bc = c;
    }
  }
  a->nspans = (len + a->span - 1) / a->span;
  return FR3D_OK;
}

size_t wgrad_partial_floats(const WgradArgs& a, int B) {
  return (size_t)B * a.nspans * a.nchunks * ((size_t)a.n_og * a.n_cg * 3 * a.Og * kWgCols + a.Cout);
}

int wgrad3_launch(const WgradArgs& args, int ci, float* dW, float* db, cudaStream_t st) {
  WgradArgs a = args;
  const size_t smem = ((size_t)a.gslots * (3 * a.Og / 8) + (size_t)a.slots * kWgX) * kWgPlane;
  FR3D_TRY(smem_optin(reinterpret_cast<const void*>(k_wgrad3), smem));
  const int units = a.B * a.nspans * a.nchunks, npairs = a.n_og * a.n_cg;
  const int total = npairs * 3 * a.Og * kWgCols;
  a.bias_partials = a.partials + (size_t)units * total;
  FR3D_TRY(launch_on(true, k_wgrad3, units * npairs, kWgThreads, smem, st, a));
  // threads per element: about eight units each, so that the loads of a layer with few elements fill the chip
  const int ry = units >= 512 ? 32 : (units >= 128 ? 16 : (units >= 32 ? 4 : 1)), rx = kWgRedThreads / ry;
  return launch_on(true, k_wgrad_reduce, (total + a.Cout + rx - 1) / rx, dim3(rx, ry), 0, st, a, units, ci, dW, db);
}

}  // namespace fr3d
