// Batched target log-prob and gradient kernels ("list of vectors" evaluation,
// Section 2.1): every chain is one row, only the event axis is reduced, so a
// chain's result never depends on another chain's.
//
//   STD_NORMAL  lp = -|x|^2/2, g = -x                      (warp per chain)
//   FUNNEL      closed form with one row reduction          (warp per chain)
//   CORR_GAUSS  G = -X P as one C x D x D product, lp = <x, g>/2
//   LOGREG      Z = Theta X^T (C x N x D), R = y - sigmoid(Z) fused into the
//               product's epilogue with the per-tile sums of y z - softplus(z);
//               G = R X - Theta (C x D x N, split over N); lp from the partials.
//
// These are the general-purpose kernels: the plain sampler calls them once per
// leapfrog step and the public gradient entry point uses them directly.
#include <cmath>

#include "hmc_device.cuh"
#include "hmc_internal.h"

namespace hmc {

std::atomic<uint64_t> g_launches{0};

// SM count of the current device (the logistic regression's split-K and
// path decisions), queried once per device; 152, a GB300's count, when no
// device can be queried.
int current_sm_count() {
  static std::atomic<int> known[64];
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 152;
  }
  if (dev < 64 && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
    cudaGetLastError();
    return 152;
  }
  if (dev < 64) known[dev].store(sms, std::memory_order_relaxed);
  return sms;
}


namespace {

// ---------------------------------------------------------------- SIMT GEMM
// C = A B over k in [k_begin, k_end), float32, each output one chain of fused
// multiply-adds in the order of k (so the tile shape does not change a bit of
// it).  A tile is BM = 16 TM rows x 64 columns; 256 threads as 16 x 16: thread
// (ty, tx) owns the rows ty TM + i and four columns -- 4 tx + j, or tx + 16 j
// where B is transposed (the order k_logreg_residual's sums keep).
//
// What bounds it: the FP32 pipe, in which fma.rn.f32x2 takes two cycles and one
// issue slot for two rows of one column, next to the shared loads.  Both
// operands are kept by k in shared memory with a thread's rows and columns
// adjacent: TM / 4 + 1 128-bit loads per 4 TM multiply-adds.  Their 16-byte
// groups are XORed with k / 4, which spreads the transposing stores over all
// banks, and the next 32 k's are on their way from memory while these are used.
// Measured, against 64 x 64 x 16 tiles with scalar shared loads and one buffer:
// X P of 4096 chains, 512 dims 90 -> 50 us (43 TFLOP/s of the 75 that a loop of
// these instructions reaches alone); a logistic regression's gradient of 2048
// chains, 20000 rows, 128 dims 931 -> 583 us.  Keeping B twice in shared memory
// (no register copies, five loads per step instead of three) was slower, 711 us.
constexpr int kBN = 64, kBK = 32, kGemmThreads = 256;

// Products over at most 16 k's leave out the zeros that fill their only step: 400000
// chains, 8 dims 80.5 -> 70.2 us (64 x 64 x 16 tiles 74.3).
constexpr int kShortK = 16;

struct Gemm {          // operands of one product; B_NT: B is [N x K] (its transpose is used)
  const float* A;
  int64_t lda;
  const float* B;
  int64_t ldb;
  int M, N, k_begin, k_end;
  bool vec_a, vec_b;   // rows start on 16 bytes: float4 loads
};

// v = row[i .. i + 3], zeros from `end` on
__device__ __forceinline__ float4 load4(const float* row, int i, int end, bool vec) {
  if (vec && i + 4 <= end) return *reinterpret_cast<const float4*>(row + i);
  float4 v;
  v.x = i < end ? row[i] : 0.f;
  v.y = i + 1 < end ? row[i + 1] : 0.f;
  v.z = i + 2 < end ? row[i + 2] : 0.f;
  v.w = i + 3 < end ? row[i + 3] : 0.f;
  return v;
}

template <int TM>
struct GemmTile {
  static constexpr int BM = 16 * TM;
  static constexpr int QA = BM * kBK / 4 / kGemmThreads;         // float4 per thread and buffer
  static constexpr int QB = kBN * kBK / 4 / kGemmThreads;
  static_assert(BM % 32 == 0 && TM % 2 == 0, "whole swizzle groups, pairs of rows");
  float a[2][kBK][BM];
  float b[2][kBK][kBN];
};

// DEPTH: k's of a step that are multiplied (fewer than kBK: a product of one step)
template <bool B_NT, int TM, int DEPTH>
__device__ __forceinline__ void gemm_tile(const Gemm& g, int m0, int n0, GemmTile<TM>& s, float (&acc)[TM][4]) {
  using T = GemmTile<TM>;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  unsigned long long c[TM / 2][4];
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) c[i][j] = 0ull;
  float4 ra[T::QA], rb[T::QB];
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // rows of eight float4; a transposed B's rows n, n + 16, n + 32, n + 48 go
  // to one warp (they are adjacent in shared memory)
  const int kq = tid & 7, ar = tid >> 3, br = (ar & 3) * 16 + (ar >> 2);
  const int bk = tid >> 4, bn = 4 * tx;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < T::QA; ++q) {
      const int r = m0 + ar + 32 * q;
      ra[q] = r < g.M ? load4(g.A + static_cast<int64_t>(r) * g.lda, k0 + 4 * kq, g.k_end, g.vec_a) : zero;
    }
#pragma unroll
    for (int q = 0; q < T::QB; ++q) {
      if (B_NT) {
        const int r = n0 + br + 8 * q;
        rb[q] = r < g.N ? load4(g.B + static_cast<int64_t>(r) * g.ldb, k0 + 4 * kq, g.k_end, g.vec_b) : zero;
      } else {
        const int k = k0 + bk + 16 * q;
        rb[q] = k < g.k_end ? load4(g.B + static_cast<int64_t>(k) * g.ldb, n0 + bn, g.N, g.vec_b) : zero;
      }
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < T::QA; ++q) {
      const int r = (ar + 32 * q) ^ (4 * kq);
      s.a[buf][4 * kq][r] = ra[q].x;
      s.a[buf][4 * kq + 1][r] = ra[q].y;
      s.a[buf][4 * kq + 2][r] = ra[q].z;
      s.a[buf][4 * kq + 3][r] = ra[q].w;
    }
#pragma unroll
    for (int q = 0; q < T::QB; ++q) {
      if (B_NT) {
        const int n = br + 8 * q, at = (4 * (n & 15) + (n >> 4)) ^ (4 * kq);
        s.b[buf][4 * kq][at] = rb[q].x;
        s.b[buf][4 * kq + 1][at] = rb[q].y;
        s.b[buf][4 * kq + 2][at] = rb[q].z;
        s.b[buf][4 * kq + 3][at] = rb[q].w;
      } else {
        const int k = bk + 16 * q;
        *reinterpret_cast<float4*>(&s.b[buf][k][bn ^ (4 * (k >> 2))]) = rb[q];
      }
    }
  };
  fetch(g.k_begin);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = g.k_begin; k0 < g.k_end; k0 += kBK, buf ^= 1) {
    const bool more = k0 + kBK < g.k_end;
    if (more) fetch(k0 + kBK);
#pragma unroll
    for (int kk = 0; kk < DEPTH; ++kk) {
      const int u = kk >> 2;
      unsigned long long av[TM / 2];
      if (TM % 4 == 0) {
#pragma unroll
        for (int i = 0; i < TM; i += 4) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&s.a[buf][kk][(ty * TM + i) ^ (4 * u)]);
          av[i / 2] = v.x;
          av[(i / 2 + 1) % (TM / 2)] = v.y;
        }
      } else {
#pragma unroll
        for (int i = 0; i < TM; i += 2)
          av[i / 2] = *reinterpret_cast<const unsigned long long*>(&s.a[buf][kk][(ty * TM + i) ^ (4 * u)]);
      }
      const float4 bq = *reinterpret_cast<const float4*>(&s.b[buf][kk][(4 * tx) ^ (4 * u)]);
      const float bv[4] = {bq.x, bq.y, bq.z, bq.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        unsigned long long bb;
        asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(bv[j]));
#pragma unroll
        for (int i = 0; i < TM / 2; ++i) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c[i][j]) : "l"(av[i]), "l"(bb));
      }
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM / 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * i][j]), "=f"(acc[2 * i + 1][j]) : "l"(c[i][j]));
}

// a thread's four adjacent columns of row m (the untransposed products)
__device__ __forceinline__ void store_cols(float* row, int n, int N, bool vec, const float (&v)[4]) {
  if (vec && n + 4 <= N) {
    *reinterpret_cast<float4*>(row + n) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (n + j < N) row[n + j] = v[j];
  }
}

// G = -X P  (corr_gauss; P symmetric so B may be read either way).  w (may be
// null): rows scaled by w[c], the vector-Jacobian product.
template <int TM, int DEPTH>
__global__ void __launch_bounds__(kGemmThreads, TM == 8 ? 2 : 3)
k_corr_gauss_grad(Gemm q, const float* __restrict__ w, float* __restrict__ g, bool vec) {
  __shared__ __align__(16) GemmTile<TM> tile;
  float acc[TM][4];
  const int m0 = blockIdx.y * (16 * TM), n0 = blockIdx.x * kBN;
  gemm_tile<false, TM, DEPTH>(q, m0, n0, tile, acc);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    if (m >= q.M) continue;
    const float wm = w ? w[m] : 1.f;
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = w ? -acc[i][j] * wm : -acc[i][j];
    store_cols(g + static_cast<int64_t>(m) * q.N, n0 + 4 * tx, q.N, vec, v);
  }
}

// lp[c] = <x_c, g_c> / 2, warp per chain
__global__ void k_half_rowdot(int C, int D, const float* __restrict__ x,
                              const float* __restrict__ g, float* __restrict__ lp) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  const float* xr = x + static_cast<int64_t>(c) * D;
  const float* gr = g + static_cast<int64_t>(c) * D;
  float s = 0.f;
  for (int d = lane; d < D; d += 32) s = fmaf(xr[d], gr[d], s);
  s = warp_sum(s);
  if (lane == 0) lp[c] = 0.5f * s;
}

// Z = Theta X^T; R = y - sigmoid(Z); lp_part[c, tile] = sum over the tile's 64
// rows of X of (y z - softplus z), or no log p at all (LP = false).  The
// epilogue is a third of the kernel at 128 dims: sigmoid and softplus share
// their exponential, the sigmoid takes one division whatever the sign of z.
template <int TM, int DEPTH, bool LP>
__global__ void __launch_bounds__(kGemmThreads, TM == 8 ? 2 : 3)
k_logreg_residual(Gemm q, const float* __restrict__ y, float* __restrict__ R, float* __restrict__ lp_part) {
  __shared__ __align__(16) GemmTile<TM> tile;
  float acc[TM][4];
  const int m0 = blockIdx.y * (16 * TM), n0 = blockIdx.x * kBN;
  gemm_tile<true, TM, DEPTH>(q, m0, n0, tile, acc);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float yv[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int n = n0 + tx + 16 * j;
    yv[j] = n < q.N ? y[n] : 0.f;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    float part = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + 16 * j;
      if (m < q.M && n < q.N) {
        const float z = acc[i][j], e = expf(-fabsf(z));
        R[static_cast<int64_t>(m) * q.N + n] = yv[j] - (z >= 0.f ? 1.f : e) / (1.f + e);
        if (LP) part += yv[j] * z - (fmaxf(z, 0.f) + log1pf(e));
      }
    }
    if (LP) {
      // the 16 threads sharing ty are one half-warp: reduce across tx
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (tx == 0 && m < q.M) lp_part[static_cast<int64_t>(m) * gridDim.x + blockIdx.x] = part;
    }
  }
}

// Gpart[s] = R[:, chunk s] X[chunk s, :]
template <int TM>
__global__ void __launch_bounds__(kGemmThreads, TM == 8 ? 2 : 3)
k_logreg_grad_partial(Gemm q, int chunk, float* __restrict__ Gpart, bool vec) {
  __shared__ __align__(16) GemmTile<TM> tile;
  float acc[TM][4];
  const int m0 = blockIdx.y * (16 * TM), n0 = blockIdx.x * kBN;
  const int rows = q.k_end;
  q.k_begin = blockIdx.z * chunk;
  q.k_end = min(rows, q.k_begin + chunk);
  gemm_tile<false, TM, kBK>(q, m0, n0, tile, acc);
  float* out = Gpart + static_cast<int64_t>(blockIdx.z) * q.M * q.N;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    if (m < q.M) store_cols(out + static_cast<int64_t>(m) * q.N, n0 + 4 * tx, q.N, vec, acc[i]);
  }
}

// g = sum_s Gpart[s] - theta; lp = sum_tiles lp_part - |theta|^2/2 (warp per
// chain).  With w: g = w[c] times that; without lp: no log p.
__global__ void k_logreg_finalize(int C, int D, int splits, int ntiles, const float* __restrict__ th,
                                  const float* __restrict__ Gpart, const float* __restrict__ lp_part,
                                  const float* __restrict__ w, float* __restrict__ g, float* __restrict__ lp) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  const int64_t row = static_cast<int64_t>(c) * D;
  float sq = 0.f;
  for (int d = lane; d < D; d += 32) {
    const float t = th[row + d];
    float acc = 0.f;
    for (int s = 0; s < splits; ++s) acc += Gpart[static_cast<int64_t>(s) * C * D + row + d];
    g[row + d] = w ? (acc - t) * w[c] : acc - t;
    sq = fmaf(t, t, sq);
  }
  if (!lp) return;
  float part = 0.f;
  for (int k = lane; k < ntiles; k += 32) part += lp_part[static_cast<int64_t>(c) * ntiles + k];
  sq = warp_sum(sq);
  part = warp_sum(part);
  if (lane == 0) lp[c] = part - 0.5f * sq;
}

__global__ void k_std_normal_grad(int C, int D, const float* __restrict__ x, float* __restrict__ lp,
                                  float* __restrict__ g) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  const int64_t row = static_cast<int64_t>(c) * D;
  float s = 0.f;
  for (int d = lane; d < D; d += 32) {
    const float v = x[row + d];
    g[row + d] = -v;
    s = fmaf(v, v, s);
  }
  s = warp_sum(s);
  if (lane == 0) lp[c] = -0.5f * s;
}

__global__ void k_funnel_grad(int C, int D, const float* __restrict__ x, float* __restrict__ lp,
                              float* __restrict__ g) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  const int64_t row = static_cast<int64_t>(c) * D;
  const float v = x[row];
  float q = 0.f;
  for (int d = 1 + lane; d < D; d += 32) q = fmaf(x[row + d], x[row + d], q);
  q = warp_sum(q);
  const float ev = expf(-v);
  const float half_n = 0.5f * static_cast<float>(D - 1);
  for (int d = 1 + lane; d < D; d += 32) g[row + d] = -ev * x[row + d];
  if (lane == 0) {
    g[row] = -v / 9.f - half_n + 0.5f * ev * q;
    lp[c] = -v * v / 18.f - half_n * v - 0.5f * ev * q;
  }
}

struct LogregPlan {
  int ntiles_n;   // 64-column blocks of the C x N residual product (one log p partial each)
  int splits;     // split of the N reduction in G = R X
  int chunk;      // rows of X per split (multiple of 16)
  size_t off_R, off_G, off_lp, bytes;
};

inline size_t align256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

LogregPlan logreg_plan(int64_t C, int D, int64_t N) {
  LogregPlan p{};
  p.ntiles_n = static_cast<int>((N + 63) / 64);
  const int64_t out_tiles = ((C + 63) / 64) * ((D + 63) / 64);
  int64_t s = (4 * static_cast<int64_t>(current_sm_count()) + out_tiles - 1) / out_tiles;
  s = std::max<int64_t>(1, std::min<int64_t>(s, (N + 511) / 512));
  int64_t chunk = (N + s - 1) / s;
  chunk = (chunk + 15) / 16 * 16;
  s = (N + chunk - 1) / chunk;
  p.splits = static_cast<int>(s);
  p.chunk = static_cast<int>(chunk);
  p.off_R = 0;
  p.off_G = align256(sizeof(float) * C * N);
  p.off_lp = p.off_G + align256(sizeof(float) * s * C * D);
  p.bytes = p.off_lp + align256(sizeof(float) * C * p.ntiles_n);
  return p;
}

inline unsigned warps_grid(int64_t C, int warps_per_block) {
  return static_cast<unsigned>((C + warps_per_block - 1) / warps_per_block);
}

// dx[c, :] = w[c] g[c, :], the vector-Jacobian product of log p from its
// gradient (dx may be g); warp per chain
__global__ void k_scale_rows(int C, int D, const float* __restrict__ w, const float* g, float* dx, bool vec) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  const int64_t row = static_cast<int64_t>(c) * D;
  const float wc = w[c];
  if (vec) {
    for (int d = 4 * lane; d < D; d += 128) {
      float4 v = *reinterpret_cast<const float4*>(g + row + d);
      v.x *= wc; v.y *= wc; v.z *= wc; v.w *= wc;
      *reinterpret_cast<float4*>(dx + row + d) = v;
    }
  } else {
    for (int d = lane; d < D; d += 32) dx[row + d] = g[row + d] * wc;
  }
}

// Rows of the tiles of an M x N product in `splits` parts, as TM: 8 (128 rows), 6
// or 4.  The larger tile loads less per multiply-add (128 rows against 64: 583
// against 661 us at 2048 x 20000 x 128, 214 against 260 us at 700 x 8000 x 301), the
// smaller one divides more evenly over the SMs (56 against 70 us at 64 x 20000 x
// 128); 96 rows make the 2048 x 128 x 20000 product in 10 splits 440 tiles, three an
// SM at most (583 -> 535 us for the whole gradient), and lose to 128 where those fill
// as many waves (29 against 21 us at 4096 x 256 x 256).
int tile_rows(int64_t M, int64_t N, int64_t splits) {
  const int64_t sms = current_sm_count();
  auto cost = [&](int tm, double rate) {
    const int64_t bm = 16 * tm, tiles = ((M + bm - 1) / bm) * ((N + kBN - 1) / kBN) * splits;
    return static_cast<double>((tiles + sms - 1) / sms * bm) / rate;
  };
  const double c8 = cost(8, 1.16), c6 = cost(6, 1.08), c4 = cost(4, 1.0);
  return c8 <= c6 && c8 <= c4 ? 8 : c6 < c4 ? 6 : 4;
}

dim3 gemm_grid(const Gemm& q, int tm, int splits = 1) {
  return dim3((q.N + kBN - 1) / kBN, (q.M + 16 * tm - 1) / (16 * tm), splits);
}

inline bool rows16(const float* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && ld % 4 == 0; }

void corr_gauss_product(int C, int D, const float* x, const float* P, const float* w, float* g, cudaStream_t s) {
  const Gemm q{x, D, P, D, C, D, 0, D, rows16(x, D), rows16(P, D)};
  const int tm = tile_rows(C, D, 1);
  const bool vec = rows16(g, D);
  auto k = D <= kShortK ? tm == 8   ? k_corr_gauss_grad<8, kShortK>
                          : tm == 6 ? k_corr_gauss_grad<6, kShortK>
                                    : k_corr_gauss_grad<4, kShortK>
           : tm == 8 ? k_corr_gauss_grad<8, kBK>
           : tm == 6 ? k_corr_gauss_grad<6, kBK>
                     : k_corr_gauss_grad<4, kBK>;
  k<<<gemm_grid(q, tm), kGemmThreads, 0, s>>>(q, w, g, vec);
}

template <bool LP>
void logreg_products(const hmc_target& t, int C, const float* x, const LogregPlan& p, float* R, float* Gp, float* lpp,
                     cudaStream_t s) {
  const int D = t.dim, N = static_cast<int>(t.n_data);
  const Gemm z{x, D, t.X, D, C, N, 0, D, rows16(x, D), rows16(t.X, D)};
  const int zm = tile_rows(C, N, 1);
  auto kz = D <= kShortK ? zm == 8   ? k_logreg_residual<8, kShortK, LP>
                           : zm == 6 ? k_logreg_residual<6, kShortK, LP>
                                     : k_logreg_residual<4, kShortK, LP>
            : zm == 8 ? k_logreg_residual<8, kBK, LP>
            : zm == 6 ? k_logreg_residual<6, kBK, LP>
                      : k_logreg_residual<4, kBK, LP>;
  kz<<<gemm_grid(z, zm), kGemmThreads, 0, s>>>(z, t.y, R, lpp);
  const Gemm r{R, N, t.X, D, C, D, 0, N, rows16(R, N), rows16(t.X, D)};
  const int gm = tile_rows(C, D, p.splits);
  auto kg = gm == 8 ? k_logreg_grad_partial<8> : gm == 6 ? k_logreg_grad_partial<6> : k_logreg_grad_partial<4>;
  kg<<<gemm_grid(r, gm, p.splits), kGemmThreads, 0, s>>>(r, p.chunk, Gp, D % 4 == 0);
}

}  // namespace

cudaError_t launch_vjp(const hmc_target& t, int64_t C64, const float* x, const float* w, float* dx,
                       float* lp_tmp, void* ws, cudaStream_t s) {
  const int C = static_cast<int>(C64), D = t.dim;
  if (t.id == HMC_T_CORR_GAUSS) {       // (the row weights in the products' epilogues, no log p)
    corr_gauss_product(C, D, x, t.P, w, dx, s);
    count_launch();
    return cudaGetLastError();
  }
  if (t.id == HMC_T_LOGREG) {
    const LogregPlan p = logreg_plan(C, D, t.n_data);
    char* base = static_cast<char*>(ws);
    float* Gp = reinterpret_cast<float*>(base + p.off_G);
    logreg_products<false>(t, C, x, p, reinterpret_cast<float*>(base + p.off_R), Gp, nullptr, s);
    k_logreg_finalize<<<warps_grid(C, 8), 256, 0, s>>>(C, D, p.splits, p.ntiles_n, x, Gp, nullptr, w, dx, nullptr);
    count_launch(3);
    return cudaGetLastError();
  }
  cudaError_t e = launch_grad(t, C, x, lp_tmp, dx, ws, s);
  if (e != cudaSuccess) return e;
  return launch_scale_rows(C, D, w, dx, dx, s);
}

cudaError_t launch_scale_rows(int64_t C, int D, const float* w, const float* g, float* dx, cudaStream_t s) {
  k_scale_rows<<<warps_grid(C, 8), 256, 0, s>>>(static_cast<int>(C), D, w, g, dx, rows16(g, D) && rows16(dx, D));
  count_launch();
  return cudaGetLastError();
}

size_t grad_workspace_bytes(const hmc_target& t, int64_t C) {
  if (t.id == HMC_T_LOGREG) return logreg_plan(C, t.dim, t.n_data).bytes;
  return 0;
}

cudaError_t launch_grad(const hmc_target& t, int64_t C64, const float* x, float* lp, float* g,
                        void* ws, cudaStream_t s, KernelTimer* timer) {
  const int C = static_cast<int>(C64), D = t.dim;
  switch (t.id) {
    case HMC_T_STD_NORMAL:
      k_std_normal_grad<<<warps_grid(C, 8), 256, 0, s>>>(C, D, x, lp, g);
      count_launch();
      break;
    case HMC_T_FUNNEL:
      k_funnel_grad<<<warps_grid(C, 8), 256, 0, s>>>(C, D, x, lp, g);
      count_launch();
      break;
    case HMC_T_CORR_GAUSS: {
      if (timer) timer->begin(s);
      corr_gauss_product(C, D, x, t.P, nullptr, g, s);
      if (timer) timer->end(s);
      count_launch();
      if (lp) {
        k_half_rowdot<<<warps_grid(C, 8), 256, 0, s>>>(C, D, x, g, lp);
        count_launch();
      }
      break;
    }
    case HMC_T_LOGREG: {
      const int N = static_cast<int>(t.n_data);
      const LogregPlan p = logreg_plan(C, D, N);
      char* base = static_cast<char*>(ws);
      float* R = reinterpret_cast<float*>(base + p.off_R);
      float* Gp = reinterpret_cast<float*>(base + p.off_G);
      float* lpp = reinterpret_cast<float*>(base + p.off_lp);
      if (timer) timer->begin(s);
      if (lp) logreg_products<true>(t, C, x, p, R, Gp, lpp, s);
      else logreg_products<false>(t, C, x, p, R, Gp, nullptr, s);
      if (timer) timer->end(s);
      k_logreg_finalize<<<warps_grid(C, 8), 256, 0, s>>>(C, D, p.splits, p.ntiles_n, x, Gp, lpp,
                                                         nullptr, g, lp);
      count_launch(3);
      break;
    }
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace hmc
