// HMC transition kernels (Section 2.1): momentum draw, leapfrog, energy,
// Metropolis-Hastings select and the dual-averaging update.
//
// Plain path (any target): one launch per operation per leapfrog step --
// begin (momentum + H_0), kick-drift, gradient, kick, ..., accept -- the
// shape a framework that evaluates a batched target op by op produces.
#include <cmath>

#include "hmc_device.cuh"
#include "hmc_internal.h"

namespace hmc {

unsigned accept_blocks(int C) { return static_cast<unsigned>((C + 7) / 8); }

namespace {

constexpr int kWarpsPerBlock = 8;

__device__ __forceinline__ void finish_block(const StepArgs& a, float prob, bool has_chain) {
  accept_block_finish<kWarpsPerBlock>(a.da, a.partials, prob, has_chain, a.C, a.t_full);
}

// ------------------------------------------------------------ plain path --
// p ~ N(0, I); xp = x; gp = g; h0 = -lp + |p|^2/2   (warp per chain)
__global__ void k_plain_begin(StepArgs a, PlainBuffers b) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= a.C) return;
  const int D = a.D;
  const int64_t row = static_cast<int64_t>(c) * D;
  const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
  float kin = 0.f;
  for (int j = lane; 4 * j < D; j += 32) {
    const float4 z = momentum4(a.seed, static_cast<uint32_t>(j), chain, a.t);
    const float zz[4] = {z.x, z.y, z.z, z.w};
    for (int i = 0; i < 4 && 4 * j + i < D; ++i) {
      const int64_t e = row + 4 * j + i;
      b.p[e] = zz[i];
      b.xp[e] = a.x[e];
      b.gp[e] = a.g[e];
      kin = fmaf(zz[i], zz[i], kin);
    }
  }
  kin = warp_sum(kin);
  if (lane == 0) b.h0[c] = -a.lp[c] + 0.5f * kin;
}

// p += eps/2 gp; xp += eps p
__global__ void k_plain_kick_drift(int64_t n, float* __restrict__ p, const float* __restrict__ gp,
                                   float* __restrict__ xp, const DAState* __restrict__ da) {
  const float eps = da->eps;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const float pi = fmaf(0.5f * eps, gp[i], p[i]);
    p[i] = pi;
    xp[i] = fmaf(eps, pi, xp[i]);
  }
}

// p += eps/2 gp
__global__ void k_plain_kick(int64_t n, float* __restrict__ p, const float* __restrict__ gp,
                             const DAState* __restrict__ da) {
  const float eps = da->eps;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    p[i] = fmaf(0.5f * eps, gp[i], p[i]);
}

// The fused implementations' form of the same steps (dense Gaussians whose rows
// the tensor maps cannot take): the elementwise steps between two gradients in
// one launch, each operation rounded as in the launches above.
// p ~ N(0, I), h0, then the first half kick (with the cached gradient) and drift
__global__ void k_merged_begin(StepArgs a, PlainBuffers b) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= a.C) return;
  const int D = a.D;
  const int64_t row = static_cast<int64_t>(c) * D;
  const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
  const float eps = a.da->eps;
  float kin = 0.f;
  for (int j = lane; 4 * j < D; j += 32) {
    const float4 z = momentum4(a.seed, static_cast<uint32_t>(j), chain, a.t);
    const float zz[4] = {z.x, z.y, z.z, z.w};
    for (int i = 0; i < 4 && 4 * j + i < D; ++i) {
      const int64_t e = row + 4 * j + i;
      kin = fmaf(zz[i], zz[i], kin);
      const float p = fmaf(0.5f * eps, a.g[e], zz[i]);
      b.p[e] = p;
      b.xp[e] = fmaf(eps, p, a.x[e]);
    }
  }
  kin = warp_sum(kin);
  if (lane == 0) b.h0[c] = -a.lp[c] + 0.5f * kin;
}

// two half kicks with the same gradient, then a drift
__global__ void k_merged_step(int64_t n, float* __restrict__ p, const float* __restrict__ gp,
                              float* __restrict__ xp, const DAState* __restrict__ da) {
  const float eps = da->eps, h = 0.5f * eps;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  auto step = [&](float g, float& pi, float& xi) {
    pi = fmaf(h, g, fmaf(h, g, pi));
    xi = fmaf(eps, pi, xi);
  };
  // (the buffers are the context's own: aligned)
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; 4 * i < n; i += stride) {
    if (4 * i + 4 <= n) {
      const float4 g = reinterpret_cast<const float4*>(gp)[i];
      float4 q = reinterpret_cast<float4*>(p)[i], x = reinterpret_cast<float4*>(xp)[i];
      step(g.x, q.x, x.x);
      step(g.y, q.y, x.y);
      step(g.z, q.z, x.z);
      step(g.w, q.w, x.w);
      reinterpret_cast<float4*>(p)[i] = q;
      reinterpret_cast<float4*>(xp)[i] = x;
    } else {
      for (int64_t k = 4 * i; k < n; ++k) step(gp[k], p[k], xp[k]);
    }
  }
}

// Random-walk proposal (Section 4.1's composition with a symmetric inner
// kernel): xp = x + eps z with z the transition's momentum draws; without a
// momentum the energies below reduce to log alpha = log p(xp) - log p(x).
__global__ void k_rw_begin(StepArgs a, PlainBuffers b, bool vec) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= a.C) return;
  const int D = a.D;
  const int64_t row = static_cast<int64_t>(c) * D;
  const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
  const float eps = a.da->eps;
  for (int j = lane; 4 * j < D; j += 32) {
    const int64_t e = row + 4 * j;
    if (vec) {
      const float4 x = *reinterpret_cast<const float4*>(a.x + e);
      const float4 z = momentum4(a.seed, static_cast<uint32_t>(j), chain, a.t);
      *reinterpret_cast<float4*>(b.xp + e) =
          make_float4(fmaf(eps, z.x, x.x), fmaf(eps, z.y, x.y), fmaf(eps, z.z, x.z), fmaf(eps, z.w, x.w));
    } else {
      const float4 z = momentum4(a.seed, static_cast<uint32_t>(j), chain, a.t);
      const float zz[4] = {z.x, z.y, z.z, z.w};
      for (int i = 0; i < 4 && 4 * j + i < D; ++i) b.xp[e + i] = fmaf(eps, zz[i], a.x[e + i]);
    }
  }
  if (lane == 0) b.h0[c] = -a.lp[c];
}

// log alpha = H_0 - H_L of chain c (warp per chain; every lane gets it).  The
// dense Gaussian's log p = <xp, gp> / 2 is formed here (a launch of its own
// would read both rows once more).
__device__ __forceinline__ float plain_log_alpha(const StepArgs& a, const PlainBuffers& b, int c,
                                                 int lane) {
  const int D = a.D;
  const int64_t row = static_cast<int64_t>(c) * D;
  float lpp;
  if (b.half_dot) {
    float s = 0.f;
#pragma unroll 4
    for (int d = lane; d < D; d += 32) s = fmaf(b.xp[row + d], b.gp[row + d], s);
    lpp = 0.5f * warp_sum(s);
    if (lane == 0) b.lpp[c] = lpp;
  } else {
    lpp = b.lpp[c];
  }
  float kin = 0.f;
  if (a.proposal != HMC_PROPOSAL_RANDOM_WALK) {
    const float h = 0.5f * a.da->eps;
#pragma unroll 4
    for (int d = lane; d < D; d += 32) {
      float p = b.p[row + d];
      if (a.merged) p = fmaf(h, b.gp[row + d], p);      // the trajectory's last half kick
      kin = fmaf(p, p, kin);
    }
    kin = 0.5f * warp_sum(kin);
  }
  const float h1 = -lpp + kin;
  float la = b.h0[c] - h1;
  if (!isfinite(la)) la = -INFINITY;
  return la;
}

// Metropolis-Hastings select of chain c given log alpha; returns min(1, alpha)
__device__ __forceinline__ float plain_select(const StepArgs& a, const PlainBuffers& b, int c, int lane,
                                              float la) {
  const int D = a.D;
  const int64_t row = static_cast<int64_t>(c) * D;
  const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
  int acc = 0;
  if (lane == 0) acc = accept_log_uniform(a.seed, chain, a.t) < la;
  acc = __shfl_sync(0xffffffffu, acc, 0);
#pragma unroll 4
  for (int d = lane; d < D; d += 32) {
    float x;
    if (acc) {
      x = b.xp[row + d];
      a.x[row + d] = x;
      a.g[row + d] = b.gp[row + d];
    } else if (a.sample_out) {
      x = a.x[row + d];
    }
    if (a.sample_out) a.sample_out[row + d] = x;
  }
  if (lane == 0) {
    if (acc) a.lp[c] = b.lpp[c];
    a.is_accepted[c] = static_cast<uint8_t>(acc);
    a.log_accept[c] = la;
    if (a.trace_acc) a.trace_acc[c] = static_cast<uint8_t>(acc);
    if (c == 0 && a.trace_eps) a.trace_eps[0] = a.da->eps;
  }
  return accept_prob(la);
}

// H_L, log alpha, Metropolis-Hastings select, traces, dual averaging
__global__ void k_plain_accept(StepArgs a, PlainBuffers b) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool has_chain = c < a.C;
  float prob = 0.f;
  if (has_chain) prob = plain_select(a, b, c, lane, plain_log_alpha(a, b, c, lane));
  finish_block(a, prob, has_chain);
}

// the split: log alpha only ...
__global__ void k_plain_ratio(StepArgs a, PlainBuffers b) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= a.C) return;
  const float la = plain_log_alpha(a, b, c, lane);
  if (lane == 0) b.la[c] = la;
}

// ... then the select from it
__global__ void k_plain_select(StepArgs a, PlainBuffers b) {
  const int c = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool has_chain = c < a.C;
  float prob = 0.f;
  if (has_chain) prob = plain_select(a, b, c, lane, b.la[c]);
  finish_block(a, prob, has_chain);
}

__global__ void k_da_init(DAState* da, float eps0, int adapt, float delta, long long num_adapt) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  da->log_eps = log(static_cast<double>(eps0));
  da->log_eps_bar = 0.0;
  da->h_bar = 0.0;
  da->mu = log(10.0 * static_cast<double>(eps0));
  da->delta = static_cast<double>(delta);
  da->last_stat = 0.0;
  da->m = 0;
  da->num_adapt = num_adapt;
  da->eps = eps0;
  da->adapt = adapt;
  da->arrive = 0u;
}

__global__ void k_philox_words(const uint32_t* __restrict__ ctr, int64_t n, uint64_t seed,
                               uint32_t* __restrict__ out) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 w = philox(c, static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
    out[4 * i] = w.x;
    out[4 * i + 1] = w.y;
    out[4 * i + 2] = w.z;
    out[4 * i + 3] = w.w;
  }
}

// one thread per (chain, Philox block)
__global__ void k_momentum(uint64_t seed, uint32_t t, int C, int D, uint32_t chain_offset,
                           float* __restrict__ out) {
  const int nblk = (D + 3) / 4;
  const int64_t total = static_cast<int64_t>(C) * nblk;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int c = static_cast<int>(i / nblk), j = static_cast<int>(i % nblk);
    const float4 z = momentum4(seed, static_cast<uint32_t>(j), static_cast<uint32_t>(c) + chain_offset, t);
    const float zz[4] = {z.x, z.y, z.z, z.w};
    for (int k = 0; k < 4 && 4 * j + k < D; ++k) out[static_cast<int64_t>(c) * D + 4 * j + k] = zz[k];
  }
}


inline unsigned elementwise_blocks(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return static_cast<unsigned>(std::min<int64_t>(b, 152 * 16));
}

}  // namespace

// whether log p of the proposal is left to plain_log_alpha
static bool plain_half_dot(const hmc_target& t, const StepArgs& a) {
  return t.id == HMC_T_CORR_GAUSS && a.K == 1;
}

// the proposal: leapfrog trajectory (HMC; MALA at L = 1) or random walk
static cudaError_t plain_proposal(const hmc_target& t, const StepArgs& a, const PlainBuffers& b,
                                  void* grad_ws, cudaStream_t s, KernelTimer* timer) {
  const int64_t n = static_cast<int64_t>(a.C) * a.D;
  auto gradient = [&](bool end) {
    // (a trajectory's middle needs no log p)
    const bool lp = end ? !plain_half_dot(t, a) : a.K > 1 || (t.id != HMC_T_CORR_GAUSS && t.id != HMC_T_LOGREG);
    cudaError_t e = launch_grad(t, a.C, b.xp, lp ? b.lpp : nullptr, b.gp, grad_ws, s, timer);
    if (e == cudaSuccess && a.K > 1) e = launch_temper(a.C, a.D, b.lpp, b.gp, a.betas, a.K, s);
    return e;
  };
  if (a.proposal == HMC_PROPOSAL_RANDOM_WALK) {
    const bool vec = a.D % 4 == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0;
    k_rw_begin<<<accept_blocks(a.C), 256, 0, s>>>(a, b, vec);
    count_launch();
    return gradient(true);
  }
  if (a.merged) {
    k_merged_begin<<<accept_blocks(a.C), 256, 0, s>>>(a, b);
    count_launch();
    for (int l = 0; l < a.L; ++l) {
      if (l > 0) {
        k_merged_step<<<elementwise_blocks((n + 3) / 4), 256, 0, s>>>(n, b.p, b.gp, b.xp, a.da);
        count_launch();
      }
      const cudaError_t e = gradient(l == a.L - 1);
      if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
  }
  k_plain_begin<<<accept_blocks(a.C), 256, 0, s>>>(a, b);
  count_launch();
  for (int l = 0; l < a.L; ++l) {
    k_plain_kick_drift<<<elementwise_blocks(n), 256, 0, s>>>(n, b.p, b.gp, b.xp, a.da);
    count_launch();
    const cudaError_t e = gradient(l == a.L - 1);
    if (e != cudaSuccess) return e;
    k_plain_kick<<<elementwise_blocks(n), 256, 0, s>>>(n, b.p, b.gp, a.da);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t launch_plain_transition(const hmc_target& t, const StepArgs& a, const PlainBuffers& bufs,
                                    void* grad_ws, cudaStream_t s, KernelTimer* timer) {
  PlainBuffers b = bufs;
  b.half_dot = plain_half_dot(t, a);
  cudaError_t e = plain_proposal(t, a, b, grad_ws, s, timer);
  if (e != cudaSuccess) return e;
  k_plain_accept<<<accept_blocks(a.C), 256, 0, s>>>(a, b);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_plain_propose(const hmc_target& t, const StepArgs& a, const PlainBuffers& bufs,
                                 void* grad_ws, cudaStream_t s) {
  PlainBuffers b = bufs;
  b.half_dot = plain_half_dot(t, a);
  cudaError_t e = plain_proposal(t, a, b, grad_ws, s, nullptr);
  if (e != cudaSuccess) return e;
  k_plain_ratio<<<accept_blocks(a.C), 256, 0, s>>>(a, b);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_plain_select(const StepArgs& a, const PlainBuffers& b, cudaStream_t s) {
  k_plain_select<<<accept_blocks(a.C), 256, 0, s>>>(a, b);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, int64_t n, uint64_t seed, uint32_t* out,
                          cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_philox_words<<<elementwise_blocks(n), 256, 0, s>>>(ctr, n, seed, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_momentum(uint64_t seed, uint32_t t, int C, int D, uint32_t chain_offset,
                            float* out, cudaStream_t s) {
  k_momentum<<<elementwise_blocks(static_cast<int64_t>(C) * ((D + 3) / 4)), 256, 0, s>>>(
      seed, t, C, D, chain_offset, out);
  count_launch();
  return cudaGetLastError();
}

// The streaming driver's moment update after kept draw k, one element per
// thread (welford_update).
__global__ void k_welford(int64_t n, const float* __restrict__ x, int64_t k, WelfordOut w) {
  const WelfordCoef q = welford_coef(k, w.bsize);
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    welford_update(w, q, k, i, x[i]);
}

cudaError_t launch_welford(int64_t n, const float* x, int64_t k, float* mean, float* m2,
                           int64_t bsize, float* bsum, float* bmean, float* bm2, cudaStream_t s) {
  k_welford<<<static_cast<unsigned>(std::min<int64_t>((n + 255) / 256, 152 * 16)), 256, 0, s>>>(
      n, x, k, WelfordOut{mean, m2, bsize, bsum, bmean, bm2});
  count_launch();
  return cudaGetLastError();
}

// Replicated batch-means effective sample size per dimension: the C nb
// batch means pooled about their grand mean (per chain, bmean / bm2 are the
// Welford mean and sum of squared deviations of its nb batch means), so
// SS = sum_c [bm2_c + nb (bmean_c - grand)^2] with grand = mean_c bmean_c,
// and ess[d] = C K (sum_c m2_c / (C (K - 1))) / (bsize SS / (C nb - 1)).  A
// block covers 8 dimensions (a 32-byte sector of each row) with 8 threads each
// striding over chains in two passes (grand mean, then sums); float64, whose
// units are few: 32 dimensions a block left 100 dimensions on 4 SMs
// (1000 chains: 133 -> 88 us).
constexpr int kBmDims = 8;
__global__ void __launch_bounds__(8 * kBmDims) k_bm_ess(int64_t C, int D, int64_t K, int64_t bsize,
                                                        const float* __restrict__ m2,
                                                        const float* __restrict__ bmean,
                                                        const float* __restrict__ bm2, float* __restrict__ ess) {
  __shared__ double a_s[8][kBmDims], b_s[8][kBmDims];
  __shared__ double grand_s[kBmDims];
  const int d = blockIdx.x * kBmDims + threadIdx.x;
  const double nb = static_cast<double>(K / bsize);
  double sb = 0.0;
  if (d < D) {
#pragma unroll 8
    for (int64_t c = threadIdx.y; c < C; c += 8) sb += static_cast<double>(bmean[c * D + d]);
  }
  a_s[threadIdx.y][threadIdx.x] = sb;
  __syncthreads();
  if (threadIdx.y == 0) {
    for (int y = 1; y < 8; ++y) sb += a_s[y][threadIdx.x];
    grand_s[threadIdx.x] = sb / static_cast<double>(C);
  }
  __syncthreads();
  const double grand = grand_s[threadIdx.x];
  double w = 0.0, ss = 0.0;
  if (d < D) {
#pragma unroll 8
    for (int64_t c = threadIdx.y; c < C; c += 8) {
      const double dev = static_cast<double>(bmean[c * D + d]) - grand;
      w += static_cast<double>(m2[c * D + d]);
      ss += static_cast<double>(bm2[c * D + d]) + nb * dev * dev;
    }
  }
  __syncthreads();
  a_s[threadIdx.y][threadIdx.x] = w;
  b_s[threadIdx.y][threadIdx.x] = ss;
  __syncthreads();
  if (threadIdx.y == 0 && d < D) {
    for (int y = 1; y < 8; ++y) {
      w += a_s[y][threadIdx.x];
      ss += b_s[y][threadIdx.x];
    }
    const double Cd = static_cast<double>(C), Kd = static_cast<double>(K);
    const double W = w / (Cd * (Kd - 1.0));
    const double sig2 = static_cast<double>(bsize) * ss / (Cd * nb - 1.0);
    ess[d] = static_cast<float>(Cd * Kd * W / sig2);
  }
}

cudaError_t launch_bm_ess(int64_t C, int D, int64_t K, int64_t bsize, const float* m2, const float* bmean,
                          const float* bm2, float* ess, cudaStream_t s) {
  k_bm_ess<<<static_cast<unsigned>((D + kBmDims - 1) / kBmDims), dim3(kBmDims, 8), 0, s>>>(C, D, K, bsize, m2,
                                                                                           bmean, bm2, ess);
  count_launch();
  return cudaGetLastError();
}

__global__ void k_temper(int64_t rows, int D, float* __restrict__ lp, float* __restrict__ g,
                         const float* __restrict__ betas, int K) {
  const int64_t n = rows * D;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t r = i / D;
    const float beta = betas[r % K];
    g[i] *= beta;
    if (i % D == 0) lp[r] *= beta;
  }
}

cudaError_t launch_temper(int64_t rows, int D, float* lp, float* g, const float* betas, int K,
                          cudaStream_t s) {
  const int64_t n = rows * D;
  k_temper<<<static_cast<unsigned>(std::min<int64_t>((n + 255) / 256, 152 * 16)), 256, 0, s>>>(
      rows, D, lp, g, betas, K);
  count_launch();
  return cudaGetLastError();
}

// Replica exchange (Section 2.2): for chain c and pair (k, k+1), k = t % 2,
// t % 2 + 2, ..., swap the two replicas' states iff
// log u < (beta_k - beta_{k+1}) (log p(x_{k+1}) - log p(x_k)), with u drawn from
// the counter generator at (k, c, t, tag 2).  Cached log p and gradient are
// tempered: the untempered values are lp / beta and g / beta.  Warp per pair.
__global__ void k_remc_swap(int64_t chains, int K, int D, float* __restrict__ x,
                            float* __restrict__ lp, float* __restrict__ g,
                            const float* __restrict__ betas, uint64_t seed, uint32_t t,
                            uint8_t* __restrict__ swapped) {
  const int npairs = K - 1;
  const int64_t w = blockIdx.x * static_cast<int64_t>(kWarpsPerBlock) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= chains * npairs) return;
  const int64_t c = w / npairs;
  const int k = static_cast<int>(w % npairs);
  if ((k & 1) != static_cast<int>(t & 1u)) {
    if (lane == 0) swapped[w] = 0;
    return;
  }
  const int64_t r0 = c * K + k, r1 = r0 + 1;
  const float b0 = betas[k], b1 = betas[k + 1];
  float raw0, raw1;
  int sw = remc_swap_accept(lp[r0], lp[r1], b0, b1, seed, static_cast<uint32_t>(k), static_cast<uint32_t>(c),
                            t, &raw0, &raw1);
  sw = __shfl_sync(0xffffffffu, sw, 0);
  if (sw) {
    for (int d = lane; d < D; d += 32) {
      const int64_t e0 = r0 * D + d, e1 = r1 * D + d;
      const float xa = x[e0], xb = x[e1];
      x[e0] = xb;
      x[e1] = xa;
      const float ga = g[e0], gb = g[e1];
      g[e0] = gb / b1 * b0;
      g[e1] = ga / b0 * b1;
    }
    if (lane == 0) {
      lp[r0] = b0 * raw1;
      lp[r1] = b1 * raw0;
    }
  }
  if (lane == 0) swapped[w] = static_cast<uint8_t>(sw);
}

cudaError_t launch_remc_swap(int64_t chains, int K, int D, float* x, float* lp, float* g,
                             const float* betas, uint64_t seed, uint32_t t, uint8_t* swapped,
                             cudaStream_t s) {
  const int64_t warps = chains * (K - 1);
  k_remc_swap<<<static_cast<unsigned>((warps + kWarpsPerBlock - 1) / kWarpsPerBlock),
                32 * kWarpsPerBlock, 0, s>>>(chains, K, D, x, lp, g, betas, seed, t, swapped);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_da_init(DAState* da, float eps0, int adapt, float delta, long long num_adapt,
                           cudaStream_t s) {
  k_da_init<<<1, 32, 0, s>>>(da, eps0, adapt, delta, num_adapt);
  count_launch();
  return cudaGetLastError();
}

}  // namespace hmc
