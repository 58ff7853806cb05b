// HMC chains of the targets whose gradient is elementwise plus row reductions
// (standard normal, funnel; Section 2.1): one launch runs a whole range of
// transitions with every chain's x, p and g in registers.
//
// Chains never talk to each other at a fixed step size, so such a range is an
// ordinary launch in which each warp runs its chains to the end; only the last
// transition reports its acceptance statistic.  While the step size adapts,
// every transition ends with the mean over all chains: the range is then a
// cooperative launch whose CTAs meet (waits bounded) after each
// transition and all apply the same dual-averaging update to a copy of the
// state.  The statistic is summed in the order of the 8-chain tiles that the
// batch's grouped launch (elementwise_tile.cuh) uses, so results do not depend
// on the launch form.
//
// What bounds it: not memory (a chain's state is read and written once per
// range, its kept samples written once) but the dependent instructions of a
// leapfrog step -- a shuffle butterfly and an exponential for the funnel -- and
// at many chains per scheduler their issue: 960 instructions per transition
// of a 100-dim chain and 10 leapfrog steps (scheduler busy 72 % at 4096
// chains), a third of them the draws.  One launch per transition paid for the
// launch, the state's round trip and a last block that finished the step-size
// update alone.  Measured, per transition: funnel, 100 dims, 10 steps, 4096
// chains 14.0 us -> 5.1 us (7.5 us while adapting), 100 chains 2.4 us (4.8);
// the 100 x 1 standard normal of 3 steps 6.0 us -> 0.33 us.  A launch of a single
// transition has nothing to carry: many chains of a whole warp take the tile
// kernel then (tiles_pay).
//
// Lanes: a chain takes G = 1..32 lanes (four dims each, NB blocks of 128 dims
// above 128); the butterfly over G lanes is the 32-lane one without its steps
// that add zeros, bit for bit.  A warp holds Q chains; its remaining
// A = 32 / (G Q) copies of them draw the momenta of A transitions at a time,
// and every lane one accept uniform of A G transitions: the draws depend on
// counters only, and for a one-dimensional chain they are most of a
// transition.
#include <algorithm>
#include <cmath>

#include "chain_sync.cuh"
#include "elementwise_tile.cuh"

namespace hmc {

namespace {

constexpr int kEwWarps = 8;

struct EwArgs {
  StepArgs s;            // s.t / s.t_full: the range's first transition
  int T;                 // transitions
  int lq;                // log2 of the chains per warp
  int nsets;             // groups of W << lq chains (W: warps per CTA)
  int vec;               // rows can be moved as float4
  long long keep_from;   // transition keep_from + k is kept draw k
  float* samples;
  float* trace_eps;
  uint8_t* trace_acc;
  unsigned* ctr;         // adapting launches: CTAs that left (0 between launches)
  int* err;
  unsigned long long* slots;   // adapting launches: [2][tiles] statistics (chain_sync.cuh)
  MeetingLimits lim;     // adapting launches: the meeting after transition i is meeting i + 1
};

template <int G>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of all tiles' slots once written, in the order of tile_partial_then_da
// (a whole warp); false after the time limit (never: nothing counts as written).
__device__ __forceinline__ bool slots_sum(const unsigned long long* slots, int ntiles, bool negative,
                                          unsigned long long wait_ns, bool never, double* sum) {
  const unsigned long long want = negative ? kSlotSign : 0ull;
  const int lane = threadIdx.x & 31;
  unsigned long long t0 = 0;
  double acc = 0.0;
  bool ok = true;
  for (int b0 = 0; b0 < ntiles && ok; b0 += 256) {
    unsigned long long w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = b0 + lane + 32 * i < ntiles ? want ^ kSlotSign : want;
    while (true) {
      // (only what is missing is read again)
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((w[i] & kSlotSign) != want) w[i] = read_slot(slots + b0 + lane + 32 * i);
      bool ready = !never;
#pragma unroll
      for (int i = 0; i < 8; ++i) ready = ready && (w[i] & kSlotSign) == want;
      if (__all_sync(0xffffffffu, ready)) break;
      const unsigned long long now = ptx::global_timer_ns();
      if (!t0) t0 = now;
      if (__any_sync(0xffffffffu, now - t0 > wait_ns)) {
        ok = false;
        break;
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += slot_value(w[i]);
  }
  *sum = warp_sum_d(acc);
  return ok;
}

// sum over all tiles in the order of tile_partial_then_da (warp 0); the loads
// of eight tiles are in flight together
__device__ __forceinline__ double tiles_sum(const double* partials, int ntiles) {
  double acc = 0.0;
  for (int b = threadIdx.x; b < ntiles; b += 256) {
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = b + 32 * i < ntiles ? __ldcg(partials + b + 32 * i) : 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += v[i];
  }
  return warp_sum_d(acc);
}

// v = s u + v and v = s u over a lane's N dims, two per instruction (each
// half rounds as the scalar instruction does)
template <int N>
__device__ __forceinline__ void axpy(float (&v)[N], float s, const float (&u)[N]) {
  if (N == 1) {
    v[0] = fmaf(s, u[0], v[0]);
  } else {
#pragma unroll
    for (int i = 0; i + 1 < N; i += 2)
      asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b64 c, {%0, %1};\n\t"
          "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
          : "+f"(v[i]), "+f"(v[i + 1])
          : "f"(s), "f"(u[i]), "f"(u[i + 1]));
  }
}

template <int N>
__device__ __forceinline__ void scale(float (&v)[N], float s, const float (&u)[N]) {
  if (N == 1) {
    v[0] = s * u[0];
  } else {
#pragma unroll
    for (int i = 0; i + 1 < N; i += 2)
      asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\t"
          "mul.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
          : "=f"(v[i]), "=f"(v[i + 1])
          : "f"(s), "f"(u[i]), "f"(u[i + 1]));
  }
}

// v / 9, correctly rounded for finite v away from the denormals (Markstein
// 1990: a quotient estimate from the rounded reciprocal, corrected by its
// exact remainder).  Used where half the dimension is subtracted next, which
// absorbs what a denormal quotient could differ by, and where a non-finite v
// rejects the transition either way.
__device__ __forceinline__ float div9(float v) {
  constexpr float y = 1.f / 9.f;
  const float q = v * y;
  return fmaf(fmaf(-9.f, q, v), y, q);
}

// 64 registers at NB = 1 (a few words spill): 32 warps per SM hold 4096 chains
// of up to 128 dims on 128 SMs, so that the adapting range keeps every chain
// in registers; past that a CTA's chains go through memory.  EL: dims per lane and block (1 for one-dimensional
// chains).  MODE: kFixed, kAdapt (cooperative), kTempered (fixed, replicas),
// kMoments (fixed, the streaming driver's running moments).
constexpr int kFixed = 0, kAdapt = 1, kTempered = 2, kMoments = 3;

template <int TARGET, int NB, int G, int EL, int MODE, int W = kEwWarps>
__global__ void __launch_bounds__(32 * W, W == 32 ? 1 : W == 16 ? 2 : NB == 1 ? 4 : NB == 2 ? 2 : 1) k_elementwise_chain(EwArgs e) {
  static_assert(NB == 1 || (G == 32 && EL == 4), "blocks past the first need the whole warp");
  constexpr bool COOP = MODE == kAdapt;
  __shared__ float prob_s[32 * W];
  __shared__ DAState da_s;
  __shared__ DACoef coef_s[32];
  __shared__ int flag_s;
  const StepArgs& a = e.s;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int Q = 1 << e.lq;
  const int j = lane & (G - 1);
  const int q = (lane / G) & (Q - 1);
  const int copy = (lane / G) >> e.lq;
  const int A = (32 / G) >> e.lq;
  const bool lead = j == 0 && copy == 0;
  const int D = a.D;
  const int64_t CD = static_cast<int64_t>(a.C) * D;
  const int ntiles = (a.C + 7) / 8;
  const bool resident = e.nsets <= static_cast<int>(gridDim.x);
  const float half_n = 0.5f * static_cast<float>(D - 1);
  if (threadIdx.x == 0) {
    flag_s = 0;
    if (COOP) da_s = *a.da;
  }
  if (COOP) __syncthreads();
  float eps = COOP ? da_s.eps : a.da->eps;
  const double n_c = static_cast<double>(a.C), inv_c = COOP ? 1.0 / n_c : 0.0;

  float x0[NB][EL], g0[NB][EL], z[EL], log_u = 0.f, lp0 = 0.f;
  bool stop = false;
  long long k = a.t_full - e.keep_from;
  for (int i = 0; i < e.T && !stop; ++i, ++k) {
    const uint32_t t = a.t + static_cast<uint32_t>(i);
    const bool last = i == e.T - 1;
    const bool keep = k >= 0;
    // (copies ahead of the current transition hold draws only while the warp
    // stays with its chains)
    const int ra = resident ? i & (A - 1) : 0, ru = resident ? i & (A * G - 1) : 0;
    // the float64 coefficients of the next 32 updates, a lane each (one at a
    // time they took 1.3 us of every adapting transition)
    if (COOP && warp == 0 && (i & 31) == 0) {
      __syncwarp();
      coef_s[lane] = da_prepare(&da_s, a.t_full + i + lane, lane);
      __syncwarp();
    }
    for (int set = blockIdx.x; set < e.nsets; set += gridDim.x) {
      const int slot = warp * Q + q;
      const int c = set * (W << e.lq) + slot;
      const bool has_chain = c < a.C;
      const int64_t row = static_cast<int64_t>(c) * D;
      const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
      if (!resident || i == 0) {
        lp0 = has_chain ? a.lp[c] : 0.f;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const int d0 = EL * (j + 32 * b);
          if (EL == 4 && e.vec) {
            float4 xv = make_float4(0.f, 0.f, 0.f, 0.f), gv = xv;
            if (has_chain && d0 < D) {
              xv = *reinterpret_cast<const float4*>(a.x + row + d0);
              gv = *reinterpret_cast<const float4*>(a.g + row + d0);
            }
            const float xx[4] = {xv.x, xv.y, xv.z, xv.w}, gg[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
            for (int u = 0; u < EL; ++u) {
              x0[b][u] = xx[u];
              g0[b][u] = gg[u];
            }
          } else {
#pragma unroll
            for (int u = 0; u < EL; ++u) {
              const bool in = has_chain && d0 + u < D;
              x0[b][u] = in ? a.x[row + d0 + u] : 0.f;
              g0[b][u] = in ? a.g[row + d0 + u] : 0.f;
            }
          }
        }
      }
      // momenta: copy `ra` of the chain drew this transition's
      float x[NB][EL], p[NB][EL], g[NB][EL];
      float kin0 = 0.f;
      auto draw_momenta = [&](uint32_t tt) {
        const float4 n = momentum4(a.seed, static_cast<uint32_t>(j), chain, tt + static_cast<uint32_t>(copy));
        const float nn[4] = {n.x, n.y, n.z, n.w};
#pragma unroll
        for (int u = 0; u < EL; ++u) z[u] = EL * j + u < D ? nn[u] : 0.f;
      };
      auto draw_uniforms = [&](uint32_t tt) {
        log_u = accept_log_uniform(a.seed, chain, tt + static_cast<uint32_t>(copy * G + j));
      };
      const bool ahead = COOP && resident && i > 0;    // drawn while the CTAs met
      if (NB == 1 && ra == 0 && !ahead) draw_momenta(t);
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if (NB == 1) {
          const int src = ((ra << e.lq) + q) * G + j;
#pragma unroll
          for (int u = 0; u < EL; ++u) p[b][u] = G == 32 ? z[u] : __shfl_sync(0xffffffffu, z[u], src);
        } else {
          const float4 n = momentum4(a.seed, static_cast<uint32_t>(j + 32 * b), chain, t);
          const float nn[4] = {n.x, n.y, n.z, n.w};
#pragma unroll
          for (int u = 0; u < EL; ++u) p[b][u] = EL * (j + 32 * b) + u < D ? nn[u] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < EL; ++u) {
          x[b][u] = x0[b][u];
          g[b][u] = g0[b][u];
          kin0 = fmaf(p[b][u], p[b][u], kin0);
        }
      }
      if (ru == 0 && !ahead) draw_uniforms(t);
      const float lu = __shfl_sync(0xffffffffu, log_u, (((ru / G) << e.lq) + q) * G + (ru & (G - 1)));
      kin0 = 0.5f * group_sum<G>(kin0);
      const float h = 0.5f * eps;
      float lp1 = 0.f;
      float beta = 1.f;       // replica exchange: this row targets p^beta
      if (MODE == kTempered) beta = a.betas[c % a.K];
      // drift, then the gradient there; with `end` also log p
      auto drift_grad = [&](bool end) {
        float qs = 0.f;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          axpy(x[b], eps, p[b]);
#pragma unroll
          for (int u = 0; u < EL; ++u) {
            // the funnel's reduction runs over x_1.. only (dim 0 is v)
            const float w = TARGET == HMC_T_FUNNEL && b == 0 && u == 0 && j == 0 ? 0.f : x[b][u];
            qs = fmaf(w, w, qs);
          }
        }
        if (TARGET == HMC_T_STD_NORMAL) {
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int u = 0; u < EL; ++u) g[b][u] = -x[b][u];
          if (end) lp1 = -0.5f * group_sum<G>(qs);
        } else {  // funnel: v is dim 0 (lane 0 of the chain, block 0, word 0)
          const float v = __shfl_sync(0xffffffffu, x[0][0], lane & ~(G - 1));
          const float ev = expf(-v);
          qs = group_sum<G>(qs);
#pragma unroll
          for (int b = 0; b < NB; ++b) scale(g[b], -ev, x[b]);
          const float gv = fmaf(0.5f * ev, qs, -div9(v) - half_n);
          g[0][0] = j == 0 ? gv : g[0][0];
          if (end) lp1 = fmaf(-0.5f * ev, qs, fmaf(-half_n, v, -v * v / 18.f));
        }
        if (MODE == kTempered) {
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int u = 0; u < EL; ++u) g[b][u] *= beta;
          if (end) lp1 *= beta;
        }
      };
      // dims past D keep x = p = g = 0 throughout (g = -x and -e^-v x vanish)
      auto half_kick = [&] {
#pragma unroll
        for (int b = 0; b < NB; ++b) axpy(p[b], h, g[b]);
      };
      half_kick();
      for (int l = 1; l < a.L; ++l) {
        drift_grad(false);
        half_kick();
        half_kick();
      }
      drift_grad(true);
      half_kick();
      float kin1 = 0.f;
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int u = 0; u < EL; ++u) kin1 = fmaf(p[b][u], p[b][u], kin1);
      kin1 = 0.5f * group_sum<G>(kin1);
      const float h0 = -lp0 + kin0, h1 = -lp1 + kin1;
      float la = h0 - h1;
      if (!isfinite(la)) la = -INFINITY;
      const bool acc = lu < la;
      if (acc) lp0 = lp1;
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int u = 0; u < EL; ++u) {
          x0[b][u] = acc ? x[b][u] : x0[b][u];
          g0[b][u] = acc ? g[b][u] : g0[b][u];
        }
      if (has_chain && copy == 0) {
        const bool put = !resident || last;
        if (keep) {
          float* sample = e.samples ? e.samples + k * CD + row : nullptr;
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            const int d0 = EL * (j + 32 * b);
            if (sample) {
              if (EL == 4 && e.vec) {
                if (d0 < D)
                  *reinterpret_cast<float4*>(sample + d0) =
                      make_float4(x0[b][0], x0[b][1 % EL], x0[b][2 % EL], x0[b][3 % EL]);
              } else {
#pragma unroll
                for (int u = 0; u < EL; ++u)
                  if (d0 + u < D) sample[d0 + u] = x0[b][u];
              }
            }
            if (MODE == kMoments) {      // the streaming driver's running moments
              int64_t idx[EL];
              uint32_t valid = 0u;
#pragma unroll
              for (int u = 0; u < EL; ++u) {
                idx[u] = row + d0 + u;
                if (d0 + u < D) valid |= 1u << u;
              }
              welford_update_n<EL>(a.w, welford_coef(k, a.w.bsize), k, idx, x0[b], valid);
            }
          }
          if (lead) {
            if (e.trace_acc) e.trace_acc[k * a.C + c] = static_cast<uint8_t>(acc);
            if (c == 0 && e.trace_eps) e.trace_eps[k] = eps;
          }
        }
        if (put) {
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int u = 0; u < EL; ++u) {
              const int d = EL * (j + 32 * b) + u;
              if (d < D) {
                a.x[row + d] = x0[b][u];
                a.g[row + d] = g0[b][u];
              }
            }
          if (lead) {
            a.lp[c] = lp0;
            a.is_accepted[c] = static_cast<uint8_t>(acc);
            a.log_accept[c] = la;
          }
        }
      }
      if (COOP || last) {
        // per 8-chain tile: the acceptance probabilities in chain order
        if (lead) prob_s[slot] = has_chain ? accept_prob(la) : 0.f;
        __syncthreads();
        const int tiles = (W / 8) << e.lq, tile = set * tiles + static_cast<int>(threadIdx.x);
        if (threadIdx.x < tiles && tile < ntiles) {
          double sum = 0.0;
          for (int w = 0; w < 8; ++w) sum += static_cast<double>(prob_s[8 * threadIdx.x + w]);
          if (COOP) put_slot(e.slots + (i & 1 ? ntiles : 0) + tile, sum, (i & 2) != 0);
          else a.partials[tile] = sum;
        }
        if (!resident) __syncthreads();      // prob_s is the next set's
        if (COOP && resident) {
          // the next transition's draws, while the statistics travel
          if (NB == 1 && ((i + 1) & (A - 1)) == 0) draw_momenta(t + 1);
          if (((i + 1) & (A * G - 1)) == 0) draw_uniforms(t + 1);
        }
      }
    }
    if (COOP) {
      // every tile's statistic, then the same update in every CTA
      if (warp == 0) {
        double sum;
        const bool ok = slots_sum(e.slots + (i & 1 ? ntiles : 0), ntiles, (i & 2) != 0, e.lim.wait_ns,
                                 i + 1 == e.lim.unreachable_gen, &sum);
        if (lane == 0) {
          if (ok) {
            da_apply_sum(&da_s, coef_s[i & 31], sum, n_c, inv_c, a.t_full + i);
          } else {
            atomicExch(e.err, 4);
            flag_s = 1;
          }
        }
      }
      __syncthreads();
      stop = flag_s != 0;
      eps = da_s.eps;
    }
  }
  if (COOP) {
    leave_adapting(a.da, &da_s, e.ctr, e.slots, 2 * ntiles);
  } else if (warp == 0) {
    // the last CTA to finish applies the last transition's statistic
    __syncwarp();
    unsigned mine = 0u;
    if (lane == 0) {
      __threadfence();
      mine = atomicAdd(&a.da->arrive, 1u) == gridDim.x - 1u ? 1u : 0u;
      __threadfence();
    }
    if (__shfl_sync(0xffffffffu, mine, 0)) {
      const double sum = tiles_sum(a.partials, ntiles);
      if (lane == 0) {
        da_update(a.da, sum / static_cast<double>(a.C), a.t_full + e.T - 1);
        a.da->arrive = 0u;
      }
    }
  }
}

cudaError_t launch_adapting(void (*kernel)(EwArgs), int threads, const EwArgs& e, int sms, cudaStream_t s) {
  int occ = 0;
  const cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, 0);
  if (err != cudaSuccess) return err;
  if (occ < 1) return cudaErrorLaunchOutOfResources;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(std::min(e.nsets, sms * occ)));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, e);
}

template <int TARGET, int NB, int G, int EL>
cudaError_t launch_range(EwArgs& e, bool adapting, int sms, cudaStream_t s) {
  if (e.s.w.mean) {
    k_elementwise_chain<TARGET, NB, G, EL, kMoments><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    return cudaGetLastError();
  }
  if (!adapting) {
    k_elementwise_chain<TARGET, NB, G, EL, kFixed><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    return cudaGetLastError();
  }
  // One CTA per SM while that holds all chains: every CTA polls every tile's
  // slot, so fewer, larger CTAs poll less (funnel, 100 dims, 4096 chains:
  // 11.7 us a transition with 512 CTAs of 8 warps, 8.8 us with 128 of 32; at
  // 1300 chains 41 CTAs of 32 warps took 7.3 us, 82 of 16 take 5.3 us).
  if (NB == 1 && e.nsets > 2 * sms) {
    e.nsets = (e.nsets + 3) / 4;
    return launch_adapting(k_elementwise_chain<TARGET, 1, G, EL, kAdapt, 32>, 1024, e, sms, s);
  }
  if (NB == 1 && e.nsets > sms) {
    e.nsets = (e.nsets + 1) / 2;
    return launch_adapting(k_elementwise_chain<TARGET, 1, G, EL, kAdapt, 16>, 512, e, sms, s);
  }
  return launch_adapting(k_elementwise_chain<TARGET, NB, G, EL, kAdapt>, 32 * kEwWarps, e, sms, s);
}

template <int TARGET>
cudaError_t launch_target(EwArgs& e, int G, bool adapting, int sms, cudaStream_t s) {
  const int nblk = (e.s.D + 3) / 4;
  if (e.s.K > 1) {         // one transition between two exchange steps
    if (nblk > 128) k_elementwise_chain<TARGET, 8, 32, 4, kTempered><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    else if (nblk > 64) k_elementwise_chain<TARGET, 4, 32, 4, kTempered><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    else if (nblk > 32) k_elementwise_chain<TARGET, 2, 32, 4, kTempered><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    else k_elementwise_chain<TARGET, 1, 32, 4, kTempered><<<e.nsets, 32 * kEwWarps, 0, s>>>(e);
    return cudaGetLastError();
  }
  if (nblk > 128) return launch_range<TARGET, 8, 32, 4>(e, adapting, sms, s);
  if (nblk > 64) return launch_range<TARGET, 4, 32, 4>(e, adapting, sms, s);
  if (nblk > 32) return launch_range<TARGET, 2, 32, 4>(e, adapting, sms, s);
  if (TARGET == HMC_T_STD_NORMAL && e.s.D == 1) return launch_range<HMC_T_STD_NORMAL, 1, 1, 1>(e, adapting, sms, s);
  switch (G) {
    case 1: return launch_range<TARGET, 1, 1, 4>(e, adapting, sms, s);
    case 2: return launch_range<TARGET, 1, 2, 4>(e, adapting, sms, s);
    case 4: return launch_range<TARGET, 1, 4, 4>(e, adapting, sms, s);
    case 8: return launch_range<TARGET, 1, 8, 4>(e, adapting, sms, s);
    case 16: return launch_range<TARGET, 1, 16, 4>(e, adapting, sms, s);
    default: return launch_range<TARGET, 1, 32, 4>(e, adapting, sms, s);
  }
}

// One transition, a warp per chain (elementwise_tile.cuh), without what the chain
// launch carries from one transition to the next.
template <int TARGET, int NB>
__global__ void __launch_bounds__(256) k_fused_elementwise(StepArgs a) {
  elementwise_tile<TARGET, NB>(a, static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x));
}

template <int TARGET>
void launch_tiles(const StepArgs& a, cudaStream_t s) {
  const int nblk = (a.D + 3) / 4;
  const unsigned grid = accept_blocks(a.C);
  if (nblk <= 32) k_fused_elementwise<TARGET, 1><<<grid, 256, 0, s>>>(a);
  else if (nblk <= 64) k_fused_elementwise<TARGET, 2><<<grid, 256, 0, s>>>(a);
  else if (nblk <= 128) k_fused_elementwise<TARGET, 4><<<grid, 256, 0, s>>>(a);
  else k_fused_elementwise<TARGET, 8><<<grid, 256, 0, s>>>(a);
}

// Whether a launch of one transition takes them: for chains of a whole warp where
// they come in more than one round, so that registers per thread (48 of the tile, 64
// to 128 of the chain launch) set how many loads are in flight.  Measured, chain
// launch / tiles: 2000 x 300 1.35, 20000 x 200 1.5, 20000 x 128 1.3 with one leapfrog
// step; 2000 x 200 and 1000 x 500 1.0; below 65 dims 0.9 to 0.2 (chains share a warp there).
// With many steps the funnel's chain launch is the shorter one up to 128 dims (0.95).
bool tiles_pay(int target_id, const StepArgs& a, int sms) {
  if (a.D > 128) return a.C > 8 * sms;
  return a.D > 64 && a.C > 16 * sms && (target_id == HMC_T_STD_NORMAL || a.L < 8);
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

cudaError_t launch_elementwise_chain(int target_id, const StepArgs& a, bool adapting, int T, long long keep_from,
                                     float* samples, float* trace_eps, uint8_t* trace_acc, const ChainSync& sync,
                                     cudaStream_t s, KernelTimer* timer) {
  if (a.D > kFusedElementwiseMaxDim || T < 1) return cudaErrorInvalidValue;
  if (target_id != HMC_T_STD_NORMAL && target_id != HMC_T_FUNNEL) return cudaErrorInvalidValue;
  if (adapting && (a.K > 1 || a.w.mean)) return cudaErrorInvalidValue;
  const int sms = current_sm_count();
  if (T == 1 && !adapting && !a.w.mean && tiles_pay(target_id, a, sms)) {
    StepArgs t = a;
    const long long k = a.t_full - keep_from;
    t.sample_out = k >= 0 && samples ? samples + k * a.C * static_cast<int64_t>(a.D) : nullptr;
    t.trace_eps = k >= 0 && trace_eps ? trace_eps + k : nullptr;
    t.trace_acc = k >= 0 && trace_acc ? trace_acc + k * a.C : nullptr;
    if (timer) timer->begin(s);
    if (target_id == HMC_T_STD_NORMAL) launch_tiles<HMC_T_STD_NORMAL>(t, s);
    else launch_tiles<HMC_T_FUNNEL>(t, s);
    if (timer) timer->end(s);
    count_launch();
    return cudaGetLastError();
  }
  EwArgs e{};
  e.s = a;
  e.T = T;
  e.keep_from = keep_from;
  e.samples = samples;
  e.trace_eps = trace_eps;
  e.trace_acc = trace_acc;
  e.ctr = sync.left;
  e.err = sync.err;
  e.slots = sync.slots;
  e.lim = meeting_limits();
  e.vec = a.D % 4 == 0 && aligned16(a.x) && aligned16(a.g) && aligned16(samples);
  int G = a.K > 1 ? 32 : 1;
  while (G < 32 && 4 * G < a.D) G *= 2;
  // one chain per warp while that is at most two warps per scheduler (its
  // spare lanes then draw ahead); more chains pack into a warp
  while ((a.C >> e.lq) > 8 * sms && (G << e.lq) < 32) ++e.lq;
  const int per_set = kEwWarps << e.lq;
  e.nsets = (a.C + per_set - 1) / per_set;
  if (timer) timer->begin(s);
  const cudaError_t r = target_id == HMC_T_STD_NORMAL ? launch_target<HMC_T_STD_NORMAL>(e, G, adapting, sms, s)
                                                      : launch_target<HMC_T_FUNNEL>(e, G, adapting, sms, s);
  if (timer) timer->end(s);
  count_launch();
  return r;
}

}  // namespace hmc
