// HMC chains of a small Bayesian logistic regression (Section 2.1): one launch
// runs a range of transitions with the data in every SM's shared memory.
//
// A group of 256 threads advances one chain; a CTA holds 1, 2 or 4 groups, which
// share the data.  The arithmetic, sum by sum, is that of the 8-chain tile
// (logreg_tile.cuh), which the batch's grouped launch runs and which works
// through the rows 16 at a time: z in even and odd dims, each 16-row block's
// contribution to the gradient on its own, the blocks added in order.  Only the
// order of the additions is a chain: the 16-row blocks are independent, so the
// group computes all rows' z at once, then all (block, dim) contributions at
// once, and only adds N / 16 numbers per dim one after the other -- three
// barriers per gradient where the tile takes three per 16 rows.  Measured, 64
// chains, 800 rows, 11 dims, 10 leapfrog steps: 486 us per transition (8 CTAs,
// 50 row blocks in series) -> 18.6 us, 23.8 us while adapting; 1000 chains, 500
// rows, 8 dims 32.6 us.  What bounds it now: the latency of shared-memory loads
// and dependent additions between the three barriers (the schedulers issue in
// 24 % of the cycles; 512 threads per chain gave 10 % at 64 chains and lost 50 %
// at 1000).
//
// Adapting transitions meet through one slot per chain (chain_sync.cuh) and sum
// them in the tile's order, so results do not depend on the launch form.
#include <algorithm>
#include <cmath>

#include "chain_sync.cuh"
#include "logreg_tile.cuh"

namespace hmc {

namespace {

constexpr int kLrGroup = 256;                 // threads per chain
constexpr int kLrMaxGroups = 4;
constexpr size_t kLrChainSmemMax = 216 * 1024;   // with the static part, within 227 KB
constexpr int64_t kLrChainMaxRows = 2048;     // as the tile's own launch

// Shared-memory layout in floats.  Rows come in blocks of 16; a row's stride ld
// is 2 mod 4 (float2 reads of 16 consecutive rows hit distinct banks) and a
// block's stride is the row length mod 32, rounded up to even, so that
// consecutive (block, dim) pairs do too.  The blocks' contributions are kept
// by dim (stride ps, 4 mod 8: float4 reads of 8 dims hit distinct banks), with
// zeros past the last block.
struct LrLayout {
  int ld, block, nblk, dpad, ps;
  int off_y, off_group, group;                // data labels; first group's area and its size
  int res, ll, part, th, pm, z, x0, g0, gn, scal; // offsets inside a group's area
  size_t bytes(int groups) const { return sizeof(float) * (static_cast<size_t>(off_group) + static_cast<size_t>(group) * groups); }
};

__host__ __device__ inline LrLayout lr_layout(int N, int D) {
  LrLayout l;
  l.ld = (D + 1) / 4 * 4 + 2;                 // >= D, 2 mod 4
  l.nblk = (N + 15) / 16;
  const int want = (D + 1) / 2 * 2 % 32, have = 16 * l.ld % 32;
  l.block = 16 * l.ld + (want - have + 32) % 32;
  l.dpad = (l.ld + 3) / 4 * 4;                // (zeros past D)
  l.ps = (l.nblk + 3) / 8 * 8 + 4;            // >= nblk, 4 mod 8
  l.off_y = (l.nblk * l.block + 3) / 4 * 4;
  l.off_group = l.off_y + 16 * l.nblk;
  l.res = 0;
  l.ll = l.res + 16 * l.nblk;
  l.part = l.ll + 16 * l.nblk;
  l.th = l.part + l.ps * D;
  l.pm = l.th + l.dpad;
  l.z = l.pm + l.dpad;                        // [2][dpad] momenta, by transition parity
  l.x0 = l.z + 2 * l.dpad;
  l.g0 = l.x0 + l.dpad;
  l.gn = l.g0 + l.dpad;
  l.scal = l.gn + l.dpad;
  l.group = l.scal + 24;
  return l;
}

struct LrChainArgs {
  StepArgs s;                // s.t / s.t_full: the range's first transition
  const float* X;
  const float* y;
  int N, T, groups;
  int rounds;                // chains per group, one after the other
  long long keep_from;       // transition keep_from + k is kept draw k
  float* samples;
  float* trace_eps;
  uint8_t* trace_acc;
  ChainSync sync;            // one slot per chain
  MeetingLimits lim;         // adapting launches: the meeting after transition i is meeting i + 1
};

template <int GT>
__device__ __forceinline__ void group_sync(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(GT) : "memory");
}

// z of R rows (first r, GT apart) and what follows from it.  LD: the row
// stride where it is known (then the padding's zeros are added too: no change).
template <int GT, int R, int LD>
__device__ __forceinline__ void rows_pass(const LrLayout& l, const float* Xs, const float* ys, float* grp, int N, int D,
                                          int r, bool need_lp) {
  const float* xr[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int row = min(r + GT * i, N - 1);
    xr[i] = Xs + (row >> 4) * l.block + (row & 15) * (LD ? LD : l.ld);
  }
  float ze[R], zo[R];
#pragma unroll
  for (int i = 0; i < R; ++i) ze[i] = zo[i] = 0.f;
  const float2* th = reinterpret_cast<const float2*>(grp + l.th);
  auto two_dims = [&](int d) {
    const float2 t = th[d >> 1];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float2 x = *reinterpret_cast<const float2*>(xr[i] + d);
      ze[i] = fmaf(x.x, t.x, ze[i]);
      zo[i] = fmaf(x.y, t.y, zo[i]);
    }
  };
  if (LD) {
#pragma unroll
    for (int d = 0; d < LD; d += 2) two_dims(d);
  } else {
#pragma unroll 4
    for (int d = 0; d < D; d += 2) two_dims(d);    // (odd D: the padding column is zero)
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int row = r + GT * i;
    if (row >= N) break;
    const float z = ze[i] + zo[i], yv = ys[row];
    grp[l.res + row] = yv - lr::sigmoid_stable(z);
    if (need_lp) grp[l.ll + row] = yv * z - lr::softplus_stable(z);
  }
}

// The sum over C chains of the written slots, tile by tile (eight in chain
// order), the tiles as tile_partial_then_da adds them; all threads, the value
// in warp 0.  wait_ns > 0: poll until written; false after that time (never:
// nothing counts as written).
__device__ __forceinline__ bool tile_slots_sum(const unsigned long long* slots, int C, bool negative,
                                               unsigned long long wait_ns, bool never, double* sum) {
  __shared__ double tile_s[kLrGroup * kLrMaxGroups];
  __shared__ int gave_up;
  const int ntiles = (C + 7) / 8;
  if (threadIdx.x == 0) gave_up = 0;
  __syncthreads();
  const unsigned long long want = negative ? kSlotSign : 0ull;
  unsigned long long t0 = 0;
  double acc = 0.0;
  for (int base = 0; base < ntiles; base += static_cast<int>(blockDim.x)) {
    const int tile = base + static_cast<int>(threadIdx.x);
    if (tile < ntiles) {
      unsigned long long w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = 8 * tile + i < C ? want ^ kSlotSign : want;
      bool ready = false;
      while (!ready) {
        ready = !never;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if ((w[i] & kSlotSign) != want) w[i] = read_slot(slots + 8 * tile + i);
#pragma unroll
        for (int i = 0; i < 8; ++i) ready = ready && (w[i] & kSlotSign) == want;
        if (wait_ns == 0) break;
        if (!ready) {
          const unsigned long long now = ptx::global_timer_ns();
          if (!t0) t0 = now;
          if (now - t0 > wait_ns) {
            gave_up = 1;
            break;
          }
        }
      }
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < 8; ++i) s += slot_value(w[i]);
      tile_s[threadIdx.x] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32)
      for (int b = threadIdx.x; b < static_cast<int>(blockDim.x) && base + b < ntiles; b += 32) acc += tile_s[b];
    if (base + static_cast<int>(blockDim.x) < ntiles) __syncthreads();
  }
  if (threadIdx.x < 32) *sum = warp_sum_d(acc);
  return gave_up == 0;
}

template <bool COOP, int LD>
__global__ void __launch_bounds__(kLrGroup * kLrMaxGroups, 1) k_logreg_chain(LrChainArgs e) {
  constexpr int GT = kLrGroup, kW = GT / 32;      // the last warps of a group take the end's sums
  extern __shared__ float4 smem_lr[];
  __shared__ DAState da_s;
  __shared__ DACoef coef_s[32];
  __shared__ int flag_s;
  const StepArgs& a = e.s;
  const int D = a.D, N = e.N, C = a.C;
  const LrLayout l = lr_layout(N, D);
  float* base = reinterpret_cast<float*>(smem_lr);
  float* Xs = base;
  float* ys = base + l.off_y;
  const int group = threadIdx.x / GT, tid = threadIdx.x % GT, warp = tid >> 5, lane = tid & 31;
  float* grp = base + l.off_group + group * l.group;
  float* th = grp + l.th;
  float* pm = grp + l.pm;
  float* x0 = grp + l.x0;
  float* g0 = grp + l.g0;
  float* gn = grp + l.gn;
  float* scal = grp + l.scal;      // 0 lp0, 1 log u, 2 log-lik sum, 3 |theta|^2, 4 kin0, 5 accepted, 8-23 log-lik sums by row mod 16
  const int64_t CD = static_cast<int64_t>(C) * D;

  // the data, with zeros past the last row and dim
  for (int i = threadIdx.x; i < l.nblk * l.block; i += blockDim.x) Xs[i] = 0.f;
  for (int i = threadIdx.x; i < 16 * l.nblk; i += blockDim.x) ys[i] = i < N ? e.y[i] : 0.f;
  for (int i = tid; i < l.group; i += GT) grp[i] = 0.f;
  if (threadIdx.x == 0) {
    flag_s = 0;
    if (COOP) da_s = *a.da;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < N * D; i += blockDim.x) {
    const int r = i / D, d = i - r * D;
    Xs[(r >> 4) * l.block + (r & 15) * l.ld + d] = e.X[i];
  }
  float eps = COOP ? da_s.eps : a.da->eps;
  const double n_c = static_cast<double>(C), inv_c = COOP ? 1.0 / n_c : 0.0;
  const bool resident = e.rounds == 1;
  // this thread's first (block, dim) and the step to its next
  const int b_first = tid / D, d_first = tid - b_first * D, dq = GT / D, dr = GT - dq * D;
  __syncthreads();

  long long k = a.t_full - e.keep_from;
  for (int i = 0; i < e.T; ++i, ++k) {
    const uint32_t t = a.t + static_cast<uint32_t>(i);
    const bool last = i == e.T - 1, keep = k >= 0;
    unsigned long long* slots = e.sync.slots + (COOP && (i & 1) ? C : 0);
    if (COOP && (i & 31) == 0 && threadIdx.x < 32) {
      __syncwarp();
      coef_s[lane] = da_prepare(&da_s, a.t_full + i + lane, lane);
      __syncwarp();
    }
    for (int round = 0; round < e.rounds; ++round) {
      const int c = (round * e.groups + group) * static_cast<int>(gridDim.x) + static_cast<int>(blockIdx.x);
      if (c >= C) break;                       // uniform in the group
      const int64_t row = static_cast<int64_t>(c) * D;
      const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
      float* z = grp + l.z + (resident && (i & 1) ? l.dpad : 0);
      float* z_next = grp + l.z + (i & 1 ? 0 : l.dpad);
      const bool draw_early = resident && D <= GT / 2;      // threads past the dims draw the next momenta
      // begin: p0 ~ N(0, I), half kick with the cached gradient, first drift
      for (int d = tid; d < D; d += GT) {
        if (!resident || i == 0) {
          x0[d] = a.x[row + d];
          g0[d] = a.g[row + d];
        }
        if (!draw_early || i == 0) z[d] = momentum1(a.seed, static_cast<uint32_t>(d), chain, t);
        const float p = fmaf(0.5f * eps, g0[d], z[d]);
        pm[d] = p;
        th[d] = fmaf(eps, p, x0[d]);
      }
      if (tid == 0 && (!resident || i == 0)) scal[0] = a.lp[c];
      group_sync<GT>(group);
      for (int step = 1; step <= a.L; ++step) {
        const bool end = step == a.L;
        // all rows: z, residual (and at the end the log-likelihood)
        if (N <= GT) {
          if (tid < N) rows_pass<GT, 1, LD>(l, Xs, ys, grp, N, D, tid, end);
        } else if (N <= 2 * GT) {
          rows_pass<GT, 2, LD>(l, Xs, ys, grp, N, D, tid, end);
        } else if (N <= 3 * GT) {
          rows_pass<GT, 3, LD>(l, Xs, ys, grp, N, D, tid, end);
        } else {
          for (int r = tid; r < N; r += 4 * GT) rows_pass<GT, 4, LD>(l, Xs, ys, grp, N, D, r, end);
        }
        group_sync<GT>(group);
        // all (16-row block, dim) contributions to the gradient
        {
          int b = b_first, d = d_first;
          for (int q = tid; q < l.nblk * D; q += GT) {
            const float4* rs = reinterpret_cast<const float4*>(grp + l.res + 16 * b);
            const float* xp = Xs + b * l.block + d;
            float acc = 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float4 rv = rs[u];
              const int ld = LD ? LD : l.ld;
              acc = fmaf(rv.x, xp[(4 * u) * ld], acc);
              acc = fmaf(rv.y, xp[(4 * u + 1) * ld], acc);
              acc = fmaf(rv.z, xp[(4 * u + 2) * ld], acc);
              acc = fmaf(rv.w, xp[(4 * u + 3) * ld], acc);
            }
            grp[l.part + d * l.ps + b] = acc;
            b += dq;
            d += dr;
            if (d >= D) {
              d -= D;
              ++b;
            }
          }
        }
        group_sync<GT>(group);
        // the blocks in order, the prior, kick and drift
        const float kick = end ? 0.5f * eps : eps;
        for (int d = tid; d < D; d += GT) {
          const float4* pp = reinterpret_cast<const float4*>(grp + l.part + d * l.ps);
          float g = 0.f;
#pragma unroll 4
          for (int b = 0; b < l.ps / 4; ++b) {
            const float4 v = pp[b];
            g += v.x;
            g += v.y;
            g += v.z;
            g += v.w;
          }
          const float tv = th[d];
          g -= tv;
          const float p = fmaf(kick, g, pm[d]);
          pm[d] = p;
          if (end) gn[d] = g;
          else th[d] = fmaf(eps, p, tv);
        }
        if (step == 1) {
          if (draw_early && !last && tid >= GT / 2 && tid - GT / 2 < D)
            z_next[tid - GT / 2] = momentum1(a.seed, static_cast<uint32_t>(tid - GT / 2), chain, t + 1);
          if (tid == GT - 1) scal[1] = accept_log_uniform(a.seed, chain, t);
        }
        if (end) {
          if (warp == kW - 1) {                // log-likelihood: 16 sums over the blocks, then their sum
            if (lane < 16) {
              const float* ll = grp + l.ll + lane;
              float lpb = 0.f;                 // (rows past N hold zeros)
              for (int b = 0; b < l.nblk; b += 16) {
                float v[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) v[u] = b + u < l.nblk ? ll[16 * (b + u)] : 0.f;
#pragma unroll
                for (int u = 0; u < 16; ++u) lpb += v[u];
              }
              scal[8 + lane] = lpb;
            }
            __syncwarp();
            if (lane == 0) {
              float lp = 0.f;
#pragma unroll
              for (int r = 0; r < 16; ++r) lp += scal[8 + r];
              scal[2] = lp;
            }
          } else if (warp == kW - 2) {
            float sq = 0.f;
            for (int d = lane; d < D; d += 32) sq = fmaf(th[d], th[d], sq);
            sq = warp_sum(sq);
            if (lane == 0) scal[3] = sq;
          } else if (warp == kW - 3) {
            float kin0 = 0.f;
            for (int d = lane; d < D; d += 32) kin0 = fmaf(z[d], z[d], kin0);
            kin0 = 0.5f * warp_sum(kin0);
            if (lane == 0) scal[4] = kin0;
          }
        }
        group_sync<GT>(group);
      }
      if (warp == 0) {
        float kin1 = 0.f;
        for (int d = lane; d < D; d += 32) kin1 = fmaf(pm[d], pm[d], kin1);
        kin1 = 0.5f * warp_sum(kin1);
        if (lane == 0) {
          const float lp0 = scal[0], kin0 = scal[4], lp1 = scal[2] - 0.5f * scal[3];
          float la = (-lp0 + kin0) - (-lp1 + kin1);
          if (!isfinite(la)) la = -INFINITY;
          const bool acc = scal[1] < la;
          scal[5] = acc ? 1.f : 0.f;
          if (acc) scal[0] = lp1;
          if (COOP) put_slot(slots + c, static_cast<double>(accept_prob(la)), (i & 2) != 0);
          else if (last) put_slot(slots + c, static_cast<double>(accept_prob(la)), false);
          if (!resident || last) a.lp[c] = scal[0];
          if (last) {
            a.is_accepted[c] = acc ? 1 : 0;
            a.log_accept[c] = la;
          }
          if (keep && e.trace_acc) e.trace_acc[k * C + c] = acc ? 1 : 0;
          if (keep && c == 0 && e.trace_eps) e.trace_eps[k] = eps;
        }
      }
      group_sync<GT>(group);
      const bool acc = scal[5] != 0.f;
      for (int d = tid; d < D; d += GT) {
        if (acc) {
          x0[d] = th[d];
          g0[d] = gn[d];
        }
        const float xv = x0[d];
        if (!resident || last) {
          a.x[row + d] = xv;
          a.g[row + d] = g0[d];
        }
        if (keep && e.samples) e.samples[k * CD + row + d] = xv;
        if (keep && a.w.mean) welford_update(a.w, welford_coef(k, a.w.bsize), k, row + d, xv);
      }
    }
    if (COOP) {
      double sum = 0.0;
      const bool ok = tile_slots_sum(slots, C, (i & 2) != 0, e.lim.wait_ns, i + 1 == e.lim.unreachable_gen, &sum);
      if (threadIdx.x == 0) {
        if (ok) {
          da_apply_sum(&da_s, coef_s[i & 31], sum, n_c, inv_c, a.t_full + i);
        } else {
          atomicExch(e.sync.err, 4);
          flag_s = 1;
        }
      }
      __syncthreads();
      if (flag_s) break;
      eps = da_s.eps;
    }
  }
  if (COOP) {
    leave_adapting(a.da, &da_s, e.sync.left, e.sync.slots, 2 * static_cast<int64_t>(C));
  } else {
    // the last CTA to finish applies the last transition's statistic
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      flag_s = atomicAdd(&a.da->arrive, 1u) == gridDim.x - 1u ? 1 : 0;
      __threadfence();
    }
    __syncthreads();
    if (flag_s) {
      double sum = 0.0;
      tile_slots_sum(e.sync.slots, C, false, 0, false, &sum);
      __syncthreads();
      if (threadIdx.x == 0) {
        da_update(a.da, sum / static_cast<double>(C), a.t_full + e.T - 1);
        a.da->arrive = 0u;
      }
      for (int c = threadIdx.x; c < C; c += blockDim.x) e.sync.slots[c] = kEmptySlot;
    }
  }
}

}  // namespace

// the kernel for row stride ld: data of 7 to 22 dims (a posterior of some
// hundred rows that takes this path) has its stride compiled in
template <bool COOP>
void (*lr_chain_kernel(int ld))(LrChainArgs) {
  switch (ld) {
    case 10: return k_logreg_chain<COOP, 10>;
    case 14: return k_logreg_chain<COOP, 14>;
    case 18: return k_logreg_chain<COOP, 18>;
    case 22: return k_logreg_chain<COOP, 22>;
    default: return k_logreg_chain<COOP, 0>;
  }
}

size_t logreg_chain_sync_bytes(int64_t C) { return 16 + 16 * static_cast<size_t>(C); }

bool logreg_chain_supported(const hmc_target& t) {
  return t.id == HMC_T_LOGREG && t.dim <= lr::kLrMaxDim && t.n_data <= kLrChainMaxRows &&
         lr_layout(static_cast<int>(t.n_data), t.dim).bytes(1) <= kLrChainSmemMax;
}

// a chain per CTA while every chain gets an SM of its own, then two and four
// groups per CTA, as far as their areas fit
static int chain_groups(const LrLayout& l, int64_t C, int sms) {
  int g = 1;
  while (g < kLrMaxGroups && C > sms * g && l.bytes(2 * g) <= kLrChainSmemMax) g *= 2;
  return g;
}

// Whether a launch of this kind takes the chain kernel, or the 8-chain tiles
// (logreg_tile.cuh), a launch per transition: the shorter one by these estimates of a
// transition in us.  The tiles work through their 16-row blocks one after another but
// keep up to 64 chains on an SM; the chain kernel has all blocks in flight and `g`
// chains on an SM, so C chains take `rounds` rounds, each with what a transition costs
// beside its gradients (in a launch of one transition also the data's way into shared
// memory).  Fitted to both kernels' times at 4400 points, 17-1500 rows, 4-512 dims,
// 64-30000 chains, 1-20 steps, all three kinds (median error 7 and 5 %); the choice is off by
// more than 10 % at 1 % of them.  Tile time / chain time measured: 17 x 4 and 2400
// chains 0.85 in a fixed range of 10 steps, 0.42 one transition of one step; 64 x 4 and
// 5000 chains 1.22 and 0.35; 200 x 4 and 5000 chains 2.83 and 0.66; 800 x 11 and 64
// chains 26 and 15.
bool logreg_chain_pays(const hmc_target& t, int64_t C, int L, ChainKind kind) {
  const int N = static_cast<int>(t.n_data), D = t.dim, sms = current_sm_count();
  const LrLayout l = lr_layout(N, D);
  const int g = chain_groups(l, C, sms);
  const double nd = static_cast<double>(N) * D, m = static_cast<double>(C) / (8.0 * sms);
  const double tiles =
      9.9 + 1.6 * m + (static_cast<double>(L) * l.nblk + 1.0) * std::max(0.88 + 0.022 * D, m * (0.38 + 0.015 * D));
  const double rounds = std::ceil(std::ceil(static_cast<double>(C) / g) / sms);
  const double gradient = 0.50 + 0.012 * l.nblk + 0.36e-4 * g * nd + 0.0064 * D;
  const double once = kind == ChainKind::kFixed ? 1.6 : kind == ChainKind::kAdapting ? 3.8 : 4.2;
  const double round = kind == ChainKind::kFixed ? 3.8 : kind == ChainKind::kAdapting ? 4.5 : 7.5 + 3.2e-4 * nd;
  return once + rounds * (round + L * gradient) <= tiles;
}

cudaError_t logreg_chain_setup() {
  // the attribute belongs to the kernels, shared by every context: the maximum
  cudaError_t e = cudaSuccess;
  for (auto k : {lr_chain_kernel<false>(10), lr_chain_kernel<false>(14), lr_chain_kernel<false>(18),
                 lr_chain_kernel<false>(22), lr_chain_kernel<false>(0), lr_chain_kernel<true>(10),
                 lr_chain_kernel<true>(14), lr_chain_kernel<true>(18), lr_chain_kernel<true>(22),
                 lr_chain_kernel<true>(0)})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLrChainSmemMax));
  return e;
}

cudaError_t launch_logreg_chain(const hmc_target& t, const StepArgs& a, bool adapting, int T, long long keep_from,
                                float* samples, float* trace_eps, uint8_t* trace_acc, const ChainSync& sync,
                                cudaStream_t s, KernelTimer* timer) {
  if (!logreg_chain_supported(t) || T < 1 || a.K > 1) return cudaErrorInvalidValue;
  if (T == 1 && !adapting && !logreg_chain_pays(t, a.C, a.L, ChainKind::kOne)) {
    StepArgs one = a;
    const long long k = a.t_full - keep_from;
    if (k >= 0) {
      one.sample_out = samples ? samples + k * a.C * static_cast<int64_t>(a.D) : nullptr;
      one.trace_eps = trace_eps ? trace_eps + k : nullptr;
      one.trace_acc = trace_acc ? trace_acc + k * a.C : nullptr;
    }
    cudaError_t r = launch_logreg_fused_transition(t, one, s, timer);
    if (r == cudaSuccess && k >= 0 && a.w.mean)
      r = launch_welford(static_cast<int64_t>(a.C) * a.D, a.x, k, a.w.mean, a.w.m2, a.w.bsize, a.w.bsum, a.w.bmean,
                         a.w.bm2, s);
    return r;
  }
  LrChainArgs e{};
  e.s = a;
  e.X = t.X;
  e.y = t.y;
  e.N = static_cast<int>(t.n_data);
  e.T = T;
  e.keep_from = keep_from;
  e.samples = samples;
  e.trace_eps = trace_eps;
  e.trace_acc = trace_acc;
  e.sync = sync;
  e.lim = meeting_limits();
  const LrLayout l = lr_layout(e.N, t.dim);
  // (past four groups a CTA, more chains per group)
  const int sms = current_sm_count();
  e.groups = chain_groups(l, a.C, sms);
  const int need = (a.C + e.groups - 1) / e.groups;
  // an adapting range's CTAs must all be resident (one per SM is always)
  const int grid = adapting ? std::min(need, sms) : need;
  e.rounds = (need + grid - 1) / grid;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(static_cast<unsigned>(kLrGroup * e.groups));
  cfg.dynamicSmemBytes = l.bytes(e.groups);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = adapting ? 1 : 0;
  if (timer) timer->begin(s);
  auto kernel = adapting ? lr_chain_kernel<true>(l.ld) : lr_chain_kernel<false>(l.ld);
  const cudaError_t r = cudaLaunchKernelEx(&cfg, kernel, e);
  if (timer) timer->end(s);
  count_launch();
  return r;
}

}  // namespace hmc
