// The No-U-Turn Sampler with the recursion unrolled (Section 2.3), for the
// targets whose gradient is elementwise plus row reductions (standard
// normal, funnel).  One warp per chain; chains build their trees
// independently, so a warp's lanes never diverge and different chains' tree
// sizes cost nothing to each other.  A launch runs one transition, or -- where
// the step size is fixed (no adaptation in the range) -- a run of
// transitions, so that each chain's tree sizes average out over the run
// instead of every transition waiting for the deepest tree of all chains.
//
// The transition is Hoffman and Gelman's efficient NUTS (slice variable u)
// as a loop: doubling j grows a subtree of 2^j leapfrog steps (step v_j eps)
// from the trajectory's end on side v_j; at leaf k every span of 2^i leaves
// that closes is checked for a U-turn against its first leaf, which is the
// only state kept per level -- O(max_depth) states, not the 2^depth
// trajectory.  The chain's working (x, p, g) lives in registers (lane owns
// dims 4 (lane + 32 b) .. + 3); the span starts live in shared memory where
// the occupancy allows (else in the per-chain scratch), the two trajectory
// ends and the two candidates in a per-chain scratch of kNutsSlots slots of
// D floats.
//
// What bounds it is the time of one leaf of the longest chain, a warp alone on its
// scheduler for most of a launch: the instructions of a leaf one after another,
// with every branch that is taken and every shuffle level waited for.  So a
// leaf's gradient does not wait for its own sum of squares: x of leaf k + 1 needs
// only leaf k's gradient, and its sum of squares rides in leaf k's butterfly with
// |p|^2 and the U-turn dot products (the exponential of the funnel's v runs
// beneath it); the usual leaf has no branch but the loop's; an even leaf is kept
// once for all the spans it opens.  Measured: a leaf of the 100-dim funnel 646 -> 537
// ns at 1024 chains (1000 -> 832 us for 20 transitions), 800 -> 731 ns at 4096,
// 1577 -> 1471 at 16384, of the 10-dim one 617 -> 509; 500 dims, 1000 chains 1050 -> 867.
//
// The random streams and the choice rule are those of nuts_common.cuh.
#include <cmath>

#include "nuts_common.cuh"

namespace hmc {

namespace {

constexpr int kWarps = 4;

struct NutsArgs {
  StepArgs s;                      // transition s.t_full is the launch's first
  float* scratch;                  // [C][kNutsSlots][Dp]
  int Dp;                          // D rounded up to 4
  int max_depth;
  unsigned long long* leaves;      // [0] leapfrog steps (gradient evaluations), [1] critical
                                   // path (the launches' longest chains), [2] this launch's longest
  int T;                           // transitions in this launch (T > 1: none adapts)
  long long keep_from;             // transition whose new state is kept sample 0
  float* samples;                  // [K][C][D] kept states, or null
  float* trace_eps;                // [K] step size per kept transition, or null
  uint8_t* trace_acc;              // [K][C] moved flags, or null
};

// shared-memory span starts: 2 (max_depth - 1) rows of Dp floats per warp
size_t span_smem_bytes(int Dp, int max_depth) {
  return static_cast<size_t>(kWarps) * 2 * (max_depth > 1 ? max_depth - 1 : 0) * Dp * sizeof(float);
}

// Forms of the kernel.  Resident blocks per SM set the registers a thread may have.
// kWide: for calls whose chains all fit so.  kPlain: as many blocks as a leaf's state
// allows without spills on its critical path (funnel, 4096 x 100: 1458 us for 20
// transitions at 5 blocks, 1869 at 7; standard normal, 4096 x 7: 491 at 7, 550 at 5).
// kLean (past 256 dims): four blocks, for which a leaf forms its own sum of squares
// first and nothing of the next leaf: with every scheduler's slots full the
// instructions count and not a leaf's latency.  20 transitions of the funnel in one
// launch, kPlain / kLean: 2000 x 400 1.31, 4096 x 300 1.19, 3000 x 400 0.98; of the standard
// normal, 4096 x 260 1.11.  A launch of one transition, which ends with its deepest
// trees, is the shorter in kPlain for the funnel (1300 x 300 0.90), unless these are
// shallow and its three blocks do not hold all chains (2000 x 300, depth 3: 1.4; 4096 x
// 400, depth 3: 1.2; 2400 x 400 as depth 5 1.4, 10 1.0).
constexpr int kPlain = 0, kWide = 1, kLean = 2;
constexpr int nuts_blocks(int target, int nb, int form) {
  return form == kWide ? (nb == 1 ? 4 : 2)
         : form == kLean ? 4
         : target == HMC_T_FUNNEL ? (nb == 1 ? 5 : nb == 2 ? 4 : 3) : nb == 1 ? 7 : 4;
}

template <int TARGET, int NB, bool SMEM, int FORM>
__global__ void __launch_bounds__(32 * kWarps, nuts_blocks(TARGET, NB, FORM)) k_nuts(NutsArgs na) {
  // the next leaf's position held over this leaf's decisions; the open pair's
  // first leaf in registers
  constexpr bool kKeepNext = FORM == kWide || (TARGET == HMC_T_FUNNEL && NB == 1), kKeepFirst = kKeepNext && NB == 1;
  extern __shared__ float4 span_smem[];
  const StepArgs& a = na.s;
  const int warp = threadIdx.x >> 5;
  const int c = blockIdx.x * kWarps + warp;
  const int lane = threadIdx.x & 31;
  const bool has_chain = c < a.C;
  float prob = 0.f;
  if (has_chain) {
    const int D = a.D;
    const int64_t row = static_cast<int64_t>(c) * D;
    const int64_t CD = static_cast<int64_t>(a.C) * D;
    const uint32_t chain = static_cast<uint32_t>(c) + a.chain_offset;
    const float eps = a.da->eps;
    float* base = na.scratch + static_cast<int64_t>(c) * kNutsSlots * na.Dp;
    float4* spans = span_smem + static_cast<int64_t>(warp) * 2 * (na.max_depth - 1) * (na.Dp / 4);
    float x[NB][4], p[NB][4], g[NB][4];
    auto slot4 = [&](int s, int b) {
      return reinterpret_cast<float4*>(base + static_cast<int64_t>(s) * na.Dp) + (lane + 32 * b);
    };
    // span row r = 2 (i - 1) (x) or 2 (i - 1) + 1 (p)
    auto span4 = [&](int r, int b) {
      return SMEM ? spans + r * (na.Dp / 4) + (lane + 32 * b) : slot4(kSlotSpan + r, b);
    };
    auto in_slot = [&](int b) { return 4 * (lane + 32 * b) < na.Dp; };
    auto put = [&](float4* q, const float (&v)[NB][4], int b) {
      *q = make_float4(v[b][0], v[b][1], v[b][2], v[b][3]);
    };
    auto get = [&](const float4* q, float (&v)[NB][4], int b) {
      const float4 w = *q;
      v[b][0] = w.x; v[b][1] = w.y; v[b][2] = w.z; v[b][3] = w.w;
    };
    auto store = [&](int s, const float (&v)[NB][4]) {
#pragma unroll
      for (int b = 0; b < NB; ++b)
        if (in_slot(b)) put(slot4(s, b), v, b);
    };
    auto load = [&](int s, float (&v)[NB][4]) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        v[b][0] = v[b][1] = v[b][2] = v[b][3] = 0.f;
        if (in_slot(b)) get(slot4(s, b), v, b);
      }
    };
    auto dot = [&](const float (&u)[NB][4], const float (&w)[NB][4]) {
      float acc = 0.f;
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc = fmaf(u[b][i], w[b][i], acc);
      return warp_sum(acc);
    };
    // both ends' U-turn tests: (dx . pa) < 0 or (dx . pb) < 0
    auto u_turn = [&](const float (&dx)[NB][4], const float (&pa)[NB][4], const float (&pb)[NB][4]) {
      float d1 = 0.f, d2 = 0.f;
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          d1 = fmaf(dx[b][i], pa[b][i], d1);
          d2 = fmaf(dx[b][i], pb[b][i], d2);
        }
      warp_sum2(d1, d2);
      return d1 < 0.f || d2 < 0.f;
    };
    const float half_n = 0.5f * static_cast<float>(D - 1);

    // dim 0 of the funnel is v (lane 0, b 0, i 0); every lane keeps copies of
    // its position, momentum and gradient, and the row sums leave it out: its
    // terms are added to them afterwards
    auto is_v = [&](int b, int i) { return TARGET == HMC_T_FUNNEL && b == 0 && i == 0 && lane == 0; };
    auto lane0 = [&](const float (&u)[NB][4]) { return __shfl_sync(0xffffffffu, u[0][0], 0); };

    // the chain's state at the start of the launch
    float lp = a.lp[c];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int d = 4 * (lane + 32 * b) + i;
        x[b][i] = d < D ? a.x[row + d] : 0.f;
        g[b][i] = d < D ? a.g[row + d] : 0.f;
      }
    unsigned long long leaves_total = 0ull;
    int moved = 0;
    for (int r = 0; r < na.T; ++r) {
      const long long t_full = a.t_full + r;
      const uint32_t t = static_cast<uint32_t>(t_full);
      // start: p0 ~ N(0, I), H0, log U
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int j = lane + 32 * b;
        const float4 z = momentum4(a.seed, static_cast<uint32_t>(j), chain, t);
        const float zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) p[b][i] = 4 * j + i < D ? zz[i] : 0.f;
      }
      const float H0 = -lp + 0.5f * dot(p, p);
      const float logU = accept_log_uniform(a.seed, chain, t);
      store(kSlotLeft, x); store(kSlotLeft + 1, p); store(kSlotLeft + 2, g);
      store(kSlotRight, x); store(kSlotRight + 1, p); store(kSlotRight + 2, g);
      int cand = kSlotCand, sub = kSlotSub;     // trade places when the subtree's is taken
      store(cand, x); store(cand + 1, g);
      float lp_end[2] = {lp, lp};     // [0]: left, [1]: right
      float lpm = lp;
      uint32_t n = 1;
      moved = 0;
      float a_sum = 0.f;
      uint32_t n_a = 0;
      const uint32_t dirs = nuts_word0(a.seed, 0u, chain, t, kNutsTagDirection);
      for (int jd = 0; jd < na.max_depth; ++jd) {
        const int v = ((dirs >> jd) & 1u) ? 1 : -1;
        const float ev = static_cast<float>(v) * eps;
        const float hv = 0.5f * ev;
        const int side = v > 0 ? kSlotRight : kSlotLeft;
        load(side, x); load(side + 1, p); load(side + 2, g);
        lp = lp_end[v > 0 ? 1 : 0];
        uint32_t n_sub = 0;
        bool ok_sub = true;
        float lps = 0.f;
        const int leaves = 1 << jd;
        // the first leaf's position: half a kick, the drift; its sum of squares
        const float sv = static_cast<float>(v);
        float v0 = lane0(x), p0 = lane0(p), g0 = lane0(g), q = 0.f;
        p0 = fmaf(hv, g0, p0);
        v0 = fmaf(ev, p0, v0);
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            p[b][i] = fmaf(hv, g[b][i], p[b][i]);
            x[b][i] = fmaf(ev, p[b][i], x[b][i]);
            if (!is_v(b, i)) q = fmaf(x[b][i], x[b][i], q);
          }
        float em = 0.f;
        if (FORM != kLean) {
          em = expf(-v0);
          q = warp_sum(q);
        }
        // first leaf of the span of two leaves in progress
        float xf[NB][4], pf[NB][4];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int i = 0; i < 4; ++i) xf[b][i] = pf[b][i] = 0.f;
        float xf0 = 0.f, pf0 = 0.f;
        // the subtree-choice words of 128 leaves at a time, four per lane
        auto words = [&](int k) {
          return philox(make_uint4(static_cast<uint32_t>((k >> 2) + lane), chain, t, kNutsTagSubtree + jd),
                        static_cast<uint32_t>(a.seed), static_cast<uint32_t>(a.seed >> 32));
        };
        uint4 wsub4 = words(0);
        int k = 0;
        for (;;) {
          const int kq = k & 3;
          const uint32_t wsub = __shfl_sync(0xffffffffu, kq == 0 ? wsub4.x : kq == 1 ? wsub4.y : kq == 2 ? wsub4.z : wsub4.w,
                                            (k >> 2) & 31);
          if (FORM == kLean) {
            em = expf(-v0);
            q = 0.f;
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                if (!is_v(b, i)) q = fmaf(x[b][i], x[b][i], q);
                xf[b][i] = pf[b][i] = 0.f;      // (not carried from leaf to leaf)
              }
            q = warp_sum(q);
          }
          // the gradient at the drifted x, whose sum of squares is known, and the
          // second half kick
          if (TARGET == HMC_T_FUNNEL) g0 = v0 * (-1.f / 9.f) - half_n + 0.5f * em * q;
          const float p0n = fmaf(hv, g0, p0);
          lp = TARGET == HMC_T_FUNNEL ? v0 * v0 * (-1.f / 18.f) - half_n * v0 - 0.5f * em * q : -0.5f * q;
          if (!kKeepFirst && (k & 1)) {
            const int o = k == 1 ? jd : __ffs(k - 1) - 1;
#pragma unroll
            for (int b = 0; b < NB; ++b)
              if (in_slot(b)) {
                get(span4(2 * (o - 1), b), xf, b);
                get(span4(2 * (o - 1) + 1, b), pf, b);
              }
          }
          // |p|^2, the next leaf's sum of squares and, for the span of two leaves
          // that closes at an odd one, its U-turn dot products dx . pf and
          // dx . p, dx = sv (x - xf) against its first leaf (xf, pf)
          float xn[NB][4], pn[NB][4], pp = 0.f, qn = 0.f, d1 = 0.f, d2 = 0.f;
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              g[b][i] = is_v(b, i) ? g0 : TARGET == HMC_T_FUNNEL ? -em * x[b][i] : -x[b][i];
              p[b][i] = fmaf(hv, g[b][i], p[b][i]);
              if (FORM != kLean) {
                pn[b][i] = fmaf(hv, g[b][i], p[b][i]);
                xn[b][i] = fmaf(ev, pn[b][i], x[b][i]);
              }
              if (!is_v(b, i)) {
                pp = fmaf(p[b][i], p[b][i], pp);
                if (FORM != kLean) qn = fmaf(xn[b][i], xn[b][i], qn);
                const float dx = sv * (x[b][i] - xf[b][i]);
                d1 = fmaf(dx, pf[b][i], d1);
                d2 = fmaf(dx, p[b][i], d2);
              }
            }
          const float p0h = fmaf(hv, g0, p0n), v0n = fmaf(ev, p0h, v0);
          if (FORM == kLean) {
            pp = warp_sum(pp);
            if (k & 1) warp_sum2(d1, d2);
          } else {
            em = expf(-v0n);
            warp_sum4(qn, pp, d1, d2);
          }
          if (TARGET == HMC_T_FUNNEL) {
            const float dx0 = sv * (v0 - xf0);
            d1 = fmaf(dx0, pf0, d1);
            d2 = fmaf(dx0, p0n, d2);
          }
          const float H = -lp + 0.5f * (TARGET == HMC_T_FUNNEL ? fmaf(p0n, p0n, pp) : pp);
          const bool finite = isfinite(H);
          // U-turn, divergence
          ok_sub = !((k & 1) && (d1 < 0.f || d2 < 0.f)) && finite && !(H - H0 >= kNutsDeltaMax - logU);
          const float pr = accept_prob(H0 - H);
          a_sum += finite ? pr : 0.f;
          const bool valid = finite && logU <= H0 - H;
          n_sub += valid;
          if (valid && nuts_take(wsub, 1u, n_sub)) {
            store(sub, x);
            store(sub + 1, g);
            lps = lp;
          }
          // an even leaf opens spans of 2^i leaves for every i with 2^i | k: kept
          // once, in the row of the largest (no other leaf of that row comes
          // before they close)
          if (!(k & 1) && jd) {
            const int o = k ? __ffs(k) - 1 : jd;
#pragma unroll
            for (int b = 0; b < NB; ++b)
              if (in_slot(b)) {
                put(span4(2 * (o - 1), b), x, b);
                put(span4(2 * (o - 1) + 1, b), p, b);
              }
          }
          // longer spans that close here (2^i | k + 1)
          if ((k & 3) == 3) {
            const int close = __ffs(k + 1) - 1;
            for (int i = 2; i <= close && ok_sub; ++i) {
              const int first = k + 1 - (1 << i), o = first ? __ffs(first) - 1 : jd;
              float dx[NB][4], pg[NB][4];
#pragma unroll
              for (int b = 0; b < NB; ++b) {
                dx[b][0] = dx[b][1] = dx[b][2] = dx[b][3] = 0.f;
                pg[b][0] = pg[b][1] = pg[b][2] = pg[b][3] = 0.f;
                if (in_slot(b)) {
                  get(span4(2 * (o - 1), b), dx, b);
                  get(span4(2 * (o - 1) + 1, b), pg, b);
                }
              }
#pragma unroll
              for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int e = 0; e < 4; ++e) dx[b][e] = sv * (x[b][e] - dx[b][e]);
              if (u_turn(dx, pg, p)) ok_sub = false;
            }
          }
          if (++k == leaves || !ok_sub) break;
          // on to the next leaf (k is its number)
          float hv2 = hv, ev2 = ev;
          if (!kKeepNext) asm volatile("" : "+f"(hv2), "+f"(ev2));
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (kKeepFirst) {
                xf[b][i] = k & 1 ? x[b][i] : xf[b][i];
                pf[b][i] = k & 1 ? p[b][i] : pf[b][i];
              }
              if (kKeepNext) {
                x[b][i] = xn[b][i];
                p[b][i] = pn[b][i];
              } else {          // formed again: held over the decisions they cost registers
                p[b][i] = fmaf(hv2, g[b][i], p[b][i]);
                x[b][i] = fmaf(ev2, p[b][i], x[b][i]);
              }
            }
          xf0 = k & 1 ? v0 : xf0;
          pf0 = k & 1 ? p0n : pf0;
          v0 = v0n;
          p0 = p0h;
          q = qn;
          if (__builtin_expect((k & 127) == 0, 0)) wsub4 = words(k);
        }
        n_a += k;
        if (!ok_sub) break;
        store(side, x); store(side + 1, p); store(side + 2, g);
        lp_end[v > 0 ? 1 : 0] = lp;
        if (n_sub > 0 && nuts_take(nuts_word0(a.seed, static_cast<uint32_t>(jd), chain, t, kNutsTagTop), n_sub, n)) {
          const int was = cand;
          cand = sub;
          sub = was;
          lpm = lps;
          moved = 1;
        }
        n += n_sub;
        // the whole trajectory's ends
        float xl[NB][4], pl[NB][4], xr[NB][4], pr[NB][4];
        load(kSlotLeft, xl); load(kSlotLeft + 1, pl);
        load(kSlotRight, xr); load(kSlotRight + 1, pr);
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int q = 0; q < 4; ++q) xr[b][q] -= xl[b][q];
        if (u_turn(xr, pl, pr)) break;
      }
      // the new state
      load(cand, x);
      load(cand + 1, g);
      lp = lpm;
      prob = a_sum / static_cast<float>(n_a);
      leaves_total += n_a;
      const long long k = t_full - na.keep_from;
      if (k >= 0) {
        if (na.samples) {
          float* out = na.samples + k * CD + row;
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int d = 4 * (lane + 32 * b) + i;
              if (d < D) out[d] = x[b][i];
            }
        }
        if (lane == 0) {
          if (na.trace_acc) na.trace_acc[k * a.C + c] = static_cast<uint8_t>(moved);
          if (c == 0 && na.trace_eps) na.trace_eps[k] = eps;
        }
      }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int d = 4 * (lane + 32 * b) + i;
        if (d < D) {
          a.x[row + d] = x[b][i];
          a.g[row + d] = g[b][i];
        }
      }
    if (lane == 0) {
      a.lp[c] = lp;
      a.is_accepted[c] = static_cast<uint8_t>(moved);
      a.log_accept[c] = logf(prob);
      atomicAdd(na.leaves, leaves_total);
      atomicMax(na.leaves + 2, leaves_total);
    }
  }
  // the last transition's statistic (the only one that can adapt)
  const bool last = accept_tile_finish<kWarps>(a.da, a.partials, prob, has_chain, a.C, a.t_full + na.T - 1,
                                               static_cast<int>(blockIdx.x), static_cast<int>(gridDim.x));
  // the launch lasts at least as long as its longest chain's leaves: the
  // critical path (the block that arrived last adds it)
  if (last && threadIdx.x == 0) {
    __threadfence();
    na.leaves[1] += atomicExch(na.leaves + 2, 0ull);
  }
}

template <int TARGET, int NB, bool SMEM, int FORM>
cudaError_t launch_v(const NutsArgs& na, size_t smem, cudaStream_t s) {
  const unsigned grid = nuts_grid(na.s.C);
  k_nuts<TARGET, NB, SMEM, FORM><<<grid, 32 * kWarps, SMEM ? smem : 0, s>>>(na);
  count_launch();
  return cudaGetLastError();
}

// resident blocks per SM with the span starts in scratch and in shared memory
// (0: they do not fit)
template <int TARGET, int NB, int FORM>
cudaError_t residency(size_t smem, int* glob, int* shared) {
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(glob, k_nuts<TARGET, NB, false, FORM>, 32 * kWarps, 0);
  *shared = 0;
  if (e == cudaSuccess && smem > 0 && smem <= kNutsSpanSmemMax)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(shared, k_nuts<TARGET, NB, true, FORM>, 32 * kWarps, smem);
  return e;
}

inline bool all_resident(const NutsArgs& na, int blocks, int sms) {
  return static_cast<int64_t>(blocks) * kWarps * sms >= na.s.C;
}

// More chains than the wide form holds.  Span starts in shared memory unless
// they cost resident chains: as many blocks per SM as the scratch form, or
// enough for every chain.
template <int TARGET, int NB, int FORM>
cudaError_t launch_many(const NutsArgs& na, size_t smem, bool wide, int sms, cudaStream_t s) {
  int glob = 0, shared = 0;
  const cudaError_t e = residency<TARGET, NB, FORM>(smem, &glob, &shared);
  if (e != cudaSuccess) return e;
  if (shared > 0 && (shared >= glob || all_resident(na, shared, sms))) return launch_v<TARGET, NB, true, FORM>(na, smem, s);
  return wide ? launch_v<TARGET, NB, false, kWide>(na, 0, s) : launch_v<TARGET, NB, false, FORM>(na, 0, s);
}

template <int TARGET, int NB>
cudaError_t launch_nb(const NutsArgs& na, cudaStream_t s) {
  const size_t smem = span_smem_bytes(na.Dp, na.max_depth);
  const int sms = current_sm_count();
  int glob = 0, shared = 0;
  const cudaError_t e = residency<TARGET, NB, kWide>(smem, &glob, &shared);
  if (e != cudaSuccess) return e;
  // the wide form where all its chains are resident at once: 1024 x 100 funnel
  // 832 us for 20 transitions (837 at 5 blocks), 1000 x 500 1605 against 1813,
  // but 2000 x 200 standard normal 362 us against 262, in two waves
  if (all_resident(na, shared, sms)) return launch_v<TARGET, NB, true, kWide>(na, smem, s);
  const bool wide = all_resident(na, glob, sms);
  if constexpr (NB == 4) {
    // (shallow trees end together: a second round of blocks is what counts there)
    const bool shallow = na.max_depth <= (all_resident(na, nuts_blocks(TARGET, NB, kLean), sms) ? 7 : 6) &&
                         !all_resident(na, nuts_blocks(TARGET, NB, kPlain), sms);
    if (TARGET == HMC_T_STD_NORMAL || na.T > 1 || shallow) return launch_many<TARGET, NB, kLean>(na, smem, wide, sms, s);
  }
  if constexpr (NB < 4 || TARGET == HMC_T_FUNNEL) return launch_many<TARGET, NB, kPlain>(na, smem, wide, sms, s);
  return cudaErrorInvalidValue;      // (not reached)
}

template <int TARGET>
cudaError_t launch_t(const NutsArgs& na, cudaStream_t s) {
  const int nb = (na.s.D + 127) / 128;
  if (nb <= 1) return launch_nb<TARGET, 1>(na, s);
  if (nb == 2) return launch_nb<TARGET, 2>(na, s);
  return launch_nb<TARGET, 4>(na, s);
}

template <int TARGET, int NB, int FORM>
cudaError_t allow_smem() {
  return cudaFuncSetAttribute(k_nuts<TARGET, NB, true, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kNutsSpanSmemMax));
}

template <int TARGET>
cudaError_t allow_smem_target() {
  cudaError_t e = allow_smem<TARGET, 1, kWide>();
  if (e == cudaSuccess) e = allow_smem<TARGET, 2, kWide>();
  if (e == cudaSuccess) e = allow_smem<TARGET, 4, kWide>();
  if (e == cudaSuccess) e = allow_smem<TARGET, 1, kPlain>();
  if (e == cudaSuccess) e = allow_smem<TARGET, 2, kPlain>();
  if (e == cudaSuccess) e = allow_smem<TARGET, 4, kLean>();
  if constexpr (TARGET == HMC_T_FUNNEL) {
    if (e == cudaSuccess) e = allow_smem<TARGET, 4, kPlain>();
  }
  return e;
}

}  // namespace

bool nuts_supported(const hmc_target& t) {
  return (t.id == HMC_T_STD_NORMAL || t.id == HMC_T_FUNNEL) && t.dim <= kNutsMaxDim;
}

size_t nuts_scratch_floats(const hmc_target& t, int64_t C) {
  return static_cast<size_t>(C) * kNutsSlots * ((t.dim + 3) / 4 * 4);
}

unsigned nuts_grid(int64_t C) { return static_cast<unsigned>((C + kWarps - 1) / kWarps); }

cudaError_t nuts_prepare() {
  const cudaError_t e = allow_smem_target<HMC_T_STD_NORMAL>();
  return e != cudaSuccess ? e : allow_smem_target<HMC_T_FUNNEL>();
}

cudaError_t launch_nuts_transitions(const hmc_target& t, const StepArgs& a, float* scratch,
                                    int max_depth, unsigned long long* leaves, int T,
                                    long long keep_from, float* samples, float* trace_eps,
                                    uint8_t* trace_acc, cudaStream_t s, KernelTimer* timer) {
  NutsArgs na{a, scratch, (t.dim + 3) / 4 * 4, max_depth, leaves, T, keep_from, samples, trace_eps,
              trace_acc};
  if (timer) timer->begin(s);
  cudaError_t e = t.id == HMC_T_FUNNEL ? launch_t<HMC_T_FUNNEL>(na, s) : launch_t<HMC_T_STD_NORMAL>(na, s);
  if (timer) timer->end(s);
  return e;
}

cudaError_t launch_nuts_transition(const hmc_target& t, const StepArgs& a, float* scratch,
                                   int max_depth, unsigned long long* leaves, cudaStream_t s,
                                   KernelTimer* timer) {
  return launch_nuts_transitions(t, a, scratch, max_depth, leaves, 1, a.t_full, a.sample_out,
                                 a.trace_eps, a.trace_acc, s, timer);
}

}  // namespace hmc
