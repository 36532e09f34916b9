// mt_transfer.cu -- weights (Eq. 3), normalisation (Sec. 1.1), exchange
// (Eq. 4, Eq. 7) and the A + B -> E reaction (Sec. 3, Sec. 7), in two
// passes: pass 1 forms the row sums r_i = sum_j nu_ij (self included) and
// stores 1 / r_i; pass 2 forms dM_i = 1/2 sum_j P_ij (M_j - M_i) for A and B,
// updates, reacts and reduces the per-step observables.
//
// Neighbour search variants:
//   walk  (1-d cell list) particles are sorted by position, so the pairs of
//         particle p are the contiguous slots around p whose tick distance is
//         <= Smax; each thread walks left and right until it leaves range.
//   cell2 (2-d cell list) candidates are the 3 x 3 block of cells around the
//         particle's cell (cell width > Smax), contiguous per row.
//   all pairs, with (BRUTE) or without (FULL, the paper's full-matrix
//         reference) the cutoff: mt_allpairs.cu.
// Precision: mixw(PR) = false is IEEE binary64 throughout; mixw(PR) = true forms
// weights and normalised weights in binary32 and updates the double-binary32
// masses with compensated additions.
#include "mt_fixed.cuh"

namespace mt {

// ------------------------------------------------------------ observables --
// After every step (every path): sum A, sum B, sum (A - B) and mean A of each
// realisation, one ring row per step (sum A and sum B are conserved by the
// symmetric transfer, sum (A - B) by the reaction too: the conservative
// components of Sec. 3).  Each realisation's slot range is cut
// into fixed chunks of kObsChunk slots (the state keeps a realisation's
// particles in its own range); a CTA sums one chunk -- each thread its
// strided slots in order, then fixed shuffle trees -- in the precision's
// own arithmetic (binary64, or double-binary32 in MIXED), and the CTA that
// completes a realisation's last chunk adds its chunk sums (thread-strided
// in order, then the block tree).  The result depends on
// the state only, not on how the step was scheduled.

// A thread's sums over its slots, in slot order: binary64, or in MIXED
// Sum2-style compensated sums of the double-binary32 masses (each high part
// added with Knuth's two-sum, the rounding errors and the low parts collected
// in a second term; as accurate here as double-binary32 additions, at a third
// of the operations).
template <int PR>
struct ThreadObs;
template <>
struct ThreadObs<false> {  // binary64 masses
  Obs3<double> v{};
  __device__ __forceinline__ void add(double a, double b) {
    v = obs3_add(v, Obs3<double>{a, b, a - b});
  }
  __device__ __forceinline__ Obs3<double> value() const { return v; }
};
template <>
struct ThreadObs<true> {  // double-binary32 masses
  kahan a{0.f, 0.f}, b{0.f, 0.f}, d{0.f, 0.f};
  static __device__ __forceinline__ void put(kahan& k, float hi, float lo) {
    const df e = two_sum(k.s, hi);
    k.s = e.hi;
    k.c = __fadd_rn(k.c, __fadd_rn(e.lo, lo));
  }
  __device__ __forceinline__ void add(df A, df B) {
    put(a, A.hi, A.lo);
    put(b, B.hi, B.lo);
    put(d, A.hi, A.lo);
    put(d, -B.hi, -B.lo);
  }
  __device__ __forceinline__ Obs3<df> value() const {
    return {fast_two_sum(a.s, a.c), fast_two_sum(b.s, b.c), fast_two_sum(d.s, d.c)};
  }
};

// PREV: the state at the step's start (obs_snapshot, by k_obs_snapshot or
// the predicted-segment kernel), while
// the step runs beside it (it writes the other mass buffer); otherwise the
// current state (left > 0: only if left - 1 of the running graph's steps are
// still to do).  Either writes the row of the step the state follows.
template <int PR, bool PREV>
__global__ void __launch_bounds__(kThreads) k_obs(Dev d, int left) {
  chained();
  using MS = Mass<PR>;
  using MV = typename MS::V;
  constexpr int kPer = kObsChunk / kThreads;  // slots per thread
  __shared__ Obs3<MV> s_w[kThreads / 32];
  __shared__ bool s_last;
  Ctrl* c = d.ctrl;
  // (both fixed before the launch: every CTA agrees)
  if (PREV && !c->obs_prev_todo) return;
  if (left > 0 && c->todo != left - 1) return;
  const unsigned long long step = PREV ? c->obs_step : c->step;
  const int ch = blockIdx.x;
  const unsigned long long* M = d.M[PREV ? c->obs_mc : c->mcur];
  // this thread's slots: loaded together, then added in slot order
  const long long a0 = d.ochunk[ch], a1 = d.ochunk[ch + 1];
  MV va[kPer], vb[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const long long p = a0 + threadIdx.x + (long long)k * kThreads;
    va[k] = p < a1 ? MS::load(M, p) : MV{};
    vb[k] = p < a1 ? MS::load(M, d.n + p) : MV{};
  }
  ThreadObs<PR == MT_MIXED_DF32> acc;
#pragma unroll
  for (int k = 0; k < kPer; ++k) acc.add(va[k], vb[k]);
  const Obs3<MV> t = obs3_block<MV, kThreads>(acc.value(), s_w);
  MV* part = reinterpret_cast<MV*>(d.opart);  // 8-byte words, 4 per chunk
  const int r = d.ochr[ch];
  const Real R = d.rt[r];
  if (threadIdx.x == 0) {
    part[4 * ch + 0] = t.a;
    part[4 * ch + 1] = t.b;
    part[4 * ch + 2] = t.d;
    __threadfence();
    s_last = atomicAdd(&d.ocnt[r], 1) + 1 == R.nch;
  }
  __syncthreads();
  if (!s_last) return;
  // the realisation's last chunk: thread t adds its chunks t, t + 256, ...
  // in order (four in flight), then the block tree
  __threadfence();
  auto get = [&](int k) {
    return Obs3<MV>{ldcg_obs(&part[4 * k + 0]), ldcg_obs(&part[4 * k + 1]),
                    ldcg_obs(&part[4 * k + 2])};
  };
  const int k1 = R.ch0 + R.nch;
  Obs3<MV> u{};
  int k = R.ch0 + threadIdx.x;
  for (; k + 3 * kThreads < k1; k += 4 * kThreads) {
    const Obs3<MV> p0 = get(k), p1 = get(k + kThreads), p2 = get(k + 2 * kThreads),
                   p3 = get(k + 3 * kThreads);
    u = obs3_add(obs3_add(obs3_add(obs3_add(u, p0), p1), p2), p3);
  }
  for (; k < k1; k += kThreads) u = obs3_add(u, get(k));
  u = obs3_block<MV, kThreads>(u, s_w);
  if (threadIdx.x == 0) {
    const long long row = (long long)((step - 1) % (unsigned long long)d.observe_cap);
    obs_row(d, row, r, R.n, u);
    d.ocnt[r] = 0;
    c->obs_done_step = step;
  }
}

__global__ void k_obs_snapshot(Dev d) { obs_snapshot(d.ctrl); }

cudaError_t launch_obs_snapshot(const Dev& d, cudaStream_t s) {
  if (d.observe_cap <= 0 || d.nochunk <= 0) return cudaSuccess;
  k_obs_snapshot<<<1, 1, 0, s>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_obs_prev(const Dev& d, int precision, cudaStream_t s) {
  if (d.observe_cap <= 0 || d.nochunk <= 0) return cudaSuccess;
  if (precision == MT_MIXED_DF32)
    k_obs<MT_MIXED_DF32, true><<<d.nochunk, kThreads, 0, s>>>(d, 0);
  else
    k_obs<MT_FP64, true><<<d.nochunk, kThreads, 0, s>>>(d, 0);  // binary64 masses
  return cudaGetLastError();
}

static cudaError_t obs_of_state(const Dev& d, int precision, int left, cudaStream_t s) {
  if (d.observe_cap <= 0 || d.nochunk <= 0) return cudaSuccess;
  if (precision == MT_MIXED_DF32)
    launch_chained(k_obs<MT_MIXED_DF32, false>, d.nochunk, kThreads, 0, s, d, left);
  else
    launch_chained(k_obs<MT_FP64, false>, d.nochunk, kThreads, 0, s, d, left);  // binary64 masses
  return cudaGetLastError();
}

cudaError_t launch_obs(const Dev& d, int precision, cudaStream_t s) {
  return obs_of_state(d, precision, 0, s);
}

cudaError_t launch_obs_step(const Dev& d, int precision, int j, int steps, cudaStream_t s) {
  return obs_of_state(d, precision, steps - j + 1, s);
}

// ================================================================ 1-d walk ==

// Calls f(q, D) for the neighbours of the particle in sorted slot p at x, left
// ones (nearest first), then right ones.  id: the particle's (periodic walls:
// the walks go around its realisation's ring; 2 Smax < L and a walk that comes
// round has crossed the wall (ring_gap), so no slot is reached from both sides).
template <class F>
__device__ __forceinline__ void walk_visit(const Dev& d, const long long* Xs, long long p,
                                           long long x, int id, F&& f) {
  if (!d.periodic) {
    for (long long q = p - 1; q >= 0; --q) {
      const long long D = x - Xs[q];
      if (D > d.S) break;
      f(q, D);
    }
    for (long long q = p + 1; q < d.n; ++q) {
      const long long D = Xs[q] - x;
      if (D > d.S) break;
      f(q, D);
    }
  } else {
    const Ring g = ring_of(d, id);
    for (long long k = 1; k < g.n; ++k) {
      const long long q = ring_step(g, p, -k);
      const long long D = ring_gap(g, q, Xs[q], p, x);
      if (D > d.S) break;
      f(q, D);
    }
    for (long long k = 1; k < g.n; ++k) {
      const long long q = ring_step(g, p, k);
      const long long D = ring_gap(g, p, x, q, Xs[q]);
      if (D > d.S) break;
      f(q, D);
    }
  }
}

constexpr int kWalkBins = 64;  // neighbour-count bins of the exchange's lanes

// Pass 1; also gathers id and masses (every species) into the sorted slots and
// leaves the neighbour count, clipped to the bins, in src.
template <int PR>
__global__ void __launch_bounds__(kThreads) k_rowsum_walk(Dev d) {
  chained();
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  if (!mixw(PR)) __syncthreads();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const long long* Xs = d.X[xc ^ 1];
  const int s = d.src[p], id = d.id[xc][s];
  gather_masses(d, mc, p, s);
  gather_species(d, mc, p, s);
  T r = T(1);  // self: nu_pp = 1
  int c = 0;
  walk_visit(d, Xs, p, Xs[p], id, [&](long long, long long D) {
    r += W::near(d, D, s_tab);
    ++c;
  });
  store_rinv<mixw(PR)>(d, p, r);
  d.id[xc ^ 1][p] = id;
  d.src[p] = c < kWalkBins ? c : kWalkBins - 1;
}

// Pass 2 for all species at once (NP pairs of them: the weights, the search and
// the reads of 1 / r serve every species): A and B (pair 0) react.  The
// binary64 instructions of a pair hold their pipe ~19 cycles per warp whatever
// lanes are active, and neighbour counts of a sparse system spread from 0 to
// twice their mean: the CTA's particles are handed to its lanes in order of
// their counts (a counting sort; each particle's sums are the same whatever
// lane forms them), which halves the warp iterations at four neighbours.
// N = 4 10^5, periodic, four species: 123 us in two passes -> 61 us (step 181 ->
// 96 us, with separations wrapped by an addition instead of a 64-bit division).
template <int PR, int NP>
__global__ void __launch_bounds__(kThreads) k_exchange_walk(Dev d) {
  chained();
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  __shared__ int s_hist[kWalkBins];
  __shared__ unsigned char s_lane[kThreads];
  const long long b0 = (long long)blockIdx.x * kThreads;
  const int n_here = (int)min((long long)kThreads, d.n - b0);
  const int tid = threadIdx.x;
  const int bin = tid < n_here ? d.src[b0 + tid] : kWalkBins - 1;
  if (tid < kWalkBins) s_hist[tid] = 0;
  __syncthreads();
  const int at = tid < n_here ? atomicAdd(&s_hist[bin], 1) : 0;
  __syncthreads();
  if (tid < 32) {
    const int h0 = s_hist[2 * tid], h1 = s_hist[2 * tid + 1];
    int inc = h0 + h1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (tid >= o) inc += t;
    }
    s_hist[2 * tid] = inc - h0 - h1;
    s_hist[2 * tid + 1] = inc - h1;
  }
  __syncthreads();
  if (tid < n_here) s_lane[s_hist[bin] + at] = (unsigned char)tid;
  __syncthreads();
  if (tid >= n_here) return;
  const long long p = b0 + s_lane[tid];
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const long long* Xs = d.X[xc ^ 1];
  const unsigned long long* M = d.M[mc ^ 1];
  unsigned long long* Mn = d.M[mc];
  // species 2 k and 2 k + 1 (an odd count repeats the last, not stored)
  const long long last = (long long)(d.nspec - 1) * d.n;
  auto off = [&](int k) { return NP == 1 ? k * d.n : min((long long)k * d.n, last); };
  const T ip = load_rinv<mixw(PR)>(d, p);
  MV m[2 * NP];
  typename MS::Acc dm[2 * NP] = {};
#pragma unroll
  for (int k = 0; k < 2 * NP; ++k) m[k] = MS::load(M, off(k) + p);
  walk_visit(d, Xs, p, Xs[p], d.periodic ? d.id[xc ^ 1][p] : 0, [&](long long q, long long D) {
    const T P = normalised<T>(d.norm, W::near(d, D, s_tab), ip, load_rinv<mixw(PR)>(d, q));
#pragma unroll
    for (int k = 0; k < 2 * NP; ++k) MS::acc(dm[k], P, MS::diff(MS::load(M, off(k) + q), m[k]));
  });
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    MS::update(m[2 * k], m[2 * k + 1], dm[2 * k], dm[2 * k + 1], k == 0 ? d.react : 0);
    MS::store(Mn, off(2 * k) + p, m[2 * k]);
    if (2 * k + 1 < d.nspec) MS::store(Mn, off(2 * k + 1) + p, m[2 * k + 1]);
  }
}

// ======================================================= 1-d dense tiles ==
// Dense neighbourhoods (tens to thousands of neighbours per particle): a CTA
// takes 256 consecutive sorted slots.  Each particle first finds its exact
// neighbour slots [jl, jr) (itself included) from the cell starts; the
// union over the CTA is one contiguous range, staged through shared memory
// in chunks of kTileChunk.  Each warp walks the union of its lanes' ranges
// with every lane reading the same slot (a shared-memory broadcast) and
// keeping the pair when the slot lies in its own range: an index test, no
// branch, and no data-dependent exit.  Inside the cutoff |dX| < 2^30, so the
// separation is the difference of the positions' low 32-bit words.  The
// particle itself adds nu_pp = 1 to r_p and an exact zero flux.

constexpr int kTileChunk = 512;
constexpr int kTileGroup = 16;  // row-sum terms added plainly before compensation

// Exact neighbour slots [jl, jr) of the particle at x: every sorted slot q
// with |X_q - x| <= Smax.  The bounds lie in the cells of x -/+ Smax.
__device__ __forceinline__ void exact_range(const Dev& d, const long long* Xs, long long x,
                                            long long& jl, long long& jr) {
  long long c = cell_of(d, x - d.S, 0);
  long long q = d.start[c], e = d.start[c + 1];
  while (q < e && Xs[q] < x - d.S) ++q;
  jl = q;
  c = cell_of(d, x + d.S, 0);
  q = d.start[c];
  e = d.start[c + 1];
  while (q < e && Xs[q] <= x + d.S) ++q;
  jr = q;
}

// The CTA's and the warp's candidate ranges from the lanes' exact ranges.
struct TileRanges {
  long long lo, hi;    // CTA: union of its particles' ranges
  long long wlo, whi;  // warp: union of its lanes' ranges (empty if no lane is valid)
};
__device__ __forceinline__ TileRanges tile_ranges(long long jl, long long jr, long long b0,
                                                  long long b1, long long* s_lohi) {
  const long long p = b0 + threadIdx.x;
  const long long w0 = b0 + (threadIdx.x & ~31);
  const int last = w0 < b1 ? (int)min(31LL, b1 - 1 - w0) : 0;
  TileRanges t;
  t.wlo = __shfl_sync(0xffffffffu, jl, 0);
  t.whi = __shfl_sync(0xffffffffu, jr, last);
  if (w0 >= b1) t.wlo = t.whi = 0;
  if (p == b0) s_lohi[0] = jl;
  if (p == b1 - 1) s_lohi[1] = jr;
  __syncthreads();
  t.lo = s_lohi[0];
  t.hi = s_lohi[1];
  return t;
}

template <int PR>
__global__ void __launch_bounds__(kThreads) k_rowsum_tile(Dev d) {
  chained();
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  __shared__ unsigned int s_x[kTileChunk];
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  __shared__ long long s_lohi[2];
  const long long b0 = (long long)blockIdx.x * kThreads;
  const long long b1 = min(b0 + (long long)kThreads, d.n);
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const long long* Xs = d.X[xc ^ 1];
  const long long p = b0 + threadIdx.x;
  const bool valid = p < b1;
  const long long x = valid ? Xs[p] : 0;
  long long jl = 0, jr = 0;
  if (valid) exact_range(d, Xs, x, jl, jr);
  const TileRanges t = tile_ranges(jl, jr, b0, b1, s_lohi);
  const unsigned int x32 = (unsigned int)x;
  // The weights are summed plainly in groups of kTileGroup candidates (two
  // chains) and each group's sum enters a compensated sum: the group sums'
  // rounding (at most kTileGroup terms of at most 1) stays near binary32's
  // precision relative to r_p, at a plain addition per weight.
  RowSum<mixw(PR)> r(T(0));
  for (long long c0 = t.lo; c0 < t.hi; c0 += kTileChunk) {
    const int nc = (int)min((long long)kTileChunk, t.hi - c0);
    for (int i = threadIdx.x; i < nc; i += kThreads) s_x[i] = (unsigned int)Xs[c0 + i];
    __syncthreads();
    const int j0 = (int)(max(t.wlo, c0) - c0), j1 = (int)(min(t.whi, c0 + nc) - c0);
    const int ql = (int)(jl - c0);
    const unsigned int qn = (unsigned int)(jr - jl);
    auto term = [&](int j) {
      const T w = W::near(d, (int)(s_x[j] - x32), s_tab);
      return (unsigned int)(j - ql) < qn ? w : T(0);
    };
    int j = j0;
    for (; j + kTileGroup <= j1; j += kTileGroup) {
      T g0 = T(0), g1 = T(0);
#pragma unroll
      for (int k = 0; k < kTileGroup; k += 2) {
        g0 += term(j + k);
        g1 += term(j + k + 1);
      }
      r.add(g0 + g1);
    }
    T g = T(0);
    for (; j < j1; ++j) g += term(j);
    r.add(g);
    __syncthreads();
  }
  if (!valid) return;
  store_rinv<mixw(PR)>(d, p, r.value());
  const int s = d.src[p];
  d.id[xc ^ 1][p] = d.id[xc][s];
  gather_masses(d, mc, p, s);
}

template <int PR, bool TR>
__global__ void __launch_bounds__(kThreads) k_exchange_tile(Dev d, int sp) {
  chained();
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ unsigned int s_x[kTileChunk];
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  __shared__ T s_r[kTileChunk];
  __shared__ MV s_a[kTileChunk];
  __shared__ MV s_b[kTileChunk];
  __shared__ long long s_lohi[2];
  const long long b0 = (long long)blockIdx.x * kThreads;
  const long long b1 = min(b0 + (long long)kThreads, d.n);
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const SpeciesPair sq = species_pair<TR>(d, sp);
  const long long* Xs = d.X[xc ^ 1];
  const unsigned long long* MA = d.M[mc ^ 1] + sq.oa;
  const unsigned long long* MB = d.M[mc ^ 1] + sq.ob;
  const long long p = b0 + threadIdx.x;
  const bool valid = p < b1;
  const long long x = valid ? Xs[p] : 0;
  long long jl = 0, jr = 0;
  if (valid) exact_range(d, Xs, x, jl, jr);
  const TileRanges t = tile_ranges(jl, jr, b0, b1, s_lohi);
  const unsigned int x32 = (unsigned int)x;
  // SYM: P = w (1/(2 r_p) + 1/(2 r_q)), the halves exact; ROW: P = w / r_p (the
  // staged 1/r_q is 0).  (Sums of 2 P overflow for masses beyond half of
  // binary64's range, whose weighted means are finite.)
  const bool sym = d.norm != MT_NORM_ROW;
  const T scale = sym ? T(0.5) : T(1);
  MV A{}, B{};
  T ip = T(0);
  if (valid) {
    A = MS::load(MA, p);
    B = MS::load(MB, p);
    ip = scale * load_rinv<mixw(PR)>(d, p);
  }
  // two accumulator sets (even and odd candidates) halve the dependent
  // chain of compensated additions
  typename MS::Acc dA{}, dB{}, dA1{}, dB1{};
  for (long long c0 = t.lo; c0 < t.hi; c0 += kTileChunk) {
    const int nc = (int)min((long long)kTileChunk, t.hi - c0);
    for (int i = threadIdx.x; i < nc; i += kThreads) {
      s_x[i] = (unsigned int)Xs[c0 + i];
      s_r[i] = sym ? scale * load_rinv<mixw(PR)>(d, c0 + i) : T(0);
      s_a[i] = MS::load(MA, c0 + i);
      s_b[i] = MS::load(MB, c0 + i);
    }
    __syncthreads();
    const int j0 = (int)(max(t.wlo, c0) - c0), j1 = (int)(min(t.whi, c0 + nc) - c0);
    const int ql = (int)(jl - c0);
    const unsigned int qn = (unsigned int)(jr - jl);
    auto pair = [&](int j, typename MS::Acc& a, typename MS::Acc& b) {
      const T w = W::near(d, (int)(s_x[j] - x32), s_tab);
      const T P = (unsigned int)(j - ql) < qn ? w * (ip + s_r[j]) : T(0);
      MS::acc(a, P, MS::diff(s_a[j], A));
      MS::acc(b, P, MS::diff(s_b[j], B));
    };
    int j = j0;
    for (; j + 1 < j1; j += 2) {
      pair(j, dA, dB);
      pair(j + 1, dA1, dB1);
    }
    if (j < j1) pair(j, dA, dB);
    __syncthreads();
  }
  dA = acc_merge(dA, dA1);
  dB = acc_merge(dB, dB1);
  if (valid) {
    MS::update(A, B, dA, dB, TR ? 0 : d.react);
    MS::store(d.M[mc] + sq.oa, p, A);
    if (sq.store_b) MS::store(d.M[mc] + sq.ob, p, B);
  }
  if (!TR) finish_step(d, 1, 0);
}

// MT_MIXED's exchange over the same tiles with the flux sums in exact integer
// arithmetic (mt_fixed.cuh): the binary64 form above spends its time in four
// binary64 instructions per ordered pair (~76 of ~80 cycles per warp and
// pair at the paper's density); here a pair is ~55 integer and binary32
// instructions, issue-bound.  Each chunk's masses, and the rows' own, are
// converted with the largest exponent among them, and a chunk's sum is rounded
// to binary64 once.  Where the chunk, or a row, has marked masses, their rests are
// summed too, in binary32 (six instructions more).  A lane whose sum still does
// not outweigh its error (FixAcc::keeps: deep in a front's tail) sums the chunk
// again, in binary64, a species at a time.  N = 10^6 at 200 per unit length: 4.09 ->
// 1.09 ms (step 4.47 -> 1.42 ms); 27 realisations of 5000, two segregated
// components, eighth step: 162 us (without rests, rows of small masses in
// binary64: 196).
template <bool TR>
__global__ void __launch_bounds__(kThreads, 4) k_exchange_tile_fix(Dev d, int sp) {
  chained();
  using W = Weight<true, 1>;
  using MS = Mass<MT_MIXED>;
  constexpr int kWarps = kThreads / 32, kPer = kTileChunk / kThreads;
  __shared__ uint2 s_xr[kTileChunk];       // low word of the position, 1 / r
  __shared__ longlong2 s_ab[kTileChunk];   // fixed masses
  __shared__ float2 s_rest[kTileChunk];    // their rests, where the chunk has marked masses
  __shared__ long long s_lohi[2];
  __shared__ int s_e[kWarps][2];  // largest exponents
  __shared__ int s_mark[2];       // fix_flags of the chunk's masses
  const long long b0 = (long long)blockIdx.x * kThreads;
  const long long b1 = min(b0 + (long long)kThreads, d.n);
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const SpeciesPair sq = species_pair<TR>(d, sp);
  const long long* Xs = d.X[xc ^ 1];
  const unsigned long long* MA = d.M[mc ^ 1] + sq.oa;
  const unsigned long long* MB = d.M[mc ^ 1] + sq.ob;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long p = b0 + threadIdx.x;
  const bool valid = p < b1;
  const long long x = valid ? Xs[p] : 0;
  long long jl = 0, jr = 0;
  if (valid) exact_range(d, Xs, x, jl, jr);
  const TileRanges t = tile_ranges(jl, jr, b0, b1, s_lohi);
  const unsigned int x32 = (unsigned int)x;
  // SYM: the integer sums take 2 P and are halved; the binary64 sums take P
  // (those of 2 P overflow for masses beyond half of binary64's range)
  const bool sym = d.norm != MT_NORM_ROW;
  const float p_scale = sym ? 0.5f : 1.0f;
  const unsigned long long Ab = valid ? MA[p] : 0, Bb = valid ? MB[p] : 0;
  const float ip = valid ? load_rinv<true>(d, p) : 0.0f;
  double dA = 0.0, dB = 0.0;
  for (long long c0 = t.lo; c0 < t.hi; c0 += kTileChunk) {
    const int nc = (int)min((long long)kTileChunk, t.hi - c0);
    unsigned long long va[kPer], vb[kPer];
    int ea = fix_exponent(Ab), eb = fix_exponent(Bb);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = threadIdx.x + k * kThreads;
      va[k] = i < nc ? MA[c0 + i] : 0;
      vb[k] = i < nc ? MB[c0 + i] : 0;
      if (i < nc) {
        s_xr[i] = make_uint2((unsigned int)Xs[c0 + i],
                             sym ? __float_as_uint(load_rinv<true>(d, c0 + i)) : 0u);
      }
      ea = max(ea, fix_exponent(va[k]));
      eb = max(eb, fix_exponent(vb[k]));
    }
    ea = __reduce_max_sync(0xffffffffu, ea);
    eb = __reduce_max_sync(0xffffffffu, eb);
    if (lane == 0) {
      s_e[warp][0] = ea;
      s_e[warp][1] = eb;
    }
    if (threadIdx.x < 2) s_mark[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      ea = max(ea, s_e[w][0]);
      eb = max(eb, s_e[w][1]);
    }
    const int EA = fix_scale(ea), EB = fix_scale(eb);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = threadIdx.x + k * kThreads;
      const long long fa = to_fix(va[k], EA), fb = to_fix(vb[k], EB);
      s_ab[i] = make_longlong2(fa, fb);
      const int ma = __reduce_or_sync(0xffffffffu, fix_flags(fa));
      const int mb = __reduce_or_sync(0xffffffffu, fix_flags(fb));
      if (lane == 0) {
        if (ma) atomicOr(&s_mark[0], ma);
        if (mb) atomicOr(&s_mark[1], mb);
      }
    }
    const long long fa = to_fix(Ab, EA), fb = to_fix(Bb, EB);
    // (every lane stages the rests if any has a marked mass: its own may lie in
    // another chunk)
    const bool rests = __syncthreads_or(((s_mark[0] | s_mark[1]) & 1) || ((fa | fb) & 1));
    if (rests) {
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int i = threadIdx.x + k * kThreads;
        s_rest[i] = i < nc ? make_float2(fix_rest(MA[c0 + i], EA), fix_rest(MB[c0 + i], EB))
                           : make_float2(0.0f, 0.0f);
      }
      __syncthreads();
    }
    const int j0 = (int)(max(t.wlo, c0) - c0), j1 = (int)(min(t.whi, c0 + nc) - c0);
    const int ql = (int)(jl - c0);
    const unsigned int qn = (unsigned int)(jr - jl);
    // this lane's slots of the chunk
    const int l0 = (int)(max(jl, c0) - c0), l1 = (int)(min(jr, c0 + nc) - c0);
    FixAcc qa, qb;
    if (!rests) {
#pragma unroll 2
      for (int j = j0; j < j1; ++j) {
        const uint2 xr = s_xr[j];
        const longlong2 ab = s_ab[j];
        const float w = W::near(d, (int)(xr.x - x32), nullptr);
        FixP P = fix_p(w * (ip + __uint_as_float(xr.y)));
        if ((unsigned int)(j - ql) >= qn) P.p = 0;
        qa.add(ab.x - fa, P);
        qb.add(ab.y - fb, P);
      }
    } else {
      const float ra = fix_rest(Ab, EA), rb = fix_rest(Bb, EB);
      float sa = 0.0f, sb = 0.0f;
#pragma unroll 2
      for (int j = j0; j < j1; ++j) {
        const uint2 xr = s_xr[j];
        const longlong2 ab = s_ab[j];
        const float2 rest = s_rest[j];
        const float w = W::near(d, (int)(xr.x - x32), nullptr);
        float Pf = w * (ip + __uint_as_float(xr.y));
        FixP P = fix_p(Pf);
        if ((unsigned int)(j - ql) >= qn) {
          P.p = 0;
          Pf = 0.0f;
        }
        qa.add(ab.x - fa, P);
        qb.add(ab.y - fb, P);
        sa = __fmaf_rn(Pf, rest.x - ra, sa);
        sb = __fmaf_rn(Pf, rest.y - rb, sb);
      }
      qa.add_rest(sa);
      qb.add_rest(sb);
    }
    if (l0 < l1) {
      // (halved in the exponent, which is far from binary64's ends)
      double ca = qa.value(EA - sym), cb = qb.value(EB - sym);
      const int halvings = sym ? 2 : 1;
      const bool one = ip >= 0x1p-19f;
      const bool fixa = fix_covers(EA) && qa.keeps(fa, halvings, s_mark[0] | fix_flags(fa), one);
      const bool fixb = fix_covers(EB) && qb.keeps(fb, halvings, s_mark[1] | fix_flags(fb), one);
      // (a species at a time: in a tail of one the other is large)
      auto again = [&](const unsigned long long* M, double own) {
        double sum = 0.0;
#pragma unroll 1
        for (int j = l0; j < l1; ++j) {
          const float P = W::near(d, (int)(s_xr[j].x - x32), nullptr) *
                          (ip + __uint_as_float(s_xr[j].y)) * p_scale;
          MS::acc(sum, P, MS::diff(MS::load(M, c0 + j), own));
        }
        return sum;
      };
      if (!fixa) ca = again(MA, __longlong_as_double((long long)Ab));
      if (!fixb) cb = again(MB, __longlong_as_double((long long)Bb));
      dA += ca;
      dB += cb;
    }
    __syncthreads();
  }
  if (valid) {
    double A = __longlong_as_double((long long)Ab), B = __longlong_as_double((long long)Bb);
    MS::update(A, B, dA, dB, TR ? 0 : d.react);
    MS::store(d.M[mc] + sq.oa, p, A);
    if (sq.store_b) MS::store(d.M[mc] + sq.ob, p, B);
  }
  if (!TR) finish_step(d, 1, 0);
}

template <int PR, bool TR>
static void launch_exchange_tile(const Dev& d, unsigned int g, cudaStream_t s, int sp) {
  if constexpr (PR == MT_MIXED) {
    if (d.fix) {
      k_exchange_tile_fix<TR><<<g, kThreads, 0, s>>>(d, sp);
      return;
    }
  }
  k_exchange_tile<PR, TR><<<g, kThreads, 0, s>>>(d, sp);
}

// ================================================== 1-d SPaM (stored P) ==
// The SPaM form of Sec. 6: the nonzero weights of the step's transfer
// matrix are stored and both passes read them, so each unordered pair's
// exponential is evaluated once.  In sorted order the nonzeros of row p are
// the contiguous slots around p: cnt_l(p) to the left and cnt_r(p) to the
// right.  The band keeps nu(p, p + k), k = 1 .. min(cnt_r(p), band_cap), in
// tiles of 32 slots: entry (p, k) is at ((p / 32) band_cap + k - 1) 32 +
// p % 32, so a warp reading its right neighbours streams one contiguous
// block, and reading its left neighbours (entries (p - k, k)) streams two
// adjacent ones.  Weights past the band are recomputed from the positions.
//   band_build     right neighbours: nu stored, right part of r_p, cnt_r;
//                  left count cnt_l; ids and masses into the sorted slots
//   band_rowsum    left part of r_p from the band -> 1 / r_p
//   band_exchange  Eq. 4 / 7 with the stored weights

__device__ __forceinline__ long long band_at(const Dev& d, long long q, long long k) {
  return (((q >> 5) * d.band_cap) + (k - 1)) * 32 + (q & 31);
}

// The slots a particle's walks cover: with periodic walls its realisation's
// ring; else the whole sorted range (realisations are separated by more than
// Smax, so the cutoff ends every walk inside its own realisation).
__device__ __forceinline__ Ring walk_ring(const Dev& d, int id) {
  return d.periodic ? ring_of(d, id) : Ring{0, d.n, 0};
}

// Slot k steps to the right (left for k < 0) of p.
__device__ __forceinline__ long long ring(const Dev& d, const Ring& g, long long p, long long k) {
  return d.periodic ? ring_step(g, p, k) : p + k;
}

// The longest right and left walks from slot p.
__device__ __forceinline__ long long walk_right(const Dev& d, const Ring& g, long long p) {
  return d.periodic ? g.n - 1 : d.n - 1 - p;
}
__device__ __forceinline__ long long walk_left(const Dev& d, const Ring& g, long long p) {
  return d.periodic ? g.n - 1 : p;
}

// Tick distance from slot q up to slot p (p to the right of q; reflecting walls:
// a higher slot).
__device__ __forceinline__ long long gap(const Ring& g, const long long* Xs, long long q,
                                         long long p) {
  return ring_gap(g, q, Xs[q], p, Xs[p]);
}

template <int PR>
__global__ void __launch_bounds__(kThreads) k_band_build(Dev d) {
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  if (!mixw(PR)) __syncthreads();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const long long* Xs = d.X[xc ^ 1];
  T* band = static_cast<T*>(d.band);
  const int s = d.src[p];
  const Ring g = walk_ring(d, d.id[xc][s]);
  RowSum<mixw(PR)> r(T(0));
  long long k = 1;
  const long long kr = walk_right(d, g, p);
  for (; k <= kr; ++k) {
    const long long D = gap(g, Xs, p, ring(d, g, p, k));
    if (D > d.S) break;
    const T w = W::near(d, D, s_tab);
    if (k <= d.band_cap) band[band_at(d, p, k)] = w;
    r.add(w);
  }
  d.cnt[p] = (int)(k - 1);
  const long long kl = walk_left(d, g, p);
  for (k = 1; k <= kl; ++k)
    if (gap(g, Xs, ring(d, g, p, -k), p) > d.S) break;
  d.cnt[d.n + p] = (int)(k - 1);
  static_cast<T*>(d.rinv)[p] = r.value();  // right part of r_p, completed by band_rowsum
  d.id[xc ^ 1][p] = d.id[xc][s];
  gather_masses(d, mc, p, s);
}

template <int PR>
__global__ void __launch_bounds__(kThreads) k_band_rowsum(Dev d) {
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  if (!mixw(PR)) __syncthreads();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const T* band = static_cast<const T*>(d.band);
  const int xc = d.ctrl->xcur;
  const Ring g = walk_ring(d, d.id[xc ^ 1][p]);
  RowSum<mixw(PR)> r(T(1));  // self
  r.add(static_cast<const T*>(d.rinv)[p]);  // right part
  const int kl = d.cnt[d.n + p];
  const int kb = kl < d.band_cap ? kl : d.band_cap;
#pragma unroll 4
  for (int k = 1; k <= kb; ++k) r.add(band[band_at(d, ring(d, g, p, -k), k)]);
  if (kl > kb) {
    const long long* Xs = d.X[xc ^ 1];
    for (int k = kb + 1; k <= kl; ++k) r.add(W::near(d, gap(g, Xs, ring(d, g, p, -k), p), s_tab));
  }
  store_rinv<mixw(PR)>(d, p, r.value());
}

// (MT_MIXED_DF32 is compiled for five CTAs per SM: 1.9 10^5 particles at 116 per unit
// length 575 -> 455 us per step, five species 1250 -> 876.  The wall's length is read
// again where weights past the band need it, so that it holds no registers in
// the loops over the band.)
template <int PR, bool TR>
__global__ void __launch_bounds__(kThreads, PR == MT_MIXED_DF32 ? 5 : 0)
    k_band_exchange(Dev d, int sp) {
  using W = Weight<mixw(PR), 1>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) exp_table<kThreads>(s_tab);
  if (!mixw(PR)) __syncthreads();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  const bool valid = p < d.n;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const SpeciesPair sq = species_pair<TR>(d, sp);
  MV A{}, B{};
  if (valid) {
    const long long* Xs = d.X[xc ^ 1];
    const Ring g = walk_ring(d, d.id[xc ^ 1][p]);
    const unsigned long long* MA = d.M[mc ^ 1] + sq.oa;
    const unsigned long long* MB = d.M[mc ^ 1] + sq.ob;
    const T* band = static_cast<const T*>(d.band);
    const T ip = load_rinv<mixw(PR)>(d, p);
    A = MS::load(MA, p);
    B = MS::load(MB, p);
    typename MS::Acc dA{}, dB{};
    auto pair = [&](long long q, T w) {
      const T P = normalised<T>(d.norm, w, ip, load_rinv<mixw(PR)>(d, q));
      MS::acc(dA, P, MS::diff(MS::load(MA, q), A));
      MS::acc(dB, P, MS::diff(MS::load(MB, q), B));
    };
    auto wall = [&]() -> long long { return d.periodic ? ring_of(d, d.id[xc ^ 1][p]).Lq : 0; };
    const int kl = d.cnt[d.n + p], kr = d.cnt[p];
    const int bl = kl < d.band_cap ? kl : d.band_cap;
    const int br = kr < d.band_cap ? kr : d.band_cap;
#pragma unroll 2
    for (int k = 1; k <= bl; ++k) {
      const long long q = ring(d, g, p, -k);
      pair(q, band[band_at(d, q, k)]);
    }
    if (kl > bl) {
      const long long x = Xs[p], Lq = wall();
      for (int k = bl + 1; k <= kl; ++k) {
        const long long q = ring(d, g, p, -k);
        pair(q, W::near(d, x - Xs[q] + (p < q ? Lq : 0), s_tab));
      }
    }
#pragma unroll 2
    for (int k = 1; k <= br; ++k) pair(ring(d, g, p, k), band[band_at(d, p, k)]);
    if (kr > br) {
      const long long x = Xs[p], Lq = wall();
      for (int k = br + 1; k <= kr; ++k) {
        const long long q = ring(d, g, p, k);
        pair(q, W::near(d, Xs[q] - x + (q < p ? Lq : 0), s_tab));
      }
    }
    MS::update(A, B, dA, dB, TR ? 0 : d.react);
    MS::store(d.M[mc] + sq.oa, p, A);
    if (sq.store_b) MS::store(d.M[mc] + sq.ob, p, B);
  }
  if (!TR) finish_step(d, 1, 0);
}

// =============================================================== 2-d cells ==
// The sort has put positions, ids and masses into the cells' slots.  Pass 1
// forms the row sums and notes each particle's neighbours in src (free after
// the sort): kNone, the slot of the only one, or kMany; it lists the particles
// that have any (in the old positions' buffer, free after the sort; the count
// in Ctrl::nbig, reset by the move).  Pass 2 streams the masses of the others
// through the reaction -- in the sparse systems of the workloads (0.1
// neighbours per particle) nine in ten -- and works off the list with full
// warps, so that the binary64 instructions of the exchange are issued for
// warps of particles that need them.  N = 10^6 at one particle per 100 units of
// area: pass 1 43 -> 31 us (all cell starts loaded ahead, one loop over all
// candidates, a box test of two subtractions per axis), pass 2 51 -> 16 us.
constexpr int kNone = -1, kMany = -2;

// Calls f(q, dx, dy) for every other slot q within the cutoff of slot p at
// (x, y), and self() for p, in slot order: the 3 x 3 block of cells around its
// cell (reflecting walls), or the wrapped cell spans (PER, minimum-image
// separations).  (The lanes of a warp meet themselves in different
// iterations: with p among the pairs, nearly every iteration evaluated a
// weight.)  AHEAD: a candidate's coordinates are loaded while the one before it
// is tested, since a warp with many candidates (a pile) waits for them: 10^4
// particles, most in a few cells, MT_MIXED 1057 -> 873 us per step (with the three
// runs' loops before: 931), and 30000 at one per unit of area 58 -> 54;
// MT_MIXED_DF32's exchange and MT_MIXED's of further species, which have no
// registers left for it, do without (DF32, 10^6 at one per unit of area: 293 against
// 282 us).
template <bool PER, bool AHEAD, class F, class G>
__device__ __forceinline__ void cell2_visit(const Dev& d, const long long* Xs, int p, long long x,
                                            long long y, F&& f, G&& self) {
  if (PER) {
    cells2_visit(d, x, y, [&](int q0, int q1) {
      long long xn = q0 < q1 ? Xs[q0] : 0, yn = q0 < q1 ? Xs[d.n + q0] : 0;
      for (int q = q0; q < q1; ++q) {
        const long long dx = min_image(xn - x, d.Lq[0]);
        const long long dy = min_image(yn - y, d.Lq[1]);
        if (q + 1 < q1) {
          xn = Xs[q + 1];
          yn = Xs[d.n + q + 1];
        }
        if (q == p) {
          self();
          continue;
        }
        if (in_range2(dx, dy, d.S)) f(q, dx, dy);
      }
    });
    return;
  }
  const int ncx = (int)d.ncx, ncy = (int)d.ncy;  // (at most 2^28 cells)
  const int kx = min((int)(x >> d.cshift), ncx - 1), ky = min((int)(y >> d.cshift), ncy - 1);
  const int kx0 = max(kx - 1, 0), kx1 = min(kx + 1, ncx - 1);
  int a[3], b[3];  // the rows' runs of slots, loaded together
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int row = ky - 1 + i;
    const bool in = row >= 0 && row < ncy;
    a[i] = in ? d.start[row * ncx + kx0] : 0;
    b[i] = in ? d.start[row * ncx + kx1 + 1] : 0;
  }
  // one loop over the three runs, so that a warp's lanes wait for the longest
  // sum of runs and not for the longest of each
  const int n0 = max(b[0] - a[0], 0), n1 = n0 + max(b[1] - a[1], 0), n2 = n1 + max(b[2] - a[2], 0);
  const int o1 = a[1] - n0, o2 = a[2] - n1;
  // the box |dx|, |dy| <= S: X_q - (x - S) in [0, 2 S], 2 S < 2^31
  const unsigned long long x0 = (unsigned long long)(x - d.S), y0 = (unsigned long long)(y - d.S);
  const unsigned int S2 = 2u * (unsigned int)d.S;
  const long long* Ys = Xs + d.n;
  auto slot = [&](int t) { return t + (t < n0 ? a[0] : t < n1 ? o1 : o2); };
  int next = AHEAD && n2 > 0 ? slot(0) : 0;
  long long xn = AHEAD && n2 > 0 ? Xs[next] : 0, yn = AHEAD && n2 > 0 ? Ys[next] : 0;
#pragma unroll 2
  for (int t = 0; t < n2; ++t) {
    const int q = AHEAD ? next : slot(t);
    if (!AHEAD && q == p) {
      self();
      continue;
    }
    const unsigned long long ux = (unsigned long long)(AHEAD ? xn : Xs[q]) - x0;
    const unsigned long long uy = (unsigned long long)(AHEAD ? yn : Ys[q]) - y0;
    if (AHEAD && t + 1 < n2) {
      next = slot(t + 1);
      xn = Xs[next];
      yn = Ys[next];
    }
    if (AHEAD && q == p) {
      self();
      continue;
    }
    if ((unsigned int)(ux >> 32) | (unsigned int)(uy >> 32)) continue;
    if ((unsigned int)ux > S2 || (unsigned int)uy > S2) continue;
    const int dx = (int)((unsigned int)ux - (unsigned int)d.S);
    const int dy = (int)((unsigned int)uy - (unsigned int)d.S);
    if ((unsigned long long)((long long)dx * dx) + (unsigned long long)((long long)dy * dy) <=
        (unsigned long long)d.S * (unsigned long long)d.S)
      f(q, dx, dy);
  }
}

template <int PR, bool PER>
__global__ void __launch_bounds__(kThreads) k_rowsum_cell2(Dev d) {
  chained();
  using W = Weight<mixw(PR), 2>;
  using T = typename W::T;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) {
    exp_table<kThreads>(s_tab);
    __syncthreads();
  }
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  const int xc = d.ctrl->xcur;
  int nb = kNone;
  if (p < d.n) {
    const long long* Xs = d.X[xc ^ 1];
    T r = T(0);
    int found = 0;
    cell2_visit<PER, true>(
        d, Xs, (int)p, Xs[p], Xs[d.n + p],
        [&](int q, long long dx, long long dy) {
          r += W::near2(d, dx, dy, s_tab);
          nb = found++ == 0 ? q : kMany;
        },
        [&] { r += T(1); });
    d.src[p] = nb;
    store_rinv<mixw(PR)>(d, p, r);
  }
  // the list of particles with neighbours, a CTA's together (one atomic per
  // warp on one address held the pass at 39 us)
  __shared__ int s_count[kThreads / 32], s_at;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned int m = __ballot_sync(0xffffffffu, nb != kNone);
  if (lane == 0) s_count[warp] = __popc(m);
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) {
    if (w < warp) before += s_count[w];
    total += s_count[w];
  }
  if (threadIdx.x == 0 && total > 0) s_at = atomicAdd(&d.ctrl->nbig, total);
  __syncthreads();
  if (nb != kNone)
    reinterpret_cast<int*>(d.X[xc])[s_at + before + __popc(m & ((1u << lane) - 1u))] = (int)p;
}

template <int PR, bool TR, bool PER>
__global__ void __launch_bounds__(kThreads) k_exchange_cell2(Dev d, int sp) {
  chained();
  using W = Weight<mixw(PR), 2>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ unsigned long long s_tab[exp_tab_words(PR)];
  if (!mixw(PR)) {
    exp_table<kThreads>(s_tab);
    __syncthreads();
  }
  const long long g = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (g >= d.n) return;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const SpeciesPair sq = species_pair<TR>(d, sp);
  const unsigned long long* MA = d.M[mc ^ 1] + sq.oa;
  const unsigned long long* MB = d.M[mc ^ 1] + sq.ob;
  auto store = [&](long long p, MV A, MV B) {
    MS::store(d.M[mc] + sq.oa, p, A);
    if (sq.store_b) MS::store(d.M[mc] + sq.ob, p, B);
  };
  if (d.src[g] == kNone) {
    MV A = MS::load(MA, g), B = MS::load(MB, g);
    if (!TR && d.react) MS::react(A, B);
    store(g, A, B);
  }
  if (g >= d.ctrl->nbig) return;
  // the list: one entry per thread of the first CTAs
  const long long p = reinterpret_cast<const int*>(d.X[xc])[g];
  const long long* Xs = d.X[xc ^ 1];
  const int nb = d.src[p];
  MV A = MS::load(MA, p), B = MS::load(MB, p);
  typename MS::Acc dA{}, dB{};
  const long long x = Xs[p], y = Xs[d.n + p];
  const T ip = load_rinv<mixw(PR)>(d, p);
  auto pair = [&](int q, long long dx, long long dy) {
    const T P = normalised<T>(d.norm, W::near2(d, dx, dy, s_tab), ip, load_rinv<mixw(PR)>(d, q));
    MS::acc(dA, P, MS::diff(MS::load(MA, q), A));
    MS::acc(dB, P, MS::diff(MS::load(MB, q), B));
  };
  if (nb >= 0) {
    long long dx = Xs[nb] - x, dy = Xs[d.n + nb] - y;
    if (PER) {
      dx = min_image(dx, d.Lq[0]);
      dy = min_image(dy, d.Lq[1]);
    }
    pair(nb, dx, dy);
  } else {
    cell2_visit<PER, !mixw(PR) || (PR == MT_MIXED && !TR)>(d, Xs, (int)p, x, y, pair, [] {});
  }
  MS::update(A, B, dA, dB, TR ? 0 : d.react);
  store(p, A, B);
}

// The end of a step whose passes leave it to a kernel of its own: a fence, an
// atomic on one address and a wait in every CTA of a large pass cost more
// (10^6 particles: ~10 us) than a launch.
__global__ void k_finish(Dev d, int flip_x, int flip_m) {
  chained();
  Ctrl* c = d.ctrl;
  c->step += 1;
  c->xcur ^= flip_x;
  c->mcur ^= flip_m;
}

// Species 2 and up into the sorted slots (the row-sum pass moved A and B).
__global__ void __launch_bounds__(kThreads) k_gather_species(Dev d) {
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  gather_species(d, d.ctrl->mcur, p, d.src[p]);
}

// --------------------------------------------------------------- launch --

template <int PR, bool PER>
static void cell2_passes(const Dev& d, unsigned int g, cudaStream_t s, Marker& mk) {
  mk("rowsum_cell2", s);
  launch_chained<kChainedCells>(k_rowsum_cell2<PR, PER>, g, kThreads, 0, s, d);
  for (int sp = 2; sp < d.nspec; sp += 2) {
    mk("exchange_cell2_species", s);
    launch_chained<kChainedCells>(k_exchange_cell2<PR, true, PER>, g, kThreads, 0, s, d, sp);
  }
  mk("exchange_cell2", s);
  launch_chained<kChainedCells>(k_exchange_cell2<PR, false, PER>, g, kThreads, 0, s, d, 0);
  launch_chained(k_finish, 1, 1, 0, s, d, 1, 0);
}

// The extra species' passes (pairs 2-3, 4-5, ...) run between the row sums
// and the A/B pass, which ends the step.
template <int PR>
static void transfer_t(const Dev& d, cudaStream_t s, Marker& mk) {
  const unsigned int g = (unsigned int)((d.n + kThreads - 1) / kThreads);
  if (d.dim == 1 && d.band_cap > 0) {
    mk("band_build", s);
    k_band_build<PR><<<g, kThreads, 0, s>>>(d);
    mk("band_rowsum", s);
    k_band_rowsum<PR><<<g, kThreads, 0, s>>>(d);
    if (d.nspec > 2) {
      mk("gather_species", s);
      k_gather_species<<<g, kThreads, 0, s>>>(d);
    }
    for (int sp = 2; sp < d.nspec; sp += 2) {
      mk("band_exchange_species", s);
      k_band_exchange<PR, true><<<g, kThreads, 0, s>>>(d, sp);
    }
    mk("band_exchange", s);
    k_band_exchange<PR, false><<<g, kThreads, 0, s>>>(d, 0);
  } else if (d.dim == 1 && d.tile) {
    mk("rowsum_tile", s);
    k_rowsum_tile<PR><<<g, kThreads, 0, s>>>(d);
    if (d.nspec > 2) {
      mk("gather_species", s);
      k_gather_species<<<g, kThreads, 0, s>>>(d);
    }
    for (int sp = 2; sp < d.nspec; sp += 2) {
      mk("exchange_tile_species", s);
      launch_exchange_tile<PR, true>(d, g, s, sp);
    }
    mk("exchange_tile", s);
    launch_exchange_tile<PR, false>(d, g, s, 0);
  } else if (d.dim == 1) {
    mk("rowsum_walk", s);
    launch_chained(k_rowsum_walk<PR>, g, kThreads, 0, s, d);
    mk("exchange_walk", s);
    if (d.nspec <= 2)
      launch_chained(k_exchange_walk<PR, 1>, g, kThreads, 0, s, d);
    else if (d.nspec <= 4)
      launch_chained(k_exchange_walk<PR, 2>, g, kThreads, 0, s, d);
    else if (d.nspec <= 6)
      launch_chained(k_exchange_walk<PR, 3>, g, kThreads, 0, s, d);
    else
      launch_chained(k_exchange_walk<PR, 4>, g, kThreads, 0, s, d);
    launch_chained(k_finish, 1, 1, 0, s, d, 1, 0);
  } else if (d.periodic) {
    cell2_passes<PR, true>(d, g, s, mk);
  } else {
    cell2_passes<PR, false>(d, g, s, mk);
  }
}

cudaError_t launch_transfer(const Dev& d, int search, int precision, cudaStream_t s,
                            Marker& mk) {
  if (search != MT_SEARCH_CELL)
    return launch_allpairs(d, search == MT_SEARCH_BRUTE, precision, s, mk);
  if (precision == MT_MIXED) {
    transfer_t<MT_MIXED>(d, s, mk);
  } else if (precision == MT_MIXED_DF32) {
    transfer_t<MT_MIXED_DF32>(d, s, mk);
  } else {
    transfer_t<MT_FP64>(d, s, mk);
  }
  return cudaGetLastError();
}

}  // namespace mt
