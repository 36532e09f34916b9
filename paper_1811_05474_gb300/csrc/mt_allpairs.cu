// mt_allpairs.cu -- the all-pairs searches (MT_SEARCH_BRUTE: every pair
// tested against the cutoff; MT_SEARCH_FULL: the paper's full matrix, Sec.
// 1.1) as a scan over all pairs that keeps the pairs with a nonzero weight.
//
// Every ordered pair (p, j) is tested; the weight (Eq. 3) is evaluated for
// the pairs that can have one: within the cutoff, or without a cutoff within
// Z ticks, beyond which exp(-s^2 / (8 D_mt dt)) is exactly 0 in the weights'
// precision (binary32: exponents above 110, binary64: above 746), so that the
// pair adds exact zeros to the row sum and the exchange.  At the usual
// densities that is a handful of pairs per row out of 10^3 to 10^5.
//
// A warp takes R rows.  Positions are staged in shared memory as 32-bit
// coarse coordinates X >> sh, one j per lane, and the test per pair is a
// subtraction and an unsigned comparison: it bounds the scan, about 2.5 warp
// instructions per 32 pairs with R = 8.  A lane's candidates are appended,
// in the order of j, to the row's list in shared memory (a ballot and a
// prefix count), and a full list is worked off 32 entries at a time with the
// exact 64-bit test and the weight.  Row sums in binary32 add the list's
// nonzero weights one by one in the order of j, the order (and the bits) of
// a plain loop over j; binary64 sums and the flux sums use lane partials and
// a fixed shuffle tree.
//
// Measured, one step: N = 10^3 binary64 full matrix 3.0 ms -> 40 us, N = 10^5
// binary32 weights 22.2 ms -> 4.7 ms (a thread per row and an exponential per pair
// before: 4 CTAs at N = 10^3, ~25 instructions per pair).
#include "mt_pair.cuh"

namespace mt {

constexpr int kApTile = 1024;   // j-particles staged per tile
constexpr int kApWarps = kThreads / 32;
constexpr int kApCap = 64;      // list entries per row

struct ApGrid {
  int sh;                 // coarse coordinate: X >> sh, below 2^31
  unsigned int zc;        // candidate if |difference of coarse coordinates| <= zc
  unsigned int pc[2];     // periodic walls: ... or >= pc (the wrapped image)
  int cut;                // 1: the exact cutoff test applies
};

// Row state of a warp: the candidates listed and the sums so far.
template <int PR, int R, bool EX>
struct ApRow {
  int list[R][kApCap];
  int cnt[R];
  unsigned int cx[R], cy[R];
  typename Weight<mixw(PR), 1>::T r[EX ? 1 : R];
  typename Mass<PR>::Acc da[EX ? R : 1], db[EX ? R : 1];
};

// EX = false: row sums.  EX = true: exchange of A and B and the end of the
// step (sp = 0), or of the extra species sp, sp + 1.
template <int PR, int DIM, int R, bool EX>
__global__ void __launch_bounds__(kThreads) k_allpairs(Dev d, ApGrid g, int sp) {
  using W = Weight<mixw(PR), DIM>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ unsigned int s_cx[kApTile];
  __shared__ unsigned int s_cy[DIM == 2 ? kApTile : 1];
  extern __shared__ __align__(16) unsigned char s_rows[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ApRow<PR, R, EX>& s = reinterpret_cast<ApRow<PR, R, EX>*>(s_rows)[warp];
  const long long row0 = ((long long)blockIdx.x * kApWarps + warp) * R;
  const long long n = d.n;
  const long long* X = d.X[d.ctrl->xcur];
  const int mc = d.ctrl->mcur;
  const SpeciesPair sq = sp > 0 ? species_pair<true>(d, sp) : species_pair<false>(d, 0);
  const unsigned long long* MA = d.M[mc] + sq.oa;
  const unsigned long long* MB = d.M[mc] + sq.ob;
  const unsigned int zc = g.zc, w2 = 2 * zc;
  unsigned int lx[R], ly[R];  // coarse coordinates of the rows minus zc
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long p = row0 + r < n ? row0 + r : n - 1;
    lx[r] = (unsigned int)(X[p] >> g.sh) - zc;
    ly[r] = DIM == 2 ? (unsigned int)(X[n + p] >> g.sh) - zc : 0;
    if (lane == 0) {
      s.cnt[r] = 0;
      s.cx[r] = lx[r];
      s.cy[r] = ly[r];
      if (EX) {
        s.da[r] = {};
        s.db[r] = {};
      } else {
        s.r[r] = T(0);
      }
    }
  }
  // can the pair of a row (lx, ly) and a lane's coordinates have a weight?
  auto near = [&](unsigned int cx, unsigned int cy, unsigned int x, unsigned int y) {
    const unsigned int ux = cx - x;  // difference + zc
    bool ok = ux <= w2;
    if (d.periodic) ok = ok || (unsigned int)abs((int)(ux - zc)) >= g.pc[0];
    if (DIM == 2) {
      const unsigned int uy = cy - y;
      bool oky = uy <= w2;
      if (d.periodic) oky = oky || (unsigned int)abs((int)(uy - zc)) >= g.pc[1];
      ok = ok && oky;
    }
    return ok;
  };
  // work off the list of row r (every lane of the warp)
  auto flush = [&](int r) {
    __syncwarp();
    const int cnt = s.cnt[r];
    const long long p = row0 + r;
    const long long x = X[p], y = DIM == 2 ? X[n + p] : 0;
    MV A{}, B{};
    T ip = T(0);
    if (EX) {
      A = MS::load(MA, p);
      B = MS::load(MB, p);
      ip = load_rinv<mixw(PR)>(d, p);
    }
    T sum = EX ? T(0) : (mixw(PR) ? s.r[EX ? 0 : r] : T(0));
    typename MS::Acc a{}, b{};
    for (int k = 0; k < cnt; k += 32) {
      T w = T(0);
      int j = 0;
      if (k + lane < cnt) {
        j = s.list[r][k + lane];
        long long dx = X[j] - x, dy = DIM == 2 ? X[n + j] - y : 0;
        if (d.periodic) {
          dx = min_image(dx, d.Lq[0]);
          if (DIM == 2) dy = min_image(dy, d.Lq[1]);
        }
        if (!g.cut || in_range2(dx, dy, d.S)) w = W::eval(d, dx, dy);
      }
      if (EX) {
        if (w != T(0) && j != p) {
          const T P = normalised<T>(d.norm, w, ip, load_rinv<mixw(PR)>(d, j));
          MS::acc(a, P, MS::diff(MS::load(MA, j), A));
          MS::acc(b, P, MS::diff(MS::load(MB, j), B));
        }
      } else if (mixw(PR)) {
        // one by one in the order of j
        unsigned int m = __ballot_sync(0xffffffffu, w != T(0));
        while (m) {
          sum += __shfl_sync(0xffffffffu, w, __ffs(m) - 1);
          m &= m - 1;
        }
      } else {
        sum += w;
      }
    }
    if (EX) {
      a = acc_warp_sum(a);
      b = acc_warp_sum(b);
      if (lane == 0) {
        s.da[EX ? r : 0] = acc_merge(s.da[EX ? r : 0], a);
        s.db[EX ? r : 0] = acc_merge(s.db[EX ? r : 0], b);
      }
    } else {
      if (!mixw(PR)) sum = warp_sum(sum) + s.r[EX ? 0 : r];
      __syncwarp();
      if (lane == 0) s.r[EX ? 0 : r] = sum;
    }
    __syncwarp();
    if (lane == 0) s.cnt[r] = 0;
    __syncwarp();
  };
  for (long long j0 = 0; j0 < n; j0 += kApTile) {
    __syncthreads();
    for (int i = threadIdx.x; i < kApTile; i += kThreads) {
      const long long j = j0 + i;
      s_cx[i] = j < n ? (unsigned int)(X[j] >> g.sh) : 0;
      if (DIM == 2) s_cy[i] = j < n ? (unsigned int)(X[n + j] >> g.sh) : 0;
    }
    __syncthreads();
    const int nt = (int)min((long long)kApTile, n - j0);
    if (row0 >= n) continue;  // a warp without rows only stages
#pragma unroll 2
    for (int i0 = 0; i0 < nt; i0 += 32) {
      const unsigned int cx = s_cx[i0 + lane], cy = DIM == 2 ? s_cy[i0 + lane] : 0;
      bool any = false;
      if (d.periodic) {
#pragma unroll
        for (int r = 0; r < R; ++r) any |= near(cx, cy, lx[r], ly[r]);
      } else if (DIM == 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) any |= cx - lx[r] <= w2;
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) any |= cx - lx[r] <= w2 && cy - ly[r] <= w2;
      }
      if (!__any_sync(0xffffffffu, any)) continue;
      const bool in = i0 + lane < nt;
#pragma unroll 1
      for (int r = 0; r < R && row0 + r < n; ++r) {
        const bool c = in && near(cx, cy, s.cx[r], s.cy[r]);
        const unsigned int m = __ballot_sync(0xffffffffu, c);
        if (!m) continue;
        int at = s.cnt[r];
        if (at + __popc(m) > kApCap) {
          flush(r);
          at = 0;
        }
        if (c) s.list[r][at + __popc(m & ((1u << lane) - 1u))] = (int)(j0 + i0 + lane);
        __syncwarp();
        if (lane == 0) s.cnt[r] = at + __popc(m);
        __syncwarp();
      }
    }
  }
  if (row0 < n) {
    for (int r = 0; r < R && row0 + r < n; ++r) flush(r);
    const long long p = row0 + lane;
    if (lane < R && p < n) {
      if (!EX) {
        store_rinv<mixw(PR)>(d, p, s.r[EX ? 0 : lane]);
      } else {
        MV A = MS::load(MA, p), B = MS::load(MB, p);
        MS::update(A, B, s.da[EX ? lane : 0], s.db[EX ? lane : 0], sp > 0 ? 0 : d.react);
        MS::store(d.M[mc ^ 1] + sq.oa, p, A);
        if (sq.store_b) MS::store(d.M[mc ^ 1] + sq.ob, p, B);
      }
    }
  }
  if (EX && sp == 0) finish_step(d, 0, 1);
}

template <int PR, int DIM, int R, bool EX>
static cudaError_t launch_one(const Dev& d, const ApGrid& g, int sp, cudaStream_t s) {
  const size_t sm = kApWarps * sizeof(ApRow<PR, R, EX>);
  const long long rows = (long long)kApWarps * R;
  k_allpairs<PR, DIM, R, EX><<<(unsigned int)((d.n + rows - 1) / rows), kThreads, sm, s>>>(d, g, sp);
  return cudaGetLastError();
}

// Rows per warp: 8 amortise a staged coordinate's load and the vote over 8
// tests; a system that would then leave multiprocessors with less than two
// CTAs takes a row per warp (N = 10^3: 125 CTAs).
template <int PR, bool EX>
static cudaError_t launch_pr(const Dev& d, const ApGrid& g, int sp, cudaStream_t s) {
  const bool wide = d.n >= 2LL * d.nsm * kApWarps * 8;
  if (d.dim == 1)
    return wide ? launch_one<PR, 1, 8, EX>(d, g, sp, s) : launch_one<PR, 1, 1, EX>(d, g, sp, s);
  return wide ? launch_one<PR, 2, 8, EX>(d, g, sp, s) : launch_one<PR, 2, 1, EX>(d, g, sp, s);
}

// The scan's parameters; false where the list does not pay: binary32 weights
// (whose row sums add the list's entries one by one) with more than a quarter
// of all pairs in reach of one another, e.g. the paper's 50-unit domain, where
// a thread per row is faster (binary64 weights always take the list: their
// arithmetic outweighs it).
static bool ap_grid(const Dev& d, bool cut, int precision, ApGrid* g) {
  const double a = precision == MT_FP64 ? d.inv8 * d.scale * d.scale : (double)d.inv8f;
  double Z = a > 0.0 ? sqrt((precision == MT_FP64 ? 746.0 : 110.0) / a) * (1.0 + 1e-6) + 2.0 : 9e18;
  if (cut && (double)d.S < Z) Z = (double)d.S;
  double reach = 1.0;
  long long Lmax = 0;
  for (int k = 0; k < d.dim; ++k) {
    const double f = 2.0 * Z / ((double)d.Lq[k] + 1.0);
    reach *= f < 1.0 ? f : 1.0;
    Lmax = d.Lq[k] > Lmax ? d.Lq[k] : Lmax;
  }
  if (precision != MT_FP64 && reach > 0.25) return false;
  g->cut = cut ? 1 : 0;
  g->sh = 0;
  while ((Lmax >> g->sh) >= (1LL << 31)) ++g->sh;
  const long long z = Z < (double)Lmax ? (long long)Z + 1 : Lmax;
  const long long zc = (z >> g->sh) + 1;
  g->zc = (unsigned int)(zc < (1LL << 31) - 1 ? zc : (1LL << 31) - 1);
  for (int k = 0; k < 2; ++k) {
    const long long p = ((d.Lq[k] - z) >> g->sh) - 1;
    g->pc[k] = p > 0 ? (unsigned int)p : 0u;
  }
  return true;
}

template <int PR>
static cudaError_t allpairs_t(const Dev& d, const ApGrid& g, cudaStream_t s, Marker& mk) {
  mk(g.cut ? "rowsum_brute" : "rowsum_full", s);
  cudaError_t e = launch_pr<PR, false>(d, g, 0, s);
  for (int sp = 2; sp < d.nspec && e == cudaSuccess; sp += 2) {
    mk(g.cut ? "exchange_brute_species" : "exchange_full_species", s);
    e = launch_pr<PR, true>(d, g, sp, s);
  }
  mk(g.cut ? "exchange_brute" : "exchange_full", s);
  return e == cudaSuccess ? launch_pr<PR, true>(d, g, 0, s) : e;
}

bool launch_allpairs(const Dev& d, bool cut, int precision, cudaStream_t s, Marker& mk,
                     cudaError_t* e) {
  ApGrid g;
  if (!ap_grid(d, cut, precision, &g)) return false;
  *e = precision == MT_MIXED        ? allpairs_t<MT_MIXED>(d, g, s, mk)
       : precision == MT_MIXED_DF32 ? allpairs_t<MT_MIXED_DF32>(d, g, s, mk)
                                    : allpairs_t<MT_FP64>(d, g, s, mk);
  return true;
}

}  // namespace mt
