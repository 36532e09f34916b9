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
// A warp takes R rows, a lane one j.  The test uses coarse coordinates X >> sh
// of 24 bits as binary32 numbers, staged in shared memory: their differences
// are exact, and a subtraction per row (FMA pipe) and a three-input minimum of
// magnitudes per two rows (ALU pipe, half rate) leave one comparison and one
// vote per R rows and 32 pairs, which bounds the scan: ~1.9 warp instructions
// per row and 32 pairs with R = 16.  Lanes that see a row note it in a bit
// mask; only the rows of the mask are looked at.  A lane's candidates are
// appended, in the order of j, to the row's list in shared memory (a ballot
// and a prefix count), and a full list is worked off 32 entries at a time with
// the exact 64-bit test and the weight.  Row sums in binary32 add the list's
// nonzero weights one by one in the order of j, the order (and the bits) of
// a plain loop over j (but for direct tiles); binary64 sums and the flux sums use lane partials and
// a fixed shuffle tree.
//
// Where much of the matrix is nonzero (a dense system, particles piled at one
// place, in whatever order they are numbered) a list costs more than the pairs:
// a group of 32 candidates takes ~60 warp instructions and, in binary32 row
// sums, 32 dependent additions.  With binary32 weights a CTA that met more than
// a given share of its pairs in one tile therefore takes the next one directly
// (ap_direct): a lane per row and share of the columns, every weight evaluated,
// until a tile holds fewer again.  (Binary64 weights outweigh their list: 1.5
// times as long directly with a quarter of all pairs in reach, 0.83 with all.)
// The first tile of more than two is a short one, so that little is listed
// before the first choice.  The shares are where the two forms take as long, at N = 2 10^4
// and 5 10^4, one per unit length on a part of the domain:
//   row sums            directly 0.86 ms and 2.9 ms; by lists 1.8 and 4.7 with
//                       1/21 and 1/27 of the pairs in reach: 1/32
//   DF32's exchange     2.1 and 7.9; 2.1 with 1/14, 7.9 with 1/11: 1/8
//   MIXED's exchange    4.5 and 20.5; 4.6 with 1/4, 14.7 with 1/4: 1/4
// N = 2 10^4, all in reach: 25.5 ms -> 6.5 ms (MIXED), 19.9 -> 3.2 (DF32); a thread
// per row, which systems with more than 1/4 of the pairs in reach by their domain
// took before: 10.5 and 4.0 ms, and N = 5000 on 50 units 2.35 and 1.01 ms -> 0.43
// and 0.24.
//
// Measured, one step: N = 10^3 binary64 full matrix 3.0 ms -> 35 us, N = 10^5
// binary32 weights 22.2 ms -> 2.6 ms (a thread per row and an exponential per
// pair before: 4 CTAs at N = 10^3, ~25 instructions per pair; the same lists
// behind an integer comparison and a predicate per row: 4.7 ms; behind 16-bit
// add-minimum pairs: 5.3 ms).
#include <cmath>

#include "mt_pair.cuh"

namespace mt {

constexpr int kApTile = 2048;   // j-particles staged per tile
constexpr int kApThreads = 128;
constexpr int kApWarps = kApThreads / 32;
constexpr int kApCap = 64;      // list entries per row
constexpr int kApFirst = 256;   // j-particles in the first tile of more than two
// The next tile is taken directly if more than this share of the last one's
// pairs (its inverse) had a weight (binary32 weights).
constexpr int dense(int precision, bool exchange) {
  return !exchange ? 32 : precision == MT_MIXED_DF32 ? 8 : 4;
}

struct ApGrid {
  int sh;         // coarse coordinate: X >> sh, below 2^24
  float zc;       // candidate if the coarse distance is at most zc (per axis)
  float half[2];  // periodic walls: half the coarse domain length
  int cut;        // 1: the exact cutoff test applies
};

__device__ __forceinline__ float min_abs3(float a, float b, float c) {
  float r;
  asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Row state of a warp: the candidates listed and the sums so far.
template <int PR, int R, bool EX>
struct ApRow {
  int list[R][kApCap];
  typename Weight<mixw(PR), 1>::T r[EX ? 1 : R];
  typename Mass<PR>::Acc da[EX ? R : 1], db[EX ? R : 1];
};

// One tile directly: columns [j0, j0 + nt) staged exactly, kApThreads at a time
// (stage: 40 bytes each), lane l taking row l % R and every (32 / R)-th of them;
// the lanes' sums join the row's at the end.  Every thread of the CTA calls it
// (nr = 0: a warp without rows).  Returns the lane's number of nonzero weights.
template <int PR, int DIM, int R, bool EX, bool PER>
__device__ __forceinline__ int ap_direct(const Dev& d, const ApGrid& g, long long j0, int nt,
                                         long long row0, int nr, unsigned char* stage,
                                         ApRow<PR, R, EX>& s, const long long* X,
                                         const unsigned long long* MA,
                                         const unsigned long long* MB) {
  using W = Weight<mixw(PR), DIM>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  long long* sx = reinterpret_cast<long long*>(stage);
  long long* sy = sx + kApThreads;
  MV* sa = reinterpret_cast<MV*>(sy + kApThreads);
  MV* sb = sa + kApThreads;
  T* sr = reinterpret_cast<T*>(sb + kApThreads);
  const int lane = threadIdx.x & 31, r = lane % R;
  const bool mine = r < nr;
  const long long p = row0 + r;
  const long long x = mine ? X[p] : 0, y = mine && DIM == 2 ? X[d.n + p] : 0;
  MV A{}, B{};
  T ip = T(0);
  if (EX && mine) {
    A = MS::load(MA, p);
    B = MS::load(MB, p);
    ip = load_rinv<mixw(PR)>(d, p);
  }
  T sum = T(0);
  typename MS::Acc a{}, b{};
  int found = 0;
  for (int c0 = 0; c0 < nt; c0 += kApThreads) {
    const int nc = min(nt - c0, kApThreads);
    __syncthreads();
    if ((int)threadIdx.x < nc) {
      const int i = threadIdx.x;
      const long long j = j0 + c0 + i;
      sx[i] = X[j];
      if (DIM == 2) sy[i] = X[d.n + j];
      if (EX) {
        sa[i] = MS::load(MA, j);
        sb[i] = MS::load(MB, j);
        sr[i] = load_rinv<mixw(PR)>(d, j);
      }
    }
    __syncthreads();
    for (int i = lane / R; mine && i < nc; i += 32 / R) {
      long long dx = sx[i] - x, dy = DIM == 2 ? sy[i] - y : 0;
      if (PER) {
        dx = min_image(dx, d.Lq[0]);
        if (DIM == 2) dy = min_image(dy, d.Lq[1]);
      }
      if (g.cut && !in_range2(dx, dy, d.S)) continue;
      const T w = W::eval(d, dx, dy);
      if (w == T(0)) continue;
      ++found;
      if (!EX) {
        sum += w;
      } else if (j0 + c0 + i != p) {
        const T P = normalised<T>(d.norm, w, ip, sr[i]);
        MS::acc(a, P, MS::diff(sa[i], A));
        MS::acc(b, P, MS::diff(sb[i], B));
      }
    }
  }
  __syncwarp();
  if constexpr (EX) {
#pragma unroll
    for (int o = 16; o >= R; o >>= 1) {
      a = acc_merge(a, acc_shfl_xor(a, o));
      b = acc_merge(b, acc_shfl_xor(b, o));
    }
    if (lane < nr) {
      s.da[lane] = acc_merge(s.da[lane], a);
      s.db[lane] = acc_merge(s.db[lane], b);
    }
  } else {
#pragma unroll
    for (int o = 16; o >= R; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane < nr) s.r[lane] += sum;
  }
  __syncwarp();
  return found;
}

// PER: periodic walls.  EX = false: row sums.  EX = true: exchange of A and B and the end of the
// step (sp = 0), or of the extra species sp, sp + 1.
template <int PR, int DIM, int R, bool EX, bool PER>
__global__ void __launch_bounds__(kApThreads, R < 16 ? 10 : DIM == 1 ? 8 : 6) k_allpairs(Dev d, ApGrid g, int sp) {
  using W = Weight<mixw(PR), DIM>;
  using T = typename W::T;
  using MS = Mass<PR>;
  using MV = typename MS::V;
  __shared__ __align__(16) float s_cx[kApTile];  // (ap_direct: its stage)
  static_assert(kApTile * sizeof(float) >= kApThreads * 40, "ap_direct's stage");
  __shared__ int s_found[2];  // pairs with a weight (candidates) in the last tile
  __shared__ float s_cy[DIM == 2 ? kApTile : 1];
  extern __shared__ __align__(16) unsigned char s_rows[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ApRow<PR, R, EX>& s = reinterpret_cast<ApRow<PR, R, EX>*>(s_rows)[warp];
  const long long row0 = ((long long)blockIdx.x * kApWarps + warp) * R;
  const long long n = d.n;
  const int nr = row0 < n ? (int)min((long long)R, n - row0) : 0;
  const long long* X = d.X[d.ctrl->xcur];
  const int mc = d.ctrl->mcur;
  const SpeciesPair sq = sp > 0 ? species_pair<true>(d, sp) : species_pair<false>(d, 0);
  const unsigned long long* MA = d.M[mc] + sq.oa;
  const unsigned long long* MB = d.M[mc] + sq.ob;
  auto coarse = [&](int a, long long j) {
    return __int2float_rn((int)(X[(long long)a * n + j] >> g.sh));
  };
  float rx[R], ry[R];  // coarse coordinates of the rows (missing rows repeat the last)
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long p = row0 + r < n ? row0 + r : n - 1;
    rx[r] = coarse(0, p);
    ry[r] = DIM == 2 ? coarse(1, p) : 0.0f;
  }
  if (lane < nr) {
    if (EX) {
      s.da[EX ? lane : 0] = {};
      s.db[EX ? lane : 0] = {};
    } else {
      s.r[EX ? 0 : lane] = T(0);
    }
  }
  int mycnt = 0;  // lane r: entries in the list of row r
  int cnt1 = 0;   // R = 1: the row's, in every lane
  // coarse distance of a lane's coordinates to row r (the larger of the axes')
  auto dist = [&](float cx, float cy, int r) {
    float u = cx - rx[r], v = DIM == 2 ? cy - ry[r] : 0.0f;
    if (PER) {  // min(|u|, L - |u|)
      u = g.half[0] - fabsf(fabsf(u) - g.half[0]);
      if (DIM == 2) v = g.half[1] - fabsf(fabsf(v) - g.half[1]);
    }
    return DIM == 2 ? fmaxf(fabsf(u), fabsf(v)) : u;
  };
  // work off the list of row r (every lane of the warp)
  auto flush = [&](int r) {
    __syncwarp();
    const int cnt = __shfl_sync(0xffffffffu, mycnt, r);
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
        if (PER) {
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
    if (lane == r) mycnt = 0;
  };
  // tiles of kApTile, the first of more than two shorter
  int nt = mixw(PR) && n > 2 * kApTile ? kApFirst : (int)min((long long)kApTile, n);
  const int cta_rows = (int)min((long long)(kApWarps * R),
                                n - (long long)blockIdx.x * (kApWarps * R));
  int found = 0, par = 0;  // this warp's pairs with a weight in the tile
  bool direct = false;
  if (threadIdx.x < 2) s_found[threadIdx.x] = 0;
  for (long long j0 = 0; j0 < n;) {
    if (mixw(PR) && j0 > 0) {
      if (lane == 0 && found) atomicAdd(&s_found[par], found);
      __syncthreads();
      direct = s_found[par] > cta_rows * nt / dense(PR, EX);
      par ^= 1;
      found = 0;
    }
    if (j0 > 0) nt = (int)min((long long)kApTile, n - j0);
    __syncthreads();
    if constexpr (mixw(PR)) {
      if (threadIdx.x == 0) s_found[par ^ 1] = 0;
      if (direct) {
        found = __reduce_add_sync(0xffffffffu, ap_direct<PR, DIM, R, EX, PER>(
            d, g, j0, nt, row0, nr, reinterpret_cast<unsigned char*>(s_cx), s, X, MA, MB));
        j0 += nt;
        continue;
      }
    }
    // (the last group of 32 is filled up)
    for (int i = threadIdx.x; i < ((nt + 31) & ~31); i += kApThreads) {
      const long long j = j0 + i;
      s_cx[i] = j < n ? coarse(0, j) : 0.0f;
      if (DIM == 2) s_cy[i] = j < n ? coarse(1, j) : 0.0f;
    }
    __syncthreads();
    j0 += nt;
    if (nr == 0) continue;  // a warp without rows only stages
    const long long jt = j0 - nt;
#pragma unroll 2
    for (int i0 = 0; i0 < nt; i0 += 32) {
      const float cx = s_cx[i0 + lane], cy = DIM == 2 ? s_cy[i0 + lane] : 0.0f;
      if (R == 1) {  // one row: a vote is the list's next entries
        const bool c = i0 + lane < nt && fabsf(dist(cx, cy, 0)) <= g.zc;
        const unsigned int m = __ballot_sync(0xffffffffu, c);
        if (m == 0) continue;
        if (cnt1 + __popc(m) > kApCap) {
          mycnt = cnt1;
          flush(0);
          cnt1 = 0;
        }
        if (c) s.list[0][cnt1 + __popc(m & ((1u << lane) - 1u))] = (int)(jt + i0 + lane);
        cnt1 += __popc(m);
        if (mixw(PR)) found += __popc(m);
        continue;
      }
      float m = 3.0e38f;
#pragma unroll
      for (int r = 0; r < R; r += 2)
        m = min_abs3(dist(cx, cy, r), dist(cx, cy, r + 1 < R ? r + 1 : r), m);
      if (!__any_sync(0xffffffffu, m <= g.zc)) continue;
      unsigned int mine = 0;
#pragma unroll
      for (int r = 0; r < R; ++r) mine |= fabsf(dist(cx, cy, r)) <= g.zc ? 1u << r : 0u;
      if (i0 + lane >= nt) mine = 0;
      unsigned int rows = __reduce_or_sync(0xffffffffu, mine) & ((1u << nr) - 1u);
#pragma unroll 1
      for (; rows; rows &= rows - 1) {
        const int r = __ffs(rows) - 1;
        const bool c = (mine >> r) & 1u;
        const unsigned int m = __ballot_sync(0xffffffffu, c);
        int at = __shfl_sync(0xffffffffu, mycnt, r);
        if (at + __popc(m) > kApCap) {
          flush(r);
          at = 0;
        }
        if (c) s.list[r][at + __popc(m & ((1u << lane) - 1u))] = (int)(jt + i0 + lane);
        if (lane == r) mycnt = at + __popc(m);
        if (mixw(PR)) found += __popc(m);
      }
    }
  }
  if (nr > 0) {
    if (R == 1) mycnt = cnt1;
#pragma unroll 1
    for (int r = 0; r < nr; ++r) flush(r);
    const long long p = row0 + lane;
    if (lane < nr) {
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
  const unsigned int grid = (unsigned int)((d.n + rows - 1) / rows);
  if (d.periodic)
    k_allpairs<PR, DIM, R, EX, true><<<grid, kApThreads, sm, s>>>(d, g, sp);
  else
    k_allpairs<PR, DIM, R, EX, false><<<grid, kApThreads, sm, s>>>(d, g, sp);
  return cudaGetLastError();
}

// Rows per warp: 16 amortise a staged coordinate's load, the comparison and
// the vote over 24 instructions; a system that would then leave
// multiprocessors with less than two CTAs takes 4 or 1 (N = 10^3: 250 CTAs).
template <int PR, int DIM, bool EX>
static cudaError_t launch_rows(const Dev& d, const ApGrid& g, int sp, cudaStream_t s) {
  const long long fill = 2LL * d.nsm * kApWarps;
  if (d.n >= 16 * fill) return launch_one<PR, DIM, 16, EX>(d, g, sp, s);
  if (d.n >= 4 * fill) return launch_one<PR, DIM, 4, EX>(d, g, sp, s);
  return launch_one<PR, DIM, 1, EX>(d, g, sp, s);
}

template <int PR, bool EX>
static cudaError_t launch_pr(const Dev& d, const ApGrid& g, int sp, cudaStream_t s) {
  return d.dim == 1 ? launch_rows<PR, 1, EX>(d, g, sp, s) : launch_rows<PR, 2, EX>(d, g, sp, s);
}

// The scan's parameters.
static ApGrid ap_grid(const Dev& d, bool cut, int precision) {
  ApGrid g;
  const double a = precision == MT_FP64 ? d.inv8 * d.scale * d.scale : (double)d.inv8f;
  double Z = a > 0.0 ? sqrt((precision == MT_FP64 ? 746.0 : 110.0) / a) * (1.0 + 1e-6) + 2.0 : 9e18;
  if (cut && (double)d.S < Z) Z = (double)d.S;
  long long Lmax = d.Lq[0];
  if (d.dim == 2 && d.Lq[1] > Lmax) Lmax = d.Lq[1];
  g.cut = cut ? 1 : 0;
  g.sh = 0;
  while ((Lmax >> g.sh) >= (1LL << 24)) ++g.sh;
  // rounding of both coordinates, and of the coarse half length and of its
  // differences (half a unit each): two more units
  g.zc = (float)(std::floor(std::ldexp(Z < (double)Lmax ? Z : (double)Lmax, -g.sh)) + 3.0);
  for (int k = 0; k < 2; ++k) g.half[k] = (float)std::ldexp((double)d.Lq[k], -g.sh - 1);
  return g;
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

cudaError_t launch_allpairs(const Dev& d, bool cut, int precision, cudaStream_t s, Marker& mk) {
  const ApGrid g = ap_grid(d, cut, precision);
  if (precision == MT_MIXED) return allpairs_t<MT_MIXED>(d, g, s, mk);
  if (precision == MT_MIXED_DF32) return allpairs_t<MT_MIXED_DF32>(d, g, s, mk);
  return allpairs_t<MT_FP64>(d, g, s, mk);
}

}  // namespace mt
