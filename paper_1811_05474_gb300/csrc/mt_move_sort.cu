// mt_move_sort.cu -- the random-walk move (Eq. 2, Sec. 3 walls) and the
// cell-list build: a counting sort of particles by cell key (histogram,
// single-pass look-back scan, atomic scatter, then a sort inside each cell
// that makes the order unique).  The uniform grid replaces the paper's
// KD-tree fixed-radius search (Sec. 2.1).
#include "mt_internal.cuh"

namespace mt {

// ------------------------------------------------------------------ move --
// Moves every particle once (unless !MOVE) and histograms its cell key
// (if HIST).  Thread 0 also resets the per-step counters of the sort.
template <int DIM, bool MOVE, bool HIST>
__global__ void __launch_bounds__(kThreads) k_move(Dev d) {
  chained();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  Ctrl* c = d.ctrl;
  if (p == 0) {
    c->tile_ctr = 0;
    c->nbig = 0;
    c->epoch += 1;
  }
  if (p >= d.n) return;
  const int xc = c->xcur;
  long long* X = d.X[xc];
  long long pos[2] = {X[p], DIM == 2 ? X[d.n + p] : 0};
  if (MOVE) {
    const int id = d.id[xc][p];
    // realisation of the particle (always 0 in 2-d, where base = 0)
    long long base = 0, Lq = d.rLq, off = 0;
    unsigned int real = d.rreal;
    int loc = id;
    if (DIM == 1 && !d.single) {
      const Real* R = d.rt + (id >> d.lbits);
      base = R->base;
      Lq = R->Lq;
      off = R->off;
      real = R->real;
      loc &= d.lmask;
    }
    float z[2];
    const float* noise = c->noise;
    if (noise) {
      z[0] = noise[off + loc];
      if (DIM == 2) z[1] = noise[d.n + loc];
    } else {
      const unsigned long long st = c->step;
      const uint4 u = philox4x32_10(
          make_uint4((unsigned int)loc, (unsigned int)st, (unsigned int)(st >> 32), real),
          d.key0, d.key1);
      const float2 g = box_muller(u.x, u.y);
      z[0] = g.x;
      z[1] = g.y;
    }
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      // Eq. 2 on the grid: drift + rint(b * xi), then the wall mirror.
      const long long step = walk_ticks(d.bq, z[a]);
      if (d.periodic && a == 0)
        pos[0] = base + wrap(pos[0] - base + d.drift[0] + step, Lq);
      else if (d.periodic)
        pos[a] = wrap(pos[a] + d.drift[a] + step, d.Lq[a]);
      else if (a == 0)
        pos[0] = base + reflect(pos[0] - base + d.drift[0] + step, Lq);
      else
        pos[a] = reflect(pos[a] + d.drift[a] + step, d.Lq[a]);
      X[(long long)a * d.n + p] = pos[a];
    }
  }
  // its arrival number in the cell (kept in rinv until the row sums)
  if (HIST)
    static_cast<int*>(d.rinv)[p] = atomicAdd(&d.count[cell_of(d, pos[0], pos[1])], 1);
}

// ------------------------------------------------------------------ scan --
// Exclusive scan of count[] into start[] (and count[] := 0), one pass with
// decoupled look-back.  Tiles are handed out in launch order by a ticket, so
// a tile only waits on tiles already running; the wait is bounded anyway and
// raises kErrTimeout instead of hanging.  A warp takes 512 consecutive counts,
// four per lane and load (coalesced 16-byte accesses), and the tile's first
// warp looks back over 32 status words at a time.  Bound: 8 bytes read and 8
// written per cell; 1.56 10^6 cells: 36 -> 14 us (a thread's 16 consecutive
// counts one by one, one thread looking back word by word).
// Status word: [63:48] epoch tag, [47:46] flag (1 aggregate, 2 prefix),
// [45:0] value.
__device__ __forceinline__ unsigned long long pack(unsigned long long tag, unsigned long long flag,
                                                   long long v) {
  return (tag << 48) | (flag << 46) | ((unsigned long long)v & ((1ULL << 46) - 1));
}

__device__ __forceinline__ int warp_inclusive(int v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

__global__ void __launch_bounds__(kThreads) k_scan(Dev d) {
  chained();
  constexpr int kWarps = kThreads / 32, kVec = kScanItems / 4;
  __shared__ int s_tile;
  __shared__ int s_warp[kWarps];
  __shared__ long long s_excl;
  Ctrl* c = d.ctrl;
  if (threadIdx.x == 0) s_tile = (int)atomicAdd(&c->tile_ctr, 1u);
  __syncthreads();
  const long long tile = s_tile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // counts k0 + 128 i + 4 lane .. + 3 (at most 2^31 particles in all)
  const long long k0 = tile * kScanTile + warp * (32 * kScanItems) + 4 * lane;
  int4 v[kVec];
  int excl[kVec];  // within the warp's counts
  int run = 0;
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    const long long k = k0 + 128 * i;
    if (k + 3 < d.ncell) {
      v[i] = *reinterpret_cast<const int4*>(d.count + k);
      *reinterpret_cast<int4*>(d.count + k) = make_int4(0, 0, 0, 0);
    } else {
      int w[4];
      for (int e = 0; e < 4; ++e) {
        w[e] = k + e < d.ncell ? d.count[k + e] : 0;
        if (k + e < d.ncell) d.count[k + e] = 0;
      }
      v[i] = make_int4(w[0], w[1], w[2], w[3]);
    }
  }
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    const int sum = v[i].x + v[i].y + v[i].z + v[i].w;
    const int inc = warp_inclusive(sum, lane);
    excl[i] = run + inc - sum;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) s_warp[warp] = run;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if (w < warp) before += s_warp[w];
    total += s_warp[w];
  }
  if (warp == 0) {
    const unsigned long long tag = (c->epoch % 65535ULL) + 1ULL;
    volatile unsigned long long* st = d.scan_status;
    long long sum = 0;
    if (tile == 0) {
      // (the test hook withholds this word: every later tile's wait then
      // runs out and raises kErrTimeout)
      if (lane == 0 && !c->scan_hold) atomicExch(&d.scan_status[0], pack(tag, 2, total));
    } else {
      if (lane == 0) atomicExch(&d.scan_status[tile], pack(tag, 1, total));
      const long long limit = c->spin_limit > 0 ? c->spin_limit : kSpinLimit;
      long long t = tile - 1, spins = 0;
      for (;;) {  // tiles t, t - 1, ... t - 31 (before tile 0: an empty prefix)
        const unsigned long long w = t - lane >= 0 ? st[t - lane] : pack(tag, 2, 0);
        const unsigned long long flag = (w >> 46) & 3ULL;
        const bool ready = (w >> 48) == tag && flag != 0;
        const unsigned int prefix = __ballot_sync(0xffffffffu, ready && flag == 2);
        const unsigned int missing = __ballot_sync(0xffffffffu, !ready);
        const int last = prefix ? __ffs(prefix) - 1 : 31;  // words up to the first prefix count
        if (missing & (0xffffffffu >> (31 - last))) {
          if (++spins > limit) {
            if (lane == 0) raise_error(c, kErrTimeout, tile);
            break;
          }
          continue;
        }
        long long part = lane <= last ? (long long)(w & ((1ULL << 46) - 1)) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        sum += part;
        if (prefix) break;
        t -= 32;
      }
      if (lane == 0) atomicExch(&d.scan_status[tile], pack(tag, 2, sum + total));
    }
    if (lane == 0) s_excl = sum;
  }
  __syncthreads();
  const int base = (int)s_excl + before;
#pragma unroll
  for (int i = 0; i < kVec; ++i) {
    const long long k = k0 + 128 * i;
    int4 o;
    o.x = base + excl[i];
    o.y = o.x + v[i].x;
    o.z = o.y + v[i].y;
    o.w = o.z + v[i].z;
    if (k + 3 < d.ncell) {
      *reinterpret_cast<int4*>(d.start + k) = o;
    } else {
      const int w[4] = {o.x, o.y, o.z, o.w};
      for (int e = 0; e < 4; ++e)
        if (k + e < d.ncell) d.start[k + e] = w[e];
    }
    // the end of the last cell
    if (d.ncell - 1 >= k && d.ncell - 1 < k + 4) {
      const int e = (int)(d.ncell - 1 - k);
      d.start[d.ncell] = e == 0 ? o.y : e == 1 ? o.z : e == 2 ? o.w : o.w + v[i].w;
    }
  }
}

// --------------------------------------------------------------- scatter --
// The slot before the sort into its cell's slots, in arrival order (1-d: the
// position too).
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_scatter(Dev d) {
  chained();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const int xc = d.ctrl->xcur;
  const long long* X = d.X[xc];
  const long long x = X[p], y = DIM == 2 ? X[d.n + p] : 0;
  const long long slot = (long long)d.start[cell_of(d, x, y)] + static_cast<const int*>(d.rinv)[p];
  if (slot < 0 || slot >= d.n) {
    raise_error(d.ctrl, kErrIndex, slot);
    return;
  }
  if (DIM == 1) d.X[xc ^ 1][slot] = x;
  d.src[slot] = (int)p;
}

// 2-d: a particle's final slot is its cell's first slot plus the number of the
// cell's particles with a smaller src (the slot before the sort), which makes
// the order unique whatever order they arrived in; it takes its position, id
// and masses (every species) there.  One thread per particle: a cell of m
// particles costs m^2 reads of src, less than the m^2 pair tests that the two
// transfer passes spend on it (a cell is wider than the cutoff).  Bound: the
// chain of dependent reads src, position, cell start (10^6 particles: 16 us;
// with the large cells' sort and the gather of ids and masses, which the row
// sums did, it takes the place of 25 us; two particles per thread: no faster).
__global__ void __launch_bounds__(kThreads) k_place2(Dev d) {
  chained();
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const long long s = d.src[p];
  if (s < 0 || s >= d.n) {  // (a scan that timed out leaves slots unset)
    raise_error(d.ctrl, kErrIndex, s);
    return;
  }
  const long long* X = d.X[xc];
  const long long x = X[s], y = X[d.n + s];
  const long long c = cell_of(d, x, y);
  const int a = max(d.start[c], 0), b = (int)min((long long)d.start[c + 1], d.n);
  long long f = a;
  for (int q = a; q < b; ++q) f += d.src[q] < s ? 1 : 0;
  if (f >= d.n) {
    raise_error(d.ctrl, kErrIndex, f);
    return;
  }
  long long* Y = d.X[xc ^ 1];
  Y[f] = x;
  Y[d.n + f] = y;
  d.id[xc ^ 1][f] = d.id[xc][s];
  gather_masses(d, mc, f, s);
  gather_species(d, mc, f, s);
}

// ------------------------------------------------------------- cell sort --
// 1-d: order inside a cell by (x, src), which makes the whole array sorted by
// position.  src is the slot before the sort, so the result does not depend
// on the order of arrival.
__device__ __forceinline__ bool before(long long xa, int sa, long long xb, int sb) {
  return xa < xb || (xa == xb && sa < sb);
}

__global__ void __launch_bounds__(kThreads) k_cellsort(Dev d) {
  chained();
  const long long k = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (k >= d.ncell) return;
  const int a = d.start[k], b = d.start[k + 1];
  const int len = b - a;
  if (len < 2) return;
  if (len > kSmallCell) {
    const int slot = atomicAdd(&d.ctrl->nbig, 1);
    if (slot < d.nbig_cap)
      d.big[slot] = (int)k;
    else
      raise_error(d.ctrl, kErrIndex, k);
    return;
  }
  long long* X = d.X[d.ctrl->xcur ^ 1];
  int* src = d.src;
  for (int i = a + 1; i < b; ++i) {
    const long long xi = X[i];
    const int si = src[i];
    int j = i - 1;
    while (j >= a && before(xi, si, X[j], src[j])) {
      X[j + 1] = X[j];
      src[j + 1] = src[j];
      --j;
    }
    X[j + 1] = xi;
    src[j + 1] = si;
  }
}

// Large cells: one CTA per cell, bitonic sort with every comparator
// ascending (partner i ^ (2j - 1) in the first stage of each merge), which
// sorts any length when positions >= len are treated as +infinity.
__global__ void __launch_bounds__(1024) k_bigsort(Dev d) {
  chained();
  __shared__ long long s_key[kBigSortCap];
  __shared__ int s_src[kBigSortCap];
  Ctrl* c = d.ctrl;
  const int nbig = min(c->nbig, d.nbig_cap);
  long long* X = d.X[c->xcur ^ 1];
  int* src = d.src;
  for (int b = blockIdx.x; b < nbig; b += gridDim.x) {
    const long long k = d.big[b];
    const int a = d.start[k];
    const int len = d.start[k + 1] - a;
    const bool shared = len <= kBigSortCap;
    long long* key = shared ? s_key : X + a;
    int* tag = shared ? s_src : src + a;
    if (shared) {
      for (int i = threadIdx.x; i < len; i += blockDim.x) {
        s_key[i] = X[a + i];
        s_src[i] = src[a + i];
      }
    }
    __syncthreads();
    long long np2 = 1;
    while (np2 < len) np2 <<= 1;
    for (long long m = 2; m <= np2; m <<= 1) {
      for (long long j = m >> 1; j > 0; j >>= 1) {
        for (long long i = threadIdx.x; i < np2; i += blockDim.x) {
          const long long l = (j == (m >> 1)) ? (i ^ (m - 1)) : (i ^ j);
          if (l > i && l < len) {
            const long long xi = key[i], xl = key[l];
            if (before(xl, tag[l], xi, tag[i])) {
              key[i] = xl;
              key[l] = xi;
              const int ts = tag[i];
              tag[i] = tag[l];
              tag[l] = ts;
            }
          }
        }
        __syncthreads();
      }
    }
    if (shared) {
      for (int i = threadIdx.x; i < len; i += blockDim.x) {
        X[a + i] = s_key[i];
        src[a + i] = s_src[i];
      }
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------- permute --
// After a 1-d sort without a transfer (upload): gather id and masses into the
// sorted slots, then the next kernel flips the selectors.
__global__ void __launch_bounds__(kThreads) k_permute(Dev d) {
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= d.n) return;
  const int xc = d.ctrl->xcur, mc = d.ctrl->mcur;
  const int s = d.src[p];
  d.id[xc ^ 1][p] = d.id[xc][s];
  gather_masses(d, mc, p, s);
  gather_species(d, mc, p, s);
}

__global__ void k_flip(Dev d, int fx, int fm) {
  d.ctrl->xcur ^= fx;
  d.ctrl->mcur ^= fm;
}

// -------------------------------------------------------------- philox --
__global__ void k_philox(uint4 c, unsigned int k0, unsigned int k1, long long n,
                         unsigned int* out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 r = philox4x32_10(make_uint4(c.x + (unsigned int)i, c.y, c.z, c.w), k0, k1);
  out[4 * i + 0] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

// ------------------------------------------------------------ launchers --
static unsigned int blocks_for(long long n, int t) { return (unsigned int)((n + t - 1) / t); }

cudaError_t launch_move(const Dev& d, bool move, bool hist, cudaStream_t s) {
  const unsigned int g = blocks_for(d.n, kThreads);
  if (d.dim == 1) {
    if (move && hist) launch_chained(k_move<1, true, true>, g, kThreads, 0, s, d);
    else if (move) launch_chained(k_move<1, true, false>, g, kThreads, 0, s, d);
    else launch_chained(k_move<1, false, true>, g, kThreads, 0, s, d);
  } else {
    if (move && hist) launch_chained(k_move<2, true, true>, g, kThreads, 0, s, d);
    else if (move) launch_chained(k_move<2, true, false>, g, kThreads, 0, s, d);
    else launch_chained(k_move<2, false, true>, g, kThreads, 0, s, d);
  }
  return cudaGetLastError();
}

cudaError_t launch_sort(const Dev& d, cudaStream_t s, Marker& mk) {
  const unsigned int gs = blocks_for(d.ncell, kScanTile);
  mk("scan", s);
  launch_chained(k_scan, gs, kThreads, 0, s, d);
  const unsigned int gp = blocks_for(d.n, kThreads);
  mk("scatter", s);
  if (d.dim == 1) {
    launch_chained(k_scatter<1>, gp, kThreads, 0, s, d);
    mk("cellsort", s);
    launch_chained(k_cellsort, blocks_for(d.ncell, kThreads), kThreads, 0, s, d);
    mk("bigsort", s);
    launch_chained(k_bigsort, (unsigned int)(d.nbig_cap < 304 ? d.nbig_cap : 304), 1024, 0, s, d);
  } else {
    launch_chained(k_scatter<2>, gp, kThreads, 0, s, d);
    mk("place", s);
    launch_chained(k_place2, gp, kThreads, 0, s, d);
  }
  return cudaGetLastError();
}

cudaError_t launch_permute(const Dev& d, cudaStream_t s) {
  if (d.dim == 1) k_permute<<<blocks_for(d.n, kThreads), kThreads, 0, s>>>(d);
  k_flip<<<1, 1, 0, s>>>(d, 1, 1);  // (2-d: placed by the sort)
  return cudaGetLastError();
}

// The built-in random walk's normals of particles given by their indices in
// a system (the counter a single handle uses for caller index gid): one per
// axis, axis-major.
__global__ void k_walk_normals(const long long* gid, long long n, unsigned long long step,
                               unsigned int real, unsigned int k0, unsigned int k1, int dim,
                               float* out) {
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const long long id = gid[p];
  const uint4 u = philox4x32_10(
      make_uint4((unsigned int)id, (unsigned int)step, (unsigned int)(step >> 32), real), k0, k1);
  const float2 g = box_muller(u.x, u.y);
  out[p] = g.x;
  if (dim == 2) out[n + p] = g.y;
}

cudaError_t launch_walk_normals(const long long* gid, long long n, unsigned long long step,
                                unsigned int real, unsigned int k0, unsigned int k1, int dim,
                                float* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_walk_normals<<<blocks_for(n, 256), 256, 0, s>>>(gid, n, step, real, k0, k1, dim, out);
  return cudaGetLastError();
}

cudaError_t launch_philox(uint4 c, unsigned int k0, unsigned int k1, long long n,
                          unsigned int* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_philox<<<blocks_for(n, 256), 256, 0, s>>>(c, k0, k1, n, out);
  return cudaGetLastError();
}

}  // namespace mt
