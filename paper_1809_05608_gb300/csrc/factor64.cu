// FP64 block-Thomas elimination of the per-(ray, species) systems (the FP64 path, the adjoint and the
// C ABI; see blocktri.cu for the twisted elimination and the structure it exploits).
//
// Two launches: the two halves of every system as independent work, zones 0..m-1 top-down and zones
// n_r-1..m+1 bottom-up, then the middle zones m = n_r/2, whose blocks receive both Schur terms (read
// back from the factor array).
//
// What bounds it: the FP64 units, one in each quarter of an SM, which every warp instruction holds for 64
// cycles however few lanes work (a warp alone gets one FP64 instruction in 64 cycles; four warps on
// the four quarters one in 16).  So a block's columns are dealt to the four warps of a CTA, warp w
// holding columns c = w mod 4, which puts an equal share of every pivot step on all four quarters,
// and the lanes of a warp are the rows: NP / RPL lanes per half, lane c with rows c and c + NP/2 (RPL = 2)
// or row c (RPL = 1), as many halves per warp as fit.  RPL = 2 fills 30 of 32 lanes at NP = 20 (three
// halves a CTA, 11 FP64 instructions per warp and pivot step); in launches of up to four CTAs per SM the chain of
// the pivot search counts instead, and RPL = 1 halves the FMAs behind it.
// Both do the same operations on every entry in the same order, those of one thread per row, so the
// factors are the same bit for bit.  Measured (one factorisation, 512 zones x 20 groups; against
// thread-per-row CTAs of four systems with two CTA barriers a step): 64 rays, RPL = 1, 7.68 -> 4.49 ms
// (RPL = 2 6.9); 256 rays, RPL = 2, 11.9 -> 10.6 ms (RPL = 1 16.7; 85 % of the FP64 units' time);
// one ray of 64 x 12, RPL = 1, 0.393 -> 0.225 ms (RPL = 2 0.44).
#include "async.cuh"
#include "mgfld_internal.cuh"

namespace mgfld {

template <int NP, int RPL>
struct Quad {
  static constexpr int L = NP / RPL;                     // lanes per half
  static constexpr int S = 32 / L;                       // halves per CTA
  static constexpr int CW = NP / 4;                      // columns per warp
  static constexpr int LK = (L + 3) / 4 * 4;             // candidate keys, in 16-byte pieces
  // resident CTAs: five three-half CTAs an SM take the 683 of 256 rays x 20 groups in one wave
  static constexpr int MINB = RPL == 1 ? 1 : (NP <= 20 ? 5 : (NP <= 24 ? 4 : 2));
  static_assert(NP % 4 == 0 && L * RPL == NP, "columns dealt to four warps");
  struct Smem {
    double tile[S][NP][NP + 1];                          // the inverse in natural order
    double f[2][S][NP];                                  // each row's multiplier of the current / next step
    double ucol[S][NP];                                  // column scaling of the next zone's Schur term
    alignas(16) double next[S][NP * NP];                 // the next zone's blocks (n x n, dense)
    alignas(16) int cand[S][LK];                         // pivot-search keys, the larger of a lane's rows
    int best[2][S];                                      // pivot row of the current / next step
    int pivrow[S][NP];                                   // row chosen at each step
  };
};

// Gauss-Jordan inversion in place with partial pivoting (implicit row exchanges); a[q][j] is row c0 + q L,
// column 4 j + w.  Per pivot step p: every row is updated with one FMA per entry, a -= f pivot_row, f
// chosen so that the pivot row itself becomes pivot_row / pivot (f = 1 - 1/pivot); the pivot row's
// entries come from its lane of the same warp.  The warp that holds column p + 1 updates it first,
// searches it for the next pivot and publishes the next multipliers while the others (and its own
// other columns) are still in the FP64 units; one CTA barrier per step, at which the publisher only
// arrives (two barriers in turn: nobody publishes step p + 2, whose multipliers take step p's place,
// before everybody has come to step p + 1's).  The inverse then goes through
// shared memory to its natural order (row r holds row step of it, column p belongs to row pivrow[p]).
template <int NP, int RPL>
__device__ inline void invert64(double (&a)[RPL][NP / 4], typename Quad<NP, RPL>::Smem &sm, int g, int c0, int w) {
  using C = Quad<NP, RPL>;
  constexpr int L = C::L, LK = C::LK, CW = C::CW;
  const unsigned full = 0xffffffffu;
  bool used[RPL];
  int step[RPL];
#pragma unroll
  for (int q = 0; q < RPL; ++q) {
    used[q] = false;
    step[q] = 0;
  }
  // search column p (its entries v, in this warp) and publish step p: pivot row and multipliers; the
  // column itself takes its value after the step
  auto publish = [&](int p, double (&v)[RPL]) {
    int key = -1;
#pragma unroll
    for (int q = 0; q < RPL; ++q)
      if (!used[q]) key = max(key, pivot_key(v[q], c0 + q * L));
    sm.cand[g][c0] = key;
    __syncwarp();
    int k = -1;
#pragma unroll
    for (int j = 0; j < LK / 4; ++j) {
      const int4 x = reinterpret_cast<const int4 *>(sm.cand[g])[j];
      k = max(k, max(max(x.x, x.y), max(x.z, x.w)));
    }
    const int best = 31 - (k & 31);
    const int src = g * L + (best >= L ? best - L : best);
    double pv = __shfl_sync(full, v[0], src);
    if (RPL == 2) {
      const double p1 = __shfl_sync(full, v[RPL - 1], src);
      if (best >= L) pv = p1;
    }
    const double inv = recip(pv);
    const int buf = p & 1;
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
      const bool me = c0 + q * L == best;
      const double f = fma(me ? -1.0 : v[q], inv, me ? 1.0 : 0.0);
      sm.f[buf][g][c0 + q * L] = f;
      v[q] = me ? inv : -f;
    }
    if (c0 == 0) {
      sm.best[buf][g] = best;
      sm.pivrow[g][p] = best;
    }
    // (the publisher need not wait for its own step: it goes on with its other columns)
    asm volatile("bar.arrive %0, 128;" ::"r"(1 + buf) : "memory");
  };
  if (w == 0) {
    double v[RPL];
#pragma unroll
    for (int q = 0; q < RPL; ++q) v[q] = a[q][0];
    publish(0, v);
#pragma unroll
    for (int q = 0; q < RPL; ++q) a[q][0] = v[q];
  }
#pragma unroll 1
  for (int jj = 0; jj < CW; ++jj) {
    // (the arrays turn by one column every four steps: column 4 jj + w is a[.][0])
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int p = 4 * jj + s, buf = s & 1;
      if (w != s) asm volatile("bar.sync %0, 128;" ::"r"(1 + buf) : "memory");
      else __syncwarp();
      const int best = sm.best[buf][g];
      const int src = g * L + (best >= L ? best - L : best);
      double f[RPL];
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        f[q] = sm.f[buf][g][c0 + q * L];
        if (c0 + q * L == best) {
          used[q] = true;
          step[q] = p;
        }
      }
      constexpr int N1 = CW > 1 ? 1 : 0;
      const int nx = s < 3 ? 0 : N1;                     // slot and warp of column p + 1
      const bool next = w == ((s + 1) & 3) && (s < 3 || jj + 1 < CW);
      auto pivot_entry = [&](int j) {
        const double x0 = __shfl_sync(full, a[0][j], src);
        if (RPL == 1) return x0;
        const double x1 = __shfl_sync(full, a[RPL - 1][j], src);
        return best >= L ? x1 : x0;
      };
      if (next) {
        const double pr = pivot_entry(nx);
        double v[RPL];
#pragma unroll
        for (int q = 0; q < RPL; ++q) v[q] = fma(-f[q], pr, a[q][nx]);
        publish(p + 1, v);
#pragma unroll
        for (int q = 0; q < RPL; ++q) a[q][nx] = v[q];
      }
#pragma unroll
      for (int j = 0; j < CW; ++j) {
        if ((next && j == nx) || (j == 0 && w == s)) continue;       // done above; column p itself
        const double pr = pivot_entry(j);
#pragma unroll
        for (int q = 0; q < RPL; ++q) a[q][j] = fma(-f[q], pr, a[q][j]);
      }
    }
    if (CW > 1) {
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        const double t = a[q][0];
#pragma unroll
        for (int j = 0; j + 1 < CW; ++j) a[q][j] = a[q][j + 1];
        a[q][CW - 1] = t;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < CW; ++j) {
    const int c = sm.pivrow[g][4 * j + w];
#pragma unroll
    for (int q = 0; q < RPL; ++q) sm.tile[g][step[q]][c] = a[q][j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < CW; ++j)
#pragma unroll
    for (int q = 0; q < RPL; ++q) a[q][j] = sm.tile[g][c0 + q * L][4 * j + w];
}

// middle = 0: item j is half j & 1 of system j / 2; 1: item j is the middle zone of system j.  Rows and
// columns beyond the real group count n (<= NP) are padded with the identity.
template <int NP, int RPL>
__global__ void __launch_bounds__(128, Quad<NP, RPL>::MINB)
k_factor64(int n, int n_r, int n_sys, const double *__restrict__ diag, const double *__restrict__ lower,
           const double *__restrict__ upper, double *dinv, const int *__restrict__ ray_list, int middle,
           int al16, const int *__restrict__ n_dev) {
  using C = Quad<NP, RPL>;
  constexpr int L = C::L, S = C::S, CW = C::CW;
  __shared__ typename C::Smem sm;
  const int n_items = (middle ? 1 : 2) * listed_sys(n_sys, n_dev, NS);
  if ((long)blockIdx.x * S >= n_items) return;           // the whole CTA
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane < S * L ? lane / L : S - 1;         // lanes that hold no half go along with the last
  const int c0 = lane < S * L ? lane % L : L - 1;        // lane of the last one
  const long item = (long)blockIdx.x * S + g;
  const bool valid = item < n_items;
  const int m = n_r / 2;
  const int half = middle ? 0 : (int)(item & 1);         // 0: zones 0..m-1 top-down, 1: zones n_r-1..m+1 bottom-up
  const long sys = valid ? listed_system(middle ? item : item >> 1, ray_list, NS) : 0;
  const int len = middle ? 1 : (half == 0 ? m : n_r - 1 - m);   // zones of this item
  const int steps = middle ? 1 : m;                      // of the CTA
  auto zone = [&](int j) { return middle ? m : (half == 0 ? j : n_r - 1 - j); };
  auto row_of = [&](int z, int r) { return ((size_t)sys * n_r + z) * n + r; };
  if (c0 < C::LK - L) sm.cand[g][L + c0] = -1;           // the keys that fill the last 16-byte piece

  // The next zone's blocks arrive in shared memory by asynchronous copies of all threads while a zone is
  // inverted, its couplings in registers.  al16: blocks of whole 16-byte pieces on 16-byte boundaries.
  const int nn = n * n;
  auto fetch = [&](int j) {
#pragma unroll
    for (int h = 0; h < S; ++h) {
      const long it = (long)blockIdx.x * S + h;
      const int hf = middle ? 0 : (int)(it & 1);
      if (it >= n_items || j >= (middle ? 1 : (hf == 0 ? m : n_r - 1 - m))) continue;
      const long sy = listed_system(middle ? it : it >> 1, ray_list, NS);
      const int z = middle ? m : (hf == 0 ? j : n_r - 1 - j);
      const double *src = diag + ((size_t)sy * n_r + z) * nn;
      if (al16)
        for (int e = 2 * threadIdx.x; e < nn; e += 256) cp_async16(&sm.next[h][e], src + e);
      else
        for (int e = threadIdx.x; e < nn; e += 128) cp_async8(&sm.next[h][e], src + e);
    }
    cp_async_commit();
  };
  double a[RPL][CW], l[RPL], u[RPL];
  auto couplings = [&](int j) {
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
      const int r = c0 + q * L;
      const bool real = valid && j < len && r < n;
      const size_t zr = row_of(real ? zone(j) : 0, real ? r : 0);
      l[q] = real ? (half == 0 ? lower[zr] : upper[zr]) : 0.0;
      u[q] = real ? (half == 0 ? upper[zr] : lower[zr]) : 0.0;
    }
  };
  fetch(0);
  couplings(0);
  for (int j = 0; j < steps; ++j) {
    const bool active = valid && j < len;
    cp_async_wait_all();
    __syncthreads();                                     // the blocks, and the last zone's inverse and couplings
    // this zone's rows, minus the previous zone's Schur term diag(l) Dinv diag(u)
#pragma unroll
    for (int q = 0; q < RPL; ++q) {
      const int r = c0 + q * L;
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        const int col = 4 * c + w;
        const double d = (active && r < n && col < n) ? sm.next[g][r * n + col] : (col == r ? 1.0 : 0.0);
        a[q][c] = (j > 0 && active) ? fma(-(l[q] * a[q][c]), sm.ucol[g][col], d) : d;
      }
    }
    if (middle) {
      // diag_m - diag(l_m) D'^{-1}_{m-1} diag(u_{m-1}) - diag(u_m) D''^{-1}_{m+1} diag(l_{m+1})
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const int nb = side == 0 ? m - 1 : m + 1;
        if (nb < 0 || nb >= n_r || !valid) continue;
        const double *sc = (side == 0 ? upper : lower) + row_of(nb, 0);
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
          const int r = c0 + q * L;
          if (r >= n) continue;
          const double *inv = dinv + row_of(nb, r) * n;
          const double cl = side == 0 ? l[q] : u[q];
#pragma unroll
          for (int c = 0; c < CW; ++c)
            if (4 * c + w < n) a[q][c] = fma(-(cl * inv[4 * c + w]), sc[4 * c + w], a[q][c]);
        }
      }
    }
    __syncthreads();                                     // every thread has read the blocks and the scaling
    if (w == 0) {
#pragma unroll
      for (int q = 0; q < RPL; ++q) sm.ucol[g][c0 + q * L] = active ? u[q] : 0.0;
    }
    if (j + 1 < steps) {                                 // in flight while this zone is inverted
      fetch(j + 1);
      couplings(j + 1);
    }
    invert64<NP, RPL>(a, sm, g, c0, w);
    // the inverse to the factor array, whole blocks by all threads
#pragma unroll
    for (int h = 0; h < S; ++h) {
      const long it = (long)blockIdx.x * S + h;
      const int hf = middle ? 0 : (int)(it & 1);
      if (it >= n_items || j >= (middle ? 1 : (hf == 0 ? m : n_r - 1 - m))) continue;
      const long sy = listed_system(middle ? it : it >> 1, ray_list, NS);
      const int z = middle ? m : (hf == 0 ? j : n_r - 1 - j);
      double *out = dinv + ((size_t)sy * n_r + z) * nn;
      for (int e = threadIdx.x; e < nn; e += 128) out[e] = sm.tile[h][e / n][e % n];
    }
  }
}

template <int NP, int RPL>
static cudaError_t run_factor64(int n, int n_r, int n_sys, const double *diag, const double *lower, const double *upper,
                                double *dinv, const int *ray_list, cudaStream_t s, const int *n_dev) {
  constexpr int S = Quad<NP, RPL>::S;
  const int al16 = n % 2 == 0 && ((uintptr_t)diag & 15u) == 0;
  if (n_r > 1)
    k_factor64<NP, RPL><<<(unsigned)((2 * (long)n_sys + S - 1) / S), 128, 0, s>>>(n, n_r, n_sys, diag, lower, upper, dinv,
                                                                                ray_list, 0, al16, n_dev);
  k_factor64<NP, RPL><<<(unsigned)((n_sys + S - 1) / S), 128, 0, s>>>(n, n_r, n_sys, diag, lower, upper, dinv, ray_list, 1,
                                                                     al16, n_dev);
  return cudaGetLastError();
}

cudaError_t launch_factor64(int n, int n_r, int n_sys, const double *diag, const double *lower, const double *upper,
                            double *dinv, const int *ray_list, cudaStream_t s, const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  // RPL = 1 up to four CTAs per SM (1.3 us a pivot step at one CTA, 0.9 of the FP64 units' time at four),
  // RPL = 2 beyond (half the FP64 instructions per half) from 20 rows on; below, launch_factor takes a thread per
  // row there, and always up to 4 rows.
  MGFLD_DISPATCH_NP(n, {
    if constexpr (NP >= 20) {
      if (2 * (long)n_sys > 4L * kSMs * Quad<NP, 1>::S)
        return (run_factor64<NP, 2>(n, n_r, n_sys, diag, lower, upper, dinv, ray_list, s, n_dev));
    }
    if constexpr (NP == 4) return cudaErrorInvalidValue;
    else return (run_factor64<NP, 1>(n, n_r, n_sys, diag, lower, upper, dinv, ray_list, s, n_dev));
  })
}

}  // namespace mgfld
