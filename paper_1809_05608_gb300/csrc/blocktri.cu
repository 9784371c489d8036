// Batched block-Thomas elimination for the per-(ray, species) systems of Eq. a62ae.
//
// Structure exploited: the off-diagonal blocks are diagonal (the flux coefficient is
// frozen), so the Schur update of a zone is a diagonal scaling of its neighbour's
// inverse, e.g. D'_i = D_i - diag(l_i) D'^{-1}_{i-1} diag(u_{i-1}): no dense block product,
// hence no tensor-core contraction on this path.  Each dense block is inverted in
// place by Gauss-Jordan elimination with partial pivoting.
//
// Two-sided ("twisted") elimination: every system is eliminated top-down over zones
// 0..m-1 and bottom-up over zones n_r-1..m+1 at the same time, the two halves meeting at
// the middle zone m = n_r/2, whose block receives both Schur terms.  The substitution runs
// the same way (inward to the middle, then outward).  The sequential chain along the zones,
// which bounds these latency-limited kernels, is half as long, and there are twice as many
// independent instruction streams; the arithmetic is unchanged.
//
// The FP64 elimination of fewer systems is in factor64.cu, the ring-fed substitution in solve.cu.
#include "async.cuh"
#include "mgfld_internal.cuh"

namespace mgfld {

template <int NP>
struct Pack {
  static constexpr int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }
  // Half-systems per CTA: a multiple of 32 threads and even (both halves of a system share a CTA).
  static constexpr int SPC0 = 32 / gcd(NP, 32);
  static constexpr int SPC = SPC0 % 2 == 0 ? SPC0 : 2 * SPC0;
  static constexpr int THREADS = SPC * NP;
};

template <int NP>
__device__ inline int max_key(const int *__restrict__ c) {
  static_assert(NP % 4 == 0, "padded block sizes are multiples of 4");
  int m[NP / 4];
#pragma unroll
  for (int j = 0; j < NP / 4; ++j) {
    const int4 v = reinterpret_cast<const int4 *>(c)[j];
    m[j] = max(max(v.x, v.y), max(v.z, v.w));
  }
#pragma unroll
  for (int w = 1; w < NP / 4; w *= 2)
#pragma unroll
    for (int j = 0; j + w < NP / 4; j += 2 * w) m[j] = max(m[j], m[j + w]);
  return m[0];
}

// FP64 elimination of many systems: one thread per block row, SPC half-systems per CTA, every lane at work where
// k_factor64 leaves some of each warp idle; the same operations on every entry, the same inverses.  Per pivot
// step: barrier; every row reads the NP candidate keys of its system (NP/4 vector loads, a
// depth-log2 max tree); the pivot row publishes itself; barrier; every row forms its multiplier
// with one FMA and updates its NP entries.  The entry of the next pivot column is updated
// first and its key published at once, so that the next search only waits for that one FMA
// while the other NP - 1 drain through the FP64 pipe, which bounds it.
template <int NP>
__global__ void __launch_bounds__(Pack<NP>::THREADS, NP <= 20 ? 4 : 1)
k_factor(int n, int n_r, int n_sys, const double *__restrict__ diag, const double *__restrict__ lower,
         const double *__restrict__ upper, double *__restrict__ dinv, const int *__restrict__ ray_list,
         const int *__restrict__ n_dev) {
  constexpr int SPC = Pack<NP>::SPC;
  __shared__ double tile[SPC][NP][NP + 1];           // natural-order inverse of the previous zone
  __shared__ __align__(16) double prow[SPC][NP];     // pivot row of the current step
  __shared__ __align__(16) int cand[SPC][NP];        // pivot-search keys
  __shared__ double ushr[SPC][NP];                   // coupling to the next zone: the column scaling of its Schur term
  __shared__ int pivrow[SPC][NP];                    // row chosen at each step
  __shared__ double pinv[SPC];                       // 1 / pivot of the current step

  const int s = threadIdx.x / NP, r = threadIdx.x % NP;
  const int half = s & 1;                            // 0: zones 0..m top-down, 1: zones n_r-1..m+1 bottom-up
  const int n_sys_e = listed_sys(n_sys, n_dev, NS);
  if ((long)blockIdx.x * (SPC / 2) >= n_sys_e) return;   // the whole CTA
  const long jsys = (long)blockIdx.x * (SPC / 2) + (s >> 1);
  const bool valid = jsys < n_sys_e;
  const long sys = valid ? listed_system(jsys, ray_list, NS) : 0;
  const int m = n_r / 2;
  const int len = half == 0 ? m + 1 : n_r - 1 - m;   // zones of this half; all threads step m + 1 times

  // Each zone's rows are loaded when the zone starts: an FP64 zone step holds the pipe for far
  // longer than a memory round trip, and the registers of a prefetch would cost resident CTAs.
  for (int j = 0; j <= m; ++j) {
    const bool active = j < len;                     // inactive (bottom half, j >= len): dummy identity
    const int i = half == 0 ? j : n_r - 1 - j;
    const bool real = valid && active && r < n;
    const size_t zrow = ((size_t)sys * n_r + (real ? i : 0)) * n + r;   // (sys, i, r)
    double a[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) a[c] = (real && c < n) ? diag[zrow * n + c] : ((c == r) ? 1.0 : 0.0);
    const double lr = (real && j > 0) ? (half == 0 ? lower[zrow] : upper[zrow]) : 0.0;
    if (j > 0 && active) {
#pragma unroll
      for (int c = 0; c < NP; ++c) a[c] = fma(-(lr * tile[s][r][c]), ushr[s][c], a[c]);
    }
    if (half == 0 && j == m && n_r - 1 > m) {
      // Middle zone: also subtract the bottom-up half's term diag(u_m) D''^{-1}_{m+1} diag(l_{m+1})
      // (that half finished at step len - 1 < m; its tile and coupling are kept).
      const double um = real ? upper[zrow] : 0.0;
#pragma unroll
      for (int c = 0; c < NP; ++c) a[c] = fma(-(um * tile[s + 1][r][c]), ushr[s + 1][c], a[c]);
    }

    // Gauss-Jordan inversion in place with partial pivoting (implicit row exchanges).
    bool used = false;
    int my_step = 0;
    cand[s][r] = pivot_key(a[0], r);
#pragma unroll
    for (int pstep = 0; pstep < NP; ++pstep) {
      __syncthreads();
      const int best = 31 - (max_key<NP>(cand[s]) & 31);
      const bool me = (r == best);
      if (me) {
        // The pivot entry was updated first in the previous step, so its reciprocal is
        // formed while the rest of this row is still in the FP64 pipe.
        pinv[s] = recip(a[pstep]);
#pragma unroll
        for (int c = 0; c < NP; c += 2)
          *reinterpret_cast<double2 *>(&prow[s][c]) = make_double2(a[c], a[c + 1]);
        pivrow[s][pstep] = r;
        used = true;
        my_step = pstep;
      }
      __syncthreads();
      const double inv = pinv[s];
      // Uniform update for every row: a -= f * pivot_row, with f chosen so that the pivot row
      // itself becomes pivot_row / pivot (f = 1 - 1/pivot): one FMA either way.  The pivot
      // column itself is overwritten below, so its update is skipped.
      const double f = fma(me ? -1.0 : a[pstep], inv, me ? 1.0 : 0.0);
      if (pstep + 1 < NP) {
        a[pstep + 1] = fma(-f, prow[s][pstep + 1], a[pstep + 1]);
        cand[s][r] = used ? -1 : pivot_key(a[pstep + 1], r);
      }
      // the rest of the pivot row read from shared memory as it is used (16-byte pieces)
#pragma unroll
      for (int c = 0; c < NP; c += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(&prow[s][c]);
        if (c != pstep + 1 && c != pstep) a[c] = fma(-f, v.x, a[c]);
        if (c + 1 != pstep + 1 && c + 1 != pstep) a[c + 1] = fma(-f, v.y, a[c + 1]);
      }
      a[pstep] = me ? inv : -f;
    }
    // Row r now holds row my_step of the inverse, with column c belonging to input row pivrow[c].
    __syncthreads();
    if (active) {
#pragma unroll
      for (int c = 0; c < NP; ++c) tile[s][my_step][pivrow[s][c]] = a[c];
      ushr[s][r] = real ? (half == 0 ? upper[zrow] : lower[zrow]) : 0.0;
    }
    __syncthreads();
    if (real) {
      double *out = dinv + zrow * n;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c < n) out[c] = tile[s][r][c];
    }
  }
}

// FP64 substitution for many systems (spr per ray; the pair systems among them), and with factors that a caller of the C ABI
// holds off the 16-byte boundaries that the ring-fed one (solve.cu) needs; the same operations in the same order (one thread per block row, the
// two halves of each system in the same CTA, stepping together): forward g_i = Dinv_i (r_i -
// l_i g_{i-1}) for i < m and h_i = Dinv_i (r_i - u_i h_{i+1}) for i > m, the middle
// x_m = Dinv_m (r_m - l_m g_{m-1} - u_m h_{m+1}), then back outward from m.  The forward results
// are kept in x (which may alias rhs: each zone's rhs is read before its x is written).
template <int NP>
__global__ void __launch_bounds__(Pack<NP>::THREADS)
k_solve(int n, int n_r, int n_sys, int spr, const double *__restrict__ dinv, const double *__restrict__ lower,
        const double *__restrict__ upper, const double *rhs, double *x, const int *__restrict__ ray_list,
        const int *__restrict__ n_dev) {
  constexpr int SPC = Pack<NP>::SPC;
  __shared__ double v[SPC][NP];
  __shared__ double mid[SPC / 2][NP];               // h_{m+1}, then x_m
  const int s = threadIdx.x / NP, r = threadIdx.x % NP;
  const int half = s & 1, sl = s >> 1;
  const int n_sys_e = listed_sys(n_sys, n_dev, spr);
  if ((long)blockIdx.x * (SPC / 2) >= n_sys_e) return;   // the whole CTA
  const long jsys = (long)blockIdx.x * (SPC / 2) + sl;
  const bool valid = jsys < n_sys_e;
  const long sys = valid ? listed_system(jsys, ray_list, spr) : 0;
  const bool realr = valid && r < n;
  const size_t base = (size_t)sys * n_r * n;
  const int m = n_r / 2, B = n_r - 1 - m;
  const int F = half == 0 ? m : B;

  auto rowdot = [&](int z, bool real) {
    const double *src = dinv + (base + (size_t)z * n + r) * n;
    double acc0 = 0.0, acc1 = 0.0;
    if (real) {
#pragma unroll
      for (int c = 0; c < NP; c += 2) {
        if (c < n) acc0 = fma(src[c], v[s][c], acc0);
        if (c + 1 < n) acc1 = fma(src[c + 1], v[s][c + 1], acc1);
      }
    }
    return acc0 + acc1;
  };
  // Forward (all threads step m times for the barriers; a half past its F steps idles).
  double prev = 0.0;
  for (int j = 0; j < m; ++j) {
    const bool act = j < F;
    const bool real = realr && act;
    const int z = half == 0 ? j : n_r - 1 - j;
    const size_t zr = base + (size_t)(real ? z : 0) * n + r;
    const double c = (real && j > 0) ? (half == 0 ? lower[zr] : upper[zr]) : 0.0;
    const double b = real ? rhs[zr] : 0.0;
    v[s][r] = real ? b - c * prev : 0.0;
    __syncthreads();
    const double g = rowdot(z, real);
    if (real) {
      x[zr] = g;
      prev = g;
    }
    __syncthreads();
  }
  if (half == 1) mid[sl][r] = B > 0 ? prev : 0.0;
  __syncthreads();
  if (half == 0) {
    const size_t zr = base + (size_t)m * n + r;
    const double l = (realr && m > 0) ? lower[zr] : 0.0;
    const double u = (realr && m < n_r - 1) ? upper[zr] : 0.0;
    v[s][r] = realr ? rhs[zr] - l * prev - u * mid[sl][r] : 0.0;
  }
  __syncthreads();
  if (half == 0) {
    const double xm = rowdot(m, realr);
    if (realr) x[base + (size_t)m * n + r] = xm;
    prev = xm;
  }
  __syncthreads();
  if (half == 0) mid[sl][r] = prev;
  __syncthreads();
  if (half == 1) prev = mid[sl][r];
  // Backward: top x_i = g_i - Dinv_i (u_i x_{i+1}), i = m-1..0; bottom x_i = h_i - Dinv_i (l_i x_{i-1}).
  for (int j = 0; j < m; ++j) {
    const bool act = j < F;
    const bool real = realr && act;
    const int z = half == 0 ? m - 1 - j : m + 1 + j;
    const size_t zr = base + (size_t)(real ? z : 0) * n + r;
    const double c = real ? (half == 0 ? upper[zr] : lower[zr]) : 0.0;
    v[s][r] = real ? c * prev : 0.0;
    __syncthreads();
    const double acc = rowdot(z, real);
    if (real) {
      const double xi = x[zr] - acc;
      x[zr] = xi;
      prev = xi;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Thread-per-row elimination of systems of any block width up to 64 rows
// (the coupled nu / antinu blocks of the pair process: 2 n_e rows), in FP64 or FP32, with
// `spr` systems per ray (the launch's j-th system is system j % spr of ray ray_list[j / spr]).
// Partial pivoting through integer
// keys (6 row bits for blocks wider than 32), the next zone's rows fetched one zone ahead, the
// pivot row read from shared memory where it is used; shared memory sized at launch.
template <int NP, typename T>
struct RowCta {
  static constexpr int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }
  static constexpr int SPC0 = 32 / gcd(NP, 32);
  static constexpr int SPC = SPC0 % 2 == 0 ? SPC0 : 2 * SPC0;   // half-systems per CTA (even)
  static constexpr int THREADS = SPC * NP;
  static constexpr int KB = NP > 32 ? 6 : 5;                     // row bits of a pivot key
  static constexpr size_t TILE = sizeof(T) * SPC * NP * (NP + 1); // natural-order inverse of the previous zone
  static constexpr size_t PROW = sizeof(T) * SPC * NP;           // pivot row of the current step
  static constexpr size_t USHR = sizeof(T) * SPC * NP;           // column scaling of the next zone's Schur term
  static constexpr size_t PINV = 16 * SPC;                       // 1 / pivot (16-byte slots)
  static constexpr size_t CAND = sizeof(int) * SPC * NP;         // pivot-search keys
  static constexpr size_t PIVR = sizeof(int) * SPC * NP;         // row chosen at each step
  static constexpr size_t BYTES = TILE + PROW + USHR + PINV + CAND + PIVR;
};

template <int KB> __device__ inline int row_key(double x, int r) {
  const unsigned hi = (unsigned)((unsigned long long)__double_as_longlong(x) >> 32) & 0x7fffffffu;
  return (int)((hi & ~((1u << KB) - 1u)) | (unsigned)((1 << KB) - 1 - r));
}
template <int KB> __device__ inline int row_key(float x, int r) {
  const unsigned b = (unsigned)__float_as_int(x) & 0x7fffffffu;
  return (int)((b & ~((1u << KB) - 1u)) | (unsigned)((1 << KB) - 1 - r));
}
__device__ inline double recip_t(double d) { return recip(d); }
__device__ inline float recip_t(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float e = fmaf(-d, r, 1.f);
  return isfinite(r) ? fmaf(r, e, r) : r;
}

template <int NP, typename TIn, typename T>
__global__ void __launch_bounds__(RowCta<NP, T>::THREADS)
k_factor_rows(int n, int n_r, int n_sys, int spr, const TIn *__restrict__ diag, const T *__restrict__ lower,
              const T *__restrict__ upper, T *__restrict__ dinv, const int *__restrict__ ray_list,
              const int *__restrict__ bad, const int *__restrict__ n_dev) {
  using C = RowCta<NP, T>;
  constexpr int SPC = C::SPC, KB = C::KB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T (*tile)[NP][NP + 1] = reinterpret_cast<T (*)[NP][NP + 1]>(smem_raw);
  T (*prow)[NP] = reinterpret_cast<T (*)[NP]>(smem_raw + C::TILE);
  T (*ushr)[NP] = reinterpret_cast<T (*)[NP]>(smem_raw + C::TILE + C::PROW);
  T *pinv = reinterpret_cast<T *>(smem_raw + C::TILE + C::PROW + C::USHR);          // stride 16 bytes
  int (*cand)[NP] = reinterpret_cast<int (*)[NP]>(smem_raw + C::TILE + C::PROW + C::USHR + C::PINV);
  int (*pivrow)[NP] = reinterpret_cast<int (*)[NP]>(smem_raw + C::TILE + C::PROW + C::USHR + C::PINV + C::CAND);
  constexpr int PS = 16 / sizeof(T);                 // pinv slot stride in elements

  const int s = threadIdx.x / NP, r = threadIdx.x % NP;
  const int half = s & 1;                            // 0: zones 0..m top-down, 1: zones n_r-1..m+1 bottom-up
  const int n_sys_e = listed_sys(n_sys, n_dev, spr);
  if ((long)blockIdx.x * (SPC / 2) >= n_sys_e) return;   // the whole CTA
  if (bad) {                                         // only where the unpivoted elimination failed
    bool any = false;
    for (int c = 0; c < SPC / 2; ++c) {
      const long js = (long)blockIdx.x * (SPC / 2) + c;
      any = any || (js < n_sys_e && bad[js]);
    }
    if (!any) return;                                // the whole CTA
  }
  const long jsys = (long)blockIdx.x * (SPC / 2) + (s >> 1);
  const bool valid = jsys < n_sys_e;
  const long sys = valid ? listed_system(jsys, ray_list, spr) : 0;
  const int m = n_r / 2;
  const int len = half == 0 ? m + 1 : n_r - 1 - m;   // zones of this half; all threads step m + 1 times
  const T one = T(1), zero = T(0);

  T nxt[NP];
  T nl = zero;
  auto load_row = [&](int j) {
    const bool act = valid && j < len && r < n;
    const int z = half == 0 ? j : n_r - 1 - j;
    const size_t zr = ((size_t)sys * n_r + (act ? z : 0)) * n + r;
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      if (act && c < n) nxt[c] = (T)diag[zr * n + c];
      else nxt[c] = (c == r) ? one : zero;
    }
    nl = (act && j > 0) ? (half == 0 ? lower[zr] : upper[zr]) : zero;
  };
  load_row(0);
  for (int j = 0; j <= m; ++j) {
    const bool active = j < len;
    const int i = half == 0 ? j : n_r - 1 - j;
    const bool real = valid && active && r < n;
    const size_t zrow = ((size_t)sys * n_r + (real ? i : 0)) * n + r;
    T a[NP];
#pragma unroll
    for (int c = 0; c < NP; ++c) a[c] = nxt[c];
    const T lr = nl;
    if (j + 1 <= m) load_row(j + 1);
    if (j > 0 && active) {
#pragma unroll
      for (int c = 0; c < NP; ++c) a[c] = fma(-(lr * tile[s][r][c]), ushr[s][c], a[c]);
    }
    if (half == 0 && j == m && n_r - 1 > m) {
      const T um = real ? upper[zrow] : zero;
#pragma unroll
      for (int c = 0; c < NP; ++c) a[c] = fma(-(um * tile[s + 1][r][c]), ushr[s + 1][c], a[c]);
    }
    bool used = false;
    int my_step = 0;
    cand[s][r] = row_key<KB>(a[0], r);
#pragma unroll
    for (int pstep = 0; pstep < NP; ++pstep) {
      __syncthreads();
      int best_key = cand[s][0];
#pragma unroll
      for (int c = 1; c < NP; ++c) best_key = max(best_key, cand[s][c]);
      const int best = (1 << KB) - 1 - (best_key & ((1 << KB) - 1));
      const bool me = (r == best);
      if (me) {
        pinv[s * PS] = recip_t(a[pstep]);
#pragma unroll
        for (int c = 0; c < NP; ++c) prow[s][c] = a[c];
        pivrow[s][pstep] = r;
        used = true;
        my_step = pstep;
      }
      __syncthreads();
      const T inv = pinv[s * PS];
      const T f = fma(me ? -one : a[pstep], inv, me ? one : zero);
      if (pstep + 1 < NP) {
        a[pstep + 1] = fma(-f, prow[s][pstep + 1], a[pstep + 1]);
        cand[s][r] = used ? -1 : row_key<KB>(a[pstep + 1], r);
      }
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c != pstep + 1 && c != pstep) a[c] = fma(-f, prow[s][c], a[c]);
      a[pstep] = me ? inv : -f;
    }
    __syncthreads();
    if (active) {
#pragma unroll
      for (int c = 0; c < NP; ++c) tile[s][my_step][pivrow[s][c]] = a[c];
      ushr[s][r] = real ? (half == 0 ? upper[zrow] : lower[zrow]) : zero;
    }
    __syncthreads();
    if (real) {
      T *out = dinv + zrow * n;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c < n) out[c] = tile[s][r][c];
    }
  }
}

// ---------------------------------------------------------------------------------------
// Warp-synchronous FP32 variants (MIXED precision): one warp per half of a (ray, species)
// system, lane r owns block row r (NP <= 32), no CTA-wide barriers.  FP32 arithmetic is 63x
// cheaper than FP64 on this GPU, so these kernels are bound by the dependency chain along the
// zones and by the instruction and shared-memory traffic of each zone step.
constexpr int kWarpsPerCta = 4;

// FP32 reciprocal: the hardware approximation (rcp.approx.ftz) refined by one Newton step, a
// few multiply-adds instead of the correctly rounded library reciprocal; ample for the FP32
// preconditioner.  rcp(0) = inf and rcp(NaN) = NaN as before.
__device__ inline float rcp_nr(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  const float e = fmaf(-x, r, 1.f);
  return isfinite(r) ? fmaf(r, e, r) : r;
}

// Packed FP32 helpers (two lanes of arithmetic per instruction).
__device__ inline void fma2_row(float *a, float s, const float *p, int c) {
  const float2 r = __ffma2_rn(make_float2(s, s), make_float2(p[c], p[c + 1]), make_float2(a[c], a[c + 1]));
  a[c] = r.x;
  a[c + 1] = r.y;
}

// In-place Gauss-Jordan inverse with partial pivoting of the warp's NP x NP zone block, lane r
// holding row r.  The pivot is found with a warp max reduction on integer keys (|a| bits with
// the row index in the 5 low bits), the pivot row is broadcast through a double-buffered
// shared-memory row (one 16-byte store per 4 entries by its owner, broadcast 16-byte loads by
// every lane), and the eliminations run as packed FP32 FMAs.  Returns with a[] holding row
// my_step of the inverse with column c belonging to natural column piv(c) (byte c % 4 of
// piv[c / 4]).
template <int NP>
__device__ inline void gj_invert(float *a, float (*prow)[NP + 4], int r, bool row, int &my_step, unsigned *piv) {
  const unsigned full = 0xffffffffu;
  bool used = !row;
  my_step = 0;
  int key = used ? -1 : (int)(((unsigned)__float_as_int(fabsf(a[0])) & ~31u) | (unsigned)(31 - r));
#pragma unroll
  for (int ps = 0; ps < NP; ++ps) {
    const int best = 31 - (__reduce_max_sync(full, key) & 31);
    if (ps % 4 == 0) piv[ps / 4] = (unsigned)best;      // four 8-bit pivot rows per register
    else piv[ps / 4] |= (unsigned)best << (8 * (ps % 4));
    const bool me = (r == best);
    float *pb = prow[ps & 1];
    if (me) {
      used = true;
      my_step = ps;
#pragma unroll
      for (int c = 0; c < NP; c += 4)
        *reinterpret_cast<float4 *>(pb + c) = make_float4(a[c], a[c + 1], a[c + 2], a[c + 3]);
    }
    __syncwarp();
    float pv[NP];
#pragma unroll
    for (int c = 0; c < NP; c += 4) {
      const float4 v = *reinterpret_cast<const float4 *>(pb + c);
      pv[c] = v.x;
      pv[c + 1] = v.y;
      pv[c + 2] = v.z;
      pv[c + 3] = v.w;
    }
    const float inv = rcp_nr(pv[ps]);
    const float f = fmaf(me ? -1.f : a[ps], inv, me ? 1.f : 0.f);
    // the pair holding the next pivot column first, so that the next search can start
    if (ps + 1 < NP) {
      const int cn = (ps + 1) & ~1;
      fma2_row(a, -f, pv, cn);
      key = used ? -1 : (int)(((unsigned)__float_as_int(fabsf(a[ps + 1])) & ~31u) | (unsigned)(31 - r));
#pragma unroll
      for (int c = 0; c < NP; c += 2)
        if (c != cn) fma2_row(a, -f, pv, c);
    } else {
#pragma unroll
      for (int c = 0; c < NP; c += 2) fma2_row(a, -f, pv, c);
    }
    a[ps] = me ? inv : -f;
  }
}

// CTAs per SM the FP32 factor is compiled for (its register budget): the kernel is bound by the
// latency of its pivot chain, so resident warps matter more than a few spilled registers.
#ifndef MGFLD_FW32_MINB
#define MGFLD_FW32_MINB 4
#endif

// Warps per CTA of the factor: four (two systems), two for the widest blocks so that the
// static shared memory (two row buffers and the inverse tile per warp) stays under 48 KB.
template <int NP> __host__ __device__ constexpr int fw_wpc() { return NP > 24 ? 2 : 4; }

// The C ABI's factor of arbitrary systems: partial pivoting in every zone.  At most 128 registers (NP <= 24), so that four
// CTAs (eight systems) fit on an SM and the 256-ray workload's 512 CTAs run in a single wave on 152 SMs.
template <int NP>
__global__ void __launch_bounds__(fw_wpc<NP>() * 32, MGFLD_FW32_MINB)
k_factor_w32(int n, int n_r, int n_sys, const double *__restrict__ diag, const double *__restrict__ lower,
             const double *__restrict__ upper, float *__restrict__ dinv, const int *__restrict__ ray_list,
             const int *__restrict__ n_dev) {
  static_assert(NP % 4 == 0, "rows of NP floats in 16-byte pieces");
  // tile: the natural-order inverse of each warp's last zone (read by the other half at the
  // middle zone); ushr: that zone's coupling to the next zone of the sequence; prow: pivot rows.
  constexpr int W = fw_wpc<NP>();
  __shared__ __align__(16) float tile[W][NP][NP];
  __shared__ __align__(16) float ushr[W][NP];
  __shared__ __align__(16) float prow[W][2][NP + 4];
  __shared__ __align__(16) float rowbuf[W][2][NP][NP];
  const int wid = threadIdx.x >> 5, r = threadIdx.x & 31;
  const int half = wid & 1;                          // 0: zones 0..m top-down, 1: zones n_r-1..m+1 bottom-up
  const long jsys = (long)blockIdx.x * (W / 2) + (wid >> 1);
  if (jsys >= listed_sys(n_sys, n_dev, NS)) return;  // both warps of the system leave; no barrier below
  const long sys = listed_system(jsys, ray_list, NS);
  const bool real = r < n;
  const bool row = r < NP;
  const int m = n_r / 2;
  const int len = half == 0 ? m + 1 : n_r - 1 - m;
  auto zone = [&](int j) { return half == 0 ? j : n_r - 1 - j; };
  // Next zone's rows, fetched one zone ahead into a double-buffered shared-memory block (each lane its own row, so
  // that no registers hold the prefetch), and its couplings into registers.  The coupling loads are unconditional
  // (lanes without a row read row 0) with the conditions applied when the values are consumed, so that no instruction
  // waits on a load in the zone it was issued.
  const int rr = real ? r : 0;
  double nl_raw = 0.0, nu_raw = 0.0;
  auto load_row = [&](int j) {
    const size_t zr = ((size_t)sys * n_r + zone(j)) * n + rr;
    float *dst = &rowbuf[wid][j & 1][row ? r : 0][0];
    if (row) {
#pragma unroll
      for (int c = 0; c < NP; ++c) dst[c] = (real && c < n) ? (float)diag[zr * n + c] : ((c == r) ? 1.f : 0.f);
    }
    nl_raw = half == 0 ? lower[zr] : upper[zr];
    nu_raw = half == 0 ? upper[zr] : lower[zr];
  };
  if (len > 0) load_row(0);
  for (int j = 0; j < len; ++j) {
    const int z = zone(j);
    const size_t zrow = ((size_t)sys * n_r + z) * n + r;
    const float lr = (real && j > 0) ? (float)nl_raw : 0.f;
    const float ur = real ? (float)nu_raw : 0.f;
    if (j + 1 < len) load_row(j + 1);
    // Middle zone: wait for the bottom-up half of this system (its last tile and coupling).
    const bool mid = half == 0 && j == m;
    if (mid) asm volatile("bar.sync %0, 64;" ::"r"(1 + (wid >> 1)) : "memory");
    float a[NP];
    // The zone's Schur complement from its raw rows and the previous zone's inverse (this warp's tile).
    {
      if (row) {
#pragma unroll
        for (int c = 0; c < NP; c += 4) {
          const float4 v = *reinterpret_cast<const float4 *>(&rowbuf[wid][j & 1][r][c]);
          a[c] = v.x;
          a[c + 1] = v.y;
          a[c + 2] = v.z;
          a[c + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < NP; ++c) a[c] = 0.f;
      }
      if (j > 0 && row) {
        // a -= diag(l) Dinv_prev diag(u_prev): row scale lr, column scale ushr
#pragma unroll
        for (int c = 0; c < NP; c += 4) {
          const float4 u = *reinterpret_cast<const float4 *>(&ushr[wid][c]);
          const float4 d = *reinterpret_cast<const float4 *>(&tile[wid][r][c]);
          const float2 t0 = __fmul2_rn(make_float2(-lr, -lr), make_float2(d.x, d.y));
          const float2 t1 = __fmul2_rn(make_float2(-lr, -lr), make_float2(d.z, d.w));
          const float2 r0 = __ffma2_rn(t0, make_float2(u.x, u.y), make_float2(a[c], a[c + 1]));
          const float2 r1 = __ffma2_rn(t1, make_float2(u.z, u.w), make_float2(a[c + 2], a[c + 3]));
          a[c] = r0.x;
          a[c + 1] = r0.y;
          a[c + 2] = r1.x;
          a[c + 3] = r1.y;
        }
      }
      if (mid && n_r - 1 > m && row) {
        // the bottom-up half's Schur term diag(u_m) D''^{-1}_{m+1} diag(l_{m+1}) as well
#pragma unroll
        for (int c = 0; c < NP; ++c) a[c] = a[c] - (ur * tile[wid ^ 1][r][c]) * ushr[wid ^ 1][c];
      }
    }
    int my_step;
    unsigned piv[NP / 4];
    gj_invert<NP>(a, prow[wid], r, row, my_step, piv);
    __syncwarp();                  // every lane has read the previous zone's tile row
    if (row) {
#pragma unroll
      for (int c = 0; c < NP; ++c) tile[wid][my_step][(piv[c / 4] >> (8 * (c % 4))) & 0xffu] = a[c];
    }
    __syncwarp();
    if (row) ushr[wid][r] = ur;   // column scaling of this zone's Schur term in the next zone
    if (real) {
      float *out = dinv + zrow * n;
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c < n) out[c] = tile[wid][r][c];
    }
    __syncwarp();
  }
  if (half == 1) asm volatile("bar.sync %0, 64;" ::"r"(1 + (wid >> 1)) : "memory");
}

// ---------------------------------------------------------------------------------------
// FP32 factor of the outer iteration with two block rows per lane (the mixed path's zone blocks,
// M-matrices: no row exchanges).  L = NP/2 lanes hold a half-system, lane m rows m and m + L, and a
// warp holds S = 32 / L half-systems (three at NP = 20); warp 0 of a
// CTA takes the top-down halves and warp 1 the bottom-up halves of the same S systems.  Every pivot row
// is read from shared memory once per lane for its two rows, so a broadcast serves twice the rows and S
// systems at once: the shared-memory traffic per system, which bounds a one-row-per-lane kernel, drops
// about threefold.  Gauss-Jordan with 2 x 2 pivot blocks: the owners of rows p and p + 1 publish both,
// every lane inverts the pivot block in closed form (one reciprocal of its determinant) and
// eliminates with the two multipliers (a_p, a_{p+1}) P^{-1}; leading 2 x 2 blocks of the Schur
// complements of an M-matrix are nonsingular, so no exchanges are needed.  The Schur term of the next
// zone is formed from the lane's own rows of the inverse, still in registers (row r of the inverse stays
// with the lane of row r); the next zone's rows and couplings arrive by asynchronous copies issued one
// zone ahead.  A zone whose 2 x 2 pivot block is singular or not finite leaves its inverse non-finite, and the
// outer iteration reports ENAN for the ray.  Where the launch keeps flags (padded and pair blocks), a system is done again
// with partial pivoting unless its pivot blocks are those of an M-matrix: determinant and diagonal entries positive, no
// entry above kGrowth times the raw one (elimination only takes from an M-matrix's diagonal).  An iterate with
// occupations outside [0, 1] makes blocks that are none, and an unnoticed small pivot there factors without a correct
// digit.  (The check, in integers: a step at 173 rays of 301 x 13 3.75 -> 3.75 ms, 3.78 with FP32 comparisons; with pairs
// at 256 rays of 512 x 20 25.37 -> 25.48 ms.)
// Bound by the issue slots of the row updates; measured at 1024 rays of 512 x 20: 2.05 ms.  (Publishing the next
// pivots before the other row is updated, as k_factor_wide does, spills here: 2.50 ms.)
template <int NP>
struct Row2 {
  static constexpr int L = NP / 2;                 // lanes per half-system
  static constexpr int S = 32 / L;                 // half-systems per warp
  static constexpr int PAD = (NP / 4) % 2 ? NP : NP + 4;   // pivot-row stride: an odd number of
                                                           // 16-byte pieces (conflict-free reads)
};

constexpr float kGrowth = 4.f;
// 0 < d <= top by the bit patterns (top's, 0 if it is not positive; NaN and negative d are above it)
__device__ inline unsigned growth_limit(float raw) { return raw > 0.f ? __float_as_uint(kGrowth * raw) : 0u; }
__device__ inline bool in_range(float d, unsigned top) { return __float_as_uint(d) - 1u < top; }

// CTAs per SM the two-rows-per-lane factor is compiled for (its register budget).
template <int NP>
__host__ __device__ constexpr int row2_minb() { return NP <= 20 ? 9 : 6; }

// FULL: n = NP, rows in 16-byte pieces; otherwise rows and columns beyond n are padded with the
// identity.  spr: systems per ray.  FLAG: bad[listed system] is set to whether a pivot block was not an
// M-matrix's.
template <int NP, bool FULL, bool FLAG>
__global__ void __launch_bounds__(64, row2_minb<NP>())
k_factor_row2(int n_, int n_r, int n_sys, int spr, const float *__restrict__ diag, const float *__restrict__ lower,
              const float *__restrict__ upper, float *__restrict__ dinv, const int *__restrict__ ray_list,
              int *__restrict__ bad, const int *__restrict__ n_dev) {
  using C = Row2<NP>;
  constexpr int L = C::L, S = C::S, PD = C::PAD;
  const int n = FULL ? NP : n_;
  static_assert(NP % 4 == 0 && L % 2 == 0, "pivot pairs in one lane pair, rows in 16-byte pieces");
  // The next zone's rows and couplings arrive by cp.async, per warp (each lane copies and later
  // reads only its own two rows: 80-byte rows are conflict-free for its 16-byte reads); after its
  // last zone the bottom-up warp leaves its last inverse in its row buffer for the middle zone of
  // the top-down warp.
  __shared__ __align__(16) float rows[2][S][NP][NP];       // the next zone's rows, per warp
  __shared__ __align__(16) float cpl[2][S][2][NP];         // its couplings (to the previous / next zone)
  __shared__ __align__(16) float prow[2][2][S][2][PD];     // per warp, double-buffered pivot row pairs
  __shared__ __align__(16) float ucol[2][S][NP];           // column scaling of the next zone's Schur term
  __shared__ int okb[S];                                   // the bottom-up half's pivots were fine
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = wid;                                    // 0: zones 0..m top-down, 1: n_r-1..m+1 bottom-up
  const int g = lane / L, mm = lane % L;                   // half-system of the warp, lane in it
  const int n_sys_e = listed_sys(n_sys, n_dev, spr);
  const long j0 = (long)blockIdx.x * S;
  if (j0 >= n_sys_e) return;                               // the whole CTA
  const long jsys = j0 + g;
  const bool valid = g < S && jsys < n_sys_e;
  const long sys = valid ? listed_system(jsys, ray_list, spr) : 0;
  const int gs = g < S ? g : 0;                            // shared-memory slot (idle lanes use 0)
  const int m = n_r / 2;
  const int len = half == 0 ? m + 1 : n_r - 1 - m;
  auto zone = [&](int j) { return half == 0 ? j : n_r - 1 - j; };
  const int r0 = mm, r1 = mm + L;                          // this lane's two rows
  // a padded row: the identity (its lane's own rows only; no copy touches columns beyond n)
  if (!FULL && g < S) {
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      rows[wid][gs][r0][c] = c == r0 ? 1.f : 0.f;
      rows[wid][gs][r1][c] = c == r1 ? 1.f : 0.f;
    }
    cpl[wid][gs][0][r0] = cpl[wid][gs][0][r1] = cpl[wid][gs][1][r0] = cpl[wid][gs][1][r1] = 0.f;
  }
  auto issue = [&](int j) {                                // rows and couplings of zone j
    if (valid && j < len) {
      const size_t zb = ((size_t)sys * n_r + zone(j)) * n;
      const float *lin = half == 0 ? lower : upper, *lout = half == 0 ? upper : lower;
      if (FULL) {
#pragma unroll
        for (int c = 0; c < NP; c += 4) {
          cp_async16(&rows[wid][gs][r0][c], diag + (zb + r0) * NP + c);
          cp_async16(&rows[wid][gs][r1][c], diag + (zb + r1) * NP + c);
        }
        cp_async4(&cpl[wid][gs][0][r0], lin + zb + r0);
        cp_async4(&cpl[wid][gs][0][r1], lin + zb + r1);
        cp_async4(&cpl[wid][gs][1][r0], lout + zb + r0);
        cp_async4(&cpl[wid][gs][1][r1], lout + zb + r1);
      } else {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const int r = p == 0 ? r0 : r1;
          if (r < n) {
            const float *src = diag + (zb + r) * n;
            float *dst = &rows[wid][gs][r][0];
            if (n % 2 == 0)
              for (int c = 0; c < n; c += 2) cp_async8(dst + c, src + c);
            else
              for (int c = 0; c < n; ++c) cp_async4(dst + c, src + c);
            cp_async4(&cpl[wid][gs][0][r], lin + zb + r);
            cp_async4(&cpl[wid][gs][1][r], lout + zb + r);
          }
        }
      }
    }
    cp_async_commit();
  };
  float (*midt)[NP][NP] = rows[1];                         // the bottom-up warp's last inverse
  float a0[NP], a1[NP];
  bool ok = true;
  issue(0);
  for (int j = 0; j < len; ++j) {
    cp_async_wait_all();
    __syncwarp();
    // the zone's rows minus the Schur term of the previous zone: row r gets
    // -l_r (row r of the previous inverse, this lane's registers) * u_prev (column scaling)
    // (lanes without a system run on whatever their slot holds: they store nothing, and a slot
    // without a system is read by its own lanes only)
    const unsigned top0 = growth_limit(rows[wid][gs][r0][r0]), top1 = growth_limit(rows[wid][gs][r1][r1]);   // (FLAG)
    const float l0 = cpl[wid][gs][0][r0], l1 = cpl[wid][gs][0][r1];   // used from the second zone on
    const float u0 = cpl[wid][gs][1][r0], u1 = cpl[wid][gs][1][r1];
#pragma unroll
    for (int c = 0; c < NP; c += 4) {
      float4 x0 = *reinterpret_cast<const float4 *>(&rows[wid][gs][r0][c]);
      float4 x1 = *reinterpret_cast<const float4 *>(&rows[wid][gs][r1][c]);
      if (j > 0) {
        const float4 u = *reinterpret_cast<const float4 *>(&ucol[wid][gs][c]);
        x0.x = fmaf(-(l0 * a0[c]), u.x, x0.x);
        x0.y = fmaf(-(l0 * a0[c + 1]), u.y, x0.y);
        x0.z = fmaf(-(l0 * a0[c + 2]), u.z, x0.z);
        x0.w = fmaf(-(l0 * a0[c + 3]), u.w, x0.w);
        x1.x = fmaf(-(l1 * a1[c]), u.x, x1.x);
        x1.y = fmaf(-(l1 * a1[c + 1]), u.y, x1.y);
        x1.z = fmaf(-(l1 * a1[c + 2]), u.z, x1.z);
        x1.w = fmaf(-(l1 * a1[c + 3]), u.w, x1.w);
      }
      a0[c] = x0.x; a0[c + 1] = x0.y; a0[c + 2] = x0.z; a0[c + 3] = x0.w;
      a1[c] = x1.x; a1[c + 1] = x1.y; a1[c + 2] = x1.z; a1[c + 3] = x1.w;
    }
    __syncwarp();                                          // every lane has read the rows and ucol
    issue(j + 1);
    if (half == 0 && j == m) {
      // middle zone: wait for the bottom-up half (which arrives once, after its last zone, whatever
      // its length) and subtract its term diag(u_m) D''^{-1}_{m+1} diag(l_{m+1}) as well
      asm volatile("bar.sync 1, 64;" ::: "memory");
      if (n_r - 1 > m) {
#pragma unroll
        for (int c = 0; c < NP; ++c) {
          const float lc = ucol[1][gs][c];
          a0[c] = fmaf(-(u0 * midt[gs][r0][c]), lc, a0[c]);
          a1[c] = fmaf(-(u1 * midt[gs][r1][c]), lc, a1[c]);
        }
      }
    }
    // Gauss-Jordan inversion with 2 x 2 pivot blocks (rows p, p + 1: lanes p % L and p % L + 1 of
    // slot p / L, known at compile time)
#pragma unroll
    for (int b = 0; b < NP / 2; ++b) {
      const int p = 2 * b, sl = p / L, pl = p % L;
      float (*pb)[2][PD] = prow[wid][b & 1];
      if (g < S && (mm == pl || mm == pl + 1)) {          // lanes beyond the S half-systems publish nothing
        float *dst = pb[gs][mm - pl];
#pragma unroll
        for (int c = 0; c < NP; c += 4) {
          if (sl == 0) *reinterpret_cast<float4 *>(dst + c) = make_float4(a0[c], a0[c + 1], a0[c + 2], a0[c + 3]);
          else *reinterpret_cast<float4 *>(dst + c) = make_float4(a1[c], a1[c + 1], a1[c + 2], a1[c + 3]);
        }
      }
      __syncwarp();
      const float2 q0 = *reinterpret_cast<const float2 *>(&pb[gs][0][p]);
      const float2 q1 = *reinterpret_cast<const float2 *>(&pb[gs][1][p]);
      const float det = fmaf(q0.x, q1.y, -(q0.y * q1.x));
      const float idet = rcp_nr(det);
      if (FLAG) {
        ok = ok && idet > 0.f && (p + 2 < NP || idet < INFINITY);   // (an infinite one makes the next NaN)
        if (mm == pl || mm == pl + 1) ok = ok && in_range(mm == pl ? q0.x : q1.y, sl == 0 ? top0 : top1);
      }
      const float i00 = q1.y * idet, i01 = -q0.y * idet, i10 = -q1.x * idet, i11 = q0.x * idet;
      // multipliers of the two rows: owners take the rows of P^{-1} times the pivot rows
      float f00, f01, f10, f11;
      if (sl == 0 && mm == pl) { f00 = 1.f - i00; f01 = -i01; }
      else if (sl == 0 && mm == pl + 1) { f00 = -i10; f01 = 1.f - i11; }
      else { f00 = fmaf(a0[p], i00, a0[p + 1] * i10); f01 = fmaf(a0[p], i01, a0[p + 1] * i11); }
      if (sl == 1 && mm == pl) { f10 = 1.f - i00; f11 = -i01; }
      else if (sl == 1 && mm == pl + 1) { f10 = -i10; f11 = 1.f - i11; }
      else { f10 = fmaf(a1[p], i00, a1[p + 1] * i10); f11 = fmaf(a1[p], i01, a1[p + 1] * i11); }
#pragma unroll
      for (int c = 0; c < NP; c += 4) {
        const float4 v0 = *reinterpret_cast<const float4 *>(&pb[gs][0][c]);
        const float4 v1 = *reinterpret_cast<const float4 *>(&pb[gs][1][c]);
        float2 lo = __ffma2_rn(make_float2(-f00, -f00), make_float2(v0.x, v0.y), make_float2(a0[c], a0[c + 1]));
        float2 hi = __ffma2_rn(make_float2(-f00, -f00), make_float2(v0.z, v0.w), make_float2(a0[c + 2], a0[c + 3]));
        lo = __ffma2_rn(make_float2(-f01, -f01), make_float2(v1.x, v1.y), lo);
        hi = __ffma2_rn(make_float2(-f01, -f01), make_float2(v1.z, v1.w), hi);
        a0[c] = lo.x; a0[c + 1] = lo.y; a0[c + 2] = hi.x; a0[c + 3] = hi.y;
        lo = __ffma2_rn(make_float2(-f10, -f10), make_float2(v0.x, v0.y), make_float2(a1[c], a1[c + 1]));
        hi = __ffma2_rn(make_float2(-f10, -f10), make_float2(v0.z, v0.w), make_float2(a1[c + 2], a1[c + 3]));
        lo = __ffma2_rn(make_float2(-f11, -f11), make_float2(v1.x, v1.y), lo);
        hi = __ffma2_rn(make_float2(-f11, -f11), make_float2(v1.z, v1.w), hi);
        a1[c] = lo.x; a1[c + 1] = lo.y; a1[c + 2] = hi.x; a1[c + 3] = hi.y;
      }
      if (sl == 0 && mm == pl) { a0[p] = i00; a0[p + 1] = i01; }
      else if (sl == 0 && mm == pl + 1) { a0[p] = i10; a0[p + 1] = i11; }
      else { a0[p] = -f00; a0[p + 1] = -f01; }
      if (sl == 1 && mm == pl) { a1[p] = i00; a1[p + 1] = i01; }
      else if (sl == 1 && mm == pl + 1) { a1[p] = i10; a1[p + 1] = i11; }
      else { a1[p] = -f10; a1[p + 1] = -f11; }
    }
    // the inverse rows to the factor buffer, and this zone's coupling to the next zone of the
    // sequence (column scaling of the next Schur term) to the warp's shared row
    if (valid) {
      float *o0 = dinv + (((size_t)sys * n_r + zone(j)) * n + r0) * n;
      float *o1 = dinv + (((size_t)sys * n_r + zone(j)) * n + r1) * n;
      if (FULL) {
#pragma unroll
        for (int c = 0; c < NP; c += 4) {
          *reinterpret_cast<float4 *>(o0 + c) = make_float4(a0[c], a0[c + 1], a0[c + 2], a0[c + 3]);
          *reinterpret_cast<float4 *>(o1 + c) = make_float4(a1[c], a1[c + 1], a1[c + 2], a1[c + 3]);
        }
      } else {
#pragma unroll
        for (int c = 0; c < NP; ++c) {
          if (r0 < n && c < n) o0[c] = a0[c];
          if (r1 < n && c < n) o1[c] = a1[c];
        }
      }
    }
    if (g < S) {
      ucol[wid][gs][r0] = u0;
      ucol[wid][gs][r1] = u1;
    }
    if (half == 1 && j == len - 1 && g < S) {
      // the bottom-up half's last inverse for the middle zone of the top-down half
#pragma unroll
      for (int c = 0; c < NP; ++c) {
        midt[gs][r0][c] = a0[c];
        midt[gs][r1][c] = a1[c];
      }
    }
    __syncwarp();
  }
  cp_async_wait_all();
  if (FLAG) {
    // every lane of the half-system
    constexpr unsigned lanes = 0xffffffffu >> (32 - L);
    ok = ((__ballot_sync(0xffffffffu, ok) >> (gs * L)) & lanes) == lanes;
  }
  if (half == 1) {
    if (FLAG && g < S && mm == 0) okb[gs] = ok;            // (read after the barrier, the top half's last zone)
    asm volatile("bar.sync 1, 64;" ::: "memory");
  } else if (FLAG && valid && mm == 0) {
    bad[jsys] = !(ok && okb[gs]);
  }
}

// The same factor, a warp per half-system, for launches that leave most of the chip idle and for the pair systems:
// lane (g, m) holds C columns of the R rows m, m + L, ..., the columns dealt to G groups of L lanes (three groups
// of 8, 8 and 4 columns of two rows at NP = 20, of 16, 16 and 8 columns of four rows at NP = 40), so that a
// pivot costs a lane a third of the row updates; the multipliers' two columns come from their group by shuffles.
// The rows that hold the next pivots are updated and published first, the others while those stores are
// under way.  Every entry takes the same operations in the same order as in k_factor_row2: the same inverses.
// Bound by the latency of the pivot chain; measured against k_factor_row2 (512 zones): 32 rays of 20 groups
// 609 -> 325 us, 256 rays 900 -> 689 us, 173 rays of 301 x 13 431 -> 318 us, 256 rays of 40-row pair systems
// 2.83 -> 2.26 ms (one row per thread with CTA barriers and partial pivoting, k_factor_rows: 8.0 ms).
template <int NP>
struct Wide {
  static constexpr int R = NP > 32 ? 4 : 2;                    // rows per lane
  static constexpr int L = NP / R;                             // lanes per column group
  static constexpr int G0 = 32 / L < NP / 4 ? 32 / L : NP / 4;
  static constexpr int C = ((NP + G0 - 1) / G0 + 3) / 4 * 4;   // columns per lane
  static constexpr int G = (NP + C - 1) / C;                   // column groups
  static constexpr int W = G * C;                              // padded row
};

template <int NP, bool FULL, bool FLAG>
__global__ void __launch_bounds__(64)
k_factor_wide(int n_, int n_r, int n_sys, int spr, const float *__restrict__ diag, const float *__restrict__ lower,
              const float *__restrict__ upper, float *__restrict__ dinv, const int *__restrict__ ray_list,
              int *__restrict__ bad, const int *__restrict__ n_dev) {
  using Q = Wide<NP>;
  constexpr int R = Q::R, L = Q::L, C = Q::C, G = Q::G, W = Q::W;
  static_assert(NP % 4 == 0 && L % 2 == 0 && L * G <= 32, "pivot pairs in one lane pair, rows in 16-byte pieces");
  const int n = FULL ? NP : n_;
  // (columns from NP to W stay zero throughout)
  __shared__ __align__(16) float rows[2][NP][W];           // the next zone's rows, per warp
  __shared__ __align__(16) float cpl[2][2][NP];            // its couplings (to the previous / next zone)
  __shared__ __align__(16) float prow[2][2][2][W];         // per warp, double-buffered pivot row pairs
  __shared__ __align__(16) float ucol[2][W];               // column scaling of the next zone's Schur term
  __shared__ int okb;                                      // the bottom-up half's pivots were fine
  const int half = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool act = lane < L * G;                           // the other lanes repeat the first group's and store nothing
  const int cg = act ? lane / L : 0, mm = lane % L, c0 = cg * C;
  const long jsys = blockIdx.x;
  if (jsys >= listed_sys(n_sys, n_dev, spr)) return;       // the whole CTA
  const size_t sys = (size_t)listed_system(jsys, ray_list, spr);
  const int m = n_r / 2;
  const int len = half == 0 ? m + 1 : n_r - 1 - m;
  auto zone = [&](int j) { return half == 0 ? j : n_r - 1 - j; };
  if (act) {
    // what no copy touches: the identity, without couplings
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = mm + i * L;
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (r >= n || c0 + c >= n) rows[half][r][c0 + c] = c0 + c == r ? 1.f : 0.f;
      if (cg == 0 && r >= n) cpl[half][0][r] = cpl[half][1][r] = 0.f;
    }
    if (mm == 0) {
#pragma unroll
      for (int c = 0; c < C; ++c) ucol[half][c0 + c] = 0.f;
    }
  }
  __syncwarp();
  auto issue = [&](int j) {                                // rows and couplings of zone j
    if (act && j < len) {
      const size_t zb = (sys * n_r + zone(j)) * n;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = mm + i * L;
        if (FULL || r < n) {
          const float *src = diag + (zb + r) * n + c0;
          float *dst = &rows[half][r][c0];
          if (FULL) {
#pragma unroll
            for (int c = 0; c < C; c += 4)
              if (c0 + c < NP) cp_async16(dst + c, src + c);
          } else if (n % 2 == 0) {
            for (int c = 0; c < C && c0 + c < n; c += 2) cp_async8(dst + c, src + c);
          } else {
            for (int c = 0; c < C && c0 + c < n; ++c) cp_async4(dst + c, src + c);
          }
          if (cg == 0) {
            cp_async4(&cpl[half][0][r], (half == 0 ? lower : upper) + zb + r);
            cp_async4(&cpl[half][1][r], (half == 0 ? upper : lower) + zb + r);
          }
        }
      }
    }
    cp_async_commit();
  };
  float (*midt)[W] = rows[1];                              // the bottom-up warp's last inverse
  float a[R][C];
  bool ok = true;
  issue(0);
  for (int j = 0; j < len; ++j) {
    cp_async_wait_all();
    __syncwarp();
    // the zone's rows minus the Schur term of the previous zone
    float u[R];
    unsigned top[R];                                       // (FLAG)
#pragma unroll
    for (int i = 0; i < R; ++i) {
      top[i] = growth_limit(rows[half][mm + i * L][mm + i * L]);
      const float l = cpl[half][0][mm + i * L];
      u[i] = cpl[half][1][mm + i * L];
#pragma unroll
      for (int c = 0; c < C; c += 4) {
        float4 x = *reinterpret_cast<const float4 *>(&rows[half][mm + i * L][c0 + c]);
        if (j > 0) {
          const float4 v = *reinterpret_cast<const float4 *>(&ucol[half][c0 + c]);
          x.x = fmaf(-(l * a[i][c]), v.x, x.x);
          x.y = fmaf(-(l * a[i][c + 1]), v.y, x.y);
          x.z = fmaf(-(l * a[i][c + 2]), v.z, x.z);
          x.w = fmaf(-(l * a[i][c + 3]), v.w, x.w);
        }
        a[i][c] = x.x; a[i][c + 1] = x.y; a[i][c + 2] = x.z; a[i][c + 3] = x.w;
      }
    }
    __syncwarp();                                          // every lane has read the rows, couplings and ucol
    issue(j + 1);
    if (half == 0 && j == m) {
      // middle zone: wait for the bottom-up half and subtract its term diag(u_m) D''^{-1}_{m+1} diag(l_{m+1})
      asm volatile("bar.sync 1, 64;" ::: "memory");
      if (n_r - 1 > m) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const float lc = ucol[1][c0 + c];
#pragma unroll
          for (int i = 0; i < R; ++i) a[i][c] = fmaf(-(u[i] * midt[mm + i * L][c0 + c]), lc, a[i][c]);
        }
      }
    }
    // rows p and p + 1 to the pivot buffer
    auto publish = [&](int p) {
      if (act && (mm == p % L || mm == p % L + 1)) {
        float *dst = &prow[half][(p / 2) & 1][mm - p % L][c0];
        const float (&x)[C] = a[p / L];
#pragma unroll
        for (int c = 0; c < C; c += 4) *reinterpret_cast<float4 *>(dst + c) = make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]);
      }
    };
    publish(0);
#pragma unroll
    for (int b = 0; b < NP / 2; ++b) {
      const int p = 2 * b, pl = p % L, pg = p / C, pc = p % C;
      const float (*pb)[W] = prow[half][b & 1];
      // columns p and p + 1 of this lane's rows, from the group that holds them
      float xp[R], yp[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        xp[i] = __shfl_sync(0xffffffffu, a[i][pc], pg * L + mm);
        yp[i] = __shfl_sync(0xffffffffu, a[i][pc + 1], pg * L + mm);
      }
      __syncwarp();
      const float2 q0 = *reinterpret_cast<const float2 *>(&pb[0][p]);
      const float2 q1 = *reinterpret_cast<const float2 *>(&pb[1][p]);
      float4 v0[C / 4], v1[C / 4];
#pragma unroll
      for (int c = 0; c < C; c += 4) {
        v0[c / 4] = *reinterpret_cast<const float4 *>(&pb[0][c0 + c]);
        v1[c / 4] = *reinterpret_cast<const float4 *>(&pb[1][c0 + c]);
      }
      const float det = fmaf(q0.x, q1.y, -(q0.y * q1.x));
      const float idet = rcp_nr(det);
      if (FLAG) {
        ok = ok && idet > 0.f && (p + 2 < NP || idet < INFINITY);   // (an infinite one makes the next NaN)
        if (mm == pl || mm == pl + 1) ok = ok && in_range(mm == pl ? q0.x : q1.y, top[p / L]);
      }
      const float i00 = q1.y * idet, i01 = -q0.y * idet, i10 = -q1.x * idet, i11 = q0.x * idet;
      // one row: minus its two multipliers times the pivot rows; what its columns p and p + 1 become is minus the
      // multipliers (x, y) P^{-1}, in the owners' rows P^{-1}
      auto update = [&](int i) {
        float f0 = fmaf(xp[i], i00, yp[i] * i10), f1 = fmaf(xp[i], i01, yp[i] * i11);
        float z0 = -f0, z1 = -f1;
        if (i == p / L && mm == pl) { z0 = i00; z1 = i01; f0 = 1.f - i00; f1 = -i01; }
        if (i == p / L && mm == pl + 1) { z0 = i10; z1 = i11; f0 = -i10; f1 = 1.f - i11; }
        float (&x)[C] = a[i];
#pragma unroll
        for (int c = 0; c < C; c += 4) {
          const float4 v = v0[c / 4], t = v1[c / 4];
          float2 lo = __ffma2_rn(make_float2(-f0, -f0), make_float2(v.x, v.y), make_float2(x[c], x[c + 1]));
          float2 hi = __ffma2_rn(make_float2(-f0, -f0), make_float2(v.z, v.w), make_float2(x[c + 2], x[c + 3]));
          lo = __ffma2_rn(make_float2(-f1, -f1), make_float2(t.x, t.y), lo);
          hi = __ffma2_rn(make_float2(-f1, -f1), make_float2(t.z, t.w), hi);
          x[c] = lo.x; x[c + 1] = lo.y; x[c + 2] = hi.x; x[c + 3] = hi.y;
        }
        if (cg == pg) {
          x[pc] = z0;
          x[pc + 1] = z1;
        }
      };
      const int next = b + 1 < NP / 2 ? (p + 2) / L : 0;     // the slot of the next pivots
      update(next);
      if (b + 1 < NP / 2) publish(p + 2);
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (i != next) update(i);
    }
    if (act) {
      const size_t zb = (sys * n_r + zone(j)) * n;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const int r = mm + i * L;
        float *o = dinv + (zb + r) * n + c0;
        if (FULL) {
#pragma unroll
          for (int c = 0; c < C; c += 4)
            if (c0 + c < NP) *reinterpret_cast<float4 *>(o + c) = make_float4(a[i][c], a[i][c + 1], a[i][c + 2], a[i][c + 3]);
        } else if (r < n) {
#pragma unroll
          for (int c = 0; c < C; ++c)
            if (c0 + c < n) o[c] = a[i][c];
        }
        if (cg == 0) ucol[half][r] = u[i];
        if (half == 1 && j == len - 1) {
#pragma unroll
          for (int c = 0; c < C; ++c) midt[r][c0 + c] = a[i][c];
        }
      }
    }
    __syncwarp();
  }
  cp_async_wait_all();
  if (FLAG) ok = __all_sync(0xffffffffu, ok) != 0;
  if (half == 1) {
    if (FLAG && lane == 0) okb = ok;                       // (read after the barrier, the top half's last zone)
    asm volatile("bar.sync 1, 64;" ::: "memory");
  } else if (FLAG && lane == 0) {
    bad[jsys] = !(ok && okb);
  }
}

// Forward/back substitution with the twisted FP32 factors, two warps per system (the top-down
// and bottom-up halves), lane r owning block row r; the halves meet at the middle zone m through
// shared memory and a two-warp named barrier.
template <int NP>
__global__ void __launch_bounds__(kWarpsPerCta * 32)
k_solve_w32(int n, int n_r, int n_sys, const float *__restrict__ dinv, const double *__restrict__ lower,
            const double *__restrict__ upper, const double *__restrict__ rhs, double *__restrict__ x,
            const int *__restrict__ ray_list, const int *__restrict__ n_dev) {
  __shared__ float hbuf[kWarpsPerCta / 2][32], xbuf[kWarpsPerCta / 2][32];
  const unsigned full = 0xffffffffu;
  const int wid = threadIdx.x >> 5, r = threadIdx.x & 31;
  const int half = wid & 1, slot = wid >> 1;
  const long jsys = (long)blockIdx.x * (kWarpsPerCta / 2) + slot;
  if (jsys >= listed_sys(n_sys, n_dev, NS)) return;
  const long sys = listed_system(jsys, ray_list, NS);
  const bool real = r < n;
  const size_t base = (size_t)sys * n_r * n;
  const int m = n_r / 2, B = n_r - 1 - m;
  // Power-of-two scaling of the right-hand side (FP32 range), the same in both halves.
  double mx = 0.0;
  if (real)
    for (int i = 0; i < n_r; ++i) mx = fmax(mx, fabs(rhs[base + (size_t)i * n + r]));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(full, mx, off));
  double scale = 1.0;
  if (mx > 0.0 && isfinite(mx)) {
    int e;
    frexp(mx, &e);
    scale = ldexp(1.0, -e);
  }
  auto matvec = [&](int z, float v) {
    const float *src = dinv + (base + (size_t)z * n + (real ? r : 0)) * n;
    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
    for (int c = 0; c < NP; c += 2) {
      const float v0 = __shfl_sync(full, v, c), v1 = __shfl_sync(full, v, c + 1);
      if (c < n) acc0 = fmaf(src[c], v0, acc0);
      if (c + 1 < n) acc1 = fmaf(src[c + 1], v1, acc1);
    }
    return acc0 + acc1;
  };
  auto bar = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + slot) : "memory"); };
  bar();                       // both halves have read rhs for the scale before x (may alias rhs) is written
  // Forward: top g_i = Dinv_i (r_i - l_i g_{i-1}), i < m; bottom h_i = Dinv_i (r_i - u_i h_{i+1}), i > m.
  const int flen = half == 0 ? m : B;
  float prev = 0.f;
  for (int j = 0; j < flen; ++j) {
    const int z = half == 0 ? j : n_r - 1 - j;
    const size_t zr = base + (size_t)z * n + r;
    const float c = (real && j > 0) ? (float)(half == 0 ? lower[zr] : upper[zr]) : 0.f;
    const float v = real ? (float)(rhs[zr] * scale) - c * prev : 0.f;
    const float g = matvec(z, v);
    if (real) x[zr] = (double)g;
    prev = g;
  }
  if (half == 1) hbuf[slot][r] = B > 0 ? prev : 0.f;
  bar();
  if (half == 0) {
    // Middle zone: x_m = Dinv_m (r_m - l_m g_{m-1} - u_m h_{m+1}).
    const size_t zr = base + (size_t)m * n + r;
    const float l = (real && m > 0) ? (float)lower[zr] : 0.f;
    const float u = (real && m < n_r - 1) ? (float)upper[zr] : 0.f;
    const float v = real ? (float)(rhs[zr] * scale) - l * prev - u * hbuf[slot][r] : 0.f;
    const float xm = matvec(m, v);
    if (real) x[zr] = (double)xm / scale;
    xbuf[slot][r] = xm;
    prev = xm;
  }
  bar();
  if (half == 1) prev = xbuf[slot][r];
  // Backward: top x_i = g_i - Dinv_i (u_i x_{i+1}), i = m-1..0; bottom x_i = h_i - Dinv_i (l_i x_{i-1}), i = m+1..
  for (int j = 0; j < flen; ++j) {
    const int z = half == 0 ? m - 1 - j : m + 1 + j;
    const size_t zr = base + (size_t)z * n + r;
    const float c = real ? (float)(half == 0 ? upper[zr] : lower[zr]) : 0.f;
    const float gz = real ? (float)x[zr] : 0.f;
    const float xi = gz - matvec(z, real ? c * prev : 0.f);
    if (real) x[zr] = (double)xi / scale;
    prev = xi;
  }
}

template <int NP>
static cudaError_t run_solve(int n, int n_r, int n_sys, int spr, const void *dinv, const double *lower,
                             const double *upper, const double *rhs, double *x, const int *ray_list,
                             cudaStream_t s, const int *n_dev) {
  constexpr int SPS = Pack<NP>::SPC / 2;             // systems per CTA
  const unsigned grid = (unsigned)((n_sys + SPS - 1) / SPS);
  k_solve<NP><<<grid, Pack<NP>::THREADS, 0, s>>>(n, n_r, n_sys, spr, (const double *)dinv, lower, upper, rhs, x,
                                                 ray_list, n_dev);
  return cudaGetLastError();
}

// Which FP64 factor: k_factor64 splits a half-system's columns over the four warps of a CTA (the shorter chain);
// k_factor keeps more lanes at work.  k_factor64 / k_factor over 64 zones, us: 4 rows 187 / 93 at 400 systems;
// 8 rows 1200 systems 223 / 222, 2400 387 / 280; 12 rows 400 265 / 386, 1200 530 / 475, 2400 1085 / 739; 16 rows 400 393 /
// 588, 1600 1406 / 1085; 24 rows 400 1183 / 1407, 800 2324 / 1927, 2400 5975 / 4762; 32 rows 800 3916 / 5331, 4000 17452 /
// 19177.  At 20 rows both fill the SMs in whole CTAs (4 systems a CTA of k_factor, 3 halves of k_factor64, 2.6 times
// the time a CTA): 1200 1874 / 1565, 1600 2191 / 2196, 2400 3193 / 2911, 4000 4871 / 5025.
template <int NP>
static bool many_rows64(long n_sys) {
  auto up = [](long a, long b) { return (a + b - 1) / b; };
  if (NP == 4) return true;
  if (NP <= 16) return n_sys > 2 * kSMs * (32 / NP);         // beyond k_factor64's one row per lane
  if (NP == 20) return 13 * up(n_sys, 4 * kSMs) < 5 * up(2 * n_sys, 3 * kSMs);
  return NP < 32 && n_sys > 4 * kSMs;
}

cudaError_t launch_factor(int n, int n_r, int n_sys, const double *diag, const double *lower, const double *upper,
                          void *dinv, int precision, const int *ray_list, cudaStream_t s, const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  if (precision != MGFLD_MIXED)
    MGFLD_DISPATCH_NP(n, {
      if (!many_rows64<NP>(n_sys))
        return launch_factor64(n, n_r, n_sys, diag, lower, upper, (double *)dinv, ray_list, s, n_dev);
      constexpr int SPS = Pack<NP>::SPC / 2;
      k_factor<NP><<<(unsigned)((n_sys + SPS - 1) / SPS), Pack<NP>::THREADS, 0, s>>>(n, n_r, n_sys, diag, lower, upper,
                                                                                  (double *)dinv, ray_list, n_dev);
      return cudaGetLastError();
    })
  MGFLD_DISPATCH_NP(n, constexpr int W = fw_wpc<NP>();
                    const unsigned grid = (unsigned)((n_sys + W / 2 - 1) / (W / 2));
                    k_factor_w32<NP><<<grid, W * 32, 0, s>>>(n, n_r, n_sys, diag, lower, upper,
                                                                             (float *)dinv, ray_list, n_dev);
                    return cudaGetLastError())
}

template <int NP, typename TIn, typename T>
static cudaError_t run_factor_rows(int nb, int n_r, int n_sys, int spr, const TIn *diag, const T *lower,
                                   const T *upper, T *dinv, const int *ray_list, const int *bad,
                                   cudaStream_t s, const int *n_dev) {
  using C = RowCta<NP, T>;
  const unsigned grid = (unsigned)((n_sys + C::SPC / 2 - 1) / (C::SPC / 2));
  if (C::BYTES > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_factor_rows<NP, TIn, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)C::BYTES);
    if (e != cudaSuccess) return e;
  }
  k_factor_rows<NP, TIn, T><<<grid, C::THREADS, C::BYTES, s>>>(nb, n_r, n_sys, spr, diag, lower, upper, dinv, ray_list,
                                                               bad, n_dev);
  return cudaGetLastError();
}

template <int NP>
static cudaError_t run_factor_gj(int n, int n_r, int n_sys, int spr, const float *diag, const float *lower,
                                   const float *upper, float *dinv, const int *ray_list, int *bad, cudaStream_t s,
                                   const int *n_dev) {
  if ((n != NP || NP > 32) && !bad) return cudaErrorInvalidValue;   // the padded and the widest kernels store flags
  // A warp per half-system up to about four half-systems on each of the 4 kSMs warp schedulers (two of small
  // blocks, of which k_factor_row2 takes five to sixteen a warp), and for the pair systems' wide blocks at any
  // number.  Both sides, wide / row2, 256 zones: 1216 systems of 12 groups 186 / 173 us, 608 128 / 148 us; of 16
  // groups 1216 247 / 259 us; of 24 groups 1216 521 / 578 us; 512 zones of 20 groups: 1024 689 / 900 us, 1536 1092 /
  // 1035 us, 4096 2330 / 2048 us; 128 zones of 40-row blocks: 1536 1661 / 2060 us.
  if constexpr (NP <= 32) {
    if (n_sys > (NP < 16 ? 4 : 8) * kSMs) {
      constexpr int S = Row2<NP>::S;
      const unsigned grid = (unsigned)((n_sys + S - 1) / S);
      const auto kern = n == NP ? (bad ? k_factor_row2<NP, true, true> : k_factor_row2<NP, true, false>)
                                : k_factor_row2<NP, false, true>;
      kern<<<grid, 64, 0, s>>>(n, n_r, n_sys, spr, diag, lower, upper, dinv, ray_list, bad, n_dev);
      return cudaGetLastError();
    }
  }
  // (without flags: whole blocks of the single species)
  const auto kern = n != NP ? k_factor_wide<NP, false, true>
                            : (bad ? k_factor_wide<NP, true, true> : k_factor_wide<NP, true, (NP > 32)>);
  kern<<<n_sys, 64, 0, s>>>(n, n_r, n_sys, spr, diag, lower, upper, dinv, ray_list, bad, n_dev);
  return cudaGetLastError();
}

// FP32 (bad: n_sys flags of scratch): the blocks of the outer iteration are, up to the sign of the
// antineutrinos' rows and columns, M-matrices (the pair process couples the partners with
// non-negative entries, and its weighted column sums cancel against the diagonal as those of the
// scattering do) while the occupations are between 0 and 1, so they are eliminated without row exchanges, two
// rows per lane; a system whose pivot blocks are not an M-matrix's is done again with partial pivoting.
cudaError_t launch_factor_rows(int nb, int n_r, int n_sys, int spr, const void *diag, const void *lower,
                               const void *upper, void *dinv, int fp32, int *bad, const int *ray_list, cudaStream_t s,
                               const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  if (nb > 48) return cudaErrorInvalidValue;
  if (fp32) {
    const float *d = (const float *)diag, *l = (const float *)lower, *u = (const float *)upper;
    float *out = (float *)dinv;
    MGFLD_DISPATCH_NPW(nb, {
      const cudaError_t e = run_factor_gj<NP>(nb, n_r, n_sys, spr, d, l, u, out, ray_list, bad, s, n_dev);
      if (e != cudaSuccess) return e;
      return (run_factor_rows<NP, float, float>(nb, n_r, n_sys, spr, d, l, u, out, ray_list, bad, s, n_dev));
    })
  } else {
    MGFLD_DISPATCH_NPW(nb, return (run_factor_rows<NP, double, double>(nb, n_r, n_sys, spr, (const double *)diag,
                                                                          (const double *)lower, (const double *)upper,
                                                                          (double *)dinv, ray_list, nullptr, s, n_dev)))
  }
}

cudaError_t launch_factor_f32(int n, int n_r, int n_sys, const float *diag, const float *lower32,
                              const float *upper32, float *dinv, int *bad, const int *ray_list, cudaStream_t s,
                              const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  // padded blocks (28 rows among them, a multiple of 4 that is no padded size): with flags, and a system whose
  // pivot blocks are not an M-matrix's again with partial pivoting
  MGFLD_DISPATCH_NP(n, {
    const cudaError_t e = run_factor_gj<NP>(n, n_r, n_sys, NS, diag, lower32, upper32, dinv, ray_list,
                                            n == NP ? nullptr : bad, s, n_dev);
    if (e != cudaSuccess || n == NP) return e;
    constexpr int NW = (NP + 7) / 8 * 8;
    return (run_factor_rows<NW, float, float>(n, n_r, n_sys, NS, diag, lower32, upper32, dinv, ray_list, bad, s, n_dev));
  })
}

// FP64 substitution, up to how many systems the ring-fed one (a warp per half-system, n of its 32 lanes at work: the
// shorter chain, but more FP64 instructions for the same rows) is the faster one; beyond, the thread per row of k_solve
// keeps every lane at work.  Ring / k_solve over 256 zones: 20 groups 256 systems 261 / 843 us, 1216 852 / 949, 1280 911 / 1052, 2048 1413 /
// 1221 us; 12 groups 1280 637 / 639; 8 groups 1280 446 / 468, 2048 649 / 491; blocks of 16 and of up to 4 rows
// (bank conflicts; few lanes) 1280 998 / 757 and 282 / 177 us.
static inline int ring64_systems(int n) { return (n <= 4 || (n > 12 && n <= 16) ? 5 : 8) * kSMs; }

cudaError_t launch_solve(int n, int n_r, int n_sys, const void *dinv, const double *lower,
                         const double *upper, const double *rhs, double *x, int precision,
                         const int *ray_list, cudaStream_t s, const int *n_dev, int *err) {
  if (n_sys == 0) return cudaSuccess;
  if (precision == MGFLD_MIXED) {
    const unsigned grid = (unsigned)((n_sys + kWarpsPerCta / 2 - 1) / (kWarpsPerCta / 2));
    MGFLD_DISPATCH_NP(n, k_solve_w32<NP><<<grid, kWarpsPerCta * 32, 0, s>>>(n, n_r, n_sys, (const float *)dinv,
                                                                          lower, upper, rhs, x, ray_list, n_dev);
                         return cudaGetLastError())
  } else if (n_sys <= ring64_systems(n) && ((uintptr_t)dinv & 15u) == 0) {
    return launch_solve_ring64(n, n_r, n_sys, NS, (const double *)dinv, lower, upper, rhs, x, ray_list, err, s, n_dev);
  } else {
    // more systems, or a caller's factors off the 16-byte boundaries that bulk copies start on
    MGFLD_DISPATCH_NP(n, return (run_solve<NP>(n, n_r, n_sys, NS, dinv, lower, upper, rhs, x, ray_list, s, n_dev)))
  }
}

// The pair systems' FP64 substitution (nb = 2 n_e rows, two systems per ray; as above, and the rings of wide blocks
// leave room for few CTAs an SM: three of 32 rows, two of 40, one of 48): the ring up to the launches that its CTAs
// hold at once, the thread per row beyond.  Ring / thread per row over 64 zones, us: 4 rows 608 systems 52 / 55, 720
// 61 / 55; 8 rows 608 53 / 61, 800 75 / 65; 12 rows 608 88 / 99, 800 125 / 111; 16 rows 912 133 / 165, 1216 252 / 187;
// 18 rows 456 184 / 193, 608 231 / 204; 24 rows 456 192 / 229, 608 239 / 234; 26 rows 128 193 / 170, 304 197 / 226, 456
// 236 / 240; 32 rows 152 211 / 203, 304 239 / 242, 380 296 / 280; 40 rows 304 270 / 363, 340 509 / 408; 48 rows 152
// 321 / 410, 180 635 / 459, 4096 8453 / 4231.
static inline bool ring64_pair(int nb, int n_sys) {
  if (nb <= 16) return n_sys <= (nb == 16 ? 6 : 4) * kSMs;
  if (nb <= 24) return n_sys <= 3 * kSMs;
  if (nb <= 32) return n_sys > kSMs && n_sys <= 2 * kSMs;    // (few systems: the row kernel's shorter chain)
  return n_sys <= (nb <= 40 ? 2 : 1) * kSMs;
}

cudaError_t launch_solve_pair64(int nb, int n_r, int n_sys, const double *dinv, const double *lower, const double *upper,
                                const double *rhs, double *x, const int *ray_list, int *err, cudaStream_t s,
                                const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  if (nb > 48) return cudaErrorInvalidValue;
  if (ring64_pair(nb, n_sys))
    return launch_solve_ring64(nb, n_r, n_sys, 2, dinv, lower, upper, rhs, x, ray_list, err, s, n_dev);
  MGFLD_DISPATCH_NPW(nb, return (run_solve<NP>(nb, n_r, n_sys, 2, dinv, lower, upper, rhs, x, ray_list, s, n_dev)))
}

}  // namespace mgfld
