// Substitution with the twisted block-Thomas factors (blocktri.cu), streamed through shared memory.
#include <type_traits>

#include "async.cuh"
#include "mgfld_internal.cuh"
#include "warp.cuh"

namespace mgfld {

// Per-system power-of-two scaling of the FP32 solve: k such that max |rhs| 2^k lies in [1/2, 1) (from
// the largest exponent, so the maximum is taken over the upper words of the bit patterns: integer pipe
// only), then the scaled right-hand side rounded to FP32 once, so that the substitution reads FP32
// values.  One CTA per listed system (spr systems per ray); its cnt = n_r x n right-hand side is
// contiguous.  A thread keeps its first kKeep entries in registers between the two uses (whole systems
// up to 16384 entries), all their loads in flight at once; 256 threads where that holds the system, so that
// short ones leave room for more CTAs.  Measured at 32 / 1024 rays of 512 x 20: 25 -> 7 us / 175 ->
// 107 us; at 173 rays of 301 x 13: 17 -> 9 us (256 threads, one load after another, the second pass
// from L2 before).
constexpr int kKeep = 16;
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
k_sysmax(int cnt, const double *__restrict__ rhs, const int *__restrict__ ray_list, int spr, int *__restrict__ sys_exp,
         float *__restrict__ rhs32, const int *__restrict__ n_dev) {
  if ((int)blockIdx.x >= listed_sys(gridDim.x, n_dev, spr)) return;   // the whole block
  const size_t base = (size_t)listed_system(blockIdx.x, ray_list, spr) * cnt;
  __shared__ unsigned red[32];
  double v[kKeep];
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    const int e = threadIdx.x + j * THREADS;
    v[j] = e < cnt ? rhs[base + e] : 0.0;
  }
  unsigned m = 0u;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) m = max(m, abs_hi_word(v[j]));
  for (int e = threadIdx.x + kKeep * THREADS; e < cnt; e += THREADS) m = max(m, abs_hi_word(rhs[base + e]));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  const unsigned wm = (threadIdx.x & 31) < THREADS / 32 ? red[threadIdx.x & 31] : 0u;
  const int k = scale_of_max(__reduce_max_sync(0xffffffffu, wm));
  if (threadIdx.x == 0) sys_exp[blockIdx.x] = k;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    const int e = threadIdx.x + j * THREADS;
    if (e < cnt) rhs32[base + e] = d2f_exp2(v[j], k);
  }
  for (int e = threadIdx.x + kKeep * THREADS; e < cnt; e += THREADS) rhs32[base + e] = d2f_exp2(rhs[base + e], k);
}

cudaError_t launch_sysmax(int n, int n_r, int n_sys, const double *rhs, const int *ray_list, int spr, int *sys_exp,
                          float *rhs32, cudaStream_t s, const int *n_dev) {
  const int cnt = n * n_r;
  if (cnt <= 256 * kKeep)
    k_sysmax<256><<<n_sys, 256, 0, s>>>(cnt, rhs, ray_list, spr, sys_exp, rhs32, n_dev);
  else
    k_sysmax<1024><<<n_sys, 1024, 0, s>>>(cnt, rhs, ray_list, spr, sys_exp, rhs32, n_dev);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Ring-fed substitution, one CTA per system: warp 0 takes the top-down half (zones 0..m-1, then the
// middle zone m, then back up from m-1 to 0), warp 1 the bottom-up half (zones n_r-1..m+1, then
// back down from m+1); the halves meet at the middle through shared memory and CTA barriers.
// Lane r owns block row r (RPL rows r, r + NP/RPL, .. of blocks wider than a warp); the zone vector is
// broadcast through shared memory.
//
// The zones of a half go in groups of K consecutive ones, S groups in a ring: a group's inverse
// blocks are contiguous in memory and arrive by one bulk copy (completion counted on an mbarrier),
// its right-hand sides (inward sweep) or forward results (outward sweep) and couplings by cp.async
// pieces of all lanes.  A bulk copy starts on a 16-byte boundary and moves whole 16-byte pieces;
// where a group is not such a piece itself (odd n) the copy takes the aligned pieces that cover it
// and the rows are read from the remainder.  (Those pieces never leave the factor array: it starts
// on such a boundary and its 4 n_ray systems fill whole pieces.)  Every wait is bounded: on timeout
// the warp flags `err` (where there is one), waits (bounded) for its copies in flight, and carries
// on with a row of NaN, which the result shows.
//
// What bounds it: large launches the HBM bandwidth of the blocks, each read twice (the inward and
// the outward sweep); small ones the chain of a zone step, v = b - l prev, its broadcast, the dot
// product.  So a step holds little else: copies, their bookkeeping and their waits once per
// group, and the next step's row and vector entries fetched into registers right after the dot
// product that frees them.  Measured
// at 32 / 1024 rays of 512 x 20: 149 -> 89 us / 1146 -> 1080 us (one zone per slot and queue entry
// before); at 173 rays of 301 x 13 (odd n, on the chain's own global loads before): 650 -> 100 us; the
// pair systems of 256 rays of 512 x 20 (40-row blocks, a thread per row with CTA barriers before): 2060 ->
// 530 us.
template <int NP, int RPL, typename T>
struct Ring {
  // Zones per group: groups of up to 16 KB, two of them per half, so that the two rings of a CTA leave
  // room for four CTAs an SM at NP = 20.  Longer groups spread the bookkeeping of a group over more
  // steps, a third and fourth slot cost CTAs.  Substitutions of 32 and 1024 rays of 512 x 20
  // (us each, with the scaling): K = 2, S = 4 195 / 1379; K = 4, S = 2 156 / 1291; K = 4, S = 4 138 /
  // 1267; K = 8, S = 4 119 / 1436; K = 8, S = 2 122 / 1267.
  static constexpr int K = NP * NP * (int)sizeof(T) <= 1600 ? 8 : (NP * NP * (int)sizeof(T) <= 4096 ? 4 : 2);
  static constexpr int S = 2;
  static constexpr int LN = NP / RPL;                               // lanes with rows
  static constexpr int BLK = K * NP * NP * (int)sizeof(T) + 16;     // a slot: K blocks and the margins of odd n
  static constexpr int VEC = K * NP;                                // elements of one vector of a slot
  static constexpr int HALF = S * BLK + (2 * S * VEC + 2 * NP) * (int)sizeof(T);   // bytes of one warp
  static constexpr int BYTES = 2 * HALF + 2 * NP * (int)sizeof(T) + 2 * S * 8;
  static_assert(NP % 4 == 0 && LN <= 32 && (S & (S - 1)) == 0, "rows in 16-byte pieces, a power-of-two ring");
};

__device__ inline void load4(const float *p, float *a) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w;
}
__device__ inline void load4(const double *p, double *a) {
  const double2 u = *reinterpret_cast<const double2 *>(p), v = *reinterpret_cast<const double2 *>(p + 2);
  a[0] = u.x; a[1] = u.y; a[2] = v.x; a[3] = v.y;
}
// s[0..3] += a[0..3] v[0..3] (packed for FP32)
__device__ inline void fma4(const float *a, const float *v, float *s) {
  const float2 lo = __ffma2_rn(make_float2(a[0], a[1]), make_float2(v[0], v[1]), make_float2(s[0], s[1]));
  const float2 hi = __ffma2_rn(make_float2(a[2], a[3]), make_float2(v[2], v[3]), make_float2(s[2], s[3]));
  s[0] = lo.x; s[1] = lo.y; s[2] = hi.x; s[3] = hi.y;
}
// (FP64: two sums, of the even and of the odd columns, in ascending order)
__device__ inline void fma4(const double *a, const double *v, double *s) {
#pragma unroll
  for (int c = 0; c < 4; ++c) s[c & 1] = fma(a[c], v[c], s[c & 1]);
}
__device__ inline float sum4(const float *s) { return (s[0] + s[1]) + (s[2] + s[3]); }
__device__ inline double sum4(const double *s) { return s[0] + s[1]; }
// The result in the caller's units: FP32 sweeps ran on a right-hand side scaled by 2^-k.  An ordinary
// value is moved to FP64 and scaled by its bit pattern; the others (and every value where 2^k takes
// FP32's range out of FP64's, which its 11-bit exponent allows) go through f2d_exp2.
__device__ inline double unscaled(float v, int k) {
  const unsigned b = __float_as_uint(v), mag = b & 0x7fffffffu;
  if (mag - 0x00800000u >= 0x7f000000u || k < -800 || k > 800) return f2d_exp2(v, k);
  return __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + ((unsigned)(896 + k) << 20))), (int)(b << 29));
}
__device__ inline double unscaled(double v, int) { return v; }

// rhs, x and g may be one array (T = double): every zone's rhs is read before its g is written and
// its g before its x.  vec16: n sizeof(T) is a multiple of 16 and the vectors are 16-byte aligned.
template <int NP, int RPL, typename T, bool FULL>
__global__ void __launch_bounds__(64)
k_solve_ring(int n, int n_r, int n_sys, int spr, const T *__restrict__ dinv, const T *__restrict__ lower,
             const T *__restrict__ upper, const T *rhs, double *x, T *g, const int *__restrict__ ray_list,
             const int *__restrict__ sys_exp, int *err, int vec16, const int *__restrict__ n_dev) {
  using R = Ring<NP, RPL, T>;
  constexpr int K = R::K, S = R::S, LN = R::LN;
  extern __shared__ __align__(128) unsigned char sm[];
  const unsigned full = 0xffffffffu;
  const int half = threadIdx.x >> 5, r = threadIdx.x & 31;
  const long jsys = blockIdx.x;
  if (jsys >= listed_sys(n_sys, n_dev, spr)) return;        // whole CTA
  const long sys = listed_system(jsys, ray_list, spr);
  unsigned char *ring = sm + half * R::HALF;                // [S][BLK]
  T *vec = reinterpret_cast<T *>(ring + S * R::BLK);        // [S][2][K n]: (rhs or g, coupling) of a group
  T *vbuf = vec + 2 * S * R::VEC;                           // [2][NP]: the zone vector of even and odd steps
  T *hbuf = reinterpret_cast<T *>(sm + 2 * R::HALF), *xbuf = hbuf + NP;   // h_{m+1} and x_m
  unsigned long long *bar = reinterpret_cast<unsigned long long *>(xbuf + NP) + half * S;
  bool real[RPL];
  int row[RPL];                                             // this lane's rows (0 where it has none: unused)
#pragma unroll
  for (int p = 0; p < RPL; ++p) {
    real[p] = r < LN && r + p * LN < n;
    row[p] = real[p] ? r + p * LN : 0;
  }
  const int nn = n * n;
  const unsigned blk = (unsigned)(nn * (int)sizeof(T));
  const int unscale = sizeof(T) == 4 ? -sys_exp[jsys] : 0;  // rhs was scaled by 2^k before rounding
  const int m = n_r / 2, B = n_r - 1 - m;
  const int F = half == 0 ? m : B;                          // zones of this half
  const int NG = (F + K - 1) / K;                           // its groups, counted inward
  const int NU = 2 * NG + (half == 0 ? 1 : 0);              // ring uses: inward, (the middle zone,) outward
  const size_t sb = (size_t)sys * n_r * n;
  const T *dsys = dinv + sb * n;
  const T *rhs_s = rhs + sb, *cin = (half == 0 ? lower : upper) + sb, *cout = (half == 0 ? upper : lower) + sb;
  T *g_s = g + sb;
  double *x_s = x + sb;
  const unsigned base15 = (unsigned)(uintptr_t)dsys & 15u;
  // group v: cnt zones from zone lo
  auto count_of = [&](int v) { return min(K, F - v * K); };
  auto low_of = [&](int v, int cnt) { return half == 0 ? v * K : n_r - v * K - cnt; };
  // bytes between a zone's block and the 16-byte boundary a copy from it starts on
  auto margin = [&](int lo) { return FULL ? 0u : (base15 + (unsigned)lo * blk) & 15u; };
  if (r == 0) {
    for (int k = 0; k < S; ++k) mbar_init(&bar[k], 1);
    mbar_fence_init();
  }
  for (int c = r; c < 2 * NP; c += 32) vbuf[c] = T(0);      // rows beyond n stay zero
  __syncwarp();
  bool ok = true;                                           // warp-uniform: no wait has given up
  auto issue = [&](int u) {                                 // the block copy of ring use u
    if (r == 0 && u < NU && ok) {
      int lo = m, cnt = 1;
      if (half != 0 || u != NG) {
        const int v = u < NG ? u : 2 * NG - (half == 0 ? 0 : 1) - u;
        cnt = count_of(v);
        lo = low_of(v, cnt);
      }
      const unsigned mg = margin(lo);
      const unsigned bytes = FULL ? (unsigned)cnt * blk : (mg + (unsigned)cnt * blk + 15u) & ~15u;
      unsigned long long *b = &bar[u & (S - 1)];
      mbar_expect_tx(b, bytes);
      bulk_g2s(ring + (u & (S - 1)) * R::BLK, reinterpret_cast<const unsigned char *>(dsys + (size_t)lo * nn) - mg,
               bytes, b);
    }
  };
  auto fill = [&](int slot, int v, const T *a, const T *c) {   // the vectors of group v, one copy group
    if (v >= 0 && v < NG) {
      const int cnt = count_of(v), lo = low_of(v, cnt);
      const T *pa = a + lo * n, *pc = c + lo * n;
      T *d = vec + 2 * slot * R::VEC;
      if (vec16) {
        constexpr int P = 16 / (int)sizeof(T);
        for (int e = r * P; e < cnt * n; e += 32 * P) {
          cp_async16(d + e, pa + e);
          cp_async16(d + R::VEC + e, pc + e);
        }
      } else {
        for (int e = r; e < cnt * n; e += 32) {
          cp_async_elem(d + e, pa + e);
          cp_async_elem(d + R::VEC + e, pc + e);
        }
      }
    }
    cp_async_commit();
  };
  auto wait = [&](int u) {                                  // ring use u has arrived
    if (!ok) return;
    unsigned long long *b = &bar[u & (S - 1)];
    const unsigned parity = (unsigned)((u / S) & 1);
    ok = warp_wait([&]() { return mbar_try_wait(b, parity); }, [&]() { return mbar_wait_bounded(b, parity); },
                   [&](bool v) { return __all_sync(full, v) != 0; });
    if (!ok) {                                              // give up: flag and drain own copies
      if (r == 0) {
        if (err) atomicExch(err, 1);
        for (int v = u; v <= ring_last_issued(u, S, NU); ++v)   // (the one waited for among them)
          mbar_wait_bounded(&bar[v & (S - 1)], (unsigned)((v / S) & 1));
      }
      __syncwarp();
    }
  };
  T a[RPL][NP], bq[RPL], cq[RPL], prev[RPL];                // the next step's rows and vector entries
  // where they come from: byte offsets in shared memory of this lane's (first) row of the zone's
  // block and of its entry of the zone's vectors
  const int row_b = row[0] * n * (int)sizeof(T), ent_b = row[0] * (int)sizeof(T);
  const int next_row = LN * n * (int)sizeof(T), next_ent = LN * (int)sizeof(T);
  int rp = 0, vp = 0;
  auto load_rows = [&]() {
#pragma unroll
    for (int p = 0; p < RPL; ++p) {
      const T *src = reinterpret_cast<const T *>(sm + rp + (p > 0 && real[p] ? p * next_row : 0));
      if (FULL) {
#pragma unroll
        for (int c = 0; c < NP; c += 4) load4(src + c, &a[p][c]);
      } else {
#pragma unroll
        for (int c = 0; c < NP; ++c) a[p][c] = c < n ? src[c] : T(0);
      }
    }
  };
  auto load_vec = [&]() {
#pragma unroll
    for (int p = 0; p < RPL; ++p) {
      const T *src = reinterpret_cast<const T *>(sm + vp + (p > 0 && real[p] ? p * next_ent : 0));
      bq[p] = src[0];
      cq[p] = src[R::VEC];
    }
  };
  // the first step of ring use u: zone li of the group from zone lo, its vectors in slot `vs`
  auto open_use = [&](int u, int lo, int li, int vs) {
    __syncwarp();                                           // every lane's vector pieces have arrived
    wait(u);
    rp = half * R::HALF + (u & (S - 1)) * R::BLK + (int)margin(lo) + li * (int)blk + row_b;
    vp = half * R::HALF + S * R::BLK + (2 * vs * R::VEC + li * n) * (int)sizeof(T) + ent_b;
    load_rows();
    load_vec();
    if (!ok) {
#pragma unroll
      for (int p = 0; p < RPL; ++p) bq[p] = T(NAN);
    }
  };
  const int vb_b = half * R::HALF + S * R::BLK + 2 * S * R::VEC * (int)sizeof(T);   // the broadcast buffers
  auto dot = [&](int buf, T *out) {
    const T *vb = reinterpret_cast<const T *>(sm + vb_b) + buf * NP;
    T s[RPL][4];
#pragma unroll
    for (int p = 0; p < RPL; ++p) s[p][0] = s[p][1] = s[p][2] = s[p][3] = T(0);
#pragma unroll
    for (int c = 0; c < NP; c += 4) {
      T v[4];
      load4(vb + c, v);
#pragma unroll
      for (int p = 0; p < RPL; ++p) fma4(&a[p][c], v, s[p]);
    }
#pragma unroll
    for (int p = 0; p < RPL; ++p) out[p] = sum4(s[p]);
  };
  int tog = 0;                                              // broadcast buffer of the next step (odd K)
  auto broadcast = [&](int buf, const T *val) {
    T *vb = reinterpret_cast<T *>(sm + vb_b + ent_b) + buf * NP;
#pragma unroll
    for (int p = 0; p < RPL; ++p)
      if (real[p]) vb[p * LN] = val[p];
    __syncwarp();
  };
  // The cnt steps of ring use u (group v): inward prev = Dinv (b - c prev), stored in g; outward
  // prev = b - Dinv (c prev), stored in x.  `refill` is called once every lane holds the last rows
  // and entries of the use before it in registers (after the first broadcast barrier), when that
  // one's slot is free for the use S - 1 ahead.  WHOLE: cnt = K, no test per step.
  auto steps = [&](auto whole, auto outward, int cnt, int z0, int dir, auto refill) {
    constexpr bool WHOLE = decltype(whole)::value, OUT = decltype(outward)::value;
    const int rstep = dir * (int)blk, vstep = dir * n * (int)sizeof(T), ostep = dir * n;
    T *gp = g_s + z0 * n + row[0];
    double *xp = x_s + z0 * n + row[0];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      if (WHOLE || i < cnt) {
        T val[RPL], d[RPL];
#pragma unroll
        for (int p = 0; p < RPL; ++p) val[p] = OUT ? cq[p] * prev[p] : fma(-cq[p], prev[p], bq[p]);
        const int buf = K % 2 == 0 ? i & 1 : tog;
        if (K % 2) tog ^= 1;
        broadcast(buf, val);
        if (i == 0) refill();
        dot(buf, d);
#pragma unroll
        for (int p = 0; p < RPL; ++p) prev[p] = OUT ? bq[p] - d[p] : d[p];
        if (WHOLE ? i + 1 < K : i + 1 < cnt) {
          rp += rstep;
          vp += vstep;
          load_rows();
          load_vec();
        }
#pragma unroll
        for (int p = 0; p < RPL; ++p)
          if (real[p]) {
            if (OUT) xp[p * LN] = unscaled(prev[p], unscale);
            else gp[p * LN] = prev[p];
          }
        gp += ostep;
        xp += ostep;
      }
    }
  };

  // the middle zone's right-hand side and couplings (top-down half), fetched up front
  const int zm = m * n;
  T bm[RPL], lm[RPL], um[RPL];
#pragma unroll
  for (int p = 0; p < RPL; ++p) {
    bm[p] = rhs_s[zm + row[p]];
    lm[p] = m > 0 ? cin[zm + row[p]] : T(0);
    um[p] = m < n_r - 1 ? cout[zm + row[p]] : T(0);
    prev[p] = T(0);
  }
  for (int u = 0; u < S; ++u) issue(u);
  for (int d = 0; d < S; ++d) fill(d, d, rhs_s, cin);
  const std::true_type yes;
  const std::false_type no;
  // Inward: top g_i = Dinv_i (r_i - l_i g_{i-1}), bottom h_i = Dinv_i (r_i - u_i h_{i+1}).
  const int dz = half == 0 ? 1 : -1;
  if (NG > 0) {
    const int cnt = count_of(0);
    cp_async_wait_group<S - 1>();
    open_use(0, low_of(0, cnt), half == 0 ? 0 : cnt - 1, 0);
#pragma unroll
    for (int p = 0; p < RPL; ++p) cq[p] = T(0);
  }
  for (int v = 0; v < NG; ++v) {
    const int cnt = count_of(v), z0 = half == 0 ? v * K : n_r - 1 - v * K;
    auto refill = [&]() {
      if (v == 0) return;
      issue(v - 1 + S);
      fill((v - 1) & (S - 1), v - 1 + S, rhs_s, cin);
    };
    if (cnt == K) steps(yes, no, K, z0, dz, refill);
    else steps(no, no, cnt, z0, dz, refill);
    if (v + 1 < NG) {
      const int cnt1 = count_of(v + 1);
      cp_async_wait_group<S - 2>();
      open_use(v + 1, low_of(v + 1, cnt1), half == 0 ? 0 : cnt1 - 1, (v + 1) & (S - 1));
    }
  }
  cp_async_wait_all();
  __syncwarp();                                             // every lane's g is written
  for (int d = 0; d < S; ++d) fill(d, NG - 1 - d, g_s, cout);
  if (half == 1) {
#pragma unroll
    for (int p = 0; p < RPL; ++p)
      if (real[p]) hbuf[row[p]] = prev[p];                  // zero when the half is empty
  }
  __syncthreads();
  int u = NG;
  if (half == 0) {
    // Middle zone: x_m = Dinv_m (r_m - l_m g_{m-1} - u_m h_{m+1}).
    wait(u);
    rp = (u & (S - 1)) * R::BLK + (int)margin(m) + row_b;
    load_rows();
    T val[RPL], d[RPL];
#pragma unroll
    for (int p = 0; p < RPL; ++p) {
      val[p] = bm[p] - lm[p] * prev[p] - um[p] * hbuf[row[p]];
      if (!ok) val[p] = T(NAN);
    }
    __syncwarp();
    broadcast(0, val);
    if (u > 0) issue(u - 1 + S);
    dot(0, d);
    __syncwarp();
#pragma unroll
    for (int p = 0; p < RPL; ++p) prev[p] = d[p];
#pragma unroll
    for (int p = 0; p < RPL; ++p)
      if (real[p]) {
        x_s[zm + row[p]] = unscaled(prev[p], unscale);
        xbuf[row[p]] = prev[p];
      }
    ++u;
  }
  __syncthreads();
  if (half == 1) {
#pragma unroll
    for (int p = 0; p < RPL; ++p) prev[p] = xbuf[row[p]];
  }
  // Outward: top x_i = g_i - Dinv_i (u_i x_{i+1}); bottom x_i = h_i - Dinv_i (l_i x_{i-1}).
  if (NG > 0) {
    const int cnt = count_of(NG - 1);
    cp_async_wait_group<S - 1>();
    open_use(u, low_of(NG - 1, cnt), half == 0 ? cnt - 1 : 0, 0);
  }
  for (int w = 0; w < NG; ++w, ++u) {
    const int v = NG - 1 - w, cnt = count_of(v), lo = low_of(v, cnt), z0 = half == 0 ? lo + cnt - 1 : lo;
    auto refill = [&]() {
      if (u > 0) issue(u - 1 + S);
      if (w > 0) fill((w - 1) & (S - 1), NG - 1 - (w - 1 + S), g_s, cout);
    };
    if (cnt == K) steps(yes, yes, K, z0, -dz, refill);
    else steps(no, yes, cnt, z0, -dz, refill);
    if (w + 1 < NG) {
      const int cnt1 = count_of(v - 1);
      cp_async_wait_group<S - 2>();
      open_use(u + 1, low_of(v - 1, cnt1), half == 0 ? cnt1 - 1 : 0, (w + 1) & (S - 1));
    }
  }
  cp_async_wait_all();
}

template <int NP, int RPL, typename T>
static cudaError_t run_ring(int n, int n_r, int n_sys, int spr, const T *dinv, const T *lower, const T *upper,
                            const T *rhs, double *x, T *g, const int *ray_list, const int *sys_exp, int *err,
                            cudaStream_t s, const int *n_dev) {
  using R = Ring<NP, RPL, T>;
  const auto kern = n == NP ? k_solve_ring<NP, RPL, T, true> : k_solve_ring<NP, RPL, T, false>;
  if (R::BYTES > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, R::BYTES);
    if (e != cudaSuccess) return e;
  }
  const uintptr_t all = (uintptr_t)lower | (uintptr_t)upper | (uintptr_t)rhs | (uintptr_t)g;
  const int vec16 = (n * sizeof(T)) % 16 == 0 && (all & 15u) == 0;
  kern<<<n_sys, 64, R::BYTES, s>>>(n, n_r, n_sys, spr, dinv, lower, upper, rhs, x, g, ray_list, sys_exp, err, vec16,
                                   n_dev);
  return cudaGetLastError();
}

cudaError_t launch_solve_ring(int n, int n_r, int n_sys, int spr, const void *dinv, const float *lower32,
                              const float *upper32, const double *rhs, float *rhs32, double *x, float *g32,
                              const int *ray_list, int *sys_exp, int *err, cudaStream_t s, const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  const cudaError_t e = launch_sysmax(n, n_r, n_sys, rhs, ray_list, spr, sys_exp, rhs32, s, n_dev);
  if (e != cudaSuccess) return e;
  const float *f = (const float *)dinv;
  if (spr != NS) {
    if (n > 48) return cudaErrorInvalidValue;
    MGFLD_DISPATCH_NPW(n, return (run_ring<NP, (NP > 32 ? 2 : 1), float>(n, n_r, n_sys, spr, f, lower32, upper32, rhs32,
                                                                         x, g32, ray_list, sys_exp, err, s, n_dev)))
  }
  MGFLD_DISPATCH_NP(n, return (run_ring<NP, 1, float>(n, n_r, n_sys, spr, f, lower32, upper32, rhs32, x, g32, ray_list,
                                                      sys_exp, err, s, n_dev)))
}

// FP64 factors (dinv on a 16-byte boundary; rhs and x may be one array; err or null).  Bound by the latency of a zone
// step in small launches and by the FP64 units, with 20 of 32 lanes at work, in large ones: the 22 instructions of a row
// and step take the units 0.29 of the 0.50 ms at 64 rays of 512 x 20 and 1.17 of the 1.63 ms at 256.  Per substitution at
// 64 / 256 rays 1770 -> 495 us / 1834 -> 1634 us, one ray of 64 x 12 115 -> 45 us (a thread per row and CTA barriers
// before, which is the faster one beyond about 1200 systems: launch_solve, launch_solve_pair64).
cudaError_t launch_solve_ring64(int n, int n_r, int n_sys, int spr, const double *dinv, const double *lower,
                                const double *upper, const double *rhs, double *x, const int *ray_list, int *err,
                                cudaStream_t s, const int *n_dev) {
  if (n_sys == 0) return cudaSuccess;
  if (spr != NS) {
    if (n > 48) return cudaErrorInvalidValue;
    MGFLD_DISPATCH_NPW(n, return (run_ring<NP, (NP > 16 ? 2 : 1), double>(n, n_r, n_sys, spr, dinv, lower, upper, rhs, x, x,
                                                                          ray_list, nullptr, err, s, n_dev)))
  }
  MGFLD_DISPATCH_NP(n, return (run_ring<NP, 1, double>(n, n_r, n_sys, spr, dinv, lower, upper, rhs, x, x, ray_list,
                                                       nullptr, err, s, n_dev)))
}

}  // namespace mgfld
