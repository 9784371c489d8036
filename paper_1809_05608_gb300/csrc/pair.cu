// The synthetic pair process (Eq. d14, zeroth moment, Legendre order 0) in the implicit step.
//
// Each neutrino species q is made and destroyed together with its partner qbar (nu_e with
// nubar_e, nu_mu,tau with nubar_mu,tau), group by group:
//   S_pair,k = C [(1 - psi_k) sum_k' w_k' Phi^p(eps_k, eps_k') (1 - psibar_k')
//                 - psi_k sum_k' w_k' chi_q(k, k') Phi^a(eps_k, eps_k') psibar_k'],
// the annihilation kernel Phi^a = pair_coef per zone, the creation kernel Phi^p =
// e^{-(eps + eps')/T} Phi^a (Eq. d12 with the pair energy eps + eps' given to the e-e+ pair), and
// chi the angular correction of the annihilation kernel (Eqs. d16-d22; 1 unless enabled).  The
// process couples the two species of a pair in every zone, so the Newton system is solved per
// (ray, pair) with coupled 2 n x 2 n zone blocks: rows and columns (s n + k), s = 0 for the
// neutrino and 1 for the antineutrino of the pair; the couplings to the neighbouring zones stay
// diagonal.  Vectors of that system are laid out [ray][pair][zone][2 n].
#include "mgfld_internal.cuh"

namespace mgfld {

// The pair kernels of every zone, threads (zone, species q, group k): species q's weighted annihilation kernel
//   pkill[q][k][k'] = C w_k' chi_q(k, k') Phi^a,
// and the weighted creation kernel, shared by the species,
//   pmake[k][k'] = C w_k' Phi^p(eps_k, eps_k') = C w_k' Phi^a e^{-eps_k/T} e^{-eps_k'/T},
// with its row sums.  chi = min(chi_1, chi_2) (Eq. d21): chi_1 = 1 - eta eta' / 6 (Eq. d16, the
// flux factors eta of species q at eps_k and of its partner at eps_k', the input eta1 clamped to
// [0, 1]), chi_2 = (8 + (mu mu' - 3)(1 + mu)(1 + mu')) / 8 (Eq. d19) with the cone edges
// mu = max(sign(x) sqrt|x|, -1), x = 1 - (R_nu / R_i)^2 (Eqs. d17, d22), R_nu each species' and
// group's neutrinosphere at psi^n and R_i the zone centre.  chi_q(k, k') = chi_qbar(k', k), so it is
// formed once per pair of species into shared memory (chi_2 = 1 + (m mu' - 3 m8) (1 + mu') with m = mu m8,
// m8 = (1 + mu) / 8), and the kernels leave from there with consecutive threads on consecutive
// columns.  Bound by the FP64 units; measured at 256 rays of 512 x 20: 4412 -> 2630 us (a thread per
// row, which formed chi of both species and stored its row 160 bytes from the next thread's, before).
static inline int pair_zones_per_block(int n) {
  // whole warps where some number of zones gives them
  for (int z = 256 / (NS * n); z > 0; --z)
    if (z * NS * n % 32 == 0) return z;
  return 256 / (NS * n) > 0 ? 256 / (NS * n) : 1;
}
// per zone: e^{-eps/T} and weights, the flux factors, mu and 1 + mu of every species, chi of both pairs,
// e^{-eps/T} e^{-eps'/T}
__host__ __device__ inline size_t pair_zone_doubles(int n) { return (size_t)(2 + 3 * NS) * n + 3 * (size_t)n * (n + 1); }

__global__ void k_pair(Prob p, Ws w, const double *__restrict__ T, int zpb) {
  extern __shared__ double sm[];
  const int n = p.n, per = NS * n, ld = n + 1;
  const int zl = threadIdx.x / per, rem = threadIdx.x % per, q = rem / n, k = rem % n;
  const unsigned nz = (unsigned)(p.n_ray * p.n_r);
  const unsigned zi = blockIdx.x * (unsigned)zpb + zl;
  const bool live = zl < zpb && zi < nz;
  double *ez = sm + (size_t)(live ? zl : 0) * pair_zone_doubles(n);
  double *wl = ez + n, *eta = wl + n, *mu = eta + NS * n, *mu1 = mu + NS * n, *chi = mu1 + NS * n;
  double *mk = chi + 2 * (size_t)n * ld;
  if (live) {
    const int ray = (int)(zi / (unsigned)p.n_r), i = (int)(zi - (unsigned)ray * p.n_r);
    const double inv_a = 1.0 / lapse_at(p, ray, i);
    if (q == 0) {
      ez[k] = exp(-(w.E[k] * inv_a) / T[zi]);
      wl[k] = kCNes * p.pair[zi] * (w.W[k] * inv_a * inv_a * inv_a);
    }
    const size_t g = (((size_t)ray * NS + q) * p.n_r + i) * n + k;
    eta[rem] = p.eta1 ? fmin(fmax(p.eta1[g], 0.0), 1.0) : 0.0;
    const double *re = p.r_edge + (size_t)ray * (p.n_r + 1);
    const double rc = 0.5 * (re[i] + re[i + 1]);
    const double rr = w.rnu[((size_t)ray * NS + q) * n + k] / rc;
    const double x = 1.0 - rr * rr;
    const double m = fmax(x > 0.0 ? sqrt(x) : (x < 0.0 ? -sqrt(-x) : 0.0), -1.0);
    mu[rem] = m;
    mu1[rem] = 1.0 + m;
  }
  __syncthreads();
  if (live) {
    // chi of the even species of the pair, row k, every other column; every fourth column of e e'
    const int pp = q >> 1, qe = 2 * pp, qb = qe + 1;
    double *row = chi + ((size_t)pp * n + k) * ld;
    if (p.pair_chi) {
      const double e6 = eta[qe * n + k] / 6.0, m8 = 0.125 * mu1[qe * n + k], m = mu[qe * n + k] * m8, m3 = -3.0 * m8;
      for (int kp = q & 1; kp < n; kp += 2) {
        const double c1 = fma(-e6, eta[qb * n + kp], 1.0);
        const double c2 = fma(fma(m, mu[qb * n + kp], m3), mu1[qb * n + kp], 1.0);
        row[kp] = ord_key(c1) < ord_key(c2) ? c1 : c2;        // the minimum, on the integer pipe
      }
    } else {
      for (int kp = q & 1; kp < n; kp += 2) row[kp] = 1.0;
    }
    const double ek = ez[k];
    for (int kp = q; kp < n; kp += NS) mk[(size_t)k * ld + kp] = ek * ez[kp];
  }
  __syncthreads();
  if (!live) return;
  // column k of every row (consecutive threads: consecutive columns)
  const double wk = wl[k];
  const double *x = chi + (size_t)(q >> 1) * n * ld + ((q & 1) ? k * ld : k);
  const int xs = (q & 1) ? 1 : ld;
  double *kill = w.pkill + ((size_t)zi * NS + q) * n * n + k, *make = w.pmake + (size_t)zi * n * n + k;
  for (int r = 0; r < n; ++r) kill[(size_t)r * n] = wk * x[r * xs];
  for (int r = q; r < n; r += NS) make[(size_t)r * n] = wk * mk[(size_t)r * ld + k];
  if (q == 0) {
    double ms = 0.0;
    for (int kp = 0; kp < n; ++kp) ms += wl[kp] * mk[(size_t)k * ld + kp];
    w.pmsum[(size_t)zi * n + k] = ms;
  }
}

cudaError_t launch_pair(const Prob &p, const Ws &w, const double *T, cudaStream_t s) {
  const int zpb = pair_zones_per_block(p.n);
  const size_t nz = (size_t)p.n_ray * p.n_r;
  const size_t sm = sizeof(double) * zpb * pair_zone_doubles(p.n);
  if (sm > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  k_pair<<<(unsigned)((nz + zpb - 1) / zpb), zpb * NS * p.n, sm, s>>>(p, w, T, zpb);
  return cudaGetLastError();
}

// Residual and Jacobian rows of the coupled pair systems (Eqs. a58, a59 with the sources of
// Eqs. a55, d8 and d14), one thread per (ray, species q, zone i, group k) equation, as k_assemble
// with the frozen flux coefficients, plus the pair sums
//   make = sum_k' pmake[k][k'] (1 - psibar_k') = pmsum_k - sum pmake psibar,  kill = sum pkill psibar,
// S += (1 - psi_k) make - psi_k kill.  Row (s n + k) of the zone's 2 n x 2 n block: the species'
// own NES block with the diagonal, and the partner's columns
//   dG_k / d psibar_k' = (1 - psi_k) pmake[k][k'] + psi_k pkill[k][k'].
// src_out (FP64): the converged sources (psi layout) for Eq. a62b and the ledgers.  Bound by the
// FP64 multiply-adds of the sums, 4 n a row: 1.95 ms a pass at 256 rays of 512 x 20.
template <typename TD>
__global__ void k_assemble_pair(Prob p, Ws w, const double *__restrict__ psi, TD *__restrict__ diag,
                                double *__restrict__ lower, double *__restrict__ upper, double *__restrict__ rhs,
                                const int *__restrict__ list, int n_list, const int *__restrict__ jac_flag,
                                double *__restrict__ src_out, int first, const int *__restrict__ n_dev) {
  const int n = p.n, n2 = 2 * n;
  const unsigned per_ray = (unsigned)(NS * p.n_r * n);
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (unsigned)listed(n_list, n_dev) * per_ray) return;
  const unsigned rl = t / per_ray;
  const int ray = list ? list[rl] : (int)rl;
  const unsigned local = t - rl * per_ray;
  const unsigned kq = local / (unsigned)n;
  const int k = (int)(local - kq * n);
  const int q = (int)(kq % NS);
  const int i = (int)(kq / NS);
  const int pq = q >> 1, sq = q & 1, qb = q ^ 1;
  const size_t g = (((size_t)ray * NS + q) * p.n_r + i) * n + k;
  const size_t gc = (((size_t)ray * 2 + pq) * p.n_r + i) * n2 + (size_t)sq * n + k;
  const size_t zi = (size_t)ray * p.n_r + i;
  const int last = p.n_r - 1;
  const double *z = w.zone + zi * ZC_N;
  const double pre = z[ZC_PRE];
  const double inv_acdt = z[ZC_INV_ACDT];

  const double *ps = psi + (g - k);
  const double *pb = psi + (((size_t)ray * NS + qb) * p.n_r + i) * n;
  const double pk = ps[k];
  const double *fin = w.phin + (zi * n + k) * n;
  const double *fout = w.phout + (zi * n + k) * n;
  double gain = 0.0, lp = 0.0;
  if (first) {
    gain = w.g0[g];
    lp = w.l0[g];
  } else {
    for (int kp = 0; kp < n; ++kp) {
      const double pv = ps[kp];
      gain += fin[kp] * pv;
      lp += fout[kp] * pv;
    }
  }
  constexpr bool MIXED = sizeof(TD) == 4;
  const double *mk = w.pmake + (zi * n + k) * n;
  const double *kl = w.pkill + ((zi * NS + q) * n + k) * n;
  double mb = 0.0, kb = 0.0;
  for (int kp = 0; kp < n; ++kp) {
    const double v = pb[kp];
    mb = fma(mk[kp], v, mb);
    kb = fma(kl[kp], v, kb);
  }
  const double make = w.pmsum[zi * n + k] - mb, kill = kb;
  const double j = w.jbuf[g];
  if (MIXED) {
    // the sums kept for the final sources (k_src_pair; the pair sums in the storage of 1/lambda and lambda,
    // which the neutrinosphere scan has consumed)
    if (!first) {
      w.g0[g] = gain;
      w.l0[g] = lp;
    }
    w.kinv[g] = mb;
    w.lam[g] = kb;
  }
  const double loss = w.rsum[zi * n + k] - lp;
  const double kap = scaled(p, p.kabs, g, q, k);
  const double S = j * (1.0 - pk) - kap * pk + ((1.0 - pk) * gain - pk * loss) + ((1.0 - pk) * make - pk * kill);
  if (!MIXED && src_out) {
    src_out[g] = S;
    return;
  }
  const double al_out = w.alpha[g];
  const double al_in = i > 0 ? w.alpha[g - n] : 0.0;
  const double gh = (i == last) ? w.ghost[((size_t)ray * NS + q) * n + k] : 0.0;
  const double p_right = i < last ? ps[k + n] : gh * pk;
  const double p_left = i > 0 ? ps[k - (ptrdiff_t)n] : pk;
  const double flux_out = -al_out * (p_right - pk);
  const double flux_in = -al_in * (pk - p_left);
  const double sh = p.u ? w.shock[g] : 0.0;
  const double G = (pk - w.psi_n[g]) * inv_acdt + pre * (flux_out - flux_in + sh) - S;
  rhs[gc] = -G;
  if (jac_flag && !jac_flag[ray]) return;
  const double jdiag = al_out * (1.0 - gh) + al_in;
  const double dg = inv_acdt + pre * jdiag + j + kap + (gain + loss) + (make + kill);
  const double c_low = pre * al_in, c_up = i < last ? pre * al_out : 0.0;
  TD *row = diag + gc * n2;
  const int own = sq * n, part = (1 - sq) * n;
  if (sizeof(TD) == 4 && w.phin32) {
    // FP32 rows (the preconditioner of the FP64 refinement): operands converted on the integer
    // pipe (truncated), the partner's columns from FP32 copies of the pair kernels
    const float *fi = w.phin32 + (zi * n + k) * n, *fd = w.phd32 + (zi * n + k) * n;
    const float pf = d2f_exp2(pk, 0);
    const float dgf = (float)dg;
    for (int kp = 0; kp < n; ++kp) {
      const float e = fmaf(pf, fd[kp], -fi[kp]);
      row[own + kp] = TD(kp == k ? e + dgf : e);
    }
    for (int kp = 0; kp < n; ++kp) {
      const float m = d2f_exp2(mk[kp], 0);
      row[part + kp] = TD(fmaf(pf, d2f_exp2(kl[kp], 0) - m, m));
    }
  } else {
    const double *fd = w.phd + (zi * n + k) * n;
    for (int kp = 0; kp < n; ++kp) {
      const double e = fma(pk, fd[kp], -fin[kp]);
      row[own + kp] = TD(kp == k ? e + dg : e);
    }
    for (int kp = 0; kp < n; ++kp) row[part + kp] = TD(fma(pk, kl[kp] - mk[kp], mk[kp]));
  }
  lower[gc] = -c_low;
  upper[gc] = -c_up;
  if (w.lower32) {
    w.lower32[gc] = d2f_exp2(-c_low, 0);
    w.upper32[gc] = d2f_exp2(-c_up, 0);
  }
}

// The converged sources of the mixed path, as k_src_mixed forms them: the sums of the ray's last residual
// plus the kernels times the last, sub-tolerance correction in FP32 (the kernels' leading 24 bits), a
// thread per (zone, species, group), the block's corrections staged as FP32.  The FP32 sums lose 2^-23 of that
// correction, which stays below the rounding of the FP64 sums only where the correction is small: for a ray that did
// not converge, or with `full` (a tolerance above 2^-30), the FP64 sums are formed again at psi, as k_assemble_pair
// forms them.
constexpr int kSrcPairThreads = 256;
__global__ void __launch_bounds__(kSrcPairThreads)
k_src_pair(Prob p, Ws w, const double *__restrict__ psi, double *__restrict__ src, bool full) {
  extern __shared__ float xs[];                              // the block's zones, [zone][species][group]
  const int n = p.n, n2 = 2 * n;
  const unsigned zrows = (unsigned)(NS * n), zpb = blockDim.x / zrows;
  const unsigned total = (unsigned)(p.n_ray * p.n_r);
  const unsigned zs = threadIdx.x / zrows, zi = blockIdx.x * zpb + zs, e = threadIdx.x - zs * zrows;
  const int q = (int)(e / (unsigned)n), k = (int)(e - (unsigned)q * n);
  const bool in = zi < total;
  const unsigned ray = in ? zi / (unsigned)p.n_r : 0, i = in ? zi - ray * (unsigned)p.n_r : 0;
  if (in)
    xs[threadIdx.x] = (float)w.x[(((size_t)ray * 2 + (q >> 1)) * p.n_r + i) * n2 + (size_t)(q & 1) * n + k];
  __syncthreads();
  if (!in) return;
  const size_t g = (((size_t)ray * NS + q) * p.n_r + i) * n + k, zr = ((size_t)zi * n + k) * n;
  const float *fi = w.phin32 + zr, *fd = w.phd32 + zr;
  const double *mk = w.pmake + zr, *kl = w.pkill + (((size_t)zi * NS + q) * n + k) * n;
  const double pk = psi[g], q1 = 1.0 - pk;
  const double kap = scaled(p, p.kabs, g, q, k);
  if (full || w.status[ray] != MGFLD_OK) {                   // (uniform over a zone)
    const double *ps = psi + (g - k), *pb = psi + (((size_t)ray * NS + (q ^ 1)) * p.n_r + i) * n;
    const double *fin = w.phin + zr, *fout = w.phout + zr;
    double gain = 0.0, lp = 0.0, mb = 0.0, kb = 0.0;
    for (int kp = 0; kp < n; ++kp) {
      const double pv = ps[kp], v = pb[kp];
      gain += fin[kp] * pv;
      lp += fout[kp] * pv;
      mb = fma(mk[kp], v, mb);
      kb = fma(kl[kp], v, kb);
    }
    const double make = w.pmsum[(size_t)zi * n + k] - mb, loss = w.rsum[(size_t)zi * n + k] - lp, j = w.jbuf[g];
    src[g] = j * q1 - kap * pk + (q1 * gain - pk * loss) + (q1 * make - pk * kb);
    return;
  }
  const float *dx = xs + zs * zrows + (size_t)q * n, *dy = xs + zs * zrows + (size_t)(q ^ 1) * n;
  float dg = 0.f, dl = 0.f, dm = 0.f, dk = 0.f;
  for (int kp = 0; kp < n; ++kp) {
    const float d = dx[kp], a = fi[kp], y = dy[kp];
    dg = fmaf(a, d, dg);
    dl = fmaf(a - fd[kp], d, dl);
    dm = fmaf(d2f_exp2(mk[kp], 0), y, dm);
    dk = fmaf(d2f_exp2(kl[kp], 0), y, dk);
  }
  const float pf = d2f_exp2(pk, 0);
  // (1 - psi) (dgain - dmake) + psi (dlp - dkill): the FP32 part of the sources
  const float corr = fmaf(1.f - pf, dg - dm, pf * (dl - dk));
  const double up = w.g0[g] + (w.pmsum[(size_t)zi * n + k] - w.kinv[g]);
  const double down = (w.rsum[(size_t)zi * n + k] - w.l0[g]) + w.lam[g];
  double S = fma(q1, up, fma(-pk, down, (double)corr));
  S = fma(w.jbuf[g], q1, fma(-kap, pk, S));
  src[g] = S;
}

cudaError_t launch_src_pair(const Prob &p, const Ws &w, const double *psi, double *src, double tol, cudaStream_t s) {
  const unsigned zrows = (unsigned)(NS * p.n), zpb = kSrcPairThreads / zrows, zones = (unsigned)(p.n_ray * p.n_r);
  k_src_pair<<<(zones + zpb - 1) / zpb, zpb * zrows, sizeof(float) * zpb * zrows, s>>>(p, w, psi, src,
                                                                                       tol > 0x1p-30);
  return cudaGetLastError();
}

cudaError_t launch_assemble_pair(const Prob &p, const Ws &w, const double *psi, void *diag, int diag_fp32,
                                 double *lower, double *upper, double *rhs, const int *list, int n_list,
                                 const int *jac_flag, cudaStream_t s, double *src_out, int first, const int *n_dev) {
  const size_t total = (size_t)n_list * NS * p.n_r * p.n;
  if (total == 0) return cudaSuccess;
  const unsigned B = 256;
  const unsigned grid = (unsigned)((total + B - 1) / B);
  if (diag_fp32)
    k_assemble_pair<float><<<grid, B, 0, s>>>(p, w, psi, (float *)diag, lower, upper, rhs, list, n_list, jac_flag,
                                              src_out, first, n_dev);
  else
    k_assemble_pair<double><<<grid, B, 0, s>>>(p, w, psi, (double *)diag, lower, upper, rhs, list, n_list, jac_flag,
                                               src_out, first, n_dev);
  return cudaGetLastError();
}

}  // namespace mgfld
