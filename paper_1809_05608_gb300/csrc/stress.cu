// Neutrino stress and lapse update (Sec. "Solution of the Transport Equations", Eqs. a62e-a62l).
//
// mgfld_stress_lapse evaluates the transport step's coefficients at the state it is given (the
// same setup kernels; the flux limiter of every edge is kept), then
//   k_stress: per edge i+1/2: f = -(4 pi/(hc)^3)/3 sum_q N_q sum_k F (X_{i+1} - X_i)
//             A_{i+1/2} / Delta M_{i+1/2}, X = eps^3 d eps psi0 on each zone's comoving grid
//             (Eqs. a62e-a62f), and the zone value, the mean of its two edges (Eq. a62i);
//   k_lapse:  a block per ray: the enclosed rest mass, the exterior lapse at the
//             outer edge (Eq. a62k), and the inward product of Eq. a62l written as one exponential
//             of a suffix sum, a_i = a_I exp(sum_{j >= i} x_j), x_j the bracket over rho c^2.
// Readings: the stress term of Eq. a62l is Delta M f / (4 pi R^2) (a force per area, as the
// pressure difference beside it); Eq. a62k carries the square root of the Schwarzschild lapse;
// the scan starts with a_I = a_{I+1/2}; the outer edge uses the transport's ghost zone and the
// centre edge carries no stress; the enclosed mass adds the caller's mass inside the innermost
// edge to sum rho V.
#include "mgfld_internal.cuh"

namespace mgfld {

constexpr double kG = 6.67430e-8;            // cm^3 g^-1 s^-2
constexpr double kMeVErg = 1.602176634e-6;

cudaError_t launch_setup(const Prob &p, const Ws &w, const double *psi, const double *ye, const double *T,
                         cudaStream_t s);

// A block per run of zones of a ray, in three phases over shared memory: X of every (zone, species, group)
// once, a thread per element, rows read whole; the limited differences; the group sums, a thread per
// (edge, species); the force, a thread per edge, and the zone values from the edges beside them.  Each
// edge is formed once (the run's first inner edge again).  Bound by the FP64 units; measured at 256 rays
// of 512 x 20: 303 -> 170 us (a thread per zone with both its edges before).
constexpr int kStressZones = 12, kStressThreads = 256;     // (31 KB of shared memory at 32 groups)
__global__ void __launch_bounds__(kStressThreads)
k_stress(Prob p, Ws w, const double *__restrict__ psi, double *__restrict__ f_edge, double *__restrict__ f_zone) {
  extern __shared__ double st_sm[];
  const int n = p.n, row = NS * n, last = p.n_r - 1;
  double *X = st_sm;                                        // [zones + 2][NS n]: eps^3 d eps psi / W E, zone lo + z
  double *lx = X + (size_t)(kStressZones + 2) * row;        // [zones + 1][NS n]: F (X_{i+1} - X_i)
  double *ia4 = lx + (size_t)(kStressZones + 1) * row;      // [zones + 2]
  double *sum = ia4 + kStressZones + 2;                     // [zones + 1][NS]
  double *fe = sum + (size_t)(kStressZones + 1) * NS;       // [zones + 1]
  const int runs = (p.n_r + kStressZones - 1) / kStressZones;
  const int ray = (int)blockIdx.x / runs, i0 = ((int)blockIdx.x - ray * runs) * kStressZones;
  // edges lo .. hi - 1 (edge i between zones i and i + 1), zones lo .. hi
  const int lo = i0 > 0 ? i0 - 1 : 0, hi = min(i0 + kStressZones, p.n_r), edges = hi - lo;
  const double *zr = w.zone + ((size_t)ray * p.n_r + lo) * ZC_N;
  for (int z = threadIdx.x; z <= edges && lo + z <= last; z += (int)blockDim.x) {
    const double ia = zr[(size_t)z * ZC_N + ZC_INV_A];
    ia4[z] = ia * ia * ia * ia;
  }
  __syncthreads();
  // (the block is whole rows of NS n threads: a thread keeps its species and group)
  const int e = threadIdx.x % row, q = e / n, k = e - q * n, z0 = threadIdx.x / row, dz = blockDim.x / row;
  const size_t sys = (size_t)ray * NS + q, g0 = (sys * p.n_r + lo) * n + k;
  for (int z = z0; z <= edges; z += dz)
    X[(size_t)z * row + e] = lo + z <= last ? psi[g0 + (size_t)z * n] * ia4[z]
                                            : w.ghost[sys * n + k] * (psi[g0 + (size_t)(z - 1) * n] * ia4[z - 1]);
  __syncthreads();
  for (int z = z0; z < edges; z += dz) {
    const size_t o = (size_t)z * row + e;
    lx[o] = w.lim[g0 + (size_t)z * n] * (X[o + row] - X[o]);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < edges * NS; t += (int)blockDim.x) {
    const double *l = lx + (size_t)t * n;                   // (edge, species) rows are consecutive
    double sq = 0.0;
    for (int k = 0; k < n; ++k) sq += l[k] * w.WE[k];
    sum[t] = sq;
  }
  __syncthreads();
  if ((int)threadIdx.x < edges) {
    const int z = threadIdx.x, i = lo + z;
    const double *zc = zr + (size_t)z * ZC_N;
    const double dM = p.rho[(size_t)ray * p.n_r + i] * zc[ZC_VOL];
    const double dMe = i < last ? 0.5 * (dM + p.rho[(size_t)ray * p.n_r + i + 1] * zc[ZC_N + ZC_VOL]) : dM;
    double s = 0.0;
    for (int q = 0; q < NS; ++q) s += stat_weight(q) * sum[z * NS + q];
    const double *re = p.r_edge + (size_t)ray * (p.n_r + 1);
    const double A = 4.0 * kPi * re[i + 1] * re[i + 1];
    const double f = -kFourPiHC3 / 3.0 * kMeVErg * s * A / dMe;
    fe[z] = f;
    if (f_edge && i >= i0) f_edge[(size_t)ray * p.n_r + i] = f;
  }
  __syncthreads();
  if (f_zone && (int)threadIdx.x < hi - i0) {
    const int i = i0 + threadIdx.x;
    f_zone[(size_t)ray * p.n_r + i] = 0.5 * (fe[i - lo] + (i > 0 ? fe[i - 1 - lo] : 0.0));
  }
}

// One block per ray, every thread a run of consecutive zones: the enclosed rest mass (block sum), x_j of
// the edges j + 1/2 below the last zone into scratch, and their suffix sums by runs, warps and the block.  Measured at
// 256 rays of 512 zones: 60 -> 23 us (a warp per ray, x_j formed twice, before).  Short rays take as many warps as
// they have zones for: 4000 rays of 64 zones 111 -> 48 us (62 with the warp per ray).
constexpr int kLapseThreads = 256;
__global__ void __launch_bounds__(kLapseThreads)
k_lapse(Prob p, const double *__restrict__ pres, const double *__restrict__ m_inner,
        const double *__restrict__ f_edge, const double *__restrict__ vol_src, int vol_stride,
        double *scratch, double *__restrict__ lapse) {
  __shared__ double wsum[2][kLapseThreads / 32];
  const int ray = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int nr = p.n_r, threads = (int)blockDim.x, warps = threads / 32, c = (nr + threads - 1) / threads;
  const double *rho = p.rho + (size_t)ray * nr, *pr = pres + (size_t)ray * nr, *fe = f_edge + (size_t)ray * nr;
  const double *re = p.r_edge + (size_t)ray * (nr + 1);
  const double *vol = vol_src + (size_t)ray * nr * vol_stride;
  double *xs = scratch + (size_t)ray * nr;
  double m = 0.0;
  for (int i = t; i < nr; i += threads) {
    const double dM = rho[i] * vol[(size_t)i * vol_stride];
    m += dM;
    double x = 0.0;
    if (i < nr - 1) {
      const double rho_e = 0.5 * (rho[i] + rho[i + 1]);
      const double dM_e = 0.5 * (dM + rho[i + 1] * vol[(size_t)(i + 1) * vol_stride]);
      const double R = re[i + 1];
      x = (pr[i + 1] - pr[i] - dM_e / (4.0 * kPi * R * R) * fe[i]) / (rho_e * kC * kC);
    }
    xs[i] = x;
  }
  for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
  if (lane == 0) wsum[0][wid] = m;
  __syncthreads();
  m = m_inner ? m_inner[ray] : 0.0;
  for (int j = 0; j < warps; ++j) m += wsum[0][j];
  const double a_out = sqrt(1.0 - 2.0 * kG * m / (kC * kC * re[nr]));
  // suffix sums: this run's, of the lanes above in the warp, of the warps above
  const int lo = min(t * c, nr), hi = min(lo + c, nr);
  double acc = 0.0;
  for (int i = hi - 1; i >= lo; --i) acc += xs[i];
  double v = acc;
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_down_sync(0xffffffffu, v, o);
    if (lane + o < 32) v += u;
  }
  if (lane == 0) wsum[1][wid] = v;
  __syncthreads();
  double run = v - acc;
  for (int j = wid + 1; j < warps; ++j) run += wsum[1][j];
  for (int i = hi - 1; i >= lo; --i) {
    run += xs[i];
    lapse[(size_t)ray * nr + i] = a_out * exp(run);
  }
}

}  // namespace mgfld

using namespace mgfld;

extern "C" mgfld_status mgfld_stress_lapse(const mgfld_dims *dims, const mgfld_problem *prob,
                                           const mgfld_state *state, const mgfld_stress_io *io, void *ws,
                                           size_t ws_bytes, void *stream) {
  if (!dims_ok(dims) || !prob_ok(prob) || !state || !state->psi || !state->ye || !state->T || !io || !ws)
    return MGFLD_EINVAL;
  if (io->lapse && !io->p) return MGFLD_EINVAL;
  if (((uintptr_t)ws & 255u) != 0) return MGFLD_EINVAL;
  const Layout L = make_layout(dims->n_ray, dims->n_r, dims->n_e, MGFLD_FP64);
  if (ws_bytes < L.total) return MGFLD_ENOMEM;
  cudaStream_t s = (cudaStream_t)stream;
  Ws w = resolve(ws, L);
  w.lim = w.lower;                       // the limiter of every edge (lower is free here)
  Prob p = make_prob(dims, prob);
  p.u = nullptr;                         // the shock terms do not enter the stress
  if (launch_setup(p, w, state->psi, state->ye, state->T, s) != cudaSuccess) return MGFLD_ECUDA;
  // the edge stress is needed by the lapse even when the caller does not keep it
  double *fe = io->f_edge ? io->f_edge : w.rhs;
  const int runs = (dims->n_r + kStressZones - 1) / kStressZones;
  const size_t sm = sizeof(double) * ((size_t)(2 * kStressZones + 3) * NS * dims->n_e + kStressZones + 2 + (kStressZones + 1) * (NS + 1));
  // (whole rows, no more of them than a run has zones: with few groups a block of 256 would mostly idle; the call at
  // 4000 rays of 64 zones and one group 535 -> 490 us)
  const int row = NS * dims->n_e, rows = kStressThreads / row;
  const int threads = (rows < kStressZones + 2 ? rows : kStressZones + 2) * row;
  k_stress<<<dims->n_ray * runs, threads, sm, s>>>(p, w, state->psi, fe, io->f_zone);
  if (cudaGetLastError() != cudaSuccess) return MGFLD_ECUDA;
  if (io->lapse) {
    const int lanes = (dims->n_r + 31) / 32 * 32;
    k_lapse<<<dims->n_ray, lanes < kLapseThreads ? lanes : kLapseThreads, 0, s>>>(p, io->p, io->m_inner, fe,
                                                                                  w.zone + ZC_VOL, ZC_N, w.src, io->lapse);
    if (cudaGetLastError() != cudaSuccess) return MGFLD_ECUDA;
  }
  return MGFLD_OK;
}
