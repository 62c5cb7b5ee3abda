// FP64 stage kernel of the time step and the device helpers that the other kernels share (Landau frame,
// Legendre series of the equilibrium, per-tile coefficients, tile schedules, group barriers). Included by
// rlb.cu inside its anonymous namespace; the file covers the kernel code that the FP64 profile summary was
// captured on, host code lives in rlb.cu.
#pragma once

constexpr int NT = 256;                    // threads per CTA
constexpr int GW = 64;                     // threads per velocity group (one row at a time)
constexpr int NG = NT / GW;                // velocity rows processed together
constexpr int TX = GW - 3;                 // cells per tile: their TX + 1 interfaces need GW indicator pairs
constexpr int HALO = 3;                    // WENO5 reaches three cells upwind/downwind
constexpr int RW = TX + 2 * HALO;          // staged row length
constexpr int NBC = QP_MAX * (NV_MAX + 1); // per-cell equilibrium coefficients

// Factors -k (k + 2) / ((2k + 1) (2k + 3)) of the backward recurrence of the Legendre coefficients
// (legendre_coeffs), filled once per device.
__device__ double g_leg[LEG_MAX + 1];

struct StageArgs {
  const TubeDev* tubes;
  const int2* tiles;  // (tube, first cell)
  const double* Fn;   // state at the start of the step (read at the cell only)
  const double* Fin;  // stage input (read with halo)
  double* Fout;       // stage output
  const double* tab;
  int* flag;
  int* warn;          // sticky warning bits (RLB_WARN_*) or NULL
  double a, b;        // Shu-Osher combination F_out = a F^n + b (F_in + dt L(F_in))
  int stage;          // 0, 1, 2: selects the b dt xi / dx table
  int ntiles;         // tiles of this launch
  int schedule;       // 0: one CTA per tile; 1: persistent, grid stride; 2: persistent, work counter
  int* counter;       // work counter of schedule 2 (zeroed before the launch)
  int split;          // work items per tile (<= 1: one): item k of a tile advances velocity rows
                      // [k Q / split, (k + 1) Q / split) after reducing the moments over all rows
};

// Tile loop of a stage launch. Schedule 0 gives each CTA one tile; the persistent schedules keep a grid of
// about one wave resident and hand out tiles by a grid stride or by an atomic work counter (cost-ordered
// tiles then balance uneven tubes). No CTA ever waits on another.
template <typename Body>
__device__ __forceinline__ void for_each_tile(int ntiles, int schedule, int* counter, Body body) {
  if (schedule == 0) {
    body((int)blockIdx.x);
    return;
  }
  if (schedule == 1) {
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
      __syncthreads();  // the previous tile's shared-memory readers are done
      body(t);
    }
    return;
  }
  __shared__ int next_tile;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) next_tile = atomicAdd(counter, 1);
    __syncthreads();
    const int t = next_tile;
    if (t >= ntiles) return;
    body(t);
  }
}

// --------------------------------------------------------------------------------------------------
// Device helpers
// --------------------------------------------------------------------------------------------------

// Source of a staged position x in [-HALO, Nx - 1 + GW + HALO] within its row: periodic wrap (Nx >= 3),
// zero-gradient ghosts (open boundary), or, on a halo side of a slab, the ghost cells the caller unpacked beside
// the row (left ghosts -3..-1 at ld-3..ld-1, right ghosts at Nx..Nx+2; ld >= Nx + 6 for slabs; positions past
// Nx + 2 are never read by a cell and map to Nx + 2). Always in [0, ld).
__device__ __forceinline__ int map_cell(int x, int Nx, int bc, int ld) {
  if (bc == RLB_BC_PERIODIC) {
    if (x < 0) x += Nx;
    return x % Nx;
  }
  if (x < 0) return (bc & RLB_BC_HALO_LEFT) ? ld + (x < -HALO ? -HALO : x) : 0;
  if (x >= Nx) return (bc & RLB_BC_HALO_RIGHT) ? (x > Nx + HALO - 1 ? Nx + HALO - 1 : x) : Nx - 1;
  return x;
}

// True where the fastest relaxation of a cell moving at beta, dt gamma (1 + |beta| max|xi|) / tau, is beyond the
// stable region of SSP-RK3 with WENO5 advection at the tube's Courant number (TubeDev::stiff_lim).
__device__ __forceinline__ bool stiff(const TubeDev& T, double beta) {
  const double k = T.dt * T.inv_tau * fma(fabs(beta), T.xi_max, 1.0);  // the rate without gamma = 1 / sqrt(1 - beta^2)
  return k * k > T.stiff_lim * T.stiff_lim * (1.0 - beta * beta);      // (k gamma)^2 > stiff_lim^2, no square root
}

// Landau frame from (N0, Nx, T00, T0x, Txx): e, beta, n (Landau), T, and gamma = (1 - beta^2)^-1/2 if gam_out is
// given. Returns false if non-physical. A cell at rest (T0x = 0, exactly so wherever the state is symmetric in xi)
// skips the division and square root that give beta = 0, gamma = 1 and n = N0.
__device__ __forceinline__ bool landau(const double mom[5], double& e, double& beta, double& n, double& T,
                                       double* gam_out = nullptr) {
  const double A = mom[2] + mom[4];
  const double disc = A * A - 4.0 * mom[3] * mom[3];
  e = 0.5 * ((mom[2] - mom[4]) + sqrt(disc));
  double gam = 1.0;
  if (mom[3] == 0.0) {
    beta = 0.0;
    n = mom[0];
  } else {
    beta = mom[3] / (mom[4] + e);
    gam = 1.0 / sqrt(1.0 - beta * beta);
    n = gam * (mom[0] - beta * mom[1]);
  }
  T = e / (3.0 * n);
  if (gam_out) *gam_out = gam;
  return disc >= 0.0 && e > 0.0 && fabs(beta) < 1.0 && n > 0.0 && T > 0.0;
}

// --------------------------------------------------------------------------------------------------
// Per-cell equilibrium coefficients of a tile (shared by the stage and initial-condition kernels)
// --------------------------------------------------------------------------------------------------

// Speed limits of the Legendre coefficients: a cell with |beta| beyond them is treated as non-physical. They are
// the speeds up to which the power series of (1 - beta xi)^-m, m = NPc + 2, (with the beta derivative: of its
// derivative too) falls below 1e-18 (1 - beta^2) within 16384 terms: the range the library documents.
__host__ __device__ constexpr double beta_limit(int NPc) { return NPc <= 2 ? 0.995524321007388 : 0.995025380567975; }
__host__ __device__ constexpr double beta_limit_d(int NPc) { return NPc <= 2 ? 0.994941897153004 : 0.994442517779333; }

// Legendre coefficients of (1 - beta xi)^-m: h[m - 2][k], m = 2 .. NM + 1, k = 0 .. KV, with
//   hhat_{m,k} = (2k+1)/2 int P_k(xi) (1 - beta xi)^-m dxi = h[m - 2][k] (gamma^2)^(m-1) / (m-1)!,
// gamma^2 = 1 / (1 - beta^2). b2 = beta^2, g1 = 1 - beta^2.
//
// The integrals are derivatives of the Legendre functions of the second kind Q_k(1/beta), and obey their
// recurrences (Abramowitz and Stegun, chapter 8): in k, at m = 2, with a_k = beta^k s_k c_k, s_k = s_{k-1}
// (k+1)/(2k+1):
//   c_{k-1} = c_k - k (k+2) / ((2k+1) (2k+3)) beta^2 c_{k+1},
// whose decaying solution is the wanted one; it is taken downward from c_{K+1} = 0, c_K = 1 (Miller's algorithm)
// and scaled by the closed form at k = 0. The error falls by ((1 - s)/(1 + s)), s = sqrt(1 - beta^2), per step, which
// gives K. In m:
//   m (1 - beta^2) a_{m+1,k} = (k + m - 1) beta a_{m,k-1} - (k - m + 1) a_{m,k},
// and for k = 0 the form without a_{m,-1}, m (1 - beta^2) a_{m+1,0} = m a_{m,0} + (m - 2) beta a_{m,1}.
// Against extended precision every coefficient is within a few units of FP64 rounding up to |beta| = 0.97 (as the
// positive power series in beta is, which takes 12 operations for each of its 40 terms at beta = 0.4 and 574 at 0.9;
// here about 2 operations for each of 18 and 46 steps). FP64 operations bound every kernel that calls this. With the
// series, the FP32 steps of 128 uneven moving tubes kept the FP64 pipe 85 % busy; on GB300 they went from 4.42 to 2.43
// ms, the FP32 stress tube's (half its gas in motion) from 6.5 to 5.2 ms, the 400-cell FP64 tube's from 89 to 54 us.
template <int NM, int KV>
__device__ __forceinline__ void legendre_coeffs(double beta, double b2, double g1, double (&h)[NM][KV + 1]) {
  double C[KV + 2];
  {
    // K = KV + 2 + 54 / -log2((1 - s)/(1 + s)), (1 - s)/(1 + s) = beta^2 / (1 + s)^2 (beta = 0: K = KV + 2)
    const float lr = 2.0f * __log2f(1.0f + sqrtf((float)g1)) - __log2f((float)b2);
    const int K = min(KV + 2 + (int)(54.0f / lr), LEG_MAX);
    double c1 = 1.0, c2 = 0.0;  // c_k, c_{k+1}
    for (int k = K; k > KV + 1; --k) {
      const double c0 = fma(g_leg[k], b2 * c2, c1);
      c2 = c1;
      c1 = c0;
    }
    C[KV + 1] = c1;
    C[KV] = fma(g_leg[KV + 1], b2 * c2, c1);
  }
#pragma unroll
  for (int k = KV; k >= 1; --k) C[k - 1] = fma(g_leg[k], b2 * C[k + 1], C[k]);
  const double inv = rlbdev::rcp_nr(C[0]);
  double bk = inv, sk = 1.0;  // beta^k / c_0; (2k+1) s_k
  h[0][0] = 1.0;
#pragma unroll
  for (int k = 1; k <= KV; ++k) {
    bk *= beta;
    sk *= (double)(k + 1) / (double)(2 * k + 1);
    h[0][k] = ((2 * k + 1) * sk) * (bk * C[k]);
  }
#pragma unroll
  for (int q = 1; q < NM; ++q) {
    const int m = q + 1;  // from m to m + 1
    h[q][0] = fma((m - 2) / 3.0, beta * h[q - 1][1], (double)m * h[q - 1][0]);
#pragma unroll
    for (int k = 1; k <= KV; ++k) {
      const double lead = (double)((k + m - 1) * (2 * k + 1)) / (double)(2 * k - 1);
      h[q][k] = fma(lead, beta * h[q - 1][k - 1], (double)(m - 1 - k) * h[q - 1][k]);
    }
  }
}

// The same times the per-cell factors of the equilibrium: ge[q][k] = g_q h[q][k], so that
//   F^eq_ij = sum_k B[i][k] w^xi_j P_k(xi_j),  B[i][k] = sum_q TAB_KW[i][q] ge[q][k]
// (Eq. (feqtrunc): Laguerre generating function for the radial projection, Legendre projection of each
// (1 - beta xi)^-m for the angular one; B = n/(4T^3) w^p_i sum_q s^(q+2) K[i][q] hhat_{q+2,k}, s = T/gamma, so
// that g_q = (n/T) (T gamma)^q).
template <int NPc, int NVc>
__device__ __forceinline__ void cell_coeffs(double beta, double b2, double g1, double g0, double tg,
                                            double (&ge)[NPc + 1][NVc + 1]) {
  legendre_coeffs<NPc + 1, NVc>(beta, b2, g1, ge);
  double g = g0;
#pragma unroll
  for (int q = 0; q <= NPc; ++q) {
#pragma unroll
    for (int k = 0; k <= NVc; ++k) ge[q][k] *= g;
    g *= tg;
  }
}

// Landau frame of a cell for the equilibrium: beta, beta^2, 1 - beta^2, gamma, g0 = n/T = 3 n^2/e and tg = T gamma =
// e gamma/(3n) from (N0, Nx, T00, T0x, Txx). As landau() with the refined hardware reciprocals in place of IEEE
// divisions and square roots (each corrected from its remainder where it is not itself a reciprocal), about 55
// FP64 operations instead of 150. Returns false if non-physical.
__device__ __forceinline__ bool landau_frame(const double mom[5], double& beta, double& b2, double& g1, double& gam,
                                             double& g0, double& tg) {
  const double A = mom[2] + mom[4], B2 = 2.0 * mom[3];
  const double disc = fma(A, A, -(B2 * B2));
  const double e = 0.5 * ((mom[2] - mom[4]) + rlbdev::sqrt_nr(disc));
  beta = rlbdev::div_nr(mom[3], mom[4] + e);
  b2 = beta * beta;
  g1 = fma(-beta, beta, 1.0);
  gam = rlbdev::rsqrt_nr(g1);
  const double n = gam * fma(-beta, mom[1], mom[0]);
  const double n3 = 3.0 * n;
  g0 = n3 * (n * rlbdev::rcp_nr(e));
  tg = (e * rlbdev::rcp_nr(n3)) * gam;
  return disc >= 0.0 && e > 0.0 && fabs(beta) < 1.0 && n > 0.0 && tg > 0.0;
}

struct CoefSmem {
  double ge[NP_MAX + 1][NV_MAX + 1][GW];  // cell_coeffs of the tile's cells
};

// Per-cell coefficients of one cell into column c of cs.ge (all zero for a non-physical cell).
template <int NPc, int NVc>
__device__ __forceinline__ void store_cell_coeffs(bool ok, double beta, double b2, double g1, double g0, double tg,
                                                  CoefSmem& cs, int c) {
  double ge[NPc + 1][NVc + 1];
  if (ok) {
    cell_coeffs<NPc, NVc>(beta, b2, g1, g0, tg, ge);
  } else {
#pragma unroll
    for (int q = 0; q <= NPc; ++q)
#pragma unroll
      for (int k = 0; k <= NVc; ++k) ge[q][k] = 0.0;
  }
#pragma unroll
  for (int q = 0; q <= NPc; ++q)
#pragma unroll
    for (int k = 0; k <= NVc; ++k) cs.ge[q][k][c] = ge[q][k];
}

// Fill B[i (NVc+1) + k][c] (radial rows i < Qp) for the TX cells of a tile from cs.ge: group g builds radial row
// i = g.
template <int NPc, int NVc>
__device__ __forceinline__ void build_rows(const double* tab, int Qp, const CoefSmem& cs, double (*Bs)[GW]) {
  const int c = threadIdx.x % GW, i = threadIdx.x / GW;
  if (c >= TX || i >= Qp) return;
  double KW[NPc + 1];
#pragma unroll
  for (int q = 0; q <= NPc; ++q) KW[q] = tab[TAB_KW + i * (NP_MAX + 1) + q];
#pragma unroll
  for (int k = 0; k <= NVc; ++k) {
    double B = KW[0] * cs.ge[0][k][c];
#pragma unroll
    for (int q = 1; q <= NPc; ++q) B = fma(KW[q], cs.ge[q][k][c], B);
    Bs[i * (NVc + 1) + k][c] = B;
  }
}

// --------------------------------------------------------------------------------------------------
// Stage kernel
// --------------------------------------------------------------------------------------------------

// Barrier of one 64-thread velocity group (named barrier 1 + g; barrier 0 is __syncthreads).
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(GW) : "memory"); }

struct StageSmem {
  union {
    struct {
      double red[NG][3 * QP_MAX][GW];  // per group: the radial sums S0, S1, S2 of each radial node
      CoefSmem coef;
    } a;                               // phases A and B
    struct {
      double row[2][NG][RW + 1];  // staged velocity rows (double-buffered: written before the first barrier)
      double d1[NG][RW + 1];      // first differences by position, d1[k] = row[k] - row[k-1]
      float2 dd[NG][RW + 1];      // the same differences in double-float (hi, lo)
      float2 sv[NG][3][GW];       // indicators v = S + e (double-float), one triple per pair of adjacent differences
      float2 phi[NG][GW];         // WENO correction of each interface, times 6 (double-float)
    } c;                          // phase C
  } u;
  double rate[2][GW];
  int src[RW + 1];            // source cell of each staged position (boundary condition applied)
  double B[NBC][GW];          // equilibrium coefficients B[i (NVc + 1) + k]; last, so that a launch allocates
                              // only the rows its tubes use (stage_smem_bytes)
};
// Dynamic shared memory of the FP64 stage kernel for `brows` coefficient rows.
constexpr size_t stage_smem_bytes(int brows) { return offsetof(StageSmem, B) + (size_t)brows * GW * sizeof(double); }

template <int NPc, int NVc>
__device__ void stage_tile(const StageArgs& A, const TubeDev& T, int x0, int part, int nparts, StageSmem& sm) {
  const int tid = threadIdx.x, c = tid % GW, g = tid / GW;
  const double* tab = A.tab + T.tab;
  const int Qp = T.Qp, Qxi = T.Qxi, Nx = T.Nx, ld = T.ld;
  const double* Fin = A.Fin + T.off;
  const double* Fn = A.Fn + T.off;
  double* Fout = A.Fout + T.off;
  const int x = x0 + c;
  const bool cell = (c < TX) && (x < Nx);
  for (int k = tid; k < RW; k += NT) sm.src[k] = map_cell(x0 - HALO + k, Nx, T.bc, ld);

  if (T.collide) {
    // A. moments of the stage input. The groups split the mirror pairs of directions (xi_jf = -xi_jb > 0) and
    //    keep, per radial node i, S0 = sum_j F_ij, S1 = sum_j F_ij xi_j and S2 = sum_j F_ij xi_j^2 from the sum
    //    s = F(xi) + F(-xi) and difference d = F(xi) - F(-xi) of each pair (S0 += s, S1 += d xi, S2 += s xi^2):
    //    5 FP64 operations per two populations. An odd Qxi's xi = 0 direction adds to S0 only. Then
    //    N0 = sum_i pbar_i S0_i, Nx = sum_i pbar_i S1_i, T00 = sum_i pbar_i^2 S0_i, T0x = sum_i pbar_i^2 S1_i and
    //    Txx = sum_i pbar_i^2 S2_i.
    double S[3 * QP_MAX];
#pragma unroll
    for (int k = 0; k < 3 * QP_MAX; ++k) S[k] = 0.0;
    const int hq = Qxi / 2;
    if (cell) {
      for (int jb = g; jb < hq; jb += NG) {
        const int jf = Qxi - 1 - jb;
        const double xi = tab[TAB_XI + jf], xi2 = xi * xi;
#pragma unroll
        for (int i = 0; i < QP_MAX; ++i) {
          if (i < Qp) {
            const double ff = __ldg(Fin + (size_t)(i * Qxi + jf) * ld + x);
            const double fb = __ldg(Fin + (size_t)(i * Qxi + jb) * ld + x);
            const double sum = ff + fb, dif = ff - fb;
            S[3 * i] += sum;
            S[3 * i + 1] = fma(dif, xi, S[3 * i + 1]);
            S[3 * i + 2] = fma(sum, xi2, S[3 * i + 2]);
          }
        }
      }
      if ((Qxi & 1) && g == (hq % NG)) {
#pragma unroll
        for (int i = 0; i < QP_MAX; ++i)
          if (i < Qp) S[3 * i] += __ldg(Fin + (size_t)(i * Qxi + hq) * ld + x);
      }
    }
#pragma unroll
    for (int k = 0; k < 3 * QP_MAX; ++k) sm.u.a.red[g][k][c] = S[k];
    __syncthreads();
    // B. Landau frame and Legendre coefficients (one thread per cell), then the equilibrium coefficients
    if (g == 0) {
      double beta = 0.0, b2 = 0.0, g1 = 1.0, gam = 1.0, g0 = 0.0, tg = 1.0;
      bool ok = false;
      if (cell) {
        double mom[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int i = 0; i < QP_MAX; ++i) {
          if (i < Qp) {
            double Si[3];
#pragma unroll
            for (int q = 0; q < 3; ++q)
              Si[q] = (sm.u.a.red[0][3 * i + q][c] + sm.u.a.red[1][3 * i + q][c]) +
                      (sm.u.a.red[2][3 * i + q][c] + sm.u.a.red[3][3 * i + q][c]);
            const double p1 = tab[TAB_PBAR + i], p2 = tab[TAB_PBAR2 + i];
            mom[0] = fma(p1, Si[0], mom[0]);
            mom[1] = fma(p1, Si[1], mom[1]);
            mom[2] = fma(p2, Si[0], mom[2]);
            mom[3] = fma(p2, Si[1], mom[3]);
            mom[4] = fma(p2, Si[2], mom[4]);
          }
        }
        ok = landau_frame(mom, beta, b2, g1, gam, g0, tg);
        if (ok && A.warn != nullptr && stiff(T, beta)) atomicOr(A.warn, RLB_WARN_STIFF);
        ok = ok && fabs(beta) <= beta_limit(NPc);
        if (!ok) atomicOr(A.flag, 1);
      }
      store_cell_coeffs<NPc, NVc>(ok, beta, b2, g1, g0, tg, sm.u.a.coef, c);
      // b dt gamma / tau and its beta multiple: the stage's collision rate is r0 - r1 xi_j
      const double r0 = ok ? (A.b * T.dt) * (T.inv_tau * gam) : 0.0;
      sm.rate[0][c] = r0;
      sm.rate[1][c] = ok ? r0 * beta : 0.0;
    }
    __syncthreads();
    build_rows<NPc, NVc>(tab, Qp, sm.u.a.coef, sm.B);
  }
  __syncthreads();  // sm.src (and, with collisions, the coefficients) are ready

  // C. advection + collision + Runge-Kutta combination. The work unit of a 64-thread group is a mirror pair
  //    of directions (j, Qxi - 1 - j) of one radial node, processed back to back: the nodes are symmetric, so
  //    w^xi P_k(-xi) = (-1)^k w^xi P_k(xi) and the even and odd Legendre parts of F^eq, summed once, give both
  //    rows' equilibria (the xi = 0 node of an odd Qxi is a unit of its own). Groups synchronise with named
  //    barriers only.
  const double a = A.a, b = A.b;
  const double* cxi_tab = tab + tab_cxi(Qxi) + A.stage * Qxi;
  double* d1 = sm.u.c.d1[g];
  float2* dd = sm.u.c.dd[g];
  float2* sv0 = sm.u.c.sv[g][0];
  float2* sv1 = sm.u.c.sv[g][1];
  float2* sv2 = sm.u.c.sv[g][2];
  float2* phi = sm.u.c.phi[g];
  const float2* epsf = reinterpret_cast<const float2*>(tab + tab_epsf(Qp, Qxi));
  const int hq = Qxi / 2, upr = hq + (Qxi & 1), U = Qp * upr;
  const int u_end = (part + 1) * U / nparts;
  int buf = 0;
  for (int u0 = part * U / nparts; u0 < u_end; u0 += NG) {
    const int u = u0 + g;
    if (u >= u_end) continue;  // uniform over the group
    const int i = u / upr, jA = u - i * upr;  // jA = hq: the xi = 0 node
    const int nrow = jA < hq ? 2 : 1;
    double E = 0.0, O = 0.0;  // even and odd parts of sum_k B[i][k] w^xi P_k(xi_jA) at this cell
    for (int h = 0; h < nrow; ++h, buf ^= 1) {
      const int j = h == 0 ? jA : Qxi - 1 - jA;
      const int s = i * Qxi + j;
      double* row = sm.u.c.row[buf][g];
      // stage the row with its first differences, in FP64 and split into double-float (position k needs k - 1
      // as well)
      {
        const double* src = Fin + (size_t)s * ld;
        // positions 0 .. GW-1, one per thread: the previous position's value comes from the lane below by a
        // shuffle (the first lane of each warp loads it)
        {
          const double v = __ldg(src + sm.src[c]);
          row[c] = v;
          const double below = __shfl_up_sync(0xffffffffu, v, 1);
          if (c > 0) {
            const double dk = v - ((c & 31) == 0 ? __ldg(src + sm.src[c - 1]) : below);
            d1[c] = dk;
            const rlbdev::DF q = rlbdev::df_split(dk);
            dd[c] = make_float2(q.hi, q.lo);
          }
        }
        for (int k = c + GW; k < RW; k += GW) {
          const double v = __ldg(src + sm.src[k]);
          row[k] = v;
          const double dk = v - __ldg(src + sm.src[k - 1]);
          d1[k] = dk;
          const rlbdev::DF q = rlbdev::df_split(dk);
          dd[k] = make_float2(q.hi, q.lo);
        }
      }
      // the Runge-Kutta input of this row's cell, loaded now so that its latency hides behind the limiter
      const double fnv = (A.stage != 0 && cell) ? __ldg(Fn + (size_t)s * ld + x) : 0.0;
      group_sync(g);
      const double xi = tab[TAB_XI + j];
      const bool fwd = h == 1;  // the mirror row xi_{Qxi-1-jA} > 0; the first row has xi <= 0
      // pairs: thread c owns the pair of differences at positions (p, p + 1), p = c + 1 (wind toward +x) or
      // c + 2 (toward -x); these are the pairs the TX + 1 interfaces of the tile use
      {
        const int p = c + (fwd ? 1 : 2);
        const float2 e = epsf[s], x = dd[p], y = dd[p + 1];
        rlbdev::DF va, vb, vc;
        rlbdev::weno5_pair_df({x.x, x.y}, {y.x, y.y}, fwd, {e.x, e.y}, va, vb, vc);
        sv0[c] = make_float2(va.hi, va.lo);
        sv1[c] = make_float2(vb.hi, vb.lo);
        sv2[c] = make_float2(vc.hi, vc.lo);
      }
      group_sync(g);
      // interfaces: interface c lies between cells x0 + c - 1 and x0 + c (row index c + 2 | c + 3); its value
      // is v2 + G with v2 the upwind cell; D = v2(c + 1) - v2(c) is the memory-order difference d1[c + 3]
      // (wind toward +x) or d1[c + 4] (toward -x)
      double D = 0.0;
      if (c <= TX) {
        auto get = [](const float2* a, int k) { const float2 q = a[k]; return rlbdev::DF{q.x, q.y}; };
        auto neg = [&](int k) { const float2 q = dd[k]; return rlbdev::DF{-q.x, -q.y}; };
        rlbdev::DF G;
        if (fwd) {
          D = d1[c + 3];
          G = rlbdev::weno5_combine6_df(get(sv0, c), get(sv1, c + 1), get(sv2, c + 2), get(dd, c + 1),
                                        get(dd, c + 2), get(dd, c + 3), get(dd, c + 4));
        } else {
          D = d1[c + 4];
          G = rlbdev::weno5_combine6_df(get(sv0, c + 2), get(sv1, c + 1), get(sv2, c), neg(c + 5), neg(c + 4),
                                        neg(c + 3), neg(c + 2));
        }
        phi[c] = make_float2(G.hi, G.lo);
      }
      group_sync(g);
      if (cell) {
        const double F = row[c + 3];
        // phi holds 6 G: D + (6 G_{x+1/2} - 6 G_{x-1/2}) / 6, the difference taken in double-float
        const float2 pr = phi[c + 1], pl = phi[c];
        const rlbdev::DF dG = rlbdev::df_plus({pr.x, pr.y}, {-pl.x, -pl.y});
        const double dphi = fma(rlbdev::df_widen(dG.hi), 1.0 / 6.0, fma(rlbdev::df_widen(dG.lo), 1.0 / 6.0, D));
        double out = F;
        if (A.stage != 0) out = fma(a, fnv, b * F);  // a = 0 in the first stage
        out = fma(-cxi_tab[j], dphi, out);  // - b dt xi/dx (Phi_{x+1/2} - Phi_{x-1/2})
        if (T.collide) {
          if (h == 0) {
            const double* pw = tab + TAB_XI + Qxi + jA * (NV_MAX + 1);
#pragma unroll
            for (int k = 0; k <= NVc; ++k) {
              const double t = sm.B[i * (NVc + 1) + k][c];
              if (k % 2 == 0)
                E = fma(t, pw[k], E);
              else
                O = fma(t, pw[k], O);
            }
          }
          const double feq = h == 0 ? E + O : E - O;
          const double rate = fma(-sm.rate[1][c], xi, sm.rate[0][c]);
          out = fma(rate, feq - F, out);  // + b dt gamma (1 - beta xi)/tau (F^eq - F)
        }
        Fout[(size_t)s * ld + x] = out;
      }
    }
  }
}

// SCHED is the launch's schedule (compile time, so that the one-CTA-per-tile kernel carries no tile loop).
template <int SCHED>
__global__ void __launch_bounds__(NT, 3) rlb_stage_kernel(StageArgs A) {
  extern __shared__ __align__(16) unsigned char stage_smem_raw[];
  StageSmem& sm = *reinterpret_cast<StageSmem*>(stage_smem_raw);
  const int K = A.split > 1 ? A.split : 1;
  for_each_tile(A.ntiles * K, SCHED, A.counter, [&](int item) {
    const int t = item / K, part = item - t * K;
    const int2 tl = A.tiles[t];
    const TubeDev T = A.tubes[tl.x];
    if (T.Np == 2 && T.Nv == 5)
      stage_tile<2, 5>(A, T, tl.y, part, K, sm);
    else
      stage_tile<NP_MAX, NV_MAX>(A, T, tl.y, part, K, sm);
  });
}
