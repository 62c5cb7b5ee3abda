// FP64 stage kernel of the time step and the device helpers that the other kernels share (Landau frame,
// Legendre coefficients of the equilibrium, per-tile coefficients, tile schedules, group barriers). Included by
// rlb.cu inside its anonymous namespace; host code lives in rlb.cu.
#pragma once

constexpr int NT = 256;                    // threads per CTA
constexpr int GW = 64;                     // threads per velocity group (one row at a time)
constexpr int NG = NT / GW;                // velocity rows processed together
constexpr int TX = GW - 4;                 // cells per tile: the stencils of their TX + 1 interfaces hold GW differences
constexpr int HALO = 3;                    // WENO5 reaches three cells upwind/downwind
constexpr int RW = TX + 2 * HALO;          // staged cells x0 - 3 .. x0 + TX + 2
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
                      // [k Q / split, (k + 1) Q / split); under schedules 1 and 2 each item reduces the
                      // moments over all rows, else the items are a cluster that shares them
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

// Source of a staged position x in [-HALO, Nx - 1 + TX + HALO] within its row: periodic wrap (Nx >= 3),
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

// Landau frame from (N0, Nx, T00, T0x, Txx): e, beta, n (Landau), T. Returns false if non-physical. A cell at rest
// (T0x = 0, exactly so wherever the state is symmetric in xi) skips the division and square root that give beta = 0 and
// n = N0.
__device__ __forceinline__ bool landau(const double mom[5], double& e, double& beta, double& n, double& T) {
  const double A = mom[2] + mom[4];
  const double disc = A * A - 4.0 * mom[3] * mom[3];
  e = 0.5 * ((mom[2] - mom[4]) + sqrt(disc));
  if (mom[3] == 0.0) {
    beta = 0.0;
    n = mom[0];
  } else {
    beta = mom[3] / (mom[4] + e);
    n = 1.0 / sqrt(1.0 - beta * beta) * (mom[0] - beta * mom[1]);
  }
  T = e / (3.0 * n);
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
// Largest error of a coefficient against extended precision, in units of 2^-52: Np = 2, Nv = 5: 5 up to |beta| = 0.7, 9 at
// 0.97, 12 at 0.9949; Np = 3, Nv = 8: 7 up to 0.45, 12 at 0.7, 24 at 0.97, 34 at 0.9949. The positive power series in beta
// has 8 at 0.7, 30 at 0.97 and 145 at 0.9949 for either, and takes 12 operations for each of its 40 terms at beta = 0.4
// and 574 at 0.9; here about 2 operations for each of 18 and 46 steps. FP64 operations bound every kernel that calls this. With the
// series, the FP32 steps of 128 uneven moving tubes kept the FP64 pipe 85 % busy; on GB300 they went from 4.42 to 2.43
// ms, the FP32 stress tube's (half its gas in motion) from 6.5 to 5.2 ms, the 400-cell FP64 tube's from 89 to 54 us.
template <int KV>
__device__ __forceinline__ void legendre_first(double beta, double b2, double g1, double (&h)[KV + 1]) {
  double C[KV + 2];
  {
    // K = KV + 1 + 54 / -log2((1 - s)/(1 + s)), (1 - s)/(1 + s) = beta^2 / (1 + s)^2 (beta = 0: K = KV + 1)
    const float lr = 2.0f * __log2f(1.0f + sqrtf((float)g1)) - __log2f((float)b2);
    const int K = min(KV + 1 + (int)(54.0f / lr), LEG_MAX);
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
  h[0] = 1.0;
#pragma unroll
  for (int k = 1; k <= KV; ++k) {
    bk *= beta;
    sk *= (double)(k + 1) / (double)(2 * k + 1);
    h[k] = ((2 * k + 1) * sk) * (bk * C[k]);
  }
}
// Coefficients of the step from the power m to m + 1 at order k: h' = lead beta h[k == 0 ? 1 : k - 1] + own h[k].
__host__ __device__ constexpr double leg_lead(int m, int k) {
  return k == 0 ? (m - 2) / 3.0 : (double)((k + m - 1) * (2 * k + 1)) / (double)(2 * k - 1);
}
__host__ __device__ constexpr double leg_own(int m, int k) { return k == 0 ? m : m - 1 - k; }

template <int NM, int KV>
__device__ __forceinline__ void legendre_coeffs(double beta, double b2, double g1, double (&h)[NM][KV + 1]) {
  legendre_first<KV>(beta, b2, g1, h[0]);
#pragma unroll
  for (int q = 1; q < NM; ++q) {
    const int m = q + 1;  // from m to m + 1
#pragma unroll
    for (int k = 0; k <= KV; ++k) {
      const double b = beta * h[q - 1][k == 0 ? 1 : k - 1];
      h[q][k] = leg_own(m, k) == 0.0   ? leg_lead(m, k) * b
                : leg_lead(m, k) == 0.0 ? leg_own(m, k) * h[q - 1][k]
                                        : fma(leg_lead(m, k), b, leg_own(m, k) * h[q - 1][k]);
    }
  }
}

// Per-cell factors of the equilibrium: with g[q] = c_q (n/T) (T gamma)^q (c_q: TAB_KC) and h of legendre_coeffs,
//   F^eq_ij = sum_k B[i][k] w^xi_j P_k(xi_j),  B[i][k] = sum_q (TAB_KW[i][q] g[q]) h[q][k]
// (Eq. (feqtrunc): Laguerre generating function for the radial projection, Legendre projection of each
// (1 - beta xi)^-m for the angular one; B = n/(4T^3) w^p_i sum_q s^(q+2) K[i][q] hhat_{q+2,k}, s = T/gamma).
template <int NPc>
__device__ __forceinline__ void cell_factors(const double* tab, double g0, double tg, double (&g)[NPc + 1]) {
  double t = g0;
#pragma unroll
  for (int q = 0; q <= NPc; ++q) {
    g[q] = t * tab[TAB_KC + q];
    t *= tg;
  }
}

// Landau frame of a cell for the equilibrium: beta, beta^2, 1 - beta^2, gamma, g0 = n/T = 3 n^2/e and tg = T gamma =
// e gamma/(3n) from (N0, Nx, T00, T0x, Txx). As landau() with the refined hardware reciprocals in place of IEEE
// divisions and square roots (each corrected from its remainder where it is not itself a reciprocal), about 55
// FP64 operations instead of 150. Returns false if non-physical.
__device__ __forceinline__ bool landau_frame(const double mom[5], double& beta, double& b2, double& g1, double& gam,
                                             double& g0, double& tg) {
  const double A = mom[2] + mom[4];
  double disc = 1.0, e, n;
  if (((unsigned long long)__double_as_longlong(mom[3]) << 1) == 0ull) {
    // at rest (T0x = 0, exactly so wherever the state is symmetric in xi): sqrt(A^2) = |A|, beta = 0
    e = 0.5 * ((mom[2] - mom[4]) + fabs(A));
    beta = b2 = 0.0;
    g1 = gam = 1.0;
    n = mom[0];
  } else {
    const double B2 = 2.0 * mom[3];
    disc = fma(A, A, -(B2 * B2));
    e = 0.5 * ((mom[2] - mom[4]) + rlbdev::sqrt_nr(disc));
    beta = rlbdev::div_nr(mom[3], mom[4] + e);
    b2 = beta * beta;
    g1 = fma(-beta, beta, 1.0);
    gam = rlbdev::rsqrt_nr(g1);
    n = gam * fma(-beta, mom[1], mom[0]);
  }
  const double n3 = 3.0 * n;
  g0 = n3 * (n * rlbdev::rcp_nr(e));
  tg = (e * rlbdev::rcp_nr(n3)) * gam;
  return disc >= 0.0 && e > 0.0 && fabs(beta) < 1.0 && n > 0.0 && tg > 0.0;
}

struct CoefSmem {
  double h[NP_MAX + 1][NV_MAX + 1][GW];  // Legendre coefficients of the tile's cells
  double g[NP_MAX + 1][GW];              // and their factors
};

// Coefficients and factors of one cell into column c of cs (all zero for a non-physical cell).
template <int NPc, int NVc>
__device__ __forceinline__ void store_cell_coeffs(const double* tab, bool ok, double beta, double b2, double g1, double g0, double tg,
                                                  CoefSmem& cs, int c) {
  double h[NPc + 1][NVc + 1], g[NPc + 1];
  if (ok) {
    legendre_coeffs<NPc + 1, NVc>(beta, b2, g1, h);
    cell_factors<NPc>(tab, g0, tg, g);
  } else {
#pragma unroll
    for (int q = 0; q <= NPc; ++q) {
      g[q] = 0.0;
#pragma unroll
      for (int k = 0; k <= NVc; ++k) h[q][k] = 0.0;
    }
  }
#pragma unroll
  for (int q = 0; q <= NPc; ++q) {
    cs.g[q][c] = g[q];
#pragma unroll
    for (int k = 0; k <= NVc; ++k) cs.h[q][k][c] = h[q][k];
  }
}

// B[i][k] of cell c.
template <int NPc>
__device__ __forceinline__ double row_coeff(const double* tab, int i, const CoefSmem& cs, int k, int c) {
  const double* KW = tab + TAB_KW + i * (NP_MAX + 1);
  double B = (KW[0] * cs.g[0][c]) * cs.h[0][k][c];
#pragma unroll
  for (int q = 1; q <= NPc; ++q) B = fma(KW[q] * cs.g[q][c], cs.h[q][k][c], B);
  return B;
}

// Fill B[i (NVc+1) + k][c] (radial rows i < Qp) for the TX cells of a tile from cs: group g builds radial row
// i = g. Coefficients of w^xi_j P_k(xi_j).
template <int NPc, int NVc>
__device__ __forceinline__ void build_rows(const double* tab, int Qp, const CoefSmem& cs, double (*Bs)[GW]) {
  const int c = threadIdx.x % GW, i = threadIdx.x / GW;
  if (c >= TX || i >= Qp) return;
#pragma unroll
  for (int k = 0; k <= NVc; ++k) Bs[i * (NVc + 1) + k][c] = row_coeff<NPc>(tab, i, cs, k, c);
}

// Orders up to which the stage kernel evaluates the equilibrium as a polynomial in xi (two Horner chains in xi^2) from
// monomial coefficients; above, from the Legendre ones (the change of basis loses digits as the order grows: its
// entries reach 63/8 at order 5, 429/16 at 7).
constexpr int NV_MONO = 5;

// Legendre to monomial coefficients of one column, in place: B[k] of P_k becomes B[k] of xi^k.
template <int NVc>
__device__ __forceinline__ void legendre_to_monomial(double* B, int stride) {
  static_assert(NVc == NV_MONO, "the table is for this order");
  const double b0 = B[0], b1 = B[stride], b2 = B[2 * stride], b3 = B[3 * stride], b4 = B[4 * stride], b5 = B[5 * stride];
  B[0] = fma(0.375, b4, fma(-0.5, b2, b0));
  B[stride] = fma(1.875, b5, fma(-1.5, b3, b1));
  B[2 * stride] = fma(-3.75, b4, 1.5 * b2);
  B[3 * stride] = fma(-8.75, b5, 2.5 * b3);
  B[4 * stride] = 4.375 * b4;
  B[5 * stride] = 7.875 * b5;
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
      double d1[NG][2][GW];         // first differences of a mirror pair's two rows, in wind order
      float4 dd[NG][GW];            // the same in double-float: (hi, hi', lo, lo')
      float4 sv[NG][2][GW];         // indicators v_B, v_C of each pair of adjacent differences (both rows)
      float2 phi[NG][2][GW];        // WENO correction of each interface, times 6 (double-float), by row
    } c;                            // phase C
  } u;
  double rate[2][GW];
  double cst[5];                    // 1, 1/6, the Runge-Kutta a, b, and -0, for register operands
  int src[RW + 1];                  // source cell of each staged position (boundary condition applied)
  double B[NBC][GW];                // equilibrium coefficients B[i (NVc + 1) + k]; last, so that a launch allocates
                                    // only the rows its tubes use (stage_smem_bytes)
};
// Dynamic shared memory of the FP64 stage kernel for `brows` coefficient rows.
constexpr size_t stage_smem_bytes(int brows) { return offsetof(StageSmem, B) + (size_t)brows * GW * sizeof(double); }

// Operand forms. On GB300 an FP64 FMA whose three operands are all registers issues every 16 cycles per SM; an
// addition, a multiplication, or an FMA with a constant-bank or immediate operand every 19 (measured). The hot loops
// therefore add and multiply by FMAs with a register 1 or -0 (same rounding), and keep their constants in registers
// that the compiler cannot fold (read from shared memory).
__device__ __forceinline__ double add_r(double a, double b, double one) { return fma(a, one, b); }

// Phase B of one cell: the five moments from the groups' radial sums, Landau frame, Legendre coefficients into
// sm.u.a.coef and the collision rate into sm.rate (zeros for a cell past the tube's end or a non-physical one).
template <int NPc, int NVc>
__device__ __forceinline__ void cell_phase(const StageArgs& A, const TubeDev& T, const double* tab, bool cell, int c,
                                           StageSmem& sm) {
  double beta = 0.0, b2 = 0.0, g1 = 1.0, gam = 1.0, g0 = 0.0, tg = 1.0;
  bool ok = false;
  if (cell) {
    double mom[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < QP_MAX; ++i) {
      if (i < T.Qp) {
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
  store_cell_coeffs<NPc, NVc>(tab, ok, beta, b2, g1, g0, tg, sm.u.a.coef, c);
  // b dt gamma / tau and its beta multiple: the stage's collision rate is r0 - r1 xi_j
  const double r0 = ok ? (A.b * T.dt) * (T.inv_tau * gam) : 0.0;
  sm.rate[0][c] = r0;
  sm.rate[1][c] = ok ? r0 * beta : 0.0;
}

// Thread-block clusters: barrier over the CTAs of the cluster (release / acquire), and a store to the same place of the
// shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_store(double* p, int rank, double v) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
}

// Moments, Landau frame and equilibrium coefficients of a tile shared by the nparts CTAs that split its velocity rows
// (one cluster): CTA `part` takes every cell of its share through phases A and B with the operations and the order of
// summation of the unshared path, and stores the results to all of them. Small handles only: the per-cell work was
// repeated in each of up to 8 CTAs, and with FP64 at 2 lanes per SM and clock that was two thirds of a stage.
template <int NPc, int NVc>
__device__ __forceinline__ void cluster_coeffs(const StageArgs& A, const TubeDev& T, int x0, int part, int nparts,
                                               StageSmem& sm) {
  const int tid = threadIdx.x;
  const double* tab = A.tab + T.tab;
  const int Qp = T.Qp, Qxi = T.Qxi, Nx = T.Nx, ld = T.ld, hq = Qxi / 2;
  const double* Fin = A.Fin + T.off;
  const int share = (TX + nparts - 1) / nparts, c0 = part * share;  // cells c0 .. c0 + share - 1 of the tile
  const int lg = share <= 8 ? 3 : (share <= 16 ? 4 : 5), cc = tid & ((1 << lg) - 1), c = c0 + cc;
  const bool own = cc < share && c < TX, cell = own && x0 + c < Nx;
  const double one = *const_cast<const volatile double*>(&sm.cst[0]);
  // A. one slice (every NG-th mirror pair) of one radial node per thread
  for (int w = tid >> lg; w < NG * Qp; w += NT >> lg) {
    const int gs = w & (NG - 1), i = w / NG;
    double S0 = 0.0, S1 = 0.0, S2 = 0.0;
    if (cell) {
      const double* r = Fin + (size_t)(i * Qxi) * ld + x0 + c;
#pragma unroll 2
      for (int jb = gs; jb < hq; jb += NG) {
        const int jf = Qxi - 1 - jb;
        const double ff = __ldg(r + (size_t)jf * ld), fb = __ldg(r + (size_t)jb * ld);
        const double sum = add_r(fb, ff, one), dif = fma(-fb, one, ff);
        S0 = add_r(sum, S0, one);
        S1 = fma(dif, tab[TAB_XI + jf], S1);
        S2 = fma(sum, tab[tab_xi2(Qp, Qxi) + jf], S2);
      }
      if ((Qxi & 1) && gs == (hq % NG)) S0 += __ldg(r + (size_t)hq * ld);
    }
    if (own) {
      sm.u.a.red[gs][3 * i][c] = S0;
      sm.u.a.red[gs][3 * i + 1][c] = S1;
      sm.u.a.red[gs][3 * i + 2][c] = S2;
    }
  }
  __syncthreads();
  // B. per cell, on one warp (a different scheduler in neighbouring CTAs)
  if ((tid >> 5) == (part & 3) && (tid & 31) < share && c0 + (tid & 31) < TX)
    cell_phase<NPc, NVc>(A, T, tab, x0 + c0 + (tid & 31) < Nx, c0 + (tid & 31), sm);
  __syncthreads();
  // B[i][k], a thread per radial row where the share fills the warps (the factors KW g once per row: 2 % of a launch on
  // 13 uneven tubes), else a thread per coefficient
  if (own && share > 8) {
    if ((tid >> lg) < Qp) {
#pragma unroll
      for (int k = 0; k <= NVc; ++k)
        sm.B[(tid >> lg) * (NVc + 1) + k][c] = row_coeff<NPc>(tab, tid >> lg, sm.u.a.coef, k, c);
    }
  } else if (own) {
    for (int w = tid >> lg; w < Qp * (NVc + 1); w += NT >> lg) {
      const int i = w / (NVc + 1), k = w - i * (NVc + 1);
      sm.B[w][c] = row_coeff<NPc>(tab, i, sm.u.a.coef, k, c);
    }
  }
  __syncthreads();
  if constexpr (NVc <= NV_MONO) {
    if (own && (tid >> lg) < Qp) legendre_to_monomial<NVc>(&sm.B[(tid >> lg) * (NVc + 1)][c], GW);
    __syncthreads();
  }
  cluster_sync();  // every CTA of the cluster runs: its shared memory can be written
  if (own) {
    const int rows = Qp * (NVc + 1);
    for (int w = tid >> lg; w < rows + 2; w += NT >> lg) {
      double* p = w < rows ? &sm.B[w][c] : &sm.rate[w - rows][c];
      const double v = *p;
      for (int r = 0; r < nparts; ++r)
        if (r != part) cluster_store(p, r, v);
    }
  }
  cluster_sync();  // all shares are in place, and no CTA is written to after it
}

// COOP: the nparts CTAs of a tile are one thread-block cluster and share phases A and B.
template <int NPc, int NVc, bool COOP>
__device__ void stage_tile(const StageArgs& A, const TubeDev& T, int x0, int part, int nparts, StageSmem& sm) {
  constexpr bool MONO = NVc <= NV_MONO;
  const int tid = threadIdx.x, c = tid % GW, g = tid / GW;
  const double* tab = A.tab + T.tab;
  const int Qp = T.Qp, Qxi = T.Qxi, Nx = T.Nx, ld = T.ld;
  const double* Fin = A.Fin + T.off;
  const double* Fn = A.Fn + T.off;
  double* Fout = A.Fout + T.off;
  const int x = x0 + c;
  const bool cell = (c < TX) && (x < Nx);
  for (int k = tid; k < RW; k += NT) sm.src[k] = map_cell(x0 - HALO + k, Nx, T.bc, ld);
  if (tid == 0) {
    sm.cst[0] = 1.0;
    sm.cst[1] = 1.0 / 6.0;
    sm.cst[2] = A.a;
    sm.cst[3] = A.b;
    sm.cst[4] = -0.0;
  }
  __syncthreads();

  if (COOP && T.collide) {
    cluster_coeffs<NPc, NVc>(A, T, x0, part, nparts, sm);
  } else if (T.collide) {
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
    const double one = *const_cast<const volatile double*>(&sm.cst[0]);
    if (cell) {
      for (int jb = g; jb < hq; jb += NG) {
        const int jf = Qxi - 1 - jb;
        const double xi = tab[TAB_XI + jf], xi2 = tab[tab_xi2(Qp, Qxi) + jf];
#pragma unroll
        for (int i = 0; i < QP_MAX; ++i) {
          if (i < Qp) {
            const double ff = __ldg(Fin + (size_t)(i * Qxi + jf) * ld + x);
            const double fb = __ldg(Fin + (size_t)(i * Qxi + jb) * ld + x);
            const double sum = add_r(fb, ff, one), dif = fma(-fb, one, ff);
            S[3 * i] = add_r(sum, S[3 * i], one);
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
    if (g == 0) cell_phase<NPc, NVc>(A, T, tab, cell, c, sm);
    __syncthreads();
    build_rows<NPc, NVc>(tab, Qp, sm.u.a.coef, sm.B);
    if constexpr (MONO) {
      if (c < TX && g < Qp) legendre_to_monomial<NVc>(&sm.B[g * (NVc + 1)][c], GW);
    }
    __syncthreads();  // the coefficients are ready, the union is free
  }

  // C. advection + collision + Runge-Kutta combination. The work unit of a 64-thread group is a mirror pair of
  //    directions (j, Qxi - 1 - j) of one radial node, both rows at once: the row with the wind toward -x is held in
  //    reversed order, so that every step of the limiter is the same packed operation on both rows. The even and odd
  //    parts of the equilibrium in xi, summed once, give both rows' equilibria. The xi = 0 node of an odd Qxi is a
  //    unit of its own. Groups synchronise with named barriers only, three per unit.
  const double* cxi_tab = tab + tab_cxi(Qxi) + A.stage * Qxi;
  double* d1f = sm.u.c.d1[g][0];
  double* d1r = sm.u.c.d1[g][1];
  float4* dd = sm.u.c.dd[g];
  float4* svb = sm.u.c.sv[g][0];
  float4* svc = sm.u.c.sv[g][1];
  float2* phf = sm.u.c.phi[g][0];
  float2* phr = sm.u.c.phi[g][1];
  const volatile double* cst = sm.cst;
  const rlbdev::F2 nz = rlbdev::minus_zero2();
  const float2* epsf = reinterpret_cast<const float2*>(tab + tab_epsf(Qp, Qxi));
  const int hq = Qxi / 2, upr = hq + (Qxi & 1), U = Qp * upr;
  const int u_end = (part + 1) * U / nparts;
  auto up = [](float4 q) { return rlbdev::DF2{rlbdev::f2(q.x, q.y), rlbdev::f2(q.z, q.w)}; };
  auto down = [](rlbdev::DF2 q) {
    return make_float4(rlbdev::lo_of(q.hi), rlbdev::hi_of(q.hi), rlbdev::lo_of(q.lo), rlbdev::hi_of(q.lo));
  };
  for (int u = part * U / nparts + g; u < u_end; u += NG) {
    const int i = u / upr, jb = u - i * upr;
    if (jb == hq) {  // the xi = 0 node: no advection
      if (!cell) continue;
      const size_t o = (size_t)(i * Qxi + hq) * ld + x;
      const double F = __ldg(Fin + o);
      double out = A.stage != 0 ? fma(A.a, __ldg(Fn + o), A.b * F) : F;
      if (T.collide) {
        const double* pw = tab + TAB_XI + Qxi + hq * (NV_MAX + 1);
        double E;
        if constexpr (MONO) {
          E = sm.B[i * (NVc + 1)][c] * pw[0];
        } else {
          E = 0.0;
#pragma unroll
          for (int k = 0; k <= NVc; k += 2) E = fma(sm.B[i * (NVc + 1) + k][c], pw[k], E);
        }
        out = fma(sm.rate[0][c], E - F, out);
      }
      Fout[o] = out;
      continue;
    }
    const int jf = Qxi - 1 - jb, sf = i * Qxi + jf, sb = i * Qxi + jb;
    // stage both rows as first differences in wind order, in FP64 and split into double-float: difference k lies
    // between positions k and k + 1, position p = cell x0 - 3 + p, or x0 + TX + 2 - p in the reversed row. Each lane
    // loads position c + 1; position c comes from the lane below (the first lane of each warp loads it)
    rlbdev::DF2 e1;
    {
      const double* rf = Fin + (size_t)sf * ld;
      const double* rb = Fin + (size_t)sb * ld;
      const double vf = __ldg(rf + sm.src[c + 1]), vr = __ldg(rb + sm.src[RW - 2 - c]);
      double pf = __shfl_up_sync(0xffffffffu, vf, 1), pr = __shfl_up_sync(0xffffffffu, vr, 1);
      if ((c & 31) == 0) {
        pf = __ldg(rf + sm.src[c]);
        pr = __ldg(rb + sm.src[RW - 1 - c]);
      }
      const double one = cst[0];
      const double df = fma(-pf, one, vf), dr = fma(-pr, one, vr);
      d1f[c] = df;
      d1r[c] = dr;
      const rlbdev::DF qf = rlbdev::df_split(df), qr = rlbdev::df_split(dr);
      dd[c] = make_float4(qf.hi, qr.hi, qf.lo, qr.lo);
      e1 = {rlbdev::f2(qf.hi, qr.hi), rlbdev::f2(qf.lo, qr.lo)};
    }
    // the cell's own values and Runge-Kutta inputs, loaded now so that their latency hides behind the limiter
    double Ff = 0.0, Fb = 0.0, nf = 0.0, nb = 0.0;
    if (cell) {
      Ff = __ldg(Fin + (size_t)sf * ld + x);
      Fb = __ldg(Fin + (size_t)sb * ld + x);
      if (A.stage != 0) {
        nf = __ldg(Fn + (size_t)sf * ld + x);
        nb = __ldg(Fn + (size_t)sb * ld + x);
      }
    }
    const float2 ee = epsf[sf];
    group_sync(g);
    // pairs: lane c owns the pair of differences (c, c + 1)
    const int c1 = min(c + 1, GW - 1);
    const rlbdev::DF2 e2 = up(dd[c1]);
    rlbdev::DF2 vA, vB, vC;
    rlbdev::weno5_pair_df2(e1, e2, rlbdev::f2(-ee.x), rlbdev::f2(ee.y), nz, vA, vB, vC);
    svb[c] = down(vB);
    svc[c] = down(vC);
    group_sync(g);
    // interfaces: lane c owns interface c (between cells x0 + c - 1 and x0 + c, or x0 + TX - c and x0 + TX - 1 - c in
    // the reversed row); its stencils' differences are c .. c + 3
    double Df = 0.0, Dr = 0.0;
    rlbdev::DF2 G = {rlbdev::f2(0.0f), rlbdev::f2(0.0f)};
    if (c <= TX) {
      G = rlbdev::weno5_combine6_df2(vA, up(svb[c + 1]), up(svc[c + 2]), e1, e2, up(dd[c + 2]), up(dd[c + 3]),
                                     nz);
      phf[c] = make_float2(rlbdev::lo_of(G.hi), rlbdev::lo_of(G.lo));
      phr[c] = make_float2(rlbdev::hi_of(G.hi), rlbdev::hi_of(G.lo));
      if (c < TX) {
        Df = d1f[c + 2];
        Dr = d1r[TX + 1 - c];
      }
    }
    group_sync(g);
    if (cell) {
      // flux differences: D + (6 G - 6 G') / 6, the difference of the corrections taken in double-float. The cell is
      // number c of its row and number TX - 1 - c of the reversed one
      const float2 g1f = phf[c + 1], g1r = phr[TX - c], g0r = phr[TX - 1 - c];
      const rlbdev::DF2 dG =
          rlbdev::df2_minus({rlbdev::f2(g1f.x, g1r.x), rlbdev::f2(g1f.y, g1r.y)},
                            {rlbdev::f2(rlbdev::lo_of(G.hi), g0r.x), rlbdev::f2(rlbdev::lo_of(G.lo), g0r.y)});
      const double sixth = cst[1], cxi = cxi_tab[jf];
      const double phi_f = fma(rlbdev::df_join(rlbdev::lo_of(dG.hi), rlbdev::lo_of(dG.lo)), sixth, Df);
      const double phi_b = fma(rlbdev::df_join(rlbdev::hi_of(dG.hi), rlbdev::hi_of(dG.lo)), sixth, Dr);
      double of = Ff, ob = Fb;
      if (A.stage != 0) {  // a = 0 and b = 1 in the first stage
        const double a = cst[2], b = cst[3], zero = cst[4];
        of = fma(a, nf, fma(b, Ff, zero));
        ob = fma(a, nb, fma(b, Fb, zero));
      }
      of = fma(-cxi, phi_f, of);  // - b dt |xi|/dx (Phi - Phi'), along each row's wind
      ob = fma(-cxi, phi_b, ob);
      if (T.collide) {
        const double xi = tab[TAB_XI + jf];
        const double* pw = tab + TAB_XI + Qxi + jf * (NV_MAX + 1);
        const double(*Bi)[GW] = &sm.B[i * (NVc + 1)];
        double cf, cb;  // F^eq - F
        if constexpr (MONO) {
          const double z = tab[tab_xi2(Qp, Qxi) + jf], w = pw[0];
          double E = Bi[NVc - NVc % 2][c], O = Bi[NVc - 1 + NVc % 2][c];
#pragma unroll
          for (int k = NVc - NVc % 2 - 2; k >= 0; k -= 2) E = fma(E, z, Bi[k][c]);
#pragma unroll
          for (int k = NVc - 3 + NVc % 2; k >= 1; k -= 2) O = fma(O, z, Bi[k][c]);
          cf = fma(w, fma(xi, O, E), -Ff);
          cb = fma(w, fma(-xi, O, E), -Fb);
        } else {
          double E = 0.0, O = 0.0;
#pragma unroll
          for (int k = 0; k <= NVc; ++k) {
            if (k % 2 == 0)
              E = fma(Bi[k][c], pw[k], E);
            else
              O = fma(Bi[k][c], pw[k], O);
          }
          cf = (E + O) - Ff;
          cb = (E - O) - Fb;
        }
        const double r0 = sm.rate[0][c], r1 = sm.rate[1][c];
        of = fma(fma(-r1, xi, r0), cf, of);  // + b dt gamma (1 - beta xi)/tau (F^eq - F)
        ob = fma(fma(r1, xi, r0), cb, ob);
      }
      Fout[(size_t)sf * ld + x] = of;
      Fout[(size_t)sb * ld + x] = ob;
    }
  }
}

// What bounds it: the FP64 pipe (89 % busy on the stress tube, 14.2 FP64 operations per node, 35 % of the issue
// slots). Measured on GB300, FP64 stress tube (2^20 cells x 384 velocities, half of it moving), ms per step: 46.0 with
// one row at a time in scalar double-float and Legendre-basis equilibria, 37.1 with both rows of a mirror pair packed,
// register operands and Horner equilibria, 34.8 once no conversion instruction was left in the rows (df_split,
// df_join). The relaxation-time sweep: 3.62, 2.89, 2.67. 80 registers for 3 CTAs per SM: two CTAs with 128 registers ran
// 8 % slower on the stress tube, four with 64 registers 1 % faster there and 3 % slower on the sweep.
// SCHED is the launch's schedule (compile time, so that the one-CTA-per-tile kernel carries no tile loop);
// SCHED_CLUSTER: one CTA per item, the items of a tile being one thread-block cluster.
constexpr int SCHED_CLUSTER = 3;
template <int SCHED>
__global__ void __launch_bounds__(NT, 3) rlb_stage_kernel(StageArgs A) {
  extern __shared__ __align__(16) unsigned char stage_smem_raw[];
  StageSmem& sm = *reinterpret_cast<StageSmem*>(stage_smem_raw);
  const int K = A.split > 1 ? A.split : 1;
  for_each_tile(A.ntiles * K, SCHED == SCHED_CLUSTER ? 0 : SCHED, A.counter, [&](int item) {
    const int t = item / K, part = item - t * K;
    const int2 tl = A.tiles[t];
    const TubeDev T = A.tubes[tl.x];
    if (T.Np == 2 && T.Nv == 5)
      stage_tile<2, 5, SCHED == SCHED_CLUSTER>(A, T, tl.y, part, K, sm);
    else
      stage_tile<NP_MAX, NV_MAX, SCHED == SCHED_CLUSTER>(A, T, tl.y, part, K, sm);
  });
}
