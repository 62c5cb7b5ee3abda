// Adjoint (reverse mode) of the FP64 stage kernel, and of the initial equilibrium. Included by rlb.cu inside
// its anonymous namespace, after the forward kernels (it uses their helpers).
//
// One forward stage maps F_in to F_out = a F^n + b (F_in + dt L(F_in)) with
//   L_s(x) = -(xi_j/dx) (Phi_s(x+1/2) - Phi_s(x-1/2)) + r_s(x) (F^eq_s(x) - F_s(x)),  r_s = gamma (1 - beta xi_j)/tau
// (Eq. (Boltz) with WENO5 interface values Phi and the Anderson-Witting collision; F^eq from Eq. (feqtrunc)
// with n, T, beta from the Landau frame of the moments of F_in). Given mu = dL/dF_out, the adjoint stage
// produces b (mu + dt J^T mu) for F_in, a mu for F^n and b dt sum mu dL/dlog(tau) for the relaxation time:
//   advection: psi_X = (xi/dx)(mu(X) - mu(X-1)) for the interface X between cells X-1 and X, and
//              (J^T mu)(y) += sum_X psi_X dPhi_X/dF(y) over the five-cell stencils that contain y (ghost
//              cells of the open boundary pass their share to the edge cell, periodic ones wrap);
//   collision: -r_s mu_s, plus sum_a c_a(s) gM_a with c = (pbar, pbar xi, pbar^2, pbar^2 xi, pbar^2 xi^2)
//              the moment weights and gM = d/dM [sum_s mu_s r_s (F^eq_s - F_s)] at fixed F, carried from
//              (n, T, beta) back through the Landau solve;
//   tau:       d/dlog(tau) of b dt r_s (F^eq_s - F_s) is -b dt r_s (F^eq_s - F_s).
// The equilibrium's parameter derivatives use B[i][k] = n w^p_i/4 sum_q K[i][q] T^(q-1) gamma^-(q+2)
// hhat_{q+2,k}(beta) and d hhat_{m,k}/d beta = m (k/(2k-1) hhat_{m+1,k-1} + (k+1)/(2k+3) hhat_{m+1,k+1}), the
// projection of m xi (1 - beta xi)^-(m+1).
//
// One adjoint stage is two launches. rlb_adjoint_cell_kernel reduces each cell's rows to what the collision term
// needs per cell (the rate, its beta multiple and gM); rlb_adjoint_kernel walks the rows. An adjoint tile has TXA =
// 60 cells, so that the TXA + 4 interfaces whose stencils reach its cells fit the 64 lanes of a velocity group.

constexpr int TXA = GW - 4;    // cells per adjoint tile
constexpr int AWD = TXA + 7;   // first differences F(k) - F(k - 1), k = x0-3 .. x0+TXA+3
constexpr int AWU = TXA + 6;   // staged adjoint positions x0-3 .. x0+TXA+2
constexpr int PC = 16;         // cells per CTA of the per-cell kernel
constexpr int NCELLV = 7;      // per-cell values: b dt r0, b dt r0 beta, b dt gM[5]

struct AdjArgs {
  const TubeDev* tubes;
  const int2* tiles;   // adjoint tiles (tube, first cell) of TXA cells
  const int2* ctiles;  // per-cell kernel: tiles of PC cells
  const double* Fin;   // forward stage input (read with halo)
  const double* mu;    // adjoint of the stage output (read with halo)
  double* out;         // adjoint of the stage input (mode 2, 1), or of F^n (mode 0)
  double* acc;         // adjoint accumulated for F^n over the stages of one step
  double* cellv;       // [NCELLV][nxtot], written by the per-cell kernel
  long long nxtot;
  const double* tab;
  int* flag;
  double* dlt;         // per PC-cell tile: accumulators of dL/dlog(tau)
  double a, b;         // the forward stage's Shu-Osher coefficients
  int mode;            // 2: out = b(mu + dt J^T mu), acc = a mu; 1: the same with acc += a mu;
                       // 0: out = acc + b(mu + dt J^T mu)
  int split;           // CTAs per tile: CTA k of a tile writes velocity rows [k Q / split, (k + 1) Q / split)
};

// Legendre coefficients and their beta derivatives (m = 2 .. Np+2, k <= Nv) of the tile's cells
struct AdjCoef {
  double hh[NP_MAX + 1][NV_MAX + 1][GW];
  double dh[NP_MAX + 1][NV_MAX + 1][GW];
};

// hhat and d hhat/d beta of the tile's cells, one thread per cell; cells with ok == 0 keep zeros. Ends with a barrier.
template <int NPc, int NVc>
__device__ void tile_coeffs_d(const double* cellv /* n, T, beta: [3][GW] */, int* ok, AdjCoef& co, int* flag) {
  const int c = threadIdx.x % GW, g = threadIdx.x / GW;
  if (g == 0 && c < TXA) {
    const double beta = cellv[2 * GW + c];
    if (ok[c] && !(fabs(beta) <= beta_limit_d(NPc))) {
      ok[c] = 0;
      atomicOr(flag, 1);
    }
    if (ok[c]) {
      double h[NPc + 2][NVc + 2];
      const double g1 = fma(-beta, beta, 1.0), u = 1.0 / g1;
      legendre_coeffs<NPc + 2, NVc + 1>(beta, beta * beta, g1, h);
      double f = u;  // gamma^2(m-1) / (m-1)! at m = 2
#pragma unroll
      for (int q = 0; q <= NPc; ++q) {
        const double fd = f * u;  // m times the factor of m + 1 = q + 3
#pragma unroll
        for (int k = 0; k <= NVc; ++k) {
          co.hh[q][k][c] = f * h[q][k];
          double d = (double)(k + 1) / (double)(2 * k + 3) * h[q + 1][k + 1];
          if (k > 0) d = fma((double)k / (double)(2 * k - 1), h[q + 1][k - 1], d);
          co.dh[q][k][c] = fd * d;
        }
        f *= u / (double)(q + 2);
      }
    } else {
#pragma unroll
      for (int m = 0; m <= NPc; ++m)
#pragma unroll
        for (int k = 0; k <= NVc; ++k) co.hh[m][k][c] = co.dh[m][k][c] = 0.0;
    }
  }
  __syncthreads();
}

// Derivatives of sum_{i,k} B[i][k](n, T, beta) Lam[i][k] with respect to n, T and beta at one cell.
template <int NPc, int NVc>
__device__ void eq_param_grads(const double* tab, int Qp, double n, double T, double beta, const AdjCoef& co,
                               int c, const double (*Lam)[GW] /* [i (NV_MAX+1) + k][GW] */, double& gn,
                               double& gT, double& gb) {
  const double g2 = 1.0 / (1.0 - beta * beta);  // gamma^2
  const double ig = sqrt(1.0 - beta * beta);    // 1/gamma
  double uq = ig * ig / T;                      // T^(q-1) gamma^-(q+2) at q = 0
  double an = 0.0, aT = 0.0, ab = 0.0;
#pragma unroll
  for (int q = 0; q <= NPc; ++q) {
    double sn = 0.0, sb = 0.0;
#pragma unroll
    for (int k = 0; k <= NVc; ++k) {
      double H = 0.0;  // sum_i w_i K[i][q] Lam[i][k]
      for (int i = 0; i < Qp; ++i)
        H = fma(tab[TAB_WP + i] * tab[TAB_K + i * (NP_MAX + 1) + q], Lam[i * (NV_MAX + 1) + k][c], H);
      const double hq = co.hh[q][k][c], dq = co.dh[q][k][c];
      sn = fma(hq, H, sn);
      sb = fma(fma(-(q + 2) * beta * g2, hq, dq), H, sb);
    }
    an = fma(uq, sn, an);
    aT = fma((q - 1) * uq, sn, aT);
    ab = fma(uq, sb, ab);
    uq *= T * ig;
  }
  const double q4 = 0.25 * n;
  gn = 0.25 * an;
  gT = q4 * aT / T;
  gb = q4 * ab;
}

// What the forward's Landau solve keeps for the way back.
struct LandauRev {
  double e, beta, n, T, gam, u;  // u = gamma^2
  double iden, in3, isq;         // 1/(Txx + e), 1/(3n), 1/sqrt((T00 + Txx)^2 - 4 T0x^2)
};

// As landau_frame, keeping the reciprocals; false if non-physical.
__device__ __forceinline__ bool landau_keep(const double mom[5], LandauRev& L) {
  const double A = mom[2] + mom[4], B2 = 2.0 * mom[3];
  const double disc = fma(A, A, -(B2 * B2));
  L.isq = rlbdev::rsqrt_any(disc);
  L.e = 0.5 * ((mom[2] - mom[4]) + rlbdev::sqrt_nr(disc));
  L.iden = rlbdev::rcp_nr(mom[4] + L.e);
  L.beta = rlbdev::div_nr(mom[3], mom[4] + L.e);
  const double g1 = fma(-L.beta, L.beta, 1.0);
  L.gam = rlbdev::rsqrt_nr(g1);
  L.u = rlbdev::rcp_nr(g1);
  L.n = L.gam * fma(-L.beta, mom[1], mom[0]);
  L.in3 = rlbdev::rcp_nr(3.0 * L.n);
  L.T = rlbdev::div_nr(L.e, 3.0 * L.n);
  return disc > 0.0 && L.e > 0.0 && fabs(L.beta) < 1.0 && L.n > 0.0 && L.T > 0.0;
}

// Landau solve backwards: adjoints (gn, gT, gbeta) of n, T, beta to the adjoints of the five moments.
__device__ __forceinline__ void landau_reverse(const double mom[5], const LandauRev& L, double gn, double gT, double gb,
                                               double gM[5]) {
  // T = e / (3n)
  double ge = gT * L.in3;
  gn = fma(-3.0 * gT, L.T * L.in3, gn);
  // n = gamma (N0 - beta Nx)
  gM[0] = gn * L.gam;
  gM[1] = -gM[0] * L.beta;
  gb = fma(gn, L.u * L.beta * L.n - L.gam * mom[1], gb);
  // beta = T0x / (Txx + e)
  gM[3] = gb * L.iden;
  const double gd = -gM[3] * L.beta;
  ge += gd;
  // e = ((T00 - Txx) + sqrt((T00 + Txx)^2 - 4 T0x^2)) / 2
  const double As = (mom[2] + mom[4]) * L.isq, h = 0.5 * ge;
  gM[2] = fma(h, As, h);
  gM[4] = gd + fma(h, As, -h);
  gM[3] = fma(-2.0 * ge, mom[3] * L.isq, gM[3]);
}

// Coefficients of the per-cell kernel's steps in m and of xi P_k, by order (filled at compile time).
struct LegTab {
  double lead[NP_MAX + 1][NV_MAX + 2], own[NP_MAX + 1][NV_MAX + 2];  // power m = q + 2 to m + 1
  double lo[NV_MAX + 1], hi[NV_MAX + 1];  // xi f: k/(2k-1) f_{k-1} + (k+1)/(2k+3) f_{k+1}
};
constexpr LegTab make_leg_tab() {
  LegTab t{};
  for (int q = 0; q <= NP_MAX; ++q)
    for (int k = 0; k <= NV_MAX + 1; ++k) {
      t.lead[q][k] = leg_lead(q + 2, k);
      t.own[q][k] = leg_own(q + 2, k);
    }
  for (int k = 0; k <= NV_MAX; ++k) {
    t.lo[k] = k == 0 ? 0.0 : (double)k / (double)(2 * k - 1);
    t.hi[k] = (double)(k + 1) / (double)(2 * k + 3);
  }
  return t;
}
__constant__ LegTab c_leg = make_leg_tab();

struct AdjCellSmem {
  double red[NT / PC][5][PC];             // partial sums of the slices
  double h[NP_MAX + 2][NV_MAX + 2][PC];   // Legendre coefficients (legendre_coeffs), powers 2 .. Np + 3
  double ga[NP_MAX + 1][NV_MAX + 1][PC];  // g_q h_{q,k}
  double gb[NP_MAX + 1][NV_MAX + 1][PC];  // and its beta derivative at fixed n, T
  double B[3][NBC][PC];                   // B[i][k] and its T and beta derivatives
  double cell[5][PC];                     // beta, g0 = n/T, T gamma, gamma^2, 1/T
  double rate[2][PC];                     // r0, r0 beta
  double mom[5][PC];
  double cst[2];                          // 1, -0
  int ok[PC];
};

// Per-cell part of an adjoint stage, PC cells per CTA: thread (c, slice) takes radial node i = slice / ns and every
// ns-th mirror pair of its directions, ns = 16 / Qp.
//  1. moments of the stage input; Landau frame and the first Legendre coefficients (one thread per cell); the further
//     powers, their beta derivatives and B[i][k], dB/dT, dB/dbeta with a thread per order and cell (a serial FP64
//     operation takes 64 cycles of its scheduler's FP64 unit whether one lane or 32 take part, so the per-cell work is
//     spread over the CTA);
//  2. Lam[i][k] = sum_j mu_ij r_ij w^xi_j P_k(xi_j) and S0 = sum mu (F^eq - F), S1 = sum mu xi (F^eq - F) over the
//     slice, Lam at once contracted with B, dB/dT and dB/dbeta (dB/dn = B/n);
//  3. the sums of the slices, then back through the Landau frame.
// As a part of each CTA of the row kernel it was repeated `split` times on small handles. On GB300 one adjoint stage of
// the 2048-cell, 96-velocity inverse problem took 177 us; now this kernel takes 29 (its serial per-cell steps bound
// it) and the rows 48. 16 tubes of about 1590 cells and 72 velocities: 783 us, now 156 + 363.
template <int NPc, int NVc>
__device__ void adjoint_cells(const AdjArgs& A, const TubeDev& T, int tile, int x0, AdjCellSmem& sm) {
  constexpr int NS = NT / PC;
  const int tid = threadIdx.x, c = tid % PC, sl = tid / PC;
  const double* tab = A.tab + T.tab;
  const int Qp = T.Qp, Qxi = T.Qxi, Nx = T.Nx, ld = T.ld, hq = Qxi / 2;
  const double* Fin = A.Fin + T.off;
  const double* mu = A.mu + T.off;
  const int x = x0 + c;
  const bool cell = x < Nx;
  const int ns = NS / Qp, i = sl / ns, js = sl - i * ns;
  const bool on = cell && i < Qp;
  if (tid == 0) {
    sm.cst[0] = 1.0;
    sm.cst[1] = -0.0;
  }
  __syncthreads();
  const double one = *const_cast<const volatile double*>(&sm.cst[0]);
  const double nz = *const_cast<const volatile double*>(&sm.cst[1]);
  {
    double S0 = 0.0, S1 = 0.0, S2 = 0.0;
    if (on) {
      for (int jb = js; jb < hq; jb += ns) {
        const int jf = Qxi - 1 - jb;
        const double ff = __ldg(Fin + (size_t)(i * Qxi + jf) * ld + x), fb = __ldg(Fin + (size_t)(i * Qxi + jb) * ld + x);
        const double s = fma(ff, one, fb);
        S0 = fma(s, one, S0);
        S1 = fma(fma(-fb, one, ff), tab[TAB_XI + jf], S1);
        S2 = fma(s, tab[tab_xi2(Qp, Qxi) + jf], S2);
      }
      if ((Qxi & 1) && js == 0) S0 += __ldg(Fin + (size_t)(i * Qxi + hq) * ld + x);
    }
    sm.red[sl][0][c] = S0;
    sm.red[sl][1][c] = S1;
    sm.red[sl][2][c] = S2;
  }
  __syncthreads();
  // the radial sums of the slices, one thread per node, sum and cell
  if (sl < 3 * Qp) {
    const int r = sl / 3, q = sl - 3 * r;
    double s = 0.0;
    for (int k = 0; k < ns; ++k) s = fma(sm.red[r * ns + k][q][c], one, s);
    sm.B[0][sl][c] = s;
  }
  __syncthreads();
  LandauRev L{};
  bool ok = false;
  if (tid < PC) {
    double mom[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int r = 0; r < Qp; ++r) {
      const double p1 = tab[TAB_PBAR + r], p2 = tab[TAB_PBAR2 + r];
      const double S0 = sm.B[0][3 * r][c], S1 = sm.B[0][3 * r + 1][c], S2 = sm.B[0][3 * r + 2][c];
      mom[0] = fma(p1, S0, mom[0]);
      mom[1] = fma(p1, S1, mom[1]);
      mom[2] = fma(p2, S0, mom[2]);
      mom[3] = fma(p2, S1, mom[3]);
      mom[4] = fma(p2, S2, mom[4]);
    }
    ok = cell && landau_keep(mom, L) && fabs(L.beta) <= beta_limit_d(NPc);
    if (cell && !ok) atomicOr(A.flag, 1);
    if (ok) {
      double h[NVc + 2];
      legendre_first<NVc + 1>(L.beta, L.beta * L.beta, fma(-L.beta, L.beta, 1.0), h);
#pragma unroll
      for (int k = 0; k <= NVc + 1; ++k) sm.h[0][k][c] = h[k];
    }
    const double iT = ok ? 3.0 * L.n * rlbdev::rcp_nr(L.e) : 0.0;
    const double r0 = ok ? T.inv_tau * L.gam : 0.0;
    sm.cell[0][c] = ok ? L.beta : 0.0;
    sm.cell[1][c] = ok ? L.n * iT : 0.0;
    sm.cell[2][c] = ok ? L.T * L.gam : 0.0;
    sm.cell[3][c] = ok ? L.u : 0.0;
    sm.cell[4][c] = iT;
    sm.rate[0][c] = r0;
    sm.rate[1][c] = ok ? r0 * L.beta : 0.0;
    sm.ok[c] = ok ? 1 : 0;
#pragma unroll
    for (int f = 0; f < 5; ++f) sm.mom[f][c] = mom[f];
  }
  __syncthreads();
  const double beta = sm.cell[0][c];
#pragma unroll 1
  for (int q = 0; q <= NPc; ++q) {  // power q + 2 to q + 3
    if (sl <= NVc + 1 && sm.ok[c])
      sm.h[q + 1][sl][c] =
          fma(c_leg.lead[q][sl], beta * sm.h[q][sl == 0 ? 1 : sl - 1][c], c_leg.own[q][sl] * sm.h[q][sl][c]);
    __syncthreads();
  }
  if (sl <= NVc) {
    double g = sm.cell[1][c];
    const double u = sm.cell[3][c], tg = sm.cell[2][c];
#pragma unroll
    for (int q = 0; q <= NPc; ++q) {
      double a = 0.0, d = 0.0;
      if (sm.ok[c]) {
        const double h = sm.h[q][sl][c];
        d = c_leg.hi[sl] * sm.h[q + 1][sl + 1][c];
        if (sl > 0) d = fma(c_leg.lo[sl], sm.h[q + 1][sl - 1][c], d);
        const double gq = g * tab[TAB_KCA + q];
        a = gq * h;
        d = (gq * u) * fma(-(double)(q + 2) * beta, h, d);
      }
      sm.ga[q][sl][c] = a;
      sm.gb[q][sl][c] = d;
      g *= tg;
    }
  }
  __syncthreads();
  for (int w = sl; w < Qp * (NVc + 1); w += NS) {
    const int r = w / (NVc + 1), k = w - r * (NVc + 1);
    double B = 0.0, BT = 0.0, Bb = 0.0;
#pragma unroll
    for (int q = 0; q <= NPc; ++q) {
      const double K = tab[TAB_KWA + r * (NP_MAX + 1) + q], t = K * sm.ga[q][k][c];
      B += t;
      BT = fma((double)(q - 1), t, BT);
      Bb = fma(K, sm.gb[q][k][c], Bb);
    }
    sm.B[0][w][c] = B;
    sm.B[1][w][c] = BT * sm.cell[4][c];
    sm.B[2][w][c] = Bb;
  }
  __syncthreads();
  {
    double S0 = 0.0, S1 = 0.0, lam[NVc + 1];
#pragma unroll
    for (int k = 0; k <= NVc; ++k) lam[k] = 0.0;
    if (on) {
      const int o = i * (NVc + 1);
      double B[NVc + 1];
#pragma unroll
      for (int k = 0; k <= NVc; ++k) B[k] = sm.B[0][o + k][c];
      const double r0 = sm.rate[0][c], r1 = sm.rate[1][c];
      for (int jb = js; jb < hq; jb += ns) {
        const int jf = Qxi - 1 - jb;
        const size_t of = (size_t)(i * Qxi + jf) * ld + x, ob = (size_t)(i * Qxi + jb) * ld + x;
        const double ff = __ldg(Fin + of), fb = __ldg(Fin + ob), mf = __ldg(mu + of), mb = __ldg(mu + ob);
        const double xi = tab[TAB_XI + jf];
        const double* pw = tab + TAB_XI + Qxi + jf * (NV_MAX + 1);
        double E = 0.0, O = 0.0;
#pragma unroll
        for (int k = 0; k <= NVc; ++k) {
          if (k % 2 == 0)
            E = fma(B[k], pw[k], E);
          else
            O = fma(B[k], pw[k], O);
        }
        const double df = fma(mf, fma(-ff, one, fma(E, one, O)), nz), db = fma(mb, fma(-fb, one, fma(-O, one, E)), nz);
        S0 = fma(fma(df, one, db), one, S0);
        S1 = fma(fma(-db, one, df), xi, S1);
        const double t = fma(r1, xi, nz), me = fma(mf, one, mb), mo = fma(-mb, one, mf);
        const double le = fma(-t, mo, fma(r0, me, nz)), lo = fma(-t, me, fma(r0, mo, nz));
#pragma unroll
        for (int k = 0; k <= NVc; ++k) lam[k] = fma(k % 2 == 0 ? le : lo, pw[k], lam[k]);
      }
      if ((Qxi & 1) && js == 0) {
        const size_t oc = (size_t)(i * Qxi + hq) * ld + x;
        const double* pw = tab + TAB_XI + Qxi + hq * (NV_MAX + 1);
        const double m = __ldg(mu + oc);
        double E = 0.0;
#pragma unroll
        for (int k = 0; k <= NVc; k += 2) E = fma(B[k], pw[k], E);
        S0 = fma(m, E - __ldg(Fin + oc), S0);
#pragma unroll
        for (int k = 0; k <= NVc; k += 2) lam[k] = fma(m * r0, pw[k], lam[k]);
      }
    }
    double pn = 0.0, pT = 0.0, pb = 0.0;
    if (on) {
#pragma unroll
      for (int k = 0; k <= NVc; ++k) {
        pn = fma(lam[k], sm.B[0][i * (NVc + 1) + k][c], pn);
        pT = fma(lam[k], sm.B[1][i * (NVc + 1) + k][c], pT);
        pb = fma(lam[k], sm.B[2][i * (NVc + 1) + k][c], pb);
      }
    }
    sm.red[sl][0][c] = pn;
    sm.red[sl][1][c] = pT;
    sm.red[sl][2][c] = pb;
    sm.red[sl][3][c] = S0;
    sm.red[sl][4][c] = S1;
  }
  __syncthreads();
  if (sl < 5) {
    double s = 0.0;
    for (int k = 0; k < NS; ++k) s = fma(sm.red[k][sl][c], one, s);
    sm.h[0][sl][c] = s;
  }
  __syncthreads();
  if (tid < 32) {
    double dl = 0.0;
    if (tid < PC && cell) {
      double gM[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, r0 = 0.0, r1 = 0.0;
      const double bdt = A.b * T.dt;
      if (ok) {
        const double S0 = sm.h[0][3][c], S1 = sm.h[0][4][c];
        r0 = sm.rate[0][c];
        r1 = sm.rate[1][c];
        // d r_s / d beta = gamma^3 (beta - xi_j) / tau = r0 gamma^2 (beta - xi_j)
        const double gn = sm.h[0][0][c] * (3.0 * L.in3), gT = sm.h[0][1][c];
        const double gb = fma(r0 * L.u, fma(L.beta, S0, -S1), sm.h[0][2][c]);
        double mom[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) mom[f] = sm.mom[f][c];
        landau_reverse(mom, L, gn, gT, gb, gM);
        dl = -bdt * r0 * fma(-L.beta, S1, S0);
      }
      double* o = A.cellv + T.xoff + x;
      o[0] = bdt * r0;
      o[A.nxtot] = bdt * r1;
#pragma unroll
      for (int f = 0; f < 5; ++f) o[(2 + f) * A.nxtot] = bdt * gM[f];
    }
#pragma unroll
    for (int d = PC / 2; d > 0; d >>= 1) dl += __shfl_down_sync(0xffffffffu, dl, d);
    if (tid == 0) A.dlt[tile] += dl;
  }
}

__global__ void __launch_bounds__(NT) rlb_adjoint_cell_kernel(AdjArgs A) {
  extern __shared__ __align__(16) unsigned char adjc_smem_raw[];
  AdjCellSmem& sm = *reinterpret_cast<AdjCellSmem*>(adjc_smem_raw);
  const int2 tl = A.ctiles[blockIdx.x];
  const TubeDev T = A.tubes[tl.x];
  if (!T.collide) return;  // ballistic: the row kernel reads no per-cell values
  if (T.Np == 2 && T.Nv == 5)
    adjoint_cells<2, 5>(A, T, blockIdx.x, tl.y, sm);
  else
    adjoint_cells<NP_MAX, NV_MAX>(A, T, blockIdx.x, tl.y, sm);
}

struct AdjSmem {
  double drow[2][NG][AWD + 1];  // first differences of the staged F rows
  double urow[2][NG][AWU + 1];  // staged adjoint rows
  double P[NG][5][GW];          // psi_X dPhi_X/dF at the five stencil slots (memory order) of interface X
  double mom[3 * QP_MAX][GW];   // per radial node: the moment weights' share, even, xi and xi^2 parts
  double rate[2][GW];           // b dt r0, b dt r0 beta
  double cst[rlbdev::ADJ_CST];  // constants of the rows (grad_constant)
  double b;                     // the forward stage's b (a register operand)
  int srcF[TXA + 8];            // source cell of each F position x0-4 .. x0+TXA+3
  int srcU[AWU + 1];            // source cell of each staged adjoint position, -1: outside the tube (zero)
};

__device__ __forceinline__ int wrap_cell(int p, int Nx) {
  const int r = p % Nx;
  return r < 0 ? r + Nx : r;
}

// What bounds it: the FP64 pipe (92 % busy on a batch that fills the GPU): 100 FP64 operations per node.
__device__ void adjoint_rows(const AdjArgs& A, const TubeDev& T, int x0, int part, int nparts, AdjSmem& sm) {
  const int tid = threadIdx.x, c = tid % GW, g = tid / GW;
  const double* tab = A.tab + T.tab;
  const int Qp = T.Qp, Qxi = T.Qxi, Q = Qp * Qxi, Nx = T.Nx, ld = T.ld;
  const double* Fin = A.Fin + T.off;
  const double* mu = A.mu + T.off;
  double* out = A.out + T.off;
  double* acc = A.acc + T.off;
  const int x = x0 + c;
  const bool cell = (c < TXA) && (x < Nx);
  const bool periodic = T.bc == RLB_BC_PERIODIC;
  for (int k = tid; k < TXA + 8; k += NT) {
    const int p = x0 - 4 + k;
    sm.srcF[k] = periodic ? wrap_cell(p, Nx) : min(max(p, 0), Nx - 1);
  }
  for (int k = tid; k < AWU; k += NT) {
    const int p = x0 - 3 + k;
    sm.srcU[k] = periodic ? wrap_cell(p, Nx) : ((p >= 0 && p < Nx) ? p : -1);
  }
  if (tid < rlbdev::ADJ_CST) {
    sm.cst[tid] = rlbdev::grad_constant(tid);
    if (tid == 0) sm.b = A.b;
  }
  if (T.collide) {
    // the cell's rate, and gM contracted with the moment weights of radial node i = g: pbar (gM0 + xi gM1) +
    // pbar^2 (gM2 + xi gM3 + xi^2 gM4) by powers of xi
    const double* v = A.cellv + T.xoff + x;
    if (g == 0) {
      sm.rate[0][c] = cell ? v[0] : 0.0;
      sm.rate[1][c] = cell ? v[A.nxtot] : 0.0;
    }
    if (g < Qp) {
      double m0 = 0.0, m1 = 0.0, m2 = 0.0;
      if (cell) {
        const double p1 = tab[TAB_PBAR + g], p2 = tab[TAB_PBAR2 + g];
        m0 = fma(p1, v[2 * A.nxtot], p2 * v[4 * A.nxtot]);
        m1 = fma(p1, v[3 * A.nxtot], p2 * v[5 * A.nxtot]);
        m2 = p2 * v[6 * A.nxtot];
      }
      sm.mom[3 * g][c] = m0;
      sm.mom[3 * g + 1][c] = m1;
      sm.mom[3 * g + 2][c] = m2;
    }
  }
  __syncthreads();

  // rows: transposed WENO5 flux differences, collision terms, Runge-Kutta combination
  const double a = A.a, cpsi = A.b * T.dt * (2.0 / 3.0) / T.dx;  // 4/6 of b dt / dx, with weno5_grad's 6/4
  double* P0 = sm.P[g][0];
  int buf = 0;
  const int r_end = (part + 1) * Q / nparts;
  for (int s = part * Q / nparts + g; s < r_end; s += NG, buf ^= 1) {  // uniform over the group
    const int i = s / Qxi, j = s - i * Qxi;
    double* dr = sm.drow[buf][g];
    double* ur = sm.urow[buf][g];
    const volatile double* cst = sm.cst;
    const double one = cst[rlbdev::C_ONE], nz = cst[rlbdev::C_NZ];
    {
      // difference k lies between positions k and k + 1 of srcF; each lane loads position c + 1 and takes position c
      // from the lane below
      const double* fs = Fin + (size_t)s * ld;
      const double v = __ldg(fs + sm.srcF[c + 1]);
      double w = __shfl_up_sync(0xffffffffu, v, 1);
      if ((c & 31) == 0) w = __ldg(fs + sm.srcF[c]);
      dr[c] = fma(-w, one, v);
      if (c < AWD - GW) dr[GW + c] = __ldg(fs + sm.srcF[GW + 1 + c]) - __ldg(fs + sm.srcF[GW + c]);
      const double* us = mu + (size_t)s * ld;
      for (int k = c; k < AWU; k += GW) {
        const int q = sm.srcU[k];
        ur[k] = q >= 0 ? __ldg(us + q) : 0.0;
      }
    }
    const double prev = (cell && A.mode != 2) ? acc[(size_t)s * ld + x] : 0.0;  // needed at the row's end only
    group_sync(g);
    const double xi = tab[TAB_XI + j];
    const bool fwd = 2 * j + 1 > Qxi;  // xi_j > 0, decided without an FP64 comparison
    if (2 * j + 1 != Qxi) {
      // lane c: interface X = x0 - 1 + c (wind toward +x) or x0 - 2 + c (toward -x); its stencil's differences are
      // dr[c .. c+3] in memory order and mu(X), mu(X-1) are ur[c+2], ur[c+1] (resp. ur[c+1], ur[c])
      const int lo = fwd ? c + 1 : c;
      const double psi = fma(fma(xi, cpsi, nz), fma(-ur[lo], one, ur[lo + 1]), nz);
      const double e = tab[tab_eps(Qxi) + s];
      double h[4];
      rlbdev::weno5_grad(dr[fwd ? c : c + 3], dr[fwd ? c + 1 : c + 2], dr[fwd ? c + 2 : c + 1], dr[fwd ? c + 3 : c], e,
                         cst, h);
      P0[(fwd ? 0 : 4) * GW + c] = fma(-psi, h[0], nz);
      P0[(fwd ? 1 : 3) * GW + c] = fma(psi, fma(-h[1], one, h[0]), nz);
      P0[2 * GW + c] = fma(psi, fma(fma(-h[2], one, h[1]), one, cst[rlbdev::C_15]), nz);
      P0[(fwd ? 3 : 1) * GW + c] = fma(psi, fma(-h[3], one, h[2]), nz);
      P0[(fwd ? 4 : 0) * GW + c] = fma(psi, h[3], nz);
    } else {
#pragma unroll
      for (int m = 0; m < 5; ++m) P0[m * GW + c] = 0.0;
    }
    group_sync(g);
    if (cell) {
      // cell y = x0 + c gathers slot m of interface lane c + 4 - m; the open boundary's ghost positions
      // (copies of the edge cells) add theirs to the edge cells
      double w = fma(P0[c + 4], one, P0[GW + c + 3]);
      w = fma(P0[2 * GW + c + 2], one, w);
      w = fma(P0[3 * GW + c + 1], one, w);
      w = fma(P0[4 * GW + c], one, w);
      if (!periodic && (x == 0 || x == Nx - 1)) {
        for (int side = 0; side < 2; ++side) {
          if ((side == 0 && x != 0) || (side == 1 && x != Nx - 1)) continue;
          for (int h = 1; h <= 3; ++h) {
            const int p = side == 0 ? -h : Nx - 1 + h;  // ghost position
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              const int lane = p - x0 + 4 - m;
              if (lane >= 0 && lane < GW) w += P0[m * GW + lane];
            }
          }
        }
      }
      const double m_ = ur[c + 3];
      if (T.collide) {
        w = fma(fma(sm.rate[1][c], xi, -sm.rate[0][c]), m_, w);
        w = fma(fma(sm.mom[3 * i + 2][c], xi, sm.mom[3 * i + 1][c]), xi, fma(sm.mom[3 * i][c], one, w));
      }
      const double val = fma(sm.b, m_, w);
      const size_t o = (size_t)s * ld + x;
      if (A.mode == 0) {
        out[o] = fma(prev, one, val);
      } else {
        out[o] = val;
        acc[o] = fma(a, m_, prev);
      }
    }
  }
}

__global__ void __launch_bounds__(NT, 2) rlb_adjoint_kernel(AdjArgs A) {
  extern __shared__ __align__(16) unsigned char adj_smem_raw[];
  AdjSmem& sm = *reinterpret_cast<AdjSmem*>(adj_smem_raw);
  const int t = blockIdx.x / A.split, part = blockIdx.x - t * A.split;
  const int2 tl = A.tiles[t];
  const TubeDev T = A.tubes[tl.x];
  adjoint_rows(A, T, tl.y, part, A.split, sm);
}

// Seed of the state from the adjoint of the five moments of each cell: dL/dF_s = sum_a c_a(s) dL/dM_a.
// gM: [5][nxtot] (field layout); seed: packed state (rows of Nx cells, tube after tube).
__global__ void __launch_bounds__(NT) rlb_moments_vjp_kernel(const TubeDev* tubes, const int2* tiles,
                                                             const double* tabs, const double* gM,
                                                             long long nxtot, double* seed) {
  const int2 tl = tiles[blockIdx.x];
  const TubeDev T = tubes[tl.x];
  const int c = threadIdx.x % GW, g = threadIdx.x / GW, x = tl.y + c;
  if (c >= TXA || x >= T.Nx) return;
  const double* tab = tabs + T.tab;
  const double* gm = gM + T.xoff + x;
  const double g0 = gm[0], g1 = gm[nxtot], g2 = gm[2 * nxtot], g3 = gm[3 * nxtot], g4 = gm[4 * nxtot];
  for (int s = g; s < T.Qp * T.Qxi; s += NG) {
    const int i = s / T.Qxi, j = s - i * T.Qxi;
    const double xi = tab[TAB_XI + j];
    const double v = tab[TAB_PBAR + i] * fma(xi, g1, g0) + tab[TAB_PBAR2 + i] * fma(xi, fma(xi, g4, g3), g2);
    seed[T.poff + (size_t)s * T.Nx + x] = v;
  }
}

// Adjoint of the Landau frame (e, beta, n) with respect to the moments (N0, Nx, T00, T0x, Txx), for the closed
// form of landau(): with A = T00 + Txx, r = sqrt(A^2 - 4 T0x^2), e = (T00 - Txx + r) / 2, W = Txx + e,
// beta = T0x / W, gamma = (1 - beta^2)^-1/2, n = gamma (N0 - beta Nx). Adds ge de/dM + gb dbeta/dM + gn dn/dM to
// G[5]. Returns false for a non-physical cell (G unchanged).
__device__ bool landau_vjp(const double mom[5], double ge, double gb, double gn, double G[5]) {
  double e, beta, n, Tt;
  if (!landau(mom, e, beta, n, Tt)) return false;
  const double A = mom[2] + mom[4], B = mom[3];
  const double r = sqrt(A * A - 4.0 * B * B);
  if (!(r > 0.0)) return false;
  // de/d(T00, T0x, Txx)
  const double e00 = 0.5 * (1.0 + A / r), e0x = -2.0 * B / r, exx = 0.5 * (A / r - 1.0);
  const double W = mom[4] + e, bW = beta / W;  // beta / W = T0x / W^2
  // dbeta/d(T00, T0x, Txx)
  const double b00 = -bW * e00, b0x = 1.0 / W - bW * e0x, bxx = -bW * (1.0 + exx);
  const double g2 = 1.0 / (1.0 - beta * beta), gam = sqrt(g2);
  // dn/dbeta at fixed (N0, Nx); dn/dN0 = gamma, dn/dNx = -gamma beta
  const double nb = gam * (g2 * beta * (mom[0] - beta * mom[1]) - mom[1]);
  const double gbt = gb + gn * nb;  // total adjoint of beta
  G[0] += gn * gam;
  G[1] -= gn * gam * beta;
  G[2] += ge * e00 + gbt * b00;
  G[3] += ge * e0x + gbt * b0x;
  G[4] += ge * exx + gbt * bxx;
  return true;
}

// Seed of the state from the adjoint of the fields of rlb_moments: dL/dF_s = sum_a c_a(s) G_a, where G_a is
// dL/dM_a plus the share of dL/de, dL/dv and dL/dn carried through the Landau frame of the cell's moments.
// gf: [RLB_NFIELDS][nxtot] (field layout); F: the FP64 state (padded rows) the fields were taken at; seed:
// packed state. A non-physical cell raises the flag and seeds only its moments' share.
__global__ void __launch_bounds__(NT) rlb_fields_vjp_kernel(const TubeDev* tubes, const int2* tiles,
                                                            const double* tabs, const double* F, const double* gf,
                                                            long long nxtot, double* seed, int* flag) {
  __shared__ double Gs[5][GW];
  const int2 tl = tiles[blockIdx.x];
  const TubeDev T = tubes[tl.x];
  const int c = threadIdx.x % GW, g = threadIdx.x / GW, x = tl.y + c;
  const bool cell = c < TXA && x < T.Nx;
  const double* tab = tabs + T.tab;
  if (g == 0) {
    double G[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (cell) {
      const double* f = F + T.off + x;
      double mom[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
      for (int j = 0; j < T.Qxi; ++j) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < T.Qp; ++i) {
          const double v = f[(size_t)(i * T.Qxi + j) * T.ld];
          a = fma(v, tab[TAB_PBAR + i], a);
          b = fma(v, tab[TAB_PBAR2 + i], b);
        }
        const double xi = tab[TAB_XI + j];
        mom[0] += a;
        mom[1] = fma(a, xi, mom[1]);
        mom[2] += b;
        mom[3] = fma(b, xi, mom[3]);
        mom[4] = fma(b * xi, xi, mom[4]);
      }
      const double* gx = gf + T.xoff + x;
#pragma unroll
      for (int a = 0; a < 5; ++a) G[a] = gx[a * nxtot];
      if (!landau_vjp(mom, gx[RLB_F_E * nxtot], gx[RLB_F_V * nxtot], gx[RLB_F_N * nxtot], G)) atomicOr(flag, 1);
    }
#pragma unroll
    for (int a = 0; a < 5; ++a) Gs[a][c] = G[a];
  }
  __syncthreads();
  if (!cell) return;
  const double g0 = Gs[0][c], g1 = Gs[1][c], g2 = Gs[2][c], g3 = Gs[3][c], g4 = Gs[4][c];
  for (int s = g; s < T.Qp * T.Qxi; s += NG) {
    const int i = s / T.Qxi, j = s - i * T.Qxi;
    const double xi = tab[TAB_XI + j];
    const double v = tab[TAB_PBAR + i] * fma(xi, g1, g0) + tab[TAB_PBAR2 + i] * fma(xi, fma(xi, g4, g3), g2);
    seed[T.poff + (size_t)s * T.Nx + x] = v;
  }
}

struct InitVjpSmem {
  AdjCoef co;
  double lam[NBC][GW];
  double cellv[3][GW];  // n, T, beta of the initial state
  double P[GW];
  int ok[GW];
};

// Adjoint of the initial condition F = F^eq(n, T = P/n, beta = v): from dL/dF (packed) to dL/dP, dL/dn,
// dL/dv of each cell (field layout).
template <int NPc, int NVc>
__device__ void init_vjp_tile(const TubeDev& T, const double* tab, int x0, const double* P, const double* n,
                              const double* v, const double* gF, double* gP, double* gn, double* gv, int* flag,
                              InitVjpSmem& sm) {
  const int c = threadIdx.x % GW, g = threadIdx.x / GW, x = x0 + c;
  const bool cell = c < TXA && x < T.Nx;
  const size_t k = (size_t)T.xoff + x;
  if (g == 0) {
    const double P_ = cell ? P[k] : 1.0, n_ = cell ? n[k] : 1.0, v_ = cell ? v[k] : 0.0;
    const bool ok = cell && P_ > 0.0 && n_ > 0.0 && fabs(v_) < 1.0;
    if (cell && !ok) atomicOr(flag, 1);
    sm.P[c] = P_;
    sm.cellv[0][c] = n_;
    sm.cellv[1][c] = P_ / n_;
    sm.cellv[2][c] = ok ? v_ : 0.0;
    sm.ok[c] = ok ? 1 : 0;
  }
  __syncthreads();
  tile_coeffs_d<NPc, NVc>(&sm.cellv[0][0], sm.ok, sm.co, flag);
  // Lam[i][k] = sum_j dL/dF_ij w^xi_j P_k(xi_j), radial row i summed by group i
  if (g < QP_MAX) {
    double lam[NVc + 1];
#pragma unroll
    for (int q = 0; q <= NVc; ++q) lam[q] = 0.0;
    if (cell && g < T.Qp) {
      for (int j = 0; j < T.Qxi; ++j) {
        const double f = gF[T.poff + (size_t)(g * T.Qxi + j) * T.Nx + x];
        const double* pw = tab + TAB_XI + T.Qxi + j * (NV_MAX + 1);
#pragma unroll
        for (int q = 0; q <= NVc; ++q) lam[q] = fma(f, pw[q], lam[q]);
      }
    }
#pragma unroll
    for (int q = 0; q <= NVc; ++q) sm.lam[g * (NV_MAX + 1) + q][c] = lam[q];
  }
  __syncthreads();
  if (g == 0 && cell) {
    double dn = 0.0, dT = 0.0, db = 0.0;
    if (sm.ok[c])
      eq_param_grads<NPc, NVc>(tab, T.Qp, sm.cellv[0][c], sm.cellv[1][c], sm.cellv[2][c], sm.co, c, sm.lam, dn, dT,
                               db);
    const double n_ = sm.cellv[0][c];
    gP[k] = dT / n_;
    gn[k] = dn - dT * sm.P[c] / (n_ * n_);
    gv[k] = db;
  }
}

__global__ void __launch_bounds__(NT) rlb_init_vjp_kernel(const TubeDev* tubes, const int2* tiles,
                                                          const double* tabs, const double* P, const double* n,
                                                          const double* v, const double* gF, double* gP,
                                                          double* gn, double* gv, int* flag) {
  extern __shared__ __align__(16) unsigned char ivjp_smem_raw[];
  InitVjpSmem& sm = *reinterpret_cast<InitVjpSmem*>(ivjp_smem_raw);
  const int2 tl = tiles[blockIdx.x];
  const TubeDev T = tubes[tl.x];
  if (T.Np == 2 && T.Nv == 5)
    init_vjp_tile<2, 5>(T, tabs + T.tab, tl.y, P, n, v, gF, gP, gn, gv, flag, sm);
  else
    init_vjp_tile<NP_MAX, NV_MAX>(T, tabs + T.tab, tl.y, P, n, v, gF, gP, gn, gv, flag, sm);
}
