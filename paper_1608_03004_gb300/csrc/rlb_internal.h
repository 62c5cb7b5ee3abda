// Internal declarations of the CUDA library (not part of the public ABI).
#pragma once

#include <cstdint>

#ifndef __CUDACC__
#define __host__
#define __device__
#endif

namespace rlbq {
bool gauss_legendre(int n, double* x, double* w);
bool gauss_laguerre1(int n, double* x, double* w);
double laguerre1(int l, double x);  // L^(1)_l(x)
double legendre(int k, double x);   // P_k(x)

}  // namespace rlbq

namespace rlb {

// Compile-time maxima of the orders the kernels support.
constexpr int QP_MAX = 4;
constexpr int NP_MAX = 3;             // Np < Qp <= QP_MAX
constexpr int NV_MAX = 8;
constexpr int QXI_MAX = 1024;
constexpr int LEG_MAX = 255;          // longest backward recurrence for the Legendre coefficients

// Per-tube description as the kernels see it.
struct TubeDev {
  int Qp, Qxi, Np, Nv;
  int bc;       // 0 open, 1 periodic
  int collide;  // 0: ballistic
  int Nx;       // cells
  int ld;       // row stride in doubles (padded)
  long long off;   // offset of row 0 of this tube in the state buffers
  long long xoff;  // offset of this tube's cells in the field layout
  double dx, dt, inv_tau;
  double x_left;
  int tab;      // offset of this tube's tables in the table buffer
  int index;    // position of the tube in the caller's list
  int tabf;     // offset of this tube's FP32 tables (reduced-precision storage)
  int storage;  // RLB_STORAGE_F64 / F32 / BF16
  long long poff;  // offset of this tube in the packed state layout (rows of Nx cells, tube after tube)
  double xi_max;      // largest |xi_j|
  double stiff_lim;   // rlb_stiffness_limit(xi_max dt / dx): dt gamma (1 + |beta| xi_max) / tau above it warns
};

// Layout of one tube's tables (doubles, starting at TubeDev::tab):
//   [0, QP_MAX)                 pbar_i
//   [QP_MAX, 2 QP_MAX)          pbar_i^2
//   [2 QP_MAX, 3 QP_MAX)        w^p_i
//   [3 QP_MAX, 3 QP_MAX + QP_MAX (NP_MAX+1))   K[i][q] = (-1)^q sum_{l=q}^{Np} C(l,q) L^(1)_l(pbar_i)
//                                               at [i (NP_MAX+1) + q]: the radial factor multiplying
//                                               s^(q+2) hhat_{q+2,k} in the truncated equilibrium
//   then KW[i][q] = w^p_i K[i][q] / (4 (q+1)! c_q) at [i (NP_MAX+1) + q]: the same with the factors that the
//                                               per-cell coefficients take out (legendre_coeffs), and c_q (NP_MAX+1)
//   then both again as the adjoint takes them (RADIAL_ADJ)
//   then xi_j (Qxi), then w^xi_j P_k(xi_j) at [j (NV_MAX+1) + k] (Qxi (NV_MAX+1)), zero for k > Nv,
//   then b_st dt xi_j / dx at [st Qxi + j] for the three Runge-Kutta stages, b = (1, 1/4, 2/3),
//   then per velocity s = i Qxi + j the WENO5 epsilon term e = 3 eps ws^2, ws = w^p_i w^xi_j / 2 (the limiter acts on
//   the weight-normalised population),
//   then per velocity s the same term as a float pair (hi, lo) in the 8 bytes of slot s (the FP64
//   stage kernel's double-float limiter),
//   then xi_j^2 (Qxi)
constexpr int TAB_PBAR = 0;
constexpr int TAB_PBAR2 = QP_MAX;
constexpr int TAB_WP = 2 * QP_MAX;
constexpr int TAB_K = 3 * QP_MAX;
constexpr int TAB_KW = TAB_K + QP_MAX * (NP_MAX + 1);
constexpr int TAB_KC = TAB_KW + QP_MAX * (NP_MAX + 1);
constexpr int TAB_KWA = TAB_KC + NP_MAX + 1;
constexpr int TAB_KCA = TAB_KWA + QP_MAX * (NP_MAX + 1);
constexpr int TAB_XI = TAB_KCA + NP_MAX + 1;
// Scales c_q of the radial factors by (Qp, Np) = (3, 2), (4, 2), (4, 3): the collision applies the equilibrium in every
// stage, so the rounding of these few constants is the part of its error that adds up over a run. The products
// w^p_i K[i][q] / (4 (q+1)!) of the tables' entries, divided by c_q, all lie within 5e-18 of doubles (found by a search
// over k / 2^17), where they round by up to 1e-16 themselves; the per-cell factors g_q carry c_q.
constexpr double RADIAL_SCALE[3][NP_MAX + 1] = {
    {1.0260772705078125, 1.1634902954101562, 1.6391983032226562, 1.0},
    {1.3723526000976562, 1.0144424438476562, 1.7607879638671875, 1.0},
    {1.1395034790039062, 1.322998046875, 1.6575088500976562, 1.1712188720703125}};
// The adjoint's radial factors, (c_q; K[i][q]) for the same three orders: K[i][q] c_q is w^p_i K[i][q] / (4 (q+1)!) of the
// exact rule within 3 units of 2^-53. They are doubles next to those values, found by a search over c_q = k / 2^12, whose
// sums with the doubles of pbar_i and pbar_i^2 meet the conditions under which the equilibrium keeps N^0 and T^00, each
// order to 5e-18 (three nodes: 1.5e-18). The gradient in log(tau) is a sum of collision terms that cancel to 1e-5 of
// themselves, and a bias of the equilibrium in these moments is what is left of it: with the factors above, which leave
// 6e-17 (three nodes) to 2e-16 (four), that gradient of a 2048-cell inverse problem was 1.1e-11 to 3.2e-10 off (against
// extended precision, six inputs), with these 2.7e-12 to 5.8e-11.
struct RadialAdj {
  double c[NP_MAX + 1], k[QP_MAX][NP_MAX + 1];
};
constexpr RadialAdj RADIAL_ADJ[3] = {
    {{1.7470703125, 1.785888671875, 1.6513671875, 1.0},
     {{0.22698812067910754, -0.09579887087265786, 0.00936379671476203},
      {-0.09845901057459167, 0.11533854013180392, -0.014346168879678392},
      {0.014567591963678652, -0.019539669259146054, 0.0049823721649163615}}},
    {{1.872314453125, 1.01171875, 1.6484375, 1.0},
     {{0.19708849068139514, -0.18492861394231702, 0.011819021642336381},
      {-0.062493369050982246, 0.1999439223017031, -0.017001741456455655},
      {-0.004967235280486029, -0.006673444758233741, 0.004180521551315315},
      {0.003896693125884858, -0.00834186360115231, 0.0010021982628039565}}},
    {{1.790283203125, 1.7490234375, 1.568359375, 1.353759765625},
     {{0.24211096224870726, -0.16223286611923352, 0.032964828719821135, -0.001983228517689746},
      {-0.1345696218644599, 0.2219254185983264, -0.057373046895087085, 0.0038137765996400785},
      {0.03552370267295469, -0.06637888242299789, 0.027634091072212492, -0.002243680786495522},
      {-0.0034223320248824344, 0.006686329943905031, -0.003225872896946547, 0.0004131327045451898}}}};
__host__ __device__ inline int tab_pw(int Qxi) { return TAB_XI + Qxi; }
__host__ __device__ inline int tab_cxi(int Qxi) { return TAB_XI + Qxi + Qxi * (NV_MAX + 1); }
__host__ __device__ inline int tab_eps(int Qxi) { return tab_cxi(Qxi) + 3 * Qxi; }
__host__ __device__ inline int tab_epsf(int Qp, int Qxi) { return tab_eps(Qxi) + Qp * Qxi; }
__host__ __device__ inline int tab_xi2(int Qp, int Qxi) { return tab_epsf(Qp, Qxi) + Qp * Qxi; }
inline int tab_size(int Qp, int Qxi) { return tab_xi2(Qp, Qxi) + Qxi; }
// Per-tube FP32 table of the reduced-precision path (floats, starting at TubeDev::tabf): one record of
// RP_REC floats per velocity s = i Qxi + j, 16-byte aligned, read with vector loads:
//   R_XI          xi_j
//   R_CXI + st    b_st dt xi_j / dx for the three Runge-Kutta stages
//   R_IWS         1 / ws, ws = w^p_i w^xi_j / 2 (the WENO5 limiter acts on F / ws)
//   R_WS6         ws / 6
//   R_P1, R_P2    pbar_i and pbar_i^2 as hi/lo float pairs (moment weights)
//   R_X, R_X2     xi_j and xi_j^2 as hi/lo float pairs
//   R_PW + k      w^xi_j P_k(xi_j), k <= NV_MAX (zero above Nv)
constexpr int RP_REC = 24;
constexpr int R_XI = 0, R_CXI = 1, R_IWS = 4, R_WS6 = 5, R_P1 = 6, R_P2 = 8, R_X = 10, R_X2 = 12, R_PW = 14;
static_assert(R_PW + NV_MAX + 1 <= RP_REC, "record too small");
inline int tabf_size(int Qp, int Qxi) { return Qp * Qxi * RP_REC; }

constexpr double RK_A[3] = {0.0, 0.75, 1.0 / 3.0};  // Shu-Osher SSP-RK3: F_out = a F^n + b (F_in + dt L(F_in))
constexpr double RK_B[3] = {1.0, 0.25, 2.0 / 3.0};

}  // namespace rlb
