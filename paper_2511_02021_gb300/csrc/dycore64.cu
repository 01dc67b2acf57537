// FP64 dynamical-core step ("plain method"): predictor-corrector substeps with
// a vertically implicit w/Exner column solve, then Smagorinsky diffusion.
//
// The paper states that ICON's dynamical core is a nonhydrostatic solver on the
// icosahedral-triangular C grid (Sec. "Current State of the Art"), that it is
// memory-bandwidth bound and dominated by index lookups on triangles, hexagons
// and 12 pentagons (Sec. "Separation of Concerns"), and that all data stay on
// the GPU (Sec. "Innovations Realized"). It gives no discretisation; the one
// computed here, on fields stored level-contiguous ([entity][ld], full level k =
// 0..N-1 top to bottom, half level h = 0..N with w = 0 at h = 0 and h = N), is:
//
//   O1 gradient   (psi_c2 - psi_c1) / d_e
//   O2 divergence (1/A_c) sum_e s_ce l_e u_e
//   O3 curl       (1/A_v) sum_e s_ve d_e vn_e           (counter-clockwise about v)
//   O4 vt         sum_j W_ej vn_j over 5 edges (Perot)
//   O5 K_c        sum_e kappa_ce (vn^2 + vt^2)/2
//   A_vn = -(K_c2 - K_c1)/d_e + ((zeta_v1 + zeta_v2)/2 + f_e) vt - wbar_e dvn/dz
//   A_w  = -sum_e kappa_ce [vn_ie dw/dn + vt_ie dw_v/dt] - w (w_{h-1} - w_{h+1})/(z_{h-1} - z_{h+1})
//   predictor vn* = vn + dtau (A_vn - cpd thv_e dpi/dn), column(S^n, vn*, A_w)
//   corrector vn' = vn + dtau ((A_vn0 + A_vn*)/2 - cpd thv_e* dpi*/dn),
//             column(S^n, vn', (A_w0 + A_w*)/2) with fluxes from S*
//   column: explicit predictors of rho, rho*theta_v, Exner, w with off-centring
//   beta = 0.65, tridiagonal system in w at interior half levels (Thomas,
//   no pivoting), Rayleigh damping, then back-substituted rho, Theta, Exner.
//   diffusion: K_h = cs^2 l d sqrt(D_T^2 + D_S^2) from least-squares vertex
//   velocities, vn += dt K_h L(vn), flux-form theta_v diffusion, Exner adjusted
//   at constant density.
//
// Mapping: one warp per entity (edge, cell or vertex) with lanes over levels, so
// every neighbour index is loaded once per entity and every gathered neighbour
// row is a coalesced, aligned segment; the implicit column solve runs its
// level-parallel parts the same way and only its Thomas recurrence one thread per
// column (see "column solve" below). The summation order of every stencil follows
// the operator definitions (fixed neighbour order), so results do not depend on the
// launch shape.
// FP64 division issues about eight FP64-pipe instructions on this GPU, so every
// division by a geometric or per-level constant is a multiplication by a
// precomputed reciprocal (area factors folded into the stencil weights); the
// column's three quotients per level (pi/Theta, the Thomas pivot, Theta/rho) use
// the Newton-Raphson reciprocal of recip64.h.
#include <cmath>
#include "icon_internal.h"
#include "recip64.h"

namespace icon {
namespace {

constexpr int kWarpsPerBlock = 8;

struct Geo64 {
  int64_t nc, ne, nv;
  int N, ld;
  const int *c2e, *e2c, *e2v, *v2e, *v2c, *vdeg, *e2vt, *e2q;
  const double *div_wa, *rot_wa, *inv_Ac, *vt_w, *kin_w, *lsq_w, *inv_de, *inv_le, *l_e, *d_e, *f_e, *inv_L34;
  const double *n_e, *t_e, *s_ce;
  const double *wu, *wl, *inv_dz, *inv_dz2, *qinv_dz;
  const double* cc;                        // per-level constants for the current dtau
  const double *kin_w_h, *div_wa_h;        // half the cell weights (state tables, [Nc][3])
  const double* adv_w;                     // kappa_ce / d_e (state table, [Nc][3]): w advection
  // what the stencils would otherwise form per warp (a warp serves one entity in three windows of
  // levels, so an instruction per entity costs as much as a third of one per level): per edge
  // [Ne][4] 1/d_e, f_e, d_e / (6 l_e), -cpd / (2 d_e); per cell [Nc][4] the damping Laplacian's
  // weights l_e / (A_c d_e) of the three neighbours and their sum
  const double4 *edge_c, *lap_w;
  bool merge_column, merge_stencil;        // the global grid takes the merged launches
  // terrain-following levels (the TOPO kernel variants; see terrain.cu): per-edge normal
  // slope factor times cpd / 2, full-level decay, per-entity tables [entity][ld], and the stage's
  // contravariant correction, contravariant velocity, Exner perturbation and half its
  // vertical derivative
  const double *t_hsn, *t_bf, *t_wu_e, *t_qinv_dz_e, *t_dz_e;
  const double *t_wu_c, *t_inv_dz_c, *t_inv_dzh_c, *t_wcc, *t_wcon, *t_ep, *t_hdpdz;
};

// per-level constants of the column solve for one dtau, [8][ld]: wu, wl, dtau beta cpd / dzh,
// cpd / dzh, 1/(1 + dtau r), dtau beta / dz, dtau (1 - beta) / dz, 2 beta / dz
enum { C_WU = 0, C_WL, C_CA, C_CX, C_DAMP, C_DTBDZ, C_DT1BDZ, C_2BDZ, C_COUNT };

__global__ void k_colconst64(int N, int ld, const double* __restrict__ wu, const double* __restrict__ wl,
                             const double* __restrict__ dzh, const double* __restrict__ dz,
                             const double* __restrict__ ray, double dtau, double* __restrict__ cc) {
  for (int i = threadIdx.x; i < ld; i += blockDim.x) {
    const bool interior = i > 0 && i < N;
    cc[C_WU * ld + i] = i <= N ? wu[i] : 0.0;
    cc[C_WL * ld + i] = i <= N ? wl[i] : 0.0;
    cc[C_CA * ld + i] = interior ? dtau * kBeta * kCpd / dzh[i] : 0.0;
    cc[C_CX * ld + i] = interior ? kCpd / dzh[i] : 0.0;
    cc[C_DAMP * ld + i] = i <= N ? 1.0 / (1.0 + dtau * ray[i]) : 1.0;
    cc[C_DTBDZ * ld + i] = i < N ? dtau * kBeta / dz[i] : 0.0;
    cc[C_DT1BDZ * ld + i] = i < N ? dtau * (1.0 - kBeta) / dz[i] : 0.0;
    cc[C_2BDZ * ld + i] = i < N ? 2.0 * kBeta / dz[i] : 0.0;
  }
}

// finiteness from the exponent bits (integer pipe; a floating-point compare would
// take an FP64-pipe slot)
__device__ inline bool finite_bits(double x) {
  return ((__double_as_longlong(x) >> 52) & 0x7ff) != 0x7ff;
}

// The warp-per-entity FP64 kernels are held to 64 registers (4 blocks of 8 warps per SM):
// they are bound by the FP64 pipe, and the extra warps hide more load latency than the few
// spilled registers of the rows kernel cost (R2B6/90 step 97.5 -> 94.4 ms).
__device__ inline int64_t warp_entity() {
  return (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
}

// zeta_v (full levels) and six times w_v (half levels): the plain sum of a hexagon's cells,
// scaled by 6/5 at the twelve pentagons (the 1/6 is in the edge tendency's per-edge constant)
__device__ __forceinline__ void vertex_item(const Geo64& G, const double* __restrict__ vn, const double* __restrict__ w,
                                            double* __restrict__ zeta, double* __restrict__ w_v, int64_t v) {
  if (v >= G.nv) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[6], C[6];
  double rw[6];
  for (int j = 0; j < 6; ++j) {
    E[j] = (int64_t)G.v2e[6 * v + j] * ld;
    C[j] = (int64_t)G.v2c[6 * v + j] * ld;
    rw[j] = G.rot_wa[6 * v + j];
  }
  const bool penta = G.vdeg[v] != 6;
  for (int k = lane; k < G.N; k += 32) {
    double acc = 0.0;
    for (int j = 0; j < 6; ++j) acc += rw[j] * vn[E[j] + k];
    zeta[v * ld + k] = acc;
  }
  for (int h = lane; h <= G.N; h += 32) {
    double acc = 0.0;
    for (int j = 0; j < 5; ++j) acc += w[C[j] + h];
    if (penta) acc *= 1.2;
    else acc += w[C[5] + h];
    w_v[v * ld + h] = acc;
  }
}

// vt (Perot) and 2 K_e = vn^2 + vt^2 at edges (the 1/2 is folded into k_cell_ke's weights)
__device__ __forceinline__ void edge_vt_item(const Geo64& G, const double* __restrict__ vn, double* __restrict__ vt,
                                             double* __restrict__ Ke, int64_t e) {
  if (e >= G.ne) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t S[5];
  double W[5];
  for (int j = 0; j < 5; ++j) {
    S[j] = (int64_t)G.e2vt[5 * e + j] * ld;
    W[j] = G.vt_w[5 * e + j];
  }
  for (int k = lane; k < G.N; k += 32) {
    double acc = 0.0;
    for (int j = 0; j < 5; ++j) acc += W[j] * vn[S[j] + k];
    const double v0 = vn[e * ld + k];
    vt[e * ld + k] = acc;
    Ke[e * ld + k] = fma(v0, v0, acc * acc);
  }
}

__global__ void __launch_bounds__(256, 4) k_vertex(Geo64 G, const double* __restrict__ vn, const double* __restrict__ w,
                                                double* __restrict__ zeta, double* __restrict__ w_v) {
  vertex_item(G, vn, w, zeta, w_v, warp_entity());
}

__global__ void __launch_bounds__(256) k_edge_vt(Geo64 G, const double* __restrict__ vn, double* __restrict__ vt,
                                                 double* __restrict__ Ke) {
  edge_vt_item(G, vn, vt, Ke, warp_entity());
}

// both, on small grids: neither reads what the other writes, and a launch there costs more than
// the work (the first nbv blocks take the vertices)
__global__ void __launch_bounds__(256, 4) k_vertex_edge_vt(Geo64 G, const double* __restrict__ vn,
                                                        const double* __restrict__ w, double* __restrict__ zeta,
                                                        double* __restrict__ w_v, double* __restrict__ vt,
                                                        double* __restrict__ Ke, unsigned nbv) {
  if (blockIdx.x < nbv) vertex_item(G, vn, w, zeta, w_v, warp_entity());
  else edge_vt_item(G, vn, vt, Ke, warp_entity() - (int64_t)nbv * kWarpsPerBlock);
}

// K_c at cells (from 2 K_e)
__global__ void __launch_bounds__(256) k_cell_ke(Geo64 G, const double* __restrict__ Ke, double* __restrict__ Kc) {
  const int64_t c = warp_entity();
  if (c >= G.nc) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[3];
  double kw[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    kw[s] = G.kin_w_h[3 * c + s];
  }
  for (int k = lane; k < G.N; k += 32) {
    double acc = 0.0;
    for (int s = 0; s < 3; ++s) acc += kw[s] * Ke[E[s] + k];
    Kc[c * ld + k] = acc;
  }
}

struct EdgeArgs {
  const double *vn, *w, *rho, *thv, *ex;   // stage state (S^n or S*)
  const double *vt, *Kc, *zeta, *w_v;      // diagnostics of the stage state
  const double* vn_base;                   // vn^n
  double* vn_out;                          // vn* or vn^{n+1} (may alias vn_base)
  double* Avn0;                            // stored (predictor) or read (corrector)
  double *F, *G, *a_e, *mflx;
  double dtau;
  double hinv_nsub;                        // 1 / (2 nsub), set on the host
  double hdtau;                            // dtau / 2 (set on the host)
  int corrector;
  int skip_flux;                           // fluxes formed after divergence damping instead
  int upwind_theta;                        // heat flux with the upwind theta_v (option)
};

// vn tendency and update, horizontal mass/heat fluxes, edge part of w advection.
// FP64-pipe bound, so the kernel minimises FP64 warp instructions: one pass over the
// half levels in windows of 31 (lane l of a window holds half level h = base + l and,
// for l < 31, full level k = h), each half-level interpolant and cell-pair sum formed
// once and handed to the lane below with a shuffle, factors of 1/2 folded into
// exactly-scaled constants, and the per-edge constants read from a table.
//
// TOPO (terrain-following levels): per-edge interpolation weights, the contravariant
// vertical velocity w - wcc (zero at lid and ground) in the vertical advection of vn,
// the metric correction of the pressure gradient on pi' = pi - pi_ref,
//   (pi'_c2 - pi'_c1)/d_e - sn_e bf_k (d pi'/dz at c1 and c2)/2,
// and mass fluxes through layers of thickness dz_e; w - wcc, pi' and d pi'/dz come from
// the stage's k_topo_cell.
template <bool TOPO, bool UT>
__global__ void __launch_bounds__(256, 4) k_edge_tend(Geo64 G, EdgeArgs a) {
  const int64_t e = warp_entity();
  if (e >= G.ne) return;
  const int lane = threadIdx.x & 31, ld = G.ld, N = G.N;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld;
  const int64_t v1 = (int64_t)G.e2v[2 * e] * ld, v2 = (int64_t)G.e2v[2 * e + 1] * ld;
  const int64_t eo = e * ld;
  // 1/d_e; f_e; d_e / (6 l_e) (a_e is stored times d_e, the cells' weights carry 1/d_e, and w_v is
  // six times the mean); -cpd / (2 d_e), or -cpd / d_e in the corrector. The factors 1/2 of
  // theta_e = (t1 + t2)/2 and rho_e = (rho1 + rho2)/2 are in the last one and in the column's
  // divergence weights, exact scalings by powers of two
  const double4 ec = G.edge_c[e];
  const double ide = ec.x, fe = ec.y, rt = ec.z;
  const double npg = (!TOPO && a.corrector) ? ec.w + ec.w : ec.w;
  const double hsn = TOPO ? G.t_hsn[e] : 0.0;
  const double hinv_nsub = a.hinv_nsub;
  const double* __restrict__ vn = a.vn + eo;
  const double* __restrict__ vt = a.vt + eo;
  const double dtau = a.dtau;
  for (int base = 0; base <= N; base += 31) {
    const int h = base + lane;
    const bool hv = h <= N;                    // a half level of this column
    const bool kv = lane < 31 && h < N;        // a full level owned by this lane
    // half-level interpolation weights: f(0) = f[0], f(N) = f[N-1], linear between
    const int hl = h > 0 ? (h - 1 < N - 1 ? h - 1 : N - 1) : 0;
    const int hu = h < N ? h : N - 1;
    double wa, wb;
    if (TOPO) {
      wa = (h == 0) ? 0.0 : (h >= N ? 1.0 : G.t_wu_e[eo + h]);
      wb = (h == 0) ? 1.0 : (h >= N ? 0.0 : 1.0 - wa);
    } else {
      wa = (h == 0) ? 0.0 : (h >= N ? 1.0 : G.wu[h]);
      wb = (h == 0) ? 1.0 : (h >= N ? 0.0 : G.wl[h]);
    }
    double vie = 0.0, tie = 0.0, sw = 0.0, dw = 0.0, dwv = 0.0;
    if (hv) {
      vie = wa * vn[hl] + wb * vn[hu];
      tie = wa * vt[hl] + wb * vt[hu];
      const double w1 = a.w[c1 + h], w2 = a.w[c2 + h];
      if (TOPO)
        sw = G.t_wcon[c1 + h] + G.t_wcon[c2 + h];        // 0 at the lid and the ground
      else
        sw = w1 + w2;
      dw = w2 - w1;
      dwv = a.w_v[v2 + h] - a.w_v[v1 + h];
    }
    const double vie_up = __shfl_down_sync(0xffffffffu, vie, 1);   // half level h + 1
    const double sw_up = __shfl_down_sync(0xffffffffu, sw, 1);
    if (hv && lane < 31) a.a_e[eo + h] = fma(vie, dw, (tie * rt) * dwv);
    if (kv) {
      const int k = h;
      // advective tendency: -grad K + (zeta + f) vt - wbar dvn/dz, with
      // wbar = (sum of the four w) / 4 and the 1/4 folded into the level constant
      const double zs = a.zeta[v1 + k] + a.zeta[v2 + k];
      const double dK = a.Kc[c2 + k] - a.Kc[c1 + k];
      const double T = fma(-dK, ide, fma(0.5, zs, fe) * vt[k]);
      const double A = fma(-((sw + sw_up) * (vie - vie_up)), TOPO ? G.t_qinv_dz_e[eo + k] : G.qinv_dz[k], T);
      const double t1 = a.thv[c1 + k], t2 = a.thv[c2 + k];
      const double th_s = t1 + t2;                     // 2 theta_e
      double vnew;
      if (TOPO) {
        // X: the pressure gradient over theta_e / 2, downgradient
        const double X = fma(G.t_ep[c2 + k] - G.t_ep[c1 + k], npg,
                             (hsn * G.t_bf[k]) * (G.t_hdpdz[c1 + k] + G.t_hdpdz[c2 + k]));
        if (a.corrector) {
          vnew = fma(dtau, fma(0.5, a.Avn0[eo + k] + A, th_s * X), a.vn_base[eo + k]);
        } else {
          vnew = fma(dtau, fma(th_s, X, A), a.vn_base[eo + k]);
          a.Avn0[eo + k] = A;
        }
      } else {
        const double tdx = th_s * (a.ex[c2 + k] - a.ex[c1 + k]);
        if (a.corrector) {
          vnew = fma(a.hdtau, fma(npg, tdx, a.Avn0[eo + k] + A), a.vn_base[eo + k]);
        } else {
          vnew = fma(dtau, fma(npg, tdx, A), a.vn_base[eo + k]);
          a.Avn0[eo + k] = A;
        }
      }
      a.vn_out[eo + k] = vnew;
      if (a.skip_flux) continue;
      // F = 2 rho_e vn and G = 4 rho_e vn theta_e (exactly; the column weights carry 1/2)
      double F = (a.rho[c1 + k] + a.rho[c2 + k]) * vnew;
      if (TOPO) F *= G.t_dz_e[eo + k];
      a.F[eo + k] = F;
      if constexpr (UT) a.G[eo + k] = F * (2.0 * (vnew >= 0.0 ? t1 : t2));     // upwind theta_v (option)
      else a.G[eo + k] = F * th_s;
      if (a.corrector) a.mflx[eo + k] = fma(F, hinv_nsub, a.mflx[eo + k]);
    }
  }
}

// ---------------------------------------------------------------- divergence damping (option)
// Fourth-order divergence damping of the corrector's vn^{n+1} before its fluxes are formed:
// vn -= c4 Abar^2 grad(div(grad(div vn))), Abar the mean cell area (an ICON option; the
// paper prints none). Cell divergence, cell Laplacian of it, then the edge update together
// with the corrector's mass and heat fluxes and the step-mean mass flux.
__global__ void __launch_bounds__(256, 4) k_dd_div(Geo64 G, const double* __restrict__ vn, double* __restrict__ D) {
  const int64_t c = warp_entity();
  if (c >= G.nc) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[3];
  double dw[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    dw[s] = G.div_wa[3 * c + s];
  }
  for (int k = lane; k < G.N; k += 32) D[c * ld + k] = (dw[0] * vn[E[0] + k] + dw[1] * vn[E[1] + k]) + dw[2] * vn[E[2] + k];
}

__global__ void __launch_bounds__(256, 4) k_dd_lap(Geo64 G, const double* __restrict__ D, double* __restrict__ L) {
  const int64_t c = warp_entity();
  if (c >= G.nc) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  // sum_s l_e / (A_c d_e) (D_nb - D_c), the own value's weights summed
  int64_t B[3];
  for (int s = 0; s < 3; ++s) {
    const int e = G.c2e[3 * c + s];
    const int ca = G.e2c[2 * e], cb = G.e2c[2 * e + 1];
    B[s] = (int64_t)(ca == c ? cb : ca) * ld;
  }
  const double4 w = G.lap_w[c];
  for (int k = lane; k < G.N; k += 32)
    L[c * ld + k] = fma(w.z, D[B[2] + k], fma(w.y, D[B[1] + k], fma(w.x, D[B[0] + k], -(w.w * D[c * ld + k]))));
}

struct DDArgs {
  const double *L, *rho, *thv;             // Laplacian of the divergence, stage state S*
  double *vn, *F, *G, *mflx;
  const double* dz_e;                      // layer thickness at edges (terrain-following), or NULL
  double scale, hinv_nsub;                 // c4 Abar^2, 1 / (2 nsub)
  int upwind_theta;
};

__global__ void __launch_bounds__(256, 4) k_dd_edge(Geo64 G, DDArgs a) {
  const int64_t e = warp_entity();
  if (e >= G.ne) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld, eo = e * ld;
  const double s = a.scale * G.inv_de[e];
  for (int k = lane; k < G.N; k += 32) {
    const double vn = a.vn[eo + k] - s * (a.L[c2 + k] - a.L[c1 + k]);
    a.vn[eo + k] = vn;
    double F = (a.rho[c1 + k] + a.rho[c2 + k]) * vn;      // 2 rho_e vn, as k_edge_tend
    if (a.dz_e) F *= a.dz_e[eo + k];
    a.F[eo + k] = F;
    const double t1 = a.thv[c1 + k], t2 = a.thv[c2 + k];
    a.G[eo + k] = F * (a.upwind_theta ? (vn >= 0.0 ? t1 + t1 : t2 + t2) : t1 + t2);
    a.mflx[eo + k] = fma(F, a.hinv_nsub, a.mflx[eo + k]);
  }
}

// ---------------------------------------------------------------- column solve
//
// The vertically implicit update of every column in three launches:
//   k_col_rows   one warp per cell, lanes over levels: everything that is parallel
//                over the levels (half-level interpolants, horizontal divergences,
//                explicit predictors, the linearised state equation, the w predictor
//                and, in the predictor, the tridiagonal row of every interior half
//                level). Rows go out level-major for the solve; the operands of the
//                final update stay in the cell's own rows.
//   k_col_thomas one thread per column: the Thomas recurrence on level-major rows
//                (coalesced across the warp; the corrector substitutes with the
//                predictor's factors), Rayleigh damping; the solution w overwrites
//                the right-hand side.
//   k_col_update one warp per cell, lanes over levels: the implicit parts of rho,
//                Theta and pi, theta_v = Theta / rho, the step-mean vertical mass flux.
// Only the recurrence is sequential in the level; keeping it apart lets the rest run
// with coalesced, level-contiguous loads instead of one thread walking a column.
//
// The FP64 pipe bounds all three, so whatever depends on S^n only is formed by the predictor
// and handed to the corrector in buffers that are dead meanwhile: the matrix factors, gamma,
// the half-level interpolants rho_ic and M, a = dtau beta cpd theta_ic / dzh (in the column's
// former solution buffer), the w predictor without the stages' advection, plus half the
// predictor's (in A_w's buffer), and on flat levels the parts of rho and Theta without the
// horizontal divergences and the same part of Exner's increment. The first two overwrite S^n's
// rho and theta_v, which nothing else reads until the corrector writes S^{n+1} there: the
// stencils of the corrector read S*. Exner is carried as its increment delta on S^n's: the
// pressure term of the row, -a (pi*_{h-1} - pi*_h), splits into S^n's part, which joins the
// hydrostatic residual of the w predictor (one difference of neighbouring Exner values, exact),
// and -a (delta_{h-1} - delta_h), which is small; the roundings of pi* no longer enter w.
// Corrector rows: 18 FP64 instructions per cell-level as written, 35 when it formed them again
// from S^n. R2B6/90: the column 3.35 ms per launch (mean of the stages), was 3.93.
struct ColArgs {
  // S^n [c][ld]; on flat levels the predictor leaves the explicit parts of rho and Theta
  // without the horizontal divergences in rho and thv, Exner's increment in d0
  double *rho, *thv, *d0;
  const double *ex, *w;
  const double* w_stage;                   // w of the stage state (vertical part of A_w)
  const double *F, *G, *a_e;               // edge fluxes and d_e times the w-advection edge terms
  double* ba;                              // w^n - dtau (cpd theta_ic dpi/dz + g) + (dtau/2) A_w0: [c][ld]
  double* aa;                              // dtau beta cpd theta_ic / dzh: [c][ld]
  double *lo, *di, *up, *rh;               // tridiagonal rows, level-major [h][Nc], h = 1..N-1; rh becomes w^{n+1}
  double *rx, *tx, *dx, *gm;               // rho*, Theta*, pi* - pi (explicit parts), gamma: [c][ld]
  double* gc;                              // (dtau/2) (Rd/cvd) pi / Theta of S^n: [c][ld]
  double *ri, *mm;                         // half-level rho and rho theta_v of S^n: [c][ld]
  double *rho_o, *thv_o, *ex_o, *w_o;      // S* or S^{n+1} (may alias S^n)
  double* wflx;
  unsigned* status;
  double dtau, inv_nsub;
  double hdtau, hrc, inv_dtau2;            // dtau / 2, (dtau / 2) Rd/cvd and 2 / dtau (set on the host)
  double b_new, b_old;                     // beta / nsub, (1 - beta) / nsub
  int hdamp;                               // half levels h < hdamp lie in the Rayleigh layer
};

// windows of 31 levels: lane l holds full level k = base + l and the half level above
// it (h = k); lane 31 only supplies the half level below lane 30's full level. The level above
// comes from the neighbouring lane (lane 30's is carried to the next window), never from
// memory, where this kernel has overwritten it.
// TOPO (terrain-following levels): each cell's own spacings and interpolation weights,
// thickness-weighted horizontal fluxes (already carrying dz_e) divided by the cell's dz,
// the explicit vertical fluxes with the contravariant (1 - beta) w - wcc, and the
// vertical advection of w with w - wcc; S^n stays, since those fluxes change with the stage.
template <bool TOPO>
__device__ __forceinline__ void col_rows_pred(const Geo64& G, const ColArgs& a, int64_t c) {
  const int lane = threadIdx.x & 31, ld = G.ld, N = G.N;
  const int64_t o = c * ld, nc = G.nc;
  const double* __restrict__ cc = G.cc;
  int64_t E[3];
  double dw[3], kw[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    dw[s] = G.div_wa_h[3 * c + s];         // the edge fluxes are 2 rho_e vn and 4 rho_e vn theta_e
    kw[s] = G.adv_w[3 * c + s];
  }
  const double dtau = a.dtau, hdtau = a.hdtau;
  double gam_c = 0.0, dx_c = 0.0, M_c = 0.0;          // carried: full / half level base - 1
  double rho_c = 0.0, thv_c = 0.0, ex_c = 0.0;
  for (int base = 0; base <= N; base += 31) {
    const int k = base + lane;
    const bool hv = k <= N;                            // half level k exists
    const bool kv = lane < 31 && k < N;                // full level k owned here
    double rho = 0.0, thv = 0.0, ex = 0.0;
    if (k < N) { rho = a.rho[o + k]; thv = a.thv[o + k]; ex = a.ex[o + k]; }
    double rho_m = __shfl_up_sync(0xffffffffu, rho, 1);
    double thv_m = __shfl_up_sync(0xffffffffu, thv, 1);
    double ex_m = __shfl_up_sync(0xffffffffu, ex, 1);
    if (lane == 0) { rho_m = rho_c; thv_m = thv_c; ex_m = ex_c; }
    rho_c = __shfl_sync(0xffffffffu, rho, 30);
    thv_c = __shfl_sync(0xffffffffu, thv, 30);
    ex_c = __shfl_sync(0xffffffffu, ex, 30);
    // half-level interpolants of S^n: rho_ic and M = rho_ic theta_ic
    double ri = 0.0, ti = 0.0;
    if (k == 0) { ri = rho; ti = thv; }
    else if (k == N) { ri = rho_m; ti = thv_m; }
    else if (k < N) {
      if constexpr (TOPO) {
        const double wu = G.t_wu_c[o + k], wl = 1.0 - wu;
        ri = wu * rho_m + wl * rho;
        ti = wu * thv_m + wl * thv;
      } else {
        const double wu = cc[C_WU * ld + k], wl = cc[C_WL * ld + k];
        ri = wu * rho_m + wl * rho;
        ti = wu * thv_m + wl * thv;
      }
    }
    const double M = ri * ti;
    const double wk = hv ? a.w[o + k] : 0.0;
    // TOPO: explicit part of the contravariant velocity at interior half levels
    const double ve = (TOPO && k >= 1 && k < N) ? (1.0 - kBeta) * wk - G.t_wcc[o + k] : wk;
    const double ri1 = __shfl_down_sync(0xffffffffu, ri, 1);      // half level k + 1
    const double M1 = __shfl_down_sync(0xffffffffu, M, 1);
    const double ve1 = __shfl_down_sync(0xffffffffu, (TOPO && (k < 1 || k >= N)) ? 0.0 : ve, 1);
    double gam = 0.0, dx = 0.0;
    if (kv) {
      // explicit predictors at full level k
      // Dr: the mass-flux divergence; Dt2: twice the heat-flux divergence
      double Dr = 0.0, Dt2 = 0.0;
      for (int s = 0; s < 3; ++s) Dr += dw[s] * a.F[E[s] + k];
      for (int s = 0; s < 3; ++s) Dt2 += dw[s] * a.G[E[s] + k];
      const double Th = rho * thv;
      const double gd = (a.hrc * ex) * recip64(Th);   // (dtau/2) times the state-equation factor
      a.gc[o + k] = gd;
      double rx, tx;
      if constexpr (TOPO) {
        const double v0 = k >= 1 ? ve : 0.0;
        const double idz = G.t_inv_dz_c[o + k], dti = dtau * idz;
        rx = rho - dti * ((Dr + ri * v0) - ri1 * ve1);
        const double dT = dti * ((0.5 * Dt2 + M * v0) - M1 * ve1);
        tx = Th - dT;
        dx = -(gd * a.inv_dtau2) * dT;
        gam = gd * ((2.0 * kBeta) * idz);
      } else {
        const double dt1 = cc[C_DT1BDZ * ld + k];
        const double Q = M * wk - M1 * ve1;
        gam = gd * cc[C_2BDZ * ld + k];
        const double r0 = rho - dt1 * (ri * wk - ri1 * ve1), t0 = Th - dt1 * Q;
        const double d0 = ((kBeta - 1.0) / kBeta * gam) * Q;
        rx = r0 - dtau * Dr;
        tx = t0 - hdtau * Dt2;
        dx = d0 - gd * Dt2;
        a.rho[o + k] = r0;
        a.thv[o + k] = t0;
        a.d0[o + k] = d0;
      }
      a.rx[o + k] = rx;
      a.tx[o + k] = tx;
      a.dx[o + k] = dx;
      a.gm[o + k] = gam;
    }
    if (hv && lane < 31) {
      a.ri[o + k] = ri;
      a.mm[o + k] = M;
    }
    // full level and half level above: from the lane above, or carried for lane 0
    double gam_m = __shfl_up_sync(0xffffffffu, gam, 1);
    double dx_m = __shfl_up_sync(0xffffffffu, dx, 1);
    double M_m = __shfl_up_sync(0xffffffffu, M, 1);
    if (lane == 0) { gam_m = gam_c; dx_m = dx_c; M_m = M_c; }
    if (kv && k >= 1) {
      // row of interior half level h = k: w predictor and the implicit coupling
      const int h = k;
      double hadv = 0.0;
      for (int s = 0; s < 3; ++s) hadv += kw[s] * a.a_e[E[s] + h];
      const double* ws = a.w_stage + o + h;
      double Aw, B, aa;
      if constexpr (TOPO) {
        const double idzh = G.t_inv_dzh_c[o + h];
        Aw = -hadv - G.t_wcon[o + h] * (ws[-1] - ws[1]) * (0.5 * idzh);
        B = wk + dtau * (-((kCpd * idzh) * ti) * (ex_m - ex) - kGrav);
        aa = (dtau * kBeta * kCpd * idzh) * ti;
      } else {
        Aw = -hadv - ws[0] * (ws[-1] - ws[1]) * G.inv_dz2[h];
        B = wk + dtau * (-(cc[C_CX * ld + h] * ti) * (ex_m - ex) - kGrav);
        aa = cc[C_CA * ld + h] * ti;
      }
      a.ba[o + h] = B + hdtau * Aw;
      a.aa[o + h] = aa;
      const int64_t i = (int64_t)h * nc + c;
      const double P = aa * gam_m, Q = aa * gam;
      a.lo[i] = -P * M_m;
      a.di[i] = fma(P + Q, M, 1.0);
      a.up[i] = -Q * M1;
      a.rh[i] = (B + dtau * Aw) - aa * (dx_m - dx);
    }
    gam_c = __shfl_sync(0xffffffffu, gam, 30);
    dx_c = __shfl_sync(0xffffffffu, dx, 30);
    M_c = __shfl_sync(0xffffffffu, M, 30);
  }
}

// the corrector's right-hand side and explicit parts, from what the predictor left. Flat levels
// need the level above only: windows of 32 with lane 31's carried.
template <bool TOPO>
__device__ __forceinline__ void col_rows_corr(const Geo64& G, const ColArgs& a, int64_t c) {
  const int lane = threadIdx.x & 31, ld = G.ld, N = G.N;
  const int64_t o = c * ld, nc = G.nc;
  int64_t E[3];
  double dw[3], kw[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    dw[s] = G.div_wa_h[3 * c + s];
    kw[s] = G.adv_w[3 * c + s];
  }
  const double dtau = a.dtau, hdtau = a.hdtau;
  constexpr int W = TOPO ? 31 : 32;
  double dx_c = 0.0;                                   // carried: full level base - 1
  for (int base = 0; base < N; base += W) {
    const int k = base + lane;
    const bool kv = lane < W && k < N;
    double ve = 0.0, ve1 = 0.0;
    if constexpr (TOPO) {
      if (k >= 1 && k < N) ve = (1.0 - kBeta) * a.w[o + k] - G.t_wcc[o + k];
      ve1 = __shfl_down_sync(0xffffffffu, ve, 1);
    }
    double dx = 0.0;
    if (kv) {
      double Dr = 0.0, Dt2 = 0.0;
      for (int s = 0; s < 3; ++s) Dr += dw[s] * a.F[E[s] + k];
      for (int s = 0; s < 3; ++s) Dt2 += dw[s] * a.G[E[s] + k];
      const double gd = a.gc[o + k];
      double rx, tx;
      if constexpr (TOPO) {
        const double rho = a.rho[o + k], Th = rho * a.thv[o + k], dti = dtau * G.t_inv_dz_c[o + k];
        rx = rho - dti * ((Dr + a.ri[o + k] * ve) - a.ri[o + k + 1] * ve1);
        const double dT = dti * ((0.5 * Dt2 + a.mm[o + k] * ve) - a.mm[o + k + 1] * ve1);
        tx = Th - dT;
        dx = -(gd * a.inv_dtau2) * dT;
      } else {
        rx = a.rho[o + k] - dtau * Dr;
        tx = a.thv[o + k] - hdtau * Dt2;
        dx = a.d0[o + k] - gd * Dt2;
      }
      a.rx[o + k] = rx;
      a.tx[o + k] = tx;
      a.dx[o + k] = dx;
    }
    double dx_m = __shfl_up_sync(0xffffffffu, dx, 1);
    if (lane == 0) dx_m = dx_c;
    dx_c = __shfl_sync(0xffffffffu, dx, W - 1);
    if (kv && k >= 1) {
      const int h = k;
      double hadv = 0.0;
      for (int s = 0; s < 3; ++s) hadv += kw[s] * a.a_e[E[s] + h];
      const double* ws = a.w_stage + o + h;
      double Aw;
      if constexpr (TOPO) Aw = -hadv - G.t_wcon[o + h] * (ws[-1] - ws[1]) * (0.5 * G.t_inv_dzh_c[o + h]);
      else Aw = -hadv - ws[0] * (ws[-1] - ws[1]) * G.inv_dz2[h];
      a.rh[(int64_t)h * nc + c] = (a.ba[o + h] + hdtau * Aw) - a.aa[o + h] * (dx_m - dx);
    }
  }
}

// Thomas recurrence per column on the level-major rows; the next row is loaded before
// the current one is stored so that its loads overlap the recurrence. The matrix depends on
// S^n only (rho_ic, theta_ic and the state-equation factor of the substep's start), so it is
// the same in both stages: the predictor factors it, keeping the sub-diagonal, storing
// 1 / pivot over the diagonal and up / pivot over the super-diagonal, and the corrector only
// substitutes its own right-hand side. The damped solution goes over the right-hand side.
template <bool CORR>
__device__ __forceinline__ void col_thomas(const Geo64& G, const ColArgs& a, int64_t c) {
  const int N = G.N, ld = G.ld;
  if (N < 2) return;
  const int64_t nc = G.nc;
  const double* __restrict__ cc = G.cc;
  const double* lo = a.lo;
  double *di = a.di, *up = a.up, *rh = a.rh;
  double dp = 0.0;
  if (!CORR) {
    double cp = 0.0;
    double l = lo[nc + c], d = di[nc + c], u = up[nc + c], r = rh[nc + c];
    for (int h = 1; h < N; ++h) {
      double ln = 0.0, dn = 0.0, un = 0.0, rn = 0.0;
      if (h + 1 < N) {
        const int64_t j = (int64_t)(h + 1) * nc + c;
        ln = lo[j]; dn = di[j]; un = up[j]; rn = rh[j];
      }
      const double q = recip64(h == 1 ? d : d - l * cp);
      cp = u * q;
      dp = (h == 1 ? r : r - l * dp) * q;
      const int64_t i = (int64_t)h * nc + c;
      di[i] = q;
      up[i] = cp;
      rh[i] = dp;
      l = ln; d = dn; u = un; r = rn;
    }
  } else {
    double l = lo[nc + c], q = di[nc + c], r = rh[nc + c];
    for (int h = 1; h < N; ++h) {
      double ln = 0.0, qn = 0.0, rn = 0.0;
      if (h + 1 < N) {
        const int64_t j = (int64_t)(h + 1) * nc + c;
        ln = lo[j]; qn = di[j]; rn = rh[j];
      }
      dp = (h == 1 ? r : r - l * dp) * q;
      rh[(int64_t)h * nc + c] = dp;
      l = ln; q = qn; r = rn;
    }
  }
  // back substitution
  double x = dp;
  if (N - 1 < a.hdamp) rh[(int64_t)(N - 1) * nc + c] = x * cc[C_DAMP * ld + N - 1];
  for (int h = N - 2; h >= 1; --h) {
    const int64_t i = (int64_t)h * nc + c;
    x = rh[i] - up[i] * x;
    rh[i] = h < a.hdamp ? x * cc[C_DAMP * ld + h] : x;
  }
}

// TOPO: each cell's dz, the contravariant step-mean vertical flux, and the ground w of
// the stage (its wcc, so that w - wcc = 0 there)
template <bool TOPO, bool CORR>
__device__ __forceinline__ void col_update(const Geo64& G, const ColArgs& a, int64_t c) {
  const int lane = threadIdx.x & 31, ld = G.ld, N = G.N;
  const int64_t o = c * ld, nc = G.nc;
  const double* __restrict__ cc = G.cc;
  bool bad = false;
  for (int base = 0; base < N; base += 31) {
    const int k = base + lane;
    // w^{n+1} (damped) at half level k; zero at the top and the bottom
    const double wn = (k >= 1 && k < N) ? a.rh[(int64_t)k * nc + c] : 0.0;
    const double ri = k <= N ? a.ri[o + k] : 0.0;
    const double M = k <= N ? a.mm[o + k] : 0.0;
    const double wn1 = __shfl_down_sync(0xffffffffu, wn, 1);
    const double ri1 = __shfl_down_sync(0xffffffffu, ri, 1);
    const double M1 = __shfl_down_sync(0xffffffffu, M, 1);
    if (lane < 31 && k < N) {
      const double q = M * wn - M1 * wn1;
      const double r = ri * wn - ri1 * wn1;
      const double dtb = TOPO ? a.dtau * kBeta * G.t_inv_dz_c[o + k] : cc[C_DTBDZ * ld + k];
      const double Th_n = a.tx[o + k] - dtb * q;
      const double ex_n = a.ex[o + k] + (a.dx[o + k] - a.gm[o + k] * q);
      const double rho_n = a.rx[o + k] - dtb * r;
      const double thv_n = Th_n * recip64(rho_n);
      if (CORR) {
        // (beta wn + (1 - beta) wold - wcc) / nsub with the weights divided on the host
        const double wold = a.w[o + k];
        double wc = fma(a.b_new, wn, a.b_old * wold);
        if (TOPO) wc = fma(-a.inv_nsub, G.t_wcc[o + k], wc);
        a.wflx[o + k] = fma(ri, wc, a.wflx[o + k]);
      }
      a.rho_o[o + k] = rho_n;
      a.thv_o[o + k] = thv_n;
      a.ex_o[o + k] = ex_n;
      a.w_o[o + k] = wn;
      bad |= !finite_bits(thv_n) || !finite_bits(wn) || !finite_bits(ex_n);
    }
  }
  if (lane == 0) a.w_o[o + N] = TOPO ? G.t_wcc[o + N] : 0.0;
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(a.status, 1u);
}

template <bool TOPO, bool CORR>
__device__ __forceinline__ void col_rows(const Geo64& G, const ColArgs& a, int64_t c) {
  if constexpr (CORR) col_rows_corr<TOPO>(G, a, c);
  else col_rows_pred<TOPO>(G, a, c);
}

template <bool TOPO, bool CORR>
__global__ void __launch_bounds__(256, 4) k_col_rows(Geo64 G, ColArgs a) {
  const int64_t c = warp_entity();
  if (c < G.nc) col_rows<TOPO, CORR>(G, a, c);
}

template <bool CORR>
__global__ void __launch_bounds__(128) k_col_thomas(Geo64 G, ColArgs a) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c < G.nc) col_thomas<CORR>(G, a, c);
}

template <bool TOPO, bool CORR>
__global__ void __launch_bounds__(256) k_col_update(Geo64 G, ColArgs a) {
  const int64_t c = warp_entity();
  if (c < G.nc) col_update<TOPO, CORR>(G, a, c);
}

// the three in one launch, on small grids: a block takes eight cells, one per warp in the
// level-parallel parts, and eight lanes walk their columns; the rows pass through global memory
// (the block's own barriers order them) and stay in L2. Eight cells and not 32: an SM's FP64 pipe
// takes a warp instruction every 16 cycles, so a small grid has to be spread over all SMs
// (R2B2/20: 450 us per step with 32 cells a block, 356 with eight).
template <bool TOPO, bool CORR>
__global__ void __launch_bounds__(256, 4) k_col_small(Geo64 G, ColArgs a) {
  const int64_t c0 = (int64_t)blockIdx.x * kWarpsPerBlock, c = warp_entity();
  if (c < G.nc) col_rows<TOPO, CORR>(G, a, c);
  __syncthreads();
  if (threadIdx.x < kWarpsPerBlock && c0 + threadIdx.x < G.nc) col_thomas<CORR>(G, a, c0 + threadIdx.x);
  __syncthreads();
  if (c < G.nc) col_update<TOPO, CORR>(G, a, c);
}

// ---------------------------------------------------------------- diffusion
__global__ void __launch_bounds__(256, 4) k_diff_vertex(Geo64 G, const double* __restrict__ vn, double* __restrict__ ux,
                                                     double* __restrict__ uy, double* __restrict__ uz,
                                                     double* __restrict__ zeta) {
  const int64_t v = warp_entity();
  if (v >= G.nv) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[6];
  for (int j = 0; j < 6; ++j) E[j] = (int64_t)G.v2e[6 * v + j] * ld;
  const double* lw = G.lsq_w + 18 * v;
  const double* rw = G.rot_wa + 6 * v;
  for (int k = lane; k < G.N; k += 32) {
    double x = 0.0, y = 0.0, z = 0.0, r = 0.0;
    for (int j = 0; j < 6; ++j) {
      const double q = vn[E[j] + k];
      x += lw[3 * j] * q;
      y += lw[3 * j + 1] * q;
      z += lw[3 * j + 2] * q;
      r += rw[j] * q;
    }
    ux[v * ld + k] = x;
    uy[v * ld + k] = y;
    uz[v * ld + k] = z;
    zeta[v * ld + k] = r;
  }
}

__global__ void __launch_bounds__(256) k_diff_div(Geo64 G, const double* __restrict__ vn, double* __restrict__ divc) {
  const int64_t c = warp_entity();
  if (c >= G.nc) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[3];
  double dw[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    dw[s] = G.div_wa[3 * c + s];
  }
  for (int k = lane; k < G.N; k += 32) {
    double acc = 0.0;
    for (int s = 0; s < 3; ++s) acc += dw[s] * vn[E[s] + k];
    divc[c * ld + k] = acc;
  }
}

// fourth-order background diffusion (option): L1 = L(vn) at edges, then the divergence
// and curl of L1 for the second Laplacian in k_diff_edge
__global__ void __launch_bounds__(256, 4) k_bd_lap(Geo64 G, const double* __restrict__ zeta,
                                                const double* __restrict__ divc, double* __restrict__ L1) {
  const int64_t e = warp_entity();
  if (e >= G.ne) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld;
  const int64_t v1 = (int64_t)G.e2v[2 * e] * ld, v2 = (int64_t)G.e2v[2 * e + 1] * ld;
  const double ile = G.inv_le[e], ide = G.inv_de[e];
  for (int k = lane; k < G.N; k += 32)
    L1[e * ld + k] = (divc[c2 + k] - divc[c1 + k]) * ide - (zeta[v2 + k] - zeta[v1 + k]) * ile;
}

__global__ void __launch_bounds__(256, 4) k_bd_curl(Geo64 G, const double* __restrict__ L1, double* __restrict__ zeta1) {
  const int64_t v = warp_entity();
  if (v >= G.nv) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[6];
  double rw[6];
  for (int j = 0; j < 6; ++j) {
    E[j] = (int64_t)G.v2e[6 * v + j] * ld;
    rw[j] = G.rot_wa[6 * v + j];
  }
  for (int k = lane; k < G.N; k += 32) {
    double r = 0.0;
    for (int j = 0; j < 6; ++j) r += rw[j] * L1[E[j] + k];
    zeta1[v * ld + k] = r;
  }
}

struct BDArgs {
  const double *D1, *zeta1;                // divergence and curl of L(vn); NULL: no background diffusion
  double scale;                            // c Abar^2
};

__global__ void __launch_bounds__(256, 3) k_diff_edge(Geo64 G, double* __restrict__ vn, const double* __restrict__ ux,
                                                   const double* __restrict__ uy, const double* __restrict__ uz,
                                                   const double* __restrict__ zeta, const double* __restrict__ divc,
                                                   const double* __restrict__ thv, double* __restrict__ thflx,
                                                   double dt, BDArgs bd) {
  const int64_t e = warp_entity();
  if (e >= G.ne) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t Q[4];
  for (int j = 0; j < 4; ++j) Q[j] = (int64_t)G.e2q[4 * e + j] * ld;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld;
  const int64_t v1 = (int64_t)G.e2v[2 * e] * ld, v2 = (int64_t)G.e2v[2 * e + 1] * ld;
  const double ile = G.inv_le[e], ide = G.inv_de[e], i34 = G.inv_L34[e];
  // the normal and the tangent scaled by 1/L34 and 1/l_e once per edge, and the factors of the
  // two products that K_h enters
  double n34[3], t34[3], n12[3], t12[3];
  for (int j = 0; j < 3; ++j) {
    const double n = G.n_e[3 * e + j], t = G.t_e[3 * e + j];
    n34[j] = n * i34;
    t34[j] = t * i34;
    n12[j] = n * ile;
    t12[j] = t * ile;
  }
  const double cs2ld = (kCsSmag * kCsSmag) * (G.l_e[e] * G.d_e[e]);
  const double dtk = dt * cs2ld, fk = (G.l_e[e] * ide) * cs2ld;
  for (int k = lane; k < G.N; k += 32) {
    const double d34x = ux[Q[3] + k] - ux[Q[2] + k], d34y = uy[Q[3] + k] - uy[Q[2] + k],
                 d34z = uz[Q[3] + k] - uz[Q[2] + k];
    const double d12x = ux[Q[1] + k] - ux[Q[0] + k], d12y = uy[Q[1] + k] - uy[Q[0] + k],
                 d12z = uz[Q[1] + k] - uz[Q[0] + k];
    const double DT = fma(d34z, n34[2], fma(d34y, n34[1], d34x * n34[0])) -
                      fma(d12z, t12[2], fma(d12y, t12[1], d12x * t12[0]));
    const double DS = fma(d12z, n12[2], fma(d12y, n12[1], fma(d12x, n12[0],
                      fma(d34z, t34[2], fma(d34y, t34[1], d34x * t34[0])))));
    const double D = sqrt(fma(DS, DS, DT * DT));
    const double lap = (divc[c2 + k] - divc[c1 + k]) * ide - (zeta[v2 + k] - zeta[v1 + k]) * ile;
    double vnew = fma(dtk * D, lap, vn[e * ld + k]);
    if (bd.D1) {
      const double lap2 = (bd.D1[c2 + k] - bd.D1[c1 + k]) * ide - (bd.zeta1[v2 + k] - bd.zeta1[v1 + k]) * ile;
      vnew -= bd.scale * lap2;
    }
    vn[e * ld + k] = vnew;
    thflx[e * ld + k] = (fk * D) * (thv[c2 + k] - thv[c1 + k]);
  }
}

__global__ void __launch_bounds__(256) k_diff_theta(Geo64 G, const double* __restrict__ thflx, double* __restrict__ thv,
                                                    double* __restrict__ ex, double dt) {
  const int64_t c = warp_entity();
  if (c >= G.nc) return;
  const int lane = threadIdx.x & 31, ld = G.ld;
  int64_t E[3];
  double sg[3];
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    sg[s] = G.s_ce[3 * c + s];
  }
  const double dtA = dt * G.inv_Ac[c];
  for (int k = lane; k < G.N; k += 32) {
    double acc = 0.0;
    for (int s = 0; s < 3; ++s) acc += sg[s] * thflx[E[s] + k];
    const double dth = dtA * acc;
    const double th = thv[c * ld + k];
    ex[c * ld + k] = ex[c * ld + k] * (1.0 + ((kRd / kCvd) * dth) * recip64(th));
    thv[c * ld + k] = th + dth;
  }
}

Geo64 make_geo(const icon_grid* grid, const double* cc) {
  const GridDev& g = grid->g;
  const Vertical& v = grid->vert;
  Geo64 G;
  G.nc = g.nc; G.ne = g.ne; G.nv = g.nv; G.N = v.N; G.ld = v.ld;
  G.c2e = g.c2e; G.e2c = g.e2c; G.e2v = g.e2v; G.v2e = g.v2e; G.v2c = g.v2c; G.vdeg = g.vdeg;
  G.e2vt = g.e2vt; G.e2q = g.e2q;
  G.div_wa = g.div_wa; G.rot_wa = g.rot_wa; G.inv_Ac = g.inv_Ac; G.vt_w = g.vt_w; G.kin_w = g.kin_w;
  G.lsq_w = g.lsq_w; G.inv_de = g.inv_de; G.inv_le = g.inv_le; G.l_e = g.l_e; G.d_e = g.d_e; G.f_e = g.f_e;
  G.inv_L34 = g.inv_L34; G.n_e = g.n_e; G.t_e = g.t_e; G.s_ce = g.s_ce;
  G.wu = v.d_wu; G.wl = v.d_wl; G.inv_dz = v.d_inv_dz; G.inv_dz2 = v.d_inv_dz2; G.qinv_dz = v.d_qinv_dz;
  G.cc = cc;
  G.kin_w_h = G.div_wa_h = G.adv_w = nullptr;
  G.edge_c = G.lap_w = nullptr;
  G.merge_column = G.merge_stencil = false;
  G.t_hsn = G.t_bf = G.t_wu_e = G.t_qinv_dz_e = G.t_dz_e = nullptr;
  G.t_wu_c = G.t_inv_dz_c = G.t_inv_dzh_c = G.t_wcc = G.t_wcon = G.t_ep = G.t_hdpdz = nullptr;
  return G;
}

// Merged launches on small grids, whose kernels run 2 to 4 us, about what starting one takes: the
// column's three parts up to R2B2 (1,280 cells; R2B2/20 398 us a step with 90 launches, 356 merged,
// R2B2/60 791 and 724; on R2B3 the parts fill the SMs better apart, R2B3/30 765 us against 900,
// R2B3/90 2286 against 2887), vertices with edges up to R2B3 (R2B3/30 785 us apart, 765 merged).
constexpr int64_t kMergeColumnCells = 1280, kMergeStencilCells = 5120;

template <bool TOPO, bool CORR>
void launch_column_as(const Geo64& G, const ColArgs& a, cudaStream_t st) {
  if (G.merge_column) {
    k_col_small<TOPO, CORR><<<blocks_for(G.nc, kWarpsPerBlock), 256, 0, st>>>(G, a);
    return;
  }
  const unsigned nbc = blocks_for(G.nc, kWarpsPerBlock);
  k_col_rows<TOPO, CORR><<<nbc, 256, 0, st>>>(G, a);
  k_col_thomas<CORR><<<blocks_for(G.nc, 128), 128, 0, st>>>(G, a);
  k_col_update<TOPO, CORR><<<nbc, 256, 0, st>>>(G, a);
}

template <bool TOPO>
void launch_column(const Geo64& G, const ColArgs& a, bool corr, cudaStream_t st) {
  if (corr) launch_column_as<TOPO, true>(G, a, st);
  else launch_column_as<TOPO, false>(G, a, st);
}

}  // namespace

namespace {

Geo64 state_geo(const icon_state* st) {
  const StateDev& s = st->s;
  Geo64 G = make_geo(st->grid, s.colconst);
  G.kin_w_h = s.kin_w_h;
  G.div_wa_h = s.div_wa_h;
  G.adv_w = s.adv_w;
  G.edge_c = reinterpret_cast<const double4*>(s.edge_c);
  G.lap_w = reinterpret_cast<const double4*>(s.lap_w);
  // by the cells of the global grid, so that a decomposed domain's parts launch the kernels the
  // single domain does (its promise is the same bits)
  const double cells = 4.0 * M_PI * kR * kR / st->abar;
  G.merge_column = cells < kMergeColumnCells + 0.5;
  G.merge_stencil = cells < kMergeStencilCells + 0.5;
  const TopoDev& T = s.topo;
  if (T.on) {
    G.t_hsn = T.hsn; G.t_bf = T.bf; G.t_wu_e = T.wu_e; G.t_qinv_dz_e = T.qinv_dz_e; G.t_dz_e = T.dz_e;
    G.t_wu_c = T.wu_c; G.t_inv_dz_c = T.inv_dz_c; G.t_inv_dzh_c = T.inv_dzh_c;
    G.t_wcc = T.wcc; G.t_wcon = T.wcon; G.t_ep = T.ep; G.t_hdpdz = T.hdpdz;
  }
  return G;
}

}  // namespace

// the parts of one FP64 step, in the order enqueue_step_fp64 issues them; a decomposed
// domain issues them for every part with halo exchanges between the stages
void fp64_step_begin(icon_state* st, double dt, int nsub, cudaStream_t stream) {
  StateDev& s = st->s;
  const Vertical& vg = st->grid->vert;
  const double dtau = dt / nsub;
  k_colconst64<<<1, 128, 0, stream>>>(vg.N, vg.ld, vg.d_wu, vg.d_wl, vg.d_dzh, vg.d_dz, vg.d_ray, dtau, s.colconst);
  cudaMemsetAsync(s.mflx, 0, sizeof(double) * st->grid->g.ne * vg.ld, stream);
  cudaMemsetAsync(s.wflx, 0, sizeof(double) * st->grid->g.nc * vg.ld, stream);
}

void fp64_step_stage(icon_state* st, double dt, int nsub, bool corr, cudaStream_t stream) {
  StateDev& s = st->s;
  const Geo64 G = state_geo(st);
  const TopoDev& T = s.topo;
  const bool topo = T.on;
  const double dtau = dt / nsub;
  const unsigned nbv = blocks_for(G.nv, kWarpsPerBlock), nbe = blocks_for(G.ne, kWarpsPerBlock),
                 nbc = blocks_for(G.nc, kWarpsPerBlock);
  const double* vn_st = corr ? s.vn_s : s.vn;
  const double* w_st = corr ? s.w_s : s.w;
  const double* rho_st = corr ? s.rho_s : s.rho;
  const double* thv_st = corr ? s.thv_s : s.thv;
  const double* ex_st = corr ? s.ex_s : s.ex;
  prof_begin(stream, K_VERTEX);
  if (G.merge_stencil) {
    k_vertex_edge_vt<<<nbv + nbe, 256, 0, stream>>>(G, vn_st, w_st, s.zeta, s.w_v, s.vt, s.Ke, nbv);
  } else {
    k_vertex<<<nbv, 256, 0, stream>>>(G, vn_st, w_st, s.zeta, s.w_v);
    prof_end(stream);
    prof_begin(stream, K_EDGE_VT);
    k_edge_vt<<<nbe, 256, 0, stream>>>(G, vn_st, s.vt, s.Ke);
  }
  prof_end(stream);
  prof_begin(stream, K_CELL_KE);
  k_cell_ke<<<nbc, 256, 0, stream>>>(G, s.Ke, s.Kc);
  prof_end(stream);
  if (topo) topo_stage(st, vn_st, s.vt, w_st, ex_st, stream);
  EdgeArgs ea;
  ea.vn = vn_st; ea.w = w_st; ea.rho = rho_st; ea.thv = thv_st; ea.ex = ex_st;
  ea.vt = s.vt; ea.Kc = s.Kc; ea.zeta = s.zeta; ea.w_v = s.w_v;
  ea.vn_base = s.vn;
  ea.vn_out = corr ? s.vn : s.vn_s;
  ea.Avn0 = s.Avn0;
  ea.F = s.F; ea.G = s.G; ea.a_e = s.a_e; ea.mflx = s.mflx;
  ea.dtau = dtau; ea.corrector = corr;
  ea.hinv_nsub = 0.5 / nsub;
  ea.hdtau = 0.5 * dtau;
  const bool damp = corr && st->divdamp4 > 0.0;
  ea.skip_flux = damp ? 1 : 0;
  ea.upwind_theta = st->upwind_theta ? 1 : 0;
  prof_begin(stream, K_EDGE_TEND);
  if (topo) {
    if (ea.upwind_theta) k_edge_tend<true, true><<<nbe, 256, 0, stream>>>(G, ea);
    else k_edge_tend<true, false><<<nbe, 256, 0, stream>>>(G, ea);
  } else {
    if (ea.upwind_theta) k_edge_tend<false, true><<<nbe, 256, 0, stream>>>(G, ea);
    else k_edge_tend<false, false><<<nbe, 256, 0, stream>>>(G, ea);
  }
  prof_end(stream);
  if (damp) {
    // Kc and the column's update-operand scratch are free until the column runs
    const double abar = st->abar;
    DDArgs da;
    da.L = s.col_rx; da.rho = rho_st; da.thv = thv_st;
    da.vn = s.vn; da.F = s.F; da.G = s.G; da.mflx = s.mflx;
    da.dz_e = topo ? T.dz_e : nullptr;
    da.scale = st->divdamp4 * abar * abar; da.hinv_nsub = 0.5 / nsub;
    da.upwind_theta = st->upwind_theta ? 1 : 0;
    prof_begin(stream, K_DIVDAMP);
    k_dd_div<<<nbc, 256, 0, stream>>>(G, s.vn, s.Kc);
    k_dd_lap<<<nbc, 256, 0, stream>>>(G, s.Kc, s.col_rx);
    k_dd_edge<<<nbe, 256, 0, stream>>>(G, da);
    prof_end(stream);
  }
  ColArgs ca;
  ca.rho = s.rho; ca.thv = s.thv; ca.ex = s.ex; ca.w = s.w;
  ca.w_stage = w_st;
  ca.F = s.F; ca.G = s.G; ca.a_e = s.a_e;
  ca.ba = s.Aw0; ca.aa = s.col_ws;
  ca.lo = s.col_lo; ca.di = s.col_di; ca.up = s.col_up; ca.rh = s.col_rh;
  ca.rx = s.col_rx; ca.tx = s.col_tx; ca.dx = s.col_px; ca.gm = s.col_gm; ca.d0 = s.col_d0;
  ca.ri = s.col_ri; ca.mm = s.col_mm; ca.gc = s.col_gc;
  ca.rho_o = corr ? s.rho : s.rho_s;
  ca.thv_o = corr ? s.thv : s.thv_s;
  ca.ex_o = corr ? s.ex : s.ex_s;
  ca.w_o = corr ? s.w : s.w_s;
  ca.wflx = s.wflx;
  ca.status = s.status;
  ca.dtau = dtau; ca.hdtau = 0.5 * dtau; ca.inv_nsub = 1.0 / nsub;
  ca.hrc = 0.5 * dtau * (kRd / kCvd); ca.inv_dtau2 = 2.0 / dtau;
  ca.b_new = kBeta / nsub;
  ca.b_old = (1.0 - kBeta) / nsub;
  ca.hdamp = 0;
  const std::vector<double>& ray = st->grid->vert.rayleigh;
  for (int h = 0; h <= G.N; ++h)
    if (ray[h] > 0.0) ca.hdamp = h + 1;
  prof_begin(stream, K_COLUMN);
  if (topo) launch_column<true>(G, ca, corr, stream);
  else launch_column<false>(G, ca, corr, stream);
  prof_end(stream);
}

void fp64_step_diffusion(icon_state* st, double dt, cudaStream_t stream) {
  StateDev& s = st->s;
  const Geo64 G = state_geo(st);
  const unsigned nbv = blocks_for(G.nv, kWarpsPerBlock), nbe = blocks_for(G.ne, kWarpsPerBlock),
                 nbc = blocks_for(G.nc, kWarpsPerBlock);
  prof_begin(stream, K_DIFF_VERTEX);
  k_diff_vertex<<<nbv, 256, 0, stream>>>(G, s.vn, s.uvx, s.uvy, s.uvz, s.zeta);
  prof_end(stream);
  prof_begin(stream, K_DIFF_DIV);
  k_diff_div<<<nbc, 256, 0, stream>>>(G, s.vn, s.divc);
  prof_end(stream);
  BDArgs bd;
  bd.D1 = nullptr; bd.zeta1 = nullptr; bd.scale = 0.0;
  if (st->diff4 > 0.0) {
    // scratch that is dead during diffusion: a_e (edges), two column-scratch cell arrays
    const double abar = st->abar;
    prof_begin(stream, K_DIFF4);
    k_bd_lap<<<nbe, 256, 0, stream>>>(G, s.zeta, s.divc, s.a_e);
    k_bd_curl<<<nbv, 256, 0, stream>>>(G, s.a_e, s.col_di);
    k_diff_div<<<nbc, 256, 0, stream>>>(G, s.a_e, s.col_lo);
    prof_end(stream);
    bd.D1 = s.col_lo; bd.zeta1 = s.col_di; bd.scale = st->diff4 * abar * abar;
  }
  prof_begin(stream, K_DIFF_EDGE);
  k_diff_edge<<<nbe, 256, 0, stream>>>(G, s.vn, s.uvx, s.uvy, s.uvz, s.zeta, s.divc, s.thv, s.thflx, dt, bd);
  prof_end(stream);
  prof_begin(stream, K_DIFF_THETA);
  k_diff_theta<<<nbc, 256, 0, stream>>>(G, s.thflx, s.thv, s.ex, dt);
  prof_end(stream);
}

void enqueue_step_fp64(icon_state* st, double dt, int nsub, cudaStream_t stream) {
  fp64_step_begin(st, dt, nsub, stream);
  for (int it = 0; it < nsub; ++it)
    for (int stage = 0; stage < 2; ++stage) fp64_step_stage(st, dt, nsub, stage == 1, stream);
  fp64_step_diffusion(st, dt, stream);
}

}  // namespace icon
