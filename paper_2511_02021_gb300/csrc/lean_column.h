// The per-state launches of the lean mixed column (included by dycore32.cu, inside its
// unnamed namespace): two forms of the same arithmetic.
//
//   k_mx_lean_column  one column per thread, both sweeps in the thread. What bounds it: the
//     FP64 pipe (one warp instruction per SM every 16 cycles, and no warp more than one every
//     64, dependent or not: measured), the HBM traffic of two sweeps (147 B per cell-level) and
//     the latency of the loads, which walk the column level by level. So each level's operands
//     are loaded one or two levels ahead into registers, through one restrict pointer per array
//     (the loop's own stores then order nothing), with 20 warps per SM at 102 registers rather
//     than 36 at 56 with the loads waited for.
//   k_mx_lean_tile    one block per 32 columns: the rows and the updates, which only need
//     neighbouring levels, are spread over the block's warps by runs of levels; one warp walks
//     the 32 columns in shared memory. A column's serial chain is then three FP64 operations per
//     level (elimination two, substitution one) instead of every operation of the level. It wins
//     while the grid has too few columns to fill the SMs with threads.
//
// Measured on a GB300 (us per launch, predictor / corrector; before: one thread per column, nine
// blocks of 128 per SM, loads in order, with the shape the tuner then picked for the predictor):
//     columns x levels          before      column       tile
//     1,280 x 60                88 / 103    60 / 72      23 / 25
//     20,480 x 60              125 / 183    82 / 97      53 / 72
//     81,920 x 47              167 / 211   130 / 155    134 / 190
//     81,920 x 90              320 / 403   250 / 295    273 / 397
//     327,680 x 90            1058 / 1159  954 / 1074  1047 / 1479
//     81,920 x 90, terrain     449 / 546   390 / 394    490 / 639
// Which one a state runs: lean_rule.h.
//
// Both forms, at every shape, give the same bits: which of two products is rounded before the
// multiply-add that takes the other is written out, not left to how the compiler contracts a
// loop it has unrolled.

// (Rd/cvd) pi / (rho theta_v)
__device__ __forceinline__ float lean_g(double ex, float rhof, float thvf) {
  return __fmul_rn(kRcvF, __fdividef(f64_to_f32(ex), __fmul_rn(rhof, thvf)));
}
// a b - c d with one product rounded before the subtraction: the second (FIRST) or the first. Results
// are defined by the loop these forms replaced, whose body was unrolled by two and in which the
// compiler fused one product at even steps of a sweep and the other at odd ones: the upward sweep
// below takes its levels in the same pairs (ODD), and so does the last row of the corrector, whose
// difference of Exner increments was fused when the row fell on the pair's first step (even N).
template <bool FIRST>
__device__ __forceinline__ float fma_diff(float a, float b, float c, float d) {
  return FIRST ? __fmaf_rn(a, b, -__fmul_rn(c, d)) : __fmaf_rn(-c, d, __fmul_rn(a, b));
}


// one column per thread (lane); every lane of the warp runs the loops (lanes past the last cell
// compute on cell 0 and store nothing) so that the chunk flushes stay warp-synchronous.
// AHEAD: levels loaded ahead (two on flat levels; one over terrain, whose four more tables per
// level would spill). Blocks of two warps: finer than four, and no slower at any size.
// TOPO (terrain-following levels): each cell's interpolation weights, 1/dz and 1/dzh and
// reference Exner (level-major tables) in place of the per-level constants, the contravariant
// (1 - beta) w - wcc in the explicit vertical fluxes (zero at the lid and the ground), the
// gathered divergences scaled by the cell's 1/dz, and the stage's terrain-following w at the
// ground
constexpr int kLeanThreads = 64, kLeanBlocks = 10;
template <bool CORR, bool TOPO, int AHEAD>
__global__ void __launch_bounds__(kLeanThreads, kLeanBlocks) k_mx_lean_column(MxGeo G, MxLeanArgs a) {
  constexpr int CH = 8, THREADS = kLeanThreads;
  __shared__ LeanTile<CH> Ts[THREADS / 32];
  const int N = G.N, ld = G.ld;
  const int64_t nc = G.nc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * THREADS + warp * 32, c = c0 + lane;
  if (c0 >= nc) return;
  LeanTile<CH>& T = Ts[warp];
  const bool act = c < nc;
  const int64_t cc = act ? c : 0;
  const double* __restrict__ cd = a.cd;
  const float* __restrict__ cf = a.cf;
  const double dtau = a.dtau;
  double* __restrict__ rhoP = a.rho;
  double* __restrict__ thvP = a.thv;
  double* __restrict__ exP = a.ex;
  double* __restrict__ wP = a.w;
  double* __restrict__ wflxP = a.wflx;
  double* __restrict__ BP = a.B;
  const double* __restrict__ dr64P = a.dr64;
  const float* __restrict__ dr32P = a.dr32;
  const float* __restrict__ dt32P = a.dt32;
  const float* __restrict__ aw32P = a.aw32;
  const double* __restrict__ wuP = a.t_wu_lm;
  const double* __restrict__ idzP = a.t_idz_lm;
  const double* __restrict__ idzhP = a.t_idzh_lm;
  const double* __restrict__ exrefP = a.t_exref_lm;
  double* __restrict__ dpP = a.dp;
  float* __restrict__ cpP = a.cp;
  const float* __restrict__ wccP = a.t_wcc + (TOPO ? cc * ld : 0);
#define LMV(p, k) (p)[(int64_t)(k) * nc + cc]
  // ---- downward sweep: at step j half level j becomes known, completing full level k = j - 1
  // and, for k >= 1, the row of half level h = k, which is eliminated at once
  {
    double dp_prev = 0.0, thv1 = 0.0, ex1 = 0.0, ti1 = 0.0, w1 = 0.0, ex2 = 0.0;
    float rho1f = 0.f, thv1f = 0.f, ti1f = 0.f, M1 = 0.f, M2 = 0.f, xv1 = 0.f, gam2 = 0.f, dpe2 = 0.f, cp_prev = 0.f;
    struct Lev {
      double rho, thv, ex, w, B, wu, idz, idzh;
      float dt, aw, wcc;
    };
    auto fetch = [&](int j) {
      Lev v;
      const bool full = j < N, half = j >= 1 && full, row = j >= 2 && j <= N;
      v.rho = full ? LMV(rhoP, j) : 0.0;
      v.thv = full ? LMV(thvP, j) : 0.0;
      v.ex = full ? LMV(exP, j) : 0.0;
      v.w = half ? LMV(wP, j) : 0.0;
      v.dt = j >= 1 && j <= N ? LMV(dt32P, j - 1) : 0.0f;
      v.aw = row ? LMV(aw32P, j - 1) : 0.0f;
      v.B = CORR && row ? LMV(BP, j - 1) : 0.0;
      if constexpr (TOPO) {
        v.wcc = half ? wccP[j] : 0.0f;
        v.wu = half ? LMV(wuP, j) : 0.0;
        v.idz = j >= 1 && j <= N ? LMV(idzP, j - 1) : 0.0;
        v.idzh = row ? LMV(idzhP, j - 1) : 0.0;
      }
      return v;
    };
    auto step = [&](int j, const Lev& v) {
      const double rho = v.rho, thv = v.thv, ex = v.ex;
      const float rhof = f64_to_f32(rho), thvf = f64_to_f32(thv);
      double ti = 0.0;
      float rif, tif;
      if (j == 0) {
        ti = thv;
        rif = rhof;
        tif = thvf;
      } else if (j == N) {
        ti = thv1;
        rif = rho1f;
        tif = thv1f;
      } else {
        float wu, wl;
        double wud = 0.0, wld = 0.0;
        if constexpr (TOPO) {
          wud = v.wu;
          wu = f64_to_f32(wud);
          wl = 1.0f - wu;
          if (!CORR) wld = 1.0 - wud;
        } else {
          wu = cf[LF_WU * ld + j];
          wl = cf[LF_WL * ld + j];
          if (!CORR) {
            wud = cd[LD_WU * ld + j];
            wld = cd[LD_WL * ld + j];
          }
        }
        rif = __fmaf_rn(wu, rho1f, __fmul_rn(wl, rhof));
        if (!CORR) {
          ti = __fma_rn(wud, thv1, __dmul_rn(wld, thv));
          tif = f64_to_f32(ti);
        } else {
          tif = TOPO ? __fmaf_rn(wu, thv1f, __fmul_rn(wl, thvf)) : __fmaf_rn(wl, thvf, __fmul_rn(wu, thv1f));
        }
      }
      const float Mh = __fmul_rn(rif, tif);
      const double wh = v.w;
      float xvj = f64_to_f32(wh);
      if constexpr (TOPO) xvj = (j == 0 || j == N) ? 0.0f : __fmaf_rn((float)(1.0 - kBeta), xvj, -v.wcc);
      float gam1 = 0.f, dpe1 = 0.f;
      if (j >= 1) {
        const int k = j - 1;
        const float dtk = v.dt;
        float dt1, dtb, dthe;
        if constexpr (TOPO) {
          const double idz = v.idz;
          dt1 = f64_to_f32(dtau * idz);
          dtb = f64_to_f32(dtau * kBeta * idz);
          dthe = __fmaf_rn(-dtk, f64_to_f32(idz), -__fmul_rn(dt1, fma_diff<true>(M1, xv1, Mh, xvj)));
        } else {
          dt1 = cf[LF_DT1 * ld + k];
          dtb = cf[LF_DTB * ld + k];
          dthe = __fmaf_rn(-dt1, fma_diff<true>(M1, xv1, Mh, xvj), -dtk);
        }
        const float g = lean_g(ex1, rho1f, thv1f);
        gam1 = __fmul_rn(g, dtb);
        dpe1 = __fmul_rn(g, dthe);
        if (j > 1) {
          const int h = k;
          double cpdzh;
          float ca;
          if constexpr (TOPO) {
            const double idzh = v.idzh;
            cpdzh = kCpd * idzh;
            ca = f64_to_f32(dtau * kBeta * kCpd * idzh);
          } else {
            cpdzh = cd[LD_CPDZH * ld + h];
            ca = cf[LF_CA * ld + h];
          }
          const float aa = __fmul_rn(ca, ti1f);
          double B;
          if (!CORR) {
            B = __fma_rn(-dtau, __fma_rn(__dmul_rn(cpdzh, ti1), ex2 - ex1, kGrav), w1);
            if (act) LMV(BP, h) = B;
          } else {
            B = v.B;
          }
          // an even N's last row as the unrolled loop rounded it (see fma_diff)
          const float dd = (CORR && j == N && (N & 1) == 0) ? __fmaf_rn(-g, dthe, dpe2) : __fsub_rn(dpe2, dpe1);
          const float inc = __fmaf_rn(-aa, dd, v.aw);
          const float lo = __fmul_rn(__fmul_rn(-aa, gam2), M2);
          const float di = __fmaf_rn(__fmul_rn(aa, __fadd_rn(gam2, gam1)), M1, 1.0f);
          const float up = __fmul_rn(__fmul_rn(-aa, gam1), Mh);
          const float piv = __fdividef(1.0f, __fmaf_rn(-lo, cp_prev, di));
          cp_prev = __fmul_rn(up, piv);
          dp_prev = __dmul_rn(__fma_rn(-f32_to_f64(lo), dp_prev, B + f32_to_f64(inc)), f32_to_f64(piv));
          if (act) {
            LMV(dpP, h) = dp_prev;
            LMV(cpP, h) = cp_prev;
          }
        }
      }
      gam2 = gam1;
      dpe2 = dpe1;
      M2 = M1;
      M1 = Mh;
      w1 = wh;
      xv1 = xvj;
      ti1 = ti;
      ti1f = tif;
      ex2 = ex1;
      ex1 = ex;
      thv1 = thv;
      rho1f = rhof;
      thv1f = thvf;
    };

    if constexpr (AHEAD == 1) {
      Lev a0 = fetch(0);
#pragma unroll 2
      for (int j = 0; j <= N; ++j) {
        const Lev b0 = fetch(j + 1);
        step(j, a0);
        a0 = b0;
      }
    } else {
      Lev a0 = fetch(0), a1 = fetch(1);
#pragma unroll 1
      for (int j = 0; j <= N; j += 2) {
        const Lev b0 = fetch(j + 2);
        step(j, a0);
        const Lev b1 = fetch(j + 3);
        if (j < N) step(j + 1, a1);
        a0 = b0;
        a1 = b1;
      }
    }
  }
  // ---- upward sweep: back substitution, damping and the update of full level k, between half
  // levels k and k + 1
  bool ok = true;
  {
    double x_next = 0.0;
    float xv_n = 0.f, fk_n = 0.f, wnf_n = 0.f;
    struct Lev {
      double rho, thv, ex, w, wflx, dr64, dp, wu, idz, exref;
      float dt, dr32, cp, wcc;
    };
    auto fetch = [&](int k) {
      Lev v;
      const bool in = k >= 0, half = k >= 1;
      v.rho = in ? LMV(rhoP, k) : 0.0;
      v.thv = in ? LMV(thvP, k) : 0.0;
      v.ex = in ? LMV(exP, k) : 0.0;
      v.w = half ? LMV(wP, k) : 0.0;
      v.dp = half ? LMV(dpP, k) : 0.0;
      v.cp = half ? LMV(cpP, k) : 0.0f;
      v.dt = in ? LMV(dt32P, k) : 0.0f;
      v.dr32 = !CORR && in ? LMV(dr32P, k) : 0.0f;
      v.dr64 = CORR && in ? LMV(dr64P, k) : 0.0;
      v.wflx = CORR && in ? LMV(wflxP, k) : 0.0;
      if constexpr (TOPO) {
        v.wcc = half ? wccP[k] : 0.0f;
        v.wu = half ? LMV(wuP, k) : 0.0;
        v.idz = in ? LMV(idzP, k) : 0.0;
        v.exref = in ? LMV(exrefP, k) : 0.0;
      }
      return v;
    };
    Lev a0 = fetch(N - 1), a1 = fetch(N - 2);
    double rho_k = a0.rho, thv_k = a0.thv;
    float rho_kf = f64_to_f32(rho_k), thv_kf = f64_to_f32(thv_k);
    float ri_n = rho_kf, M_n = __fmul_rn(rho_kf, thv_kf);
    auto level = [&](int k, const Lev& v, const Lev& u, auto odd) {
      constexpr bool ODD = decltype(odd)::value;
      const double rho_u = u.rho, thv_u = u.thv;
      const float rho_uf = f64_to_f32(rho_u), thv_uf = f64_to_f32(thv_u);
      const double ex_k = v.ex, w_k = v.w;
      double x = 0.0, wn = 0.0;
      if (k >= 1) {
        x = __fma_rn(-f32_to_f64(v.cp), x_next, v.dp);
        wn = k < a.hdamp ? x * cd[LD_DAMP * ld + k] : x;
      }
      x_next = x;
      const float dtk = v.dt;
      float ri_k, M_k;
      if (k == 0) {
        ri_k = rho_kf;
        M_k = __fmul_rn(rho_kf, thv_kf);
      } else if constexpr (TOPO) {
        const float wu = f64_to_f32(v.wu), wl = 1.0f - wu;
        ri_k = __fmaf_rn(wu, rho_uf, __fmul_rn(wl, rho_kf));
        M_k = __fmul_rn(ri_k, __fmaf_rn(wu, thv_uf, __fmul_rn(wl, thv_kf)));
      } else {
        const float wu = cf[LF_WU * ld + k], wl = cf[LF_WL * ld + k];
        ri_k = __fmaf_rn(wl, rho_kf, __fmul_rn(wu, rho_uf));
        M_k = __fmul_rn(ri_k, __fmaf_rn(wl, thv_kf, __fmul_rn(wu, thv_uf)));
      }
      const float wf_k = f64_to_f32(w_k);
      float xv_k = wf_k;
      if constexpr (TOPO) xv_k = k >= 1 ? __fmaf_rn((float)(1.0 - kBeta), wf_k, -v.wcc) : 0.0f;
      const float wnf = f64_to_f32(wn);
      float dtb, dt1, dthe, idzf = 1.0f;
      double idz = 0.0, exref;
      const float D = fma_diff<ODD>(M_k, xv_k, M_n, xv_n);
      if constexpr (TOPO) {
        idz = v.idz;
        idzf = f64_to_f32(idz);
        dt1 = f64_to_f32(dtau * idz);
        dtb = f64_to_f32(dtau * kBeta * idz);
        exref = v.exref;
        dthe = __fmaf_rn(-dtk, idzf, -__fmul_rn(dt1, D));
      } else {
        dtb = cf[LF_DTB * ld + k];
        dt1 = cf[LF_DT1 * ld + k];
        exref = cd[LD_EXREF * ld + k];
        dthe = __fmaf_rn(-dt1, D, -dtk);
      }
      const float g = lean_g(ex_k, rho_kf, thv_kf);
      const float q = fma_diff<ODD>(M_k, wnf, M_n, wnf_n);
      const float dTh = __fmaf_rn(-dtb, q, dthe);
      const float dex = fma_diff<true>(g, dthe, __fmul_rn(g, dtb), q);
      float s_rho, s_thv, s_exp;
      if (!CORR) {
        const float drk = v.dr32;
        const float Xe = fma_diff<ODD>(ri_k, xv_k, ri_n, xv_n), Xi = fma_diff<ODD>(ri_k, wnf, ri_n, wnf_n);
        const float t = TOPO ? __fmaf_rn(-drk, idzf, -__fmul_rn(dt1, Xe)) : __fmaf_rn(-dt1, Xe, -drk);
        const float drho = __fmaf_rn(-dtb, Xi, t);
        s_rho = __fadd_rn(rho_kf, drho);
        s_thv = thv_kf + __fdividef(__fmaf_rn(-drho, thv_kf, dTh), s_rho);
        s_exp = __fadd_rn(f64_to_f32(ex_k - exref), dex);
        ok = ok && isfinite(s_thv) && isfinite(s_exp) && isfinite(wnf);
      } else {
        double t;
        float fk;
        if constexpr (TOPO) {
          fk = __fmul_rn(ri_k, __fmaf_rn((float)kBeta, wnf, xv_k));
          t = __fma_rn(dtau * idz, f32_to_f64(fk) - f32_to_f64(fk_n), __dmul_rn(v.dr64, idz));
        } else {
          fk = __fmul_rn(ri_k, __fmaf_rn((float)(1.0 - kBeta), wf_k, __fmul_rn((float)kBeta, wnf)));
          t = __fma_rn(cd[LD_IDZ * ld + k], f32_to_f64(fk) - f32_to_f64(fk_n), v.dr64);
        }
        const double rho_n = rho_k - t;
        const float rho_nf = f64_to_f32(rho_n);
        const double thv_n = thv_k + f32_to_f64(__fdividef(__fmaf_rn(f64_to_f32(t), thv_kf, dTh), rho_nf));
        const double ex_n = ex_k + f32_to_f64(dex);
        if (act) {
          LMV(wflxP, k) = __fma_rn(f32_to_f64(fk), a.inv_nsub, v.wflx);
          LMV(rhoP, k) = rho_n;
          LMV(thvP, k) = thv_n;
          LMV(exP, k) = ex_n;
          LMV(wP, k) = wn;
        }
        s_rho = rho_nf;
        s_thv = f64_to_f32(thv_n);
        s_exp = f64_to_f32(ex_n - exref);
        ok = ok && finite64(thv_n) && finite64(ex_n) && finite64(wn);
        fk_n = fk;
      }
      const int k0 = k & ~(CH - 1);
      T.t[0][k - k0][lane] = s_rho;
      T.t[1][k - k0][lane] = s_thv;
      T.t[2][k - k0][lane] = s_exp;
      T.t[3][k - k0][lane] = wnf;
      if (k == k0) lean_flush(G, a, T, c0, k0, lane);
      wnf_n = wnf;
      ri_n = ri_k;
      M_n = M_k;
      xv_n = xv_k;
      rho_k = rho_u;
      thv_k = thv_u;
      rho_kf = rho_uf;
      thv_kf = thv_uf;
    };

    if constexpr (AHEAD == 1) {
#pragma unroll 1
      for (int k = N - 1; k >= 0; k -= 2) {
        const Lev b0 = fetch(k - 2);
        level(k, a0, a1, std::false_type{});
        const Lev b1 = fetch(k - 3);
        if (k > 0) level(k - 1, a1, b0, std::true_type{});
        a0 = b0;
        a1 = b1;
      }
    } else {
#pragma unroll 1
      for (int k = N - 1; k >= 0; k -= 2) {
        const Lev b0 = fetch(k - 2), b1 = fetch(k - 3);
        level(k, a0, a1, std::false_type{});
        if (k > 0) level(k - 1, a1, b0, std::true_type{});
        a0 = b0;
        a1 = b1;
      }
    }
  }
  if (act) {
    if constexpr (TOPO) {                                  // the ground: the stage's terrain-following w
      const float wg = wccP[N];
      a.w32[c * ld + N] = wg;
      if (CORR) LMV(wP, N) = f32_to_f64(wg);
    } else {
      a.w32[c * ld + N] = 0.0f;
      if (CORR) LMV(wP, N) = 0.0;                          // the ground (w^n there is 0 already)
    }
  }
  if (!ok && act) atomicOr(a.status, 1u);
#undef LMV
}

// one block of W warps per 32 columns; 660 (over terrain 792) bytes of shared memory per level.
// Rows and updates are split into one run of levels per warp; a run starts two rows early to
// have its neighbours' half levels (two steps more per run, instead of an exchange and a
// barrier). The warp that walks the columns changes with the block, so that the walks of the
// resident blocks spread over the SM's schedulers. W and the register budget: eight warps and
// 128 registers while a block has an SM to itself or nearly so (1,280 x 60: 23 us against 29
// with four warps), four warps and 102 registers when several share it.
template <bool CORR, bool TOPO, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) k_mx_lean_tile(MxGeo G, MxLeanArgs a) {
  extern __shared__ double lean_sm[];
  const int N = G.N, ld = G.ld;
  const int64_t nc = G.nc;
  constexpr int PT = kLeanPitch;
  double* const X = lean_sm;                               // right-hand side, dp, then w^{n+1}
  float* const P = reinterpret_cast<float*>(X + N * PT);   // sub-diagonal, then rho
  float* const Q = P + N * PT;                             // diagonal, then theta_v
  float* const R = Q + N * PT;                             // super-diagonal, cp, then pi - pi_ref
  float* const WC = R + N * PT;                            // TOPO: wcc of the tile
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * 32, c = c0 + lane;
  const bool act = c < nc;
  const int64_t cc = act ? c : 0;
  const double* __restrict__ cd = a.cd;
  const float* __restrict__ cf = a.cf;
  const double dtau = a.dtau;
  const int serial = blockIdx.x % W;                       // the warp that walks the columns
  // every array through a restrict pointer of its own: the next level's loads may pass this
  // level's stores (the in-place updates touch each element once, after its only reads)
  double* __restrict__ rhoP = a.rho;
  double* __restrict__ thvP = a.thv;
  double* __restrict__ exP = a.ex;
  double* __restrict__ wP = a.w;
  double* __restrict__ wflxP = a.wflx;
  double* __restrict__ BP = a.B;
  const double* __restrict__ dr64P = a.dr64;
  const float* __restrict__ dr32P = a.dr32;
  const float* __restrict__ dt32P = a.dt32;
  const float* __restrict__ aw32P = a.aw32;
  const double* __restrict__ wuP = a.t_wu_lm;
  const double* __restrict__ idzP = a.t_idz_lm;
  const double* __restrict__ idzhP = a.t_idzh_lm;
  const double* __restrict__ exrefP = a.t_exref_lm;
#define LMV(p, k) (p)[(int64_t)(k) * nc + cc]
  if constexpr (TOPO) {
    for (int r = warp; r < 32; r += W)
      for (int k = lane; k <= N; k += 32) WC[k * PT + r] = c0 + r < nc ? a.t_wcc[(c0 + r) * ld + k] : 0.0f;
    __syncthreads();
  }
  // ---- rows of the interior half levels, a run of them per warp
  {
    const int ch = (N - 1 + W - 1) / W;
    const int h0 = 1 + warp * ch, h1 = h0 + ch < N ? h0 + ch : N;
    if (h0 < h1) {
      double thv1 = 0.0, ex1 = 0.0, ti1 = 0.0, w1 = 0.0, ex2 = 0.0;
      float rho1f = 0.f, thv1f = 0.f, ti1f = 0.f, M1 = 0.f, M2 = 0.f, xv1 = 0.f, gam2 = 0.f, dpe2 = 0.f;
      if (h0 >= 2) {
        thv1 = LMV(thvP, h0 - 2);
        thv1f = f64_to_f32(thv1);
        rho1f = f64_to_f32(LMV(rhoP, h0 - 2));
      }
      // the loads of the next two levels are in flight while these two are computed
      struct Lev {
        double rho, thv, ex, w, B;
        float dt, aw;
      };
      auto fetch = [&](int j) {
        Lev v;
        const bool full = j < N && j <= h1, half = j >= 1 && full, row = j - 1 >= h0 && j <= h1;
        v.rho = full ? LMV(rhoP, j) : 0.0;
        v.thv = full ? LMV(thvP, j) : 0.0;
        v.ex = full ? LMV(exP, j) : 0.0;
        v.w = half ? LMV(wP, j) : 0.0;
        v.dt = j >= h0 && j <= h1 ? LMV(dt32P, j - 1) : 0.0f;
        v.aw = row ? LMV(aw32P, j - 1) : 0.0f;
        v.B = CORR && row ? LMV(BP, j - 1) : 0.0;
        return v;
      };
      auto step = [&](int j, const Lev& v) {
        const double rho = v.rho, thv = v.thv, ex = v.ex;
        const float rhof = f64_to_f32(rho), thvf = f64_to_f32(thv);
        double ti = 0.0;
        float rif, tif;
        if (j == 0) {
          ti = thv;
          rif = rhof;
          tif = thvf;
        } else if (j == N) {
          ti = thv1;
          rif = rho1f;
          tif = thv1f;
        } else {
          float wu, wl;
          double wud = 0.0, wld = 0.0;
          if constexpr (TOPO) {
            wud = LMV(wuP, j);
            wu = f64_to_f32(wud);
            wl = 1.0f - wu;
            if (!CORR) wld = 1.0 - wud;
          } else {
            wu = cf[LF_WU * ld + j];
            wl = cf[LF_WL * ld + j];
            if (!CORR) {
              wud = cd[LD_WU * ld + j];
              wld = cd[LD_WL * ld + j];
            }
          }
          rif = __fmaf_rn(wu, rho1f, __fmul_rn(wl, rhof));
          if (!CORR) {
            ti = __fma_rn(wud, thv1, __dmul_rn(wld, thv));
            tif = f64_to_f32(ti);
          } else {
            tif = TOPO ? __fmaf_rn(wu, thv1f, __fmul_rn(wl, thvf)) : __fmaf_rn(wl, thvf, __fmul_rn(wu, thv1f));
          }
        }
        const float Mh = __fmul_rn(rif, tif);
        const double wh = v.w;
        float xvj = f64_to_f32(wh);
        if constexpr (TOPO) xvj = (j == 0 || j == N) ? 0.0f : __fmaf_rn((float)(1.0 - kBeta), xvj, -WC[j * PT + lane]);
        float gam1 = 0.f, dpe1 = 0.f;
        if (j >= h0) {
          const int k = j - 1;
          const float dtk = v.dt;
          float dt1, dtb, dthe;
          if constexpr (TOPO) {
            const double idz = LMV(idzP, k);
            dt1 = f64_to_f32(dtau * idz);
            dtb = f64_to_f32(dtau * kBeta * idz);
            dthe = __fmaf_rn(-dtk, f64_to_f32(idz), -__fmul_rn(dt1, fma_diff<true>(M1, xv1, Mh, xvj)));
          } else {
            dt1 = cf[LF_DT1 * ld + k];
            dtb = cf[LF_DTB * ld + k];
            dthe = __fmaf_rn(-dt1, fma_diff<true>(M1, xv1, Mh, xvj), -dtk);
          }
          const float g = lean_g(ex1, rho1f, thv1f);
          gam1 = __fmul_rn(g, dtb);
          dpe1 = __fmul_rn(g, dthe);
          if (j > h0) {
            const int h = k;
            double cpdzh;
            float ca;
            if constexpr (TOPO) {
              const double idzh = LMV(idzhP, h);
              cpdzh = kCpd * idzh;
              ca = f64_to_f32(dtau * kBeta * kCpd * idzh);
            } else {
              cpdzh = cd[LD_CPDZH * ld + h];
              ca = cf[LF_CA * ld + h];
            }
            const float aa = __fmul_rn(ca, ti1f);
            double B;
            if (!CORR) {
              B = __fma_rn(-dtau, __fma_rn(__dmul_rn(cpdzh, ti1), ex2 - ex1, kGrav), w1);
              if (act) LMV(BP, h) = B;
            } else {
              B = v.B;
            }
            // an even N's last row as the unrolled loop rounded it (see fma_diff)
            const float dd = (CORR && j == N && (N & 1) == 0) ? __fmaf_rn(-g, dthe, dpe2) : __fsub_rn(dpe2, dpe1);
            const float inc = __fmaf_rn(-aa, dd, v.aw);
            const int i = h * PT + lane;
            P[i] = __fmul_rn(__fmul_rn(-aa, gam2), M2);
            Q[i] = __fmaf_rn(__fmul_rn(aa, __fadd_rn(gam2, gam1)), M1, 1.0f);
            R[i] = __fmul_rn(__fmul_rn(-aa, gam1), Mh);
            X[i] = B + f32_to_f64(inc);
          }
        }
        gam2 = gam1;
        dpe2 = dpe1;
        M2 = M1;
        M1 = Mh;
        w1 = wh;
        xv1 = xvj;
        ti1 = ti;
        ti1f = tif;
        ex2 = ex1;
        ex1 = ex;
        thv1 = thv;
        rho1f = rhof;
        thv1f = thvf;
      };
      Lev a0 = fetch(h0 - 1), a1 = fetch(h0);
#pragma unroll 1
      for (int j = h0 - 1; j <= h1; j += 2) {
        const Lev b0 = fetch(j + 2), b1 = fetch(j + 3);
        step(j, a0);
        if (j < h1) step(j + 1, a1);
        a0 = b0;
        a1 = b1;
      }
    }
  }
  // ---- the run of full levels this warp updates, top of the run last: an even count from the
  // ground up; what it needs of its neighbours' levels is read before they are updated
  const int cu = ((N + W - 1) / W + 1) & ~1;
  const int kt = N - 1 - warp * cu;                        // lowest level of the run
  const int kb = kt - cu + 1 > 0 ? kt - cu + 1 : 0;        // highest level of the run
  float rho_lf = 0.f, thv_lf = 0.f, wf_l = 0.f;            // level kt + 1, half level kt + 1
  float rho_uf0 = 0.f, thv_uf0 = 0.f;                      // level kb - 1
  if (kt >= 0) {
    const int kl = kt + 1 < N ? kt + 1 : N - 1;
    rho_lf = f64_to_f32(LMV(rhoP, kl));
    thv_lf = f64_to_f32(LMV(thvP, kl));
    if (kt + 1 < N) wf_l = f64_to_f32(LMV(wP, kt + 1));
    if (kb > 0) {
      rho_uf0 = f64_to_f32(LMV(rhoP, kb - 1));
      thv_uf0 = f64_to_f32(LMV(thvP, kb - 1));
    }
  }
  __syncthreads();
  // ---- elimination and back substitution, one warp, one column per lane
  if (warp == serial) {
    // the FP32 factor of the next row is formed between the two dependent FP64 operations of
    // this one
    double dp = 0.0, x0 = X[PT + lane], lo64 = f32_to_f64(P[PT + lane]);
    float piv = __fdividef(1.0f, __fmaf_rn(-P[PT + lane], 0.0f, Q[PT + lane]));
    float cp = __fmul_rn(R[PT + lane], piv);
#pragma unroll 2
    for (int h = 1; h < N; ++h) {
      const int i = h * PT + lane, n = h + 1 < N ? i + PT : i;
      const double t = __fma_rn(-lo64, dp, x0);
      const double piv64 = f32_to_f64(piv);
      R[i] = cp;
      const float lo_n = P[n];
      const float di_n = Q[n], up_n = R[n];
      x0 = X[n];
      piv = __fdividef(1.0f, __fmaf_rn(-lo_n, cp, di_n));
      cp = __fmul_rn(up_n, piv);
      dp = __dmul_rn(t, piv64);
      lo64 = f32_to_f64(lo_n);
      X[i] = dp;
    }
    double x = 0.0, d0 = dp, c64 = f32_to_f64(R[(N - 1) * PT + lane]);
#pragma unroll 2
    for (int h = N - 1; h >= 1; --h) {
      const int i = h * PT + lane, n = h > 1 ? i - PT : i;
      x = __fma_rn(-c64, x, d0);
      d0 = X[n];
      c64 = f32_to_f64(R[n]);
      X[i] = x;
    }
    X[lane] = 0.0;                                         // the lid
  }
  __syncthreads();
  // ---- updates of the full levels; Rayleigh damping of w, whose half level below the run is
  // read before its own warp damps it in place
  auto damped = [&](double x, int h) { return h < a.hdamp ? x * cd[LD_DAMP * ld + h] : x; };
  float wnf_n = kt >= 0 && kt + 1 < N ? f64_to_f32(damped(X[(kt + 1) * PT + lane], kt + 1)) : 0.0f;
  __syncthreads();
  bool ok = true;
  if (kt >= 0) {
    // half level kt + 1
    float ri_n, M_n, xv_n = 0.f, fk_n = 0.f;
    // the loads of the next two levels are in flight while these two are computed
    struct Lev {
      double rho, thv, ex, w, wflx, dr64;
      float dt, dr32;
    };
    auto fetch = [&](int k) {
      Lev v;
      const bool in = k >= kb;
      v.rho = in ? LMV(rhoP, k) : 0.0;
      v.thv = in ? LMV(thvP, k) : 0.0;
      v.ex = in ? LMV(exP, k) : 0.0;
      v.w = in && k >= 1 ? LMV(wP, k) : 0.0;
      v.dt = in ? LMV(dt32P, k) : 0.0f;
      v.dr32 = !CORR && in ? LMV(dr32P, k) : 0.0f;
      v.dr64 = CORR && in ? LMV(dr64P, k) : 0.0;
      v.wflx = CORR && in ? LMV(wflxP, k) : 0.0;
      return v;
    };
    Lev a0 = fetch(kt), a1 = fetch(kt - 1);
    double rho_k = a0.rho, thv_k = a0.thv;
    float rho_kf = f64_to_f32(rho_k), thv_kf = f64_to_f32(thv_k);
    if (kt + 1 == N) {
      ri_n = rho_kf;
      M_n = __fmul_rn(rho_kf, thv_kf);
    } else {
      const int h = kt + 1;
      float wu, wl;
      if constexpr (TOPO) {
        wu = f64_to_f32(LMV(wuP, h));
        wl = 1.0f - wu;
        ri_n = __fmaf_rn(wu, rho_kf, __fmul_rn(wl, rho_lf));
        M_n = __fmul_rn(ri_n, __fmaf_rn(wu, thv_kf, __fmul_rn(wl, thv_lf)));
        xv_n = __fmaf_rn((float)(1.0 - kBeta), wf_l, -WC[h * PT + lane]);
      } else {
        wu = cf[LF_WU * ld + h];
        wl = cf[LF_WL * ld + h];
        ri_n = __fmaf_rn(wl, rho_lf, __fmul_rn(wu, rho_kf));
        M_n = __fmul_rn(ri_n, __fmaf_rn(wl, thv_lf, __fmul_rn(wu, thv_kf)));
        xv_n = wf_l;
      }
      if (CORR)
        fk_n = TOPO ? __fmul_rn(ri_n, __fmaf_rn((float)kBeta, wnf_n, xv_n))
                    : __fmul_rn(ri_n, __fmaf_rn((float)(1.0 - kBeta), wf_l, __fmul_rn((float)kBeta, wnf_n)));
    }
    auto level = [&](int k, const Lev& v, const Lev& u, auto odd) {
      constexpr bool ODD = decltype(odd)::value;
      const double rho_u = u.rho, thv_u = u.thv;
      const float rho_uf = k > kb ? f64_to_f32(rho_u) : rho_uf0, thv_uf = k > kb ? f64_to_f32(thv_u) : thv_uf0;
      const double ex_k = v.ex, w_k = v.w;
      const double wn = damped(X[k * PT + lane], k);
      const float dtk = v.dt;
      float ri_k, M_k;
      if (k == 0) {
        ri_k = rho_kf;
        M_k = __fmul_rn(rho_kf, thv_kf);
      } else if constexpr (TOPO) {
        const float wu = f64_to_f32(LMV(wuP, k)), wl = 1.0f - wu;
        ri_k = __fmaf_rn(wu, rho_uf, __fmul_rn(wl, rho_kf));
        M_k = __fmul_rn(ri_k, __fmaf_rn(wu, thv_uf, __fmul_rn(wl, thv_kf)));
      } else {
        const float wu = cf[LF_WU * ld + k], wl = cf[LF_WL * ld + k];
        ri_k = __fmaf_rn(wl, rho_kf, __fmul_rn(wu, rho_uf));
        M_k = __fmul_rn(ri_k, __fmaf_rn(wl, thv_kf, __fmul_rn(wu, thv_uf)));
      }
      const float wf_k = f64_to_f32(w_k);
      float xv_k = wf_k;
      if constexpr (TOPO) xv_k = k >= 1 ? __fmaf_rn((float)(1.0 - kBeta), wf_k, -WC[k * PT + lane]) : 0.0f;
      const float wnf = f64_to_f32(wn);
      float dtb, dt1, dthe, idzf = 1.0f;
      double idz = 0.0, exref;
      const float D = fma_diff<ODD>(M_k, xv_k, M_n, xv_n);
      if constexpr (TOPO) {
        idz = LMV(idzP, k);
        idzf = f64_to_f32(idz);
        dt1 = f64_to_f32(dtau * idz);
        dtb = f64_to_f32(dtau * kBeta * idz);
        exref = LMV(exrefP, k);
        dthe = __fmaf_rn(-dtk, idzf, -__fmul_rn(dt1, D));
      } else {
        dtb = cf[LF_DTB * ld + k];
        dt1 = cf[LF_DT1 * ld + k];
        exref = cd[LD_EXREF * ld + k];
        dthe = __fmaf_rn(-dt1, D, -dtk);
      }
      const float g = lean_g(ex_k, rho_kf, thv_kf);
      const float q = fma_diff<ODD>(M_k, wnf, M_n, wnf_n);
      const float dTh = __fmaf_rn(-dtb, q, dthe);
      const float dex = fma_diff<true>(g, dthe, __fmul_rn(g, dtb), q);
      float s_rho, s_thv, s_exp;
      if (!CORR) {
        const float drk = v.dr32;
        const float Xe = fma_diff<ODD>(ri_k, xv_k, ri_n, xv_n), Xi = fma_diff<ODD>(ri_k, wnf, ri_n, wnf_n);
        const float t = TOPO ? __fmaf_rn(-drk, idzf, -__fmul_rn(dt1, Xe)) : __fmaf_rn(-dt1, Xe, -drk);
        const float drho = __fmaf_rn(-dtb, Xi, t);
        s_rho = __fadd_rn(rho_kf, drho);
        s_thv = thv_kf + __fdividef(__fmaf_rn(-drho, thv_kf, dTh), s_rho);
        s_exp = __fadd_rn(f64_to_f32(ex_k - exref), dex);
        ok = ok && isfinite(s_thv) && isfinite(s_exp) && isfinite(wnf);
      } else {
        double t;
        float fk;
        if constexpr (TOPO) {
          fk = __fmul_rn(ri_k, __fmaf_rn((float)kBeta, wnf, xv_k));
          t = __fma_rn(dtau * idz, f32_to_f64(fk) - f32_to_f64(fk_n), __dmul_rn(v.dr64, idz));
        } else {
          fk = __fmul_rn(ri_k, __fmaf_rn((float)(1.0 - kBeta), wf_k, __fmul_rn((float)kBeta, wnf)));
          t = __fma_rn(cd[LD_IDZ * ld + k], f32_to_f64(fk) - f32_to_f64(fk_n), v.dr64);
        }
        const double rho_n = rho_k - t;
        const float rho_nf = f64_to_f32(rho_n);
        const double thv_n = thv_k + f32_to_f64(__fdividef(__fmaf_rn(f64_to_f32(t), thv_kf, dTh), rho_nf));
        const double ex_n = ex_k + f32_to_f64(dex);
        if (act) {
          LMV(wflxP, k) = __fma_rn(f32_to_f64(fk), a.inv_nsub, v.wflx);
          LMV(rhoP, k) = rho_n;
          LMV(thvP, k) = thv_n;
          LMV(exP, k) = ex_n;
          LMV(wP, k) = wn;
        }
        s_rho = rho_nf;
        s_thv = f64_to_f32(thv_n);
        s_exp = f64_to_f32(ex_n - exref);
        ok = ok && finite64(thv_n) && finite64(ex_n) && finite64(wn);
        fk_n = fk;
      }
      const int i = k * PT + lane;
      P[i] = s_rho;
      Q[i] = s_thv;
      R[i] = s_exp;
      if (k < a.hdamp) X[i] = wn;
      wnf_n = wnf;
      ri_n = ri_k;
      M_n = M_k;
      xv_n = xv_k;
      rho_k = rho_u;
      thv_k = thv_u;
      rho_kf = rho_uf;
      thv_kf = thv_uf;
    };
#pragma unroll 1
    for (int k = kt; k >= kb; k -= 2) {
      const Lev b0 = fetch(k - 2), b1 = fetch(k - 3);
      level(k, a0, a1, std::false_type{});
      if (k > kb) level(k - 1, a1, b0, std::true_type{});
      a0 = b0;
      a1 = b1;
    }
    if (warp == 0 && act) {
      if constexpr (TOPO) {                                // the ground: the stage's terrain-following w
        const float wg = WC[N * PT + lane];
        a.w32[c * ld + N] = wg;
        if (CORR) LMV(wP, N) = f32_to_f64(wg);
      } else {
        a.w32[c * ld + N] = 0.0f;
        if (CORR) LMV(wP, N) = 0.0;                       // the ground (w^n there is 0 already)
      }
    }
  }
  if (!ok && act) atomicOr(a.status, 1u);
  __syncthreads();
  // ---- the FP32 shadows as whole level runs of each cell's [c][ld] row
  for (int r = warp; r < 32 && c0 + r < nc; r += W) {
    const int64_t o = (c0 + r) * ld;
    for (int k = lane; k < N; k += 32) {
      const int i = k * PT + r;
      a.rho32[o + k] = P[i];
      a.thv32[o + k] = Q[i];
      a.exp32[o + k] = R[i];
      a.w32[o + k] = f64_to_f32(X[i]);
    }
  }
#undef LMV
}

const TileChoice kLeanDefault = {2, LEAN_RULE};

bool lean_shape_ok(const TileChoice& t) {
  return t.lanes == 2 && (t.block == LEAN_TILE4 || t.block == LEAN_TILE8 || t.block == LEAN_RULE ||
                          t.block == LEAN_COLUMN1 || t.block == LEAN_COLUMN2);
}

// the forced form, or the one lean_rule.h gives for the current device
int lean_form(const MxGeo& G, const TileChoice& t, bool topo) {
  if (t.block != LEAN_RULE) return t.block;
  int dev = 0, sms = 152, shared = 233472, reserved = 1024;      // a GB300's, should a query fail
  if (cudaGetDevice(&dev) == cudaSuccess) {
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&shared, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  }
  return lean_form_for(G.nc, G.N, topo, sms, (size_t)shared, (size_t)reserved);
}

template <bool CORR, bool TOPO, int W, int MINB>
void launch_lean_tile(const MxGeo& G, const MxLeanArgs& a, cudaStream_t st) {
  // the limit is set for the most levels a grid can have (203 KB over terrain), the same by
  // every thread; a launch takes what its own levels need
  cudaFuncSetAttribute(k_mx_lean_tile<CORR, TOPO, W, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)lean_tile_bytes(256, TOPO));
  const size_t sm = lean_tile_bytes(G.N, TOPO);
  k_mx_lean_tile<CORR, TOPO, W, MINB><<<blocks_for(G.nc, 32), 32 * W, sm, st>>>(G, a);
}

template <bool CORR, bool TOPO>
void launch_lean_column_as(const MxGeo& G, const MxLeanArgs& a, const TileChoice& t, cudaStream_t st) {
  const unsigned nb = blocks_for(G.nc, kLeanThreads);
  switch (lean_form(G, t, TOPO)) {
    case LEAN_TILE8: launch_lean_tile<CORR, TOPO, 8, 2>(G, a, st); break;
    case LEAN_TILE4: launch_lean_tile<CORR, TOPO, 4, 5>(G, a, st); break;
    case LEAN_COLUMN1: k_mx_lean_column<CORR, TOPO, 1><<<nb, kLeanThreads, 0, st>>>(G, a); break;
    default: k_mx_lean_column<CORR, TOPO, 2><<<nb, kLeanThreads, 0, st>>>(G, a);
  }
}

template <bool CORR>
void launch_lean_column(const MxGeo& G, const MxLeanArgs& a, const TileChoice& t, bool topo, cudaStream_t st) {
  if (topo) launch_lean_column_as<CORR, true>(G, a, t, st);
  else launch_lean_column_as<CORR, false>(G, a, t, st);
}
