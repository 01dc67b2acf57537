// The FP32 stencils of one mixed-precision state (included by dycore32.cu, inside its unnamed
// namespace): four consecutive levels per lane in 128-bit loads.
//
// What bounds them: the gathers of neighbour rows. With one level per lane and load, a lane kept
// 4 bytes per load in flight and spent most of its instructions on addresses, and every kernel
// here ran at about half the HBM rate. A lane now holds a quad of levels: a quarter of the loads
// and of the index arithmetic, four times the bytes in flight per load. LPE lanes share an
// entity (neighbour indices and weights are loaded once per lane and serve its quads); rows are
// ld long, a multiple of 32 levels, so a quad never leaves its row. Levels past the last one
// are computed and stored into the rows' padding, which nothing reads as a level.
// Every level's arithmetic is that of the one-level form, in the same order.
// Per launch (GB300, R2B6 / 90 levels, us, one level per lane -> this form): vertices 131 -> 81, edge
// diagnostics 125 -> 92, kinetic energy 121 -> 100, edge tendency 531 -> 377, gather (which formed the
// damping's edge update) 557 -> 269, damping 275 -> 449 (with that update), diffusion at vertices and
// cells 258 -> 158, at edges 889 -> 356, of theta_v 794 -> 326.
struct F4 {
  float v[4];
};
__device__ __forceinline__ F4 ld4(const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  return F4{{t.x, t.y, t.z, t.w}};
}
__device__ __forceinline__ void st4(float* p, const F4& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}
// acc + w x, level by level
__device__ __forceinline__ void fma4(F4& acc, float w, const F4& x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) acc.v[i] = __fmaf_rn(w, x.v[i], acc.v[i]);
}

// m += w x on a quad of an FP64 row (whole 16-byte words: element by element, every store wrote a
// quarter of each 32-byte sector it touched)
__device__ __forceinline__ void add4(double* m, const F4& x, double w) {
  double2* q = reinterpret_cast<double2*>(m);
  double2 a = q[0], b = q[1];
  a.x = __fma_rn(f32_to_f64(x.v[0]), w, a.x);
  a.y = __fma_rn(f32_to_f64(x.v[1]), w, a.y);
  b.x = __fma_rn(f32_to_f64(x.v[2]), w, b.x);
  b.y = __fma_rn(f32_to_f64(x.v[3]), w, b.y);
  q[0] = a;
  q[1] = b;
}

// warp w, lanes [sub*LPE, (sub+1)*LPE) handle entity w * (32/LPE) + sub
#define QUAD_PROLOGUE(LPE, COUNT)                                                        \
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;             \
  const int64_t item = gw * (32 / (LPE)) + (int64_t)((threadIdx.x & 31) / (LPE));        \
  const int lane = (int)(threadIdx.x & ((LPE) - 1));                                     \
  if (item >= (COUNT)) return;

// O3 curl (full levels) and the vertex mean of w (half levels)
template <int LPE>
__device__ __forceinline__ void mx_vertex_quads(const MxGeo& G, const float* __restrict__ vn,
                                                const float* __restrict__ w, float* __restrict__ zeta,
                                                float* __restrict__ w_v, int64_t v, int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2, nh = (G.N + 4) >> 2;
  int64_t E[6], C[6];
  float rw[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    E[j] = (int64_t)G.v2e[6 * v + j] * ld;
    C[j] = (int64_t)G.v2c[6 * v + j] * ld;
    rw[j] = G.rot_w32[6 * v + j];
  }
  const int deg = G.vdeg[v];
  const float inv_deg = 1.0f / (float)deg;
  for (int q = lane; q < nh; q += LPE) {
    const int k = 4 * q;
    if (q < nq) {
      F4 acc{};
#pragma unroll
      for (int j = 0; j < 6; ++j) fma4(acc, rw[j], ld4(vn + E[j] + k));
      st4(zeta + v * ld + k, acc);
    }
    F4 acc{};
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const F4 x = ld4(w + C[j] + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j < 5 || deg == 6) acc.v[i] += x.v[i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc.v[i] *= inv_deg;
    st4(w_v + v * ld + k, acc);
  }
}

// O4 vt
template <int LPE>
__device__ __forceinline__ void mx_edge_diag_quads(const MxGeo& G, const float* __restrict__ vn, float* __restrict__ vt,
                                                   int64_t e, int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t S[5];
  float W[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    S[j] = (int64_t)G.e2vt[5 * e + j] * ld;
    W[j] = G.vt_w32[5 * e + j];
  }
  for (int q = lane; q < nq; q += LPE) {
    F4 acc{};
#pragma unroll
    for (int j = 0; j < 5; ++j) fma4(acc, W[j], ld4(vn + S[j] + 4 * q));
    st4(vt + e * ld + 4 * q, acc);
  }
}

template <int LPE>
__global__ void __launch_bounds__(512) k_mx_vertex(MxGeo G, const float* __restrict__ vn, const float* __restrict__ w,
                                                   float* __restrict__ zeta, float* __restrict__ w_v) {
  QUAD_PROLOGUE(LPE, G.nv)
  mx_vertex_quads<LPE>(G, vn, w, zeta, w_v, item, lane);
}

template <int LPE>
__global__ void __launch_bounds__(512) k_mx_edge_diag(MxGeo G, const float* __restrict__ vn, float* __restrict__ vt) {
  QUAD_PROLOGUE(LPE, G.ne)
  mx_edge_diag_quads<LPE>(G, vn, vt, item, lane);
}

// both in one launch, on small grids (neither reads what the other writes; the first nbv blocks
// take the vertices)
__global__ void __launch_bounds__(128) k_mx_vertex_edge(MxGeo G, const float* __restrict__ vn,
                                                        const float* __restrict__ w, float* __restrict__ zeta,
                                                        float* __restrict__ w_v, float* __restrict__ vt, unsigned nbv) {
  const int lane = threadIdx.x & 7;
  const int64_t item = (int64_t)blockIdx.x * 16 + (threadIdx.x >> 3);
  if (blockIdx.x < nbv) {
    if (item < G.nv) mx_vertex_quads<8>(G, vn, w, zeta, w_v, item, lane);
  } else if (item - (int64_t)nbv * 16 < G.ne) {
    mx_edge_diag_quads<8>(G, vn, vt, item - (int64_t)nbv * 16, lane);
  }
}

// O5 K_c = sum_e kappa_ce (vn_e^2 + vt_e^2)/2
template <int LPE>
__device__ __forceinline__ void mx_cell_ke_quads(const MxGeo& G, const float* __restrict__ vn,
                                                 const float* __restrict__ vt, float* __restrict__ Kc, int64_t c,
                                                 int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t E[3];
  float kw[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    kw[s] = G.kin_w32[3 * c + s];
  }
  for (int q = lane; q < nq; q += LPE) {
    F4 acc{};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const F4 a = ld4(vn + E[s] + 4 * q), b = ld4(vt + E[s] + 4 * q);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        acc.v[i] = __fmaf_rn(kw[s], 0.5f * __fmaf_rn(a.v[i], a.v[i], __fmul_rn(b.v[i], b.v[i])), acc.v[i]);
    }
    st4(Kc + c * ld + 4 * q, acc);
  }
}

template <int LPE>
__global__ void __launch_bounds__(512) k_mx_cell_ke(MxGeo G, const float* __restrict__ vn, const float* __restrict__ vt,
                                                    float* __restrict__ Kc) {
  QUAD_PROLOGUE(LPE, G.nc)
  mx_cell_ke_quads<LPE>(G, vn, vt, Kc, item, lane);
}

// vn tendency and update, horizontal flux integrals, edge part of the w advection. A lane holds
// the half levels of its quad and the one below it (five: the interpolants the quad's full levels
// difference; the fifth is formed again by the next lane rather than shuffled). Where a sum has
// two products, the one rounded first is written out, as the one-level form had it. TOPO
// (terrain-following levels): per-edge interpolation weights, w - wcc in the vertical advection,
// the metric correction of the pressure gradient (exp is then against the per-cell reference),
// fluxes through dz_e. ROUND_PG: the predictor subtracts the rounded pressure gradient instead of
// fusing the product (the persistent ensemble's results are defined so).
template <int LPE, bool TOPO, bool ROUND_PG = false>
__device__ __forceinline__ void mx_edge_tend_quads(const MxGeo& G, const MxEdgeArgs& a, int64_t e, int lane) {
  const int ld = G.ld, N = G.N, nh = (N + 4) >> 2;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld;
  const int64_t v1 = (int64_t)G.e2v[2 * e] * ld, v2 = (int64_t)G.e2v[2 * e + 1] * ld;
  const float ide = G.inv_de32[e], ile = G.inv_le32[e], fe = G.f_e32[e], le = G.l_e32[e];
  const float cide = (float)kCpd * ide;
  const float csn = TOPO ? a.t_csn[e] : 0.0f;
  const int64_t o = e * ld;
  const float* __restrict__ vn = a.vn + o;
  const float* __restrict__ vt = a.vt + o;
  const float* __restrict__ w = a.w;
  const float* __restrict__ ws = TOPO ? a.t_wcon : a.w;      // the vertical velocity that advects vn
  const float* __restrict__ wv = a.w_v;
  const float* __restrict__ wu32 = TOPO ? a.t_wu_e + o : G.wu32;
  const float* __restrict__ wl32 = G.wl32;
  const float* __restrict__ idz32 = TOPO ? a.t_inv_dz_e + o : G.inv_dz32;
  float* __restrict__ ae_o = a.a_e + o;
  const float* vnb_o = a.vn_base + o;      // vn_base, Avn0 and vn_out may be one buffer
  float* avn_o = a.Avn0 + o;
  float* vout_o = a.vn_out + o;
  float* __restrict__ phi_o = a.phi + o;
  float* __restrict__ gth_o = a.gth + o;
  double* __restrict__ mflx_o = a.mflx + o;
  const bool corr = a.corrector != 0, skip = a.skip_flux != 0, upw = a.upwind_theta != 0;
  const float dtau = a.dtau;
  const double inv_nsub = a.inv_nsub;
  auto half = [](float wa, float xa, float wb, float xb) {
    return __fmaf_rn(wa, xa, __fmul_rn(wb, xb));
  };
  for (int q = lane; q < nh; q += LPE) {
    const int k0 = 4 * q;
    const bool below = k0 + 4 <= N;        // the half level below the quad exists
    float vie[5], sw[5];
    {
      const F4 x = ld4(vn + k0), t = ld4(vt + k0), wu = ld4(wu32 + k0);
      F4 wl;
      if constexpr (TOPO) {
#pragma unroll
        for (int i = 0; i < 4; ++i) wl.v[i] = 1.0f - wu.v[i];
      } else {
        wl = ld4(wl32 + k0);
      }
      const float xm = k0 > 0 ? vn[k0 - 1] : 0.0f, tm = k0 > 0 ? vt[k0 - 1] : 0.0f;
      const float xp = k0 + 4 < N ? vn[k0 + 4] : 0.0f;
      const F4 w1 = ld4(w + c1 + k0), w2 = ld4(w + c2 + k0), y1 = ld4(wv + v1 + k0), y2 = ld4(wv + v2 + k0);
      F4 ae;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int h = k0 + i;
        const float xu = i ? x.v[i ? i - 1 : 0] : xm, tu = i ? t.v[i ? i - 1 : 0] : tm;
        vie[i] = h == 0 ? x.v[i] : (h >= N ? xu : half(wu.v[i], xu, wl.v[i], x.v[i]));
        const float tie = h == 0 ? t.v[i] : (h >= N ? tu : half(wu.v[i], tu, wl.v[i], t.v[i]));
        const float dw = w2.v[i] - w1.v[i], dwv = y2.v[i] - y1.v[i];
        if (!TOPO) sw[i] = w1.v[i] + w2.v[i];
        ae.v[i] = __fmaf_rn(__fmul_rn(vie[i], dw), ide, __fmul_rn(__fmul_rn(tie, dwv), ile));
      }
      st4(ae_o + k0, ae);
      if (k0 >= N) continue;
      if constexpr (TOPO) {
        const F4 s1 = ld4(ws + c1 + k0), s2 = ld4(ws + c2 + k0);
#pragma unroll
        for (int i = 0; i < 4; ++i) sw[i] = s1.v[i] + s2.v[i];                  // 0 at the lid and the ground
      }
      vie[4] = sw[4] = 0.0f;
      if (below) {
        const float wa = wu32[k0 + 4], wb = TOPO ? 1.0f - wa : wl32[k0 + 4];
        vie[4] = k0 + 4 >= N ? x.v[3] : half(wa, x.v[3], wb, xp);
        sw[4] = ws[c1 + k0 + 4] + ws[c2 + k0 + 4];
      }
    }
    const F4 z1 = ld4(a.zeta + v1 + k0), z2 = ld4(a.zeta + v2 + k0);
    const F4 K1 = ld4(a.Kc + c1 + k0), K2 = ld4(a.Kc + c2 + k0), t = ld4(vt + k0), iz = ld4(idz32 + k0);
    const F4 t1 = ld4(a.thv + c1 + k0), t2 = ld4(a.thv + c2 + k0);
    const F4 p1 = ld4(a.exp + c1 + k0), p2 = ld4(a.exp + c2 + k0), vb = ld4(vnb_o + k0);
    F4 A, vo, av{}, bf{}, d1{}, d2{};
    if (corr) av = ld4(avn_o + k0);
    if constexpr (TOPO) {
      bf = ld4(a.t_bf + k0);
      d1 = ld4(a.t_hdpdz + c1 + k0);
      d2 = ld4(a.t_hdpdz + c2 + k0);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float wbar = 0.25f * (sw[i] + sw[i + 1]);
      const float zeta_e = 0.5f * (z1.v[i] + z2.v[i]);
      A.v[i] = -(K2.v[i] - K1.v[i]) * ide + (zeta_e + fe) * t.v[i] - wbar * (vie[i] - vie[i + 1]) * iz.v[i];
      const float th_e = 0.5f * (t1.v[i] + t2.v[i]);
      float px;
      if constexpr (TOPO) px = (p2.v[i] - p1.v[i]) * cide - (csn * bf.v[i]) * (d1.v[i] + d2.v[i]);
      else px = __fmul_rn(p2.v[i] - p1.v[i], cide);
      if (corr)
        vo.v[i] = __fmaf_rn(dtau, __fmaf_rn(0.5f, av.v[i] + A.v[i], -__fmul_rn(th_e, px)), vb.v[i]);
      else
        vo.v[i] = __fmaf_rn(dtau, ROUND_PG ? __fsub_rn(A.v[i], __fmul_rn(th_e, px)) : __fmaf_rn(-th_e, px, A.v[i]), vb.v[i]);
    }
    if (!corr) st4(avn_o + k0, A);
    st4(vout_o + k0, vo);
    if (skip) continue;
    const F4 r1 = ld4(a.rho + c1 + k0), r2 = ld4(a.rho + c2 + k0);
    F4 F, g, dz{};
    if constexpr (TOPO) dz = ld4(a.t_dz_e + o + k0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      F.v[i] = 0.5f * (r1.v[i] + r2.v[i]) * vo.v[i];
      if constexpr (TOPO) F.v[i] *= dz.v[i];
      g.v[i] = (le * F.v[i]) * (upw ? (vo.v[i] >= 0.0f ? t1.v[i] : t2.v[i]) : 0.5f * (t1.v[i] + t2.v[i]));
    }
    st4(phi_o + k0, F);
    st4(gth_o + k0, g);
    if (corr) add4(mflx_o + k0, F, inv_nsub);
  }
}

// 64 registers, so 1,024 threads per SM in blocks of any size the tile may have
template <int LPE, bool TOPO>
__global__ void __launch_bounds__(512, 2) k_mx_edge_tend(MxGeo G, MxEdgeArgs a) {
  QUAD_PROLOGUE(LPE, G.ne)
  mx_edge_tend_quads<LPE, TOPO>(G, a, item, lane);
}

// ---- fourth-order divergence damping of the corrector's vn^{n+1}: cell divergence, its cell
// Laplacian, then the edge update (eight lanes per entity, four entities per warp)
constexpr int kQuadLanes = 8;

template <int LPE>
__device__ __forceinline__ void mx_div_quads(const MxGeo& G, const float* __restrict__ vn, float* __restrict__ D,
                                             int64_t c, int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t E[3];
  float dw[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    dw[s] = G.div_w32[3 * c + s];
  }
  for (int q = lane; q < nq; q += LPE) {
    const F4 x0 = ld4(vn + E[0] + 4 * q), x1 = ld4(vn + E[1] + 4 * q), x2 = ld4(vn + E[2] + 4 * q);
    F4 d;
#pragma unroll
    for (int i = 0; i < 4; ++i) d.v[i] = dw[0] * x0.v[i] + dw[1] * x1.v[i] + dw[2] * x2.v[i];
    st4(D + c * ld + 4 * q, d);
  }
}

__global__ void __launch_bounds__(256) k_mx_dd_div(MxGeo G, const float* __restrict__ vn, float* __restrict__ D) {
  QUAD_PROLOGUE(kQuadLanes, G.nc)
  mx_div_quads<kQuadLanes>(G, vn, D, item, lane);
}

template <int LPE>
__device__ __forceinline__ void mx_dd_lap_quads(const MxGeo& G, const float* __restrict__ D, float* __restrict__ L,
                                                int64_t c, int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t B[3];
  float wt[3];
  bool out[3];                                               // c is the edge's first cell
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int e = G.c2e[3 * c + s];
    const int ca = G.e2c[2 * e], cb = G.e2c[2 * e + 1];
    out[s] = ca == c;
    B[s] = (int64_t)(out[s] ? cb : ca) * ld;
    wt[s] = G.div_w32[3 * c + s] * G.inv_de32[e];
  }
  for (int q = lane; q < nq; q += LPE) {
    const F4 m = ld4(D + c * ld + 4 * q);                    // own row once, not once per edge
    const F4 x0 = ld4(D + B[0] + 4 * q), x1 = ld4(D + B[1] + 4 * q), x2 = ld4(D + B[2] + 4 * q);
    F4 l;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float g0 = out[0] ? x0.v[i] - m.v[i] : m.v[i] - x0.v[i];
      const float g1 = out[1] ? x1.v[i] - m.v[i] : m.v[i] - x1.v[i];
      const float g2 = out[2] ? x2.v[i] - m.v[i] : m.v[i] - x2.v[i];
      l.v[i] = wt[0] * g0 + wt[1] * g1 + wt[2] * g2;
    }
    st4(L + c * ld + 4 * q, l);
  }
}

__global__ void __launch_bounds__(256) k_mx_dd_lap(MxGeo G, const float* __restrict__ D, float* __restrict__ L) {
  QUAD_PROLOGUE(kQuadLanes, G.nc)
  mx_dd_lap_quads<kQuadLanes>(G, D, L, item, lane);
}

// the damping's edge update with the corrector's fluxes and the FP64 step-mean mass flux. A kernel
// of its own: formed inside the corrector's gather by both cells of every edge, it saved the
// fluxes' round trip but held so many neighbour rows that the gather spilled at 64 registers and
// waited on its loads at 80. R2B6/90, per step: gather 4.63 and damping 0.64 ms with it fused,
// 2.72 and 2.25 ms apart (this kernel 322 us per launch, 5.5 TB/s of its 60 B per cell-level)
__global__ void __launch_bounds__(256, 4) k_mx_dd_edge(MxGeo G, MxDDArgs a) {
  QUAD_PROLOGUE(kQuadLanes, G.ne)
  const int64_t e = item;
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld, o = e * ld;
  const float sc = a.scale * G.inv_de32[e], le = G.l_e32[e];
  for (int q = lane; q < nq; q += kQuadLanes) {
    const int k = 4 * q;
    const F4 v = ld4(a.vn + o + k), L1 = ld4(a.L + c1 + k), L2 = ld4(a.L + c2 + k);
    const F4 r1 = ld4(a.rho + c1 + k), r2 = ld4(a.rho + c2 + k), t1 = ld4(a.thv + c1 + k), t2 = ld4(a.thv + c2 + k);
    F4 dz{}, vd, F, g;
    if (a.dz_e) dz = ld4(a.dz_e + o + k);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      vd.v[i] = __fmaf_rn(-sc, L2.v[i] - L1.v[i], v.v[i]);
      F.v[i] = 0.5f * (r1.v[i] + r2.v[i]) * vd.v[i];
      if (a.dz_e) F.v[i] *= dz.v[i];
      g.v[i] = (le * F.v[i]) * (a.upwind_theta ? (vd.v[i] >= 0.0f ? t1.v[i] : t2.v[i]) : 0.5f * (t1.v[i] + t2.v[i]));
    }
    st4(a.vn + o + k, vd);
    st4(a.phi + o + k, F);
    st4(a.gth + o + k, g);
    add4(a.mflx + o + k, F, a.inv_nsub);
  }
}

// ---- diffusion: least-squares vertex velocity and O3 curl of vn
template <int LPE>
__device__ __forceinline__ void mx_diff_vertex_quads(const MxGeo& G, const float* __restrict__ vn,
                                                     float* __restrict__ ux, float* __restrict__ uy,
                                                     float* __restrict__ uz, float* __restrict__ zeta, int64_t v,
                                                     int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t E[6];
  float L[18], R[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) E[j] = (int64_t)G.v2e[6 * v + j] * ld;
#pragma unroll
  for (int j = 0; j < 18; ++j) L[j] = G.lsq_w32[18 * v + j];
#pragma unroll
  for (int j = 0; j < 6; ++j) R[j] = G.rot_w32[6 * v + j];
  for (int q = lane; q < nq; q += LPE) {
    F4 x{}, y{}, z{}, r{};
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const F4 u = ld4(vn + E[j] + 4 * q);
      fma4(x, L[3 * j], u);
      fma4(y, L[3 * j + 1], u);
      fma4(z, L[3 * j + 2], u);
      fma4(r, R[j], u);
    }
    const int64_t o = v * ld + 4 * q;
    st4(ux + o, x);
    st4(uy + o, y);
    st4(uz + o, z);
    st4(zeta + o, r);
  }
}

// vertices first, then O2 divergence at the cells; both only read vn
template <int LPE>
__global__ void __launch_bounds__(512, 2) k_mx_diff_vertex(MxGeo G, const float* __restrict__ vn, float* __restrict__ ux,
                                                        float* __restrict__ uy, float* __restrict__ uz,
                                                        float* __restrict__ zeta, float* __restrict__ divc) {
  QUAD_PROLOGUE(LPE, G.nv + G.nc)
  if (item < G.nv) mx_diff_vertex_quads<LPE>(G, vn, ux, uy, uz, zeta, item, lane);
  else mx_div_quads<LPE>(G, vn, divc, item - G.nv, lane);
}

// diffusion: Smagorinsky K_h, vn += dt K_h L(vn), theta_v flux; D1 and zeta1 (fourth-order
// background diffusion, an option) or NULL
template <int LPE>
__device__ __forceinline__ void mx_diff_edge_quads(const MxGeo& G, float* __restrict__ vn, const float* __restrict__ ux,
                                                   const float* __restrict__ uy, const float* __restrict__ uz,
                                                   const float* __restrict__ zeta, const float* __restrict__ divc,
                                                   const float* __restrict__ thv, float* __restrict__ thflx, float dt,
                                                   const float* __restrict__ D1, const float* __restrict__ zeta1,
                                                   float bd_scale, int64_t e, int lane) {
  const int ld = G.ld, nq = (G.N + 3) >> 2;
  int64_t Q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) Q[j] = (int64_t)G.e2q[4 * e + j] * ld;
  const int64_t c1 = (int64_t)G.e2c[2 * e] * ld, c2 = (int64_t)G.e2c[2 * e + 1] * ld;
  const int64_t v1 = (int64_t)G.e2v[2 * e] * ld, v2 = (int64_t)G.e2v[2 * e + 1] * ld;
  const float nx = G.n_e32[3 * e], ny = G.n_e32[3 * e + 1], nz = G.n_e32[3 * e + 2];
  const float tx = G.t_e32[3 * e], ty = G.t_e32[3 * e + 1], tz = G.t_e32[3 * e + 2];
  const float ide = G.inv_de32[e], ile = G.inv_le32[e], i34 = G.L34inv32[e], le = G.l_e32[e];
  const float cs2ld = (float)(kCsSmag * kCsSmag) * le / ide;
  for (int q = lane; q < nq; q += LPE) {
    const int k = 4 * q;
    const F4 x3 = ld4(ux + Q[3] + k), x2 = ld4(ux + Q[2] + k), x1 = ld4(ux + Q[1] + k), x0 = ld4(ux + Q[0] + k);
    const F4 y3 = ld4(uy + Q[3] + k), y2 = ld4(uy + Q[2] + k), y1 = ld4(uy + Q[1] + k), y0 = ld4(uy + Q[0] + k);
    const F4 z3 = ld4(uz + Q[3] + k), z2 = ld4(uz + Q[2] + k), z1 = ld4(uz + Q[1] + k), z0 = ld4(uz + Q[0] + k);
    const F4 d1 = ld4(divc + c1 + k), d2 = ld4(divc + c2 + k), c1z = ld4(zeta + v1 + k), c2z = ld4(zeta + v2 + k);
    const F4 t1 = ld4(thv + c1 + k), t2 = ld4(thv + c2 + k), vb = ld4(vn + e * ld + k);
    F4 vo, fl;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float ax = x3.v[i] - x2.v[i], ay = y3.v[i] - y2.v[i], az = z3.v[i] - z2.v[i];
      const float bx = x1.v[i] - x0.v[i], by = y1.v[i] - y0.v[i], bz = z1.v[i] - z0.v[i];
      const float DT = (ax * nx + ay * ny + az * nz) * i34 - (bx * tx + by * ty + bz * tz) * ile;
      const float DS = (ax * tx + ay * ty + az * tz) * i34 + (bx * nx + by * ny + bz * nz) * ile;
      const float Kh = cs2ld * sqrtf(DT * DT + DS * DS);
      const float lap = (d2.v[i] - d1.v[i]) * ide - (c2z.v[i] - c1z.v[i]) * ile;
      vo.v[i] = vb.v[i] + dt * Kh * lap;
      fl.v[i] = le * Kh * (t2.v[i] - t1.v[i]) * ide;
    }
    if (D1) {
      const F4 e1 = ld4(D1 + c1 + k), e2 = ld4(D1 + c2 + k), f1 = ld4(zeta1 + v1 + k), f2 = ld4(zeta1 + v2 + k);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float lap2 = (e2.v[i] - e1.v[i]) * ide - (f2.v[i] - f1.v[i]) * ile;
        vo.v[i] -= bd_scale * lap2;
      }
    }
    st4(vn + e * ld + k, vo);
    st4(thflx + e * ld + k, fl);
  }
}

__global__ void __launch_bounds__(256, 2) k_mx_diff_edge(MxGeo G, float* __restrict__ vn, const float* __restrict__ ux,
                                                         const float* __restrict__ uy, const float* __restrict__ uz,
                                                         const float* __restrict__ zeta,
                                                         const float* __restrict__ divc, const float* __restrict__ thv,
                                                         float* __restrict__ thflx, float dt,
                                                         const float* __restrict__ D1, const float* __restrict__ zeta1,
                                                         float bd_scale) {
  QUAD_PROLOGUE(kQuadLanes, G.ne)
  mx_diff_edge_quads<kQuadLanes>(G, vn, ux, uy, uz, zeta, divc, thv, thflx, dt, D1, zeta1, bd_scale, item, lane);
}

// ---- diffusion of theta_v: FP32 increment, FP64 accumulation, Exner at constant density,
// shadows refreshed. A block takes 32 cells and 32 levels at a time: eight lanes per cell gather
// the edges' fluxes by quads of levels, the increments cross to level-major order through shared
// memory for the FP64 update (32 consecutive cells per level), the refreshed shadows cross back.
__global__ void __launch_bounds__(256, 4) k_mx_diff_theta(MxGeo G, const float* __restrict__ thflx,
                                                          double* __restrict__ thv, double* __restrict__ ex,
                                                          float* __restrict__ thv32, float* __restrict__ exp32, float dt,
                                                          const double* __restrict__ exref_lm) {
  __shared__ float s0[32][33], s1[32][33];
  const int N = G.N, ld = G.ld, tid = threadIdx.x, grp = tid >> 3, lane = tid & 7;
  const int64_t nc = G.nc, c0 = (int64_t)blockIdx.x * 32, c = c0 + grp;
  int64_t E[3] = {0, 0, 0};
  float sg[3] = {0.f, 0.f, 0.f}, dtA = 0.f;
  if (c < nc) {
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      E[s] = (int64_t)G.c2e[3 * c + s] * ld;
      sg[s] = G.s_ce32[3 * c + s];
    }
    dtA = dt * (float)G.inv_Ac[c];
  }
  for (int k0 = 0; k0 < N; k0 += 32) {
    const int kq = k0 + 4 * lane;
    if (c < nc && kq < N) {
      const F4 x0 = ld4(thflx + E[0] + kq), x1 = ld4(thflx + E[1] + kq), x2 = ld4(thflx + E[2] + kq);
#pragma unroll
      for (int i = 0; i < 4; ++i) s0[4 * lane + i][grp] = dtA * (sg[0] * x0.v[i] + sg[1] * x1.v[i] + sg[2] * x2.v[i]);
    }
    __syncthreads();
    const int cl = tid & 31;
    for (int r = tid >> 5; r < 32; r += 8) {
      const int k = k0 + r;
      if (k >= N || c0 + cl >= nc) continue;
      const int64_t i = (int64_t)k * nc + c0 + cl;
      const float dth = s0[r][cl];
      const double th = thv[i], exo = ex[i];
      const double th_n = th + f32_to_f64(dth);
      const double ex_n = exo + exo * f32_to_f64(kRcvF * dth / f64_to_f32(th));
      thv[i] = th_n;
      ex[i] = ex_n;
      s0[r][cl] = f64_to_f32(th_n);
      s1[r][cl] = f64_to_f32(ex_n - (exref_lm ? exref_lm[i] : G.ex_ref[k]));
    }
    __syncthreads();
    if (c < nc && kq < N) {
      F4 a, b;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a.v[i] = s0[4 * lane + i][grp];
        b.v[i] = s1[4 * lane + i][grp];
      }
      st4(thv32 + c * ld + kq, a);
      st4(exp32 + c * ld + kq, b);
    }
    __syncthreads();
  }
}

// ---- gather of the lean column's stage inputs: a block takes 32 consecutive cells, eight lanes
// per cell gather its edges by quads of levels (32 levels per pass), and the results cross to
// level-major order through shared memory (32 consecutive cells per level). CORR: the
// predictor's A_w is averaged in as the rows are written, where it is read coalesced. TOPO
// (terrain-following levels): the vertical advection of w with w - wcc and the cell's own 1/dzh;
// the divergences stay per unit thickness and the column scales them by the cell's 1/dz.
template <bool CORR, bool TOPO>
__global__ void __launch_bounds__(256, 4) k_mx_lean_gather(MxGeo G, MxLeanArgs a) {
  __shared__ double sd[CORR ? 32 : 1][33];
  __shared__ float sf[CORR ? 2 : 3][32][33];                 // dtau D_Theta, A_w, dtau D_rho (predictor)
  const int N = G.N, ld = G.ld;
  const int64_t nc = G.nc, c0 = (int64_t)blockIdx.x * 32;
  const int tid = threadIdx.x, lane = tid & 7, cl = tid >> 3;
  const float dtau32 = (float)a.dtau;
  // the cell's neighbours and weights, held for every pass over the levels
  const bool act = c0 + cl < nc;
  const int64_t c = act ? c0 + cl : 0, o = c * ld;
  const float4 cw = a.cw32[c];
  int64_t E[3];
  float sg[3], kw[3];
  double dwt[3];
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    E[s] = (int64_t)G.c2e[3 * c + s] * ld;
    sg[s] = G.s_ce32[3 * c + s];
    kw[s] = G.kin_w32[3 * c + s];
    if (CORR) dwt[s] = a.dwa_t[3 * c + s];
  }
  for (int k0 = 0; k0 < N; k0 += 32) {
    const int k = k0 + 4 * lane;
    if (act && k < N) {
      F4 ae[3], F[3], Gt[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        ae[s] = ld4(a.a_e + E[s] + k);
        F[s] = ld4(a.phi + E[s] + k);
        Gt[s] = ld4(a.gth + E[s] + k);
      }
      const F4 w = ld4(a.w_stage + o + k);
      const float wm = k > 0 ? a.w_stage[o + k - 1] : 0.0f, wp = k + 4 <= N ? a.w_stage[o + k + 4] : 0.0f;
      F4 wc{}, iz;
      if constexpr (TOPO) {
        wc = ld4(a.t_wcon + o + k);
        iz = ld4(a.t_inv_dzh + o + k);
      } else {
        iz = ld4(G.inv_dz2_32 + k);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 4 * lane + i;
        // conversions on the integer pipe: the hardware ones are FP64-pipe operations, a warp
        // instruction per SM every 16 cycles
        if (CORR)
          sd[r][cl] = (dwt[0] * f32_to_f64(F[0].v[i]) + dwt[1] * f32_to_f64(F[1].v[i])) + dwt[2] * f32_to_f64(F[2].v[i]);
        else
          sf[2][r][cl] = (cw.x * F[0].v[i] + cw.y * F[1].v[i]) + cw.z * F[2].v[i];
        sf[0][r][cl] = (sg[0] * Gt[0].v[i] + sg[1] * Gt[1].v[i] + sg[2] * Gt[2].v[i]) * cw.w;
        const float hadv = kw[0] * ae[0].v[i] + kw[1] * ae[1].v[i] + kw[2] * ae[2].v[i];
        const float wu = i ? w.v[i ? i - 1 : 0] : wm, wd = i < 3 ? w.v[i < 3 ? i + 1 : 3] : wp;
        float Aw;
        if constexpr (TOPO) Aw = -hadv - wc.v[i] * (wu - wd) * (0.5f * iz.v[i]);
        else Aw = -hadv - w.v[i] * (wu - wd) * iz.v[i];
        sf[1][r][cl] = Aw;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = (tid >> 5) + 8 * i, ci = tid & 31, kk = k0 + r;
      if (c0 + ci >= nc || kk >= N) continue;
      const int64_t j = (int64_t)kk * nc + c0 + ci;
      if (CORR) a.dr64[j] = sd[r][ci];
      else a.dr32[j] = sf[2][r][ci];
      a.dt32[j] = sf[0][r][ci];
      if (kk >= 1) {
        float Aw = sf[1][r][ci];
        if (CORR) Aw = 0.5f * (a.Aw0[j] + Aw);
        else a.Aw0[j] = Aw;
        a.aw32[j] = dtau32 * Aw;
      }
    }
    __syncthreads();
  }
}
