// weno_tiles1d.cuh -- the 1D stage kernels (Euler and scalar equations) of
// the central-upwind WENO right-hand side, templated on the stencil
// half-width r.  Included by weno_tiles.cuh inside its namespaces; it uses
// the helpers defined there (stage_control, load_scheme, block_max_atomic, ...).
#pragma once

// ---------------------------------------------------------------------------
// 1D stage kernel: NC = 3 (Euler) or 1 (scalar advection).  Tile of
// kT1 = 127 cells, 128 faces, one face per thread.
// Planes: 0 rho, 1 m, 2 E, 3 u, 4 H, 5 sqrt(rho), 6-8 F  (advection: 0 u).
// Sixth-order Euler projects differences of adjacent cells, as the 2D
// kernel does (euler2d_tile6): dd holds per cell pair d rho, dm, dE, dF1, dF2
// (dF0 = dm), and the centre values come back as 4 F_i + 2 (F_{i+1} - F_i)
// after the back-projection.
// ---------------------------------------------------------------------------
// The centre values of a sixth-order 1D Euler face between cells L and L+1 of
// the staged fluxes pl[6..8] (R L = I).  With dd, FP64 differences:
// 4 F_hat += 4 F_L + 2 dF of pair L; without, from the fields' 6 h: the face
// gets 2 F_hat, F_L + F_{L+1} and a twelfth of what backproject3 gives.
template <int REG>
__device__ __forceinline__ void add_centre3(const double (*pl)[REG], const double *dd, int nd,
                                            int L, double &F0, double &F1, double &F2) {
  if (dd) {
    F0 = fma(4.0, pl[6][L], fma(2.0, dd[nd + L], F0));
    F1 = fma(4.0, pl[7][L], fma(2.0, dd[3 * nd + L], F1));
    F2 = fma(4.0, pl[8][L], fma(2.0, dd[4 * nd + L], F2));
  } else {
    F0 = fma(1.0 / 12.0, F0, pl[6][L] + pl[6][L + 1]);
    F1 = fma(1.0 / 12.0, F1, pl[7][L] + pl[7][L + 1]);
    F2 = fma(1.0 / 12.0, F2, pl[8][L] + pl[8][L + 1]);
  }
}

// The projected differences of field m of face f in FP64 from the staged cells.
template <int REG>
__device__ __forceinline__ void wide_differences3(const double (*pl)[REG], int f, int m,
                                                  const FaceState &fs, double (&dw)[5],
                                                  double (&dg)[5]) {
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const int k = f + j;
    dw[j] = project3_field(fs, m, pl[0][k + 1] - pl[0][k], pl[1][k + 1] - pl[1][k],
                           pl[2][k + 1] - pl[2][k]);
    dg[j] = project3_field(fs, m, pl[6][k + 1] - pl[6][k], pl[7][k + 1] - pl[7][k],
                           pl[8][k + 1] - pl[8][k]);
  }
}
// The packed differences of a face for the integer path.
template <int ND>
struct PackedFace3 {
  const fx::u64 *pf;
  __device__ __forceinline__ fx::u64 operator()(int s, int q, int j) const {
    return pf[(s ? (q == 0 ? 1 : 2 + q) : q) * ND + j];
  }
};
// Face f with all its fields in FP64 from the staged cells: what the integer
// path leaves out.  al: the speed maxima; out: the face.
template <int REG, int AI>
__device__ __noinline__ void face_wide3(const double (*pl)[REG], int f, double gm1,
                                        const unsigned long long *al, int alpha_single,
                                        const SchemeParams &scheme, double *out) {
  FaceState fs = {};
  const int kL = f + 2, kR = f + 3;
  roe_face(pl[5][kL], pl[3][kL], 0.0, pl[4][kL], pl[5][kR], pl[3][kR], 0.0, pl[4][kR], gm1, fs);
  double h[3];
#pragma unroll 1
  for (int m = 0; m < 3; ++m) {
    double dw[5], dg[5];
    const double A = field_speed(alpha_single, al, m, 3);
    wide_differences3<REG>(pl, f, m, fs, dw, dg);
    h[m] = 6.0 * pair_wide<AI, true>(-A * dw[2], dw, dg, A, scheme.rp[m == 1 ? 0 : 1]);
  }
  double F0, F1, F2;
  backproject3(fs, h[0], h[1], h[2], F0, F1, F2);
  add_centre3<REG>(pl, nullptr, 0, kL, F0, F1, F2);
  out[0] = F0;
  out[1] = F1;
  out[2] = F2;
}

// Lanes per face of the latency layout and its cells per 128-thread tile: a
// scalar's positive and negative flux (2); for Euler a characteristic field
// each (3: p != 1 and FP32 reconstruction), or each flux of a field (6, five
// faces a warp so that a face's lanes can shuffle).
__host__ __device__ constexpr int lanes1d(int nc, bool p1, int prec) {
  return nc == 1 ? 2 : (p1 && prec == 0 ? 6 : 3);
}
__host__ __device__ constexpr int cells_lanes1d(int lanes) {
  return lanes == 2 ? 63 : (lanes == 3 ? 41 : 19);
}

template <int NC, int T, int R = 3, int LANES = 1>
constexpr size_t smem_line1d() {
  return sizeof(double) * (((NC == 3) ? 9 : 2) * (T + 2 * R) + (T + 1) * NC +
                           (LANES > 1 ? (T + 1) * NC : 0) +
                           ((NC == 3 && R == 3) ? 5 * (T + 2 * R - 1) : 0));
}

// One tile of T cells (T + 1 faces) of a 1D stage with a stencil of
// half-width R (order 2R).  LANES threads share a face: 1 (blockDim = T + 1,
// the throughput layout), or, for problems too small to fill the GPU, where a
// stage's time is one thread's chain of operations, lanes1d() of them.  Every
// lane layout runs the same arithmetic per field, so the results are bitwise
// identical.
// sm: dynamic shared memory of smem_line1d<NC, T, R, LANES>() bytes.
template <int NC, int AI, bool P1, int PREC, int T, int R = 3, int LANES = 1>
__device__ __forceinline__ void line1d_tile(const StageArgs &a, long long b, long long tile,
                                            bool zeroing_block, double *sm) {
  static_assert(R == 3 || PREC == 0, "FP32 reconstruction is sixth order only");
  static_assert(LANES == 1 || (R == 3 && LANES == lanes1d(NC, P1, PREC) && (NC == 3 || PREC == 0)),
                "lane layouts: sixth order, see lanes1d");
  constexpr int REG = T + 2 * R, N = 2 * R;
  constexpr int NP = (NC == 3) ? 9 : 2;
  double(*pl)[REG] = reinterpret_cast<double(*)[REG]>(sm);
  double(*fl)[NC] = reinterpret_cast<double(*)[NC]>(sm + NP * REG);
  double *const hb = sm + NP * REG + (T + 1) * NC;  // LANES > 1: per-field fluxes
  constexpr bool kDiff = (NC == 3 && R == 3);
  constexpr int ND = REG - 1;  // cell pairs of the tile
  double *const dd = hb + (LANES > 1 ? (T + 1) * NC : 0);  // kDiff: [5][ND]
  // p = 1 in FP64: packed differences, projected on the integer pipes
  constexpr bool kPacked = kDiff && P1 && PREC == 0;
  fx::u64 *const dp = reinterpret_cast<fx::u64 *>(dd);
  const long long i0 = tile * T;
  double dt;
  if (!stage_control(a, b, tile == 0, zeroing_block, dt)) return;
  const long long nx = a.nx;
  const double *Ub = a.Uin + b * NC * nx;
  const double gm1 = a.gamma - 1.0;
  const int tid = threadIdx.x;
  // the scheme's constants and speeds, published by the barrier after the staging
  __shared__ SchemeParams s_scheme;
  load_scheme(a, s_scheme);
  const ReconParams *const s_rp = s_scheme.rp;
  const Recon32 &s_r32 = s_scheme.r32;
  __shared__ Speeds s_sp;
  if constexpr (kPacked) make_speeds(a, b, 3, s_sp);

  for (int k = tid; k < REG; k += blockDim.x) {
    const long long gi = ghost(i0 - R + k, nx, a.bc_x);
    if (NC == 1) {
      const double u = Ub[gi];
      if (!(u == u) || fabs(u) > 1.7e308) record_status(a.status, 3, a.stage, b, 0, gi);
      pl[0][k] = u;
      pl[1][k] = scalar_flux(a.system, a.adv_speed, u);
    } else {
      const double rho = Ub[gi], m = Ub[nx + gi], E = Ub[2 * nx + gi];
      const double rs = rsqrt_pos(rho);
      const double ir = rs * rs;
      const double u = m * ir;
      const double p = gm1 * (E - 0.5 * (m * u));
      if (!(pos_finite(rho) && pos_finite(p))) record_status(a.status, 3, a.stage, b, 0, gi);
      const double rH = E + p;
      pl[0][k] = rho;
      pl[1][k] = m;
      pl[2][k] = E;
      pl[3][k] = u;
      pl[4][k] = rH * ir;
      pl[5][k] = rho * rs;
      pl[6][k] = m;
      pl[7][k] = fma(m, u, p);
      pl[8][k] = rH * u;
    }
  }
  __syncthreads();
  if constexpr (kDiff) {
    for (int k = tid; k < ND; k += blockDim.x) {
      const double d[5] = {pl[0][k + 1] - pl[0][k], pl[1][k + 1] - pl[1][k],
                           pl[2][k + 1] - pl[2][k], pl[7][k + 1] - pl[7][k],
                           pl[8][k + 1] - pl[8][k]};
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        if constexpr (kPacked)
          dp[q * ND + k] = fx::pack(d[q]);
        else
          dd[q * ND + k] = d[q];
      }
    }
    __syncthreads();
  }

  if constexpr (LANES == 3) {
    // one characteristic field per thread; the field-0 thread back-projects
    const int f = tid / 3, q = tid - 3 * f;
    const bool act = (f <= T) && (i0 + f - 1 < nx);
    FaceState fs;
    if (act) {
      const int kL = f + 2, kR = f + 3;
      if (!roe_face(pl[5][kL], pl[3][kL], 0.0, pl[4][kL], pl[5][kR], pl[3][kR], 0.0, pl[4][kR],
                    gm1, fs) && q == 0)
        record_status(a.status, 3, a.stage, b, 0, i0 + f);
      const unsigned long long *al = a.alpha_in + b * 8;
      const double A = field_speed(a, al, q, 3);
      double h;
      double dW[5], dG[5];  // the field's projected differences over pairs f .. f+4
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const int k = f + j;
        dW[j] = project3_field(fs, q, dd[k], dd[ND + k], dd[2 * ND + k]);
        dG[j] = project3_field(fs, q, dd[ND + k], dd[3 * ND + k], dd[4 * ND + k]);
      }
      if constexpr (PREC == 1)
        h = field_flux_f32d<P1>(dW, dG, A, s_r32);
      else
        h = field_flux<AI, P1>(dW, dG, A, s_rp[q == 1 ? 0 : 1], 0.0);
      hb[3 * f + q] = h;
    }
    __syncthreads();
    if (act && q == 0) {
      double F0, F1, F2;
      backproject3(fs, hb[3 * f], hb[3 * f + 1], hb[3 * f + 2], F0, F1, F2);
      add_centre3<REG>(pl, dd, ND, f + 2, F0, F1, F2);
      fl[f][0] = F0;
      fl[f][1] = F1;
      fl[f][2] = F2;
    }
  } else if constexpr (LANES == 6) {
    // lane l < 30 of a warp: face 5 warp + l / 6, field (l % 6) % 3, and of its
    // pair of lanes the first projects the state and reconstructs the positive
    // flux, the second the physical flux and the mirrored negative one
    const int lane = tid & 31, l = min(lane, 29), r = l % 6, q = r % 3, sgn = r / 3;
    const int f = min(5 * (tid >> 5) + l / 6, T);
    const bool act = lane < 30 && i0 + f - 1 < nx;
    const int other = lane < 30 ? lane + (sgn ? -3 : 3) : lane;
    FaceState fs = {};
    const int kL = f + 2, kR = f + 3;
    if (!roe_face(pl[5][kL], pl[3][kL], 0.0, pl[4][kL], pl[5][kR], pl[3][kR], 0.0, pl[4][kR], gm1,
                  fs) && act && r == 0)
      record_status(a.status, 3, a.stage, b, 0, i0 + f);
    const PackedFace3<ND> diff = {dp + f};
    int E[3], B0, B2, top;
    const int ea = s_sp.ea[0], eb = s_sp.eb[0];
    const bool in = face_exponents<3>(ea, eb, diff, E, B0, B2, top);
    const fx::LeftRows<3> rows = face_rows<3>(fs, E, B0, B2, ea, eb);
    // all fields of a face that has one left to FP64 go there (face_wide3); a
    // warp of such faces skips the integer path
    const bool ok = in && rows.emax < 2047 &&
                    (top == 0 || !uneven_face<3>(fs, rows, ea, eb, pl[5][kL], pl[5][kR], diff));
    const ReconParams &rp = s_rp[q == 1 ? 0 : 1];
    bool wide = !ok;
    double h = 0.0;
    if (__any_sync(0xffffffffu, ok)) {
      fx::i64 v[5];
      const int as = sgn ? ea : 0, as1 = sgn ? eb : 0;
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const fx::u64 d[3] = {diff(sgn, 0, j), diff(sgn, 1, j), diff(sgn, 2, j)};
        const fx::Proj p = fx::project<3>(rows, E, as, as1, d);
        v[j] = q == 1 ? fx::entropy<3>(rows, as, as1, p) : (q == 0 ? p.z + p.tc : p.z - p.tc);
      }
      const int k0 = (q == 1 ? rows.ue + eb : rows.um + ea) - 1592;
      h = field_lanes<AI>(v, s_sp.ka[0][q], k0, ok, sgn, other, rp, wide);
    }
    const unsigned todo = __ballot_sync(0xffffffffu, wide);
    if (todo != 0) {
      const bool mine = (todo >> (l - r) & 63u) != 0;
      ZA6Part part = {0.0, 1.0};
      double base = 0.0;
      if (mine) {
        double dw[5], dg[5];
        const double A = field_speed(a, a.alpha_in + b * 8, q, 3);
        wide_differences3<REG>(pl, f, q, fs, dw, dg);
        base = -A * dw[2];
        part = recon_wide<AI, true>(dw, dg, A, sgn, rp);
      }
      const ZA6Part mate = {__shfl_sync(0xffffffffu, part.num, other),
                            __shfl_sync(0xffffffffu, part.den, other)};
      if (mine && sgn == 0) h = 6.0 * pair_flux(base, part, mate);
    }
    const double h1 = __shfl_sync(0xffffffffu, h, min(lane + 1, 31)),
                 h2 = __shfl_sync(0xffffffffu, h, min(lane + 2, 31));
    if (act && r == 0) {
      double F0, F1, F2;
      backproject3(fs, h, h1, h2, F0, F1, F2);
      add_centre3<REG>(pl, nullptr, 0, kL, F0, F1, F2);
      fl[f][0] = F0;
      fl[f][1] = F1;
      fl[f][2] = F2;
    }
  } else if constexpr (LANES == 2) {
    // the positive (even lane) and the mirrored negative flux (odd lane) of a
    // scalar face, the operations of field_flux: the corrections meet by a lane
    // shuffle, and so do the FP64 parts where a face of the warp needs those
    const int f = tid >> 1, sgn = tid & 1;
    const bool act = (f <= T) && (i0 + f - 1 < nx);
    double dw[5] = {}, dg[5] = {}, xw[5] = {};
    double A = 0.0, base = 0.0;
    bool fixed = false, flat = false, lost = false;
    fx::i64 c = 0;
    const ReconParams &rp = s_rp[0];
    double scale = 0.0;
    if (act) {
      A = scalar_alpha_of(a.system, a.adv_speed, a.ustar, a.alpha_in + b * 8);
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        dw[j] = pl[0][f + j + 1] - pl[0][f + j];
        dg[j] = pl[1][f + j + 1] - pl[1][f + j];
        xw[j] = __dmul_rn(A, dw[j]);
      }
      const double centre = pl[1][f + 2] + pl[1][f + 3];
      base = __dsub_rn(centre, xw[2]);
      if constexpr (P1) {
        const int es = fx::top_exponent(xw, dg);
        fixed = es >= rp.es_lo && es <= rp.es_hi && !fx::uneven(xw, dg, es, centre);
        fx::i64 x[5], g[5];
        if (fixed) {
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            x[j] = fx::to_fixed(xw[j], es);
            g[j] = fx::to_fixed(dg[j], es);
          }
          fixed = !fx::lost_pair(x, g);
        }
        if (fixed) {
          fx::i64 d[5];
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            if (sgn)
              d[4 - j] = x[j] - g[j];
            else
              d[j] = x[j] + g[j];
          }
          c = recon_fixed<AI>(d, es - 1079, rp);
          scale = fx::scale_back(es);
        } else {
          unsigned long long any = 0;
#pragma unroll
          for (int j = 0; j < 5; ++j)
            any |= (unsigned long long)(__double_as_longlong(xw[j]) | __double_as_longlong(dg[j])) << 1;
          flat = any == 0;
        }
      }
    }
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    double h = flat ? base : __fma_rn((double)c, scale, base);
    // (a flux that the integer path gives up takes its face along)
    const unsigned gone = __ballot_sync(0xffffffffu, lost) >> (tid & 30) & 3u;
    const bool wide = act && !flat && (!fixed || gone != 0);
    if (__any_sync(0xffffffffu, wide)) {
      ZA6Part part = {0.0, 1.0};
      if (wide) part = recon_wide<AI, P1>(dw, dg, A, sgn, rp);
      const ZA6Part mate = {__shfl_xor_sync(0xffffffffu, part.num, 1),
                            __shfl_xor_sync(0xffffffffu, part.den, 1)};
      if (wide) h = pair_flux(base, part, mate);
    }
    if (act && sgn == 0) fl[f][0] = h;
  } else {
    const int f = tid;  // face between cells i0+f-1 and i0+f; stencil f..f+2R-1
    if (f <= T && i0 + f - 1 < nx) {
      if (NC == 1) {
        const double A = scalar_alpha_of(a.system, a.adv_speed, a.ustar, a.alpha_in + b * 8);
        double h;
        if constexpr (PREC == 1) {
          double w[6], g[6];
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            w[j] = pl[0][f + j];
            g[j] = pl[1][f + j];
          }
          h = field_flux_f32<P1>(w, g, A, s_r32);
        } else if constexpr (R == 3) {
          double dw[5], dg[5];
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            dw[j] = pl[0][f + j + 1] - pl[0][f + j];
            dg[j] = pl[1][f + j + 1] - pl[1][f + j];
          }
          h = field_flux<AI, P1>(dw, dg, A, s_rp[0], pl[1][f + 2] + pl[1][f + 3]);
        } else {
          const ReconParams rp = s_rp[0];
          double pp[N], mm[N];  // f^+ in stencil order, f^- mirrored
#pragma unroll
          for (int j = 0; j < N; ++j) {
            const double v = pl[0][f + j], fv = pl[1][f + j];
            pp[j] = fma(A, v, fv);
            mm[N - 1 - j] = fma(-A, v, fv);
          }
          h = pair_flux_r<R>(za_r<R, AI, P1>(pp, rp), za_r<R, AI, P1>(mm, rp));
        }
        fl[f][0] = h;  // 2 F (the split without 1/2); 1/2 goes with 1/dx
      } else {
        const int kL = f + R - 1, kR = f + R;
        FaceState fs;
        if (!roe_face(pl[5][kL], pl[3][kL], 0.0, pl[4][kL], pl[5][kR], pl[3][kR], 0.0, pl[4][kR],
                      gm1, fs))
          record_status(a.status, 3, a.stage, b, 0, i0 + f);
        const unsigned long long *al = a.alpha_in + b * 8;
        const double A1 = field_speed(a, al, 0, 3), A2 = field_speed(a, al, 1, 3),
                     A3 = field_speed(a, al, 2, 3);
        double h1, h2, h3;
        bool done = true;
        if constexpr (kPacked) {
          double hs[3];
          done = face_fields<3, AI>(
              fs, pl[5][kL], pl[5][kR], s_sp.ka[0], s_sp.ea[0], s_sp.eb[0], PackedFace3<ND>{dp + f},
              [&](int m) -> const ReconParams & { return s_rp[m == 1 ? 0 : 1]; }, hs);
          h1 = hs[0];
          h2 = hs[1];
          h3 = hs[2];
        } else if constexpr (R == 3) {
          double dW[3][5], dG[3][5];  // projected differences over pairs f .. f+4
#pragma unroll
          for (int j = 0; j < 5; ++j) {
            const int k = f + j;
            project3(fs, dd[k], dd[ND + k], dd[2 * ND + k], dW[0][j], dW[1][j], dW[2][j]);
            project3(fs, dd[ND + k], dd[3 * ND + k], dd[4 * ND + k], dG[0][j], dG[1][j],
                     dG[2][j]);
          }
          if constexpr (PREC == 1) {
            h1 = field_flux_f32d<P1>(dW[0], dG[0], A1, s_r32);
            h2 = field_flux_f32d<P1>(dW[1], dG[1], A2, s_r32);
            h3 = field_flux_f32d<P1>(dW[2], dG[2], A3, s_r32);
          } else {
            h1 = field_flux<AI, P1>(dW[0], dG[0], A1, s_rp[1], 0.0);
            h2 = field_flux<AI, P1>(dW[1], dG[1], A2, s_rp[0], 0.0);
            h3 = field_flux<AI, P1>(dW[2], dG[2], A3, s_rp[1], 0.0);
          }
        } else {
          const ReconParams rp4 = s_rp[1], rp2 = s_rp[0];
          double p1[N], p2[N], p3[N], m1[N], m2[N], m3[N];  // f^- mirrored
#pragma unroll
          for (int j = 0; j < N; ++j) {
            const int k = f + j;
            double w1, w2, w3, g1, g2, g3;
            project3(fs, pl[0][k], pl[1][k], pl[2][k], w1, w2, w3);
            project3(fs, pl[6][k], pl[7][k], pl[8][k], g1, g2, g3);
            p1[j] = fma(A1, w1, g1);
            m1[N - 1 - j] = fma(-A1, w1, g1);
            p2[j] = fma(A2, w2, g2);
            m2[N - 1 - j] = fma(-A2, w2, g2);
            p3[j] = fma(A3, w3, g3);
            m3[N - 1 - j] = fma(-A3, w3, g3);
          }
          h1 = pair_flux_r<R>(za_r<R, AI, P1>(p1, rp4), za_r<R, AI, P1>(m1, rp4));
          h2 = pair_flux_r<R>(za_r<R, AI, P1>(p2, rp2), za_r<R, AI, P1>(m2, rp2));
          h3 = pair_flux_r<R>(za_r<R, AI, P1>(p3, rp4), za_r<R, AI, P1>(m3, rp4));
        }
        double F0, F1, F2;
        backproject3(fs, h1, h2, h3, F0, F1, F2);
        if constexpr (R == 3)
          add_centre3<REG>(pl, kPacked ? nullptr : dd, ND, kL, F0, F1, F2);
        fl[f][0] = F0;
        fl[f][1] = F1;
        fl[f][2] = F2;
        if constexpr (kPacked)
          if (!done) face_wide3<REG, AI>(pl, f, gm1, al, a.alpha_single, s_scheme, &fl[f][0]);
      }
    }
  }
  __syncthreads();

  // the faces hold 4 F for Euler off the packed path, else 2 F
  const double idx = (NC == 3 && !kPacked ? 0.25 : 0.5) * s_scheme.rdx;
  unsigned long long m3v[3] = {0ull, 0ull, 0ull};
  const bool want_alpha = (NC == 3 || a.system >= 2) && (a.mode == 0) && (a.alpha_out != nullptr);
  if (tid < T && i0 + tid < nx) {
    const long long gi = i0 + tid;
    const long long o = b * NC * nx + gi;
    double uo[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const double L = -(fl[tid + 1][q] - fl[tid][q]) * idx;
      if (a.mode == 1) {
        uo[q] = L;
      } else {
        const double uin = (NC == 1) ? pl[0][tid + R] : pl[q][tid + R];
        const double base_s = fma(dt, L, uin);
        uo[q] = (a.a_n != 0.0) ? fma(a.a_n, a.Un[o + q * nx], a.a_s * base_s) : a.a_s * base_s;
      }
      a.Uout[o + q * nx] = uo[q];
    }
    if (want_alpha && NC == 1) {  // scalar: keys of max u and max -u
      if (!(uo[0] == uo[0]) || fabs(uo[0]) > 1.7e308) record_status(a.status, 3, a.stage, b, 0, gi);
      m3v[0] = okey(uo[0]);
      m3v[1] = okey(-uo[0]);
    } else if (want_alpha) {
      const double ir = rcp_pos(uo[0]);
      const double u = uo[1] * ir;
      const double p = gm1 * (uo[NC - 1] - 0.5 * (uo[1] * u));
      if (!(pos_finite(uo[0]) && pos_finite(p))) record_status(a.status, 3, a.stage, b, 0, gi);
      const double cs = sqrt_pos(a.gamma * p * ir);
      m3v[0] = abs_bits(u - cs);
      m3v[1] = abs_bits(u);
      m3v[2] = abs_bits(u + cs);
    }
  }
  if (want_alpha) {
    const int slot[3] = {0, 1, 2};
    const int dup[3] = {-1, -1, -1};
    block_max_atomic<3>(m3v, a.alpha_out + b * 8, slot, dup);
  }
}

// Three blocks an SM for the Euler faces on the integer pipes: the compiler
// would take 220 registers (two blocks; 64 x 1600 cells: 173 us a step, 151 with three).
template <int NC, int AI, bool P1, int PREC, int R = 3>
__global__ void __launch_bounds__(kThreads1D, (NC == 3 && R == 3 && P1 && PREC == 0) ? 3 : 0)
    k_line1d(const __grid_constant__ StageArgs a) {
  extern __shared__ double sm[];
  pdl_start();
  line1d_tile<NC, AI, P1, PREC, kT1, R>(a, blockIdx.y, blockIdx.x,
                                        blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0, sm);
}

// Latency layout of small 1D problems (lanes1d).
template <int NC, int AI, bool P1, int PREC>
__global__ void __launch_bounds__(kThreads1D) k_line1d_lanes(const __grid_constant__ StageArgs a) {
  extern __shared__ double sm[];
  pdl_start();
  constexpr int kL = lanes1d(NC, P1, PREC);
  line1d_tile<NC, AI, P1, PREC, cells_lanes1d(kL), 3, kL>(
      a, blockIdx.y, blockIdx.x, blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0, sm);
}
