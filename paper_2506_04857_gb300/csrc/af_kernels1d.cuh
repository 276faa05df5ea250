// af_kernels1d.cuh -- the 1D AF scheme (Sec. 4: the 1D tests use the 1D AF
// scheme with the LLF FVS and without the Godunov-Powell source), included at
// the end of af_kernels.cu (the passes) and af_kernels_lat.cu (the step of a
// short grid in one launch) so that it shares the 2D device functions.
//
// The 1D problem runs on the 2D data structures with ny = 1: class 0 holds the
// cell averages (nx), class 1 the interface point values (nxa = nx, or nx + 1
// for outflow; point f is the left face of cell f), pd[4] and uc the cell
// centre values.  With one row the y-neighbours of every index map onto the
// index itself, so the shared pieces reduce to their x parts:
//   - the point update is the x-face line of Sec. 2.3 (point f-1, centre f-1,
//     point f, centre f, point f+1) without the y terms and the source;
//   - the sensor of Sec. 3.4 sees zero y-differences;
//   - the dt pass forms cfl / (max varrho_1 / dx) (the y maximum stays 0).
// Specific to 1D: the centre value of the cell parabola (6 Ubar - U_L - U_R)/4
// (Simpson), the face flux F1 of the face point value (no quadrature across
// the face), the LLF point state between neighbouring points, and the flux
// limiter of Sec. 3.2 with the two faces L, R (the 2D box with the two
// y-directions zero; no source, so U^{Lim,1} = U^LLF).
#pragma once

namespace {

// P1 (1D): point data of the points, the averages and the centre values; dt maximum
// parts: 1 the point, 2 the average, 4 the centre of index i
__device__ __forceinline__ void b1_pointdata(const AfDev &d, const AfGrid &g, int i, int reduce_dt, int parts = 7) {
  const size_t PS = (size_t)g.nxa;
  double m1 = 0.0, s1, s2;
  bool clim = false;
  if ((parts & 1) && i < g.ex[1]) {
    double U[8];
    load8(sview(d.us[1], g, 1), i, 0, U);
    point_data(U, g, d.pd[1] + i, PS, false, s1, s2);
    m1 = maxnn(m1, s1);
  }
  if ((parts & 2) && i < g.nx) {
    double A[8];
    load8(sview(d.us[0], g, 0), i, 0, A);
    point_data(A, g, d.pd[0] + i, PS, true, s1, s2);
    m1 = maxnn(m1, s1);
  }
  if ((parts & 4) && i < g.nx) {
    double A[8], uc[8];
    load8(sview(d.us[0], g, 0), i, 0, A);
    const SV P = sview(d.us[1], g, 1);
    const int ip = mface(i + 1, g.nx, g.bc);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double pl = P(i, 0, k), pr = P(ip, 0, k), v = (fma(6.0, A[k], -pl) - pr) * 0.25;
      // equal values give exactly that value (uniform data stay uniform bit for bit)
      uc[k] = ((bits(pl) ^ bits(A[k])) | (bits(pr) ^ bits(A[k]))) == 0 ? A[k] : v;
    }
    if (!clear_of_floor(uc, g)) {   // Remark 3.2
      double out[8], t1, t2;
      scaling_limiter(uc, A, g.gm1, out, t1, t2);
      clim = t1 < 1.0 || t2 < 1.0;
      for (int k = 0; k < 8; ++k) uc[k] = out[k];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) d.uc[k * PS + i] = uc[k];
    point_data(uc, g, d.pd[4] + i, PS, false, s1, s2);
  }
  count(d.st, ST_CENTER_LIMITED, clim);
  if (reduce_dt) {
    unsigned long long b1 = (unsigned long long)__double_as_longlong(m1);
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long o1 = __shfl_down_sync(0xffffffffu, b1, off);
      b1 = o1 > b1 ? o1 : b1;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&d.sc->smax[0], b1);
  }
}

// Sec. 3.3 slow path for point f: LLF state from the fluxes between f and its
// neighbouring points, scaling limiter, Remark 4.1 shrink.
__device__ __noinline__ void point_pp1(const AfDev &d, const AfGrid &g, int f, const double *UH, double dt,
                                       double *out, int &limited, int &shrunk, int &bad) {
  const int fm = mface(f - 1, g.nx, g.bc), fp = mface(f + 1, g.nx, g.bc);
  const SV P = sview(d.us[1], g, 1);
  double U[8];
  Full me, nb;
  load8(P, f, 0, U);
  full_data(U, g, me);
  double Fl[8], Fr[8];
  load8(P, fm, 0, U);
  full_data(U, g, nb);
  llf_flux_full(0, nb, me, Fl);
  load8(P, fp, 0, U);
  full_data(U, g, nb);
  llf_flux_full(0, me, nb, Fr);
  const double cxf = dt * g.rdx;
  double UL[8];
  for (int k = 0; k < 8; ++k) UL[k] = fma(-cxf, Fr[k] - Fl[k], me.U[k]);
  double t1, t2;
  scaling_limiter(UH, UL, g.gm1, out, t1, t2);
  limited = (t1 < 1.0 || t2 < 1.0);
  shrunk = 0;
  bad = 0;
  if (!in_G(out, g.gm1)) {
    shrunk = 1;
    double Us[8];
    for (int k = 0; k < 8; ++k) Us[k] = UH[k];
    Us[0] = fma(t1, UH[0], (1.0 - t1) * UL[0]);
    bool ok = false;
    for (int m = 0; m < 10 && !ok; ++m) {
      const double th = fmax(0.0, t2 - ldexp(1e-8, m));
      for (int k = 0; k < 8; ++k) out[k] = fma(th, Us[k], (1.0 - th) * UL[k]);
      ok = in_G(out, g.gm1);
    }
    if (!ok)
      for (int k = 0; k < 8; ++k) out[k] = UL[k];
    bad = !in_G(out, g.gm1);
  }
}

// P2 (1D): point update, its limiter and the RK combination; the sensor phi
// parts: 1 the point, 2 the sensor values of cell f
__device__ __forceinline__ void b1_points(const AfDev &d, const AfGrid &g, int f, double a, double b, int parts = 3,
                                          bool pois = false) {
  const size_t PS = (size_t)g.nxa;
  const double dt = pois ? nan_value() : d.sc->dt;
  int nlim = 0, nshr = 0, nbad = 0;
  if ((parts & 1) && f < g.ex[1]) {
    const int fm = mface(f - 1, g.nx, g.bc), fp = mface(f + 1, g.nx, g.bc);
    const int c0 = mcell(f - 1, g.nx, g.bc), c1 = mcell(f, g.nx, g.bc);
    const PP me = pref(d, g, 1, f, 0);
    double acc[8], dB;
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = pu(me, k);
    const PP L[5] = {pref(d, g, 1, fm, 0), pref(d, g, 4, c0, 0), me, pref(d, g, 4, c1, 0), pref(d, g, 1, fp, 0)};
    fvs_line<0, false>(L, PS, g.nxa, 0.5 * dt * g.rdx, acc, dB, 0);
    if (g.pp_on && !clear_of_floor(acc, g)) {
      double out[8];
      int lim, shr, bad;
      point_pp1(d, g, f, acc, dt, out, lim, shr, bad);
      nlim += lim;
      nshr += shr;
      nbad += bad;
      for (int k = 0; k < 8; ++k) acc[k] = out[k];
    }
    const size_t cs = (size_t)g.ex[1];
    rk_store(d.uo[1] + f, d.un[1] + f, cs, a, b, acc);
  }
  if ((parts & 2) && f < g.nx && g.kappa != 0.0) {
    double phi[4];
    sensor_phi<false>(d, g, f, 0, phi);
#pragma unroll
    for (int q = 0; q < 4; ++q) d.phi[q * PS + f] = phi[q];
  }
  if (nlim) atomicAdd(&d.st->cnt[ST_POINT_LIMITED], (unsigned long long)nlim);
  if (nshr) atomicAdd(&d.st->cnt[ST_SHRINK], (unsigned long long)nshr);
  if (nbad) {
    atomicAdd(&d.st->cnt[ST_NONADMISSIBLE], (unsigned long long)nbad);
    atomicOr(&d.st->err, AFE_NONADMISSIBLE);
  }
}

// P3 (1D): per face f, F^LLF between the adjacent averages, G = theta^s (F1(U_f) - F^LLF),
// theta^s and alpha^LLF (slots of the 2D face layout)
__device__ __forceinline__ void b1_faces(const AfDev &d, const AfGrid &g, int f) {
  const size_t PS = (size_t)g.nxa;
  int nsens = 0;
  if (f < g.ex[1]) {
    const int ca = mcell(f - 1, g.nx, g.bc), cb = mcell(f, g.nx, g.bc);
    const WV A = wview(d.pd[0], g), PW = wview(d.pd[1], g);
    const SV Ub = sview(d.us[0], g, 0);
    const double Ba[3] = {Ub(ca, 0, 4), Ub(ca, 0, 5), Ub(ca, 0, 6)};
    const double Bb[3] = {Ub(cb, 0, 4), Ub(cb, 0, 5), Ub(cb, 0, 6)};
    const double al = alpha_llf(A(ca, 0, QA_V1), A(cb, 0, QA_V1), A(ca, 0, QA_CF1), A(cb, 0, QA_CF1),
                                A(ca, 0, QA_SRHO), A(cb, 0, QA_SRHO), Ba, Bb);
    // unmapped cell indices: an outflow ghost cell's phi comes from its own (mirrored) neighbours
    const double ts = theta_s<false>(d, g, 0, f - 1, 0, f, 0);
    double *out = d.fx + f;
    double Fl[8], G[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      double Fh = 0.0;
      if (k != 4) {
        const int s = QP_F1 + fslot(0, k);
        Fh = PW(f, 0, s);
        Fl[k] = 0.5 * fma(-al, Ub(cb, 0, k) - Ub(ca, 0, k), A(ca, 0, s) + A(cb, 0, s));
      } else {
        Fl[k] = -0.5 * al * (Ub(cb, 0, k) - Ub(ca, 0, k));
      }
      G[k] = is_one(ts) ? Fh - Fl[k] : ts * (Fh - Fl[k]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      out[(QF_FLLF + k) * PS] = Fl[k];
      out[(QF_G + k) * PS] = G[k];
    }
    out[QF_TS * PS] = ts;
    out[QF_AL * PS] = al;
    nsens = ts < 0.99;
  }
  if (g.kappa != 0.0 && nsens) atomicAdd(&d.st->cnt[ST_SENSOR_LT099], 1ull);
}

// P4 (1D): per cell, U^LLF = U^{Lim,1}, the anti-diffusive fluxes H_L, H_R and
// Lambda_L, Lambda_R (or the unlimited update without PP)
// The FP64 bounds D_k = |dt/dx G_L,k| + |dt/dx G_R,k| and box certificate of 1D cell i
// for the states box_cert32 leaves undecided (not inlined; Lim1 by value, G reloaded)
__device__ __noinline__ bool box_cert64_1d(const AfDev &d, const AfGrid &g, int i, int ip, double l0, double l1,
                                           double l2, double l3, double l4, double l5, double l6, double l7,
                                           double cxf) {
  const WV FX = wview(d.fx, g);
  const double L1[8] = {l0, l1, l2, l3, l4, l5, l6, l7};
  double D[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) D[k] = absd(cxf * FX(i, 0, QF_G + k)) + absd(-cxf * FX(ip, 0, QF_G + k));
  return box_certified(L1, D, g);
}

__device__ __forceinline__ void b1_cells(const AfDev &d, const AfGrid &g, int i, double a, double b, bool pois = false) {
  const size_t PS = (size_t)g.nxa;
  int nlam = 0, ncfl = 0;
  NewtonLog nl = {0, 0};
  if (i < g.nx) {
    const double dt = pois ? nan_value() : d.sc->dt, cxf = dt * g.rdx;
    const int ip = mface(i + 1, g.nx, g.bc);
    const WV FX = wview(d.fx, g);
    const SV Ub = sview(d.us[0], g, 0);
    double Ullf[8], H[4][8], Gf[4][8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const double fl = FX(i, 0, QF_FLLF + k), fr = FX(ip, 0, QF_FLLF + k);
      const double gl = FX(i, 0, QF_G + k), gr = FX(ip, 0, QF_G + k);
      Ullf[k] = fma(-cxf, fr - fl, Ub(i, 0, k));
      H[0][k] = cxf * gl;
      H[1][k] = -cxf * gr;
      H[2][k] = 0.0;
      H[3][k] = 0.0;
      Gf[0][k] = gl;
      Gf[1][k] = gr;
      Gf[2][k] = Gf[3][k] = 0.0;
    }
    const size_t cs0 = (size_t)g.nx;
    if (!g.pp_on) {
      // no PP: the blended high-order update, then the RK combination
      double fe[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) fe[k] = Ullf[k] + H[0][k] + H[1][k];
      rk_store(d.uo[0] + i, d.un[0] + i, cs0, a, b, fe);
    } else {
      if (dt * ((FX(i, 0, QF_AL) + FX(ip, 0, QF_AL)) * g.rdx) > 1.0 + 1e-12) ncfl = 1;   // Lemma 3.1 (count only)
      double Lam[4];
      // fast path: where the box provably needs no limiting, Lambda = 1 exactly
      // (the FP32 certificates of the 2D cell pass, with the lower and upper face values 0;
      // the FP64 forms only for the states they leave undecided)
      bool fast = clear_of_floor(Ullf, g);
      if (fast)
        fast = box_cert32(Ullf, Gf, cxf, 0.0, g.c13) ||
               box_cert64_1d(d, g, i, ip, Ullf[0], Ullf[1], Ullf[2], Ullf[3], Ullf[4], Ullf[5], Ullf[6], Ullf[7], cxf);
      if (fast) {
        Lam[0] = Lam[1] = 1.0;
      } else {
        const double eps_rho = fmin(1e-13, Ullf[0]);
        const double eps_p = fmin(1e-13, pressure(Ullf, g.gm1));
        flux_limiter_box(Ullf, H, eps_rho, eps_p, g.gm1, Lam, nl);
        nlam = lt_one(Lam[0]) || lt_one(Lam[1]);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) d.lim1[k * PS + i] = Ullf[k];
      d.lam[0 * PS + i] = Lam[0];
      d.lam[1 * PS + i] = Lam[1];
    }
  }
  if (nlam) atomicAdd(&d.st->cnt[ST_LAMBDA_LT1], 1ull);
  if (ncfl) atomicAdd(&d.st->cnt[ST_CFL_VIOLATIONS], 1ull);
  if (nl.solves) {
    atomicAdd(&d.st->cnt[ST_NEWTON_SOLVES], (unsigned long long)nl.solves);
    atomicMax(&d.st->cnt[ST_NEWTON_MAXIT], (unsigned long long)nl.maxit);
  }
}

// face coefficient of face f: min(Lambda_R(f-1), Lambda_L(f)); an outflow
// boundary face takes the Lambda of its one cell
__device__ __forceinline__ double theta1(const AfGrid &g, const WV &L, int f) {
  if (g.bc == 1) {
    if (f == 0) return L(0, 0, 0);
    if (f == g.nx) return L(g.nx - 1, 0, 1);
    return minnn(L(f - 1, 0, 1), L(f, 0, 0));
  }
  return minnn(L(wrapi(f - 1, g.nx), 0, 1), L(wrapi(f, g.nx), 0, 0));
}

__device__ __forceinline__ void value1(const AfDev &d, const AfGrid &g, int i, double tl, double tr, double dt,
                                       double *out) {
  const WV FX = wview(d.fx, g), L1 = wview(d.lim1, g);
  const int ip = mface(i + 1, g.nx, g.bc);
  const double cxf = dt * g.rdx;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    out[k] = fma(cxf, fma(-tr, FX(ip, 0, QF_G + k), tl * FX(i, 0, QF_G + k)), L1(i, 0, k));
}

// P5 (1D): face coefficients, the limited update, the admissibility check, RK
__device__ __forceinline__ void b1_final(const AfDev &d, const AfGrid &g, int i, double a, double b) {
  int nface = 0;
  if (i < g.nx) {
    const double dt = d.sc->dt;
    const WV L = wview(d.lam, g);
    const double tl = theta1(g, L, i), tr = theta1(g, L, i + 1);
    double fe[8];
    value1(d, g, i, tl, tr, dt, fe);
    rk_store(d.uo[0] + i, d.un[0] + i, (size_t)g.nx, a, b, fe);
    d.thx[i] = tl;
    nface += lt_one(tl);
    if (g.bc == 1 && i == g.nx - 1) {
      d.thx[i + 1] = tr;
      nface += lt_one(tr);
    }
    bool ok = fe[0] > 0.0 && qform(fe, 0.0) > 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) ok = ok && finite_bits(fe[k]);
    if (!ok) {
      const int slot = atomicAdd(&d.st->nrepair, 1);
      if (slot < AF_MAX_REPAIR) d.st->repair[slot] = i;
      else atomicOr(&d.st->err, AFE_REPAIR_OVERFLOW);
    }
  }
  if (nface) atomicAdd(&d.st->cnt[ST_FACE_THETA_LT1], (unsigned long long)nface);
}

// Remark 4.1 for the flagged cells, one thread, in cell order (as in 2D, two faces)
__device__ void b1_repair(const AfDev &d, const AfGrid &g, double a, double b) {
  int n = d.st->nrepair;
  if (n <= 0) return;
  if (n > AF_MAX_REPAIR) n = AF_MAX_REPAIR;
  int *list = d.st->repair;
  for (int p = 1; p < n; ++p) {
    int v = list[p], q = p - 1;
    while (q >= 0 && list[q] > v) { list[q + 1] = list[q]; --q; }
    list[q + 1] = v;
  }
  const double dt = d.sc->dt;
  const size_t cs0 = (size_t)g.nx;
  unsigned long long nshr = 0, nbad = 0;
  auto face_idx = [&](int f) { return g.bc == 0 ? wrapi(f, g.nx) : f; };
  auto store = [&](int c, const double *fe) {
    for (int k = 0; k < 8; ++k)
      d.uo[0][k * cs0 + c] = a == 0.0 ? fe[k] : fma(a, d.un[0][k * cs0 + c], b * fe[k]);
  };
  for (int p = 0; p < n; ++p) {
    const int i = list[p];
    double fe[8];
    value1(d, g, i, d.thx[face_idx(i)], d.thx[face_idx(i + 1)], dt, fe);
    if (in_G(fe, g.gm1)) continue;
    nshr++;
    const double t0[2] = {d.thx[face_idx(i)], d.thx[face_idx(i + 1)]};
    for (int m = 0; m <= 10; ++m) {
      double t[2];
      for (int I = 0; I < 2; ++I) t[I] = (m < 10) ? fmax(0.0, t0[I] - ldexp(1e-8, m)) : 0.0;
      value1(d, g, i, t[0], t[1], dt, fe);
      if (in_G(fe, g.gm1) || m == 10) {
        d.thx[face_idx(i)] = t[0];
        d.thx[face_idx(i + 1)] = t[1];
        store(i, fe);
        if (!in_G(fe, g.gm1)) nbad++;
        break;
      }
    }
    for (int q = -1; q <= 1; q += 2) {
      int c = i + q;
      if (g.bc == 1 && (c < 0 || c >= g.nx)) continue;
      c = wrapi(c, g.nx);
      value1(d, g, c, d.thx[face_idx(c)], d.thx[face_idx(c + 1)], dt, fe);
      store(c, fe);
    }
  }
  d.st->nrepair = 0;
  if (nshr) {
    d.st->cnt[ST_SHRINK] += nshr;
    d.st->cnt[ST_CELL_SHRINK] += nshr;
  }
  if (nbad) {
    d.st->cnt[ST_NONADMISSIBLE] += nbad;
    d.st->err |= AFE_NONADMISSIBLE;
  }
}

#ifdef AF_LAT
// A whole step (or the stages s0..s1 of one) of a short grid in one launch of one thread-block
// cluster: the passes follow one another across a cluster barrier.  Arrays stay in global
// memory (L2), written by one CTA of the cluster and read by its neighbours after the barrier,
// whose arrive releases and whose wait acquires at cluster scope.
// What bounds it: latency.  At 800 cells a pass is about 50 threads per SM with 40 to 130
// dependent FP64 instructions of 64 cycles each, and a launch of its own costs more than that.
// threadIdx.y is a role: the point, the average and the centre of a cell side by side in the
// point-data pass, the point and the sensor in the point pass; the other passes deal the
// indices to all threads.
struct AfStages1d {
  AfDev d[3];
};
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
constexpr int kStepThreads = 128;   // of each role, at most
__global__ void __launch_bounds__(3 * kStepThreads) k1_step(const __grid_constant__ AfStages1d S,
                                                            const __grid_constant__ AfGrid g, int s0, int s1,
                                                            int reduce_dt) {
  const int bx = (int)blockDim.x, cs = (int)gridDim.x, rank = (int)blockIdx.x, role = (int)threadIdx.y;
  const int n = g.nxa;
  const bool first = rank == 0 && threadIdx.x == 0 && threadIdx.y == 0;
  // one index per thread of a role, and one per thread of the cluster; the trip counts are uniform in a block
  const int base1 = rank * bx, step1 = cs * bx, base3 = (role * cs + rank) * bx, step3 = 3 * cs * bx;
  for (int s = s0; s <= s1; ++s) {
    const AfDev &d = S.d[s];
    const double a = s == 0 ? 0.0 : (s == 1 ? 3.0 / 4.0 : 1.0 / 3.0), b = s == 0 ? 1.0 : (s == 1 ? 1.0 / 4.0 : 2.0 / 3.0);
    for (int q = base1; q < n; q += step1) b1_pointdata(d, g, q + (int)threadIdx.x, reduce_dt && s == 0, 1 << role);
    cluster_sync();
    if (reduce_dt && s == 0) {
      if (first) b_dt(d, g);
      cluster_sync();
    }
    if (role < 2)
      for (int q = base1; q < n; q += step1) b1_points(d, g, q + (int)threadIdx.x, a, b, 1 << role);
    cluster_sync();
    for (int q = base3; q < n; q += step3) b1_faces(d, g, q + (int)threadIdx.x);
    cluster_sync();
    for (int q = base3; q < n; q += step3) b1_cells(d, g, q + (int)threadIdx.x, a, b);
    cluster_sync();
    if (g.pp_on) {
      for (int q = base3; q < n; q += step3) b1_final(d, g, q + (int)threadIdx.x, a, b);
      cluster_sync();
      // every thread reads the same count: nothing changes it before the next barrier
      if (*(volatile int *)&d.st->nrepair > 0) {
        cluster_sync();
        if (first) b1_repair(d, g, a, b);
        cluster_sync();
      }
    }
  }
}
#else
// Quiet tiles of 128 indices, as in 2D (levels d.lev, one per block)
__device__ __forceinline__ int level1(const AfDev &d) { return d.lev ? d.lev[blockIdx.x] : 0; }
__global__ void __launch_bounds__(kTile1) k1_quiet1(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g) {
  pass_begin();
  const int i0 = blockIdx.x * kTile1, i = i0 + threadIdx.x;
  const SV P = sview(d.us[1], g, 1), A = sview(d.us[0], g, 0);
  bool ok = true;
  for (int s = 0; s < 8 && ok; ++s) {
    const int k = 7 - s;
    const double v = P(i0, 0, k);
    const bool eq = (i >= g.ex[1] || same_value(P(i, 0, k), v)) && (i >= g.nx || same_value(A(i, 0, k), v));
    ok = __all_sync(0xffffffffu, eq);
  }
  ok = __syncthreads_and(ok);
  if (threadIdx.x == 0) {
    if (ok) {
      double V[8];
      load8(P, i0, 0, V);
      ok = ge_pos(V[0], 1e-13) && qform_cert32(V, g.c13);
    }
    d.quiet[blockIdx.x] = ok;
  }
}
__global__ void __launch_bounds__(128) k1_quiet23(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                                  int pass) {
  pass_begin();
  b_quiet23<kTile1, 1, 1>(d, g, pass);
}
// As quiet_cfl, one dimension
__device__ __noinline__ bool quiet_cfl1(const AfDev &d, const AfGrid &g, int i) {
  double V[8];
  load8(sview(d.us[0], g, 0), i, 0, V);
  const double dt = d.sc->dt;
  const float rho = (float)V[0], bb = (float)(V[4]) * (float)(V[4]) + (float)(V[5]) * (float)(V[5]) + (float)(V[6]) * (float)(V[6]);
  const float cf = sqrtf((1.0001f * (float)(g.gamma * g.gm1) * (float)V[7] + bb) / rho);
  if (2.0f * (float)dt * (fabsf((float)V[1]) / rho + cf) * (float)g.rdx < 0.999f) return false;
  Full f;
  full_data(V, g, f);
  const double al = alpha_llf(f.v[0], f.v[0], f.cf[0], f.cf[0], f.srho, f.srho, f.B, f.B);
  return dt * ((al + al) * g.rdx) > 1.0 + 1e-12;
}

// blockIdx.y: the point, the average or the centre of a cell (one body at a time in the
// instruction cache, as in 2D)
__global__ void __launch_bounds__(128) k1_pointdata(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                                    int reduce_dt) {
  pass_begin();
  if (level1(d) > 4 && !(reduce_dt && blockIdx.y == 0 && threadIdx.x < 32)) return;
  b1_pointdata(d, g, blockIdx.x * blockDim.x + threadIdx.x, reduce_dt, 1 << blockIdx.y);
}
// blockIdx.y: the point, the sensor
__global__ void __launch_bounds__(128) k1_points(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                                 double a, double b) {
  pass_begin();
  const int lev = level1(d), i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool pois = lev > 0 && poisoned(d);
  if (blockIdx.y == 0 && lev > 0 && !pois) {
    if (i < g.ex[1]) {
      double V[8];
      load8(sview(d.us[1], g, 1), i, 0, V);
      rk_store(d.uo[1] + i, d.un[1] + i, (size_t)g.ex[1], a, b, V);
    }
    return;
  }
  if (blockIdx.y == 0 || lev <= 3) b1_points(d, g, i, a, b, 1 << blockIdx.y, pois);
}
__global__ void __launch_bounds__(128) k1_faces(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g) {
  pass_begin();
  if (level1(d) <= 2) b1_faces(d, g, blockIdx.x * blockDim.x + threadIdx.x);
}
__global__ void __launch_bounds__(128) k1_cells(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                                double a, double b) {
  pass_begin();
  const int lev = level1(d), i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool pois = lev > 0 && poisoned(d);
  if (lev > 0) {
    if (i < g.nx && threadIdx.x % 32 == 0 && quiet_cfl1(d, g, i))
      atomicAdd(&d.st->cnt[ST_CFL_VIOLATIONS], (unsigned long long)min(32, g.nx - i));
    if (i < g.nx && lev == 1 && !pois) {
      double V[8];
      load8(sview(d.us[0], g, 0), i, 0, V);
#pragma unroll
      for (int k = 0; k < 8; ++k) d.lim1[(size_t)k * g.nxa + i] = V[k];
      d.lam[i] = d.lam[(size_t)g.nxa + i] = 1.0;
    }
    if (!pois) return;
  }
  b1_cells(d, g, i, a, b, pois);
}
__global__ void __launch_bounds__(128) k1_final(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                                double a, double b) {
  pass_begin();
  const int lev = level1(d), i = blockIdx.x * blockDim.x + threadIdx.x;
  if (lev > 0 && !poisoned(d)) {
    if (i >= g.nx) return;
    double V[8];
    load8(sview(d.us[0], g, 0), i, 0, V);
    rk_store(d.uo[0] + i, d.un[0] + i, (size_t)g.nx, a, b, V);
    if (lev == 1) {
      d.thx[i] = 1.0;
      if (g.bc == 1 && i == g.nx - 1) d.thx[i + 1] = 1.0;
    }
    return;
  }
  b1_final(d, g, i, a, b);
}
__global__ void k1_dt(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g) {
  pass_begin();
  if (threadIdx.x == 0 && blockIdx.x == 0) b_dt(d, g);
}
__global__ void k1_repair(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g, double a, double b) {
  pass_begin();
  if (blockIdx.x == 0 && threadIdx.x == 0) b1_repair(d, g, a, b);
}
#endif

}  // namespace

#ifdef AF_LAT
namespace {
int step_threads(int n, int cs) {
  const int t = ((n + cs - 1) / cs + 31) / 32 * 32;
  return t < kStepThreads ? t : kStepThreads;
}
cudaLaunchConfig_t step_config(int n, int cs, cudaLaunchAttribute *at, cudaStream_t s) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(cs);
  c.blockDim = dim3(step_threads(n, cs), 3);
  c.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = cs;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}
}  // namespace

// The cluster size of k1_step on the current device for n indices: 16, else 8, else 0 (no such cluster
// fits, or it has fewer threads of a role than there are indices).  In the cluster a pass costs a
// barrier instead of a launch, on 16 SMs instead of 152: us a step of smooth data, cluster and pass by
// pass, 800 cells 86 and 118, 2047 99 and 116; with a second round of indices 2300 155 and 120, 4095
// 156 and 128 (blast 273 and 295 at 2047, 333 and 315 at 4095).
int af_lat_step1d_cluster(int n) {
  cudaFuncSetAttribute(k1_step, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  for (int cs = 16; cs >= 8 && n <= cs * kStepThreads; cs /= 2) {
    cudaLaunchAttribute at;
    cudaLaunchConfig_t c = step_config(n, cs, &at, nullptr);
    int k = 0;
    if (cudaOccupancyMaxActiveClusters(&k, k1_step, &c) == cudaSuccess && k > 0) return cs;
    cudaGetLastError();
  }
  return 0;
}
void af_lat_step1d(const AfDev *d, const AfGrid &g, int s0, int s1, int reduce_dt, int cluster, cudaStream_t s) {
  AfStages1d S;
  for (int k = 0; k < 3; ++k) S.d[k] = d[k];
  cudaLaunchAttribute at;
  cudaLaunchConfig_t c = step_config(g.nxa, cluster, &at, s);
  cudaLaunchKernelEx(&c, k1_step, S, g, s0, s1, reduce_dt);
}
#else

// threads per block: a warp until every SM has four of them, which is when the FP64 pipe is full
static unsigned threads1d(const AfGrid &g) { return g.nxa <= 152 * kTile1 ? 32 : kTile1; }
static_assert(kQuiet1Min > 152 * kTile1, "the levels of the 1D tiles are indexed by blocks of kTile1 indices");

// One 1D stage: P1 (with the dt pass when reduce_dt), P2..P5 and the repair
// pass; t (may be NULL) brackets each launch with an event pair.
void af_launch_stage1d(const AfDev &d, const AfGrid &g, double a, double b, int reduce_dt, cudaStream_t s,
                       AfEventTimer *t) {
  const unsigned nt = threads1d(g), nb = (unsigned)((g.nxa + nt - 1) / nt);
  auto timed = [&](int k, auto launch) {
    const bool on = t && t->begin(k, s);
    launch();
    if (t) t->end(on, s);
  };
  timed(AF_K_POINTDATA, [&] {
    if (d.lev) {
      pass(k1_quiet1, nb, nt, s, d, g);
      pass(k1_quiet23, (nb + 127) / 128, 128, s, d, g, 0);
      pass(k1_quiet23, (nb + 127) / 128, 128, s, d, g, 1);
    }
    pass(k1_pointdata, dim3(nb, 3), nt, s, d, g, reduce_dt);
  });
  if (reduce_dt) timed(AF_K_DT, [&] { pass(k1_dt, 1, 32, s, d, g); });
  timed(AF_K_POINTS, [&] { pass(k1_points, dim3(nb, g.kappa != 0.0 ? 2 : 1), nt, s, d, g, a, b); });
  timed(AF_K_FACES, [&] { pass(k1_faces, nb, nt, s, d, g); });
  timed(AF_K_CELLS, [&] { pass(k1_cells, nb, nt, s, d, g, a, b); });
  if (g.pp_on) {
    timed(AF_K_FINAL, [&] { pass(k1_final, nb, nt, s, d, g, a, b); });
    timed(AF_K_REPAIR, [&] { pass(k1_repair, 1, 32, s, d, g, a, b); });
  }
}
size_t af_quiet_tiles1d(const AfGrid &g) { return (size_t)((g.nxa + kTile1 - 1) / kTile1); }
void af_launch_dt1d(const AfDev &d, const AfGrid &g, cudaStream_t s) {
  const unsigned nt = threads1d(g), nb = (unsigned)((g.nxa + nt - 1) / nt);
  pass(k1_pointdata, dim3(nb, 3), nt, s, d, g, 1);
  pass(k1_dt, 1, 32, s, d, g);
}
#endif
