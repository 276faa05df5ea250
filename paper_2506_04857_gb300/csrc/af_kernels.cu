// af_kernels.cu -- sm_103a kernels of one SSP-RK3 stage of the positivity-
// preserving Active Flux scheme for 2D ideal MHD with the Godunov-Powell
// source term (Duan, Chandrashekar, Klingenberg, arXiv:2506.04857).
//
// The stage is split into five passes so that every FP64 quantity is formed
// exactly once (the FP64 pipe is the bound on GB300; the intermediates cost
// HBM traffic, of which there is plenty):
//   P1 k_pointdata : per DoF: primitives, F1, F2, spectral radii (Sec. 1, eq. cf);
//                    per cell: bi-parabola centre value + its limiter (Sec. 2.1,
//                    Remark 3.2); the running max of varrho for dt.
//   P2 k_points    : per x-face / y-face / corner: LLF-FVS update with the
//                    central Powell source (Sec. 2.3), first-order LLF point
//                    schemes and scaling limiter (Sec. 3.3), round-off shrink
//                    (Remark 4.1), RK combination; per cell: shock-sensor phi
//                    (Sec. 3.4).
//   P3 k_faces     : per face: Simpson flux (Sec. 2.2), LLF flux between the
//                    adjacent cell averages (eq. 2d_llf_flux), theta^s (Sec. 3.4).
//   P4 k_cells     : per cell: Powell source on the 3x3 Simpson nodes
//                    (eq. semi_av_src), S^LLF, the sensor blend, steps (1)-(2)
//                    of the parametrized flux limiter (Sec. 3.2) -> Lambda.
//   P5 k_final     : per cell: unique face coefficients (step (3)), limited
//                    update, round-off check, RK combination.
// Points and cells whose limiters may act go to work lists (k_points_slow,
// k_lists).  A one-thread repair kernel applies the round-off shrink of Remark
// 4.1 to the (rare) cell averages that leave the admissible set.
//
// Limiter fast paths: where the paper's limiter provably returns theta = 1
// (all tested quantities clear 1e-13 by a wide margin) the blend is skipped;
// everywhere else the full procedure runs.  Results are identical.
#include "af_stage.cuh"

namespace {

// Blocks of 256 threads per SM the batch kernels are compiled for: the fastest of a sweep (at
// most 64 registers for the point pass, 80 for the point data, 128 for the cells: a 32-run ensemble
// 21.6 -> 20.8 ms with them).
constexpr int kBatchPt = 4, kBatchPd = 3, kBatchCl = 2;
// Batches hand limited points and cells to work lists of their own runs, as single runs do: with
// the slow paths inline the point pass spilled 2.2 kB a thread.
// the nz parts of the work of a tile (DoF classes, face directions) are items of their own, one part
// after the other over all tiles
#define AF_BATCH_LOOP(nz, call)                                   \
  for (int it = blockIdx.x; it < nitems * (nz); it += gridDim.x) { \
    [[maybe_unused]] const int z = it / nitems;                    \
    const int4 w = items[it - z * nitems];                        \
    const AfRun *__restrict__ r = runs + w.x;                     \
    const int i = w.y + threadIdx.x, j = w.z + threadIdx.y;       \
    call;                                                         \
  }

__global__ void __launch_bounds__(256, kBatchPd) kb_pointdata(const AfRun *__restrict__ runs, const int4 *__restrict__ items,
                                                    int nitems, int reduce_dt) {
  AF_BATCH_LOOP(5, b_pointdata(r->d, r->g, i, j, reduce_dt, z + 1));
}
__global__ void kb_dt(const AfRun *__restrict__ runs, int nruns) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nruns) b_dt(runs[t].d, runs[t].g);
}
template <bool UP>
__global__ void __launch_bounds__(256, kBatchPt) kb_points(const AfRun *__restrict__ runs, const int4 *__restrict__ items,
                                                 int nitems, double a, double b) {
  AF_BATCH_LOOP(4, (b_points<false, UP, kPlain>(r->d, r->g, i, j, a, b, 0, z)));
}
__global__ void __launch_bounds__(256) kb_faces(const AfRun *__restrict__ runs, const int4 *__restrict__ items,
                                                int nitems) {
  AF_BATCH_LOOP(2, b_faces<false>(r->d, r->g, i, j, 0, z));
}
__global__ void __launch_bounds__(256, kBatchCl) kb_cells(const AfRun *__restrict__ runs, const int4 *__restrict__ items,
                                                int nitems, double a, double b) {
  AF_BATCH_LOOP(1, (b_cells<false, true, true>(r->d, r->g, i, j, a, b, 0)));
}
__global__ void __launch_bounds__(256) kb_final(const AfRun *__restrict__ runs, const int4 *__restrict__ items,
                                                int nitems, double a, double b) {
  AF_BATCH_LOOP(1, if (r->g.pp_on) b_final(r->d, r->g, i, j, a, b));
}
__global__ void kb_repair(const AfRun *__restrict__ runs, int nruns, double a, double b) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nruns) return;
  if (runs[t].g.pp_on) b_repair(runs[t].d, runs[t].g, a, b);
  runs[t].d.st->npq = runs[t].d.st->ncq = 0;   // the next stage's work lists start empty
}
// The work lists of all runs in one grid: the cell lists of the runs one after the other, then their
// point lists, cut into pieces that the blocks take in turn.  So one limited run among many, or a
// batch of one, has the whole chip for its lists.  A list is cut finely (a half-warp per cell, four
// lanes per point) while the lists of all runs, were they as long, would still fit the grid.
// With 8 blocks for each run's lists a step of one limited 512 x 512 lattice took 33.2 ms (the same run
// alone 3.5), with two of 768 x 768 79.6; now 3.6 and 14.6.
template <class Count, class Piece>
__device__ __forceinline__ void batch_pieces(int nruns, int fine, int &it, int &done, Count count, Piece piece) {
  const int lane = threadIdx.x & 31;
  for (int r0 = 0; r0 < nruns; r0 += 32) {
    const int mine = r0 + lane < nruns ? count(r0 + lane) : 0;
    for (unsigned m = __ballot_sync(0xffffffffu, mine > 0); m; m &= m - 1) {
      const int q = __ffs(m) - 1, n = __shfl_sync(0xffffffffu, mine, q);
      const bool shrt = (long long)n * nruns <= (long long)gridDim.x * fine;
      const int np = shrt ? (n + fine - 1) / fine : (n + kListThreads - 1) / kListThreads;
      for (; it < done + np; it += gridDim.x) piece(r0 + q, n, it - done, shrt);
      done += np;
    }
  }
}
__global__ void __launch_bounds__(kListThreads) kb_lists(const AfRun *__restrict__ runs, int nruns, double a, double b) {
  int it = blockIdx.x, done = 0;   // the block's next piece, the pieces of the lists passed
  batch_pieces(
      nruns, kListThreads / 16, it, done,
      [&](int r) { return runs[r].g.pp_on ? list_length(&runs[r].d.st->ncq, runs[r].d.cq_cap) : 0; },
      [&](int r, int n, int p, bool shrt) {
        if (shrt) cells_box_short(runs[r].d, runs[r].g, n, p);
        else cells_box_long(runs[r].d, runs[r].g, n, p * kListThreads, n);
      });
  batch_pieces(
      nruns, kListThreads / 4, it, done,
      [&](int r) { return runs[r].g.pp_on ? list_length(&runs[r].d.st->npq, runs[r].d.pq_cap) : 0; },
      [&](int r, int n, int p, bool shrt) {
        if (shrt) points_short<false>(runs[r].d, runs[r].g, a, b, n, p);
        else points_long<false>(runs[r].d, runs[r].g, a, b, n, p * kListThreads + (int)threadIdx.x, n);
      });
}

// ---------------------------------------------------------------------------
// math self-check: out = rcp(x) (op 0), ddiv(x, y) (op 1), dsqrt(x) (op 2)
// ---------------------------------------------------------------------------
// point data of the inflow state: out = [U (8)][as a point (AF_NQP)][as an average (AF_NQA)]
__global__ void k_inflow_pd(const __grid_constant__ AfGrid g, const double *U, double *out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double u[8], s1, s2;
  for (int k = 0; k < 8; ++k) out[k] = u[k] = U[k];
  point_data(u, g, out + 8, 1, false, s1, s2);
  point_data(u, g, out + 8 + AF_NQP, 1, true, s1, s2);
}
__global__ void k_math_check(int op, const double *x, const double *y, double *out, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  if (op == 0) out[t] = rcp(x[t]);
  else if (op == 1) out[t] = ddiv(x[t], y[t]);
  else if (op == 2) out[t] = dsqrt(x[t]);
  else if (op == 3) out[t] = add_i(x[t], y[t]);
  else if (op == 4) out[t] = mul_i(x[t], y[t]);
  else if (op == 5) out[t] = ge_i(x[t], y[t]) ? 1.0 : 0.0;
  else if (op == 6) out[t] = ge_pos(x[t], y[t]) ? 1.0 : 0.0;
  else if (op == 7) out[t] = gt_pos(x[t], y[t]) ? 1.0 : 0.0;
  else if (op == 8) out[t] = ge_zero(x[t]) ? 1.0 : 0.0;
  else if (op == 9) out[t] = qform_cert32(x + 8 * t, y[0]) ? 1.0 : 0.0;   // x: n states of 8
  else {                                                                  // x: n cases of 8 + 4 x 8
    double Gf[4][8];
    for (int q = 0; q < 4; ++q)
      for (int k = 0; k < 8; ++k) Gf[q][k] = x[40 * t + 8 + 8 * q + k];
    out[t] = box_cert32(x + 40 * t, Gf, y[0], y[1], y[2]) ? 1.0 : 0.0;
  }
}

// FP64 FMA throughput probe: 8 independent register chains per thread.
__global__ void k_fp64_probe(double *out, int iters) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  double a0 = 1.0 + t * 1e-9, a1 = a0 + 0.1, a2 = a0 + 0.2, a3 = a0 + 0.3;
  double a4 = a0 + 0.4, a5 = a0 + 0.5, a6 = a0 + 0.6, a7 = a0 + 0.7;
  const double m = 0.999999, c = 1e-7;
  for (int k = 0; k < iters; ++k) {
    a0 = fma(a0, m, c); a1 = fma(a1, m, c); a2 = fma(a2, m, c); a3 = fma(a3, m, c);
    a4 = fma(a4, m, c); a5 = fma(a5, m, c); a6 = fma(a6, m, c); a7 = fma(a7, m, c);
  }
  out[t] = a0 + a1 + a2 + a3 + a4 + a5 + a6 + a7;
}

// ---------------------------------------------------------------------------
// Example 4.4: the discrete divergence measures of the state bound in d.us.
// Per cell: s1 = sum_{l,m} |(div B)^{l,m}| w_l w_m dx dy over the 3x3 nodes of
// eq. (semi_av_src) (centre node: the limited centre value, as in a stage) and
// s2 = |dy/6 ([R] - [L]) + dx/6 ([T] - [B])|, the Simpson edge integral of B.n
// ([.] = corner + 4 face centre + corner).  Each block reduces its cells in a
// fixed order and writes one partial pair; a one-block pass sums the partials
// in a fixed order, so the result does not depend on scheduling.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_divb(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                              double *partials) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  double s1 = 0.0, s2 = 0.0;
  if (i < g.nx && j < g.ny) {
    const SV Ub = sview(d.us[0], g, 0), X = sview(d.us[1], g, 1), Y = sview(d.us[2], g, 2), C = sview(d.us[3], g, 3);
    const int ip = mface(i + 1, g.nx, g.bc), jp = mface(j + 1, g.ny, g.bc);
    double A[8], uc[8];
    load8(Ub, i, j, A);
    centre_value(d, g, i, j, A, uc);
    double b1[3][3], b2[3][3];   // [l][m]: l along x, m along y
    b1[0][0] = C(i, j, 4); b1[1][0] = Y(i, j, 4); b1[2][0] = C(ip, j, 4);
    b1[0][1] = X(i, j, 4); b1[1][1] = uc[4];      b1[2][1] = X(ip, j, 4);
    b1[0][2] = C(i, jp, 4); b1[1][2] = Y(i, jp, 4); b1[2][2] = C(ip, jp, 4);
    b2[0][0] = C(i, j, 5); b2[1][0] = Y(i, j, 5); b2[2][0] = C(ip, j, 5);
    b2[0][1] = X(i, j, 5); b2[1][1] = uc[5];      b2[2][1] = X(ip, j, 5);
    b2[0][2] = C(i, jp, 5); b2[1][2] = Y(i, jp, 5); b2[2][2] = C(ip, jp, 5);
    const double w[3] = {1.0 / 6.0, 2.0 / 3.0, 1.0 / 6.0};
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        double dx1, dy2;
        if (l == 0) dx1 = fma(4.0, b1[1][m], -3.0 * b1[0][m]) - b1[2][m];
        else if (l == 1) dx1 = b1[2][m] - b1[0][m];
        else dx1 = fma(3.0, b1[2][m], fma(-4.0, b1[1][m], b1[0][m]));
        if (m == 0) dy2 = fma(4.0, b2[l][1], -3.0 * b2[l][0]) - b2[l][2];
        else if (m == 1) dy2 = b2[l][2] - b2[l][0];
        else dy2 = fma(3.0, b2[l][2], fma(-4.0, b2[l][1], b2[l][0]));
        s1 = fma(w[l] * w[m], absd(fma(dx1, g.rdx, dy2 * g.rdy)), s1);
      }
    s1 *= g.dx * g.dy;
    const double right = fma(4.0, b1[2][1], b1[2][0] + b1[2][2]), left = fma(4.0, b1[0][1], b1[0][0] + b1[0][2]);
    const double top = fma(4.0, b2[1][2], b2[0][2] + b2[2][2]), bottom = fma(4.0, b2[1][0], b2[0][0] + b2[2][0]);
    s2 = absd(fma(g.dy, right - left, g.dx * (top - bottom))) * (1.0 / 6.0);
  }
  __shared__ double sh[2][128];
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  sh[0][t] = s1;
  sh[1][t] = s2;
  __syncthreads();
  for (int h = 64; h > 0; h >>= 1) {
    if (t < h) {
      sh[0][t] += sh[0][t + h];
      sh[1][t] += sh[1][t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    const size_t b = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    partials[2 * b] = sh[0][0];
    partials[2 * b + 1] = sh[1][0];
  }
}

// Run diagnostics: per block, the minimum density and pressure of each DoF
// class and the sum of the cell-average densities (AF_NDIAG partials).
__device__ __forceinline__ double nan_min(double a, double b) { return (a != a || a < b) ? a : b; }
__global__ void __launch_bounds__(128) k_diag(const __grid_constant__ AfDev d, const __grid_constant__ AfGrid g,
                                              double *partials) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  double v[AF_NDIAG];
  for (int q = 0; q < 8; ++q) v[q] = inf;
  v[8] = 0.0;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    if (i < g.ex[c] && j < g.ey[c]) {
      double U[8];
      load8(sview(d.us[c], g, c), i, j, U);
      v[c] = U[0];
      v[4 + c] = pressure(U, g.gm1);
      if (c == 0) v[8] = U[0];
    }
  }
  __shared__ double sh[AF_NDIAG][128];
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  for (int q = 0; q < AF_NDIAG; ++q) sh[q][t] = v[q];
  __syncthreads();
  for (int h = 64; h > 0; h >>= 1) {
    if (t < h) {
      for (int q = 0; q < 8; ++q) sh[q][t] = nan_min(sh[q][t], sh[q][t + h]);
      sh[8][t] += sh[8][t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    const size_t b = (size_t)blockIdx.y * gridDim.x + blockIdx.x;
    for (int q = 0; q < AF_NDIAG; ++q) partials[AF_NDIAG * b + q] = sh[q][0];
  }
}

__global__ void __launch_bounds__(256) k_diag_sum(const double *partials, int nblocks, double cell_area, double *out) {
  __shared__ double sh[AF_NDIAG][256];
  const int t = threadIdx.x;
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  double v[AF_NDIAG];
  for (int q = 0; q < 8; ++q) v[q] = inf;
  v[8] = 0.0;
  for (int k = t; k < nblocks; k += 256) {
    for (int q = 0; q < 8; ++q) v[q] = nan_min(v[q], partials[AF_NDIAG * k + q]);
    v[8] += partials[AF_NDIAG * k + 8];
  }
  for (int q = 0; q < AF_NDIAG; ++q) sh[q][t] = v[q];
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h) {
      for (int q = 0; q < 8; ++q) sh[q][t] = nan_min(sh[q][t], sh[q][t + h]);
      sh[8][t] += sh[8][t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    for (int q = 0; q < 8; ++q) out[q] = sh[q][0];
    out[8] = sh[8][0] * cell_area;
  }
}

__global__ void __launch_bounds__(256) k_divb_sum(const double *partials, int nblocks, double *out) {
  __shared__ double sh[2][256];
  const int t = threadIdx.x;
  double a = 0.0, b = 0.0;
  for (int k = t; k < nblocks; k += 256) {
    a += partials[2 * k];
    b += partials[2 * k + 1];
  }
  sh[0][t] = a;
  sh[1][t] = b;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h) {
      sh[0][t] += sh[0][t + h];
      sh[1][t] += sh[1][t + h];
    }
    __syncthreads();
  }
  if (t == 0) {
    out[0] = sh[0][0];
    out[1] = sh[1][0];
  }
}

inline dim3 grid2(int nx, int ny) { return dim3((nx + 31) / 32, (ny + 3) / 4); }

}  // namespace

// Small grids: up to two warps of a part per scheduler (152 SMs x 4 x 2 row tiles of 32).  There a
// pass is one chain of dependent operations long and the short chains of AF_LAT pay; above it the
// FP64 pipe fills and AF_LAT's additional operations cost (a step of Orszag-Tang, AF_LAT against the
// other build: 96 x 96 162 against 238 us, 128 x 128 203 and 262, 192 x 192 344 and 399, 256 x 256 592
// and 542).
bool af_small_grid(const AfGrid &g) { return (long long)af_tiles_x(g) * g.nya <= 152 * 4 * 2; }

// From 2^19 index points on: a stage then takes over a millisecond, the check about 10 us (40 us of
// 8 ms at 2048 x 2048).
bool af_quiet_grid(const AfGrid &g) { return !g.special && g.pp_on && !g.upwind && (long long)g.nxa * g.nya >= 1 << 19; }
void af_launch_quiet(const AfDev &d, const AfGrid &g, cudaStream_t s) { launch_quiet(d, g, s); }

void af_launch_pointdata(const AfDev &d, const AfGrid &g, int reduce_dt, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_pointdata(d, g, reduce_dt, s);
  else launch_pointdata(d, g, reduce_dt, s);
}
void af_launch_points(const AfDev &d, const AfGrid &g, double a, double b, int mode, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_points(d, g, a, b, mode, s);
  else launch_points(d, g, a, b, mode, s);
}
void af_launch_faces(const AfDev &d, const AfGrid &g, int mode, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_faces(d, g, mode, s);
  else launch_faces(d, g, mode, s);
}
void af_launch_cells(const AfDev &d, const AfGrid &g, double a, double b, int mode, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_cells(d, g, a, b, mode, s);
  else launch_cells(d, g, a, b, mode, s);
}
void af_launch_final(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_final(d, g, a, b, s);
  else launch_final(d, g, a, b, s);
}
void af_launch_dt(const AfDev &d, const AfGrid &g, cudaStream_t s) { pass(k_dt, 1, 32, s, d, g); }
void af_launch_repair(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) {
  pass(k_repair, 1, 32, s, d, g, a, b);
}
int af_divb_nblocks(const AfGrid &g) { const dim3 b = grid2(g.nx, g.ny); return (int)(b.x * b.y); }
int af_diag_nblocks(const AfGrid &g) { const dim3 b = grid2(g.nxa, g.nya); return (int)(b.x * b.y); }
void af_launch_diag(const AfDev &d, const AfGrid &g, double *partials, double *out, cudaStream_t s) {
  const dim3 b = grid2(g.nxa, g.nya);
  k_diag<<<b, dim3(32, 4), 0, s>>>(d, g, partials);
  k_diag_sum<<<1, 256, 0, s>>>(partials, (int)(b.x * b.y), g.dx * g.dy, out);
}
void af_launch_divb(const AfDev &d, const AfGrid &g, double *partials, double *out, cudaStream_t s) {
  const dim3 b = grid2(g.nx, g.ny);
  k_divb<<<b, dim3(32, 4), 0, s>>>(d, g, partials);
  k_divb_sum<<<1, 256, 0, s>>>(partials, (int)(b.x * b.y), out);
}
void af_launch_points_slow(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) {
  if (g.special) pass(k_points_slow<true>, kShortBlocks, kListThreads, s, d, g, a, b);
  else pass(k_points_slow<false>, kShortBlocks, kListThreads, s, d, g, a, b);
}
void af_launch_lists(const AfDev &d, const AfGrid &g, double a, double b, cudaStream_t s) {
  if (af_small_grid(g)) af_lat_lists(d, g, a, b, s);
  else launch_lists(d, g, a, b, s);
}
float af_run_fp64_probe(cudaStream_t s, double *flops) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = sms * 8, threads = 256, iters = 8192;
  double *buf = nullptr;
  if (cudaMallocAsync(&buf, sizeof(double) * blocks * threads, s) != cudaSuccess) return -1.f;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  k_fp64_probe<<<blocks, threads, 0, s>>>(buf, 64);   // warm-up
  cudaEventRecord(e0, s);
  k_fp64_probe<<<blocks, threads, 0, s>>>(buf, iters);
  cudaEventRecord(e1, s);
  cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaFreeAsync(buf, s);
  cudaStreamSynchronize(s);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  *flops = 2.0 * 8.0 * (double)iters * blocks * threads / (ms * 1e-3);
  return ms;
}

void af_launch_inflow_pd(const AfGrid &g, const double *U, double *out, cudaStream_t s) {
  k_inflow_pd<<<1, 32, 0, s>>>(g, U, out);
}

void af_launch_math_check(int op, const double *x, const double *y, double *out, long long n, cudaStream_t s) {
  if (n <= 0) return;
  k_math_check<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(op, x, y, out, n);
}

void af_launch_batch(int pass, const AfRun *runs, int nruns, const int4 *items, int nitems, dim3 block, int nblocks,
                     double a, double b, int flag, cudaStream_t s) {
  const int reduce_dt = flag;
  switch (pass) {
    case AF_K_POINTDATA: kb_pointdata<<<nblocks, block, 0, s>>>(runs, items, nitems, reduce_dt); break;
    case AF_K_DT: kb_dt<<<(nruns + 127) / 128, 128, 0, s>>>(runs, nruns); break;
    case AF_K_POINTS:
      if (flag) kb_points<true><<<nblocks, block, 0, s>>>(runs, items, nitems, a, b);
      else kb_points<false><<<nblocks, block, 0, s>>>(runs, items, nitems, a, b);
      break;
    case AF_K_FACES: kb_faces<<<nblocks, block, 0, s>>>(runs, items, nitems); break;
    case AF_K_CELLS: kb_cells<<<nblocks, block, 0, s>>>(runs, items, nitems, a, b); break;
    case AF_K_FINAL: kb_final<<<nblocks, block, 0, s>>>(runs, items, nitems, a, b); break;
    case AF_K_CELLS_SLOW:
      kb_lists<<<152 * 2, kListThreads, 0, s>>>(runs, nruns, a, b);
      break;
    case AF_K_REPAIR: kb_repair<<<(nruns + 127) / 128, 128, 0, s>>>(runs, nruns, a, b); break;
    default: break;
  }
}

int af_batch_parts(int pass) { return pass == AF_K_POINTDATA ? 5 : (pass == AF_K_POINTS ? 4 : (pass == AF_K_FACES ? 2 : 1)); }

int af_batch_occupancy(int pass, dim3 block) {
  int n = 0;
  const int threads = block.x * block.y;
  switch (pass) {
    case AF_K_POINTDATA: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kb_pointdata, threads, 0); break;
    case AF_K_POINTS: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kb_points<false>, threads, 0); break;
    case AF_K_FACES: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kb_faces, threads, 0); break;
    case AF_K_CELLS: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kb_cells, threads, 0); break;
    case AF_K_FINAL: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kb_final, threads, 0); break;
    default: n = 1;
  }
  return n > 0 ? n : 1;
}

#include "af_kernels1d.cuh"
