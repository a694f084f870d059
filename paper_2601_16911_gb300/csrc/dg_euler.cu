// Fused stage kernel for the 2D compressible Euler equations (ideal gas), DG Q_p.
//
// Same tile structure as the scalar kernel: a TX x TY tile of cells plus a one-cell
// halo of all four conserved variables is staged in shared memory (mode-major), then
//   (a)+(b) vertex candidates of the density (Sec. 5.4: the sensor is computed from
//           the density and applied to all variables), one thread per tile vertex;
//   (c)     cell-vertex sensor gamma_e and nu_e = lambda_e h_e / (2p) with
//           lambda_e = max(|v| + c) over the cell's volume and face Gauss nodes;
//   (d)     SC weights: alpha~_q from the density's pointwise indicator, the
//           dissipation f_q of each conserved variable redistributed separately, so
//           each variable keeps its own cell dissipation rate (eq. alphaq);
//   (e)     HLL face fluxes with Davis wave-speed estimates, the volume flux and the
//           viscous term by sum factorisation, M^{-1}, and the SSP-RK3 combination.
//           As in the scalar kernel, every flux is evaluated as its deviation from the
//           flux of the cell's mean state (exact: a constant flux has zero residual),
//           so FP32 rounding is relative to the variation inside the cell.
// Non-positive density or pressure at any node raises the positivity bit of the
// status word (the computation continues; nothing traps).
#include "dg_scalar_kernel.cuh"

namespace cvw {
namespace {

constexpr int NV = 4;


// Mean state of a cell and the derived quantities the deviation fluxes need.
struct EulerMean {
  float U[NV];      // rho, m_x, m_y, E of the cell mean
  float vx, vy, H;  // mean velocity, E + p of the mean state
  float irho;       // 1 / rho of the mean
};

__device__ __forceinline__ EulerMean euler_mean(float g, const float* Ub) {
  EulerMean M;
#pragma unroll
  for (int v = 0; v < NV; ++v) M.U[v] = Ub[v];
  const float ir = 1.0f / Ub[0];
  M.irho = ir;
  M.vx = Ub[1] * ir;
  M.vy = Ub[2] * ir;
  const float p = (g - 1.0f) * (Ub[3] - 0.5f * (Ub[1] * M.vx + Ub[2] * M.vy));
  M.H = Ub[3] + p;
  return M;
}

// a*b - c*d with the rounding of c*d compensated (Kahan's FMA form): the result is
// accurate relative to itself even when the two products nearly cancel.
__device__ __forceinline__ f2 diff_of_products(f2 a, f2 b, float c, f2 d) {
  const f2 nw = mul2(dup2(-c), d);       // -w
  const f2 ne = fma2(dup2(c), d, nw);    // c*d - w, exactly
  return sub2(fma2(a, b, nw), ne);
}

// F(Ubar + d) - F(Ubar) in x and y at a pair of nodes, written as sums of (mean quantity) x
// (deviation) so that FP32 rounding is relative to |d|:
//   dv = (dm rhobar - mbar drho) / (rho rhobar),
//   dE - dK = (dE rhobar - dm . mbar / 2) / rhobar - (mbar + dm) . dv / 2,
//   dp = (g - 1)(dE - dK),  dH = dE + dp.
// The two differences that cancel exactly in uniform flow (dv for a uniform velocity,
// dE - dK for a uniform pressure) are formed with compensated products.
__device__ __forceinline__ void euler_dflux(float g, const EulerMean& M, const f2 (&d)[NV], f2 (&dFx)[NV], f2 (&dFy)[NV]) {
  const f2 rb = dup2(M.U[0]);
  const f2 rr = mul2(rb, add2(rb, d[0]));
  const f2 ir = mk2(rcp_fast(rr.x), rcp_fast(rr.y));
  const f2 dvx = mul2(diff_of_products(d[1], rb, M.U[1], d[0]), ir);
  const f2 dvy = mul2(diff_of_products(d[2], rb, M.U[2], d[0]), ir);
  // dE rhobar - (dmx mbarx + dmy mbary) / 2, compensated
  const f2 x1 = diff_of_products(d[3], rb, 0.5f * M.U[1], d[1]);
  const f2 np2 = mul2(dup2(-0.5f * M.U[2]), d[2]);
  const f2 x = sub2(add2(x1, np2), fma2(dup2(0.5f * M.U[2]), d[2], np2));
  const f2 m1 = add2(dup2(M.U[1]), d[1]), m2 = add2(dup2(M.U[2]), d[2]);
  const f2 k = fma2(m1, dvx, mul2(m2, dvy));
  const f2 dEmK = fma2(dup2(-0.5f), k, mul2(x, dup2(M.irho)));
  const f2 dp = mul2(dup2(g - 1.0f), dEmK);
  const f2 dH = add2(d[3], dp), H = add2(dup2(M.H), dH);
  const f2 vx = dup2(M.vx), vy = dup2(M.vy);
  dFx[0] = d[1];
  dFx[1] = add2(fma2(m1, dvx, mul2(d[1], vx)), dp);
  dFx[2] = fma2(m2, dvx, mul2(d[2], vx));
  dFx[3] = fma2(H, dvx, mul2(dH, vx));
  dFy[0] = d[2];
  dFy[1] = fma2(m1, dvy, mul2(d[1], vy));
  dFy[2] = add2(fma2(m2, dvy, mul2(d[2], vy)), dp);
  dFy[3] = fma2(H, dvy, mul2(dH, vy));
}

// |v| + c at a pair of nodes of full state U, with the velocity along x (dir 0) or y (dir 1)
// and the sound speed c; flags non-positive density or pressure
__device__ __forceinline__ float euler_wave(float g, const f2 (&U)[NV], int dir, f2& vn, f2& c, bool& bad) {
  const f2 ir = mk2(rcp_fast(U[0].x), rcp_fast(U[0].y));
  const f2 vx = mul2(U[1], ir), vy = mul2(U[2], ir);
  const f2 p = mul2(dup2(g - 1.0f), fma2(dup2(-0.5f), fma2(U[1], vx, mul2(U[2], vy)), U[3]));
  bad |= !(U[0].x > 0.0f) || !(U[0].y > 0.0f) || !(p.x > 0.0f) || !(p.y > 0.0f);
  c = mk2(sqrt_fast(g * fmaxf(p.x, 0.0f) * fabsf(ir.x)), sqrt_fast(g * fmaxf(p.y, 0.0f) * fabsf(ir.y)));
  vn = dir == 0 ? vx : vy;
  const f2 v2 = fma2(vx, vx, mul2(vy, vy));
  return fmaxf(sqrt_fast(v2.x) + c.x, sqrt_fast(v2.y) + c.y);
}

// HLL flux minus F(Ubar) . n across a face with normal +x (dir 0) or +y (dir 1) at a pair of
// nodes, from the left/lower state Ubar + dL to the right/upper state Ubar + dR (reading
// A14), with Davis wave speeds from the node states' normal velocities vnl, vnr and sound
// speeds cl, cr (euler_wave).  The constant F(Ubar) drops out of every branch:
// (S_R F(Ubar) - S_L F(Ubar)) / (S_R - S_L) = F(Ubar).
__device__ __forceinline__ void hll_dev(float g, const EulerMean& M, const f2 (&dL)[NV], const f2 (&dR)[NV], f2 vnl, f2 cl,
                                        f2 vnr, f2 cr, int dir, f2 (&F)[NV]) {
  const f2 sl = mk2(fminf(vnl.x - cl.x, vnr.x - cr.x), fminf(vnl.y - cl.y, vnr.y - cr.y));
  const f2 sr = mk2(fmaxf(vnl.x + cl.x, vnr.x + cr.x), fmaxf(vnl.y + cl.y, vnr.y + cr.y));
  f2 fl[NV], fr[NV], o[NV];
  if (dir == 0) {
    euler_dflux(g, M, dL, fl, o);
    euler_dflux(g, M, dR, fr, o);
  } else {
    euler_dflux(g, M, dL, o, fl);
    euler_dflux(g, M, dR, o, fr);
  }
  const f2 inv = mk2(rcp_fast(sr.x - sl.x), rcp_fast(sr.y - sl.y));
  const f2 wl = mul2(sr, inv), wr = mul2(mul2(dup2(-1.0f), sl), inv), wd = mul2(mul2(sl, sr), inv);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const f2 m = fma2(wl, fl[v], fma2(wr, fr[v], mul2(wd, sub2(dR[v], dL[v]))));
    F[v] = mk2(sl.x >= 0.0f ? fl[v].x : sr.x <= 0.0f ? fr[v].x : m.x, sl.y >= 0.0f ? fl[v].y : sr.y <= 0.0f ? fr[v].y : m.y);
  }
}

// Calls f(ua, ub, mid) for every pair of node rows of a cell with modes c: the volume nodes (x group
// q, rows +eta_h (a) and -eta_h (b)) and the face nodes: the ends +-1 are one more x group and
// one more row pair, whose Legendre values are all 1 (their corner combination is left out).
// mid: the row pair is the one middle row.
template <int N, int MP, class F>
__device__ __forceinline__ void for_node_groups(const float* img, const f2 (&c)[NV][N][MP], F&& f) {
  using Img = PackedImage<2, N - 1>;
  constexpr int NG = Img::NG;
#pragma unroll 1
  for (int q = 0; q <= NG; ++q) {
    f2 b[MP], tb[NV][N];
    load_pairs<MP>(img + Img::BX + 2 * MP * (q < NG ? q : 0), b);
    if (q == NG) {
#pragma unroll
      for (int p = 0; p < MP; ++p) b[p] = mk2(1.0f, 1.0f);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int my = 0; my < N; ++my) {
        f2 s = mul2(b[0], c[v][my][0]);
#pragma unroll
        for (int p = 1; p < MP; ++p) s = fma2(b[p], c[v][my][p], s);
        tb[v][my] = mk2(s.x + s.y, s.x - s.y);
      }
#pragma unroll 1
    for (int h = 0; h < (q < NG ? NG + 1 : NG); ++h) {
      f2 by[N], ua[NV], ub[NV];
      load_pairs<N>(img + Img::BY + 2 * N * (h < NG ? h : 0), by);
      if (h == NG) {
#pragma unroll
        for (int my = 0; my < N; ++my) by[my] = mk2(1.0f, 1.0f);
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        f2 e = mul2(by[0], tb[v][0]), o = mul2(by[1], tb[v][1]);
#pragma unroll
        for (int my = 2; my < N; ++my) {
          if (my & 1) o = fma2(by[my], tb[v][my], o);
          else e = fma2(by[my], tb[v][my], e);
        }
        ua[v] = add2(e, o);
        ub[v] = sub2(e, o);
      }
      f(ua, ub, (N & 1) && h == NG - 1);
    }
  }
}

// Positivity limiter of one cell (readings P1-P4; Zhang and Shu's scaling limiter): the density's
// non-mean modes are scaled by th1 to keep rho >= eps_e at the volume and face Gauss nodes, then
// all non-mean modes by th2 to keep p >= eps_e, the root of p(U_bar + t dU) = eps_e found by 40
// bisection steps at the nodes that violate it.  False (and c unchanged) where the mean is not
// admissible.
template <int N, int MP>
__device__ __forceinline__ bool limit_positivity(float g, const float* img, f2 (&c)[NV][N][MP], float& th1, float& th2) {
  float Ub[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) Ub[v] = c[v][0][0].x;
  auto pres = [&](const float (&U)[NV]) { return (g - 1.0f) * (U[3] - 0.5f * (U[1] * U[1] + U[2] * U[2]) / U[0]); };
  const float pb = pres(Ub);
  th1 = th2 = 1.0f;
  if (!(Ub[0] > 0.0f && pb > 0.0f)) return false;
  const float eps = 1e-3f * fminf(Ub[0], pb);
  // the smallest density, and whether any node's pressure (with th1 = 1) is below eps
  float rmin = Ub[0];
  bool low = false;
  for_node_groups<N, MP>(img, c, [&](const f2 (&ua)[NV], const f2 (&ub)[NV], bool mid) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= 2 && mid) continue;
      const f2 (&u)[NV] = k < 2 ? ua : ub;
      const float U[NV] = {k & 1 ? u[0].y : u[0].x, k & 1 ? u[1].y : u[1].x, k & 1 ? u[2].y : u[2].x, k & 1 ? u[3].y : u[3].x};
      rmin = fminf(rmin, U[0]);
      low |= !(pres(U) >= eps);
    }
  });
  if (rmin < eps) th1 = fminf(1.0f, (Ub[0] - eps) / (Ub[0] - rmin));
  // (the pressures are taken again where the density changed or a node was low)
  if (low || th1 < 1.0f)
    for_node_groups<N, MP>(img, c, [&](const f2 (&ua)[NV], const f2 (&ub)[NV], bool mid) {
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        if (k >= 2 && mid) continue;
        float U[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) U[v] = k == 0 ? ua[v].x : k == 1 ? ua[v].y : k == 2 ? ub[v].x : ub[v].y;
        U[0] = fmaf(th1, U[0] - Ub[0], Ub[0]);
        if (!(pres(U) < eps)) continue;
        float lo = 0.0f, hi = 1.0f;  // p(lo) >= eps > p(hi)
#pragma unroll 1
        for (int it = 0; it < 40; ++it) {
          const float t = 0.5f * (lo + hi);
          float Ut[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) Ut[v] = fmaf(t, U[v] - Ub[v], Ub[v]);
          if (pres(Ut) >= eps) lo = t; else hi = t;
        }
        th2 = fminf(th2, lo);
      }
    });
  if (th1 < 1.0f || th2 < 1.0f) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const f2 f = dup2((v == 0 ? th1 : 1.0f) * th2);
#pragma unroll
      for (int my = 0; my < N; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) c[v][my][p] = mul2(c[v][my][p], f);
      c[v][0][0].x = Ub[v];
    }
  }
  return true;
}

// Shared-memory layout of the Euler stage tile (floats): four variables' cells, each laid
// out as the scalar tile's (TileLayout), then the density's vertex data (later the
// indicator), the node tabulations, the faces' projected fluxes (mode pairs,
// component-major, so that neighbouring faces lie in neighbouring banks) and the largest
// wave speed of each side of a face (later the SC factors of the four variables).
template <int P, int TX, int TY>
struct EulerLayout {
  using L = TileLayout<2, P, TX, TY>;
  static constexpr int NT = L::NT, ND = L::ND, MP = L::MP, NFACE = L::NFACE;
  static constexpr int VAR = (L::HY * L::RS + 3) / 4 * 4;        // floats of a variable's cells
  static constexpr int OFF_C = 0;                                // [NV][VAR]
  static constexpr int OFF_ST = OFF_C + NV * VAR;                // vertex data, then [ND][NT] indicator
  static constexpr int OFF_IMG = (OFF_ST + imax(L::VS * L::NVT, ND * NT) + 3) / 4 * 4;
  static constexpr int OFF_F = OFF_IMG + L::Img::FLOATS;         // [NV][MP][NFACE] pairs
  static constexpr int OFF_LAM = OFF_F + 2 * NV * MP * NFACE;    // [2][NFACE], then [NV][NT]
  static constexpr int FLOATS = OFF_LAM + imax(2 * NFACE, NV * NT);
  static constexpr size_t BYTES = sizeof(float) * (size_t)FLOATS;
};

// Minimum resident CTAs the register allocation must allow, from sweeps (us per step).
// p = 1, 512^2: 4 CTAs of 160 threads 108.7, 3 CTAs 114, 6 CTAs 114.  p = 2, 512^2: 3 CTAs 321,
// 2 CTAs 352 (but 5 % faster on meshes of one wave), 4 CTAs 360.  p = 3, 512^2: 2 CTAs at
// 255 registers 415, 3 CTAs at 168 496.  p = 4 (8x8 tiles), 300^2: 2 CTAs 494.  All forms from p = 2 on
// spill; the ones in use, stores / loads: p = 2 (168 registers) 0.45 / 0.85 KB, p = 3 0.2 / 0.5 KB, p = 4
// 1.3 / 2.3 KB, so at p = 3 what 3 CTAs lose is more spilling, not the first.
template <int P, int TX, int TY>
constexpr int euler_min_ctas() {
  return P == 1 ? 4 : P == 2 ? 3 : 2;
}
// Threads of a block: at p = 1 one warp more than the cells, at p = 4 two, to share the
// vertices and faces; at p = 2 and 3 the extra warp would cost more registers than it saves.
template <int P, int TX, int TY>
__host__ __device__ constexpr int euler_threads() {
  return TX * TY + (P == 1 ? 32 : P == 4 ? 64 : 0);
}

// One CTA per tile.  Density vertices and faces share the threads, as in the scalar kernel;
// then one thread per cell, on two-wide FMAs over mode and node pairs (dg_packed.cuh), which
// took the Q3 stage of 512^2 from 137 M to 63 M warp instructions and the step from 681 to
// 415 us (Q1 at 256^2 59 -> 39 us, Q2 131 -> 106, Q4 at 128^2 257 -> 127).  Bound by
// instruction issue (43 %) and latency at 8 warps per SM (255 registers: four variables'
// residuals and node sums are live together):
//   faces: the four projected fluxes into r (a left/lower face was projected relative to
//     the neighbour's mean, so the cell adds F(Ubar_nb) - F(Ubar) on the face's mean mode);
//   volume pass A (by node groups): flux deviation projected into r, lambda_e over the nodes;
//   volume pass B, only where the viscosity (1 - gamma_e) nu_e is non-zero: the viscous term.
// The SC weights of troubled cells (stage d) are taken before that by all threads of the
// tile, (cell, node group) and (cell, variable) at a time.
// POS: the positivity limiter on the stage's result, in registers, before it is written.
template <int P, int TX, int TY, bool POS>
__global__ void __launch_bounds__(euler_threads<P, TX, TY>(), (euler_min_ctas<P, TX, TY>()))
    dg_euler_stage(const __grid_constant__ StageArgs a, const __grid_constant__ PackedTables<2, P> T) {
  using E = EulerLayout<P, TX, TY>;
  using L = typename E::L;
  using Img = PackedImage<2, P>;
  constexpr int N = L::N, ND = L::ND, MP = L::MP, NG = L::NG, NT = L::NT, NB = euler_threads<P, TX, TY>();
  constexpr int HX = L::HX, HY = L::HY, NH = L::NH, NFACE = L::NFACE;
  extern __shared__ __align__(16) float smem[];
  float* sc = smem + E::OFF_C;
  float* st = smem + E::OFF_ST;
  float* sNq = smem + E::OFF_ST;
  const float* img = smem + E::OFF_IMG;
  f2* sF = reinterpret_cast<f2*>(smem + E::OFF_F);
  float* sLam = smem + E::OFF_LAM;
  float* sAf = smem + E::OFF_LAM;
  __shared__ int phs[NV][HY];
  __shared__ int sc_count;
  __shared__ short sc_cell[NT];
  if (threadIdx.x == 0) sc_count = 0;
  const int nx = a.nx, ny = a.ny;
  const size_t ncell = (size_t)nx * ny;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const float g = a.gas_gamma;

  // ---- load tile + halo of all variables: asynchronous copies in place ---------------------
  for (int f = threadIdx.x; f < Img::FLOATS / 4; f += NB) cp_async16(smem + E::OFF_IMG + 4 * f, a.pk_img + 4 * f);
  pdl_wait();  // everything below reads or writes what earlier kernels write
  const bool aligned = (reinterpret_cast<uintptr_t>(a.u_in) & 15) == 0;
  // Otherwise the rows of a tile that touches no x boundary are copied by 16-byte chunks, and
  // the rest (and a state that is not 16-byte aligned) float by float.
  if (!L::CHUNKED && aligned && i0 > 0 && i0 + TX < nx) {
    if constexpr (!L::CHUNKED) {
      stage_rows16_inner<ND, HX, HY, L::RS, NB, NV>(sc, E::VAR, phs[0], a.u_in, (int64_t)ncell * ND, nx, ny, i0 - 1, j0 - 1,
                                                    a.pery, a.status, CVW_EXTENT(a, lim_in));
    }
  } else {
    // whole 16-byte chunks, or floats where the state is not 16-byte aligned
    constexpr int NQ4 = ND / 4 > 0 ? ND / 4 : 1;
    const int per = L::CHUNKED && aligned ? NQ4 : ND;
    for (int f = threadIdx.x; f < NH * per; f += NB) {
      const int h = f / per, q = f - h * per, r = h / HX, cc = h - r * HX;
      int gi = i0 - 1 + cc, gj = j0 - 1 + r;
      bool in = true;
      if (gi < 0 || gi >= nx) {
        if (a.perx) gi = (gi + nx) % nx; else in = false;
      }
      if (gj < 0 || gj >= ny) {
        if (a.pery) gj = (gj + ny) % ny; else in = false;
      }
      const size_t src = ((size_t)gj * nx + gi) * ND;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const size_t s = (size_t)v * ncell * ND + src;
        if (L::CHUNKED && aligned) {
          const bool ok = in && CVW_SPAN(a.status, s + 4 * q, 4, a.lim_in);
          cp_async16z(sc + v * E::VAR + (L::cell(phs[v], cc, r) ^ (4 * q)), ok ? a.u_in + s + 4 * q : a.u_in, ok ? 16 : 0);
        } else {
          const bool ok = in && CVW_SPAN(a.status, s + q, 1, a.lim_in);
          const int dst = L::CHUNKED ? (L::cell(phs[v], cc, r) ^ (q & ~3)) + (q & 3) : r * L::RS + cc * ND + q;
          cp_async4(sc + v * E::VAR + dst, ok ? a.u_in + s + q : a.u_in, ok ? 4 : 0);
        }
      }
    }
    for (int r = threadIdx.x; r < NV * HY; r += NB) (&phs[0][0])[r] = 0;
  }
  cp_async_wait_all();
  __syncthreads();

  // ---- (a)+(b): density vertex candidates ---------------------------------------------------
  tile_vertex_phase<2, P, TX, TY, NB>(a, T, sc, phs[0], st, i0, j0, nx, ny);

  const bool sensor_only = (a.mode & kModeSensorOnly) != 0;
  const bool rk = (a.mode & kModeRK) != 0, with_un = rk && a.rk_a != 0.0f;
  const int act_x = min(TX, nx - i0), act_y = min(TY, ny - j0);
  bool bad = false;

  // ---- the tile's faces, each once: traces, HLL, projection, each side's wave speed --------------
  // In the vertex phase's barrier interval, from the block's last thread backwards: the
  // vertex phase's extra round falls on the first threads, the face phase's on the last.
#pragma unroll 1
  for (int f = NB - 1 - threadIdx.x; f < NFACE; f += NB) {
    int dirn, hx, hy;
    bool hasl, hasr, needed;
    if (f < L::NFX) {
      hy = f / (TX + 1), hx = f - hy * (TX + 1);
      needed = hy < act_y && hx <= act_x;  // a side of an active cell
      const int gl = i0 - 1 + hx;
      hasl = a.perx || gl >= 0;
      hasr = a.perx || gl + 1 < nx;
      ++hy;
      dirn = 0;
    } else {
      const int q = f - L::NFX;
      hy = q / TX, hx = q - hy * TX;
      needed = hx < act_x && hy <= act_y;
      ++hx;
      const int gl = j0 - 1 + hy;
      hasl = a.pery || gl >= 0;
      hasr = a.pery || gl + 1 < ny;
      dirn = 1;
    }
    if (!needed) continue;
    // tangential traces (non-mean modes) as mode pairs: the left/lower cell meets the face
    // with its upper side (+1), the right/upper cell with its lower side ((-1)^i along the
    // normal); a missing side (transmissive boundary) is the other side's ghost
    f2 tr[2][NV][MP];
    float um[2][NV];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const float sg = side ? -1.0f : 1.0f;
      const int cx = hx + (dirn == 0 ? side : 0), cy = hy + (dirn == 1 ? side : 0);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        f2 c[N][MP];
        load_cell<L>(sc + v * E::VAR, L::cell(phs[v], cx, cy), c);
        um[side][v] = c[0][0].x;
        c[0][0].x = 0.0f;
        if (dirn == 0) {
          float d[2 * MP];
          d[2 * MP - 1] = 0.0f;
#pragma unroll
          for (int my = 0; my < N; ++my) {
            f2 s = c[my][0];
#pragma unroll
            for (int p = 1; p < MP; ++p) s = add2(s, c[my][p]);
            d[my] = fmaf(sg, s.y, s.x);
          }
#pragma unroll
          for (int p = 0; p < MP; ++p) tr[side][v][p] = mk2(d[2 * p], d[2 * p + 1]);
        } else {
#pragma unroll
          for (int p = 0; p < MP; ++p) {
            f2 e = c[0][p], o = c[1][p];
#pragma unroll
            for (int my = 2; my < N; ++my) {
              if (my & 1) o = add2(o, c[my][p]);
              else e = add2(e, c[my][p]);
            }
            tr[side][v][p] = fma2(dup2(sg), o, e);
          }
        }
      }
    }
    if (!hasl || !hasr) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        um[0][v] = hasl ? um[0][v] : um[1][v];
        um[1][v] = hasr ? um[1][v] : um[0][v];
#pragma unroll
        for (int p = 0; p < MP; ++p) {
          tr[0][v][p] = hasl ? tr[0][v][p] : tr[1][v][p];
          tr[1][v][p] = hasr ? tr[1][v][p] : tr[0][v][p];
        }
      }
    }
    const EulerMean ML = euler_mean(g, um[0]);
    f2 h[NV][MP];
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int p = 0; p < MP; ++p) h[v][p] = mk2(0.0f, 0.0f);
    float laml = 0.0f, lamr = 0.0f;
#pragma unroll 1
    for (int q = 0; q < NG; ++q) {
      f2 b[MP], dL[NV], dR[NV], U[NV];
      load_pairs<MP>(img + Img::BX + 2 * MP * q, b);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        f2 sl = mul2(b[0], tr[0][v][0]), sr = mul2(b[0], tr[1][v][0]);
#pragma unroll
        for (int p = 1; p < MP; ++p) {
          sl = fma2(b[p], tr[0][v][p], sl);
          sr = fma2(b[p], tr[1][v][p], sr);
        }
        dL[v] = mk2(sl.x + sl.y, sl.x - sl.y);
        dR[v] = mk2(sr.x + sr.y, sr.x - sr.y);
      }
      f2 vnl, cl, vnr, cr;
#pragma unroll
      for (int v = 0; v < NV; ++v) U[v] = add2(dup2(um[0][v]), dL[v]);
      laml = fmaxf(laml, euler_wave(g, U, dirn, vnl, cl, bad));
#pragma unroll
      for (int v = 0; v < NV; ++v) U[v] = add2(dup2(um[1][v]), dR[v]);
      lamr = fmaxf(lamr, euler_wave(g, U, dirn, vnr, cr, bad));
      if (sensor_only) continue;
#pragma unroll
      for (int v = 0; v < NV; ++v) dR[v] = add2(dup2(um[1][v] - um[0][v]), dR[v]);
      f2 F[NV];
      hll_dev(g, ML, dL, dR, vnl, cl, vnr, cr, dirn, F);
      const float w = img[Img::WX + q];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const f2 sd = mul2(dup2(w), mk2(F[v].x + F[v].y, F[v].x - F[v].y));
#pragma unroll
        for (int p = 0; p < MP; ++p) h[v][p] = fma2(b[p], sd, h[v][p]);
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v)
#pragma unroll
      for (int p = 0; p < MP; ++p) sF[(v * MP + p) * NFACE + f] = h[v][p];
    sLam[f] = laml;
    sLam[NFACE + f] = lamr;
  }
  __syncthreads();
  pdl_launch_dependents();

  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int gi = i0 + tx, gj = j0 + ty;
  const size_t cell = (size_t)gj * nx + gi;
  // (the checked build also checks the cell's index in the per-cell outputs and its span of
  // u_n and u_out in the last variable)
  const bool active = (NB == NT || threadIdx.x < NT) && gi < nx && gj < ny && CVW_SPAN(a.status, cell, 1, a.lim_cell) &&
                      CVW_SPAN(a.status, ((size_t)(NV - 1) * ncell + cell) * ND, ND,
                               a.lim_in < a.lim_out ? a.lim_in : a.lim_out);
  // ---- (c) sensor from the density; lambda_e over the face nodes -------------------------------
  float gam = 1.0f, n0 = 0.0f, lam = 0.0f;
  if (active) {
    f2 c[N][MP], S[N][MP];
    load_cell<L>(sc, L::cell(phs[0], tx + 1, ty + 1), c);
    gam = cell_sensor<2, P, TX, TY>(a, T, st, c, tx, ty, n0, S);
#pragma unroll
    for (int k = 0; k < 4; ++k) lam = fmaxf(lam, sLam[((k & 1) ? NFACE : 0) + cell_face<L, TX>(k, tx, ty)]);
  }

  // ---- (d) troubled cells: the density's pointwise indicator Nq at the volume nodes, then each
  // variable's factor afac = sum w g / sum w Nq g, g = |grad u_v|^2 (alpha_{v,q} = Nq[q] afac[v];
  // alpha = 1 where afac < 0).  The tile's threads share the troubled cells' work.
  bool troubled = false, need_sc = false;
  float afac[NV];
  // mean deviations of the left (first half) and lower neighbour, zero where there is none
  // (after this stage a cell's slot is its thread's own)
  f2 dn[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const float m = active ? sc[v * E::VAR + L::cell(phs[v], tx + 1, ty + 1)] : 0.0f;
    dn[v] = mk2(active && (a.perx || gi > 0) ? sc[v * E::VAR + L::cell(phs[v], tx, ty + 1)] - m : 0.0f,
                active && (a.pery || gj > 0) ? sc[v * E::VAR + L::cell(phs[v], tx + 1, ty)] - m : 0.0f);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) afac[v] = -1.0f;
  if (!sensor_only) {
    if (active) {
      troubled = a.sc && gam < a.c_gamma && n0 > 1e-30f;
      if (a.troubled_override) {
        const int ov = a.troubled_override[cell];
        if (ov >= 0) troubled = ov && n0 > 1e-30f;
      }
    }
    need_sc = troubled && gam < 1.0f;
    if (need_sc) sc_cell[atomicAdd(&sc_count, 1)] = (short)threadIdx.x;
    if (__syncthreads_or(need_sc)) {
      const int n = sc_count;
#pragma unroll 1
      for (int t = threadIdx.x; t < n * L::NGG; t += NB) {
        const int gh = t / n, id = sc_cell[t - gh * n];
        f2 s1, s2;
        sc_node_group<2, P, TX, TY>(a, T, img, sNq, sc, phs[0], id, gh / NG, gh % NG, s1, s2);
      }
      __syncthreads();
#pragma unroll 1
      for (int t = threadIdx.x; t < n * NV; t += NB) {
        const int v = t / n, id = sc_cell[t - v * n];
        f2 c[N][MP], s1 = mk2(0.0f, 0.0f), s2 = s1;
        load_cell<L>(sc + v * E::VAR, L::cell(phs[v], id % TX + 1, id / TX + 1), c);
        c[0][0].x = 0.0f;
#pragma unroll 1
        for (int q = 0; q < NG; ++q) {
          f2 b[MP], d[MP], tb[N], td[N];
          load_pairs<MP>(img + Img::BX + 2 * MP * q, b);
          load_pairs<MP>(img + Img::DX + 2 * MP * q, d);
#pragma unroll
          for (int my = 0; my < N; ++my) {
            f2 s = mul2(b[0], c[my][0]), sd = mul2(d[0], c[my][0]);
#pragma unroll
            for (int p = 1; p < MP; ++p) {
              s = fma2(b[p], c[my][p], s);
              sd = fma2(d[p], c[my][p], sd);
            }
            tb[my] = mk2(s.x + s.y, s.x - s.y);
            td[my] = mk2(sd.x + sd.y, sd.y - sd.x);
          }
#pragma unroll 1
          for (int h = 0; h < NG; ++h) {
            f2 ua, ub, va, vb;
            node_gradient<N, MP>(img + Img::BY + 2 * N * h, img + Img::DY + 2 * N * h, tb, td, ua, ub, va, vb);
            const f2 kx = dup2(a.two_dx * a.two_dx), ky = dup2(a.two_dy * a.two_dy);
            const f2 qa = fma2(kx, mul2(ua, ua), mul2(ky, mul2(va, va)));
            const f2 qb = fma2(kx, mul2(ub, ub), mul2(ky, mul2(vb, vb)));
            const f2 w = dup2(img[Img::WX + q] * img[Img::WY + h]);
            const float* ra = sNq + N * h * NT + id;
            s1 = fma2(w, qa, s1);
            s2 = fma2(mul2(w, mk2(ra[q * NT], ra[(N - 1 - q) * NT])), qa, s2);
            if (2 * h != N - 1) {
              const float* rb = sNq + N * (N - 1 - h) * NT + id;
              s1 = fma2(w, qb, s1);
              s2 = fma2(mul2(w, mk2(rb[q * NT], rb[(N - 1 - q) * NT])), qb, s2);
            }
          }
        }
        const float t2 = s2.x + s2.y;
        sAf[v * NT + id] = t2 > 0.0f ? (s1.x + s1.y) / t2 : -1.0f;
      }
      __syncthreads();
      if (need_sc) {
#pragma unroll
        for (int v = 0; v < NV; ++v) afac[v] = sAf[v * NT + threadIdx.x];
      }
    }
  }
  if (active) {

  // ---- faces into the residual: right, left, top, bottom ---------------------------------------
  int hc[NV];
  float Ubar[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    hc[v] = v * E::VAR + L::cell(phs[v], tx + 1, ty + 1);
    Ubar[v] = sc[hc[v]];
  }
  const EulerMean M = euler_mean(g, Ubar);
  f2 r[NV][N][MP];
  if (!sensor_only) {
    // the lower faces' F(Ubar_nb) - F(Ubar), twice (its projection on the face's mean mode)
    f2 nx2[NV], ny2[NV];
    euler_dflux(g, M, dn, nx2, ny2);
    const int fR = cell_face<L, TX>(0, tx, ty), fL = cell_face<L, TX>(1, tx, ty), fT = cell_face<L, TX>(2, tx, ty),
              fB = cell_face<L, TX>(3, tx, ty);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      // r[mx,my] = -2/dx (hR[my] - (-1)^mx hL[my]) - 2/dy (hT[mx] - (-1)^my hB[mx])
      f2 ve[MP], vo[MP], hr[MP], hl[MP];
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const f2* row = sF + (v * MP + p) * NFACE;
        f2 top = row[fT], bot = row[fB];
        hr[p] = row[fR];
        hl[p] = row[fL];
        if (p == 0) {
          hl[0].x = fmaf(2.0f, nx2[v].x, hl[0].x);
          bot.x = fmaf(2.0f, ny2[v].y, bot.x);
        }
        ve[p] = mul2(dup2(a.two_dy), sub2(bot, top));
        vo[p] = mul2(dup2(-a.two_dy), add2(bot, top));
      }
#pragma unroll
      for (int my = 0; my < N; ++my) {
        const float R = (my & 1) ? hr[my / 2].y : hr[my / 2].x, Lf = (my & 1) ? hl[my / 2].y : hl[my / 2].x;
        const f2 x = mk2(-a.two_dx * (R - Lf), -a.two_dx * (R + Lf));
#pragma unroll
        for (int p = 0; p < MP; ++p) r[v][my][p] = add2(x, (my & 1) ? vo[p] : ve[p]);
      }
    }
  }

  // ---- volume pass A: flux deviation into r, lambda_e over the nodes -------------------------------
#pragma unroll 1
  for (int q = 0; q < NG; ++q) {
    f2 b[MP], tb[NV][N], hx[NV][N], hy[NV][N];
    load_pairs<MP>(img + Img::BX + 2 * MP * q, b);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      f2 c[N][MP];
      load_cell<L>(sc, hc[v], c);
      c[0][0].x = 0.0f;  // deviation: no mean mode
#pragma unroll
      for (int my = 0; my < N; ++my) {
        f2 s = mul2(b[0], c[my][0]);
#pragma unroll
        for (int p = 1; p < MP; ++p) s = fma2(b[p], c[my][p], s);
        tb[v][my] = mk2(s.x + s.y, s.x - s.y);
        hx[v][my] = hy[v][my] = mk2(0.0f, 0.0f);
      }
    }
#pragma unroll 1
    for (int h = 0; h < NG; ++h) {
      const float* yb = img + Img::BY + 2 * N * h;
      const bool mid = (N & 1) && h == NG - 1;  // the middle row: one row only
      f2 ua[NV], ub[NV], fx[NV], fy[NV], gx[NV], gy[NV];
      {
        f2 by[N];
        load_pairs<N>(yb, by);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          f2 e = mul2(by[0], tb[v][0]), o = mul2(by[1], tb[v][1]);
#pragma unroll
          for (int my = 2; my < N; ++my) {
            if (my & 1) o = fma2(by[my], tb[v][my], o);
            else e = fma2(by[my], tb[v][my], e);
          }
          ua[v] = add2(e, o);
          ub[v] = sub2(e, o);
        }
      }
      {
        f2 U[NV], vn, cs;
#pragma unroll
        for (int v = 0; v < NV; ++v) U[v] = add2(dup2(Ubar[v]), ua[v]);
        lam = fmaxf(lam, euler_wave(g, U, 0, vn, cs, bad));
        if (!mid) {
#pragma unroll
          for (int v = 0; v < NV; ++v) U[v] = add2(dup2(Ubar[v]), ub[v]);
          lam = fmaxf(lam, euler_wave(g, U, 0, vn, cs, bad));
        }
      }
      if (sensor_only) continue;
      euler_dflux(g, M, ua, fx, fy);
#pragma unroll
      for (int v = 0; v < NV; ++v) gx[v] = gy[v] = mk2(0.0f, 0.0f);
      if (!mid) euler_dflux(g, M, ub, gx, gy);
      f2 by[N], dy[N];
      load_pairs<N>(yb, by);
      load_pairs<N>(img + Img::DY + 2 * N * h, dy);
      const f2 w = dup2(img[Img::WY + h]);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const f2 xs = mul2(w, add2(fx[v], gx[v])), xd = mul2(w, sub2(fx[v], gx[v]));
        const f2 ys = mul2(w, add2(fy[v], gy[v])), yd = mul2(w, sub2(fy[v], gy[v]));
#pragma unroll
        for (int my = 0; my < N; ++my) {
          hx[v][my] = fma2(by[my], (my & 1) ? xd : xs, hx[v][my]);
          if (my > 0) hy[v][my] = fma2(dy[my], (my & 1) ? ys : yd, hy[v][my]);
        }
      }
    }
    if (sensor_only) continue;
    f2 d[MP];
    load_pairs<MP>(img + Img::BX + 2 * MP * q, b);
    load_pairs<MP>(img + Img::DX + 2 * MP * q, d);
    const float kx = a.two_dx * img[Img::WX + q], ky = a.two_dy * img[Img::WX + q];
#pragma unroll
    for (int v = 0; v < NV; ++v) project_nodes<N, MP>(b, d, kx, ky, hx[v], hy[v], r[v]);
  }
  const float nu = lam * a.nu_scale;
  if (a.gamma_out) a.gamma_out[cell] = gam;
  if (a.nu_out) a.nu_out[cell] = nu;
  if (a.lambda_out) a.lambda_out[cell] = lam;
  if (sensor_only) {
    if (bad) atomicOr(a.status, kStatPositivity);
    return;
  }
  if (a.troubled_out) a.troubled_out[cell] = troubled ? 1 : 0;
  if (a.alpha_out) {
#pragma unroll 1
    for (int q = 0; q < ND; ++q) {
      const float nq = need_sc ? sNq[q * NT + threadIdx.x] : 0.0f;
#pragma unroll
      for (int v = 0; v < NV; ++v) a.alpha_out[(cell * NV + v) * ND + q] = afac[v] >= 0.0f ? nq * afac[v] : 1.0f;
    }
  }

  // ---- volume pass B: the viscous term, where (1 - gamma_e) nu_e > 0 -----------------------------
  // Where every variable has the linear weights, the stiffness form of the Legendre basis
  // (add_stiffness); alpha-weighted cells take the quadrature.
  const float mu = (1.0f - gam) * nu;
  bool weighted = false;
#pragma unroll
  for (int v = 0; v < NV; ++v) weighted |= afac[v] >= 0.0f;
  if (mu > 0.0f && !weighted) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      f2 c[N][MP];
      load_cell<L>(sc, hc[v], c);
      c[0][0].x = 0.0f;
      add_stiffness<2, N, N, MP>(-mu * a.two_dx * a.two_dx, -mu * a.two_dy * a.two_dy, c, r[v]);
    }
  } else if (mu > 0.0f) {
#pragma unroll 1
    for (int v = 0; v < NV; ++v) {
      f2 c[N][MP], rv[N][MP];
      const float af = v == 0 ? afac[0] : v == 1 ? afac[1] : v == 2 ? afac[2] : afac[3];
      load_cell<L>(sc + v * E::VAR, L::cell(phs[v], tx + 1, ty + 1), c);
      c[0][0].x = 0.0f;
#pragma unroll
      for (int my = 0; my < N; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) rv[my][p] = mk2(0.0f, 0.0f);
#pragma unroll 1
      for (int q = 0; q < NG; ++q)
        weighted_viscous<N, MP, NT>(a, img, sNq + threadIdx.x, q, -mu * (af >= 0.0f ? af : 1.0f), af >= 0.0f, c, rv);
#pragma unroll
      for (int w = 0; w < NV; ++w)
        if (w == v) {
#pragma unroll
          for (int my = 0; my < N; ++my)
#pragma unroll
            for (int p = 0; p < MP; ++p) r[w][my][p] = add2(r[w][my][p], rv[my][p]);
        }
    }
  }

  // ---- M^{-1} and the RK combination; cells of whole 16-byte chunks are written here ----------------
  // Per variable, the cell's u_n is read in full before any of its outputs is written: only
  // this thread reads or writes the cell's span, so u_n may alias u_out, and the reads of a
  // variable go out together.  16-byte loads and stores where both states are 16-byte aligned.
  f2 fin = mk2(0.0f, 0.0f);  // stays zero while every du/dt is finite
  const bool v16 = ND % 4 == 0 && ((reinterpret_cast<uintptr_t>(a.u_out) | reinterpret_cast<uintptr_t>(a.u_n)) & 15) == 0;
  auto write_var = [&](int v) {
    auto val = [&](int m) { return (m % N) & 1 ? r[v][m / N][m % N / 2].y : r[v][m / N][m % N / 2].x; };
    float* out = a.u_out + ((size_t)v * ncell + cell) * ND;
    if (v16) {
#pragma unroll
      for (int q = 0; q < ND / 4; ++q)
        reinterpret_cast<float4*>(out)[q] = make_float4(val(4 * q), val(4 * q + 1), val(4 * q + 2), val(4 * q + 3));
    } else {
#pragma unroll
      for (int m = 0; m < ND; ++m) out[m] = val(m);
    }
  };
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    f2 c[N][MP], n[N][MP];
    load_cell<L>(sc, hc[v], c);
    if (with_un) {
      const float* un = a.u_n + ((size_t)v * ncell + cell) * ND;
      if (v16) {
#pragma unroll
        for (int q = 0; q < ND / 4; ++q) {
          const float4 x = reinterpret_cast<const float4*>(un)[q];
          const int m = 4 * q, m2 = m + 2;
          n[m / N][m % N / 2] = mk2(x.x, x.y);
          n[m2 / N][m2 % N / 2] = mk2(x.z, x.w);
        }
      } else {
#pragma unroll
        for (int my = 0; my < N; ++my)
#pragma unroll
          for (int p = 0; p < MP; ++p) n[my][p] = mk2(un[2 * p + N * my], 2 * p + 1 < N ? un[2 * p + 1 + N * my] : 0.0f);
      }
    }
#pragma unroll
    for (int my = 0; my < N; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const float ys = 0.25f * (2 * my + 1);
        f2 d = mul2(r[v][my][p], mk2(ys * (4 * p + 1), ys * (4 * p + 3)));
        if (2 * p + 1 >= N) d.y = 0.0f;
        fin = fma2(d, dup2(0.0f), fin);
        if (rk) {
          d = fma2(dup2(a.dt), d, c[my][p]);
          if (with_un) d = fma2(dup2(a.rk_b), sub2(d, n[my][p]), n[my][p]);
        }
        r[v][my][p] = d;
      }
    if constexpr (!POS) write_var(v);
  }
  if constexpr (POS) {
    float th1, th2;
    bad |= !limit_positivity<N, MP>(g, img, r, th1, th2);
#pragma unroll
    for (int v = 0; v < NV; ++v) write_var(v);
  }
  if (!(fin.x + fin.y == 0.0f)) atomicOr(a.status, kStatNonfinite);
  }  // active
  if (bad) atomicOr(a.status, kStatPositivity);
}

template <int P, int TX, int TY, bool POS>
cudaError_t launch_euler(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  using Tb = DgTables<2, P>;
  constexpr size_t smem = EulerLayout<P, TX, TY>::BYTES;
  static_assert(smem <= 220 * 1024, "tile too large for shared memory");
  auto kern = dg_euler_stage<P, TX, TY, POS>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (m->tables_bytes != sizeof(Tb)) return cudaErrorInvalidValue;
  dim3 grid((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY);
  return launch_pdl(kern, grid, dim3(euler_threads<P, TX, TY>()), smem, s, a, static_cast<const Tb*>(m->tables)->pk);
}


// Cell-local work outside the stage: one thread per cell, its coefficients in registers.
template <int P>
__device__ __forceinline__ void load_state(const StageArgs& a, const float* u, int64_t cell, int64_t ncell, f2 (&c)[NV][P + 1][(P + 2) / 2]) {
  constexpr int N = P + 1, ND = N * N, MP = (N + 1) / 2;
  const bool v16 = ND % 4 == 0 && (reinterpret_cast<uintptr_t>(u) & 15) == 0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const float* src = u + ((int64_t)v * ncell + cell) * ND;
    if (v16) {
#pragma unroll
      for (int q = 0; q < ND / 4; ++q) {
        const float4 x = reinterpret_cast<const float4*>(src)[q];
        const int m = 4 * q, m2 = m + 2;
        c[v][m / N][m % N / 2] = mk2(x.x, x.y);
        c[v][m2 / N][m2 % N / 2] = mk2(x.z, x.w);
      }
    } else {
#pragma unroll
      for (int my = 0; my < N; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) c[v][my][p] = mk2(src[2 * p + N * my], 2 * p + 1 < N ? src[2 * p + 1 + N * my] : 0.0f);
    }
  }
}
constexpr int kCellThreads = 128;

// The node tabulations into shared memory (plain copies).
template <int P>
__device__ __forceinline__ void load_image(const float* img, float* s) {
  for (int f = threadIdx.x; f < PackedImage<2, P>::FLOATS; f += kCellThreads) s[f] = img[f];
  __syncthreads();
}

// The positivity limiter on its own: u_in -> u_out (may be the same array), theta per cell.
template <int P>
__global__ void __launch_bounds__(kCellThreads)
    euler_positivity_kernel(const __grid_constant__ StageArgs a, float* __restrict__ theta_out) {
  constexpr int N = P + 1, ND = N * N, MP = (N + 1) / 2;
  __shared__ __align__(16) float img[PackedImage<2, P>::FLOATS];
  load_image<P>(a.pk_img, img);
  const int64_t ncell = (int64_t)a.nx * a.ny;
  const int64_t cell = (int64_t)blockIdx.x * kCellThreads + threadIdx.x;
  if (cell >= ncell) return;
  if (!CVW_SPAN(a.status, cell, 1, a.lim_cell) ||
      !CVW_SPAN(a.status, ((NV - 1) * ncell + cell) * ND, ND, a.lim_in < a.lim_out ? a.lim_in : a.lim_out))
    return;
  f2 c[NV][N][MP];
  load_state<P>(a, a.u_in, cell, ncell, c);
  float th1, th2;
  if (!limit_positivity<N, MP>(a.gas_gamma, img, c, th1, th2)) atomicOr(a.status, kStatPositivity);
  if (theta_out) theta_out[cell] = th1 * th2;
  if (a.u_out == a.u_in && th1 == 1.0f && th2 == 1.0f) return;  // in place: nothing changed
  const bool v16 = ND % 4 == 0 && (reinterpret_cast<uintptr_t>(a.u_out) & 15) == 0;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    float* out = a.u_out + ((int64_t)v * ncell + cell) * ND;
    auto val = [&](int m) { return (m % N) & 1 ? c[v][m / N][m % N / 2].y : c[v][m / N][m % N / 2].x; };
    if (v16) {
#pragma unroll
      for (int q = 0; q < ND / 4; ++q)
        reinterpret_cast<float4*>(out)[q] = make_float4(val(4 * q), val(4 * q + 1), val(4 * q + 2), val(4 * q + 3));
    } else {
#pragma unroll
      for (int m = 0; m < ND; ++m) out[m] = val(m);
    }
  }
}

// max lambda_e = max(|v| + c) over every cell's volume and face Gauss nodes; non-positive density
// or pressure at a node raises the status bit, as in the stage.
template <int P>
__global__ void __launch_bounds__(kCellThreads)
    euler_wavespeed_kernel(const __grid_constant__ StageArgs a, const __grid_constant__ MaxSlots out) {
  constexpr int N = P + 1, ND = N * N, MP = (N + 1) / 2;
  __shared__ __align__(16) float img[PackedImage<2, P>::FLOATS];
  load_image<P>(a.pk_img, img);
  const int64_t ncell = (int64_t)a.nx * a.ny;
  float lam = 0.0f;
  bool bad = false;
  for (int64_t cell = (int64_t)blockIdx.x * kCellThreads + threadIdx.x; cell < ncell; cell += (int64_t)gridDim.x * kCellThreads) {
    if (!CVW_SPAN(a.status, ((NV - 1) * ncell + cell) * ND, ND, a.lim_in)) continue;
    f2 c[NV][N][MP];
    load_state<P>(a, a.u_in, cell, ncell, c);
    // mean + deviation, as in the stage: one rounding at the size of the mean
    float Ubar[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Ubar[v] = c[v][0][0].x, c[v][0][0].x = 0.0f;
    for_node_groups<N, MP>(img, c, [&](const f2 (&da)[NV], const f2 (&db)[NV], bool mid) {
      f2 U[NV], vn, cs;
#pragma unroll
      for (int v = 0; v < NV; ++v) U[v] = add2(dup2(Ubar[v]), da[v]);
      lam = fmaxf(lam, euler_wave(a.gas_gamma, U, 0, vn, cs, bad));
      if (mid) return;
#pragma unroll
      for (int v = 0; v < NV; ++v) U[v] = add2(dup2(Ubar[v]), db[v]);
      lam = fmaxf(lam, euler_wave(a.gas_gamma, U, 0, vn, cs, bad));
    });
  }
  if (bad) atomicOr(a.status, kStatPositivity);
  finish_max(lam, a.status, out);
}

template <int P>
cudaError_t launch_positivity_p(const cvweno_mesh_s* m, const StageArgs& a, float* theta, cudaStream_t s) {
  const int64_t ncell = (int64_t)a.nx * a.ny;
  euler_positivity_kernel<P><<<(unsigned)((ncell + kCellThreads - 1) / kCellThreads), kCellThreads, 0, s>>>(a, theta);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_wavespeed_p(const StageArgs& a, const MaxSlots& out, cudaStream_t s) {
  const int64_t ncell = (int64_t)a.nx * a.ny, blocks = (ncell + kCellThreads - 1) / kCellThreads;
  euler_wavespeed_kernel<P><<<(unsigned)(blocks < 1216 ? blocks : 1216), kCellThreads, 0, s>>>(a, out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_stage_euler(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  if (m->dim != 2) return cudaErrorNotSupported;
  switch (m->p * 2 + (a.limit_pos ? 1 : 0)) {
    case 2: return launch_euler<1, 16, 8, false>(m, a, s);
    case 3: return launch_euler<1, 16, 8, true>(m, a, s);
    case 4: return launch_euler<2, 16, 8, false>(m, a, s);
    case 5: return launch_euler<2, 16, 8, true>(m, a, s);
    case 6: return launch_euler<3, 16, 8, false>(m, a, s);
    case 7: return launch_euler<3, 16, 8, true>(m, a, s);
    case 8: return launch_euler<4, 8, 8, false>(m, a, s);
    case 9: return launch_euler<4, 8, 8, true>(m, a, s);
    default: return cudaErrorNotSupported;
  }
}

cudaError_t launch_positivity(const cvweno_mesh_s* m, const StageArgs& a, float* theta, cudaStream_t s) {
  if (m->dim != 2 || m->desc.system != CVWENO_EULER || m->kind != CVWENO_DG) return cudaErrorNotSupported;
  switch (m->p) {
    case 1: return launch_positivity_p<1>(m, a, theta, s);
    case 2: return launch_positivity_p<2>(m, a, theta, s);
    case 3: return launch_positivity_p<3>(m, a, theta, s);
    case 4: return launch_positivity_p<4>(m, a, theta, s);
    default: return cudaErrorNotSupported;
  }
}

cudaError_t launch_wavespeed_euler(const cvweno_mesh_s* m, const StageArgs& a, const MaxSlots& out, cudaStream_t s) {
  switch (m->p) {
    case 1: return launch_wavespeed_p<1>(a, out, s);
    case 2: return launch_wavespeed_p<2>(a, out, s);
    case 3: return launch_wavespeed_p<3>(a, out, s);
    case 4: return launch_wavespeed_p<4>(a, out, s);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace cvw
