// Continuous Galerkin (CG) stage for scalar conservation laws on periodic meshes.
//
// State: values at the Gauss-Lobatto-Legendre nodes of the global lattice
// (p nx) x (p ny), node I + (p nx) J.  One RK stage is
//   K1 cg_stage_cells   tile of cells + one-cell halo: nodal -> Legendre modes, the same
//                       vertex phase and cell sensor as DG (stages a-c), the lumped-mass
//                       projection P_h grad u at the cell's own nodes (reading A13, from
//                       the local integrals of the tile and halo cells), the CG SC weights
//                       with f_q = |grad u|^2 - gamma grad u . P_h grad u (Sec. 4; A24),
//                       and the cell-local residual
//                       int grad phi . f(u) - nu_e sum_q alpha_q w_q grad phi . (grad u - gamma P_h grad u)
//                       (Sec. 2.2, CG form of eq. stab)
//   K2 cg_node_stage2d  (2D) per tile of lattice nodes: the deterministic nodal assembly
//                       r_j, du = r_j / ML_j, and the two defect-correction sweeps
//                       du <- du + ML^{-1}(r - M_C du) (reading A12) with the
//                       tensor-product consistent mass, the second writing the SSP-RK3
//                       combination (or du itself for a residual); r and the first
//                       iterate are formed on a halo of 2p nodes, so one launch suffices
//   1D: cg_node_rhs (assembly, du = r / ML) and two cg_node_sweep launches
// Nodal sums gather the cells around a node in a fixed order.
#include "dg_scalar_kernel.cuh"

namespace cvw {
namespace {

// i mod n for any int i (n > 0), without a division when i is already in range
__device__ __forceinline__ int wrap_index(int i, int n) {
  if ((unsigned)i < (unsigned)n) return i;
  i %= n;
  return i < 0 ? i + n : i;
}

// Device image of the nodal tables in the order they take in shared memory (host-built, once per
// mesh): V[m][a], the Legendre modes of the nodal basis, by mirrored node pairs g = (a = g,
// a = p - g), whose columns differ by (-1)^m only (the middle node of an even p is its own
// partner): rows of mode pairs for the x direction, every entry doubled for the y direction.
template <int DIM, int P>
struct CgImage {
  static constexpr int N = P + 1, MP = (N + 1) / 2, NG = (N + 1) / 2;
  static constexpr int VX = 0;                                    // [NG][MP] pairs
  static constexpr int VY = VX + 2 * NG * MP;                     // [NG][N] doubled
  static constexpr int FLOATS = (VY + (DIM == 2 ? 2 * NG * N : 0) + 3) / 4 * 4;
};

// The tile's cells are modes computed here, so they lie as padded mode pairs (like the vertex
// data) at every degree.
template <int DIM, int P, int TX, int TY>
struct CgCells : TileLayout<DIM, P, TX, TY> {
  using L = TileLayout<DIM, P, TX, TY>;
  static constexpr bool PADDED = true;
  static __device__ __forceinline__ int cell(const int*, int hx, int hy) { return L::vertex(hy * L::HX + hx); }
};

template <int DIM, int P, int TX, int TY>
struct CgLayout {
  using L = CgCells<DIM, P, TX, TY>;
  using Img = PackedImage<DIM, P>;
  static constexpr int N = P + 1, ND = L::ND, NH = L::NH, NT = L::NT;
  static constexpr int NNX = P * (TX + 2) + 1, NNY = DIM == 2 ? P * (TY + 2) + 1 : 1;
  // nodal rows at a 16-byte stride with room for a per-row phase of up to 3 floats
  static constexpr int NNXP = (NNX + 3 + 3) / 4 * 4;
  static constexpr int OFF_C = 0;                                              // cells
  static constexpr int OFF_ST = (L::VS * NH + 3) / 4 * 4;                      // vertex data, then stage (d)
  // as the DG tile's; in 1D, where no barrier parts the sensor from stage (d), behind the vertex data
  static constexpr int OFF_NQ = DIM == 1 ? OFF_ST + L::VS * L::NVT : OFF_ST, OFF_S12 = OFF_NQ + ND * NT;
  static constexpr int OFF_IMG = ((DIM == 1 ? OFF_S12 : OFF_ST + imax(L::VS * L::NVT, L::SCF)) + 3) / 4 * 4;
  static constexpr int OFF_VIMG = OFF_IMG + Img::FLOATS;
  // The nodal tile is dead once the halo cells are converted to modes, the local integrals
  // (pairs (x, y), [ND][NH]) once P_h grad u is gathered; then its modes
  // (pairs, [2 NY1 MP][NT]) lie there, and gamma_e of the troubled cells for the other threads.
  static constexpr int OFF_NODE = OFF_VIMG + CgImage<DIM, P>::FLOATS;
  static constexpr int OFF_B = OFF_NODE;
  static constexpr int OFF_PH = OFF_NODE, OFF_GAM = OFF_PH + 4 * L::NY1 * L::MP * NT;
  static constexpr int FLOATS = OFF_NODE + imax(imax(2 * ND * NH, NNXP * NNY), OFF_GAM - OFF_PH + NT);
  static constexpr size_t BYTES = sizeof(float) * (size_t)FLOATS;
};

// Nodal values u[b][a] (polynomial at the cell's nodes) to Legendre modes, V x V: sums and
// differences of mirrored nodes feed the even and the odd modes.
template <int DIM, int P>
__device__ __forceinline__ void nodes_to_modes(const float* vimg, const float (&u)[DIM == 2 ? P + 1 : 1][P + 1],
                                               f2 (&c)[DIM == 2 ? P + 1 : 1][(P + 2) / 2]) {
  using I = CgImage<DIM, P>;
  constexpr int N = I::N, MP = I::MP, NG = I::NG, NY1 = DIM == 2 ? N : 1;
  f2 t[NY1][MP];
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    f2 v[MP];
    load_pairs<MP>(vimg + I::VX + 2 * MP * g, v);
    const bool mid = 2 * g == P;
#pragma unroll
    for (int b = 0; b < NY1; ++b) {
      const f2 sd = mid ? mk2(u[b][g], 0.0f) : mk2(u[b][g] + u[b][P - g], u[b][g] - u[b][P - g]);
#pragma unroll
      for (int p = 0; p < MP; ++p) t[b][p] = g == 0 ? mul2(v[p], sd) : fma2(v[p], sd, t[b][p]);
    }
  }
  if constexpr (DIM == 1) {
#pragma unroll
    for (int p = 0; p < MP; ++p) c[0][p] = t[0][p];
  } else {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      f2 v[N];
      load_pairs<N>(vimg + I::VY + 2 * N * g, v);
      const bool mid = 2 * g == P;
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const f2 e = mid ? t[g][p] : add2(t[g][p], t[P - g][p]);
        const f2 o = mid ? mk2(0.0f, 0.0f) : sub2(t[g][p], t[P - g][p]);
#pragma unroll
        for (int my = 0; my < NY1; ++my)
          c[my][p] = g == 0 ? mul2(v[my], (my & 1) ? o : e) : fma2(v[my], (my & 1) ? o : e, c[my][p]);
      }
    }
  }
}

// Nodal functionals r[b][a] = sum_m V[my][b] V[mx][a] R[my][mx] of a modal one, the transpose of
// nodes_to_modes: node row by node row, handed to f(b, g, (value at a = g, value at a = p - g)).
template <int DIM, int P, class F>
__device__ __forceinline__ void modes_to_nodes_t(const float* vimg, const f2 (&R)[DIM == 2 ? P + 1 : 1][(P + 2) / 2], F&& f) {
  using I = CgImage<DIM, P>;
  constexpr int N = I::N, MP = I::MP, NG = I::NG, NY1 = DIM == 2 ? N : 1;
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    f2 v[MP], tb[NY1];
    load_pairs<MP>(vimg + I::VX + 2 * MP * g, v);
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      f2 s = mul2(v[0], R[my][0]);
#pragma unroll
      for (int p = 1; p < MP; ++p) s = fma2(v[p], R[my][p], s);
      tb[my] = mk2(s.x + s.y, s.x - s.y);
    }
    if constexpr (DIM == 1) {
      f(0, g, tb[0]);
    } else {
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        f2 w[N];
        load_pairs<N>(vimg + I::VY + 2 * N * h, w);
        f2 e = mul2(w[0], tb[0]), o = mul2(w[1], tb[1]);
#pragma unroll
        for (int my = 2; my < N; ++my) {
          if (my & 1) o = fma2(w[my], tb[my], o);
          else e = fma2(w[my], tb[my], e);
        }
        f(h, g, add2(e, o));
        if (2 * h != P) f(P - h, g, sub2(e, o));
      }
    }
  }
}

// int P_m d/dxi u (x) and d/deta (y) over the reference cell for u = sum c_m P_m: int P_mx P_kx' is 2
// for kx > mx of the other parity, int P_my P_ky 2/(2my+1) on the diagonal (1 in 1D).
template <int DIM, int N, int NY1, int MP>
__device__ __forceinline__ void gradient_moments(const f2 (&c)[NY1][MP], f2 (&gx)[NY1][MP], f2 (&gy)[NY1][MP]) {
  auto val = [&](int my, int k) { return k >= N ? 0.0f : (k & 1) ? c[my][k / 2].y : c[my][k / 2].x; };
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    const float sy = DIM == 2 ? 4.0f / (2 * my + 1) : 2.0f;
    float d[2 * MP + 2];  // d[m] = c[m+1] + c[m+3] + ...
    d[2 * MP + 1] = d[2 * MP] = 0.0f;
#pragma unroll
    for (int m = 2 * MP - 1; m >= 0; --m) d[m] = val(my, m + 1) + d[m + 2 <= 2 * MP + 1 ? m + 2 : 2 * MP];
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      gx[my][p] = mk2(sy * d[2 * p], 2 * p + 1 < N ? sy * d[2 * p + 1] : 0.0f);
      gy[my][p] = mk2(0.0f, 0.0f);
    }
  }
  if constexpr (DIM == 2) {
#pragma unroll
    for (int my = NY1 - 2; my >= 0; --my)
#pragma unroll
      for (int p = 0; p < MP; ++p) gy[my][p] = my + 3 < NY1 ? add2(c[my + 1][p], gy[my + 2 < NY1 ? my + 2 : my][p]) : c[my + 1][p];
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) gy[my][p] = mul2(gy[my][p], mk2(4.0f / (4 * p + 1), 4.0f / (4 * p + 3)));
  }
}

// lumped mass of a 1D lattice node with local index a in [0, p): its GLL weight times
// dx/2, counted twice at cell vertices (two cells share them)
template <int DIM, int P>
__device__ __forceinline__ float ml1(const CgTables<DIM, P>& C, int a, float h) {
  return (a == 0 ? 2.0f : 1.0f) * C.wl[a] * h;
}

// Values tb and x-derivatives td at the node pair of tables b (P) and d (P'), row by row.
template <int N, int NY1, int MP>
__device__ __forceinline__ void x_values(const f2 (&b)[MP], const f2 (&d)[MP], const f2 (&c)[NY1][MP], f2 (&tb)[NY1],
                                         f2 (&td)[NY1]) {
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    f2 s = mul2(b[0], c[my][0]), sd = mul2(d[0], c[my][0]);
#pragma unroll
    for (int p = 1; p < MP; ++p) {
      s = fma2(b[p], c[my][p], s);
      sd = fma2(d[p], c[my][p], sd);
    }
    tb[my] = mk2(s.x + s.y, s.x - s.y);
    td[my] = mk2(sd.x + sd.y, sd.y - sd.x);
  }
}

// The same values of modes kept in shared memory, [NY1 MP] rows NT apart.
template <int NY1, int MP, int NT>
__device__ __forceinline__ void projection_values(const f2 (&b)[MP], const f2* sp, f2 (&t)[NY1]) {
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    f2 s = mul2(b[0], sp[my * MP * NT]);
#pragma unroll
    for (int p = 1; p < MP; ++p) s = fma2(b[p], sp[(my * MP + p) * NT], s);
    t[my] = mk2(s.x + s.y, s.x - s.y);
  }
}

// The same of modes in registers.
template <int NY1, int MP>
__device__ __forceinline__ void projection_values(const f2 (&b)[MP], const f2 (&c)[NY1][MP], f2 (&t)[NY1]) {
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    f2 s = mul2(b[0], c[my][0]);
#pragma unroll
    for (int p = 1; p < MP; ++p) s = fma2(b[p], c[my][p], s);
    t[my] = mk2(s.x + s.y, s.x - s.y);
  }
}

// Threads of a block of the CG cell kernel, and the resident CTAs its registers must allow.
// KPP 256^2, us per step: p = 3, 4 CTAs of 128 threads 85.9, 4 of 160 (96 registers, spills) 91.0,
// 3 of 128 95.9, 5 of 128 92.7; p = 2, 4 CTAs 56.6, 3 69.7, 5 58.1.
template <int DIM, int P, int TX, int TY, bool FEW = false>
__host__ __device__ constexpr int cg_block_threads() {
  return TX * TY + (DIM == 1 || P == 1 || FEW ? 32 : 0);
}
template <int DIM, int P, bool FEW = false>
constexpr int cg_min_ctas() {
  return DIM == 1 || FEW ? 1 : P == 1 ? 6 : P <= 3 ? 4 : 2;
}

// One CTA per tile; bound by FP32 issue and latency at 13 warps per SM (49 % of the issue slots at
// 256^2).  On two-wide FMAs and in the modal basis (local integrals, projection and residual go
// to the nodes and back by V) the Q3 step takes 85.9 us instead of 107, Q2 56.6 instead of 65, Q1
// 29.7 instead of 42 (KPP 256^2, node kernel included).
template <int DIM, int P, int SYS, int TX, int TY, bool FEW = false>
__global__ void __launch_bounds__((cg_block_threads<DIM, P, TX, TY, FEW>()), (cg_min_ctas<DIM, P, FEW>()))
    cg_stage_cells(const __grid_constant__ StageArgs a, const __grid_constant__ PackedTables<DIM, P> T,
                   const __grid_constant__ CgTables<DIM, P> C) {
  using G = CgLayout<DIM, P, TX, TY>;
  using L = typename G::L;
  using Img = PackedImage<DIM, P>;
  using Law = ScalarLaw<SYS, DIM>;
  constexpr int N = L::N, ND = L::ND, NT = L::NT, HX = L::HX, HY = L::HY, NH = L::NH, MP = L::MP, NG = L::NG;
  constexpr int NB = cg_block_threads<DIM, P, TX, TY, FEW>();  // threads of the block
  constexpr int NNX = G::NNX, NNY = G::NNY, NNXP = G::NNXP;
  constexpr int NY1 = L::NY1, NGY = DIM == 2 ? NG : 1;
  extern __shared__ __align__(16) float smem[];
  float* sc = smem + G::OFF_C;
  float* st = smem + G::OFF_ST;
  float* sNq = smem + G::OFF_NQ;
  const float* img = smem + G::OFF_IMG;
  const float* vimg = smem + G::OFF_VIMG;
  float* snode = smem + G::OFF_NODE;
  f2* sb = reinterpret_cast<f2*>(smem + G::OFF_B);

  const int nx = a.nx, ny = DIM == 2 ? a.ny : 1;
  const int nnx = a.nnx, nny = DIM == 2 ? a.nny : 1;
  const int i0 = blockIdx.x * TX, j0 = DIM == 2 ? blockIdx.y * TY : 0;
  const float hdx = 1.0f / a.two_dx, hdy = DIM == 2 ? 1.0f / a.two_dy : 1.0f;
  __shared__ int sc_count;        // troubled cells of the tile,
  __shared__ short sc_cell[NT];   // and their threads
  if (threadIdx.x == 0) sc_count = 0;

  // ---- nodal values of the tile and its halo (periodic lattice) -------------------------
  for (int f = threadIdx.x; f < Img::FLOATS / 4; f += NB) cp_async16(smem + G::OFF_IMG + 4 * f, a.pk_img + 4 * f);
  for (int f = threadIdx.x; f < CgImage<DIM, P>::FLOATS / 4; f += NB) cp_async16(smem + G::OFF_VIMG + 4 * f, a.cg_img + 4 * f);
  pdl_wait();  // everything below reads or writes what earlier kernels write
  // Node (ix, iy) lands at snode[iy][sph[iy] + ix].  Where the tile's rows do not wrap in x
  // and the state is 16-byte aligned, each row is copied as the 16-byte chunks that cover
  // it: the first chunk starts up to 3 floats early (sph, the row's phase), the last is
  // zero-filled past the row's last node, so no read leaves the row's own span or the
  // floats just before it.  Otherwise 4-byte copies, phase 0.
  __shared__ int sph[NNY];
  {
    const int I0 = P * (i0 - 1), J0 = DIM == 2 ? P * (j0 - 1) : 0;
    const bool rows16 = I0 >= 0 && I0 + NNX <= nnx && (reinterpret_cast<uintptr_t>(a.u_in) & 15) == 0;
    if (rows16) {
      constexpr int NCH = NNXP / 4;  // chunks per row
      for (int f = threadIdx.x; f < NNY * NCH; f += NB) {
        const int iy = f / NCH, k = f - iy * NCH;
        const int J = DIM == 2 ? wrap_index(J0 + iy, nny) : 0;
        const int64_t g0 = (int64_t)J * nnx + I0;  // the row's first node
        const int ph = (int)(g0 & 3);
        const int64_t c0 = g0 - ph + 4 * k;
        const int64_t left = g0 + NNX - c0;  // wanted floats from the chunk's start on
        if (left > 0 && CVW_SPAN(a.status, c0, left >= 4 ? 4 : left, a.lim_in))
          cp_async16z(snode + iy * NNXP + 4 * k, a.u_in + c0, left >= 4 ? 16 : (int)left * 4);
        if (k == 0) sph[iy] = ph;
      }
    } else {
      for (int f = threadIdx.x; f < NNX * NNY; f += NB) {
        const int ix = f % NNX, iy = f / NNX;
        const int I = wrap_index(I0 + ix, nnx);
        const int J = DIM == 2 ? wrap_index(J0 + iy, nny) : 0;
        if (CVW_SPAN(a.status, (size_t)J * nnx + I, 1, a.lim_in)) cp_async4(snode + iy * NNXP + ix, a.u_in + (size_t)J * nnx + I, 4);
      }
      for (int iy = threadIdx.x; iy < NNY; iy += NB) sph[iy] = 0;
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // ---- every halo cell: nodal -> Legendre modes c = (V x V) u_loc -------------------------
  // The transform is applied to u_loc - u_ref: every mode but the mean is unchanged (the rows of V
  // beyond the mean sum to zero), the mean gets u_ref back, and a constant cell yields exactly zero
  // non-mean modes.  u_ref is a middle node: the even modes come from sums of mirrored nodes,
  // which about the middle nearly cancel on smooth data (about the first node they do not, and
  // round at their own size: RMS error of the second and higher even modes 2 to 5 times as large at
  // p = 2 and 4, 1.7 times at p = 3).
  for (int h = threadIdx.x; h < NH; h += NB) {
    const int hx = h % HX, hy = DIM == 2 ? h / HX : 0;
    float u[NY1][N];
#pragma unroll
    for (int b = 0; b < NY1; ++b)
#pragma unroll
      for (int aa = 0; aa < N; ++aa) u[b][aa] = snode[sph[P * hy + b] + (P * hx + aa) + NNXP * (P * hy + b)];
    const float uref = u[DIM == 2 ? P / 2 : 0][P / 2];
#pragma unroll
    for (int b = 0; b < NY1; ++b)
#pragma unroll
      for (int aa = 0; aa < N; ++aa) u[b][aa] -= uref;
    f2 c[NY1][MP];
    nodes_to_modes<DIM, P>(vimg, u, c);
    c[0][0].x += uref;
    store_vertex<L>(sc, h, c);
  }
  __syncthreads();
  // ---- (a)+(b) vertex candidates (shared with DG) ---------------------------------------
  tile_vertex_phase<DIM, P, TX, TY, NB, false, L>(a, T, sc, nullptr, st, i0, j0, nx, ny);
  // ---- P_h local integrals b_a = int phi_a grad u of every tile and halo cell (reading A13),
  // with dx dy / 4 = hdx hdy and the factor 2/dx of d/dx cancelling hdx.  From the block's last
  // thread backwards: the vertex phase's extra round (if any) falls on the first warp.
  for (int h = NB - 1 - threadIdx.x; h < NH; h += NB) {
    f2 c[NY1][MP], gx[NY1][MP], gy[NY1][MP];
    load_cell<L>(sc, L::vertex(h), c);
    gradient_moments<DIM, N, NY1, MP>(c, gx, gy);
    modes_to_nodes_t<DIM, P>(vimg, gx, [&](int b, int g, f2 v) {
      sb[(g + N * b) * NH + h].x = hdy * v.x;
      sb[(P - g + N * b) * NH + h].x = hdy * v.y;
    });
    if constexpr (DIM == 2)
      modes_to_nodes_t<DIM, P>(vimg, gy, [&](int b, int g, f2 v) {
        sb[(g + N * b) * NH + h].y = hdx * v.x;
        sb[(P - g + N * b) * NH + h].y = hdx * v.y;
      });
  }
  __syncthreads();
  pdl_launch_dependents();

  // ---- one thread per own cell (the others take part in stage (d)) --------------------------
  const int tx = threadIdx.x % TX, ty = DIM == 2 ? threadIdx.x / TX : 0;
  const int gi = i0 + tx, gj = j0 + ty;
  const size_t cell = (size_t)gj * nx + gi;
  const bool active = (NB == NT || threadIdx.x < NT) && gi < nx && gj < ny &&
                      CVW_SPAN(a.status, cell, 1, a.lim_cell);  // per-cell outputs and rloc
  const int hcx = tx + 1, hcy = DIM == 2 ? min(ty, TY - 1) + 1 : 0;
  f2 c[NY1][MP];
  load_cell<L>(sc, L::cell(nullptr, hcx, hcy), c);
  const float ubar = c[0][0].x;
  const bool sensor_only = (a.mode & kModeSensorOnly) != 0, need_lam = !(a.lambda_const > 0.0f);
  const Law law(a, ubar);
  float n0 = 0.0f, gam = 1.0f, lam = need_lam ? 0.0f : a.lambda_const;
  f2 px[NY1][MP], py[NY1][MP];  // modes of P_h grad u
  if (active) {
    gam = cell_sensor<DIM, P, TX, TY>(a, T, st, c, tx, ty, n0, px);
    // lambda_e over the volume and face Gauss nodes of the cell polynomial
    if (need_lam) {
      c[0][0].x = 0.0f;
      // (the mean's speed, never above the nodes', keeps an infinite state's speed infinite where the
      // deviations are NaN)
      lam = fmaxf(cell_speed<DIM, P>(img, law, ubar, c), law.speed(ubar));
    }
    if (a.gamma_out) a.gamma_out[cell] = gam;
    if (a.nu_out) a.nu_out[cell] = lam * a.nu_scale;
    if (a.lambda_out) a.lambda_out[cell] = lam;
  }
  if (sensor_only) return;

  // P_h grad u at the own cell's nodes: sum over the cells sharing each node / ML
  if (active) {
    float nx_[NY1][N], ny_[NY1][N];
#pragma unroll
    for (int bb = 0; bb < NY1; ++bb)
#pragma unroll
      for (int aa = 0; aa < N; ++aa) {
        f2 s = mk2(0.0f, 0.0f);
        // x-neighbours of the node: (halo column, local index)
        const int ncx = (aa == 0 || aa == P) ? 2 : 1;
        const int ncy = DIM == 2 ? ((bb == 0 || bb == P) ? 2 : 1) : 1;
#pragma unroll
        for (int jy = 0; jy < ncy; ++jy)
#pragma unroll
          for (int jx = 0; jx < ncx; ++jx) {
            int cx = hcx, la = aa, cy = hcy, lb = bb;
            if (aa == 0) { cx = jx == 0 ? hcx - 1 : hcx; la = jx == 0 ? P : 0; }
            if (aa == P) { cx = jx == 0 ? hcx : hcx + 1; la = jx == 0 ? P : 0; }
            if (DIM == 2 && bb == 0) { cy = jy == 0 ? hcy - 1 : hcy; lb = jy == 0 ? P : 0; }
            if (DIM == 2 && bb == P) { cy = jy == 0 ? hcy : hcy + 1; lb = jy == 0 ? P : 0; }
            s = add2(s, sb[(la + N * lb) * NH + cy * HX + cx]);
          }
        // 1 / ML of the node: the inverse lumped masses of its two 1D indices
        const float iml = C.iml[aa == P ? 0 : aa] * a.two_dx * (DIM == 2 ? C.iml[bb == P ? 0 : bb] * a.two_dy : 1.0f);
        nx_[bb][aa] = s.x * iml;
        ny_[bb][aa] = s.y * iml;
      }
    nodes_to_modes<DIM, P>(vimg, nx_, px);
    if constexpr (DIM == 2) nodes_to_modes<DIM, P>(vimg, ny_, py);
  }

  // ---- (d) SC weights (A24), f_q = |grad u|^2 - gamma grad u . P_h grad u: the troubled cells' node
  // groups shared by the tile's threads, as in the DG kernel
  bool troubled = false;
  float afac = -1.0f;
  if (active) {
    troubled = a.sc && gam < a.c_gamma && n0 > 1e-30f;
    if (a.troubled_override) {
      const int ov = a.troubled_override[cell];
      if (ov >= 0) troubled = ov && n0 > 1e-30f;
    }
  }
  const bool need_sc = troubled && gam < 1.0f;
  f2* sP = reinterpret_cast<f2*>(smem + G::OFF_PH);
  if constexpr (DIM == 1) {
    // by the cell's own thread, with the projection in its registers: cells of two to five nodes have
    // less to share than the tile's barriers cost (300 cells P1: 27.9 us per step shared, 26.6 so with
    // unrolled loops)
    if (need_sc) {
      float s1 = 0.0f, s2 = 0.0f;
#pragma unroll 1
      for (int g = 0; g < NG; ++g) {
        f2 b[MP], d[MP], tb[1], td[1], tp[1], g1, g2, nq;
        sc_node_group<DIM, P, TX, TY, false, L>(a, T, img, sNq, sc, nullptr, threadIdx.x, g, 0, g1, g2, &nq);
        load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
        load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
        f2 cc[1][MP];
        load_cell<L>(sc, L::cell(nullptr, hcx, 0), cc);
        cc[0][0].x = 0.0f;
        x_values<N, 1, MP>(b, d, cc, tb, td);
        projection_values<1, MP>(b, px, tp);
        const f2 f = mul2(dup2(-gam * a.two_dx * img[Img::WX + g]), mul2(td[0], tp[0]));
        g1 = add2(g1, f);
        g2 = fma2(nq, f, g2);
        s1 += g1.x + g1.y;
        s2 += g2.x + g2.y;
      }
      if (s1 > 0.0f && s2 > 0.0f) afac = s1 / s2;
    }
  } else {
  if (need_sc) sc_cell[atomicAdd(&sc_count, 1)] = (short)threadIdx.x;
  const bool any_sc = __syncthreads_or(need_sc);  // (and every cell has gathered the local integrals)
  // the projection's modes wait in shared memory: held in registers over the volume flux they
  // would cost the kernel a resident CTA
  if (active) {
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        sP[(my * MP + p) * NT + threadIdx.x] = px[my][p];
        if (DIM == 2) sP[((NY1 + my) * MP + p) * NT + threadIdx.x] = py[my][p];
      }
  }
  if (any_sc) {
    const int n = sc_count;
    float* sGam = smem + G::OFF_GAM;
    float* sS = smem + G::OFF_S12;
    if (need_sc) sGam[threadIdx.x] = gam;
    __syncthreads();
#pragma unroll 1
    for (int t = threadIdx.x; t < n * L::NGG; t += NB) {
      const int gh = t / n, id = sc_cell[t - gh * n], g = gh / NGY, h = gh - g * NGY;
      f2 s1, s2, nqa, nqb = mk2(0.0f, 0.0f);
      sc_node_group<DIM, P, TX, TY, false, L>(a, T, img, sNq, sc, nullptr, id, g, h, s1, s2, &nqa, &nqb);
      // grad u . P_h grad u at the group's nodes
      f2 b[MP], d[MP], tp[NY1];
      load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
      load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
      const float gm = -sGam[id];
      f2 tb[NY1], td[NY1];
      {
        f2 cc[NY1][MP];
        load_cell<L>(sc, L::cell(nullptr, id % TX + 1, DIM == 2 ? id / TX + 1 : 0), cc);
        cc[0][0].x = 0.0f;
        x_values<N, NY1, MP>(b, d, cc, tb, td);
      }
      if constexpr (DIM == 1) {
        projection_values<NY1, MP, NT>(b, sP + id, tp);
        const f2 f = mul2(dup2(gm * a.two_dx * img[Img::WX + g]), mul2(td[0], tp[0]));
        s1 = add2(s1, f);
        s2 = fma2(nqa, f, s2);
      } else {
        const float* yb_ = img + Img::BY + 2 * N * h;
        f2 xa, xb, ya, yb, pa, pb;
        node_gradient<N, MP>(yb_, img + Img::DY + 2 * N * h, tb, td, xa, xb, ya, yb);
        projection_values<NY1, MP, NT>(b, sP + id, tp);
        node_rows<N>(yb_, tp, pa, pb);
        xa = mul2(mul2(dup2(a.two_dx), xa), pa);
        xb = mul2(mul2(dup2(a.two_dx), xb), pb);
        projection_values<NY1, MP, NT>(b, sP + NY1 * MP * NT + id, tp);
        node_rows<N>(yb_, tp, pa, pb);
        const f2 w = dup2(gm * img[Img::WX + g] * img[Img::WY + h]), ky = dup2(a.two_dy);
        const f2 fa = mul2(w, fma2(mul2(ky, ya), pa, xa));
        s1 = add2(s1, fa);
        s2 = fma2(nqa, fa, s2);
        if (2 * h != N - 1) {
          const f2 fb = mul2(w, fma2(mul2(ky, yb), pb, xb));
          s1 = add2(s1, fb);
          s2 = fma2(nqb, fb, s2);
        }
      }
      sS[gh * NT + id] = s1.x + s1.y;
      sS[(L::NGG + gh) * NT + id] = s2.x + s2.y;
    }
    __syncthreads();
    if (need_sc) {
      float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
      for (int gh = 0; gh < L::NGG; ++gh) {
        s1 += sS[gh * NT + threadIdx.x];
        s2 += sS[(L::NGG + gh) * NT + threadIdx.x];
      }
      if (s1 > 0.0f && s2 > 0.0f) afac = s1 / s2;
    }
  }
  }  // DIM == 2
  if (!active) return;
  if (a.troubled_out) a.troubled_out[cell] = troubled ? 1 : 0;
  if (a.alpha_out) {
#pragma unroll 1
    for (int q = 0; q < ND; ++q) a.alpha_out[cell * ND + q] = afac >= 0.0f ? sNq[q * NT + threadIdx.x] * afac : 1.0f;
  }

  // ---- (e) modal residual R: the volume flux as deviations from f(ubar) (the constant part, which
  // lives on the cell's edges and telescopes between neighbours, is added below), and
  // -nu alpha (grad u - gamma P_h grad u)
  load_cell<L>(sc, L::cell(nullptr, hcx, hcy), c);  // again, rather than held
  c[0][0].x = 0.0f;
  const float nu = lam * a.nu_scale;
  f2 R[NY1][MP];
#pragma unroll
  for (int my = 0; my < NY1; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) R[my][p] = mk2(0.0f, 0.0f);
  float dummy = 0.0f;
  volume_flux<DIM, P>(a, img, law, ubar, c, false, true, dummy, R);
  if (afac < 0.0f) {
    // linear weights: the Gauss rule is exact, so the gradient's part is the stiffness form and
    // the projection's int P_mx' P_kx = 2 for kx < mx of the other parity, diagonal in y
    add_stiffness<DIM, N, NY1, MP>(-nu * a.two_dx * a.two_dx, -nu * a.two_dy * a.two_dy, c, R);
    const float kx = nu * gam * a.two_dx, ky = nu * gam * a.two_dy;
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      const float sy = DIM == 2 ? 4.0f / (2 * my + 1) : 2.0f;
      float even = 0.0f, odd = 0.0f;  // sums of the even and odd modes so far
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const f2 v = DIM == 1 ? px[my][p] : sP[(my * MP + p) * NT + threadIdx.x];
        const float e1 = even + v.x;
        R[my][p] = fma2(dup2(kx * sy), mk2(odd, e1), R[my][p]);
        even = e1;
        odd += v.y;
      }
    }
    if constexpr (DIM == 2) {
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        const f2 s = mul2(dup2(ky), mk2(4.0f / (4 * p + 1), 4.0f / (4 * p + 3)));
        f2 even = sP[(NY1 * MP + p) * NT + threadIdx.x], odd = mk2(0.0f, 0.0f);
#pragma unroll
        for (int my = 1; my < NY1; ++my) {
          R[my][p] = fma2(s, (my & 1) ? even : odd, R[my][p]);
          const f2 v = sP[((NY1 + my) * MP + p) * NT + threadIdx.x];
          if (my & 1) odd = my == 1 ? v : add2(odd, v);
          else even = add2(even, v);
        }
      }
    }
  } else {
    const float m = -nu * afac;
#pragma unroll 1
    for (int g = 0; g < NG; ++g) {
      f2 b[MP], d[MP], tb[NY1], td[NY1], tp[NY1], tq[NY1], hx[NY1], hy[NY1];
      load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
      load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
      x_values<N, NY1, MP>(b, d, c, tb, td);
      if constexpr (DIM == 1) projection_values<NY1, MP>(b, px, tp);
      else projection_values<NY1, MP, NT>(b, sP + threadIdx.x, tp);
      if (DIM == 2) projection_values<NY1, MP, NT>(b, sP + NY1 * MP * NT + threadIdx.x, tq);
#pragma unroll
      for (int my = 0; my < NY1; ++my) hx[my] = hy[my] = mk2(0.0f, 0.0f);
      const float* nq = sNq + threadIdx.x;
      if constexpr (DIM == 1) {
        const f2 al = mul2(dup2(m), mk2(nq[g * NT], nq[(N - 1 - g) * NT]));
        hx[0] = mul2(al, fma2(dup2(a.two_dx), td[0], mul2(dup2(-gam), tp[0])));
      } else {
#pragma unroll 1
        for (int h = 0; h < NGY; ++h) {
          const float *yb = img + Img::BY + 2 * N * h, *yd = img + Img::DY + 2 * N * h;
          f2 xa, xb, ya, yy, pa, pb, qa, qb;
          node_gradient<N, MP>(yb, yd, tb, td, xa, xb, ya, yy);
          node_rows<N>(yb, tp, pa, pb);
          node_rows<N>(yb, tq, qa, qb);
          const bool mid = (N & 1) && h == NG - 1;
          const f2 w = dup2(m * img[Img::WY + h]), kx = dup2(a.two_dx), ky = dup2(a.two_dy), gm = dup2(-gam);
          const float *na = nq + (g + N * h) * NT, *nb = nq + (g + N * (N - 1 - h)) * NT;
          const f2 la = mul2(w, mk2(na[0], na[(N - 1 - 2 * g) * NT]));
          f2 lb = mul2(w, mk2(nb[0], nb[(N - 1 - 2 * g) * NT]));
          if (mid) lb = mk2(0.0f, 0.0f);
          const f2 fx = mul2(la, fma2(gm, pa, mul2(kx, xa))), gx = mul2(lb, fma2(gm, pb, mul2(kx, xb)));
          const f2 fy = mul2(la, fma2(gm, qa, mul2(ky, ya))), gy = mul2(lb, fma2(gm, qb, mul2(ky, yy)));
          project_rows<N>(yb, yd, fx, gx, fy, gy, hx, hy);
        }
      }
      project_nodes<NY1, MP>(b, d, a.two_dx * img[Img::WX + g], a.two_dy * img[Img::WX + g], hx, hy, R);
    }
  }
  // to the nodal basis; r[a, b] scaled by the cell's Jacobian
  float r[ND];
  modes_to_nodes_t<DIM, P>(vimg, R, [&](int b, int g, f2 v) {
    r[g + N * b] = hdx * hdy * v.x;
    if (2 * g != P) r[P - g + N * b] = hdx * hdy * v.y;
  });
  // The constant part of the flux: int_K d_x phi_ab f(ubar_e) = (delta_{a,p} - delta_{a,0})
  // wl_b (dy/2) f_x(ubar_e) (likewise in y).  At the nodes of an edge between a left cell L
  // and a right cell R the two cells' terms sum to (f_x(ubar_L) - f_x(ubar_R)) wl_b dy/2;
  // each cell adds that sum for its left and bottom edges (its right and top edges are
  // its neighbours' left and bottom ones), the difference formed by the deviation formula
  // of its own law from the halo means.
  {
    float fx, fy;
    law.flux_dev(sc[L::cell(nullptr, hcx - 1, hcy)] - ubar, fx, fy);  // f(ubar_left) - f(ubar_e)
#pragma unroll
    for (int b = 0; b < NY1; ++b) r[N * b] = fmaf(fx, DIM == 2 ? C.wl[b] * hdy : 1.0f, r[N * b]);
    if constexpr (DIM == 2) {
      law.flux_dev(sc[L::cell(nullptr, hcx, hcy - 1)] - ubar, fx, fy);  // f(ubar_below) - f(ubar_e)
#pragma unroll
      for (int aa = 0; aa < N; ++aa) r[aa] = fmaf(fy, C.wl[aa] * hdx, r[aa]);
    }
  }
  // node row b of the cells of a mesh row is contiguous in rloc (mesh-owned, aligned): the warp's
  // stores and the node kernel's gathers are whole lines
  const size_t rowlen = (size_t)nx * N, row0 = DIM == 2 ? (size_t)gj * N * rowlen : 0;
#pragma unroll
  for (int b = 0; b < NY1; ++b) {
    const size_t k = row0 + b * rowlen + (size_t)gi * N;
    if (!CVW_SPAN(a.status, k, N, CVW_EXTENT(a, lim_cell) * ND)) continue;
    if constexpr (N == 4) {
      *reinterpret_cast<float4*>(a.rloc + k) = make_float4(r[N * b], r[N * b + 1], r[N * b + N - 2], r[N * b + N - 1]);
    } else if constexpr (N == 2) {
      *reinterpret_cast<float2*>(a.rloc + k) = make_float2(r[N * b], r[N * b + 1]);
    } else {
#pragma unroll
      for (int m = 0; m < N; ++m) a.rloc[k + m] = r[N * b + m];
    }
  }
}

// 1D nodal assembly r_j at lattice node I, 0 <= I < nnx: the sum of the cell-local residuals
// (which carry the telescoped flux of the cell means) over the cells containing the node, the
// left one first.  A node with local index 0 lies in cell i - 1 (as its local p) and cell i.
template <int P>
__device__ __forceinline__ float node_residual(const StageArgs& a, int I) {
  constexpr int N = P + 1;
  const int i = I / P, aa = I - i * P;
  const int cx0 = aa == 0 ? (i == 0 ? a.nx - 1 : i - 1) : i, lx0 = aa == 0 ? P : aa;
  const int64_t lim = CVW_EXTENT(a, lim_cell) * N;
  auto rl = [&](size_t k) { return CVW_SPAN(a.status, k, 1, lim) ? a.rloc[k] : 0.0f; };
  float r = rl((size_t)cx0 * N + lx0);
  if (aa == 0) r += rl((size_t)i * N);
  return r;
}

// 1D nodal assembly: r_j and du = r_j / ML_j.
template <int DIM, int P>
__global__ void cg_node_rhs(const __grid_constant__ StageArgs a, const __grid_constant__ CgTables<DIM, P> C) {
  static_assert(DIM == 1, "2D: cg_node_stage2d");
  const int64_t nn = (int64_t)a.nnx * (DIM == 2 ? a.nny : 1);
  const float hdx = 1.0f / a.two_dx, hdy = DIM == 2 ? 1.0f / a.two_dy : 1.0f;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nn; j += (int64_t)gridDim.x * blockDim.x) {
    const int I = (int)(j % a.nnx), J = (int)(j / a.nnx);
    const float r = node_residual<P>(a, I);
    const float ml = ml1(C, I % P, hdx) * (DIM == 2 ? ml1(C, J % P, hdy) : 1.0f);
    if (!CVW_SPAN(a.status, j, 1, a.lim_out)) continue;
    a.rnode[j] = r;
    a.du[j] = r / ml;
  }
}

// (M_C du) at lattice node (I, J): the consistent mass is the tensor product of the 1D
// assembled masses, so the product is a sum over the (up to two) cells containing the
// node in each direction of M1[local][b] times the nodes of that cell, x first, then y.
template <int DIM, int P>
__device__ __forceinline__ float mass_apply(const CgTables<DIM, P>& C, const float* __restrict__ du, int I, int J,
                                            int nnx, int nny, float hdx, float hdy) {
  const int ax = I % P, ay = DIM == 2 ? J % P : 0;
  const int ncx = ax == 0 ? 2 : 1, ncy = DIM == 2 ? (ay == 0 ? 2 : 1) : 1;
  float acc = 0.0f;
  for (int ky = 0; ky < ncy; ++ky) {
    // y-cell starting at lattice row J0y, node's local index ly in it
    const int ly = DIM == 2 ? (ay == 0 ? (ky == 0 ? P : 0) : ay) : 0;
    const int J0y = J - ly;
#pragma unroll
    for (int d = 0; d < (DIM == 2 ? P + 1 : 1); ++d) {
      const int Jr = DIM == 2 ? ((J0y + d) % nny + nny) % nny : 0;
      const float* rowp = du + (size_t)Jr * nnx;
      float w = 0.0f;
      for (int kx = 0; kx < ncx; ++kx) {
        const int lx = ax == 0 ? (kx == 0 ? P : 0) : ax;
        const int I0x = I - lx;
#pragma unroll
        for (int b = 0; b <= P; ++b) {
          const int i = I0x + b;  // at most p <= nnx beyond either end (two modulos instead: P3 28.5 us per step, 26.5 so)
          w = fmaf(C.M1[lx][b], rowp[i < 0 ? i + nnx : i >= nnx ? i - nnx : i], w);
        }
      }
      acc = DIM == 2 ? fmaf(C.M1[ly][d], w, acc) : w;
    }
  }
  return acc * hdx * hdy;
}

// One defect-correction sweep du_out = du_in + ML^{-1}(r - M_C du_in) (reading A12), node
// by node (1D meshes); the final sweep writes the SSP-RK3 combination (or du itself).
template <int DIM, int P>
__global__ void cg_node_sweep(const __grid_constant__ StageArgs a, const __grid_constant__ CgTables<DIM, P> C,
                              const float* __restrict__ du_in, float* __restrict__ du_out, int final_sweep) {
  const int64_t nn = (int64_t)a.nnx * (DIM == 2 ? a.nny : 1);
  const float hdx = 1.0f / a.two_dx, hdy = DIM == 2 ? 1.0f / a.two_dy : 1.0f;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nn; j += (int64_t)gridDim.x * blockDim.x) {
    if (!CVW_SPAN(a.status, j, 1, a.lim_out)) continue;  // nodal inputs, outputs and work arrays
    const int I = (int)(j % a.nnx), J = (int)(j / a.nnx);
    const float mc = mass_apply<DIM, P>(C, du_in, I, J, a.nnx, DIM == 2 ? a.nny : 1, hdx, hdy);
    const float ml = ml1(C, I % P, hdx) * (DIM == 2 ? ml1(C, J % P, hdy) : 1.0f);
    const float du = du_in[j] + (a.rnode[j] - mc) / ml;
    if (!final_sweep) {
      du_out[j] = du;
    } else if (a.mode & kModeRK) {
      float v = fmaf(a.dt, du, a.u_in[j]);
      if (a.rk_a != 0.0f) v = fmaf(a.rk_b, v - a.u_n[j], a.u_n[j]);  // plain load: u_n may alias u_out
      a.u_out[j] = v;
      if (!isfinite(v)) atomicOr(a.status, kStatNonfinite);
    } else {
      a.u_out[j] = du;
      if (!isfinite(du)) atomicOr(a.status, kStatNonfinite);
    }
  }
}

// The node phase of one 2D stage, per tile of kNdX x kNdY lattice nodes: the nodal
// assembly r and du0 = r / ML on the tile and a halo of 2p nodes, the first
// defect-correction sweep du1 = du0 + ML^{-1}(r - M_C du0) (reading A12) on the tile and a
// halo of p nodes, and the second at the tile's nodes, which writes the SSP-RK3
// combination (or du itself for a residual).  The consistent mass is the tensor product
// of the 1D assembled masses, so M_C du is applied as two passes over the window: along
// x (each node sums M1[local][b] du over the nodes of the up to two cells containing it),
// then along y.  The halo values are recomputed by every tile that needs them, in the same
// arithmetic, so neighbouring tiles agree bitwise.
// The kernel is bound by its barriers and the halo (a 32x32 tile at p = 3 forms r on 44x44 nodes):
// 32x32 tiles of 1024 threads (or 64x32 of 512, launch_cg_t) from p = 3 on, 32x16 of 512 below.
// The gathers read node rows of the cells of a mesh row, contiguous in rloc (KPP Q3 256^2 85.9 ->
// 84.4 us per step against cell by cell, both kernels).
template <int P>
__host__ __device__ constexpr int node_tile_y() { return P >= 3 ? 32 : 16; }
template <int P, int kNdX>
struct NodeLayout {
  static constexpr int kNdY = node_tile_y<P>();
  static constexpr int RX = kNdX + 4 * P, RY = kNdY + 4 * P;  // r and du0 window (halo 2p)
  static constexpr int DX = kNdX + 2 * P, DY = kNdY + 2 * P;  // du1 window (halo p)
  static constexpr size_t BYTES = sizeof(float) * (2 * RY * RX + RY * DX + DY * DX);
};

template <int P, int kNdX, int NT, int CTAS>
__global__ void __launch_bounds__(NT, CTAS)
    cg_node_stage2d(const __grid_constant__ StageArgs a, const __grid_constant__ CgTables<2, P> C) {
  using L = NodeLayout<P, kNdX>;
  constexpr int N = P + 1, kNdY = L::kNdY, RX = L::RX, RY = L::RY, DX = L::DX, DY = L::DY;
  constexpr int NO = kNdX * kNdY / NT, TR = NT / kNdX;  // output nodes of a thread, rows apart
  static_assert(NO * NT == kNdX * kNdY && TR * kNdX == NT && RX + RY <= NT, "threads of a node tile");
  extern __shared__ __align__(16) float nsm[];
  float (*sr)[RX] = reinterpret_cast<float (*)[RX]>(nsm);
  float (*sd0)[RX] = reinterpret_cast<float (*)[RX]>(nsm + RY * RX);
  float (*sd1)[DX] = reinterpret_cast<float (*)[DX]>(nsm + 2 * RY * RX);
  float* sxp = nsm + 2 * RY * RX + DY * DX;  // x-pass of M_C du0 [RY][DX], then of M_C du1 [DY][kNdX]
  __shared__ float sM1[N][N];
  // per window column rx (lattice column I0 - 2p + rx) and row ry: the offsets of the
  // local residual entries the node gathers (B: the second cell, -1 if none), the node's
  // 1D local index and its inverse 1D lumped mass
  __shared__ long long srowA[RY], srowB[RY];
  __shared__ int scolA[RX], scolB[RX], slx[RX], sly[RY];
  __shared__ float simlx[RX], simly[RY];
  const int nnx = a.nnx, nny = a.nny;
  const int I0 = blockIdx.x * kNdX, J0 = blockIdx.y * kNdY;
  const float hh = (1.0f / a.two_dx) * (1.0f / a.two_dy), k2 = a.two_dx * a.two_dy;
  if (threadIdx.x < N * N) sM1[threadIdx.x / N][threadIdx.x % N] = (&C.M1[0][0])[threadIdx.x];
  // this thread's output nodes; their RK inputs are loaded right after pdl_wait, so that their
  // latency overlaps the window (u_n may alias u_out: only this thread reads or writes
  // its nodes)
  const int tx = threadIdx.x % kNdX, ty0 = threadIdx.x / kNdX;
  const bool rk = (a.mode & kModeRK) != 0, with_un = rk && a.rk_a != 0.0f;
  float uin[NO], un[NO];
  auto own = [&](int k) { return I0 + tx < nnx && J0 + ty0 + k * TR < nny; };
  auto node = [&](int k) { return (size_t)(J0 + ty0 + k * TR) * nnx + I0 + tx; };
  // 1 / (m_l wl[l]) of 1D local index l in [0, p)
  auto iml = [&](int l) {
    float v = C.iml[0];
#pragma unroll
    for (int k = 1; k < P; ++k) v = l == k ? C.iml[k] : v;
    return v;
  };
  // A node with 1D local index 0 lies in two cells (the one before it as its local p),
  // any other in one; the nodal sum takes the cells below-left first (node_residual's order).
  if (threadIdx.x < RX) {
    const int rx = threadIdx.x, Iw = wrap_index(I0 - 2 * P + rx, nnx), i = Iw / P, aa = Iw - i * P;
    const int cx0 = aa == 0 ? (i == 0 ? a.nx - 1 : i - 1) : i;
    scolA[rx] = cx0 * N + (aa == 0 ? P : aa);
    scolB[rx] = aa == 0 ? i * N : -1;
    slx[rx] = aa;
    simlx[rx] = iml(aa);
  } else if (threadIdx.x < RX + RY) {
    const int ry = threadIdx.x - RX, Jw = wrap_index(J0 - 2 * P + ry, nny), jc = Jw / P, bb = Jw - jc * P;
    const int cy0 = bb == 0 ? (jc == 0 ? a.ny - 1 : jc - 1) : jc;
    const long long rowlen = (long long)a.nx * N;
    srowA[ry] = (cy0 * N + (bb == 0 ? P : bb)) * rowlen;
    srowB[ry] = bb == 0 ? jc * N * rowlen : -1;
    sly[ry] = bb;
    simly[ry] = iml(bb);
  }
  pdl_wait();  // everything below reads or writes what earlier kernels write
#pragma unroll
  for (int k = 0; k < NO; ++k) {
    const bool ok = own(k) && CVW_SPAN(a.status, node(k), 1, a.lim_in) && CVW_SPAN(a.status, node(k), 1, a.lim_out);
    uin[k] = ok && rk ? a.u_in[node(k)] : 0.0f;
    un[k] = ok && with_un ? a.u_n[node(k)] : 0.0f;
  }
  __syncthreads();
  // ---- r and du0 on the window: every gather of the thread in flight before the first use -----
  constexpr int NW = (RX * RY + NT - 1) / NT;
  float rv[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const int f = threadIdx.x + k * NT;
    rv[k] = 0.0f;
    if (f < RX * RY) {
      const int ry = f / RX, rx = f - ry * RX;
      const long long rA = srowA[ry], rB = srowB[ry];
      const int cA = scolA[rx], cB = scolB[rx];
      const int64_t lim = CVW_EXTENT(a, lim_cell) * (N * N);
      auto rl = [&](long long k) { return CVW_SPAN(a.status, k, 1, lim) ? a.rloc[k] : 0.0f; };
      float r = rl(rA + cA);
      if (cB >= 0) r += rl(rA + cB);
      if (rB >= 0) {
        r += rl(rB + cA);
        if (cB >= 0) r += rl(rB + cB);
      }
      rv[k] = r;
    }
  }
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const int f = threadIdx.x + k * NT;
    if (f < RX * RY) {
      const int ry = f / RX, rx = f - ry * RX;
      sr[ry][rx] = rv[k];
      sd0[ry][rx] = rv[k] * (simlx[rx] * simly[ry] * k2);
    }
  }
  __syncthreads();
  // The passes work cell by cell: a cell's p+1 nodes along the pass direction (and the p
  // nodes of the cell before it, for the node shared by both) are read once, and its p
  // outputs follow with compile-time local indices: output a of the cell sums
  // M1[a][b] over the cell's nodes, plus M1[p][b] over the previous cell's for a = 0.
  // Segment s of a line starts at the cell whose local node 0 sits at source index
  // z = out0 - a0 + s p (a0: the local index of the line's first output); the products
  // are taken in the same order as node by node, so the results are the same bits.
  auto cell_pass = [&](const float (&v)[2 * P + 1], int a) {
    float w = 0.0f;
    if (a == 0) {
#pragma unroll
      for (int b = 0; b <= P; ++b) w = fmaf(C.M1[P][b], v[b], w);
#pragma unroll
      for (int b = 0; b <= P; ++b) w = fmaf(C.M1[0][b], v[P + b], w);
    } else {
#pragma unroll
      for (int aa = 1; aa < P; ++aa)
        if (aa == a) {
#pragma unroll
          for (int b = 0; b <= P; ++b) w = fmaf(C.M1[aa][b], v[P + b], w);
        }
    }
    return w;
  };
  // ---- first sweep: x-pass over the rows of the window, columns of the du1 window ----------
  {
    constexpr int NSEG = (DX + P - 1) / P + 1;
    const int a0 = slx[P];
    for (int f = threadIdx.x; f < RY * NSEG; f += NT) {
      const int ry = f / NSEG, sg = f - ry * NSEG, z = P - a0 + sg * P;  // r-window column of node 0
      float v[2 * P + 1];
#pragma unroll
      for (int j = 0; j <= 2 * P; ++j) {
        const int col = z - P + j;
        v[j] = col >= 0 && col < RX ? sd0[ry][col] : 0.0f;
      }
#pragma unroll
      for (int a = 0; a < P; ++a) {
        const int cx = z - P + a;  // du1-window column
        if (cx >= 0 && cx < DX) sxp[ry * DX + cx] = cell_pass(v, a);
      }
    }
  }
  __syncthreads();
  // ---- first sweep: y-pass and du1 -----------------------------------------------------------
  {
    constexpr int NSEG = (DY + P - 1) / P + 1;
    const int b0 = sly[P];
    for (int f = threadIdx.x; f < DX * NSEG; f += NT) {
      const int cx = f / NSEG, sg = f - cx * NSEG, z = P - b0 + sg * P;  // r-window row of node 0
      const int rx = cx + P;
      float v[2 * P + 1];
#pragma unroll
      for (int j = 0; j <= 2 * P; ++j) {
        const int row = z - P + j;
        v[j] = row >= 0 && row < RY ? sxp[row * DX + cx] : 0.0f;
      }
#pragma unroll
      for (int a = 0; a < P; ++a) {
        const int dy = z - P + a, ry = dy + P;
        if (dy >= 0 && dy < DY) {
          const float mc = cell_pass(v, a);
          sd1[dy][cx] = sd0[ry][rx] + (sr[ry][rx] - mc * hh) * (simlx[rx] * simly[ry] * k2);
        }
      }
    }
  }
  __syncthreads();
  // ---- second sweep: x-pass over the du1 window's rows, the tile's columns ------------------
  {
    constexpr int NSEG = (kNdX + P - 1) / P + 1;
    const int a0 = slx[2 * P];
    for (int f = threadIdx.x; f < DY * NSEG; f += NT) {
      const int dy = f / NSEG, sg = f - dy * NSEG, z = P - a0 + sg * P;  // du1-window column of node 0
      float v[2 * P + 1];
#pragma unroll
      for (int j = 0; j <= 2 * P; ++j) {
        const int col = z - P + j;
        v[j] = col >= 0 && col < DX ? sd1[dy][col] : 0.0f;
      }
#pragma unroll
      for (int a = 0; a < P; ++a) {
        const int ox = z - P + a;
        if (ox >= 0 && ox < kNdX) sxp[dy * kNdX + ox] = cell_pass(v, a);
      }
    }
  }
  __syncthreads();
  pdl_launch_dependents();
  // ---- second sweep: y-pass at this thread's nodes, and the stage output --------------------
#pragma unroll
  for (int k = 0; k < NO; ++k) {
    if (!own(k)) continue;
    const size_t j = node(k);
    if (!CVW_SPAN(a.status, j, 1, a.lim_in) || !CVW_SPAN(a.status, j, 1, a.lim_out)) continue;
    const int ty = ty0 + k * TR, ay = sly[ty + 2 * P], ly0 = ay == 0 ? P : ay, dy = ty + P;
    float mc = 0.0f;
#pragma unroll
    for (int d = 0; d <= P; ++d) mc = fmaf(sM1[ly0][d], sxp[(dy - ly0 + d) * kNdX + tx], mc);
    if (ay == 0) {
#pragma unroll
      for (int d = 0; d <= P; ++d) mc = fmaf(sM1[0][d], sxp[(dy + d) * kNdX + tx], mc);
    }
    float v = sd1[dy][tx + P] + (sr[ty + 2 * P][tx + 2 * P] - mc * hh) * (simlx[tx + 2 * P] * simly[ty + 2 * P] * k2);
    if (rk) {
      v = fmaf(a.dt, v, uin[k]);
      if (with_un) v = fmaf(a.rk_b, v - un[k], un[k]);
    }
    a.u_out[j] = v;
    if (!isfinite(v)) atomicOr(a.status, kStatNonfinite);
  }
}

template <int P, int W, int NT, int CTAS>
cudaError_t launch_nodes(const StageArgs& a, const CgTables<2, P>& C, cudaStream_t s) {
  using L = NodeLayout<P, W>;
  auto kern = cg_node_stage2d<P, W, NT, CTAS>;
  if (L::BYTES > 40 * 1024) {  // (beside the static arrays)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(kern, dim3((a.nnx + W - 1) / W, (a.nny + L::kNdY - 1) / L::kNdY), dim3(NT), L::BYTES, s, a, C);
}

template <int DIM, int P, int SYS, int TX, int TY>
cudaError_t launch_cg_t(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  using Tb = DgTables<DIM, P>;
  using Cb = CgTables<DIM, P>;
  constexpr size_t smem = CgLayout<DIM, P, TX, TY>::BYTES;
  static_assert(smem <= 220 * 1024, "tile too large for shared memory");
  if (m->tables_bytes != sizeof(Tb) || m->cg_tables_bytes != sizeof(Cb)) return cudaErrorInvalidValue;
  const PackedTables<DIM, P>& T = static_cast<const Tb*>(m->tables)->pk;
  const Cb& C = *static_cast<const Cb*>(m->cg_tables);
  dim3 grid((a.nx + TX - 1) / TX, DIM == 2 ? (a.ny + TY - 1) / TY : 1);
  auto k1 = cg_stage_cells<DIM, P, SYS, TX, TY>;
  int threads = cg_block_threads<DIM, P, TX, TY>();
  // FEW: at most one block per SM, where only a block's latency counts: a warp more, so that the
  // tile's vertices take one round, and registers uncapped.  CG Q2 per step, plain / FEW: Burgers
  // 60^2 36.5 / 34.5 us, 110^2 38.4 / 37.0; on larger grids the fifth warp spills at 4 blocks per SM.
  if constexpr (DIM == 2 && P == 2) {
    if ((int64_t)grid.x * grid.y <= 152) {
      k1 = cg_stage_cells<DIM, P, SYS, TX, TY, true>;
      threads = cg_block_threads<DIM, P, TX, TY, true>();
    }
  }
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = launch_pdl(k1, grid, dim3(threads), smem, s, a, T, C);
  if (e != cudaSuccess) return e;
  if (a.mode & kModeSensorOnly) return cudaGetLastError();
  kernel_mark(m, s);
  if constexpr (DIM == 2) {
    // 32-wide tiles of 1024 threads are resident 2 per SM (2 x 152 on the chip).  From one and a half
    // such waves on, 64-wide tiles of 512 threads recompute less halo in half the waves (us per step,
    // 32 / 64 wide: KPP Q3 256^2 cells 84.7 / 82.4, 512^2 266 / 244.5, Burgers Q4 256^2 248 / 245);
    // at 324 tiles a few SMs would hold two wide ones (Q4 144^2 126.9 / 131.3).  Below p = 3 the
    // halo is thin and width gains nothing (Q1 256^2 31.4 / 31.7).
    constexpr int kNdY = node_tile_y<P>(), NT1 = 32 * kNdY;
    const int64_t tiles = (int64_t)((a.nnx + 31) / 32) * ((a.nny + kNdY - 1) / kNdY);
    const bool wide = P >= 3 && tiles > 3 * 152;
    if constexpr (P >= 3)
      e = wide ? launch_nodes<P, 64, 512, 2>(a, C, s) : launch_nodes<P, 32, NT1, 2048 / NT1>(a, C, s);
    else
      e = launch_nodes<P, 32, NT1, 2048 / NT1>(a, C, s);
    if (e != cudaSuccess) return e;
    kernel_mark(m, s);
  } else {
    const int64_t nn = m->nnode;
    const int bn = (int)((nn + 255) / 256 < 4096 ? (nn + 255) / 256 : 4096);
    cg_node_rhs<DIM, P><<<bn, 256, 0, s>>>(a, C);
    kernel_mark(m, s);
    cg_node_sweep<DIM, P><<<bn, 256, 0, s>>>(a, C, a.du, a.du2, 0);
    kernel_mark(m, s);
    cg_node_sweep<DIM, P><<<bn, 256, 0, s>>>(a, C, a.du2, nullptr, 1);
    kernel_mark(m, s);
  }
  return cudaGetLastError();
}

template <int DIM, int P>
cudaError_t launch_cg_p(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  constexpr int TX = DIM == 2 ? 16 : 128, TY = DIM == 2 ? 8 : 1;
  switch (m->desc.system) {
    case CVWENO_BURGERS: return launch_cg_t<DIM, P, CVWENO_BURGERS, TX, TY>(m, a, s);
    case CVWENO_KPP: return DIM == 2 ? launch_cg_t<DIM, P, CVWENO_KPP, TX, TY>(m, a, s) : cudaErrorNotSupported;
    case CVWENO_LINADV: return launch_cg_t<DIM, P, CVWENO_LINADV, TX, TY>(m, a, s);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace

cudaError_t launch_stage_cg(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  switch (m->dim * 10 + m->p) {
    case 11: return launch_cg_p<1, 1>(m, a, s);
    case 12: return launch_cg_p<1, 2>(m, a, s);
    case 13: return launch_cg_p<1, 3>(m, a, s);
    case 14: return launch_cg_p<1, 4>(m, a, s);
    case 21: return launch_cg_p<2, 1>(m, a, s);
    case 22: return launch_cg_p<2, 2>(m, a, s);
    case 23: return launch_cg_p<2, 3>(m, a, s);
    case 24: return launch_cg_p<2, 4>(m, a, s);
    default: return cudaErrorNotSupported;
  }
}

// CgImage<dim, p> of the mesh's nodal tables into dst (host, capacity floats); the number written.
template <int DIM, int P>
static int fill_cg_image(const void* tables, float* dst, int capacity) {
  using I = CgImage<DIM, P>;
  const CgTables<DIM, P>& C = *static_cast<const CgTables<DIM, P>*>(tables);
  if (capacity < I::FLOATS) return 0;
  for (int f = 0; f < I::FLOATS; ++f) dst[f] = 0.0f;
  for (int g = 0; g < I::NG; ++g)
    for (int m = 0; m < I::N; ++m) {
      dst[I::VX + 2 * I::MP * g + m] = C.V[m][g];
      if (DIM == 2) dst[I::VY + 2 * (I::N * g + m)] = dst[I::VY + 2 * (I::N * g + m) + 1] = C.V[m][g];
    }
  return I::FLOATS;
}

int cg_image(int dim, int p, const void* tables, float* dst, int capacity) {
  switch (dim * 10 + p) {
    case 11: return fill_cg_image<1, 1>(tables, dst, capacity);
    case 12: return fill_cg_image<1, 2>(tables, dst, capacity);
    case 13: return fill_cg_image<1, 3>(tables, dst, capacity);
    case 14: return fill_cg_image<1, 4>(tables, dst, capacity);
    case 21: return fill_cg_image<2, 1>(tables, dst, capacity);
    case 22: return fill_cg_image<2, 2>(tables, dst, capacity);
    case 23: return fill_cg_image<2, 3>(tables, dst, capacity);
    case 24: return fill_cg_image<2, 4>(tables, dst, capacity);
    default: return 0;
  }
}

}  // namespace cvw
