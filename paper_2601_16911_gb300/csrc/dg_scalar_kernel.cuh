// Fused per-stage kernel for scalar conservation laws (DG, tensor Legendre Q_p).
//
// One CTA owns a TX x TY tile of cells.  It stages the tile plus a one-cell halo of
// Legendre coefficients in shared memory and then runs every stage of the path without
// touching HBM in between:
//
//   (a)+(b) vertex phase, one thread per tile vertex: Taylor data of the (up to) four
//           cells around the vertex at that vertex (eq. taylorsol), their pointwise
//           indicators (eq. pointsnorm), Jiang-Shu weights with equal linear weights and
//           the vertex candidate t* (eq. taylorcand), gathered in the fixed slot order
//           SW, SE, NW, NE -- no atomics, so results are deterministic;
//           beside it every face of the tile once: LLF flux at its Gauss nodes,
//           projected onto the tangential modes;
//   (c)     cell phase, one thread per cell: the 2^d vertex candidates as Legendre modes
//           of the cell and in its semi-norm coordinates (Sec. 3.2 remark), Jiang-Shu
//           cell weights, the reconstruction u*, the sensor gamma_e (eq. gamma) and
//           nu_e = lambda_e h_e / (2p) (eq. lostab);
//   (e)     the faces' and the volume flux' part of the residual by sum factorisation;
//           the viscous term, in cells with linear weights as the exact stiffness form
//           of the Legendre basis;
//   (d)     in troubled cells (gamma_e < C_gamma): pointwise indicators at the Gauss nodes,
//           the dissipation-preserving weights alpha_q (eq. alphaq) and the viscous term by
//           quadrature with them;
//           M^{-1} (diagonal) and the SSP-RK3 stage combination in the epilogue.
//           Fluxes are evaluated as deviations from the flux of the cell mean (exact: a
//           constant flux has zero residual), so FP32 rounding is relative to the variation
//           within a cell, not to |f(u)|.
//
// What bounds it and why it is written in pairs: the kernel is bound by instruction issue
// and FP32 arithmetic (the working set streams through L2; KPP 1024^2 Q3 runs at 68 % of the
// issue slots, KPP 256^2 at 52 %, with only 13 warps per SM to hide latencies).  Every
// contraction runs on two-wide FMAs over mode pairs and symmetric node pairs
// (dg_packed.cuh), which took the Q3 stage from 14.6 M to 8.7 M warp instructions at 256^2.
// Per step, scalar form -> this one (GB300): KPP 256^2 Q3 81 -> 53 us, 64 Burgers meshes of
// the batch 4.66 -> 3.36 ms, linear advection 330 x 170 Q4 residual 42.8 -> 31.3 us.
//
// Code-size discipline: the loops over vertex slots, corners and node groups are rolled
// (not in 1D, where they are one to three short rounds of a latency-bound chain: CG P1 of 300
// cells 23.6 -> 23.4 us per step, P3 28.2 -> 27.7) and read their tabulations (staged in shared memory) with uniform, broadcast loads, so
// the kernel body stays within the instruction cache; only the short loops over modes are
// unrolled into registers.  All arithmetic is FP32.
#pragma once

#include "mlp_mma.cuh"
#include "stage_common.cuh"
#include "tc_tf32.cuh"

namespace cvw {

// Shared-memory layout of the tile.
// Cells (tile and halo) lie cell-major, so that a row of modes is one vector load:
//  - CHUNKED, a cell of whole 16-byte chunks (2D Q1 and Q3, 1D Q3): the chunks arrive by
//    16-byte copies in place.  The four chunks of a 2D Q3 cell are swizzled by the cell
//    index (chunk q at q ^ (h / 2 mod 4)), so that the same chunk of eight consecutive
//    cells covers all banks;
//  - otherwise (9 and 25 floats in 2D; 2, 3 and 5 in 1D) each halo row is one run of
//    cells at the phase ph[row] of its first 16-byte chunk (stage_rows16); the odd cell
//    sizes of 2D are conflict-free strides for 4-byte loads, and the row stride keeps a
//    tile row's lanes in step with the row before.
// The vertex candidates lie vertex-major in padded mode pairs, 2D Q3 swizzled alike.
// TC: the tensor-core form of the sensor (2D, p = 3, 8 x 16 tiles).  The vertex candidates
// are kept only as the split TF32 MMA operand [part][K chunk][vertex][4] (16-byte rows,
// vertex-major within a chunk), which for every corner l is a canonical operand over the
// tile's cells as it stands: the cells of a tile row (8, one core-matrix group) meet 8
// consecutive vertices, and the next tile row starts VXT vertices further on (the
// descriptor's 8-row-group stride).
template <int DIM, int P, int TX, int TY, bool TC = false>
struct TileLayout {
  using K = PackedTables<DIM, P>;
  using Img = PackedImage<DIM, P>;
  static constexpr int N = K::N, ND = K::ND, NY1 = K::NY1, MP = K::MP, NG = Img::NG, NS = ND - 1, NC = 1 << DIM;
  static constexpr int NT = TX * TY;
  static constexpr int HX = TX + 2, HY = DIM == 2 ? TY + 2 : 1, NH = HX * HY;
  static constexpr int VXT = TX + 1, VYT = DIM == 2 ? TY + 1 : 1, NVT = VXT * VYT;
  static_assert(!TC || (Img::HAS_TC && TX == 8 && NT == 128), "tensor-core form: 2D p = 3, 8 x 16 tiles");
  static constexpr bool CHUNKED = ND % 4 == 0, SWIZZLED = ND == 16, ROWS = DIM == 2 && P == 4;  // ROWS: store_rows
  static constexpr bool PADDED = false;  // cells laid out as vertex data (the CG tile)
  static constexpr int RS = CHUNKED ? HX * ND
                            : DIM == 1 ? (HX * ND + 6) / 4 * 4
                                       : TX * ND + 32 * ((2 * ND + 3 + 31) / 32);
  static constexpr int VS = SWIZZLED ? 16 : 2 * MP * NY1;         // floats of a vertex
  static constexpr int TCK = Img::TCK, TCCH = TCK / 4;            // K of the corner products, its 16-byte chunks
  static constexpr int TSA_PART = TCCH * NVT * 4;                 // floats of one part (hi or lo) of the operand
  static constexpr int OFF_C = 0;                                 // cells
  static constexpr int OFF_ST = (HY * RS + 3) / 4 * 4;            // vertices; TC: [2][TCCH][NVT][4]
  static constexpr int IMG = TC ? Img::FLOATS_ALL : Img::FLOATS;
  // stage (d), over the vertex data once every cell has its sensor: pointwise indicators
  // [ND][NT], then each node group's two sums [2][NGG][NT]
  static constexpr int NGG = DIM == 2 ? NG * NG : NG;
  static constexpr int OFF_NQ = OFF_ST, OFF_S12 = OFF_NQ + ND * NT;
  static constexpr int SCF = (ND + 2 * NGG) * NT;
  static constexpr int OFF_IMG = (OFF_ST + imax(TC ? 2 * TSA_PART : VS * NVT, SCF) + 3) / 4 * 4;  // the staged PackedImage
  static constexpr int OFF_ATC = OFF_IMG + Img::TC;               // TC: [2][NC][TCCH][TCK][4]
  // u_n of the tile's cells: CHUNKED [NT][US] (a padded stride, conflict-free for 16-byte
  // loads), otherwise [ND][NT] (ROWS tiles read u_n when they write)
  static constexpr int US = ND == 16 ? 20 : ND;
  static constexpr int OFF_UN = OFF_IMG + IMG;
  // face fluxes of the tile, projected on the tangential modes: x-faces ((TX+1) per tile
  // row), then y-faces (TX per row, TY+1 rows); then the largest wave speed at the face
  // nodes of the left/lower and of the right/upper cell
  static constexpr int NFP = DIM == 2 ? N : 1;
  static constexpr int NFX = (TX + 1) * TY, NFY = DIM == 2 ? TX * (TY + 1) : 0, NFACE = NFX + NFY;
  static constexpr int OFF_F = OFF_UN + (ROWS ? 0 : CHUNKED ? US : ND) * NT;  // [NFACE][NFP]
  static constexpr int OFF_LAM = OFF_F + NFACE * NFP;             // [2][NFACE]
  static constexpr int FLOATS = OFF_LAM + 2 * NFACE;
  static constexpr size_t BYTES = sizeof(float) * (size_t)FLOATS;
  // with the surrogate sensor: packed weights, then one 32 x 16 bf16 input block per warp
  static constexpr int OFF_MLP = (FLOATS + 3) / 4 * 4;
  static constexpr int OFF_XS = OFF_MLP + (int)(sizeof(MlpPacked) / sizeof(float));
  static constexpr size_t BYTES_MLP = sizeof(float) * (size_t)OFF_XS + (size_t)(NT / 32) * 32 * 16 * 2;

  // offset of the halo cell (hx, hy); load_cell undoes the swizzle
  static __device__ __forceinline__ int cell(const int* ph, int hx, int hy) {
    if constexpr (CHUNKED) {
      const int h = hy * HX + hx;
      return SWIZZLED ? h * 16 + ((h >> 1) & 3) * 4 : h * ND;
    } else {
      return hy * RS + ph[hy] + hx * ND;
    }
  }
  static __device__ __forceinline__ int vertex(int v) { return SWIZZLED ? v * 16 + ((v >> 1) & 3) * 4 : v * VS; }
};

// Padded mode pairs at an offset of L::vertex (vertex data, CG cells).
template <class L>
__device__ __forceinline__ void load_rows(const float* st, int off, f2 (&t)[L::NY1][L::MP]) {
  if constexpr (L::MP % 2 == 0) {
#pragma unroll
    for (int my = 0; my < L::NY1; ++my)
#pragma unroll
      for (int p = 0; p < L::MP; p += 2) {
        const float4 x = *reinterpret_cast<const float4*>(st + (L::SWIZZLED ? off ^ (4 * my) : off + 2 * (L::MP * my + p)));
        t[my][p] = mk2(x.x, x.y);
        t[my][p + 1] = mk2(x.z, x.w);
      }
  } else {
#pragma unroll
    for (int my = 0; my < L::NY1; ++my)
#pragma unroll
      for (int p = 0; p < L::MP; ++p) t[my][p] = *reinterpret_cast<const f2*>(st + off + 2 * (L::MP * my + p));
  }
}
// The coefficients of the cell at offset off, as mode pairs.
template <class L>
__device__ __forceinline__ void load_cell(const float* sc, int off, f2 (&c)[L::NY1][L::MP]) {
  constexpr int N = L::N, NY1 = L::NY1, MP = L::MP;
  if constexpr (L::PADDED) {
    load_rows<L>(sc, off, c);
  } else if constexpr (L::CHUNKED && N == 4) {
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      const float4 v = *reinterpret_cast<const float4*>(sc + (L::SWIZZLED ? off ^ (4 * my) : off));
      c[my][0] = mk2(v.x, v.y);
      c[my][1] = mk2(v.z, v.w);
    }
  } else if constexpr (L::CHUNKED) {  // 2D Q1
    const float4 v = *reinterpret_cast<const float4*>(sc + off);
    c[0][0] = mk2(v.x, v.y);
    c[NY1 - 1][0] = mk2(v.z, v.w);
  } else {
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p)
        c[my][p] = mk2(sc[off + 2 * p + N * my], 2 * p + 1 < N ? sc[off + 2 * p + 1 + N * my] : 0.0f);
  }
}

// Vertex data as mode pairs, and back.
template <class L>
__device__ __forceinline__ void load_vertex(const float* st, int v, f2 (&t)[L::NY1][L::MP]) {
  load_rows<L>(st, L::vertex(v), t);
}
template <class L>
__device__ __forceinline__ void store_vertex(float* st, int v, const f2 (&t)[L::NY1][L::MP]) {
  const int off = L::vertex(v);
  if constexpr (L::MP % 2 == 0) {
#pragma unroll
    for (int my = 0; my < L::NY1; ++my)
#pragma unroll
      for (int p = 0; p < L::MP; p += 2)
        *reinterpret_cast<float4*>(st + (L::SWIZZLED ? off ^ (4 * my) : off + 2 * (L::MP * my + p))) =
            make_float4(t[my][p].x, t[my][p].y, t[my][p + 1].x, t[my][p + 1].y);
  } else {
#pragma unroll
    for (int my = 0; my < L::NY1; ++my)
#pragma unroll
      for (int p = 0; p < L::MP; ++p) *reinterpret_cast<f2*>(st + off + 2 * (L::MP * my + p)) = t[my][p];
  }
}

// Row pairs [g][MP] of a tabulation in shared memory (8-byte rows, 16 where MP is even).
template <int MP>
__device__ __forceinline__ void load_pairs(const float* t, f2 (&b)[MP]) {
  if constexpr (MP % 2 == 0) {
#pragma unroll
    for (int p = 0; p < MP; p += 2) {
      const float4 x = *reinterpret_cast<const float4*>(t + 2 * p);
      b[p] = mk2(x.x, x.y);
      b[p + 1] = mk2(x.z, x.w);
    }
  } else {
#pragma unroll
    for (int p = 0; p < MP; ++p) b[p] = *reinterpret_cast<const f2*>(t + 2 * p);
  }
}

// Output of a 2D Q4 tile.  A thread's own 25 floats lie 25 apart in global memory, so its
// stores (and reads of u_n) would each touch a sector per lane: by rows the 256^2 Burgers
// step takes 113.5 us instead of 122.9, the 330 x 170 residual 29.6 instead of 31.4.  (At Q2
// the nine floats per thread cost less than the copy: 69 against 63 us per limited step.)
//  Its cell's slot in the tile, which no other thread reads by then, already
// has the phase of the cell's place in the array: each thread writes its result there, and
// its warp copies the tile rows of its cells as runs: out = w, or u_n + rk_b (w - u_n) where
// with_un.  off: first float of the variable.  Every lane of the warps that hold cells calls it.
template <class L, int TX, int TY>
__device__ __forceinline__ void store_rows(const StageArgs& a, const float* sc, const int* ph, int64_t off, int i0, int j0,
                                           bool with_un) {
  constexpr int ND = L::ND, RPW = 32 / TX, NCH = (TX * ND + 6) / 4;
  const int nx = a.nx, ny = a.ny, row0 = (int)(threadIdx.x / 32) * RPW, wid = min(TX, nx - i0) * ND;
  const bool vec = ((reinterpret_cast<uintptr_t>(a.u_in) | reinterpret_cast<uintptr_t>(a.u_out) |
                     (with_un ? reinterpret_cast<uintptr_t>(a.u_n) : 0)) & 15) == 0;
#pragma unroll
  for (int it = 0; it < (RPW * NCH + 31) / 32; ++it) {
    const int f = it * 32 + (threadIdx.x & 31), r = row0 + f / NCH, k = f % NCH;
    if (f >= RPW * NCH || r >= TY || j0 + r >= ny) continue;
    const int64_t g0 = off + ((int64_t)(j0 + r) * nx + i0) * ND, c = (g0 & ~(int64_t)3) + 4 * k;
    const int x0 = (int)(c - g0);  // the chunk's first float within the run
    const float* w = sc + (r + 1) * L::RS + ph[r + 1] + ND + x0;
    if (vec && x0 >= 0 && x0 + 4 <= wid) {
      if (!CVW_SPAN(a.status, c, 4, a.lim_out)) continue;
      float4 v = *reinterpret_cast<const float4*>(w);
      if (with_un) {
        const float4 n = *reinterpret_cast<const float4*>(a.u_n + c);
        v = make_float4(fmaf(a.rk_b, v.x - n.x, n.x), fmaf(a.rk_b, v.y - n.y, n.y), fmaf(a.rk_b, v.z - n.z, n.z),
                        fmaf(a.rk_b, v.w - n.w, n.w));
      }
      *reinterpret_cast<float4*>(a.u_out + c) = v;
    } else {
      for (int e = max(0, -x0); e < 4 && x0 + e < wid; ++e) {
        if (!CVW_SPAN(a.status, c + e, 1, a.lim_out)) continue;
        float v = w[e];
        if (with_un) {
          const float n = a.u_n[c + e];
          v = fmaf(a.rk_b, v - n, n);
        }
        a.u_out[c + e] = v;
      }
    }
  }
}

// Writes a 2D or 1D tile's scalar cells: by rows (store_rows) where the layout says so, each
// thread its own cell otherwise, 16 bytes at a time where it is whole chunks and the output
// aligned.  hc: the cell's slot in sc.
template <class L, int TX, int TY>
__device__ __forceinline__ void write_cell(const StageArgs& a, float* sc, const int* ph, int hc, const f2 (&c)[L::NY1][L::MP],
                                           int i0, int j0, int tx, int ty, bool active, bool with_un) {
  constexpr int N = L::N, ND = L::ND;
  auto val = [&](int m) { return (m % N) & 1 ? c[m / N][m % N / 2].y : c[m / N][m % N / 2].x; };
  if constexpr (L::ROWS) {
    if (threadIdx.x >= TX * TY) return;
    if (active) {
#pragma unroll
      for (int m = 0; m < ND; ++m) sc[hc + m] = val(m);
    }
    __syncwarp();
    store_rows<L, TX, TY>(a, sc, ph, 0, i0, j0, with_un);
  } else {
    if (!active) return;
    float* out = a.u_out + ((size_t)(L::NY1 > 1 ? j0 + ty : 0) * a.nx + i0 + tx) * ND;
    if (ND % 4 == 0 && (reinterpret_cast<uintptr_t>(a.u_out) & 15) == 0) {
#pragma unroll
      for (int q = 0; q < ND / 4; ++q)
        reinterpret_cast<float4*>(out)[q] = make_float4(val(4 * q), val(4 * q + 1), val(4 * q + 2), val(4 * q + 3));
    } else {
#pragma unroll
      for (int m = 0; m < ND; ++m) out[m] = val(m);
    }
  }
}

// Copies the packed surrogate weights into shared memory (uint4 copies; NB threads).
template <int DIM, int P, int TX, int TY, int NB = TX * TY>
__device__ __forceinline__ void stage_mlp_to_smem(const void* mlp, float* smem) {
  using L = TileLayout<DIM, P, TX, TY>;
  const uint4* src = static_cast<const uint4*>(mlp);
  uint4* dst = reinterpret_cast<uint4*>(smem + L::OFF_MLP);
  for (int i = threadIdx.x; i < (int)(sizeof(MlpPacked) / 16); i += NB) dst[i] = __ldg(src + i);
}

// Surrogate inputs of one cell (2D): per corner l, the vertex candidate's cell mean minus
// the cell mean, and its h-scaled gradient at the vertex, over ||u^e||_e + eps, clamped to
// [-8, 8].  st holds reference-coordinate Taylor data; the cell mean of the Taylor
// monomial (xi - s)^k / k! over [-1, 1] is (-s)^k 2^k / (k+1)!.
template <int P, int TX, int TY>
__device__ __forceinline__ void cell_features(const StageArgs& a, const float* st, float c0, float n0, int tx,
                                              int ty, float (&f)[kMlpIn]) {
  using L = TileLayout<2, P, TX, TY>;
  constexpr int N = L::N, MP = L::MP, VXT = L::VXT;
  float mom[N];
  {
    float v = 1.0f, fact = 1.0f;
#pragma unroll
    for (int k = 0; k < N; ++k) {  // 2^k / (k+1)!
      fact *= (float)(k + 1);
      mom[k] = v / fact;
      v *= 2.0f;
    }
  }
  const float inv_s = 1.0f / (n0 + a.eps);
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int vi = (tx + (l & 1)) + (ty + (l >> 1)) * VXT;
    const float sx = (l & 1) ? -1.0f : 1.0f, sy = (l & 2) ? -1.0f : 1.0f;
    f2 t[N][MP];
    load_vertex<L>(st, vi, t);
    float mean = 0.0f;
#pragma unroll
    for (int ky = 0; ky < N; ++ky) {
      float row = 0.0f;
#pragma unroll
      for (int kx = 0; kx < N; ++kx) {
        const float v = (kx & 1) ? t[ky][kx / 2].y * sx : t[ky][kx / 2].x;
        row = fmaf(v, mom[kx], row);
      }
      mean = fmaf(row, mom[ky] * ((ky & 1) ? sy : 1.0f), mean);
    }
    const float gx = a.h_e * a.two_dx * t[0][0].y, gy = a.h_e * a.two_dy * t[1][0].x;
    f[3 * l + 0] = fminf(8.0f, fmaxf(-8.0f, (mean - c0) * inv_s));
    f[3 * l + 1] = fminf(8.0f, fmaxf(-8.0f, gx * inv_s));
    f[3 * l + 2] = fminf(8.0f, fmaxf(-8.0f, gy * inv_s));
  }
}

// Reading S7: with the surrogate, a cell whose semi-norm is below this fraction of
// (|mean| + 1) holds rounding-level variation only; it takes gamma_e = 1 directly.
constexpr float kNearFlat = 1e-5f;

// Starts the copy of the tabulation image img (device, PackedImage<DIM, P>) into shared
// memory; it lands with the tile's first cp.async wait.  NB: threads of the block.
template <int DIM, int P, int TX, int TY, int NB = TX * TY, bool TC = false>
__device__ __forceinline__ void stage_tables_to_smem(const float* img, float* smem) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  for (int f = threadIdx.x; f < L::IMG / 4; f += NB) cp_async16(smem + L::OFF_IMG + 4 * f, img + 4 * f);
}

// Writes PackedImage<DIM, P> of T to img (one block; run once per mesh, off the stage path).
template <int DIM, int P>
__global__ void packed_image_kernel(const __grid_constant__ DgTables<DIM, P> T, float* __restrict__ img) {
  using I = PackedImage<DIM, P>;
  constexpr int N = I::N, NS = I::NS, MP = I::MP, NG = I::NG;
  for (int f = threadIdx.x; f < I::FLOATS_ALL; f += blockDim.x) {
    float v = 0.0f;
    if (f >= I::TC) {  // split corner matrix: [part][l][K chunk j][row i][e], K index 4 j + e
      constexpr int TCK = I::TCK, NC = I::NC;
      const int g = f - I::TC, part = g / (NC * TCK * TCK), r = g - part * (NC * TCK * TCK);
      const int l = r / (TCK * TCK), r2 = r - l * (TCK * TCK), j = r2 / (4 * TCK), r3 = r2 - j * (4 * TCK);
      const int i = r3 / 4, k = 4 * j + (r3 & 3);
      const float x = (i < NS && k < NS) ? (&T.A[0][0][0])[(l * NS + i) * NS + k] : 0.0f;
      const float hi = tc::tf32_rna(x);
      v = part == 0 ? hi : tc::tf32_rna(x - hi);
    } else if (f >= I::WX) {
      const int g = (f - I::WX) % NG;
      if (f < I::WY + NG) v = (f < I::WY && 2 * g == N - 1) ? 0.5f * T.w[g] : T.w[g];
    } else if (DIM == 2 && f >= I::KY) {
      const int g = (f - I::KY) / 2;
      v = (&T.Bk[0][0][0])[(g / (NG * N) * N + g / N % NG) * N + g % N];
    } else if (f >= I::KX) {
      const int g = f - I::KX, m = g % (2 * MP);
      v = m < N ? (&T.Bk[0][0][0])[(g / (2 * MP * NG) * N + g / (2 * MP) % NG) * N + m] : 0.0f;
    } else if (DIM == 2 && f >= I::BY) {
      const int g = (f - I::BY) / 2, d = g / (NG * N);
      v = d ? T.Bd[g / N % NG][g % N] : T.B[g / N % NG][g % N];
    } else {
      const int m = f % (2 * MP), g = f / (2 * MP) % NG;
      v = m < N ? (f >= I::DX ? T.Bd[g][m] : T.B[g][m]) : 0.0f;
    }
    img[f] = v;
  }
}

// Stages (a)+(b) for the tile's vertices, from the cells sc: vertex candidates t* into st,
// and (optionally) the physical vertex data to tstar_out.  NB threads of the block share
// the vertices.
template <int DIM, int P, int TX, int TY, int NB = TX * TY, bool TC = false, class L = TileLayout<DIM, P, TX, TY, TC>>
__device__ __forceinline__ void tile_vertex_phase(const StageArgs& a, const PackedTables<DIM, P>& T, const float* sc,
                                                  const int* ph, float* st, int i0, int j0, int nx, int ny) {
  constexpr int N = L::N, ND = L::ND, NY1 = L::NY1, MP = L::MP, NC = L::NC, VXT = L::VXT, NVT = L::NVT;
  const int act_x = min(TX, nx - i0), act_y = DIM == 2 ? min(TY, ny - j0) : 1;
  for (int v = threadIdx.x; v < NVT; v += NB) {
    const int va = v % VXT, vb = DIM == 2 ? v / VXT : 0;
    if (va > act_x || (DIM == 2 && vb > act_y)) continue;
    f2 acc[NY1][MP];
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) acc[my][p] = mk2(0.0f, 0.0f);
    float wsum = 0.0f;
    const int gi_w = i0 - 1 + va, gj_s = j0 - 1 + vb;
    const bool has_w = a.perx || gi_w >= 0, has_e = a.perx || gi_w + 1 < nx;
    const bool has_s = DIM == 1 || a.pery || gj_s >= 0, has_n = DIM == 1 || a.pery || gj_s + 1 < ny;
    // slots SW, SE, NW, NE: the cell right of / above the vertex touches it with its
    // left / lower corner (sign -1), the cell left of / below with its right / upper one
#pragma unroll (DIM == 1 ? NC : P <= 2 ? 2 : 1)
    for (int s = 0; s < NC; ++s) {
      const int ex = s & 1, ey = (s >> 1) & 1;
      if (!((ex ? has_e : has_w) && (ey ? has_n : has_s))) continue;
      const float sx = ex ? -1.0f : 1.0f, sy = ey ? -1.0f : 1.0f;
      f2 c[NY1][MP], t[NY1][MP];
      load_cell<L>(sc, L::cell(ph, va + ex, DIM == 2 ? vb + ey : 0), c);
      corner_taylor2<N, NY1>(c, sx, sy, t);
      f2 b2 = mk2(0.0f, 0.0f);
#pragma unroll
      for (int my = 0; my < NY1; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) b2 = fma2(mul2(T.sigma2[my][p], t[my][p]), t[my][p], b2);
      const float wt = rcp_fast(ipowf(a.eps + powq(sqrt_fast(b2.x + b2.y), a.q), a.r));
      wsum += wt;
      const f2 we = mk2(wt, wt * sx), wo = mul2(we, dup2(sy));  // t's signs sx^kx sy^ky
#pragma unroll
      for (int my = 0; my < NY1; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) acc[my][p] = fma2((my & 1) ? wo : we, t[my][p], acc[my][p]);
    }
    const f2 inv = dup2(rcp_fast(wsum));
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) acc[my][p] = mul2(acc[my][p], inv);
    auto val = [&](int k) { return (k % N) & 1 ? acc[k / N][k % N / 2].y : acc[k / N][k % N / 2].x; };
    if constexpr (TC) {
      // t*_1 .. t*_NS, zero-padded to TCK, split into TF32 hi and lo: row v of the operand
#pragma unroll
      for (int j = 0; j < L::TCCH; ++j) {
        float hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 4 * j + e + 1;
          tc::split_tf32(k < ND ? val(k < ND ? k : 0) : 0.0f, hi[e], lo[e]);
        }
        *reinterpret_cast<float4*>(st + (j * NVT + v) * 4) = make_float4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<float4*>(st + L::TSA_PART + (j * NVT + v) * 4) = make_float4(lo[0], lo[1], lo[2], lo[3]);
      }
    } else {
      store_vertex<L>(st, v, acc);
    }
    if (a.tstar_out) {
      int I = i0 + va, J = j0 + vb;
      bool own_x = (va < TX || I == nx) && I < a.vx;
      int vyn = DIM == 2 ? (a.pery ? ny : ny + 1) : 1;
      bool own_y = DIM == 1 || ((vb < TY || J == ny) && J < vyn);
      if (own_x && own_y) {
        size_t vi = (size_t)I + (size_t)a.vx * J;
        if (CVW_SPAN(a.status, vi * ND, ND, (int64_t)a.vx * vyn * ND))
#pragma unroll
          for (int k = 0; k < ND; ++k) a.tstar_out[vi * ND + k] = val(k) * T.tscale[k];
      }
    }
  }
}

// Weight of a candidate with semi-norm sqrt(b2) (eq. finalweno).
__device__ __forceinline__ float sensor_weight(const StageArgs& a, float gamma, float norm) {
  return gamma * rcp_fast(ipowf(a.eps + powq(norm, a.q), a.r));
}

// gamma_e (eq. gamma) from the semi-norm coordinates w0 of u^e and S / osum of u^{e,*}; S
// leaves as the latter's coordinates.
template <int NY1, int MP>
__device__ __forceinline__ float sensor_gamma(const StageArgs& a, const f2 (&w0)[NY1][MP], f2 (&S)[NY1][MP], float osum,
                                              float n0) {
  const f2 inv = dup2(rcp_fast(osum));
  f2 d2 = mk2(0.0f, 0.0f);
#pragma unroll
  for (int my = 0; my < NY1; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      S[my][p] = mul2(S[my][p], inv);
      const f2 df = sub2(w0[my][p], S[my][p]);
      d2 = fma2(df, df, d2);
    }
  // the limiter, the surrogate's inputs and its fallback always use the computed sensor
  const bool forced = !(a.mode & (kModeLimit | kModeFeatures));
  if (forced && a.sensor_mode == CVWENO_SENSOR_SMOOTH) return 1.0f;
  if (forced && a.sensor_mode == CVWENO_SENSOR_TROUBLED) return 0.0f;
  if (n0 <= 1e-30f) return 1.0f;
  return 1.0f - powq(fminf(1.0f, sqrt_fast(d2.x + d2.y) * rcp_fast(n0)), a.q);
}

// Stage (c) for one cell with Legendre coefficients c: the cell-vertex reconstruction
// and the sensor gamma_e (eq. gamma); n0 returns ||u^e||_e, S the semi-norm coordinates of
// u^{e,*} (dead unless the limiter reads them).
template <int DIM, int P, int TX, int TY>
__device__ __forceinline__ float cell_sensor(const StageArgs& a, const PackedTables<DIM, P>& T, const float* st,
                                             const f2 (&c)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP], int tx,
                                             int ty, float& n0,
                                             f2 (&S)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using L = TileLayout<DIM, P, TX, TY>;
  constexpr int N = L::N, NY1 = L::NY1, MP = L::MP, NC = L::NC, VXT = L::VXT;
  f2 w0[NY1][MP];
  n0 = sqrt_fast(norm_coords2<DIM, P>(T, c, w0));
  const float om0 = sensor_weight(a, 1.0f - NC * a.gamma_vertex, n0);
#pragma unroll
  for (int my = 0; my < NY1; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) S[my][p] = mul2(dup2(om0), w0[my][p]);
  float osum = om0;
#pragma unroll (DIM == 1 ? NC : P == 1 ? 2 : 1)
  for (int l = 0; l < NC; ++l) {
    const int cx = l & 1, cy = (l >> 1) & 1;
    const float gx = cx ? -1.0f : 1.0f, gy = cy ? -1.0f : 1.0f;
    f2 t[NY1][MP], v[NY1][MP];
    load_vertex<L>(st, tx + cx + (DIM == 2 ? (ty + cy) * VXT : 0), t);
    taylor_modes2<N, NY1>(t, gx, gy, v);
    // (R couples modes of equal parity only: the signs of v pass through it)
    const float b2 = norm_coords2<DIM, P>(T, v, t);
    const float om = sensor_weight(a, a.gamma_vertex, sqrt_fast(b2));
    osum += om;
    const f2 we = mk2(om, om * gx), wo = mul2(we, dup2(gy));
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) S[my][p] = fma2((my & 1) ? wo : we, t[my][p], S[my][p]);
  }
  norm_coords2<DIM, P>(T, c, w0);  // again, rather than held over the corner loop
  return sensor_gamma<NY1, MP>(a, w0, S, osum, n0);
}

// Tensor memory and completion barrier of the tensor-core form of the sensor (one
// allocation per CTA, made before the tile and freed inside it).
struct TcCtx {
  const uint32_t* slot;  // shared: TMEM base address (lane 0, first of kTcCols columns)
  uint32_t mbar;         // shared-memory address of the MMA completion mbarrier
  uint32_t* done;        // shared: warps that have read their corner products
};
constexpr uint32_t kTcCols = 64;          // 4 corners x 16 FP32 columns
constexpr uint32_t kTcPolls = 1u << 22;   // bounded wait for the corner products

// Issued by one thread once the tile's vertex candidates (the split operand) are in
// shared memory: w_l = R C_l t*_l for the four corners l of all 128 cells, into TMEM
// columns 16 l .. 16 l + 15 of the cell's lane, as A_hi B_hi + A_hi B_lo + A_lo B_hi.
template <int P, int TX, int TY>
__device__ __forceinline__ void issue_corner_products(const float* smem, const TcCtx& tcx) {
  using L = TileLayout<2, P, TX, TY, true>;
  constexpr int TCK = L::TCK, NC = L::NC;
  constexpr uint32_t ALBO = L::NVT * 16, ASBO = L::VXT * 16, APART = L::TSA_PART * 4;
  constexpr uint32_t BLBO = TCK * 16, BSBO = 8 * 16, BCORNER = TCK * TCK * 4, BPART = NC * BCORNER;
  const uint32_t id = tc::idesc_tf32(128, TCK);
  const uint32_t tsa = tc::smem_u32(smem + L::OFF_ST), atc = tc::smem_u32(smem + L::OFF_ATC);
  tc::fence_after();
  const uint32_t tmem = *tcx.slot;
#pragma unroll
  for (int l = 0; l < NC; ++l) {
    const uint32_t a0 = tsa + (((l >> 1) & 1) * L::VXT + (l & 1)) * 16, b0 = atc + l * BCORNER;
    const uint32_t d = tmem + 16 * l;
#pragma unroll
    for (int s = 0; s < TCK / 8; ++s) {
      const uint64_t ah = tc::smem_desc(a0 + 2 * s * ALBO, ALBO, ASBO);
      const uint64_t al = tc::smem_desc(a0 + APART + 2 * s * ALBO, ALBO, ASBO);
      const uint64_t bh = tc::smem_desc(b0 + 2 * s * BLBO, BLBO, BSBO);
      const uint64_t bl = tc::smem_desc(b0 + BPART + 2 * s * BLBO, BLBO, BSBO);
      tc::mma_tf32(d, ah, bh, id, s > 0);
      tc::mma_tf32(d, ah, bl, id, 1u);
      tc::mma_tf32(d, al, bh, id, 1u);
    }
  }
  tc::commit(tcx.mbar);
}

// Stage (c) as cell_sensor, with the corner products read from tensor memory
// (issue_corner_products).  Every thread of the CTA calls it (the TMEM loads are
// warp-collective), cells outside the mesh included; the last warp to have read its
// products frees the TMEM.  overlap() runs between the cell's own part and the wait for
// the tensor cores: work of the cell that does not depend on the sensor.
template <int P, int TX, int TY, class Overlap>
__device__ __forceinline__ float cell_sensor_tc(const StageArgs& a, const PackedTables<2, P>& T, const TcCtx& tcx,
                                                const f2 (&c)[PackedTables<2, P>::NY1][PackedTables<2, P>::MP],
                                                float& n0, f2 (&S)[PackedTables<2, P>::NY1][PackedTables<2, P>::MP],
                                                Overlap&& overlap) {
  using L = TileLayout<2, P, TX, TY, true>;
  constexpr int N = L::N, MP = L::MP, NC = L::NC;
  f2 w0[N][MP];
  n0 = sqrt_fast(norm_coords2<2, P>(T, c, w0));
  const float om0 = sensor_weight(a, 1.0f - NC * a.gamma_vertex, n0);
#pragma unroll
  for (int my = 0; my < N; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) S[my][p] = mul2(dup2(om0), w0[my][p]);
  float osum = om0;
  overlap();
  if (!tc::mbar_wait(tcx.mbar, 0, kTcPolls)) atomicOr(a.status, kStatTimeout);
  tc::fence_after();
  const uint32_t tmem = *tcx.slot;
  const uint32_t trow = tmem + ((threadIdx.x & ~31u) << 16);
#pragma unroll 1
  for (int l = 0; l < NC; ++l) {
    float wl[16];  // row i of the product is mode i + 1
    tc::tmem_ld16(trow + 16 * l, wl);
    auto pair = [&](int my, int p) { return mk2(my + p ? wl[2 * p + N * my - 1 < 0 ? 0 : 2 * p + N * my - 1] : 0.0f, wl[2 * p + N * my]); };
    f2 b2 = mk2(0.0f, 0.0f);
#pragma unroll
    for (int my = 0; my < N; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) b2 = fma2(pair(my, p), pair(my, p), b2);
    const float om = sensor_weight(a, a.gamma_vertex, sqrt_fast(b2.x + b2.y));
    osum += om;
#pragma unroll
    for (int my = 0; my < N; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p) S[my][p] = fma2(dup2(om), pair(my, p), S[my][p]);
  }
  // this warp is done with the TMEM; the last of the CTA's warps frees it
  tc::fence_before();
  __syncwarp();
  uint32_t arrived = 0;
  if ((threadIdx.x & 31) == 0) {
    __threadfence_block();
    arrived = atomicAdd(tcx.done, 1u);
  }
  arrived = __shfl_sync(0xffffffffu, arrived, 0);
  if (arrived == TX * TY / 32 - 1) {
    __threadfence_block();
    tc::fence_after();
    tc::tmem_dealloc(tmem, kTcCols);
  }
  return sensor_gamma<N, MP>(a, w0, S, osum, n0);
}

// Stage (e), faces: every face of the tile once (a cell-wise loop would see each interior
// face from both sides).  The LLF flux at the face's Gauss nodes minus f(ubar_l) . n, ubar_l
// the mean of the left/lower cell (of the right/upper one where the left/lower cell is
// absent at a transmissive boundary, whose ghost is the present cell's trace), projected
// onto the tangential Legendre modes: sF[face][j] = sum_q w_q P_j(xi_q) F_q.  The
// right/upper cell adds the difference of the two means' fluxes (mode 0 only).  sLam: each
// side's largest wave speed at the nodes (where lambda_e is computed).
template <int DIM, int P, int SYS, int TX, int TY, int NB = TX * TY, bool TC = false>
__device__ __forceinline__ void tile_face_phase(const StageArgs& a, const float* sc, const int* ph, const float* img,
                                                float* sF, float* sLam, int i0, int j0, int nx, int ny) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  using Img = PackedImage<DIM, P>;
  using Law = ScalarLaw<SYS, DIM>;
  constexpr int N = L::N, NY1 = L::NY1, MP = L::MP, NFX = L::NFX, NFACE = L::NFACE, NFP = L::NFP;
  const bool need_lam = !(a.lambda_const > 0.0f), need_flux = !(a.mode & kModeSensorOnly);
  // faces from the block's last thread backwards: the vertex phase's extra round falls on
  // the first warp, the face phase's on the last
#pragma unroll 1
  for (int f = NB - 1 - threadIdx.x; f < NFACE; f += NB) {
    int dirn, hx, hy;
    bool hasl, hasr;
    if (f < NFX) {
      hy = f / (TX + 1), hx = f - hy * (TX + 1);
      const int gl = i0 - 1 + hx;
      hasl = a.perx || gl >= 0;
      hasr = a.perx || gl + 1 < nx;
      if (DIM == 2) ++hy;
      dirn = 0;
    } else {
      const int g = f - NFX;
      hy = g / TX, hx = g - hy * TX + 1;
      const int gl = j0 - 1 + hy;
      hasl = a.pery || gl >= 0;
      hasr = a.pery || gl + 1 < ny;
      dirn = 1;
    }
    // traces along the face, relative to each cell's own mean, as tangential mode pairs: the
    // left/lower cell meets the face with its right/upper side, the right/upper cell with
    // its left/lower side (sign (-1)^i along the normal)
    float um[2];
    f2 tr[2][MP];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      f2 c[NY1][MP];
      load_cell<L>(sc, L::cell(ph, hx + (dirn == 0 ? side : 0), hy + (DIM == 2 && dirn == 1 ? side : 0)), c);
      um[side] = c[0][0].x;
      c[0][0].x = 0.0f;
      const float sg = side ? -1.0f : 1.0f;
      if (DIM == 1 || dirn == 0) {
        float d[2 * MP];
        d[2 * MP - 1] = 0.0f;
#pragma unroll
        for (int my = 0; my < NY1; ++my) {
          f2 s = c[my][0];
#pragma unroll
          for (int p = 1; p < MP; ++p) s = add2(s, c[my][p]);
          d[my] = fmaf(sg, s.y, s.x);
        }
#pragma unroll
        for (int p = 0; p < (DIM == 2 ? MP : 1); ++p) tr[side][p] = mk2(d[2 * p], d[2 * p + 1]);
      } else {
#pragma unroll
        for (int p = 0; p < MP; ++p) {
          f2 e = c[0][p], o = c[NY1 > 1 ? 1 : 0][p];
#pragma unroll
          for (int my = 2; my < NY1; ++my) {
            if (my & 1) o = add2(o, c[my][p]);
            else e = add2(e, c[my][p]);
          }
          tr[side][p] = fma2(dup2(sg), o, e);
        }
      }
    }
    if (!hasl) {
#pragma unroll
      for (int p = 0; p < MP; ++p) tr[0][p] = tr[1][p];
      um[0] = um[1];
    }
    if (!hasr) {
#pragma unroll
      for (int p = 0; p < MP; ++p) tr[1][p] = tr[0][p];
      um[1] = um[0];
    }
    const Law law(a, um[0]);
    const float dm = um[1] - um[0];
    float laml = 0.0f, lamr = 0.0f;
    if constexpr (DIM == 1) {
      const float vl = tr[0][0].x, vr = tr[1][0].x;
      if (need_lam) laml = law.speed(um[0] + vl), lamr = law.speed(um[1] + vr);
      if (need_flux) sF[f] = llf_dev(law, a, um[0], vl, dm + vr, 0);
    } else {
      f2 h[MP];
#pragma unroll
      for (int p = 0; p < MP; ++p) h[p] = mk2(0.0f, 0.0f);
#pragma unroll 1
      for (int g = 0; g < L::NG; ++g) {
        f2 b[MP];
        load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
        f2 sl = mul2(b[0], tr[0][0]), sr = mul2(b[0], tr[1][0]);
#pragma unroll
        for (int p = 1; p < MP; ++p) {
          sl = fma2(b[p], tr[0][p], sl);
          sr = fma2(b[p], tr[1][p], sr);
        }
        const f2 vl = mk2(sl.x + sl.y, sl.x - sl.y), vr = mk2(sr.x + sr.y, sr.x - sr.y);
        if (need_lam) {
          laml = fmaxf(laml, fmaxf(law.speed(um[0] + vl.x), law.speed(um[0] + vl.y)));
          lamr = fmaxf(lamr, fmaxf(law.speed(um[1] + vr.x), law.speed(um[1] + vr.y)));
        }
        if (need_flux) {
          const f2 F = mul2(dup2(img[Img::WX + g]), llf_dev2(law, a, um[0], vl, add2(dup2(dm), vr), dirn));
          const f2 sd = mk2(F.x + F.y, F.x - F.y);
#pragma unroll
          for (int p = 0; p < MP; ++p) h[p] = fma2(b[p], sd, h[p]);
        }
      }
      if (need_flux) {
        if constexpr (N == 4) {
          *reinterpret_cast<float4*>(sF + f * NFP) = make_float4(h[0].x, h[0].y, h[MP - 1].x, h[MP - 1].y);
        } else if constexpr (N == 2) {
          *reinterpret_cast<f2*>(sF + f * NFP) = h[0];
        } else {
#pragma unroll
          for (int j = 0; j < N; ++j) sF[f * NFP + j] = (j & 1) ? h[j / 2].y : h[j / 2].x;
        }
      }
    }
    if (need_lam) {
      sLam[f] = laml;
      sLam[NFACE + f] = lamr;
    }
  }
}

// The faces of cell (tx, ty): index of its right, left, top, bottom face.
template <class L, int TX>
__device__ __forceinline__ int cell_face(int k, int tx, int ty) {
  const int up = (k & 1) == 0;
  return k < 2 ? ty * (TX + 1) + tx + up : L::NFX + (ty + up) * TX + tx;
}

// Stage (e), the faces' part of a cell's residual from the tile's face phase (sF): a lower
// face (left/bottom) was projected relative to the neighbour's mean, so this cell adds
// f(ubar_nb) - f(ubar) (mode 0: the integral of P_j over the face is 2 delta_j0) where that
// neighbour is present.  r is set.
template <int DIM, int P, int SYS, int TX, int TY, bool TC>
__device__ __forceinline__ void face_residual(const StageArgs& a, const ScalarLaw<SYS, DIM>& law, const float* smem,
                                              float ml, float mb, float ubar, int tx, int ty, int gi, int gj,
                                              f2 (&r)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  constexpr int N = L::N, MP = L::MP, NFP = L::NFP;
  const float* sF = smem + L::OFF_F;
  if constexpr (DIM == 1) {
    const bool hasL = a.perx || gi > 0;
    const float FR = sF[tx + 1];
    const float FL = sF[tx] + (hasL ? law.flux_dev_dir(ml - ubar, 0) : 0.0f);
    // r[m] = -2/dx (FR - (-1)^m FL)
    const f2 v = mk2(-a.two_dx * (FR - FL), -a.two_dx * (FR + FL));
#pragma unroll
    for (int p = 0; p < MP; ++p) r[0][p] = v;
  } else {
    float h[4][N];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float* src = sF + cell_face<L, TX>(k, tx, ty) * NFP;
      if constexpr (N == 4) {
        const float4 x = *reinterpret_cast<const float4*>(src);
        h[k][0] = x.x, h[k][1] = x.y, h[k][2] = x.z, h[k][N - 1] = x.w;
      } else if constexpr (N == 2) {
        const f2 x = *reinterpret_cast<const f2*>(src);
        h[k][0] = x.x, h[k][1] = x.y;
      } else {
#pragma unroll
        for (int j = 0; j < N; ++j) h[k][j] = src[j];
      }
    }
    if (a.perx || gi > 0) h[1][0] = fmaf(2.0f, law.flux_dev_dir(ml - ubar, 0), h[1][0]);
    if (a.pery || gj > 0) h[3][0] = fmaf(2.0f, law.flux_dev_dir(mb - ubar, 1), h[3][0]);
    // r[mx,my] = -2/dx (hR[my] - (-1)^mx hL[my]) - 2/dy (hT[mx] - (-1)^my hB[mx])
    f2 ve[MP], vo[MP];
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      const int q = 2 * p + 1 < N ? 2 * p + 1 : 0;
      const f2 T = mk2(h[2][2 * p], h[2][q]), B = mk2(h[3][2 * p], h[3][q]);
      ve[p] = mul2(dup2(a.two_dy), sub2(B, T));
      vo[p] = mul2(dup2(-a.two_dy), add2(B, T));
    }
#pragma unroll
    for (int my = 0; my < N; ++my) {
      const f2 x = mk2(-a.two_dx * (h[0][my] - h[1][my]), -a.two_dx * (h[0][my] + h[1][my]));
#pragma unroll
      for (int p = 0; p < MP; ++p) r[my][p] = add2(x, (my & 1) ? vo[p] : ve[p]);
    }
  }
}

// Reference gradient at the four nodes (+-xi, +-eta_h) from the x-contractions tb (values) and
// td (x-derivatives): (a) at +eta_h, (b) at -eta_h.
template <int N, int MP>
__device__ __forceinline__ void node_gradient(const float* yb, const float* yd, const f2 (&tb)[N], const f2 (&td)[N],
                                              f2& xa, f2& xb, f2& ya, f2& yy) {
  f2 by[N], dy[N];
  load_pairs<N>(yb, by);
  load_pairs<N>(yd, dy);
  f2 e = mul2(by[0], td[0]), o = mul2(by[1], td[1]), ye = mk2(0.0f, 0.0f), yo = mul2(dy[1], tb[1]);
#pragma unroll
  for (int my = 2; my < N; ++my) {
    if (my & 1) {
      o = fma2(by[my], td[my], o);
      yo = fma2(dy[my], tb[my], yo);
    } else {
      e = fma2(by[my], td[my], e);
      ye = fma2(dy[my], tb[my], ye);
    }
  }
  xa = add2(e, o);
  xb = sub2(e, o);
  ya = add2(yo, ye);
  yy = sub2(yo, ye);
}

// Values at the node rows +-eta_h (a, b) of x-contractions t.
template <int N>
__device__ __forceinline__ void node_rows(const float* yb, const f2 (&t)[N], f2& a, f2& b) {
  f2 by[N];
  load_pairs<N>(yb, by);
  f2 e = mul2(by[0], t[0]), o = mul2(by[1], t[1]);
#pragma unroll
  for (int my = 2; my < N; ++my) {
    if (my & 1) o = fma2(by[my], t[my], o);
    else e = fma2(by[my], t[my], e);
  }
  a = add2(e, o);
  b = sub2(e, o);
}

// Projection over y of (weighted) x fluxes fx, gx and y fluxes fy, gy at the node rows +-eta_h.
template <int N>
__device__ __forceinline__ void project_rows(const float* yb, const float* yd, f2 fx, f2 gx, f2 fy, f2 gy, f2 (&hx)[N],
                                             f2 (&hy)[N]) {
  f2 by[N], dy[N];
  load_pairs<N>(yb, by);
  load_pairs<N>(yd, dy);
  const f2 xs = add2(fx, gx), xd = sub2(fx, gx), ys = add2(fy, gy), yd2 = sub2(fy, gy);
#pragma unroll
  for (int my = 0; my < N; ++my) {
    hx[my] = fma2(by[my], (my & 1) ? xd : xs, hx[my]);
    if (my > 0) hy[my] = fma2(dy[my], (my & 1) ? ys : yd2, hy[my]);
  }
}

// max lambda_e over the volume and face Gauss nodes of a cell (modes c without the mean ubar): the
// ends +-1 are one more x group and one more row pair, whose Legendre values are all 1 (their
// corner combination is left out).
template <int DIM, int P, class Law>
__device__ __forceinline__ float cell_speed(const float* img, const Law& law, float ubar,
                                            const f2 (&c)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using Img = PackedImage<DIM, P>;
  constexpr int N = Img::N, NY1 = Img::NY1, MP = Img::MP, NG = Img::NG;
  float lam = 0.0f;
  auto take = [&](f2 d) { lam = fmaxf(lam, fmaxf(law.speed(ubar + d.x), law.speed(ubar + d.y))); };
#pragma unroll (DIM == 1 ? 4 : 1)
  for (int g = 0; g <= NG; ++g) {
    f2 b[MP], tb[NY1];
    load_pairs<MP>(img + Img::BX + 2 * MP * (g < NG ? g : 0), b);
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      f2 s = g < NG ? mul2(b[0], c[my][0]) : c[my][0];
#pragma unroll
      for (int p = 1; p < MP; ++p) s = g < NG ? fma2(b[p], c[my][p], s) : add2(c[my][p], s);
      tb[my] = mk2(s.x + s.y, s.x - s.y);
    }
    if constexpr (DIM == 1) {
      take(tb[0]);
    } else {
#pragma unroll 1
      for (int h = 0; h < (g < NG ? NG + 1 : NG); ++h) {
        f2 by[N];
        load_pairs<N>(img + Img::BY + 2 * N * (h < NG ? h : 0), by);
        f2 e = h < NG ? mul2(by[0], tb[0]) : tb[0], o = h < NG ? mul2(by[1], tb[1]) : tb[1];
#pragma unroll
        for (int my = 2; my < NY1; ++my) {
          if (my & 1) o = h < NG ? fma2(by[my], tb[my], o) : add2(tb[my], o);
          else e = h < NG ? fma2(by[my], tb[my], e) : add2(tb[my], e);
        }
        take(add2(e, o));
        take(sub2(e, o));
      }
    }
  }
  return lam;
}

// r[mx,my] += kx P_mx' hx[my] + ky P_mx hy[my] at the node pair +-xi of tables b (P) and d (P').
template <int NY1, int MP>
__device__ __forceinline__ void project_nodes(const f2 (&b)[MP], const f2 (&d)[MP], float kx, float ky, const f2 (&hx)[NY1],
                                              const f2 (&hy)[NY1], f2 (&r)[NY1][MP]) {
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    const f2 x = mul2(dup2(kx), mk2(hx[my].x - hx[my].y, hx[my].x + hx[my].y));
#pragma unroll
    for (int p = 0; p < MP; ++p) r[my][p] = fma2(d[p], x, r[my][p]);
    if (my > 0) {
      const f2 y = mul2(dup2(ky), mk2(hy[my].x + hy[my].y, hy[my].x - hy[my].y));
#pragma unroll
      for (int p = 0; p < MP; ++p) r[my][p] = fma2(b[p], y, r[my][p]);
    }
  }
}

// Volume flux of a cell (modes c without the mean ubar) into the modal residual r, by node groups:
// the four nodes (+-xi_g, +-eta_h); lambda_e over them into lam where need_lam.
template <int DIM, int P, class Law>
__device__ __forceinline__ void volume_flux(const StageArgs& a, const float* img, const Law& law, float ubar,
                                            const f2 (&c)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP], bool need_lam,
                                            bool flux, float& lam,
                                            f2 (&r)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using Img = PackedImage<DIM, P>;
  constexpr int N = Img::N, NY1 = Img::NY1, MP = Img::MP, NG = Img::NG, NGY = DIM == 2 ? NG : 1;
#pragma unroll (DIM == 1 ? 3 : 1)
  for (int g = 0; g < NG; ++g) {
    f2 b[MP], tb[NY1];
    load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      f2 s = mul2(b[0], c[my][0]);
#pragma unroll
      for (int p = 1; p < MP; ++p) s = fma2(b[p], c[my][p], s);
      tb[my] = mk2(s.x + s.y, s.x - s.y);
    }
    f2 hx[NY1], hy[NY1];
    if constexpr (DIM == 1) {
      if (need_lam) lam = fmaxf(lam, fmaxf(law.speed(ubar + tb[0].x), law.speed(ubar + tb[0].y)));
      f2 fy;
      law.flux_dev2(tb[0], hx[0], fy);
    } else {
#pragma unroll
      for (int my = 0; my < NY1; ++my) hx[my] = hy[my] = mk2(0.0f, 0.0f);
#pragma unroll 1
      for (int h = 0; h < NGY; ++h) {
        f2 by[N];
        load_pairs<N>(img + Img::BY + 2 * N * h, by);
        f2 e = mul2(by[0], tb[0]), o = mul2(by[1], tb[NY1 > 1 ? 1 : 0]);
#pragma unroll
        for (int my = 2; my < NY1; ++my) {
          if (my & 1) o = fma2(by[my], tb[my], o);
          else e = fma2(by[my], tb[my], e);
        }
        const bool mid = (N & 1) && h == NG - 1;  // the middle row: one row only
        const f2 ua = add2(e, o), ub = sub2(e, o);
        if (need_lam) {
          lam = fmaxf(lam, fmaxf(law.speed(ubar + ua.x), law.speed(ubar + ua.y)));
          lam = fmaxf(lam, fmaxf(law.speed(ubar + ub.x), law.speed(ubar + ub.y)));
        }
        if (!flux) continue;
        f2 fx, fy, gx = mk2(0.0f, 0.0f), gy = mk2(0.0f, 0.0f);
        law.flux_dev2(ua, fx, fy);
        if (!mid) law.flux_dev2(ub, gx, gy);
        const f2 w = dup2(img[Img::WY + h]);
        const f2 xs = mul2(w, add2(fx, gx)), xd = mul2(w, sub2(fx, gx));
        const f2 ys = mul2(w, add2(fy, gy)), yd = mul2(w, sub2(fy, gy));
        f2 dy[N];
        load_pairs<N>(img + Img::DY + 2 * N * h, dy);
#pragma unroll
        for (int my = 0; my < NY1; ++my) {
          hx[my] = fma2(by[my], (my & 1) ? xd : xs, hx[my]);
          if (my > 0) hy[my] = fma2(dy[my], (my & 1) ? ys : yd, hy[my]);
        }
      }
    }
    if (!flux) continue;
    f2 d[MP];
    load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
    project_nodes<NY1, MP>(b, d, a.two_dx * img[Img::WX + g], a.two_dy * img[Img::WX + g], hx, hy, r);
  }
}

// The viscous term with linear weights: the stiffness form of the Legendre basis, which the
// Gauss rule integrates exactly and which separates: the x part of mode (mx, my) is
// kx (2 / (2 my + 1)) sum_k S[mx][k] c[k, my], S[m][k] = int P_m' P_k' = min(m,k) (min(m,k) + 1)
// for m + k even (0 otherwise), and likewise in y.
template <int DIM, int N, int NY1, int MP>
__device__ __forceinline__ void add_stiffness(float kx, float ky, const f2 (&c)[NY1][MP], f2 (&r)[NY1][MP]) {
  auto S = [](int m, int k) { const int mn = m < k ? m : k; return (float)(mn * (mn + 1)); };
#pragma unroll
  for (int my = 0; my < NY1; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      f2 sx = mul2(mk2(S(2 * p, 0), S(2 * p + 1, 1)), c[my][0]);
#pragma unroll
      for (int q = 1; q < MP; ++q) sx = fma2(mk2(S(2 * p, 2 * q), S(2 * p + 1, 2 * q + 1)), c[my][q], sx);
      r[my][p] = fma2(dup2(DIM == 2 ? kx * (2.0f / (2 * my + 1)) : kx), sx, r[my][p]);
      if (DIM == 2 && my > 0) {
        f2 sy = mk2(0.0f, 0.0f);
#pragma unroll
        for (int k = 2 - (my & 1); k < NY1; k += 2) sy = fma2(dup2(S(my, k)), c[k][p], sy);
        r[my][p] = fma2(mul2(dup2(ky), mk2(2.0f / (4 * p + 1), 2.0f / (4 * p + 3))), sy, r[my][p]);
      }
    }
}

// The alpha-weighted viscous term of a 2D cell at the nodes of x group g, by quadrature: m =
// -mu afac times the indicators nq[q * NT] (nodes q = qx + N qy), or m alone where linear.
template <int N, int MP, int NT>
__device__ __forceinline__ void weighted_viscous(const StageArgs& a, const float* img, const float* nq, int g, float m,
                                                 bool weights, const f2 (&c)[N][MP], f2 (&r)[N][MP]) {
  using Img = PackedImage<2, N - 1>;
  constexpr int NG = Img::NG;
  f2 b[MP], d[MP], tb[N], td[N], hx[N], hy[N];
  load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
  load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
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
    hx[my] = hy[my] = mk2(0.0f, 0.0f);
  }
#pragma unroll 1
  for (int h = 0; h < NG; ++h) {
    f2 xa, xb, ya, yb;
    node_gradient<N, MP>(img + Img::BY + 2 * N * h, img + Img::DY + 2 * N * h, tb, td, xa, xb, ya, yb);
    const bool mid = (N & 1) && h == NG - 1;
    const f2 w = dup2(m * img[Img::WY + h]);
    const float *qa = nq + (g + N * h) * NT, *qb = nq + (g + N * (N - 1 - h)) * NT;
    const f2 la = weights ? mul2(w, mk2(qa[0], qa[(N - 1 - 2 * g) * NT])) : w;
    f2 lb = weights ? mul2(w, mk2(qb[0], qb[(N - 1 - 2 * g) * NT])) : w;
    if (mid) lb = mk2(0.0f, 0.0f);
    const f2 fx = mul2(mul2(la, dup2(a.two_dx)), xa), gx = mul2(mul2(lb, dup2(a.two_dx)), xb);
    const f2 fy = mul2(mul2(la, dup2(a.two_dy)), ya), gy = mul2(mul2(lb, dup2(a.two_dy)), yb);
    const f2 xs = add2(fx, gx), xd = sub2(fx, gx), ys = add2(fy, gy), yd = sub2(fy, gy);
    f2 by[N], dy[N];
    load_pairs<N>(img + Img::BY + 2 * N * h, by);
    load_pairs<N>(img + Img::DY + 2 * N * h, dy);
#pragma unroll
    for (int my = 0; my < N; ++my) {
      hx[my] = fma2(by[my], (my & 1) ? xd : xs, hx[my]);
      if (my > 0) hy[my] = fma2(dy[my], (my & 1) ? ys : yd, hy[my]);
    }
  }
  project_nodes<N, MP>(b, d, a.two_dx * img[Img::WX + g], a.two_dy * img[Img::WX + g], hx, hy, r);
}

// Stage (d) for node group (g, h) of the cell of thread id: the pointwise indicators at its
// nodes into sNq, and the group's part of the two sums of eq. alphaq: w |grad u|^2 and
// w Nq |grad u|^2.
template <int DIM, int P, int TX, int TY, bool TC = false, class L = TileLayout<DIM, P, TX, TY, TC>>
__device__ __forceinline__ void sc_node_group(const StageArgs& a, const PackedTables<DIM, P>& T, const float* img,
                                              float* sNq, const float* sc, const int* ph, int id, int g, int h, f2& s1,
                                              f2& s2, f2* nqa = nullptr, f2* nqb = nullptr) {
  using Img = PackedImage<DIM, P>;
  constexpr int N = L::N, NT = L::NT, NY1 = L::NY1, MP = L::MP, NG = L::NG;
  f2 c[NY1][MP];
  load_cell<L>(sc, L::cell(ph, id % TX + 1, DIM == 2 ? id / TX + 1 : 0), c);
  c[0][0].x = 0.0f;
  // squares of the derivatives at the nodes, (a) at +eta_h, (b) at -eta_h: the sum of all
  // weighted by sigma, and |grad u|^2; the signs (-1)^k at the mirrored nodes drop out
  f2 na = mk2(0.0f, 0.0f), nb = na, ga = na, gb = na;
#pragma unroll (DIM == 1 ? 5 : 1)
  for (int kx = 0; kx < N; ++kx) {
    f2 b[MP], X[NY1];
    load_pairs<MP>(img + Img::KX + 2 * MP * (kx * NG + g), b);
#pragma unroll
    for (int my = 0; my < NY1; ++my) {
      f2 s = mul2(b[0], c[my][0]);
#pragma unroll
      for (int p = 1; p < MP; ++p) s = fma2(b[p], c[my][p], s);
      X[my] = mk2(s.x + s.y, s.x - s.y);
    }
#pragma unroll
    for (int ky = 0; ky < NY1; ++ky) {
      f2 e = X[0], o = mk2(0.0f, 0.0f);
      if constexpr (DIM == 2) {
        f2 by[N];
        load_pairs<N>(img + Img::KY + 2 * N * (ky * NG + h), by);
        e = mul2(by[0], X[0]);
        o = mul2(by[1], X[NY1 > 1 ? 1 : 0]);
#pragma unroll
        for (int my = 2; my < NY1; ++my) {
          if (my & 1) o = fma2(by[my], X[my], o);
          else e = fma2(by[my], X[my], e);
        }
      }
      const f2 da = add2(e, o), db = sub2(e, o), qa = mul2(da, da), qb = mul2(db, db);
      const f2 sg = dup2(reinterpret_cast<const float*>(&T.sigma2[ky][0])[kx]);  // (zero for the value itself)
      na = fma2(sg, qa, na);
      nb = fma2(sg, qb, nb);
      if (ky < 2) {
        const f2 sq = dup2(ky == 0 ? (kx == 1 ? a.two_dx * a.two_dx : 0.0f) : kx == 0 ? a.two_dy * a.two_dy : 0.0f);
        ga = fma2(sq, qa, ga);
        gb = fma2(sq, qb, gb);
      }
    }
  }
  const f2 w = dup2(DIM == 2 ? img[Img::WX + g] * img[Img::WY + h] : img[Img::WX + g]);
  f2 nq = mk2(sqrtf(na.x), sqrtf(na.y));
  float* row = sNq + (DIM == 2 ? N * h : 0) * NT + id;
  row[g * NT] = nq.x;
  row[(N - 1 - g) * NT] = nq.y;
  if (nqa) *nqa = nq;
  s1 = mul2(w, ga);
  s2 = mul2(mul2(w, nq), ga);
  if (DIM == 2 && 2 * h != N - 1) {
    nq = mk2(sqrtf(nb.x), sqrtf(nb.y));
    row = sNq + N * (N - 1 - h) * NT + id;
    row[g * NT] = nq.x;
    row[(N - 1 - g) * NT] = nq.y;
    if (nqb) *nqb = nq;
    s1 = fma2(w, gb, s1);
    s2 = fma2(mul2(w, nq), gb, s2);
  }
}

// The state of a resident tile: cells with halo at stride ND in in[] (this stage's) and out[] (the
// next one's), and this thread's cell at the start of the step.
template <int MP>
struct Resident {
  float *in, *out;
  const int* ph;  // a zero
  f2 un[MP];
};

// One tile of one stage: the whole path (a)-(e) for the cells [i0, i0+TX) x [j0, j0+TY)
// (SURR: the instantiation that also runs the surrogate sensor and the features mode; the
// plain instantiation carries none of that code, so its registers are unaffected)
// of the mesh described by a.  Every thread must have started the staging of the
// tabulations (stage_tables_to_smem) before the call: the tile's first cp.async wait and
// barrier complete it.  The function contains its own barriers and is called by every
// thread of the CTA.  A block of NB > TX * TY threads shares the loads, the vertices and
// the faces among all of them; its threads beyond the cells sit out the per-cell stages.
// TC: the tensor-core form of stage (c) (2D, p = 3, 8 x 16 tiles; TileLayout), with the
// CTA's TMEM allocation and MMA barrier in tcx; the TMEM is freed inside the tile.
// RES: the tile's cells (and halo) are resident in shared memory (Resident), a 1D mesh of one
// tile; nothing is loaded or stored.
template <int DIM, int P, int SYS, int TX, int TY, bool SURR = false, int NB = TX * TY, bool TC = false, bool RES = false>
__device__ __forceinline__ void scalar_tile(const StageArgs& a, const PackedTables<DIM, P>& T, int i0, int j0,
                                            float* smem, TcCtx tcx = {}, Resident<(P + 2) / 2>* res = nullptr) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  using Img = PackedImage<DIM, P>;
  using Law = ScalarLaw<SYS, DIM>;
  constexpr int N = L::N, ND = L::ND, NT = L::NT, NY1 = L::NY1, MP = L::MP, NG = L::NG;
  constexpr int NGY = DIM == 2 ? NG : 1;
  constexpr int HX = L::HX, NH = L::NH, HY = L::HY;
  static_assert(!TC || (DIM == 2 && !SURR && NB == NT), "tensor-core form: plain 2D kernel, one thread per cell");
  static_assert(!RES || (DIM == 1 && !SURR && !TC), "resident tiles: plain 1D kernel");
  float* sc = smem + L::OFF_C;
  float* st = smem + L::OFF_ST;
  const float* img = smem + L::OFF_IMG;
  float* sNq = smem + L::OFF_NQ;
  if constexpr (RES) sc = res->in;

  const int nx = a.nx, ny = DIM == 2 ? a.ny : 1;

  // ---- load tile + halo: asynchronous copies in place, all of the thread's in flight -----
  // A state that is not 16-byte aligned takes 4-byte copies.
  __shared__ int ph_rows[HY];
  __shared__ int sc_count;        // troubled cells of the tile,
  __shared__ short sc_cell[NT];   // and their threads
  int* ph = ph_rows;
  if constexpr (RES) ph = const_cast<int*>(res->ph);
  if (threadIdx.x == 0) sc_count = 0;
  if constexpr (!RES) {
  const bool aligned = (reinterpret_cast<uintptr_t>(a.u_in) & 15) == 0;
  if (L::CHUNKED && aligned) {
    constexpr int NQ4 = ND / 4 > 0 ? ND / 4 : 1;
    for (int f = threadIdx.x; f < NH * NQ4; f += NB) {
      const int h = f / NQ4, q = f - h * NQ4;
      const int r = DIM == 2 ? h / HX : 0, cc = h - r * HX;
      int gi = i0 - 1 + cc, gj = DIM == 2 ? j0 - 1 + r : 0;
      bool ok = true;
      if (gi < 0 || gi >= nx) {
        if (a.perx) gi = (gi + nx) % nx; else ok = false;
      }
      if (DIM == 2 && (gj < 0 || gj >= ny)) {
        if (a.pery) gj = (gj + ny) % ny; else ok = false;
      }
      ok = ok && CVW_SPAN(a.status, ((size_t)gj * nx + gi) * ND + 4 * q, 4, a.lim_in);
      cp_async16z(sc + (L::cell(ph, cc, r) ^ (4 * q)), ok ? a.u_in + ((size_t)gj * nx + gi) * ND + 4 * q : a.u_in,
                  ok ? 16 : 0);
    }
  } else if (!L::CHUNKED && aligned) {
    if constexpr (!L::CHUNKED) {
      if (i0 > 0 && i0 + TX < nx)
        stage_rows16_inner<ND, HX, HY, L::RS, NB, 1>(sc, 0, ph, a.u_in, 0, nx, DIM == 2 ? ny : 1, i0 - 1,
                                                     DIM == 2 ? j0 - 1 : 0, DIM == 2 && a.pery, a.status,
                                                     CVW_EXTENT(a, lim_in));
      else
        stage_rows16<ND, HX, HY, L::RS, NB>(sc, ph, a.u_in, nx, DIM == 2 ? ny : 1, i0 - 1, DIM == 2 ? j0 - 1 : 0, a.perx,
                                            DIM == 2 && a.pery, a.status, CVW_EXTENT(a, lim_in));
    }
  } else {
    for (int f = threadIdx.x; f < NH * ND; f += NB) {
      const int r = DIM == 2 ? f / (HX * ND) : 0, rem = f - r * (HX * ND), cc = rem / ND, mm = rem - cc * ND;
      int gi = i0 - 1 + cc, gj = DIM == 2 ? j0 - 1 + r : 0;
      bool ok = true;
      if (gi < 0 || gi >= nx) {
        if (a.perx) gi = (gi + nx) % nx; else ok = false;
      }
      if (DIM == 2 && (gj < 0 || gj >= ny)) {
        if (a.pery) gj = (gj + ny) % ny; else ok = false;
      }
      ok = ok && CVW_SPAN(a.status, ((size_t)gj * nx + gi) * ND + mm, 1, a.lim_in);
      const int dst = L::CHUNKED ? (L::cell(ph, cc, r) ^ (mm & ~3)) + (mm & 3) : r * L::RS + cc * ND + mm;
      cp_async4(sc + dst, ok ? a.u_in + ((size_t)gj * nx + gi) * ND + mm : a.u_in, ok ? 4 : 0);
    }
    for (int r = threadIdx.x; r < HY; r += NB) ph[r] = 0;
  }
  cp_async_wait_all();
  __syncthreads();
  }  // !RES

  // u_n of the thread's own cell (RK stages 2 and 3), read only by the output: copied after
  // the halo so that it overlaps the stages below, and awaited before the output.
  // Only this thread reads u_n or writes u_out for its cell, so u_n may alias u_out.
  const bool with_un = (a.mode & kModeRK) && a.rk_a != 0.0f, pre_un = with_un && !L::ROWS && !RES;
  const bool un16 = L::CHUNKED && (reinterpret_cast<uintptr_t>(a.u_n) & 15) == 0;
  {
    const int ogi = i0 + threadIdx.x % TX, ogj = DIM == 2 ? j0 + threadIdx.x / TX : 0;
    if (pre_un && threadIdx.x < NT && ogi < nx && ogj < ny &&
        CVW_SPAN(a.status, ((size_t)ogj * nx + ogi) * ND, ND, a.lim_in)) {
      const float* src = a.u_n + ((size_t)ogj * nx + ogi) * ND;
      float* sUn = smem + L::OFF_UN;
      if (un16) {
#pragma unroll
        for (int k = 0; k < ND / 4; ++k) cp_async16(sUn + threadIdx.x * L::US + 4 * k, src + 4 * k);
      } else {
#pragma unroll 1
        for (int m = 0; m < ND; ++m) cp_async4(sUn + (L::CHUNKED ? threadIdx.x * L::US + m : m * NT + threadIdx.x), src + m, 4);
      }
    }
  }

  // ---- (a)+(b): vertex candidates of the tile's vertices; the tile's faces ----------------
  tile_vertex_phase<DIM, P, TX, TY, NB, TC>(a, T, sc, ph, st, i0, j0, nx, ny);
  const bool sensor_only = (a.mode & kModeSensorOnly) != 0, need_lam = !(a.lambda_const > 0.0f);
  if (!(a.mode & (kModeLimit | kModeFeatures)) && !(sensor_only && !need_lam))
    tile_face_phase<DIM, P, SYS, TX, TY, NB, TC>(a, sc, ph, img, smem + L::OFF_F, smem + L::OFF_LAM, i0, j0, nx, ny);
  if constexpr (TC) tc::fence_proxy_async();  // the operand, for the tensor cores
  __syncthreads();
  if constexpr (TC) {
    if (threadIdx.x == 0) issue_corner_products<P, TX, TY>(smem, tcx);
  }
  pdl_launch_dependents();

  // ---- one thread per cell from here on (the others take part in stage (d)) ------------------
  const int tx = threadIdx.x % TX, ty = DIM == 2 ? threadIdx.x / TX : 0;
  const int gi = i0 + tx, gj = DIM == 2 ? j0 + ty : 0;
  // (the checked build also checks the cell's span of u_out and its index in the per-cell
  // outputs)
  const bool active = (NB == NT || threadIdx.x < NT) && gi < nx && gj < ny && CVW_SPAN(a.status, ((size_t)gj * nx + gi) * ND, ND, a.lim_out) &&
                      CVW_SPAN(a.status, (size_t)gj * nx + gi, 1, a.lim_cell);
  // the surrogate runs warp-wide on the tensor cores: cells outside the mesh take part
  // (on the tile's zero-filled halo data); so do they in the TC form, whose TMEM loads are
  // warp-collective
  bool use_mlp = false;
  if constexpr (DIM == 2 && SURR) use_mlp = a.mlp != nullptr && !(a.mode & (kModeLimit | kModeFeatures));
  const int hc = L::cell(ph, tx + 1, DIM == 2 ? min(ty, TY - 1) + 1 : 0);
  const size_t cell = (size_t)gj * nx + gi;
  f2 c[NY1][MP];
  load_cell<L>(sc, hc, c);
  const float ubar = c[0][0].x;
  if constexpr (RES) {
    if (!with_un) {  // the step's first stage
#pragma unroll
      for (int p = 0; p < MP; ++p) res->un[p] = c[0][p];
    }
  }
  f2 r[NY1][MP];  // the residual (TC: its faces' part is taken while the tensor cores run)

  // ---- (c) cell-vertex reconstruction and sensor --------------------------------------
  float n0 = 0.0f, gam = 1.0f;
  f2 wstar[NY1][MP];
  if constexpr (DIM == 2 && SURR) {
    if (a.mode & kModeFeatures) {
      if (!active) return;
      gam = cell_sensor<DIM, P, TX, TY>(a, T, st, c, tx, ty, n0, wstar);
      float f[kMlpIn];
      cell_features<P, TX, TY>(a, st, ubar, n0, tx, ty, f);
#pragma unroll
      for (int j = 0; j < kMlpIn; ++j) a.feat_out[cell * kMlpIn + j] = f[j];
      if (a.gamma_out) a.gamma_out[cell] = gam;
      if (a.norm_out) a.norm_out[cell] = n0;
      return;
    }
    if (use_mlp && threadIdx.x < NT) {
      n0 = sqrtf(norm_coords2<DIM, P>(T, c, wstar));
      float f[kMlpIn];
      cell_features<P, TX, TY>(a, st, ubar, n0, tx, ty, f);
      float o0 = 0.0f, o1 = 0.0f;
      const bool live = active && n0 > kNearFlat * (fabsf(ubar) + 1.0f);
      const int warp = threadIdx.x >> 5;
      // a warp whose cells are all flat to rounding (S7) skips the network
      if (__any_sync(0xffffffffu, live))
        mlp_warp(*reinterpret_cast<const MlpPacked*>(smem + L::OFF_MLP), f,
                 reinterpret_cast<__nv_bfloat16*>(smem + L::OFF_XS) + warp * 32 * 16, o0, o1);
      const float conf = 1.0f / (1.0f + __expf(-o1));
      const bool fallback = live && !(conf >= a.mlp_conf_min);
      if (a.mlp_fallbacks) {  // one atomic per warp: the count of its falling-back cells
        const unsigned am = __activemask(), fm = __ballot_sync(am, fallback);
        if (fm && (threadIdx.x & 31) == (unsigned)(__ffs(am) - 1)) atomicAdd(a.mlp_fallbacks, (unsigned)__popc(fm));
      }
      if (!live) {
        gam = 1.0f;  // flat to rounding (readings A7, S7): no network, no fallback
      } else if (!fallback) {
        gam = 1.0f / (1.0f + __expf(-o0));
      } else {
        gam = cell_sensor<DIM, P, TX, TY>(a, T, st, c, tx, ty, n0, wstar);
      }
      if (a.sensor_mode == CVWENO_SENSOR_SMOOTH) gam = 1.0f;
      if (a.sensor_mode == CVWENO_SENSOR_TROUBLED) gam = 0.0f;
    } else if (active) {
      gam = cell_sensor<DIM, P, TX, TY>(a, T, st, c, tx, ty, n0, wstar);
    }
  } else if constexpr (TC) {
    const bool faces_now = active && !(a.mode & (kModeSensorOnly | kModeLimit));
    gam = cell_sensor_tc<P, TX, TY>(a, T, tcx, c, n0, wstar, [&] {
      if (faces_now)
        face_residual<DIM, P, SYS, TX, TY, TC>(a, Law(a, ubar), smem, sc[L::cell(ph, tx, ty + 1)], sc[L::cell(ph, tx + 1, ty)],
                                               ubar, tx, ty, gi, gj, r);
    });
  } else if (active) {
    gam = cell_sensor<DIM, P, TX, TY>(a, T, st, c, tx, ty, n0, wstar);
  }

  // ---- HWENO limiter (Sec. 3): u^{e,*} = mean of u^e + R^{-1} w* on the other modes ----
  if (a.mode & kModeLimit) {
    const bool lim = active && (a.limit_all || (gam < a.c_gamma && n0 > 1e-30f));
    if (lim) {
      norm_solve2<DIM, P>(T, wstar);
      f2 bad = mk2(ubar * 0.0f, 0.0f);
#pragma unroll
      for (int my = 0; my < NY1; ++my)
#pragma unroll
        for (int p = 0; p < MP; ++p) {
          bad = fma2(wstar[my][p], dup2(0.0f), bad);
          c[my][p] = wstar[my][p];
        }
      c[0][0].x = ubar;
      if (!(bad.x + bad.y == 0.0f)) atomicOr(a.status, kStatNonfinite);
    }
    if (active && a.troubled_out) a.troubled_out[cell] = lim ? 1 : 0;
    write_cell<L, TX, TY>(a, sc, ph, hc, c, i0, j0, tx, ty, active, false);
    return;
  }

  // ---- (d) troubled cells: pointwise indicators and the SC weights ---------------------------
  // Few cells are troubled, but along a front every warp has some: a thread of its own cell
  // would run the whole evaluation for a few lanes while the tile waits (KPP 256^2 Q3: a third
  // of the stage).  The tile lists its troubled cells instead, and all its threads share
  // (cell, node group) tasks; each cell then sums its groups in a fixed order.
  bool troubled = false;
  float afac = -1.0f;  // alpha_q = Nq[q] * afac where afac >= 0, else alpha_q = 1
  // means of the left and lower neighbours (after stage (d) a cell's slot is its thread's own)
  const float ml = active ? sc[L::cell(ph, tx, DIM == 2 ? ty + 1 : 0)] : 0.0f;
  const float mb = DIM == 2 && active ? sc[L::cell(ph, tx + 1, ty)] : 0.0f;
  if (!sensor_only) {
    if (active) {
      troubled = a.sc && gam < a.c_gamma && n0 > 1e-30f;
      if (a.troubled_override) {
        const int ov = a.troubled_override[cell];
        if (ov >= 0) troubled = ov && n0 > 1e-30f;
      }
    }
    const bool need_sc = troubled && gam < 1.0f;
    if (need_sc) sc_cell[atomicAdd(&sc_count, 1)] = (short)threadIdx.x;
    if (__syncthreads_or(need_sc)) {
      const int n = sc_count;
      float* sS = smem + L::OFF_S12;
#pragma unroll 1
      for (int t = threadIdx.x; t < n * L::NGG; t += NB) {
        const int gh = t / n, id = sc_cell[t - gh * n];
        f2 s1, s2;
        sc_node_group<DIM, P, TX, TY, TC>(a, T, img, sNq, sc, ph, id, gh / NGY, gh % NGY, s1, s2);
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
        if (s2 > 0.0f) afac = s1 / s2;
      }
    }
  }
  if (active) {

  // ---- (e) faces into the residual; lambda_e over the face nodes ----------------------------
  // From here on the modes without the mean: rounding stays relative to the in-cell variation.
  if (!TC) load_cell<L>(sc, hc, c);  // again, rather than held over the sensor
  c[0][0].x = 0.0f;
  const Law law(a, ubar);
  if (!TC && !sensor_only) face_residual<DIM, P, SYS, TX, TY, TC>(a, law, smem, ml, mb, ubar, tx, ty, gi, gj, r);
  float lam = need_lam ? 0.0f : a.lambda_const;
  if (need_lam) {
    const float* sLam = smem + L::OFF_LAM;
#pragma unroll
    for (int k = 0; k < 2 * DIM; ++k) lam = fmaxf(lam, sLam[((k & 1) ? L::NFACE : 0) + cell_face<L, TX>(k, tx, ty)]);
  }

  // ---- (e) volume flux, by node groups: the four nodes (+-xi_g, +-eta_h); lambda_e over them -----
  if (!sensor_only || need_lam) {
    volume_flux<DIM, P>(a, img, law, ubar, c, need_lam, !sensor_only, lam, r);
  }
  const float nu = lam * a.nu_scale;
  if (a.gamma_out) a.gamma_out[cell] = gam;
  if (a.nu_out) a.nu_out[cell] = nu;
  if (a.lambda_out) a.lambda_out[cell] = lam;
  if (sensor_only) return;

  if (a.troubled_out) a.troubled_out[cell] = troubled ? 1 : 0;
  if (a.alpha_out) {
#pragma unroll 1
    for (int q = 0; q < ND; ++q) a.alpha_out[cell * ND + q] = afac >= 0.0f ? sNq[q * NT + threadIdx.x] * afac : 1.0f;
  }

  // ---- (e) viscous term, where (1 - gamma_e) nu_e > 0 -----------------------------------------
  const float mu = (1.0f - gam) * nu;
  if (afac < 0.0f) {
    add_stiffness<DIM, N, NY1, MP>(-mu * a.two_dx * a.two_dx, -mu * a.two_dy * a.two_dy, c, r);
  } else if (mu > 0.0f) {
    if constexpr (DIM == 2) {
#pragma unroll 1
      for (int g = 0; g < NG; ++g) weighted_viscous<N, MP, NT>(a, img, sNq + threadIdx.x, g, -mu * afac, true, c, r);
    } else {
#pragma unroll 1
      for (int g = 0; g < NG; ++g) {
        f2 b[MP], d[MP];
        load_pairs<MP>(img + Img::BX + 2 * MP * g, b);
        load_pairs<MP>(img + Img::DX + 2 * MP * g, d);
        f2 s = mul2(d[0], c[0][0]);
#pragma unroll
        for (int p = 1; p < MP; ++p) s = fma2(d[p], c[0][p], s);
        const f2 al = mk2(sNq[g * NT + threadIdx.x], sNq[(N - 1 - g) * NT + threadIdx.x]);
        const f2 h[1] = {mul2(mul2(mk2(s.x + s.y, s.y - s.x), dup2(-mu * afac * a.two_dx)), al)};
        project_nodes<1, MP>(b, d, a.two_dx * img[Img::WX + g], 0.0f, h, h, r);
      }
    }
  }

  // ---- M^{-1} and the RK combination (without u_n where the rows take it) ------------------------
  const float* sUn = smem + L::OFF_UN;  // u_n of this cell
  if (pre_un) cp_async_wait_all();
  c[0][0].x = ubar;
  f2 bad = mk2(0.0f, 0.0f);  // stays zero while every du/dt is finite
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    f2 un[MP];
    if (pre_un) {
      if constexpr (L::CHUNKED && N == 4) {
        const float4 x = *reinterpret_cast<const float4*>(sUn + threadIdx.x * L::US + 4 * my);
        un[0] = mk2(x.x, x.y);
        un[MP - 1] = mk2(x.z, x.w);
      } else {
#pragma unroll
        for (int p = 0; p < MP; ++p) {
          const int m0 = 2 * p + N * my, m1 = 2 * p + 1 < N ? m0 + 1 : m0;
          un[p] = L::CHUNKED ? mk2(sUn[threadIdx.x * L::US + m0], sUn[threadIdx.x * L::US + m1])
                             : mk2(sUn[m0 * NT + threadIdx.x], sUn[m1 * NT + threadIdx.x]);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      const float ys = DIM == 2 ? 0.25f * (2 * my + 1) : 0.5f;
      f2 d = mul2(r[my][p], mk2(ys * (4 * p + 1), 2 * p + 1 < N ? ys * (4 * p + 3) : 0.0f));
      if (2 * p + 1 >= N) d.y = 0.0f;
      bad = fma2(d, dup2(0.0f), bad);
      if (a.mode & kModeRK) {
        d = fma2(dup2(a.dt), d, c[my][p]);
        if (pre_un) d = fma2(dup2(a.rk_b), sub2(d, un[p]), un[p]);
        if constexpr (RES) {
          if (with_un) d = fma2(dup2(a.rk_b), sub2(d, res->un[p]), res->un[p]);
        }
      }
      r[my][p] = d;
    }
  }
  if (!(bad.x + bad.y == 0.0f)) atomicOr(a.status, kStatNonfinite);
  }  // active
  if (sensor_only) return;
  if constexpr (RES) {
    if (!active) return;
    // the cell, and its copies in the periodic halo
#pragma unroll
    for (int m = 0; m < ND; ++m) {
      const float v = m & 1 ? r[0][m / 2].y : r[0][m / 2].x;
      res->out[(tx + 1) * ND + m] = v;
      if (a.perx && gi == 0) res->out[(nx + 1) * ND + m] = v;
      if (a.perx && gi == nx - 1) res->out[m] = v;
    }
  } else {
    write_cell<L, TX, TY>(a, sc, ph, hc, r, i0, j0, tx, ty, active, with_un);
  }
}

template <int DIM, int P, int SYS, int TX, int TY, bool SURR, int NB = TX * TY, bool TC = false>
__device__ __forceinline__ void stage_body(const StageArgs& a, const PackedTables<DIM, P>& T) {
  extern __shared__ __align__(16) float smem[];
  TcCtx tcx = {};
  if constexpr (TC) {
    // published by the tile's first barrier (after its loads)
    __shared__ uint32_t tmem_slot, tc_done;
    __shared__ uint64_t mma_bar;
    if (threadIdx.x < 32) {
      tc::tmem_alloc(&tmem_slot, kTcCols);
      tc::fence_before();
    }
    if (threadIdx.x == 0) {
      tc::mbar_init(&mma_bar, 1);
      tc_done = 0;
    }
    tcx = TcCtx{&tmem_slot, tc::smem_u32(&mma_bar), &tc_done};
  }
  stage_tables_to_smem<DIM, P, TX, TY, NB, TC>(a.pk_img, smem);  // lands with the tile's first wait
  pdl_wait();  // everything below reads or writes what earlier kernels write
  if constexpr (SURR && DIM == 2) {
    if (a.mlp) stage_mlp_to_smem<DIM, P, TX, TY, NB>(a.mlp, smem);
  }
  scalar_tile<DIM, P, SYS, TX, TY, SURR, NB, TC>(a, T, blockIdx.x * TX, DIM == 2 ? blockIdx.y * TY : 0, smem, tcx);
}

// Threads of a block of the plain stage kernel: one warp more than the tile's cells in 1D
// and up to p = 3 in 2D, so that the tile's (TX + 1) (TY + 1) vertices take one round and
// its faces two (KPP 1024^2 Q3: 0.557 ms per step with 128 threads, 0.525 with 160).  At
// p = 4 the extra warp's registers would cost a resident CTA per SM.
template <int DIM, int P, int TX, int TY>
__host__ __device__ constexpr int stage_block_threads() {
  return DIM == 1 || P <= 3 ? TX * TY + 32 : TX * TY;
}
// Resident CTAs per SM the registers must allow.  At p = 3 the kernel takes 112 registers
// uncapped (3 CTAs of 160 threads): 4 CTAs at 96 measured 53.3 us per KPP 256^2 Q3 step,
// 3 CTAs 70, 5 CTAs 73.6 (spills); at p = 4 (152 registers) 2, 3 and 4 CTAs 31.4, 31.3,
// 32.2 us per 330 x 170 residual.
template <int DIM, int P>
constexpr int stage_min_ctas() {
  return DIM == 1 ? 1 : P == 4 ? 3 : P == 1 ? 6 : 4;
}

template <int DIM, int P, int SYS, int TX, int TY>
__global__ void __launch_bounds__(stage_block_threads<DIM, P, TX, TY>(), (stage_min_ctas<DIM, P>()))
    dg_scalar_stage(const __grid_constant__ StageArgs a, const __grid_constant__ PackedTables<DIM, P> T) {
  stage_body<DIM, P, SYS, TX, TY, false, stage_block_threads<DIM, P, TX, TY>()>(a, T);
}

// The tensor-core form of the 2D Q3 stage kernel: 8 x 16 tiles, the sensor's corner
// products on tcgen05 in split TF32 (TileLayout, issue_corner_products); 4 CTAs per SM.
template <int SYS>
__global__ void __launch_bounds__(128, 4)
    dg_scalar_stage_tc(const __grid_constant__ StageArgs a, const __grid_constant__ PackedTables<2, 3> T) {
  stage_body<2, 3, SYS, 8, 16, false, 128, true>(a, T);
}

// nsteps SSP-RK3 steps of a 1D mesh that is a single tile (nx <= TX), in one launch.  The
// state stays in shared memory (two buffers with halo, a stage reads one and writes the
// other; u_n in the registers of the cell's thread) and goes back to global memory at the end;
// a block barrier stands in for the kernel boundary.  Each stage is the stage kernel's code
// with the same block, so the results are bitwise those of three launches per step.  Bound by
// the latency of one cell's chain on 5 warps: Burgers P2, 128 cells, 10 steps 57.3 us (77.9 with
// every stage's halo through global memory).
template <int P, int SYS, int TX>
__global__ void __launch_bounds__(stage_block_threads<1, P, TX, 1>())
    dg_scalar_steps_tile(const __grid_constant__ StepArgs s, const __grid_constant__ PackedTables<1, P> T) {
  constexpr int NB = stage_block_threads<1, P, TX, 1>(), ND = P + 1;
  extern __shared__ __align__(16) float smem[];
  __shared__ __align__(16) float state[2][(TX + 2) * ND + 4];
  __shared__ int zero;
  stage_tables_to_smem<1, P, TX, 1, NB>(s.st[0].pk_img, smem);
  pdl_wait();
  const StageArgs& a0 = s.st[0];
  const int nx = a0.nx;
  if (threadIdx.x == 0) zero = 0;
  for (int f = threadIdx.x; f < (nx + 2) * ND; f += NB) {
    const int h = f / ND, m = f - h * ND;
    int i = h - 1;
    bool in = true;
    if (i < 0 || i >= nx) {
      if (a0.perx) i = (i + nx) % nx; else in = false;
    }
    state[0][f] = in && CVW_SPAN(a0.status, i * ND + m, 1, a0.lim_in) ? a0.u_in[i * ND + m] : 0.0f;
    state[1][f] = 0.0f;  // (absent halo cells read as zeros)
  }
  cp_async_wait_all();
  __syncthreads();
  Resident<(P + 2) / 2> res;
  res.in = state[0];
  res.out = state[1];
  res.ph = &zero;
#pragma unroll 1
  for (int n = 0; n < s.nsteps; ++n) {
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      scalar_tile<1, P, SYS, TX, 1, false, NB, false, true>(s.st[k], T, 0, 0, smem, {}, &res);
      __syncthreads();
      float* t = res.in;
      res.in = res.out;
      res.out = t;
    }
  }
  float* u = s.st[2].u_out;
  for (int f = threadIdx.x; f < nx * ND; f += NB)
    if (CVW_SPAN(a0.status, f, 1, a0.lim_out)) u[f] = res.in[ND + f];
}

// The surrogate instantiation takes the plain kernel's block and is held to the register
// budget of 4 resident CTAs up to p = 3 and 3 at p = 4, which the network's fragments
// would otherwise exceed.
template <int DIM, int P, int SYS, int TX, int TY>
__global__ void __launch_bounds__(stage_block_threads<DIM, P, TX, TY>(), (P >= 4 ? 3 : 4) * (128 / (TX * TY)))
    dg_scalar_stage_surrogate(const __grid_constant__ StageArgs a, const __grid_constant__ PackedTables<DIM, P> T) {
  stage_body<DIM, P, SYS, TX, TY, true, stage_block_threads<DIM, P, TX, TY>()>(a, T);
}

}  // namespace cvw
