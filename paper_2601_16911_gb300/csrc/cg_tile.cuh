// Scalar (unpacked) vertex and sensor phases.
#pragma once

#include "stage_common.cuh"
#include "tc_tf32.cuh"

namespace cvw {
namespace legacy {

// Reference Taylor data t[k] = d^k u (sx, sy) at corner (sx, sy) in {-1, 1}^2 of one
// cell whose coefficients sit at c[m * stride]:
//   t[kx + N ky] = sx^kx sy^ky sum_my E[ky][my] sy^my sum_mx E[kx][mx] sx^mx c[mx, my]
// using P_m^(k)(-1) = (-1)^(m+k) P_m^(k)(1).
template <int DIM, int P>
__device__ __forceinline__ void corner_taylor(const DgTables<DIM, P>& T, const float* c, int stride, float sx, float sy,
                                              float* t) {
  constexpr int N = P + 1;
  float px[N], py[N];
  px[0] = py[0] = 1.0f;
#pragma unroll
  for (int m = 1; m < N; ++m) {
    px[m] = px[m - 1] * sx;
    py[m] = py[m - 1] * sy;
  }
  if constexpr (DIM == 1) {
    float cl[N];
#pragma unroll
    for (int m = 0; m < N; ++m) cl[m] = c[m * stride] * px[m];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      float acc = 0.0f;
#pragma unroll
      for (int m = 0; m < N; ++m) acc = fmaf(T.E[k][m], cl[m], acc);
      t[k] = acc * px[k];
    }
  } else {
    float cl[N * N];
#pragma unroll
    for (int my = 0; my < N; ++my)
#pragma unroll
      for (int mx = 0; mx < N; ++mx) cl[mx + N * my] = c[(mx + N * my) * stride] * (px[mx] * py[my]);
    float tmp[N][N];  // [kx][my]
#pragma unroll
    for (int kx = 0; kx < N; ++kx)
#pragma unroll
      for (int my = 0; my < N; ++my) {
        float acc = 0.0f;
#pragma unroll
        for (int mx = 0; mx < N; ++mx) acc = fmaf(T.E[kx][mx], cl[mx + N * my], acc);
        tmp[kx][my] = acc;
      }
#pragma unroll
    for (int ky = 0; ky < N; ++ky)
#pragma unroll
      for (int kx = 0; kx < N; ++kx) {
        float acc = 0.0f;
#pragma unroll
        for (int my = 0; my < N; ++my) acc = fmaf(T.E[ky][my], tmp[kx][my], acc);
        t[kx + N * ky] = acc * (px[kx] * py[ky]);
      }
  }
}

// Shared-memory layout of the tile: halo coefficients, vertex candidates, the corner
// matrices (rows padded to a multiple of 4 floats for 16-byte broadcast loads), the
// 1D tabulations read with run-time node indices, and per-thread alpha~ storage.
// TC: the tensor-core form of the sensor (2D, p = 3, 8 x 16 tiles).  The vertex
// candidates are kept only as the split TF32 MMA operand [part][K chunk][vertex][4]
// (16-byte rows, vertex-major within a chunk), which for every corner l is a canonical
// operand over the tile's cells as it stands: the cells of a tile row (8, one core-matrix
// group) meet 8 consecutive vertices, and the next tile row starts VXT vertices further
// on (the descriptor's 8-row-group stride).  The image is staged from B on, with its
// tensor-core section (the split corner matrices); the alpha~ storage reuses the operand
// once the MMAs have completed.
template <int DIM, int P, int TX, int TY, bool TC = false>
struct TileLayout {
  using Tb = DgTables<DIM, P>;
  static constexpr int N = P + 1, ND = Tb::ND, NS = Tb::NS, NC = Tb::NC;
  using Img = TabImage<DIM, P>;
  static constexpr int NSP = Img::NSP;
  static constexpr int NT = TX * TY;
  static constexpr int HX = TX + 2, HY = DIM == 2 ? TY + 2 : 1, NH = HX * HY;
  static constexpr int VXT = TX + 1, VYT = DIM == 2 ? TY + 1 : 1, NVT = VXT * VYT;
  static_assert(!TC || (Img::HAS_TC && TX == 8 && NT == 128), "tensor-core form: 2D p = 3, 8 x 16 tiles");
  static constexpr int TCK = Img::TCK, TCCH = TCK / 4;            // K of the corner products, its 16-byte chunks
  static constexpr int TSA_PART = TCCH * NVT * 4;                 // floats of one part (hi or lo) of the operand
  static constexpr int OFF_SC = 0;                                // [ND][NH]
  static constexpr int OFF_ST = OFF_SC + ND * NH;                 // [ND][NVT]
  static constexpr int OFF_TSA = (OFF_SC + ND * NH + 3) / 4 * 4;  // TC: [2][TCCH][NVT][4]
  // the staged TabImage (16-byte aligned): A [NC][NS][NSP], B[q][m], Bd[q][m],
  // Bk[k][q][m], w[q] (TC: from B on, then the tensor-core section); image float f sits
  // at OFF_A + f
  static constexpr int IMG0 = TC ? Img::B : 0;
  static constexpr int IMG1 = TC ? Img::FLOATS_ALL : Img::FLOATS;
  static constexpr int OFF_A = (TC ? OFF_TSA + 2 * TSA_PART : (OFF_ST + ND * NVT + 3) / 4 * 4) - IMG0;
  static constexpr int OFF_B = OFF_A + Img::B;
  static constexpr int OFF_BD = OFF_A + Img::BD;
  static constexpr int OFF_BK = OFF_A + Img::BK;
  static constexpr int OFF_W = OFF_A + Img::W;
  static constexpr int OFF_ATC = OFF_A + Img::TC;                 // TC: [2][NC][TCCH][TCK][4]
  static constexpr int OFF_NQ = TC ? OFF_TSA : OFF_A + Img::FLOATS;  // [ND][NT] pointwise indicators
  static constexpr int OFF_UN = TC ? OFF_A + IMG1 : OFF_NQ + ND * NT;  // u_n of the tile's cells, [ND][NT] or [NT][ND]
  // the tile's loads are staged over the indicator and u_n regions (TC: over the operand)
  static constexpr int STAGING = TC ? 2 * TSA_PART : 2 * ND * NT;
  static_assert(!TC || ND * NT <= 2 * TSA_PART, "alpha~ storage must fit the operand region");
  // face fluxes of the tile, projected on the tangential modes: x-faces ((TX+1) per tile
  // row), then y-faces (TX per row, TY+1 rows)
  // (degrees 2 and 3, from measurements: at p = 1 the face work per cell is too small to
  // pay for the face phase's own law evaluations and its uneven rounds before the
  // barrier; at p = 4 the batch kernel, at its register cap, lost time; the surrogate
  // instantiation at p = 2, held to 96 registers, keeps the cell-wise faces)
  static constexpr bool SHARED_FACES = P == 2 || P == 3;
  static constexpr int NFP = DIM == 2 ? N : 1;
  static constexpr int NFX = (TX + 1) * TY, NFY = DIM == 2 ? TX * (TY + 1) : 0, NFACE = NFX + NFY;
  static constexpr int OFF_F = OFF_UN + ND * NT;                  // [NFACE][NFP]
  static constexpr int FLOATS = OFF_F + (SHARED_FACES ? NFACE * NFP : 0);
  static constexpr size_t BYTES = sizeof(float) * (size_t)FLOATS;
};

// Starts the copy of the tabulation image img (device, TabImage<DIM, P>) into shared
// memory; it lands with the tile's first cp.async wait.  NB: threads of the block.
template <int DIM, int P, int TX, int TY, int NB = TX * TY, bool TC = false>
__device__ __forceinline__ void stage_tables_to_smem(const float* img, float* smem) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  for (int f = L::IMG0 / 4 + threadIdx.x; f < L::IMG1 / 4; f += NB) cp_async16(smem + L::OFF_A + 4 * f, img + 4 * f);
}

// Writes TabImage<DIM, P> of T to img (one block; run once per mesh, off the stage path).
template <int DIM, int P>
__global__ void tab_image_kernel(const __grid_constant__ DgTables<DIM, P> T, float* __restrict__ img) {
  using I = TabImage<DIM, P>;
  constexpr int N = I::N, NS = I::NS, NSP = I::NSP;
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
    } else if (f < I::B) {
      const int l = f / (NS * NSP), rem = f - l * (NS * NSP), i = rem / NSP, j = rem - i * NSP;
      v = j < NS ? T.A[l][i][j] : 0.0f;
    } else if (f < I::BD) {
      v = (&T.B[0][0])[f - I::B];
    } else if (f < I::BK) {
      v = (&T.Bd[0][0])[f - I::BD];
    } else if (f < I::W) {
      v = (&T.Bk[0][0][0])[f - I::BK];
    } else if (f < I::W + N) {
      v = T.w[f - I::W];
    }
    img[f] = v;
  }
}

// Stages (a)+(b) for the tile's vertices, from the halo coefficients sc (mode-major):
// vertex candidates t* into st, and (optionally) the physical vertex data to tstar_out.
// NB threads of the block share the vertices.
template <int DIM, int P, int TX, int TY, int NB = TX * TY, bool TC = false>
__device__ __forceinline__ void tile_vertex_phase(const StageArgs& a, const DgTables<DIM, P>& T, const float* sc,
                                                  float* st, int i0, int j0, int nx, int ny) {
  using L = TileLayout<DIM, P, TX, TY, TC>;
  constexpr int ND = L::ND, NC = L::NC, HX = L::HX, NH = L::NH, VXT = L::VXT, NVT = L::NVT;
  const int act_x = min(TX, nx - i0), act_y = DIM == 2 ? min(TY, ny - j0) : 1;
  for (int v = threadIdx.x; v < NVT; v += NB) {
    int va = v % VXT, vb = DIM == 2 ? v / VXT : 0;
    if (va > act_x || (DIM == 2 && vb > act_y)) continue;
    float acc[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) acc[k] = 0.0f;
    float wsum = 0.0f;
    const int gi_w = i0 - 1 + va, gj_s = j0 - 1 + vb;
    const bool has_w = a.perx || gi_w >= 0, has_e = a.perx || gi_w + 1 < nx;
    const bool has_s = DIM == 1 || a.pery || gj_s >= 0, has_n = DIM == 1 || a.pery || gj_s + 1 < ny;
    const float* base = sc + (DIM == 2 ? vb * HX : 0) + va;
    // slots SW, SE, NW, NE: the cell right of / above the vertex touches it with its
    // left / lower corner (sign -1), the cell left of / below with its right / upper one
#pragma unroll (DIM == 1 || P <= 2 ? NC : 1)
    for (int s = 0; s < NC; ++s) {
      const int ex = s & 1, ey = (s >> 1) & 1;
      if (!((ex ? has_e : has_w) && (ey ? has_n : has_s))) continue;
      float t[ND];
      corner_taylor<DIM, P>(T, base + ex + (DIM == 2 ? ey * HX : 0), NH, ex ? -1.0f : 1.0f, ey ? -1.0f : 1.0f, t);
      float b2 = 0.0f;
#pragma unroll
      for (int k = 1; k < ND; ++k) b2 = fmaf(T.sigma[k] * t[k], t[k], b2);
      const float wt = rcp_fast(ipowf(a.eps + powq(sqrt_fast(b2), a.q), a.r));
      wsum += wt;
#pragma unroll
      for (int k = 0; k < ND; ++k) acc[k] = fmaf(wt, t[k], acc[k]);
    }
    const float inv = rcp_fast(wsum);
    if constexpr (TC) {
      // t*_1 .. t*_NS, zero-padded to TCK, split into TF32 hi and lo: row v of the operand
#pragma unroll
      for (int j = 0; j < L::TCCH; ++j) {
        float hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 4 * j + e + 1;
          tc::split_tf32(k < ND ? acc[k < ND ? k : 0] * inv : 0.0f, hi[e], lo[e]);
        }
        *reinterpret_cast<float4*>(st + (j * NVT + v) * 4) = make_float4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<float4*>(st + L::TSA_PART + (j * NVT + v) * 4) = make_float4(lo[0], lo[1], lo[2], lo[3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < ND; ++k) st[k * NVT + v] = acc[k] * inv;
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
          for (int k = 0; k < ND; ++k) a.tstar_out[vi * ND + k] = acc[k] * inv * T.tscale[k];
      }
    }
  }
}

// Stage (c) for one cell with Legendre coefficients c: the cell-vertex reconstruction
// and the sensor gamma_e (eq. gamma); n0 returns ||u^e||_e.
template <int DIM, int P, int TX, int TY>
__device__ __forceinline__ float cell_sensor(const StageArgs& a, const DgTables<DIM, P>& T, const float* st,
                                             const float* sA, const float* c, int tx, int ty, float& n0,
                                             float* wstar) {
  using L = TileLayout<DIM, P, TX, TY>;
  constexpr int NS = L::NS, NC = L::NC, NSP = L::NSP, VXT = L::VXT, NVT = L::NVT;
  float w0[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    float acc = 0.0f;
#pragma unroll
    for (int j = i; j < NS; ++j) acc = fmaf(T.R[i][j], c[j + 1], acc);
    w0[i] = acc;
  }
  float n0sq = 0.0f;
#pragma unroll
  for (int i = 0; i < NS; ++i) n0sq = fmaf(w0[i], w0[i], n0sq);
  n0 = sqrt_fast(n0sq);
  const float om0 = (1.0f - NC * a.gamma_vertex) * rcp_fast(ipowf(a.eps + powq(n0, a.q), a.r));
  float S[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) S[i] = om0 * w0[i];
  float osum = om0;
#pragma unroll (DIM == 1 || P <= 2 ? NC : 1)
  for (int l = 0; l < NC; ++l) {
    const int vi = (tx + (l & 1)) + (DIM == 2 ? (ty + ((l >> 1) & 1)) * VXT : 0);
    float tl[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) tl[k] = k < NS ? st[(k + 1) * NVT + vi] : 0.0f;
    const float4* Al = reinterpret_cast<const float4*>(sA + l * NS * NSP);
    float wl[NS];
    float b2 = 0.0f;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      float acc = 0.0f;
#pragma unroll
      for (int j4 = 0; j4 < NSP / 4; ++j4) {
        const float4 q4 = Al[i * (NSP / 4) + j4];
        acc = fmaf(q4.x, tl[4 * j4 + 0], acc);
        acc = fmaf(q4.y, tl[4 * j4 + 1], acc);
        acc = fmaf(q4.z, tl[4 * j4 + 2], acc);
        acc = fmaf(q4.w, tl[4 * j4 + 3], acc);
      }
      wl[i] = acc;
      b2 = fmaf(acc, acc, b2);
    }
    const float om = a.gamma_vertex * rcp_fast(ipowf(a.eps + powq(sqrt_fast(b2), a.q), a.r));
    osum += om;
#pragma unroll
    for (int i = 0; i < NS; ++i) S[i] = fmaf(om, wl[i], S[i]);
  }
  const float inv = rcp_fast(osum);
  float d2 = 0.0f;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    float df = w0[i] - S[i] * inv;
    wstar[i] = S[i] * inv;  // semi-norm coordinates of u^{e,*} (dead unless the limiter reads it)
    d2 = fmaf(df, df, d2);
  }
  // the limiter, the surrogate's inputs and its fallback always use the computed sensor
  const bool forced = !(a.mode & (kModeLimit | kModeFeatures));
  if (forced && a.sensor_mode == CVWENO_SENSOR_SMOOTH) return 1.0f;
  if (forced && a.sensor_mode == CVWENO_SENSOR_TROUBLED) return 0.0f;
  if (n0 <= 1e-30f) return 1.0f;
  return 1.0f - powq(fminf(1.0f, sqrt_fast(d2) * rcp_fast(n0)), a.q);
}

}  // namespace legacy
}  // namespace cvw
