// Packed (two-wide) FP32 building blocks of the stage kernels.
//
// Why packed: sm_103a issues a scalar FP32 FMA on every second cycle of a scheduler (measured
// on the GB300 with independent chains: 70 FMA per SM and cycle), while the two-wide
// fma.rn.f32x2 reaches 120, so a contraction written in scalar FMAs runs at about half the
// rate, and twice the issue slots, of a packed one.
//
// What is paired:
//   - the Legendre modes 2i and 2i + 1 of one row (fixed my): (even, odd) in x.  A row of N
//     modes is MP = ceil(N/2) pairs, the last one padded with a zero mode when N is odd.
//     A contraction over mx then leaves its even and odd part in the two halves, which is
//     what both ends need: at a corner s = +-1 the sum is even + s odd, and at the two Gauss
//     nodes +-xi of a symmetric pair it is even + odd and even - odd.  One pair of partial
//     sums therefore serves both signs, and no sign is multiplied into the coefficients.
//   - the two Gauss nodes +-xi of a symmetric pair, once the x-contraction is done: the
//     y-contraction, the flux and the projection back run on both nodes at once, with the
//     same even/odd split over my for the two rows +-eta.  The middle node of an odd rule is
//     its own mirror image: in x it takes both halves with half its weight each, in y it
//     takes one row.
//
// What is skipped: the derivatives at a corner and the Taylor -> Legendre map are triangular
// (P_m^(k) = 0 for k > m; a monomial of degree k has no modes above k), and the semi-norm's
// Gram matrix couples only modes of equal parity in x and in y (both integrals vanish
// otherwise), so its Cholesky factor has one small triangular block per parity class.  At
// Q3 that is 80 instead of 128 products per corner transform and 36 instead of 120 per
// factor product; the four corner maps R C_l (225 products each) become two triangular
// passes of 40 and one factor product.
#pragma once

#include "cvweno_internal.cuh"

namespace cvw {

using f2 = float2;
__device__ __forceinline__ f2 mk2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }

// P_m^(k)(1) = (m + k)! / (2^k k! (m - k)!), zero for k > m.
__device__ constexpr float kCornerE[5][5] = {
    {1, 1, 1, 1, 1}, {0, 1, 3, 6, 10}, {0, 0, 3, 15, 45}, {0, 0, 0, 15, 105}, {0, 0, 0, 0, 105}};
// Legendre mode m of (xi + 1)^k / k!: (2m+1) 2^k k! / ((k-m)! (k+m+1)!), zero for m > k; about
// the other end (xi - 1) the sign is (-1)^(m+k).
__device__ constexpr float kTaylorT[5][5] = {{1.0, 1.0, 2.0 / 3, 1.0 / 3, 2.0 / 15},
                                             {0.0, 1.0, 1.0, 3.0 / 5, 4.0 / 15},
                                             {0.0, 0.0, 1.0 / 3, 1.0 / 3, 4.0 / 21},
                                             {0.0, 0.0, 0.0, 1.0 / 15, 1.0 / 15},
                                             {0.0, 0.0, 0.0, 0.0, 1.0 / 105}};

// a + e * b for a compile-time coefficient pair e (zero and unit halves are folded away by
// the callers' unrolling where both halves agree).
template <bool FIRST>
__device__ __forceinline__ f2 coef_fma(float ex, float ey, f2 v, f2 acc) {
  if (FIRST) return ex == 1.0f && ey == 1.0f ? v : mul2(mk2(ex, ey), v);
  return ex == 1.0f && ey == 1.0f ? add2(v, acc) : fma2(mk2(ex, ey), v, acc);
}

// Reference Taylor data of one cell at its corner (sx, sy), up to the signs sx^kx sy^ky (the
// caller's weights carry them): t[ky][kx] = sum E[ky][my] sy^my E[kx][mx] sx^mx c[my][mx].
template <int N, int NY1>
__device__ __forceinline__ void corner_taylor2(const f2 (&c)[NY1][(N + 1) / 2], float sx, float sy,
                                               f2 (&t)[NY1][(N + 1) / 2]) {
  constexpr int MP = (N + 1) / 2;
  f2 tmp[NY1][MP];
#pragma unroll
  for (int my = 0; my < NY1; ++my) {
    float d[2 * MP];
    d[2 * MP - 1] = 0.0f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      if (k == N - 1) {  // one mode only
        const float cm = (k & 1) ? c[my][k / 2].y * sx : c[my][k / 2].x;
        d[k] = kCornerE[k][k] * cm;
        continue;
      }
      f2 acc = mk2(0.0f, 0.0f);
#pragma unroll
      for (int p = k / 2; p < MP; ++p) {
        const float ex = kCornerE[k][2 * p], ey = 2 * p + 1 < N ? kCornerE[k][2 * p + 1] : 1.0f;  // padded mode is 0
        acc = p == k / 2 ? coef_fma<true>(ex, ey, c[my][p], acc) : coef_fma<false>(ex, ey, c[my][p], acc);
      }
      d[k] = fmaf(sx, acc.y, acc.x);
    }
#pragma unroll
    for (int p = 0; p < MP; ++p) tmp[my][p] = mk2(d[2 * p], d[2 * p + 1]);
  }
  if constexpr (NY1 == 1) {
#pragma unroll
    for (int p = 0; p < MP; ++p) t[0][p] = tmp[0][p];
  } else {
#pragma unroll
    for (int my = 1; my < NY1; my += 2)
#pragma unroll
      for (int p = 0; p < MP; ++p) tmp[my][p] = mul2(tmp[my][p], dup2(sy));
#pragma unroll
    for (int k = 0; k < NY1; ++k)
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        f2 acc = coef_fma<true>(kCornerE[k][k], kCornerE[k][k], tmp[k][p], mk2(0.0f, 0.0f));
#pragma unroll
        for (int my = k + 1; my < NY1; ++my) acc = coef_fma<false>(kCornerE[k][my], kCornerE[k][my], tmp[my][p], acc);
        t[k][p] = acc;
      }
  }
}

// Legendre modes of a vertex candidate t (Taylor data about a corner of the cell), up to the
// signs gx^mx gy^my: g = +1 where the vertex is the cell's left/lower end, -1 at the other.
// The value t[0][0].x only enters the mean, which no caller reads.
template <int N, int NY1>
__device__ __forceinline__ void taylor_modes2(const f2 (&t)[NY1][(N + 1) / 2], float gx, float gy,
                                              f2 (&v)[NY1][(N + 1) / 2]) {
  constexpr int MP = (N + 1) / 2;
  f2 tmp[NY1][MP];
#pragma unroll
  for (int ky = 0; ky < NY1; ++ky) {
    float d[2 * MP];
    d[2 * MP - 1] = 0.0f;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      if (m == N - 1) {
        d[m] = kTaylorT[m][m] * ((m & 1) ? t[ky][m / 2].y * gx : t[ky][m / 2].x);
        continue;
      }
      f2 acc = mk2(0.0f, 0.0f);
#pragma unroll
      for (int p = m / 2; p < MP; ++p) {
        const float ex = kTaylorT[m][2 * p], ey = 2 * p + 1 < N ? kTaylorT[m][2 * p + 1] : 0.0f;
        acc = p == m / 2 ? coef_fma<true>(ex, ey, t[ky][p], acc) : coef_fma<false>(ex, ey, t[ky][p], acc);
      }
      d[m] = fmaf(gx, acc.y, acc.x);
    }
#pragma unroll
    for (int p = 0; p < MP; ++p) tmp[ky][p] = mk2(d[2 * p], d[2 * p + 1]);
  }
  if constexpr (NY1 == 1) {
#pragma unroll
    for (int p = 0; p < MP; ++p) v[0][p] = tmp[0][p];
  } else {
#pragma unroll
    for (int ky = 1; ky < NY1; ky += 2)
#pragma unroll
      for (int p = 0; p < MP; ++p) tmp[ky][p] = mul2(tmp[ky][p], dup2(gy));
#pragma unroll
    for (int m = 0; m < NY1; ++m)
#pragma unroll
      for (int p = 0; p < MP; ++p) {
        f2 acc = coef_fma<true>(kTaylorT[m][m], kTaylorT[m][m], tmp[m][p], mk2(0.0f, 0.0f));
#pragma unroll
        for (int ky = m + 1; ky < NY1; ++ky) acc = coef_fma<false>(kTaylorT[m][ky], kTaylorT[m][ky], tmp[ky][p], acc);
        v[m][p] = acc;
      }
  }
}

// Semi-norm coordinates w = R v, by parity class (PackedTables::R2), and their square sum.
template <int DIM, int P>
__device__ __forceinline__ float norm_coords2(const PackedTables<DIM, P>& T, const f2 (&v)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP],
                                              f2 (&w)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using K = PackedTables<DIM, P>;
  constexpr int NY1 = K::NY1, MP = K::MP;
  f2 s = mk2(0.0f, 0.0f);
  int e = 0;
#pragma unroll
  for (int my = 0; my < NY1; ++my)
#pragma unroll
    for (int p = 0; p < MP; ++p) {
      f2 acc = mul2(T.R2[e++], v[my][p]);
#pragma unroll
      for (int qy = my; qy < NY1; qy += 2)
#pragma unroll
        for (int q = 0; q < MP; ++q) {
          if (qy == my && q <= p) continue;
          acc = fma2(T.R2[e++], v[qy][q], acc);
        }
      w[my][p] = acc;
      s = my + p == 0 ? mul2(acc, acc) : fma2(acc, acc, s);
    }
  return s.x + s.y;
}

// Modes v with R v = w (back substitution within each parity class; the mean's slot is
// left zero).
template <int DIM, int P>
__device__ __forceinline__ void norm_solve2(const PackedTables<DIM, P>& T, f2 (&w)[PackedTables<DIM, P>::NY1][PackedTables<DIM, P>::MP]) {
  using K = PackedTables<DIM, P>;
  constexpr int NY1 = K::NY1, MP = K::MP;
  int e = K::NR2;
#pragma unroll
  for (int my = NY1 - 1; my >= 0; --my)
#pragma unroll
    for (int p = MP - 1; p >= 0; --p) {
      f2 acc = w[my][p];
#pragma unroll
      for (int qy = my + (NY1 - 1 - my) / 2 * 2; qy >= my; qy -= 2)
#pragma unroll
        for (int q = MP - 1; q >= 0; --q) {
          if (qy == my && q <= p) continue;
          const f2 r = T.R2[--e];
          acc = fma2(mk2(-r.x, -r.y), w[qy][q], acc);
        }
      const f2 d = T.R2[--e];
      w[my][p] = mk2(my + p == 0 ? 0.0f : acc.x / d.x, 2 * p + 1 < K::N ? acc.y / d.y : 0.0f);
    }
}

}  // namespace cvw
