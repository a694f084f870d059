// C ABI of the cell-vertex WENO library: mesh lifecycle, stage dispatch, SSP-RK3,
// projection of analytic initial data and the FP64 reductions (conservation totals
// and CFL wave speed -- the only FP64 arithmetic on the device).
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include "cvweno_internal.cuh"

using namespace cvw;

namespace {

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 304;  // 2 x 152 SMs
constexpr int kRedOut = 4 * kRedBlocks;  // d_red: partials of up to four variables, then results [8], slots [2]
constexpr int kProjN = 12;       // projection rule points per direction

inline cudaStream_t S(void* s) { return reinterpret_cast<cudaStream_t>(s); }

inline cvweno_status cuda_status(cudaError_t e) { return e == cudaSuccess ? CVWENO_OK : CVWENO_ERR_CUDA; }

// ---- analytic initial data --------------------------------------------------------------

struct ProjTables {
  float x[kProjN];
  float wP[kProjN][kMaxP + 1];  // weight times Legendre value at the projection nodes
};

// The projection rule and its Legendre values (FP64), built once per process.
struct ProjRule {
  double x[kProjN], w[kProjN], P[kProjN][kMaxP + 1];
  bool ok;
  ProjRule() {
    static_assert(kProjN <= kMaxGaussRule, "projection rule larger than the Gauss rule builder");
    ok = gauss_rule(kProjN, x, w);
    for (int q = 0; ok && q < kProjN; ++q) legendre_values(x[q], kMaxP, P[q]);
  }
};
const ProjRule& proj_rule() {
  static const ProjRule rule;
  return rule;
}

struct ProjArgs {
  float* u;
  int nx, ny, dim, nd, n, nvar, type;
  double x0, y0, dx, dy, lx, ly, gas_gamma;
  float prm[64];
};

__device__ void prim_to_cons(float g, float rho, float vx, float vy, float p, float* U) {
  U[0] = rho;
  U[1] = rho * vx;
  U[2] = rho * vy;
  U[3] = p / (g - 1.0f) + 0.5f * rho * (vx * vx + vy * vy);
}

__device__ void ic_eval(const ProjArgs& a, float x, float y, float* U) {
  const float* P = a.prm;
  const float twopi = 6.28318530717958647692f;
  switch (a.type) {
    case CVWENO_IC_CONST:
      for (int v = 0; v < 4; ++v) U[v] = P[v];
      break;
    case CVWENO_IC_SINE_STEP:
      U[0] = P[0] * sinf(twopi * P[1] * (x - (float)a.x0) / (float)a.lx) + (x >= P[3] ? P[2] : 0.0f);
      break;
    case CVWENO_IC_CIRCLE: {
      float rx = x - P[0], ry = y - P[1];
      U[0] = (rx * rx + ry * ry <= P[2] * P[2]) ? P[3] : P[4];
      break;
    }
    case CVWENO_IC_QUADRANTS: {
      int qd = (x >= P[0] ? 1 : 0) + 2 * (y >= P[1] ? 1 : 0);
      const float* s = P + 2 + 4 * qd;
      prim_to_cons((float)a.gas_gamma, s[0], s[1], s[2], s[3], U);
      break;
    }
    case CVWENO_IC_FOURIER: {
      int M = (int)P[0];
      float acc = 0.0f;
      for (int j = 0; j < M && j < 15; ++j) {
        const float* md = P + 1 + 4 * j;
        acc += md[0] * sinf(twopi * (md[1] * (x - (float)a.x0) / (float)a.lx + md[2] * (y - (float)a.y0) / (float)a.ly) +
                            md[3]);
      }
      U[0] = acc;
      break;
    }
    case CVWENO_IC_POLY: {
      float acc = 0.0f, yp = 1.0f;
      for (int j = 0; j < 5; ++j) {
        float xp = 1.0f;
        for (int i = 0; i < 5; ++i) {
          acc += P[i + 5 * j] * xp * yp;
          xp *= x;
        }
        yp *= y;
      }
      U[0] = acc;
      break;
    }
    case CVWENO_IC_DENSITY_WAVE: {
      float rho = 1.0f + P[0] * sinf(twopi * (P[1] * (x - (float)a.x0) / (float)a.lx +
                                              P[2] * (y - (float)a.y0) / (float)a.ly));
      prim_to_cons((float)a.gas_gamma, rho, P[3], P[4], P[5], U);
      break;
    }
    default:
      U[0] = U[1] = U[2] = U[3] = 0.0f;
  }
}

// L2 projection c_m = (2mx+1)(2my+1)/4 sum_ab w_a w_b P_mx(a) P_my(b) u0(x_a, y_b) (2D), by sum
// factorisation: each row b of nodes is contracted over x first.  Four lanes per cell take
// three rows each and add their sums by shuffles, so that a small mesh still fills warps and a
// cell's chain is a quarter as long.
constexpr int kProjLanes = 4, kProjRows = kProjN / kProjLanes, kProjThreads = 128;

template <int DIM, int N, int NVAR>
__global__ void __launch_bounds__(kProjThreads) project_kernel(const __grid_constant__ ProjArgs a,
                                                               const __grid_constant__ ProjTables T) {
  constexpr int NY1 = DIM == 2 ? N : 1, ND = N * NY1, R = DIM == 2 ? kProjRows : 1;
  const int64_t ncell = (int64_t)a.nx * a.ny;
  const int lane = threadIdx.x % kProjLanes;
  // whole warps stay in the loop (the shuffles are warp-wide); cells past the end are clamped
  for (int64_t e0 = (blockIdx.x * (int64_t)kProjThreads + (threadIdx.x & ~31)) / kProjLanes; e0 < ncell;
       e0 += (int64_t)gridDim.x * kProjThreads / kProjLanes) {
    const int64_t mine = e0 + (threadIdx.x & 31) / kProjLanes, e = mine < ncell ? mine : ncell - 1;
    const int i = (int)(e % a.nx), j = (int)(e / a.nx);
    const double xc = a.x0 + (i + 0.5) * a.dx, yc = DIM == 2 ? a.y0 + (j + 0.5) * a.dy : 0.0;
    auto node_x = [&](int q) { return (float)(xc + 0.5 * a.dx * T.x[q]); };
    auto node_y = [&](int q) { return DIM == 2 ? (float)(yc + 0.5 * a.dy * T.x[q]) : 0.0f; };
    // row k of this lane is b = lane + 4 k (1D: the one row, on lane 0)
    float s[R][NVAR][N];
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
      for (int v = 0; v < NVAR; ++v)
#pragma unroll
        for (int m = 0; m < N; ++m) s[k][v][m] = 0.0f;
    float y[R];
#pragma unroll
    for (int k = 0; k < R; ++k) y[k] = node_y(lane + kProjLanes * k);
#pragma unroll 1
    for (int q = 0; q < kProjN; ++q) {
      const float x = node_x(q);
#pragma unroll
      for (int k = 0; k < R; ++k) {
        float U[4];
        ic_eval(a, x, y[k], U);
#pragma unroll
        for (int v = 0; v < NVAR; ++v)
#pragma unroll
          for (int m = 0; m < N; ++m) s[k][v][m] = fmaf(T.wP[q][m], U[v], s[k][v][m]);
      }
    }
    // over the lane's rows, then over the lanes
    float c[NVAR][ND];
#pragma unroll
    for (int v = 0; v < NVAR; ++v)
#pragma unroll
      for (int m = 0; m < ND; ++m) {
        float acc;
        if constexpr (DIM == 2) {
          acc = 0.0f;
#pragma unroll
          for (int k = 0; k < R; ++k) acc = fmaf(T.wP[lane + kProjLanes * k][m / N], s[k][v][m % N], acc);
#pragma unroll
          for (int d = 1; d < kProjLanes; d *= 2) acc += __shfl_xor_sync(0xffffffffu, acc, d, kProjLanes);
        } else {
          acc = s[0][v][m];
        }
        c[v][m] = acc * (DIM == 2 ? 0.25f * (2 * (m % N) + 1) * (2 * (m / N) + 1) : 0.5f * (2 * m + 1));
      }
    if (mine >= ncell) continue;
    // lane l writes modes l, l + 4, ...
#pragma unroll
    for (int v = 0; v < NVAR; ++v)
#pragma unroll
      for (int m0 = 0; m0 < ND; m0 += kProjLanes) {
        float o = c[v][m0];
#pragma unroll
        for (int l = 1; l < kProjLanes; ++l)
          if (m0 + l < ND && lane == l) o = c[v][m0 + l < ND ? m0 + l : m0];
        if (m0 + lane < ND) a.u[((size_t)v * ncell + e) * ND + m0 + lane] = o;
      }
  }
}

// A 2D Fourier datum in closed form.  About the cell's centre, sin(A_c + B_c + d_a + d_b) with
// offsets d the same in every cell, so the rule's sums over x and y separate: per mode a cell
// needs the sine and cosine of its two centre phases, and the projections of sin and cos of the
// offsets (host, FP64).  The centre phases are formed in turns, as the product of i + 1/2 with a
// two-float ratio, and reduced before they are rounded.  Bound by the stores and by FP32 issue:
// 512^2 Q3 with four modes: 9.8 us (2.63 ms with 144 full evaluations and a dense projection per
// cell, 0.104 ms with one-dimensional phases at the nodes).
struct FourierArgs {
  float* u;
  int nx, ny, modes;
  float rx[15][2], ry[15][2];                  // turns per cell in x and y (two-float)
  float cx[15][kMaxP + 1], sx[15][kMaxP + 1];  // (2m+1)/2 sum_a w_a P_m(a) (cos, sin)(d_a)
  float cy[15][kMaxP + 1], sy[15][kMaxP + 1];  // likewise in y
  float amp_cos[15], amp_sin[15];              // amplitude times cosine and sine of the phase
};
constexpr int kFourierThreads = 128;

// sin and cos of 2 pi (i + 1/2) r, r = r[0] + r[1]
__device__ __forceinline__ void turn_sincos(int i, const float (&r)[2], float& s, float& c) {
  const float h = (float)i + 0.5f, p = h * r[0];
  const float lo = fmaf(h, r[1], fmaf(h, r[0], -p));
  sincospif(2.0f * ((p - rintf(p)) + lo), &s, &c);
}

template <int N>
__global__ void __launch_bounds__(kFourierThreads) project_fourier_kernel(const __grid_constant__ FourierArgs a) {
  constexpr int ND = N * N;
  const int64_t ncell = (int64_t)a.nx * a.ny;
  for (int64_t e = blockIdx.x * (int64_t)kFourierThreads + threadIdx.x; e < ncell; e += (int64_t)gridDim.x * kFourierThreads) {
    const int i = (int)(e % a.nx), j = (int)(e / a.nx);
    float c[ND];
#pragma unroll
    for (int m = 0; m < ND; ++m) c[m] = 0.0f;
#pragma unroll 1
    for (int k = 0; k < a.modes; ++k) {
      float sa, ca, sb0, cb0;
      turn_sincos(i, a.rx[k], sa, ca);
      turn_sincos(j, a.ry[k], sb0, cb0);
      const float sb = fmaf(sb0, a.amp_cos[k], cb0 * a.amp_sin[k]), cb = fmaf(cb0, a.amp_cos[k], -sb0 * a.amp_sin[k]);
      float S[N], C[N];  // x projections of sin and cos of A
#pragma unroll
      for (int m = 0; m < N; ++m) {
        S[m] = fmaf(sa, a.cx[k][m], ca * a.sx[k][m]);
        C[m] = fmaf(ca, a.cx[k][m], -sa * a.sx[k][m]);
      }
#pragma unroll
      for (int my = 0; my < N; ++my) {
        const float s = fmaf(sb, a.cy[k][my], cb * a.sy[k][my]), t = fmaf(cb, a.cy[k][my], -sb * a.sy[k][my]);
#pragma unroll
        for (int m = 0; m < N; ++m) c[m + N * my] = fmaf(S[m], t, fmaf(C[m], s, c[m + N * my]));
      }
    }
    float* o = a.u + e * ND;
    if (ND % 4 == 0 && (reinterpret_cast<uintptr_t>(a.u) & 15) == 0) {
#pragma unroll
      for (int q = 0; q < ND / 4; ++q)
        reinterpret_cast<float4*>(o)[q] = make_float4(c[4 * q], c[4 * q + 1], c[4 * q + 2], c[4 * q + 3]);
    } else {
#pragma unroll
      for (int m = 0; m < ND; ++m) o[m] = c[m];
    }
  }
}

cudaError_t launch_project_fourier(cvweno_mesh m, const float* prm, const ProjRule& R, float* u, cudaStream_t s) {
  FourierArgs a;
  memset(&a, 0, sizeof(a));
  a.u = u;
  a.nx = m->nx;
  a.ny = m->ny;
  a.modes = (int)prm[0] < 0 ? 0 : (int)prm[0] < 15 ? (int)prm[0] : 15;
  auto direction = [&](double k, int n, float (&r)[2], float* c, float* sn) {
    const double turns = k / n;  // per cell
    r[0] = (float)turns;
    r[1] = (float)(turns - (double)r[0]);
    double cs[kMaxP + 1] = {0.0}, ss[kMaxP + 1] = {0.0};
    for (int q = 0; q < kProjN; ++q) {
      const double d = M_PI * turns * R.x[q], cd = R.w[q] * cos(d), sd = R.w[q] * sin(d);
      for (int mm = 0; mm <= m->p; ++mm) {
        cs[mm] += 0.5 * (2 * mm + 1) * R.P[q][mm] * cd;
        ss[mm] += 0.5 * (2 * mm + 1) * R.P[q][mm] * sd;
      }
    }
    for (int mm = 0; mm <= m->p; ++mm) c[mm] = (float)cs[mm], sn[mm] = (float)ss[mm];
  };
  for (int k = 0; k < a.modes; ++k) {
    const float* md = prm + 1 + 4 * k;
    direction(md[1], m->nx, a.rx[k], a.cx[k], a.sx[k]);
    direction(md[2], m->ny, a.ry[k], a.cy[k], a.sy[k]);
    a.amp_cos[k] = (float)(md[0] * cos((double)md[3]));
    a.amp_sin[k] = (float)(md[0] * sin((double)md[3]));
  }
  int64_t blocks = (m->ncell + kFourierThreads - 1) / kFourierThreads;
  if (blocks > 65535) blocks = 65535;
  switch (m->p) {
    case 1: project_fourier_kernel<2><<<(int)blocks, kFourierThreads, 0, s>>>(a); break;
    case 2: project_fourier_kernel<3><<<(int)blocks, kFourierThreads, 0, s>>>(a); break;
    case 3: project_fourier_kernel<4><<<(int)blocks, kFourierThreads, 0, s>>>(a); break;
    case 4: project_fourier_kernel<5><<<(int)blocks, kFourierThreads, 0, s>>>(a); break;
    default: return cudaErrorNotSupported;
  }
  return cudaGetLastError();
}

template <int DIM, int N>
cudaError_t launch_project(const ProjArgs& a, const ProjTables& T, cudaStream_t s) {
  const int64_t ncell = (int64_t)a.nx * a.ny;
  int64_t blocks = (ncell * kProjLanes + kProjThreads - 1) / kProjThreads;
  if (blocks > 65535) blocks = 65535;
  if constexpr (DIM == 2) {
    if (a.nvar == 4) {
      project_kernel<DIM, N, 4><<<(int)blocks, kProjThreads, 0, s>>>(a, T);
      return cudaGetLastError();
    }
  }
  project_kernel<DIM, N, 1><<<(int)blocks, kProjThreads, 0, s>>>(a, T);
  return cudaGetLastError();
}

// CG: interpolation at the GLL nodes of the periodic lattice (reading A25)
__global__ void project_cg_kernel(const __grid_constant__ ProjArgs a, const __grid_constant__ ProjTables T,
                                  int p, int nnx, int nny, const float* __restrict__ xg_dev) {
  (void)T;
  const int64_t nn = (int64_t)nnx * nny;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nn; j += (int64_t)gridDim.x * blockDim.x) {
    const int I = (int)(j % nnx), J = (int)(j / nnx);
    const int i = I / p, ai = I % p, jj = J / p, bj = J % p;
    const float x = (float)(a.x0 + (i + 0.5) * a.dx + 0.5 * a.dx * xg_dev[ai]);
    const float y = a.dim == 2 ? (float)(a.y0 + (jj + 0.5) * a.dy + 0.5 * a.dy * xg_dev[bj]) : 0.0f;
    float U[4];
    ic_eval(a, x, y, U);
    a.u[j] = U[0];
  }
}

// ---- FP64 reductions --------------------------------------------------------------------

// CG: partial sums of ML_j u_j (FP64) with the lumped mass of each lattice node
__global__ void sum_cg_partial(const float* __restrict__ u, int nnx, int nny, int p, const double* __restrict__ ml1x,
                               const double* __restrict__ ml1y, double* __restrict__ partial) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  const int64_t nn = (int64_t)nnx * nny;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nn; j += (int64_t)gridDim.x * blockDim.x) {
    const int I = (int)(j % nnx), J = (int)(j / nnx);
    acc += ml1x[I % p] * ml1y[J % p] * (double)u[j];
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

// DG conservation totals in one launch: block (b, v) sums mode 0 of a grid-stride slice of
// variable v (FP64) into partial[v][b]; the last block to finish adds each variable's partials
// in a fixed order into out[v].  The counter wraps to zero with the call's last block: calls that
// overlap on one mesh (which share the partials, so their own totals are undefined) leave it
// zero all the same, where a reset by the last block could leave a remainder for every later call.
__global__ void __launch_bounds__(kRedThreads) sum_mode0_kernel(const float* __restrict__ u, int64_t n, int stride,
                                                                double* __restrict__ partial, double* __restrict__ out,
                                                                unsigned* done) {
  __shared__ double sh[kRedThreads / 32];
  __shared__ bool last;
  const int nb = gridDim.x, nvar = gridDim.y, v = blockIdx.y, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  auto warp_sum = [](double x) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    return x;
  };
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)kRedThreads + threadIdx.x; i < n; i += (int64_t)nb * kRedThreads)
    acc += (double)u[((int64_t)v * n + i) * stride];
  acc = warp_sum(acc);
  if (lane == 0) sh[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kRedThreads / 32; ++w) acc += sh[w];
    partial[v * kRedBlocks + blockIdx.x] = acc;
    __threadfence();
    last = atomicInc(done, (unsigned)(nb * nvar) - 1) == (unsigned)(nb * nvar) - 1;  // back to zero by itself
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (warp < nvar) {  // one warp per variable
    acc = 0.0;
    for (int b = lane; b < nb; b += 32) acc += __ldcg(partial + warp * kRedBlocks + b);
    acc = warp_sum(acc);
    if (lane == 0) out[warp] = acc;
  }
}

__global__ void max_partial(const float* __restrict__ x, int64_t n, double* __restrict__ partial) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc = fmax(acc, (double)x[i]);
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

// single block: out[0] = sum (or max) of partial[0..n) in a fixed order
__global__ void finish_reduce(const double* __restrict__ partial, int n, int is_max, double* __restrict__ out) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc = is_max ? fmax(acc, partial[i]) : acc + partial[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] = is_max ? fmax(sh[threadIdx.x], sh[threadIdx.x + s]) : sh[threadIdx.x] + sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

StageArgs base_args(const cvweno_mesh_s* m) {
  StageArgs a;
  memset(&a, 0, sizeof(a));
  const cvweno_params& p = m->desc.params;
  a.status = m->d_status;
  set_check_extents(a, m->chk_state >= 0 ? m->chk_state : m->nstate, m->chk_cell >= 0 ? m->chk_cell : m->ncell);
  a.nx = m->nx;
  a.ny = m->ny;
  a.perx = m->desc.bc[0] == CVWENO_PERIODIC;
  a.pery = m->dim == 2 && m->desc.bc[2] == CVWENO_PERIODIC;
  a.vx = m->vx;
  a.two_dx = (float)(2.0 / m->dx);
  a.two_dy = (float)(2.0 / m->dy);
  a.nu_scale = (float)(m->h / (2.0 * m->p));
  a.h_e = (float)m->h;
  a.pk_img = m->d_pkimg;
  a.cg_img = m->d_cgimg;
  a.mlp = m->surrogate;
  a.mlp_conf_min = m->surrogate_conf_min;
  a.mlp_fallbacks = m->surrogate_fallbacks;
  a.eps = (float)p.eps;
  a.r = (int)p.r;
  a.q = (float)p.q;
  a.gamma_vertex = (float)p.gamma_vertex;
  a.c_gamma = (float)p.c_gamma;
  a.lambda_const = (float)p.lambda_const;
  a.sc = p.sc_quadrature;
  a.sensor_mode = p.sensor_mode;
  a.limit_all = 0;
  a.adv_vx = (float)p.adv_vx;
  a.adv_vy = (float)p.adv_vy;
  a.gas_gamma = (float)p.gas_gamma;
  a.rk_b = 1.0f;
  a.nnx = m->nnx;
  a.nny = m->nny;
  a.rloc = m->d_rloc;
  a.rnode = m->d_r;
  a.du = m->d_du;
  a.du2 = m->d_du2;
  return a;
}

cudaError_t launch(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  if (m->kind == CVWENO_CG) return launch_stage_cg(m, a, s);  // marks after each kernel itself
  cudaError_t e = m->desc.system == CVWENO_EULER ? launch_stage_euler(m, a, s) : launch_stage(m, a, s);
  kernel_mark(m, s);
  return e;
}

// Clears a raised status word that has been read, and its code.
cvweno_status take_status(cvweno_mesh m, int st, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  if (st) {
    e = cudaMemsetAsync(m->d_status, 0, sizeof(int), s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  }
  if (st & kStatCheck) return CVWENO_ERR_CHECK;
  if (st & kStatPositivity) return CVWENO_ERR_POSITIVITY;
  if (st & kStatNonfinite) return CVWENO_ERR_NONFINITE;
  if (st & kStatTimeout) return CVWENO_ERR_TIMEOUT;
  return CVWENO_OK;
}

cvweno_status read_status(cvweno_mesh m, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(m->h_status, m->d_status, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  return take_status(m, *m->h_status, s);
}

cvweno_status rk_stage(cvweno_mesh m, const float* in, const float* un, float* out, float ra, float rb, float dt,
                       cudaStream_t s, bool limit_pos = false) {
  NvtxRange range("rk_stage");
  StageArgs a = base_args(m);
  a.u_in = in;
  a.u_n = un;
  a.u_out = out;
  a.rk_a = ra;
  a.rk_b = rb;
  a.dt = dt;
  a.limit_pos = limit_pos;
  a.mode = kModeRK;
  return cuda_status(launch(m, a, s));
}

cvweno_status limit_stage(cvweno_mesh m, const float* in, float* out, cudaStream_t s) {
  StageArgs a = base_args(m);
  a.u_in = in;
  a.u_out = out;
  a.mode = kModeLimit;
  return cuda_status(launch(m, a, s));
}

cvweno_status positivity_stage(cvweno_mesh m, float* x, cudaStream_t s) {
  StageArgs a = base_args(m);
  a.u_in = x;
  a.u_out = x;
  cudaError_t e = launch_positivity(m, a, nullptr, s);
  kernel_mark(m, s);
  return cuda_status(e);
}

// A 1D scalar DG mesh of one tile without a limiter runs its steps in one launch, unless
// kernel timing asks for the stages one by one.
bool steps_in_one_launch(cvweno_mesh m) {
  return m->dim == 1 && m->kind != CVWENO_CG && m->desc.system != CVWENO_EULER && !m->desc.params.positivity &&
         !m->desc.params.hweno_limiter && !m->timing && m->nx <= kTile1D;
}

cvweno_status enqueue_steps_one_launch(cvweno_mesh m, float* u, float dt, int nsteps, cudaStream_t s) {
  StepArgs sa;
  const float* in[3] = {u, m->d_u1, m->d_u2};
  float* out[3] = {m->d_u1, m->d_u2, u};
  const float ra[3] = {0.0f, 0.75f, 1.0f / 3.0f}, rb[3] = {1.0f, 0.25f, 2.0f / 3.0f};
  for (int k = 0; k < 3; ++k) {
    StageArgs& a = sa.st[k];
    a = base_args(m);
    a.u_in = in[k];
    a.u_n = u;
    a.u_out = out[k];
    a.rk_a = ra[k];
    a.rk_b = rb[k];
    a.dt = dt;
    a.mode = kModeRK;
  }
  sa.nsteps = nsteps;
  return cuda_status(launch_steps_1d_tile(m, sa, s));
}

cvweno_status enqueue_step(cvweno_mesh m, float* u, float dt, cudaStream_t s) {
  if (steps_in_one_launch(m)) return enqueue_steps_one_launch(m, u, dt, 1, s);
  if (m->desc.params.positivity) {
    // every stage result is limited (reading P3): the limiter is cell-local, so the stage
    // kernel applies it before it writes; with timing on it is a launch of its own
    if (!m->timing) {
      cvweno_status st = rk_stage(m, u, u, m->d_u1, 0.0f, 1.0f, dt, s, true);
      if (st == CVWENO_OK) st = rk_stage(m, m->d_u1, u, m->d_u2, 0.75f, 0.25f, dt, s, true);
      if (st == CVWENO_OK) st = rk_stage(m, m->d_u2, u, u, 1.0f / 3.0f, 2.0f / 3.0f, dt, s, true);
      return st;
    }
    m->tcount = 0;
    kernel_mark(m, s);
    cvweno_status st = rk_stage(m, u, u, m->d_u1, 0.0f, 1.0f, dt, s);
    if (st == CVWENO_OK) st = positivity_stage(m, m->d_u1, s);
    if (st == CVWENO_OK) st = rk_stage(m, m->d_u1, u, m->d_u2, 0.75f, 0.25f, dt, s);
    if (st == CVWENO_OK) st = positivity_stage(m, m->d_u2, s);
    if (st == CVWENO_OK) st = rk_stage(m, m->d_u2, u, u, 1.0f / 3.0f, 2.0f / 3.0f, dt, s);
    if (st == CVWENO_OK) st = positivity_stage(m, u, s);
    return st;
  }
  if (m->timing) {
    m->tcount = 0;
    kernel_mark(m, s);
  }
  if (m->desc.params.hweno_limiter) {
    // every stage result is limited (reading A27); the limiter reads neighbours, so it
    // runs out of place: stages write d_u1, the limiter writes d_u2 (the last one u)
    cvweno_status st = rk_stage(m, u, u, m->d_u1, 0.0f, 1.0f, dt, s);
    if (st == CVWENO_OK) st = limit_stage(m, m->d_u1, m->d_u2, s);
    if (st == CVWENO_OK) st = rk_stage(m, m->d_u2, u, m->d_u1, 0.75f, 0.25f, dt, s);
    if (st == CVWENO_OK) st = limit_stage(m, m->d_u1, m->d_u2, s);
    if (st == CVWENO_OK) st = rk_stage(m, m->d_u2, u, m->d_u1, 1.0f / 3.0f, 2.0f / 3.0f, dt, s);
    if (st == CVWENO_OK) st = limit_stage(m, m->d_u1, u, s);
    return st;
  }
  cvweno_status st = rk_stage(m, u, u, m->d_u1, 0.0f, 1.0f, dt, s);
  if (st == CVWENO_OK) st = rk_stage(m, m->d_u1, u, m->d_u2, 0.75f, 0.25f, dt, s);
  if (st == CVWENO_OK) st = rk_stage(m, m->d_u2, u, u, 1.0f / 3.0f, 2.0f / 3.0f, dt, s);
  return st;
}

}  // namespace

namespace cvw {
StageArgs stage_base_args(const cvweno_mesh_s* m) { return base_args(m); }

void kernel_mark(const cvweno_mesh_s* mc, cudaStream_t s) {
  cvweno_mesh_s* m = const_cast<cvweno_mesh_s*>(mc);
  if (!m->timing || m->tcount >= kMaxMarks) return;
  // inside stream capture the record becomes an event-record node of the graph, so the
  // events time every replay
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &cs);
  cudaEventRecordWithFlags(m->tev[m->tcount++], s, cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : 0);
}
}  // namespace cvw

extern "C" {

void cvweno_default_params(cvweno_params* p) {
  if (!p) return;
  p->eps = 1e-6;
  p->r = 2.0;
  p->q = 1.0;
  p->gamma_vertex = 1e-3;
  p->c_gamma = 0.9;
  p->sc_quadrature = 1;
  p->sensor_mode = CVWENO_SENSOR_COMPUTED;
  p->lambda_const = 0.0;
  p->gas_gamma = 1.4;
  p->adv_vx = 1.0;
  p->adv_vy = 0.0;
}

const char* cvweno_status_string(cvweno_status s) {
  switch (s) {
    case CVWENO_OK: return "ok";
    case CVWENO_ERR_ARG: return "invalid argument";
    case CVWENO_ERR_CUDA: return "CUDA runtime error";
    case CVWENO_ERR_NONFINITE: return "non-finite value produced";
    case CVWENO_ERR_POSITIVITY: return "non-positive density or pressure";
    case CVWENO_ERR_TIMEOUT: return "bounded device wait timed out";
    case CVWENO_ERR_UNSUPPORTED: return "unsupported configuration";
    case CVWENO_ERR_NOMEM: return "out of memory";
    case CVWENO_ERR_CHECK: return "bounds check failed (checked build)";
  }
  return "unknown status";
}

cvweno_status cvweno_mesh_destroy(cvweno_mesh m) {
  if (!m) return CVWENO_OK;
  if (m->d_u1) cudaDeviceSynchronize();
  cudaFree(m->d_u1);
  cudaFree(m->d_u2);
  cudaFree(m->d_lambda);
  cudaFree(m->d_red);
  cudaFree(m->d_status);
  cudaFree(m->d_rloc);
  cudaFree(m->d_r);
  cudaFree(m->d_du);
  cudaFree(m->d_du2);
  cudaFree(m->d_cg_xg);
  cudaFree(m->d_cg_ml);
  cudaFree(m->d_cgimg);
  cudaFree(m->d_pkimg);
  cudaFreeHost(m->h_status);
  cudaFreeHost(m->h_red);
  for (int i = 0; i < kMaxMarks; ++i)
    if (m->tev[i]) cudaEventDestroy(m->tev[i]);
  free(m->cell_vertices);
  free(m->vertex_cells);
  free(m->colour);
  free(m->tables);
  free(m->cg_tables);
  free(m);
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_create(const cvweno_mesh_desc* d, cvweno_mesh* out) {
  if (!d || !out) return CVWENO_ERR_ARG;
  *out = nullptr;
  if (d->dim != 1 && d->dim != 2) return CVWENO_ERR_ARG;
  if (d->nx < 1 || (d->dim == 2 && d->ny < 1)) return CVWENO_ERR_ARG;
  if (d->nx > (1 << 24) || (d->dim == 2 && d->ny > (1 << 20))) return CVWENO_ERR_ARG;
  if (!(d->x1 > d->x0) || (d->dim == 2 && !(d->y1 > d->y0))) return CVWENO_ERR_ARG;
  for (int i = 0; i < 4; ++i)
    if (d->bc[i] != CVWENO_PERIODIC && d->bc[i] != CVWENO_TRANSMISSIVE) return CVWENO_ERR_ARG;
  if ((d->bc[0] == CVWENO_PERIODIC) != (d->bc[1] == CVWENO_PERIODIC)) return CVWENO_ERR_ARG;
  if (d->dim == 2 && (d->bc[2] == CVWENO_PERIODIC) != (d->bc[3] == CVWENO_PERIODIC)) return CVWENO_ERR_ARG;
  if (d->system < CVWENO_BURGERS || d->system > CVWENO_EULER) return CVWENO_ERR_ARG;
  const cvweno_params& p = d->params;
  if (!(p.eps > 0.0) || !(p.q >= 1.0) || !(p.gamma_vertex > 0.0) || (1 << d->dim) * p.gamma_vertex >= 1.0)
    return CVWENO_ERR_ARG;
  if (p.sensor_mode < 0 || p.sensor_mode > 2) return CVWENO_ERR_ARG;
  if (p.hweno_limiter != 0 && p.hweno_limiter != 1) return CVWENO_ERR_ARG;
  if (p.hweno_limiter && (d->kind != CVWENO_DG || d->system == CVWENO_EULER)) return CVWENO_ERR_UNSUPPORTED;
  if (p.positivity != 0 && p.positivity != 1) return CVWENO_ERR_ARG;
  if (p.positivity && (d->kind != CVWENO_DG || d->system != CVWENO_EULER)) return CVWENO_ERR_UNSUPPORTED;
  if (d->kind != CVWENO_DG && d->kind != CVWENO_CG) return CVWENO_ERR_ARG;
  // CG: scalar laws on periodic meshes (no boundary flux term is implemented)
  if (d->kind == CVWENO_CG && (d->system == CVWENO_EULER || d->bc[0] != CVWENO_PERIODIC ||
                               (d->dim == 2 && d->bc[2] != CVWENO_PERIODIC)))
    return CVWENO_ERR_UNSUPPORTED;
  if (d->degree < 1 || d->degree > kMaxP) return CVWENO_ERR_UNSUPPORTED;
  if (p.r != floor(p.r) || p.r < 1.0 || p.r > 8.0) return CVWENO_ERR_UNSUPPORTED;
  if ((d->system == CVWENO_KPP || d->system == CVWENO_EULER) && d->dim != 2) return CVWENO_ERR_UNSUPPORTED;

  cvweno_mesh m = (cvweno_mesh)calloc(1, sizeof(cvweno_mesh_s));
  if (!m) return CVWENO_ERR_NOMEM;
  m->desc = *d;
  m->chk_state = m->chk_cell = -1;
  cudaGetDevice(&m->device);
  m->dim = d->dim;
  m->p = d->degree;
  m->n = d->degree + 1;
  m->nd = d->dim == 2 ? m->n * m->n : m->n;
  m->nq = m->nd;
  m->nvar = d->system == CVWENO_EULER ? 4 : 1;
  m->ncorner = 1 << d->dim;
  m->nx = d->nx;
  m->ny = d->dim == 2 ? d->ny : 1;
  m->vx = d->bc[0] == CVWENO_PERIODIC ? m->nx : m->nx + 1;
  m->vy = d->dim == 2 ? (d->bc[2] == CVWENO_PERIODIC ? m->ny : m->ny + 1) : 1;
  m->ncell = (int64_t)m->nx * m->ny;
  m->nvert = (int64_t)m->vx * m->vy;
  m->kind = d->kind;
  m->nnx = d->kind == CVWENO_CG ? m->p * m->nx : 0;
  m->nny = d->kind == CVWENO_CG ? (d->dim == 2 ? m->p * m->ny : 1) : 0;
  m->nnode = (int64_t)m->nnx * m->nny;
  m->nstate = d->kind == CVWENO_CG ? m->nnode * m->nvar : m->ncell * m->nd * m->nvar;
  m->dx = (d->x1 - d->x0) / m->nx;
  m->dy = d->dim == 2 ? (d->y1 - d->y0) / m->ny : 1.0;
  m->h = d->dim == 2 ? sqrt(m->dx * m->dx + m->dy * m->dy) : m->dx;

  cvweno_status st = build_tables(m);
  if (st != CVWENO_OK) { cvweno_mesh_destroy(m); return st; }
  cudaError_t e = cudaSuccess;
  size_t sbytes = sizeof(float) * (size_t)m->nstate;
  if (e == cudaSuccess) e = cudaMalloc(&m->d_u1, sbytes);
  if (e == cudaSuccess) e = cudaMalloc(&m->d_u2, sbytes);
  if (e == cudaSuccess) e = cudaMalloc(&m->d_lambda, sizeof(float) * (size_t)m->ncell);
  if (e == cudaSuccess) e = cudaMalloc(&m->d_pkimg, sizeof(float) * (size_t)packed_image_floats(m->dim, m->p));
  if (e == cudaSuccess) e = launch_packed_image(m->dim, m->p, m->tables, m->d_pkimg, 0);
  if (e == cudaSuccess) e = cudaStreamSynchronize(0);
  if (m->kind == CVWENO_CG) {
    if (e == cudaSuccess) e = cudaMalloc(&m->d_rloc, sizeof(float) * (size_t)m->ncell * m->nd);
    if (m->dim == 1) {  // 2D meshes keep the node phase in one kernel's shared memory
      if (e == cudaSuccess) e = cudaMalloc(&m->d_du2, sizeof(float) * (size_t)m->nnode);
      if (e == cudaSuccess) e = cudaMalloc(&m->d_r, sizeof(float) * (size_t)m->nnode);
      if (e == cudaSuccess) e = cudaMalloc(&m->d_du, sizeof(float) * (size_t)m->nnode);
    }
    float cimg[kMaxCgImage];
    const int nimg = cg_image(m->dim, m->p, m->cg_tables, cimg, kMaxCgImage);
    if (nimg == 0) e = cudaErrorInvalidValue;
    if (e == cudaSuccess) e = cudaMalloc(&m->d_cgimg, sizeof(float) * nimg);
    if (e == cudaSuccess) e = cudaMemcpy(m->d_cgimg, cimg, sizeof(float) * nimg, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&m->d_cg_xg, sizeof(float) * (kMaxP + 1));
    if (e == cudaSuccess) e = cudaMalloc(&m->d_cg_ml, sizeof(double) * 2 * (kMaxP + 1));
    if (e == cudaSuccess) {
      float xg[kMaxP + 1];
      double ml[2 * (kMaxP + 1)];
      for (int i = 0; i <= kMaxP; ++i) {
        xg[i] = i <= m->p ? (float)m->cg_xg[i] : 0.0f;
        const double w = i <= m->p ? m->cg_wl[i] * (i == 0 ? 2.0 : 1.0) : 0.0;  // vertex nodes: two cells
        ml[i] = w * 0.5 * m->dx;
        ml[kMaxP + 1 + i] = m->dim == 2 ? w * 0.5 * m->dy : 1.0;
      }
      e = cudaMemcpy(m->d_cg_xg, xg, sizeof(xg), cudaMemcpyHostToDevice);
      if (e == cudaSuccess) e = cudaMemcpy(m->d_cg_ml, ml, sizeof(ml), cudaMemcpyHostToDevice);
    }
  }
  if (e == cudaSuccess) e = cudaMalloc(&m->d_red, sizeof(double) * (kRedOut + 10));
  if (e == cudaSuccess) e = cudaMemset(m->d_red, 0, sizeof(double) * (kRedOut + 10));
  if (e == cudaSuccess) e = cudaMalloc(&m->d_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(m->d_status, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMallocHost(&m->h_status, sizeof(int));
  if (e == cudaSuccess) e = cudaMallocHost(&m->h_red, sizeof(double) * 8);
  if (e != cudaSuccess) {
    cvweno_mesh_destroy(m);
    return e == cudaErrorMemoryAllocation ? CVWENO_ERR_NOMEM : CVWENO_ERR_CUDA;
  }
  *out = m;
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_info(cvweno_mesh m, int64_t* ncells, int64_t* ndof, int* nvars, int64_t* nverts,
                               int* nquad) {
  if (!m) return CVWENO_ERR_ARG;
  if (ncells) *ncells = m->ncell;
  if (ndof) *ndof = m->nd;
  if (nvars) *nvars = m->nvar;
  if (nverts) *nverts = m->nvert;
  if (nquad) *nquad = m->nq;
  return CVWENO_OK;
}

cvweno_status cvweno_state_size(cvweno_mesh m, int64_t* nstate) {
  if (!m || !nstate) return CVWENO_ERR_ARG;
  *nstate = m->nstate;
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_tables(cvweno_mesh m, int32_t* cell_vertices, int32_t* vertex_cells, int32_t* colour) {
  if (!m) return CVWENO_ERR_ARG;
  if (cell_vertices) memcpy(cell_vertices, m->cell_vertices, sizeof(int32_t) * m->ncell * m->ncorner);
  if (vertex_cells) memcpy(vertex_cells, m->vertex_cells, sizeof(int32_t) * m->nvert * m->ncorner);
  if (colour) memcpy(colour, m->colour, sizeof(int32_t) * m->ncell);
  return CVWENO_OK;
}

cvweno_status cvweno_project(cvweno_mesh m, int ic_type, const double* ic_params, float* u, void* stream) {
  if (!m || !ic_params || !u) return CVWENO_ERR_ARG;
  if (ic_type < CVWENO_IC_CONST || ic_type > CVWENO_IC_DENSITY_WAVE) return CVWENO_ERR_ARG;
  if ((ic_type == CVWENO_IC_QUADRANTS || ic_type == CVWENO_IC_DENSITY_WAVE) != (m->nvar == 4) &&
      ic_type != CVWENO_IC_CONST)
    return CVWENO_ERR_ARG;
  ProjArgs a;
  memset(&a, 0, sizeof(a));
  a.u = u;
  a.nx = m->nx;
  a.ny = m->ny;
  a.dim = m->dim;
  a.nd = m->nd;
  a.n = m->n;
  a.nvar = m->nvar;
  a.type = ic_type;
  a.x0 = m->desc.x0;
  a.y0 = m->desc.y0;
  a.dx = m->dx;
  a.dy = m->dy;
  a.lx = m->desc.x1 - m->desc.x0;
  a.ly = m->dim == 2 ? m->desc.y1 - m->desc.y0 : 1.0;
  a.gas_gamma = m->desc.params.gas_gamma;
  for (int i = 0; i < 64; ++i) a.prm[i] = (float)ic_params[i];
  // Gauss nodes/weights of the 12-point projection rule and Legendre values there.
  const ProjRule& R = proj_rule();
  if (!R.ok) return CVWENO_ERR_ARG;
  if (m->kind != CVWENO_CG && m->dim == 2 && ic_type == CVWENO_IC_FOURIER)
    return cuda_status(launch_project_fourier(m, a.prm, R, u, S(stream)));
  ProjTables T;
  for (int q = 0; q < kProjN; ++q) {
    T.x[q] = (float)R.x[q];
    for (int mm = 0; mm <= kMaxP; ++mm) T.wP[q][mm] = (float)(R.w[q] * R.P[q][mm]);
  }
  if (m->kind == CVWENO_CG) {
    int blocks = (int)((m->nnode + 255) / 256);
    if (blocks > 65535) blocks = 65535;
    project_cg_kernel<<<blocks, 256, 0, S(stream)>>>(a, T, m->p, m->nnx, m->nny, m->d_cg_xg);
    return cuda_status(cudaGetLastError());
  }
  cudaError_t e = cudaErrorNotSupported;
  switch (m->dim * 10 + m->p) {
    case 11: e = launch_project<1, 2>(a, T, S(stream)); break;
    case 12: e = launch_project<1, 3>(a, T, S(stream)); break;
    case 13: e = launch_project<1, 4>(a, T, S(stream)); break;
    case 14: e = launch_project<1, 5>(a, T, S(stream)); break;
    case 21: e = launch_project<2, 2>(a, T, S(stream)); break;
    case 22: e = launch_project<2, 3>(a, T, S(stream)); break;
    case 23: e = launch_project<2, 4>(a, T, S(stream)); break;
    case 24: e = launch_project<2, 5>(a, T, S(stream)); break;
  }
  return cuda_status(e);
}

cvweno_status cvweno_vertex_data(cvweno_mesh m, const float* u, float* tstar, void* stream) {
  if (!m || !u || !tstar) return CVWENO_ERR_ARG;
  NvtxRange range("cvweno_vertex_data");
  StageArgs a = base_args(m);
  a.u_in = u;
  a.tstar_out = tstar;
  a.mode = kModeSensorOnly;
  return cuda_status(launch(m, a, S(stream)));
}

cvweno_status cvweno_sensor(cvweno_mesh m, const float* u, float* gamma, float* nu, void* stream) {
  if (!m || !u) return CVWENO_ERR_ARG;
  NvtxRange range("cvweno_sensor");
  StageArgs a = base_args(m);
  a.u_in = u;
  a.gamma_out = gamma;
  a.nu_out = nu;
  a.mode = kModeSensorOnly;
  return cuda_status(launch(m, a, S(stream)));
}

cvweno_status cvweno_positivity(cvweno_mesh m, const float* u, float* out, float* theta, void* stream) {
  if (!m || !u || !out) return CVWENO_ERR_ARG;
  if (m->kind != CVWENO_DG || m->desc.system != CVWENO_EULER || m->dim != 2) return CVWENO_ERR_UNSUPPORTED;
  StageArgs a = base_args(m);
  a.u_in = u;
  a.u_out = out;
  return cuda_status(launch_positivity(m, a, theta, S(stream)));
}

cvweno_status cvweno_limit(cvweno_mesh m, const float* u, float* out, int all_cells, int32_t* troubled,
                           void* stream) {
  if (!m || !u || !out || u == out) return CVWENO_ERR_ARG;
  if (m->kind != CVWENO_DG || m->desc.system == CVWENO_EULER) return CVWENO_ERR_UNSUPPORTED;
  NvtxRange range("cvweno_limit");
  StageArgs a = base_args(m);
  a.u_in = u;
  a.u_out = out;
  a.troubled_out = troubled;
  a.limit_all = all_cells ? 1 : 0;
  a.mode = kModeLimit;
  return cuda_status(launch(m, a, S(stream)));
}

cvweno_status cvweno_residual_ex(cvweno_mesh m, const float* u, const int32_t* troubled_override, float* dudt,
                                 float* gamma, float* nu, float* alpha, int32_t* troubled, void* stream) {
  if (!m || !u || !dudt || u == dudt) return CVWENO_ERR_ARG;
  NvtxRange range("cvweno_residual");
  StageArgs a = base_args(m);
  a.u_in = u;
  a.u_n = u;
  a.u_out = dudt;
  a.gamma_out = gamma;
  a.nu_out = nu;
  a.alpha_out = alpha;
  a.troubled_out = troubled;
  a.troubled_override = troubled_override;
  a.mode = kModeResidual;
  return cuda_status(launch(m, a, S(stream)));
}

cvweno_status cvweno_residual(cvweno_mesh m, const float* u, float* dudt, void* stream) {
  return cvweno_residual_ex(m, u, nullptr, dudt, nullptr, nullptr, nullptr, nullptr, stream);
}

cvweno_status cvweno_max_wavespeed(cvweno_mesh m, const float* u, double* lam, void* stream) {
  if (!m || !u || !lam) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  StageArgs a = base_args(m);
  a.u_in = u;
  cudaError_t e;
  double* out = m->d_red + kRedOut;
  if (m->kind == CVWENO_CG || (m->desc.system != CVWENO_EULER && m->desc.params.lambda_const > 0.0) || m->surrogate) {
    // CG cells' polynomials come from the stage kernel; a constant speed needs no pass, but takes
    // this way for the same answer on an empty status; with the network attached the call is one
    // more evaluation of the sensor, whose fallbacks are counted
    a.lambda_out = m->d_lambda;
    a.mode = kModeSensorOnly;
    e = launch(m, a, s);
    if (e == cudaSuccess) {
      max_partial<<<kRedBlocks, kRedThreads, 0, s>>>(m->d_lambda, m->ncell, m->d_red);
      finish_reduce<<<1, kRedThreads, 0, s>>>(m->d_red, kRedBlocks, 1, out);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->h_red, out, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return CVWENO_ERR_CUDA;
    cvweno_status st = read_status(m, s);  // synchronises
    if (st != CVWENO_OK) return st;
  } else {
    // one pass over the cells, one copy of the maximum and the status word
    unsigned* slots = reinterpret_cast<unsigned*>(out + 8);
    const MaxSlots ms{slots, slots + 1, out, reinterpret_cast<int*>(out + 1)};
    e = m->desc.system == CVWENO_EULER ? launch_wavespeed_euler(m, a, ms, s) : launch_wavespeed_scalar(m, a, ms, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->h_red, out, 2 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return CVWENO_ERR_CUDA;
    int bits;
    memcpy(&bits, m->h_red + 1, sizeof(bits));
    cvweno_status st = take_status(m, bits, s);
    if (st != CVWENO_OK) return st;
  }
  *lam = m->h_red[0];
  return CVWENO_OK;
}

cvweno_status cvweno_step(cvweno_mesh m, float* u, double dt, double cfl, double* dt_used, void* stream) {
  if (!m || !u) return CVWENO_ERR_ARG;
  NvtxRange range("cvweno_step");
  cudaStream_t s = S(stream);
  if (!(dt > 0.0)) {
    if (!(cfl > 0.0)) return CVWENO_ERR_ARG;
    double lam = 0.0;
    cvweno_status st = cvweno_max_wavespeed(m, u, &lam, stream);
    if (st != CVWENO_OK) return st;
    if (!(lam > 0.0)) return CVWENO_ERR_ARG;
    double hmin = m->dim == 2 ? fmin(m->dx, m->dy) : m->dx;
    dt = cfl * hmin / (m->dim * lam);
  }
  if (dt_used) *dt_used = dt;
  return enqueue_step(m, u, (float)dt, s);
}

cvweno_status cvweno_advance(cvweno_mesh m, float* u, double dt, int nsteps, void* stream) {
  if (!m || !u || !(dt > 0.0) || nsteps < 0) return CVWENO_ERR_ARG;
  NvtxRange range("cvweno_advance");
  if (nsteps > 0 && steps_in_one_launch(m)) return enqueue_steps_one_launch(m, u, (float)dt, nsteps, S(stream));
  for (int i = 0; i < nsteps; ++i) {
    cvweno_status st = enqueue_step(m, u, (float)dt, S(stream));
    if (st != CVWENO_OK) return st;
  }
  return CVWENO_OK;
}

cvweno_status cvweno_mass_total(cvweno_mesh m, const float* u, double* totals, void* stream) {
  if (!m || !u || !totals) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  if (m->kind == CVWENO_CG) {
    // sum_j ML_j u_j with ML_j = ml1x(I mod p) ml1y(J mod p)
    sum_cg_partial<<<kRedBlocks, kRedThreads, 0, s>>>(u, m->nnx, m->nny, m->p, m->d_cg_ml, m->d_cg_ml + (kMaxP + 1),
                                                     m->d_red);
    finish_reduce<<<1, kRedThreads, 0, s>>>(m->d_red, kRedBlocks, 0, m->d_red + kRedOut);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->h_red, m->d_red + kRedOut, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return CVWENO_ERR_CUDA;
    totals[0] = m->h_red[0];
    return CVWENO_OK;
  }
  // int_{K_e} u_h = |K_e| * (Legendre mode 0)
  const double vol = m->dim == 2 ? m->dx * m->dy : m->dx;
  const int64_t nb = (m->ncell + kRedThreads - 1) / kRedThreads;
  unsigned* slots = reinterpret_cast<unsigned*>(m->d_red + kRedOut + 8);
  sum_mode0_kernel<<<dim3((unsigned)(nb < kRedBlocks ? nb : kRedBlocks), m->nvar), kRedThreads, 0, s>>>(
      u, m->ncell, m->nd, m->d_red, m->d_red + kRedOut, slots + 2);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(m->h_red, m->d_red + kRedOut, sizeof(double) * m->nvar, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  for (int v = 0; v < m->nvar; ++v) totals[v] = m->h_red[v] * vol;
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_set_kernel_timing(cvweno_mesh m, int enable) {
  if (!m) return CVWENO_ERR_ARG;
  if (enable && !m->tev[0])
    for (int i = 0; i < kMaxMarks; ++i)
      if (cudaEventCreate(&m->tev[i]) != cudaSuccess) return CVWENO_ERR_CUDA;
  m->timing = enable ? 1 : 0;
  if (enable) m->tcount = 0;  // disabling keeps the last step's events readable
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_set_tensor_cores(cvweno_mesh m, int enable) {
  if (!m || (enable != 0 && enable != 1)) return CVWENO_ERR_ARG;
  if (enable && !(m->dim == 2 && m->kind == CVWENO_DG && m->p == 3 && m->desc.system != CVWENO_EULER))
    return CVWENO_ERR_UNSUPPORTED;
  m->tensor_cores = enable;
  return CVWENO_OK;
}

cvweno_status cvweno_mesh_set_check_extents(cvweno_mesh m, int64_t state_floats, int64_t cells) {
  if (!m || state_floats > m->nstate || cells > m->ncell || ((state_floats < 0) != (cells < 0)))
    return CVWENO_ERR_ARG;
#ifdef CVWENO_CHECK
  m->chk_state = state_floats;
  m->chk_cell = cells;
  return CVWENO_OK;
#else
  return CVWENO_ERR_UNSUPPORTED;
#endif
}

cvweno_status cvweno_kernel_times(cvweno_mesh m, float* ms, int capacity, int* count) {
  if (!m || !count || capacity < 0 || (capacity > 0 && !ms)) return CVWENO_ERR_ARG;
  *count = 0;
  if (!m->tev[0] || m->tcount < 2) return CVWENO_OK;
  if (cudaEventSynchronize(m->tev[m->tcount - 1]) != cudaSuccess) return CVWENO_ERR_CUDA;
  const int n = m->tcount - 1 < capacity ? m->tcount - 1 : capacity;
  for (int i = 0; i < n; ++i)
    if (cudaEventElapsedTime(&ms[i], m->tev[i], m->tev[i + 1]) != cudaSuccess) return CVWENO_ERR_CUDA;
  *count = n;
  return CVWENO_OK;
}

cvweno_status cvweno_status_check(cvweno_mesh m, void* stream) {
  if (!m) return CVWENO_ERR_ARG;
  return read_status(m, S(stream));
}

}  // extern "C"
