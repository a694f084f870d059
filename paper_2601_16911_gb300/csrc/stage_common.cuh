// Pieces shared by the stage kernels: scalar helpers, the scalar laws in deviation form,
// asynchronous copies and programmatic dependent launch.
#pragma once

#include <utility>

#include "dg_packed.cuh"

namespace cvw {

__device__ __forceinline__ float ipowf(float x, int r) {
  if (r == 2) return x * x;  // the paper's r
  float y = x;
  for (int i = 1; i < r; ++i) y *= x;
  return y;
}

// The general power is out of line: it is cold at the paper's q = 1, and inlined at every
// call site it crowds the instruction cache of the stage kernels.
static __device__ __noinline__ float powf_cold(float x, float q) { return powf(x, q); }
__device__ __forceinline__ float powq(float x, float q) { return q == 1.0f ? x : powf_cold(x, q); }

// Reciprocal and square root in PTX's approximate forms (relative error about 2^-22, no
// range check and no slow path), for the nonlinear weights and norms of stages (b)-(c)
// and the node-wise flux paths, which need FP32 precision, not correct rounding.
__device__ __forceinline__ float rcp_fast(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ float sqrt_fast(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- scalar fluxes, evaluated as deviations from the cell mean -------------------------
// A law object is built per cell from its mean ubar.  flux_dev returns
// f(ubar + d) - f(ubar) in forms whose rounding is relative to |d|; llf_dev returns the
// LLF flux minus f(ubar) . n.  The constant f(ubar) cancels exactly between the volume
// and face terms of every test function, so it is never formed.
template <int SYS, int DIM>
struct ScalarLaw;

template <int DIM>
struct ScalarLaw<CVWENO_BURGERS, DIM> {
  float ubar;
  __device__ __forceinline__ ScalarLaw(const StageArgs&, float ub) : ubar(ub) {}
  __device__ __forceinline__ float dev(float d) const { return d * fmaf(0.5f, d, ubar); }
  __device__ __forceinline__ void flux_dev(float d, float& fx, float& fy) const {
    fx = dev(d);
    fy = fx;
  }
  __device__ __forceinline__ float flux_dev_dir(float d, int) const { return dev(d); }
  __device__ __forceinline__ f2 flux_dev_dir2(f2 d, int) const { return mul2(d, fma2(dup2(0.5f), d, dup2(ubar))); }
  __device__ __forceinline__ void flux_dev2(f2 d, f2& fx, f2& fy) const { fx = fy = flux_dev_dir2(d, 0); }
  // |f'(u)| (Euclidean) for nu_e, and |f'(u) . n| for an axis-aligned face
  __device__ __forceinline__ float speed(float u) const { return DIM == 2 ? 1.41421356237f * fabsf(u) : fabsf(u); }
  __device__ __forceinline__ float nspeed(float u, int) const { return fabsf(u); }
};

// sin d and cos d - 1 for |d| <= 1 from their Maclaurin series, Horner in d^2, to the
// d^11 and d^12 terms: the first omitted terms are below 2e-10 at |d| = 1, far under one
// FP32 ulp, and cos d - 1 comes without cancellation.
__device__ __forceinline__ void sin_cosm1_small(float d, float& s, float& cm1) {
  const float z = d * d;
  float ps = fmaf(z, -1.0f / 39916800.0f, 1.0f / 362880.0f);
  ps = fmaf(z, ps, -1.0f / 5040.0f);
  ps = fmaf(z, ps, 1.0f / 120.0f);
  ps = fmaf(z, ps, -1.0f / 6.0f);
  s = fmaf(d * z, ps, d);
  float pc = fmaf(z, 1.0f / 479001600.0f, -1.0f / 3628800.0f);
  pc = fmaf(z, pc, 1.0f / 40320.0f);
  pc = fmaf(z, pc, -1.0f / 720.0f);
  pc = fmaf(z, pc, 1.0f / 24.0f);
  pc = fmaf(z, pc, -0.5f);
  cm1 = z * pc;
}

// sin d and cos d - 1 for the deviations beyond |d| = 1 (a few multiples of pi inside a
// KPP cell): Cody and Waite's reduction d = k pi/2 + r, |r| <= pi/4, with pi/2 split into
// an FP32 head and tail and the FMA products exact, then the series above for r and the
// quadrant k mod 4.  cos d - 1 is taken from cos r - 1 where cos d = cos r (no
// cancellation); in the other quadrants cos d is at most cos(pi/4) and c - 1 does not
// cancel.  Accurate to a few FP32 ulps while k pi/2's tail stays below half an ulp of r,
// i.e. for |d| up to about 1e3 (a KPP state lies within [pi/4, 7 pi/2] by the maximum
// principle); a non-finite d gives non-finite results, which the stage flags.
__device__ __forceinline__ void sin_cosm1_reduced(float d, float& s, float& cm1) {
  const float k = rintf(d * 0.636619772f);      // nearest multiple of pi/2
  float r = fmaf(-k, 1.57079637f, d);            // pi/2 rounded to FP32 ...
  r = fmaf(-k, -4.37113883e-8f, r);              // ... and the rest of pi/2
  float sr, cr1;
  sin_cosm1_small(r, sr, cr1);
  switch ((int)k & 3) {
    case 0: s = sr; cm1 = cr1; break;
    case 1: s = cr1 + 1.0f; cm1 = -sr - 1.0f; break;
    case 2: s = -sr; cm1 = -cr1 - 2.0f; break;
    default: s = -(cr1 + 1.0f); cm1 = sr - 1.0f; break;
  }
}

// Both for a pair of deviations: the series on the pair, after the reduction of the halves
// beyond |d| = 1 (k = 0 for the others, whose value is the plain series).
__device__ __forceinline__ void sin_cosm1_2(f2 d, f2& s, f2& cm1) {
  const bool big = fabsf(d.x) > 1.0f || fabsf(d.y) > 1.0f;
  f2 r = d;
  float kx = 0.0f, ky = 0.0f;
  if (big) {
    kx = fabsf(d.x) > 1.0f ? rintf(d.x * 0.636619772f) : 0.0f;
    ky = fabsf(d.y) > 1.0f ? rintf(d.y * 0.636619772f) : 0.0f;
    r = fma2(mk2(-kx, -ky), dup2(1.57079637f), r);
    r = fma2(mk2(-kx, -ky), dup2(-4.37113883e-8f), r);
  }
  const f2 z = mul2(r, r);
  f2 ps = fma2(z, dup2(-1.0f / 39916800.0f), dup2(1.0f / 362880.0f));
  ps = fma2(z, ps, dup2(-1.0f / 5040.0f));
  ps = fma2(z, ps, dup2(1.0f / 120.0f));
  ps = fma2(z, ps, dup2(-1.0f / 6.0f));
  s = fma2(mul2(r, z), ps, r);
  f2 pc = fma2(z, dup2(1.0f / 479001600.0f), dup2(-1.0f / 3628800.0f));
  pc = fma2(z, pc, dup2(1.0f / 40320.0f));
  pc = fma2(z, pc, dup2(-1.0f / 720.0f));
  pc = fma2(z, pc, dup2(1.0f / 24.0f));
  pc = fma2(z, pc, dup2(-0.5f));
  cm1 = mul2(z, pc);
  if (big) {
    const f2 sr = s, cr = cm1;
    const int qx = (int)kx & 3, qy = (int)ky & 3;
    s.x = (qx & 1) ? cr.x + 1.0f : sr.x;
    cm1.x = (qx & 1) ? -sr.x : cr.x;  // cos d - 1 (+1 where the quadrant is odd)
    s.y = (qy & 1) ? cr.y + 1.0f : sr.y;
    cm1.y = (qy & 1) ? -sr.y : cr.y;
    // k = 2, 3: both change sign (cos d = -cos r: cos d - 1 = -(cos r - 1) - 2)
    if (qx & 2) s.x = -s.x, cm1.x = -cm1.x;
    if (qy & 2) s.y = -s.y, cm1.y = -cm1.y;
    cm1.x -= (qx & 1) ? 1.0f : (qx & 2) ? 2.0f : 0.0f;
    cm1.y -= (qy & 1) ? 1.0f : (qy & 2) ? 2.0f : 0.0f;
  }
}

template <int DIM>
struct ScalarLaw<CVWENO_KPP, DIM> {
  float sb, cb;  // sin(ubar), cos(ubar)
  __device__ __forceinline__ ScalarLaw(const StageArgs&, float ub) {
    float cm1;
    sin_cosm1_reduced(ub, sb, cm1);
    cb = 1.0f + cm1;
  }
  // sin(ub + d) - sin(ub) = sin(ub)(cos d - 1) + cos(ub) sin d, and likewise for cos.
  // Deviations inside a cell are mostly small: the series above; otherwise the reduced
  // series (sin_cosm1_reduced).
  __device__ __forceinline__ void flux_dev(float d, float& fx, float& fy) const {
    float s, cm1;
    if (fabsf(d) <= 1.0f) {
      sin_cosm1_small(d, s, cm1);
    } else {
      sin_cosm1_reduced(d, s, cm1);
    }
    fx = fmaf(sb, cm1, cb * s);
    fy = fmaf(cb, cm1, -sb * s);
  }
  __device__ __forceinline__ float flux_dev_dir(float d, int dir) const {
    float fx, fy;
    flux_dev(d, fx, fy);
    return dir == 0 ? fx : fy;
  }
  __device__ __forceinline__ void flux_dev2(f2 d, f2& fx, f2& fy) const {
    f2 s, cm1;
    sin_cosm1_2(d, s, cm1);
    fx = fma2(dup2(sb), cm1, mul2(dup2(cb), s));
    fy = fma2(dup2(cb), cm1, mul2(dup2(-sb), s));
  }
  __device__ __forceinline__ f2 flux_dev_dir2(f2 d, int dir) const {
    f2 s, cm1;
    sin_cosm1_2(d, s, cm1);
    return fma2(dup2(dir == 0 ? sb : cb), cm1, mul2(dup2(dir == 0 ? cb : -sb), s));
  }
  __device__ __forceinline__ float speed(float) const { return 1.0f; }
  __device__ __forceinline__ float nspeed(float u, int dir) const {
    return dir == 0 ? fabsf(cosf(u)) : fabsf(sinf(u));
  }
};

template <int DIM>
struct ScalarLaw<CVWENO_LINADV, DIM> {
  float vx, vy, ubar;
  __device__ __forceinline__ ScalarLaw(const StageArgs& a, float ub) : vx(a.adv_vx), vy(a.adv_vy), ubar(ub) {}
  __device__ __forceinline__ void flux_dev(float d, float& fx, float& fy) const {
    fx = vx * d;
    fy = vy * d;
  }
  __device__ __forceinline__ float flux_dev_dir(float d, int dir) const { return (dir == 0 ? vx : vy) * d; }
  __device__ __forceinline__ f2 flux_dev_dir2(f2 d, int dir) const { return mul2(dup2(dir == 0 ? vx : vy), d); }
  __device__ __forceinline__ void flux_dev2(f2 d, f2& fx, f2& fy) const {
    fx = mul2(dup2(vx), d);
    fy = mul2(dup2(vy), d);
  }
  __device__ __forceinline__ float speed(float) const { return DIM == 2 ? sqrtf(vx * vx + vy * vy) : fabsf(vx); }
  __device__ __forceinline__ float nspeed(float, int dir) const { return fabsf(dir == 0 ? vx : vy); }
};

// LLF flux in direction dir (0 = x, 1 = y) minus f(ubar) . n, from the left/lower
// state ubar + dL to the right/upper state ubar + dR (reading A14).
template <class Law>
__device__ __forceinline__ float llf_dev(const Law& law, const StageArgs& a, float ubar, float dL, float dR, int dir) {
  const float lam = a.lambda_const > 0.0f ? a.lambda_const
                                          : fmaxf(law.nspeed(ubar + dL, dir), law.nspeed(ubar + dR, dir));
  return 0.5f * (law.flux_dev_dir(dL, dir) + law.flux_dev_dir(dR, dir)) - 0.5f * lam * (dR - dL);
}

// The same at a pair of face nodes.
template <class Law>
__device__ __forceinline__ f2 llf_dev2(const Law& law, const StageArgs& a, float ubar, f2 dL, f2 dR, int dir) {
  f2 lam = dup2(a.lambda_const);
  if (!(a.lambda_const > 0.0f)) {
    lam.x = fmaxf(law.nspeed(ubar + dL.x, dir), law.nspeed(ubar + dR.x, dir));
    lam.y = fmaxf(law.nspeed(ubar + dL.y, dir), law.nspeed(ubar + dR.y, dir));
  }
  const f2 f = add2(law.flux_dev_dir2(dL, dir), law.flux_dev_dir2(dR, dir));
  return fma2(mul2(dup2(-0.5f), lam), sub2(dR, dL), mul2(dup2(0.5f), f));
}

// 4-byte asynchronous global -> shared copy (zero-filled when src_bytes == 0), so that a
// thread keeps all of its tile loads in flight at once instead of waiting on each.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int src_bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Programmatic dependent launch.  A stage kernel launched with programmatic stream
// serialisation may start while the previous kernel on its stream finishes: before
// pdl_wait() it touches only data that no kernel of the current step writes (the
// tabulation image, shared memory); pdl_wait() returns once the previous kernel has
// completed and its writes are visible.  pdl_launch_dependents() lets the next kernel
// start once every CTA of this one has passed it.  Both are no-ops without the launch
// attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// Host: launches kern with programmatic stream serialisation, so that it may start while
// the previous kernel on stream s finishes (the kernel must call pdl_wait() before it
// touches anything that kernel writes).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned); the
// zero-filling form copies src_bytes (0 or 16) and fills the rest with zeros.
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src));
}
__device__ __forceinline__ void cp_async16z(float* dst, const float* src, int src_bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(src_bytes));
}

// Starts the copy of R rows of W consecutive columns of a row-major global array (at src +
// off, nrow rows of ncol columns, each column E floats) into shared memory: row r, column c lands at
// dst[r * RS + ph[r] + c * E + e].  Global row r0 + r and column c0 + c wrap (periodic) or,
// outside the array, read as zeros.  The row's in-range columns are one run in global
// memory; ph[r] is its offset within a 16-byte chunk, so the run's whole chunks are copied
// 16 bytes at a time (src 16-byte aligned required) and only its head and tail (under 4
// floats each, 6 at most when the run has no whole chunk) and the wrapped or absent
// columns float by float.  One warp per row (rows of many chunks).  Requires
// RS >= W * E + 3; the copies land with the thread's next cp.async wait, the zeros and
// ph[] with the next barrier.
template <int E, int W, int R, int RS, int NT>
__device__ __forceinline__ void stage_rows16(float* dst, int* ph, const float* src, int ncol, int nrow, int c0,
                                             int r0, bool perc, bool perr, int* status, int64_t lim, int64_t off = 0) {
  static_assert(RS >= W * E + 3 && RS % 4 == 0, "staging row too short");
  constexpr int NW = NT / 32;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int c_lo = max(0, -c0), c_hi = min(W - 1, ncol - 1 - c0);  // in-range columns
  const int cr = max(c_hi + 1, c_lo), nout = (c_lo + W - cr) * E;  // columns [0, c_lo), [cr, W)
#pragma unroll 1
  for (int r = warp; r < R; r += NW) {
    int gr = r0 + r;
    bool row_ok = true;
    if (gr < 0 || gr >= nrow) {
      if (perr) gr = ((gr % nrow) + nrow) % nrow; else row_ok = false;
    }
    float* d = dst + r * RS;
    if (!row_ok) {
      for (int e = lane; e < W * E; e += 32) d[e] = 0.0f;
      if (lane == 0) ph[r] = 0;
      continue;
    }
    const int64_t gbase = off + ((int64_t)gr * ncol + c0) * E;  // global float of column 0
    const int p = (int)(gbase & 3);
    if (lane == 0) ph[r] = p;
    d += p;
    const int64_t dofs = (int64_t)r * RS + p - gbase;  // staging float of global float x: x + dofs
    // body: the whole 16-byte chunks of the in-range run [g0, g1)
    const int64_t g0 = gbase + (int64_t)c_lo * E, g1 = c_hi < c_lo ? g0 : gbase + (int64_t)(c_hi + 1) * E;
    const int64_t b0 = (g0 + 3) & ~(int64_t)3, b1 = g1 & ~(int64_t)3;
    const bool body = b0 < b1;
    if (body)
      for (int64_t x = b0 + 4 * lane; x < b1; x += 128)
        if (CVW_SPAN(status, x, 4, lim) && CVW_SPAN(status, x + dofs, 4, R * RS)) cp_async16(d + (x - gbase), src + x);
    // head and tail of the run (or the whole run when it has no whole chunk)
    const int nh = body ? (int)(b0 - g0) : (int)(g1 - g0), nt = body ? (int)(g1 - b1) : 0;
    if (lane < nh) {
      if (CVW_SPAN(status, g0 + lane, 1, lim) && CVW_SPAN(status, g0 + lane + dofs, 1, R * RS))
        cp_async4(d + (g0 + lane - gbase), src + g0 + lane, 4);
    } else if (lane < nh + nt) {
      if (CVW_SPAN(status, b1 + lane - nh, 1, lim) && CVW_SPAN(status, b1 + lane - nh + dofs, 1, R * RS))
        cp_async4(d + (b1 + lane - nh - gbase), src + b1 + lane - nh, 4);
    }
    for (int j = lane; j < nout; j += 32) {
      const int cj = j / E, e = j - cj * E;
      const int c = cj < c_lo ? cj : cr + (cj - c_lo);
      if (perc) {
        const int gc = ((c0 + c) % ncol + ncol) % ncol;
        if (CVW_SPAN(status, off + ((int64_t)gr * ncol + gc) * E + e, 1, lim) &&
            CVW_SPAN(status, (int64_t)r * RS + p + c * E + e, 1, R * RS))
          cp_async4(d + c * E + e, src + off + ((int64_t)gr * ncol + gc) * E + e, 4);
      } else {
        d[c * E + e] = 0.0f;
      }
    }
  }
}

// The same rows for NV arrays (array v at src + v * var, staged at dst + v * dstv, phases at ph +
// v * R) where every column is in range: a row is the 16-byte chunks that cover its run, the
// first up to 3 floats early (floats of the same array), the last zero-filled past the run, so
// one flat loop over the chunks serves them.  Rows outside the array wrap or read as zeros.
// Requires RS >= W * E + 6.
template <int E, int W, int R, int RS, int NT, int NV>
__device__ __forceinline__ void stage_rows16_inner(float* dst, int dstv, int* ph, const float* src, int64_t var, int ncol,
                                                   int nrow, int c0, int r0, bool perr, int* status, int64_t lim) {
  constexpr int NCH = (W * E + 6) / 4;
  static_assert(RS >= 4 * NCH && RS % 4 == 0, "staging row too short");
  for (int f = threadIdx.x; f < R * NCH; f += NT) {
    const int r = f / NCH, k = f - r * NCH;
    int gr = r0 + r;
    bool ok = true;
    if (gr < 0 || gr >= nrow) {
      if (perr) gr = ((gr % nrow) + nrow) % nrow; else ok = false;
    }
    const int64_t row = ((int64_t)gr * ncol + c0) * E;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int64_t g0 = v * var + row, c = (g0 & ~(int64_t)3) + 4 * k;
      const int left = (int)(g0 + W * E - c);
      const int n = !ok || left <= 0 ? 0 : left < 4 ? left : 4;
      const bool in = n > 0 && CVW_SPAN(status, c, n, lim);
      if (k == 0) ph[v * R + r] = (int)(g0 & 3);
      cp_async16z(dst + v * dstv + r * RS + 4 * k, in ? src + c : src, in ? 4 * n : 0);
    }
  }
}

// Ends a kernel that maximises x >= 0 over its threads (every thread calls it once): the block's
// maximum goes into the slots; the last block publishes the result with the status word
// and leaves the slots zero for the next call.
__device__ __forceinline__ void finish_max(float x, int* status, const MaxSlots& out) {
  __shared__ unsigned best;
  if (threadIdx.x == 0) best = 0;
  __syncthreads();
  const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(x));
  if ((threadIdx.x & 31) == 0) atomicMax(&best, w);
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicMax(out.best, best);
    __threadfence();
    if (atomicInc(out.done, gridDim.x - 1) == gridDim.x - 1) {  // back to zero by itself (sum_mode0_kernel)
      __threadfence();
      *out.max = (double)__uint_as_float(atomicExch(out.best, 0u));
      *out.status = atomicOr(status, 0);
    }
  }
}

}  // namespace cvw
