// Instantiations of the fused scalar stage kernel for uniform quadrilateral meshes.
#include "dg_scalar_launch.cuh"

namespace cvw {

cudaError_t launch_stage_1d(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s);
cudaError_t launch_stage_surrogate(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s);

cudaError_t launch_stage(const cvweno_mesh_s* m, const StageArgs& a, cudaStream_t s) {
  if (m->dim == 1) return launch_stage_1d(m, a, s);
  if ((a.mlp && !(a.mode & kModeLimit)) || (a.mode & kModeFeatures)) return launch_stage_surrogate(m, a, s);
  constexpr int TX = 16, TY = 8;
  if (m->tensor_cores && m->p == 3) {
    switch (m->desc.system) {
      case CVWENO_BURGERS: return launch_scalar_tc<CVWENO_BURGERS>(m, a, s);
      case CVWENO_KPP: return launch_scalar_tc<CVWENO_KPP>(m, a, s);
      case CVWENO_LINADV: return launch_scalar_tc<CVWENO_LINADV>(m, a, s);
      default: return cudaErrorNotSupported;
    }
  }
  switch (m->p * 10 + m->desc.system) {
    case 10 + CVWENO_BURGERS: return launch_scalar<2, 1, CVWENO_BURGERS, TX, TY>(m, a, s);
    case 20 + CVWENO_BURGERS: return launch_scalar<2, 2, CVWENO_BURGERS, TX, TY>(m, a, s);
    case 30 + CVWENO_BURGERS: return launch_scalar<2, 3, CVWENO_BURGERS, TX, TY>(m, a, s);
    case 40 + CVWENO_BURGERS: return launch_scalar<2, 4, CVWENO_BURGERS, TX, TY>(m, a, s);
    case 10 + CVWENO_KPP: return launch_scalar<2, 1, CVWENO_KPP, TX, TY>(m, a, s);
    case 20 + CVWENO_KPP: return launch_scalar<2, 2, CVWENO_KPP, TX, TY>(m, a, s);
    case 30 + CVWENO_KPP: return launch_scalar<2, 3, CVWENO_KPP, TX, TY>(m, a, s);
    case 40 + CVWENO_KPP: return launch_scalar<2, 4, CVWENO_KPP, TX, TY>(m, a, s);
    case 10 + CVWENO_LINADV: return launch_scalar<2, 1, CVWENO_LINADV, TX, TY>(m, a, s);
    case 20 + CVWENO_LINADV: return launch_scalar<2, 2, CVWENO_LINADV, TX, TY>(m, a, s);
    case 30 + CVWENO_LINADV: return launch_scalar<2, 3, CVWENO_LINADV, TX, TY>(m, a, s);
    case 40 + CVWENO_LINADV: return launch_scalar<2, 4, CVWENO_LINADV, TX, TY>(m, a, s);
    default: return cudaErrorNotSupported;
  }
}

namespace {
template <int DIM, int P>
cudaError_t packed_image(const void* t, float* dst, cudaStream_t s) {
  packed_image_kernel<DIM, P><<<1, 256, 0, s>>>(*static_cast<const DgTables<DIM, P>*>(t), dst);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_packed_image(int dim, int p, const void* t, float* dst, cudaStream_t s) {
  if (!t || !dst) return cudaErrorInvalidValue;
  switch (dim * 10 + p) {
    case 11: return packed_image<1, 1>(t, dst, s);
    case 12: return packed_image<1, 2>(t, dst, s);
    case 13: return packed_image<1, 3>(t, dst, s);
    case 14: return packed_image<1, 4>(t, dst, s);
    case 21: return packed_image<2, 1>(t, dst, s);
    case 22: return packed_image<2, 2>(t, dst, s);
    case 23: return packed_image<2, 3>(t, dst, s);
    case 24: return packed_image<2, 4>(t, dst, s);
    default: return cudaErrorNotSupported;
  }
}

namespace {
// max lambda_e over the volume and face Gauss nodes: one thread per cell, its coefficients in
// registers.
constexpr int kSpeedThreads = 128;
template <int DIM, int P, int SYS>
__global__ void __launch_bounds__(kSpeedThreads)
    scalar_wavespeed_kernel(const __grid_constant__ StageArgs a, const __grid_constant__ MaxSlots out) {
  using Img = PackedImage<DIM, P>;
  constexpr int N = Img::N, NY1 = Img::NY1, MP = Img::MP, ND = N * NY1;
  __shared__ __align__(16) float img[Img::FLOATS];
  for (int f = threadIdx.x; f < Img::FLOATS; f += kSpeedThreads) img[f] = a.pk_img[f];
  __syncthreads();
  const int64_t ncell = (int64_t)a.nx * (DIM == 2 ? a.ny : 1);
  float lam = 0.0f;
  for (int64_t cell = (int64_t)blockIdx.x * kSpeedThreads + threadIdx.x; cell < ncell;
       cell += (int64_t)gridDim.x * kSpeedThreads) {
    if (!CVW_SPAN(a.status, cell * ND, ND, a.lim_in)) continue;
    f2 c[NY1][MP];
#pragma unroll
    for (int my = 0; my < NY1; ++my)
#pragma unroll
      for (int p = 0; p < MP; ++p)
        c[my][p] = mk2(a.u_in[cell * ND + 2 * p + N * my], 2 * p + 1 < N ? a.u_in[cell * ND + 2 * p + 1 + N * my] : 0.0f);
    const float ubar = c[0][0].x;
    c[0][0].x = 0.0f;
    const ScalarLaw<SYS, DIM> law(a, ubar);
    lam = fmaxf(lam, cell_speed<DIM, P>(img, law, ubar, c));
  }
  finish_max(lam, a.status, out);
}

template <int DIM, int P>
cudaError_t launch_wavespeed_t(int system, const StageArgs& a, const MaxSlots& out, cudaStream_t s) {
  const int64_t ncell = (int64_t)a.nx * (DIM == 2 ? a.ny : 1), n = (ncell + kSpeedThreads - 1) / kSpeedThreads;
  const unsigned blocks = (unsigned)(n < 1216 ? n : 1216);  // 8 per SM
  switch (system) {
    case CVWENO_BURGERS: scalar_wavespeed_kernel<DIM, P, CVWENO_BURGERS><<<blocks, kSpeedThreads, 0, s>>>(a, out); break;
    case CVWENO_LINADV: scalar_wavespeed_kernel<DIM, P, CVWENO_LINADV><<<blocks, kSpeedThreads, 0, s>>>(a, out); break;
    case CVWENO_KPP:
      if constexpr (DIM == 2) {
        scalar_wavespeed_kernel<DIM, P, CVWENO_KPP><<<blocks, kSpeedThreads, 0, s>>>(a, out);
        break;
      }
      return cudaErrorNotSupported;
    default: return cudaErrorNotSupported;
  }
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_wavespeed_scalar(const cvweno_mesh_s* m, const StageArgs& a, const MaxSlots& out, cudaStream_t s) {
  switch (m->dim * 10 + m->p) {
    case 11: return launch_wavespeed_t<1, 1>(m->desc.system, a, out, s);
    case 12: return launch_wavespeed_t<1, 2>(m->desc.system, a, out, s);
    case 13: return launch_wavespeed_t<1, 3>(m->desc.system, a, out, s);
    case 14: return launch_wavespeed_t<1, 4>(m->desc.system, a, out, s);
    case 21: return launch_wavespeed_t<2, 1>(m->desc.system, a, out, s);
    case 22: return launch_wavespeed_t<2, 2>(m->desc.system, a, out, s);
    case 23: return launch_wavespeed_t<2, 3>(m->desc.system, a, out, s);
    case 24: return launch_wavespeed_t<2, 4>(m->desc.system, a, out, s);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace cvw

namespace cvw {
namespace {
// sin d and cos d - 1 as the KPP flux forms them (sin_cosm1_2, both halves).
__global__ void kpp_sincos_kernel(const float* __restrict__ d, float* __restrict__ out, int n) {
  for (int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 2 * gridDim.x * blockDim.x) {
    f2 s, cm1;
    sin_cosm1_2(mk2(d[i], i + 1 < n ? d[i + 1] : 0.0f), s, cm1);
    out[i] = s.x;
    out[n + i] = cm1.x;
    if (i + 1 < n) out[i + 1] = s.y, out[n + i + 1] = cm1.y;
  }
}
}  // namespace
}  // namespace cvw

extern "C" cvweno_status cvweno_kpp_sincos(const float* d, float* out, int n, void* stream) {
  if (n < 0 || (n > 0 && (!d || !out))) return CVWENO_ERR_ARG;
  if (n == 0) return CVWENO_OK;
  const int threads = 256, blocks = (n + threads - 1) / threads < 1024 ? (n + threads - 1) / threads : 1024;
  cvw::kpp_sincos_kernel<<<blocks, threads, 0, static_cast<cudaStream_t>(stream)>>>(d, out, n);
  return cudaGetLastError() == cudaSuccess ? CVWENO_OK : CVWENO_ERR_CUDA;
}
