// Casida pair-spectrum launcher (fp32 spectra, bf16 hi/lo panel)
#include "dense.cuh"
#include "poisson_launch.cuh"
#include "poisson_spectrum.cuh"

namespace rsx {

// wsq[kx][iy][iz] = sqrt(w_kx * vhat[kx][iy][iz] * h^3), w = 1 at kx = 0, Mx/2 and 2
// otherwise (vhat = ghat h^3 / N_pad): the Casida panel weights
static __global__ void k_spectrum_weights(const float* __restrict__ vhat, int Hx, int Hy, int Hz, int Mx, float h3,
                                   float* __restrict__ wsq) {
  const size_t n = (size_t)Hx * Hy * Hz;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int kx = (int)(i / ((size_t)Hy * Hz));
    const float w = (kx == 0 || 2 * kx == Mx) ? 1.0f : 2.0f;
    wsq[i] = sqrtf(w * vhat[i] * h3);
  }
}

size_t spectrum_weight_elems(const Geom& g) {
  const size_t rows = (size_t)g.Hx * (g.My / 2 + 1);
  return rows * 64 * line_j(g.Az) + rows * (g.Mz / 2 + 1);
}

cudaError_t launch_spectrum_weights(const Geom& g, const float* vhat, float h3, float* wl, cudaStream_t s) {
  float* wsq = wl + (size_t)g.Hx * (g.My / 2 + 1) * 64 * line_j(g.Az);   // folded weights behind the lane-order ones
  k_spectrum_weights<<<512, 256, 0, s>>>(vhat, g.Hx, g.My / 2 + 1, g.Mz / 2 + 1, g.Mx, h3, wsq);
  return launch_lane_order<float>(g, wsq, wl, 8, s);
}

cudaError_t launch_spectrum_f32(const Geom& g, int nq, const Cx<float>* inter, const Cx<float>* tw8,
                                const float* wl, uint16_t* hi, uint16_t* lo, int nrb, cudaStream_t s) {
  if (nq <= 0) return cudaSuccess;
  if (g.Ay != g.Az) return cudaErrorInvalidValue;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const long long nwork = (long long)nq * g.Hx;
  switch (g.Ay) {
#define RSX_CASE(a)                                                                                  \
  case a: {                                                                                          \
    using S = Split8<float, a, spec_groups(a)>;                                                      \
    const int nt = 8 * spec_lines(a);                                                                \
    const size_t smem = sizeof(Cx<float>) * ((size_t)spec_lines(a) * S::SCR + (size_t)(8 * a) * spec_pitch(a)); \
    auto k = k_spectrum<a>;                                                                          \
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    if (e != cudaSuccess) return e;                                                                  \
    int per_sm = 1;                                                                                  \
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nt, smem) != cudaSuccess) {        \
      cudaGetLastError();                                                                            \
      per_sm = 1;                                                                                    \
    }                                                                                                \
    const long long cap = (long long)(per_sm > 0 ? per_sm : 1) * nsm;                                \
    const int grid = (int)(nwork < cap ? nwork : cap);                                               \
    k<<<grid, nt, smem, s>>>(g, nq, inter, tw8, wl, hi, lo, nrb);                                    \
    return cudaGetLastError();                                                                       \
  }
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rsx
