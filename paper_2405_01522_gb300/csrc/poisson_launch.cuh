// Launchers of the pair Poisson passes for one precision R (included once per TU).
#pragma once
#include <utility>

#include "poisson_pass2.cuh"

namespace rsx {

#define RSX_FOR_EACH_A(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(10) X(12) X(14)

inline bool axis_supported_impl(int A) {
  switch (A) {
#define RSX_CASE(a) case a: return true;
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return false;
  }
}

template <class K>
inline cudaError_t set_smem(K k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Launch, with programmatic stream serialisation (see pdl_wait) when pdl is set.  It pays where
// the passes are launch latency: a 32^3 Poisson solve takes 7.5 us instead of 14.3 in stream
// order.  Where every SM has work it costs: CTAs set up early take their places while the
// kernel before still runs, and the persistent pass 2 ends up unevenly dealt (96^3 x 512
// pairs 6.76 -> 6.89 ms, FP64 32^3 x 16 279 -> 349 us, the uneven batch 4.44 -> 4.75 ms); the
// line lies at one plane of pass 2 per SM (solve_pairs).
template <class... P, class... Q>
inline cudaError_t launch_pdl(bool pdl, void (*k)(P...), long long grid, int block, size_t smem, cudaStream_t s, Q&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, std::forward<Q>(args)...);
}

// ---- pass 2 (k_pass2): the plane in shared memory where it fits beside the line scratch
// (and p2_global does not ask otherwise), else in global scratch
template <typename R>
size_t pass2_smem_bytes(const Geom& g, bool* fits) {
  size_t sc = 0, pl = 0;
  switch (g.Ay) {
#define RSX_CASE(a)               \
  case a:                         \
    sc = p2_scratch_bytes<R, a>(); \
    pl = p2_plane_bytes<R, a>();   \
    break;
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: break;
  }
  const bool f = g.p2_global == 0 && sc + pl <= (size_t)g.smem_optin;
  if (fits) *fits = f;
  return f ? sc + pl : sc;
}

template <typename R>
size_t pass2_gscratch_bytes(const Geom& g, int grid) {
  return (size_t)grid * g.nz * p2_pitch<R>(g.Ay) * sizeof(Cx<R>);
}

// edges whose plane fits in shared memory: FP32 all, FP64 up to 64
template <typename R, int A>
inline auto pass2_kernel(bool dsmem) {
  if constexpr (p2_scratch_bytes<R, A>() + p2_plane_bytes<R, A>() <= 232448) {
    if (dsmem) return k_pass2<R, A, true>;
  }
  return k_pass2<R, A, false>;
}

// both variants (a context may switch p2_global)
template <typename R>
cudaError_t prepare_pass2(const Geom& g, int* ctas) {
  Geom gs = g;
  gs.p2_global = 0;
  bool fits = false;
  const size_t smem = pass2_smem_bytes<R>(gs, &fits);
  gs.p2_global = 1;
  const size_t smem_g = pass2_smem_bytes<R>(gs, nullptr);
  *ctas = 1;
  switch (g.Ay) {
#define RSX_CASE(a)                                                                                            \
  case a: {                                                                                                    \
    cudaError_t e = set_smem(pass2_kernel<R, a>(false), smem_g);                                               \
    if (e != cudaSuccess || !fits) return e;                                                                   \
    auto k = pass2_kernel<R, a>(true);                                                                         \
    e = set_smem(k, smem);                                                                                     \
    int nb = 0;                                                                                                \
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, p2_threads<R>(a), smem);   \
    *ctas = nb > 0 ? nb : 1;                                                                                   \
    return e;                                                                                                  \
  }
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}

template <typename R>
cudaError_t launch_pass2(const Geom& g, int nq, Cx<R>* inter, const Cx<R>* twl, const R* vlanes, R* gscratch, int grid,
                         cudaStream_t s) {
  if (nq <= 0) return cudaSuccess;
  if (g.Ay != g.Az) return cudaErrorInvalidValue;
  bool fits = false;
  const size_t smem = pass2_smem_bytes<R>(g, &fits);
  if (!fits && gscratch == nullptr) return cudaErrorInvalidValue;
  switch (g.Ay) {
#define RSX_CASE(a)                                                                                  \
  case a: {                                                                                          \
    auto k = pass2_kernel<R, a>(fits);                                                               \
    return launch_pdl(g.pdl, k, grid, p2_threads<R>(a), smem, s, g, nq, inter, twl, vlanes, (Cx<R>*)gscratch); \
  }
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rsx
