// pass 1 (x forward) launchers, both precisions
#include "poisson_launch.cuh"
#include "poisson_xpass.cuh"

namespace rsx {

template <typename R, int A>
constexpr size_t pass1_smem() {
  using X = XWarp<R, A>;
  return sizeof(Cx<R>) * kXWarps * (size_t)(X::SCR > X::TILE ? X::SCR : X::TILE);
}

template <typename R>
cudaError_t prepare_pass1(const Geom& g) {
  switch (g.Ax) {
#define RSX_CASE(a) \
  case a: return set_smem(k_pass1<R, a>, pass1_smem<R, a>());
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t prepare_pass1<float>(const Geom&);
template cudaError_t prepare_pass1<double>(const Geom&);

template <typename R>
cudaError_t launch_pass1(const Geom& g, const PairMap<R>& pm, int q0, int nq, Cx<R>* inter,
                         const Cx<R>* twx, cudaStream_t s) {
  if (nq <= 0) return cudaSuccess;
  const long long noct = (long long)g.nz * (g.ny / 8), nob = (noct + kXWarps - 1) / kXWarps;
  const int G = g.p1_group > 0 ? (g.p1_group < nq ? g.p1_group : nq) : 0;
  Geom gg = g;
  gg.p1_group = G;
  const long long nblk = G > 0 ? (long long)((nq + G - 1) / G) * G * nob : nob * nq;
  if (nblk > 0x7fffffffLL) return cudaErrorInvalidValue;
  switch (g.Ax) {
#define RSX_CASE(a)                                                                                  \
  case a: {                                                                                          \
    const size_t smem = pass1_smem<R, a>();                                                           \
    auto k = k_pass1<R, a>;                                                                          \
    return launch_pdl(gg.pdl, k, nblk, 32 * kXWarps, smem, s, gg, pm, q0, nq, inter, twx);                   \
  }
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_pass1<float>(const Geom&, const PairMap<float>&, int, int, Cx<float>*,
                                         const Cx<float>*, cudaStream_t);
template cudaError_t launch_pass1<double>(const Geom&, const PairMap<double>&, int, int, Cx<double>*,
                                          const Cx<double>*, cudaStream_t);

bool axis_supported(int A) { return axis_supported_impl(A); }

}  // namespace rsx
