// pass 3 (x inverse + exchange accumulation) launchers, both precisions
#include "poisson_launch.cuh"
#include "poisson_xpass.cuh"

namespace rsx {

template <typename R, int A>
constexpr size_t pass3_smem() {
  using X = XWarp<R, A>;
  return sizeof(Cx<R>) * kXWarps * (size_t)(X::SCR + X::TILE);
}

template <typename R>
cudaError_t prepare_pass3(const Geom& g) {
  switch (g.Ax) {
#define RSX_CASE(a) \
  case a: return set_smem(k_pass3<R, a>, pass3_smem<R, a>());
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t prepare_pass3<float>(const Geom&);
template cudaError_t prepare_pass3<double>(const Geom&);

template <typename R>
cudaError_t launch_pass3(const Geom& g, const PairMap<R>& pm, int q0, int p0, int np, int pot, const Cx<R>* inter,
                         const Cx<R>* twx, R* out, cudaStream_t s) {
  if (np <= 0) return cudaSuccess;
  const long long noct = (long long)g.nz * (g.ny / 8), nblk = (noct + kXWarps - 1) / kXWarps * np;
  if (nblk > 0x7fffffffLL) return cudaErrorInvalidValue;
  switch (g.Ax) {
#define RSX_CASE(a)                                                                                  \
  case a: {                                                                                          \
    const size_t smem = pass3_smem<R, a>();                                                           \
    auto k = k_pass3<R, a>;                                                                          \
    return launch_pdl(g.pdl, k, nblk, 32 * kXWarps, smem, s, g, pm, q0, p0, np, pot, inter, twx, out);      \
  }
    RSX_FOR_EACH_A(RSX_CASE)
#undef RSX_CASE
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_pass3<float>(const Geom&, const PairMap<float>&, int, int, int, int, const Cx<float>*,
                                         const Cx<float>*, float*, cudaStream_t);
template cudaError_t launch_pass3<double>(const Geom&, const PairMap<double>&, int, int, int, int, const Cx<double>*,
                                          const Cx<double>*, double*, cudaStream_t);

}  // namespace rsx
