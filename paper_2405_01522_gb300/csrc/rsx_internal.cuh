// Internal declarations shared by the CUDA translation units of librsx.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#include "fft_small.cuh"

namespace rsx {

// The pair Poisson solve by pruned, zero-padded FFT convolution.  The potential of a pair
// density rho = f1 f2 on the box (nz, ny, nx) is
//     V = h^3/N_pad * IDFT( ghat * DFT(rho zero-padded to (2nz, 2ny, 2nx)) )
// restricted to the box (Sec. 3.1: Eq. 2's integral as a Poisson problem at O(N log N); padding
// twice the box makes the periodic convolution the isolated one).  Three passes:
//   pass 1  x forward, real-to-complex (two rows y, y+1 packed as one complex line), output
//           I[q][kx][z][y], kx in [0, Mx/2]: (Mx/2+1) nz ny complex      (poisson_xpass.cuh)
//   pass 2  per (q, kx): y forward on nz rows, z forward + multiply by ghat + z inverse on My
//           columns, y inverse keeping y < ny; in place on I             (poisson_pass2.cuh)
//   pass 3  per output p: x inverse complex-to-real of every pair of p's list, keeping x < nx,
//           and out_p -= partner * V (Eq. 2's sum over j)                (poisson_xpass.cuh)
// Only nz of the 2nz z-planes and ny of the 2ny rows are non-zero, so the x transforms run on
// nz ny rows and the y transforms on nz rows per kx; I is 4x smaller than a padded half
// spectrum.  The line transforms are in poisson_lines.cuh.

// Which pair densities a batch holds and which pairs each output accumulates.
//   PROD: pair q = b * na + a  has density A[a] * B[b]  (exchange: A = phi, B = psi;
//         Casida: A = virtual, B = occupied, so q = i * n_virt + a);
//         output p (an element of B) accumulates pairs q = p * na + a, partner A[a].
//   SYM:  unique pairs a <= b of one set A (upper triangle, row-major);
//         output p accumulates every pair containing p, partner the other orbital.
//   LIST: pairs and outputs of several independent orbital sets (the uneven batch):
//         pair q has density plist[2q] * plist[2q + 1]; output p is orbital i of a set of
//         nocc orbitals phi whose symmetric pairs start at q0 (SYM order within the set),
//         accumulates -sum_e phi_e V[phi_i phi_e] and is written to olist[p].out.
enum PairMode { kProd = 0, kSym = 1, kList = 2 };

template <typename R>
struct OutRef {
  const R* phi;   // the output's orbital set [nocc][N]
  R* out;         // the output array [N]
  int nocc, i, q0, pad;
};

template <typename R>
struct PairMap {
  int mode;
  const R* A;
  const R* B;
  int na, nb;
  size_t N;  // points per orbital
  const R* const* plist = nullptr;   // LIST: two orbital pointers per pair
  const OutRef<R>* olist = nullptr;  // LIST: one entry per output

  __device__ __forceinline__ void pair(int q, const R*& f1, const R*& f2) const {
    if (mode == kProd) {
      const int b = q / na, a = q - b * na;
      f1 = A + (size_t)a * N;
      f2 = B + (size_t)b * N;
    } else if (mode == kSym) {
      int i = 0, rem = q;
      while (rem >= na - i) { rem -= na - i; ++i; }
      f1 = A + (size_t)i * N;
      f2 = A + (size_t)(i + rem) * N;
    } else {
      f1 = plist[2 * q];
      f2 = plist[2 * q + 1];
    }
  }
  __device__ __forceinline__ int nentries(int p) const { return mode == kList ? olist[p].nocc : na; }
  // entry e of output p: pair index and the orbital multiplied into the accumulator
  __device__ __forceinline__ void entry(int p, int e, int& q, const R*& partner) const {
    if (mode == kProd) {
      q = p * na + e;
      partner = A + (size_t)e * N;
    } else if (mode == kSym) {
      const int i = p < e ? p : e, j = p < e ? e : p;
      q = i * na - i * (i - 1) / 2 + (j - i);
      partner = A + (size_t)e * N;
    } else {
      const OutRef<R> o = olist[p];
      const int i = o.i < e ? o.i : e, j = o.i < e ? e : o.i;
      q = o.q0 + i * o.nocc - i * (i - 1) / 2 + (j - i);
      partner = o.phi + (size_t)e * N;
    }
  }
  // the array output p (local index pl of a launch starting at out) is written to
  __device__ __forceinline__ R* out_row(int p, R* out, int pl) const {
    return mode == kList ? olist[p].out : out + (size_t)pl * N;
  }
};

struct Geom {
  int nz, ny, nx;     // box
  int Mz, My, Mx;     // padded (2n)
  int Az, Ay, Ax;     // M / 16
  int Hx;             // Mx / 2 + 1 (half spectrum along x)
  int smem_optin;     // shared memory a CTA may opt into on the context's device (bytes)
  int p1_group;       // tuning: pass-1 block order (0: pair-major; G > 0: pairs fastest in groups of G)
  int p2_global;      // tuning: 1 = the y/z pass keeps its work plane in global scratch even where
                      // shared memory would hold it (0 = shared memory whenever it fits)
  int* dbg = nullptr; // bounds-checked builds: the status word an out-of-range index is reported in
  bool pdl = false;   // launch the passes with programmatic stream serialisation (launch_pdl)
  int dbg_nq = 0;     // bounds-checked builds: pairs the launch's intermediate holds (0: unknown)
  __host__ __device__ size_t N() const { return (size_t)nz * ny * nx; }
  __host__ __device__ size_t inter_elems() const { return (size_t)Hx * nz * ny; }  // complex per pair
};

// Bounds-checked builds (-DRSX_CHECKED, `librsx_checked.so`): the FFT passes test the
// indices they compute against the arrays they address, report the first violation as
// RSX_EBOUNDS in the context's status word and skip the access.  In the normal build the
// test is the constant true and compiles away.
#ifdef RSX_CHECKED
__device__ inline bool in_range_checked(int* dbg, long long i, long long n) {
  if (i >= 0 && i < n) return true;
  if (dbg) atomicMax(dbg, 7);   // RSX_EBOUNDS
  return false;
}
#define RSX_IN_RANGE(g, i, n) ::rsx::in_range_checked((g).dbg, (long long)(i), (long long)(n))
#else
#define RSX_IN_RANGE(g, i, n) true
#endif

// Kernel attributes of the three passes for geometry g on the current device (once per context:
// the launchers below make no attribute calls).  ctas: resident CTAs per SM of pass 2's
// shared-memory variant.
template <typename R>
cudaError_t prepare_pass1(const Geom& g);
template <typename R>
cudaError_t prepare_pass2(const Geom& g, int* ctas);
template <typename R>
cudaError_t prepare_pass3(const Geom& g);

// ---- launchers (defined per precision in poisson_f32.cu / poisson_f64.cu)
template <typename R>
cudaError_t launch_pass1(const Geom& g, const PairMap<R>& pm, int q0, int nq, Cx<R>* inter,
                         const Cx<R>* twx, cudaStream_t s);
// twl: w_M^{-t k1}, t < lanes, k1 < M / lanes (lanes per line: 8, or 16 in FP32 at edge 112);
// vlanes: the kernel table in the y/z pass's lane order (launch_vhat_lanes)
template <typename R>
cudaError_t launch_pass2(const Geom& g, int nq, Cx<R>* inter, const Cx<R>* twl, const R* vlanes, R* gscratch, int grid,
                         cudaStream_t s);
template <typename R>
cudaError_t launch_pass3(const Geom& g, const PairMap<R>& pm, int q0, int p0, int np, int pot, const Cx<R>* inter,
                         const Cx<R>* twx, R* out, cudaStream_t s);
// forward y/z transform of each pair plane, weighted by sqrt(w_G vhat(G) h^3) and split
// into bf16 hi/lo of the K panel, tile-major [ld/64][nrb][128][64] (nrb row blocks of 128).
// tw8: w_M^{-t k1}, t < 8, k1 < M / 8; wl: launch_spectrum_weights
cudaError_t launch_spectrum_f32(const Geom& g, int nq, const Cx<float>* inter, const Cx<float>* tw8,
                                const float* wl, uint16_t* hi, uint16_t* lo, int nrb, cudaStream_t s);
// panel weights sqrt(w_kx vhat h^3) in lane order, spectrum_weight_elems(g) floats
size_t spectrum_weight_elems(const Geom& g);
cudaError_t launch_spectrum_weights(const Geom& g, const float* vhat, float h3, float* wl, cudaStream_t s);
template <typename R>
size_t pass2_smem_bytes(const Geom& g, bool* fits);
template <typename R>
size_t pass2_gscratch_bytes(const Geom& g, int grid);   // global plane scratch of a launch of `grid` CTAs
bool axis_supported(int A);

}  // namespace rsx
