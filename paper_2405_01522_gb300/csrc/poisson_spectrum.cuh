// Casida pair spectra: y and z forward transforms of each transition's x spectrum, weighted,
// split into bf16 hi + lo and written to the K panel (poisson_lines.cuh, poisson_pass2.cuh).
#pragma once
#include <cuda_bf16.h>

#include "poisson_pass2.cuh"

namespace rsx {

// Lines per CTA (8 lanes each) and CTAs per SM asked of the compiler.  Without the z inverse A = 14
// pays on 8 lanes here: 56 lines (128 registers a thread, 416 bytes of spill stores) take 16.1 us
// per transition at 112^3, 28 lines 36; 16 lanes x A took 20.6.
__host__ __device__ constexpr int spec_lines(int A) { return A == 14 ? 56 : A == 10 ? 40 : p2_lines<float>(A); }
__host__ __device__ constexpr int spec_min_ctas(int A) { return p2_min_ctas<float>(A); }
__host__ __device__ constexpr int spec_pitch(int A) { return 16 * A + 2; }   // as p2_pitch on 8 lanes
__host__ __device__ constexpr int spec_groups(int A) { return A >= 8 ? 1 : line_j(A); }

// Persistent grid over (kx, transition q), transitions fastest: the CTAs in flight fill the same
// 128 x 64 panel tiles (rows = transitions).  Per plane: y forward of the nz rows into the work
// plane, then z forward of the My columns; the spectra leave registers as
//   S_q(G) = sqrt(w_kx ghat(G) h^6 / N_pad) (Re, Im) R_q(G), w = 1 at kx = 0, Mx/2 and 2 otherwise,
// split into bf16 hi + lo.  K sums over G, so the order of G along a panel row is free: within a
// column (kx, ky) it is the lanes' own, 16-byte pieces (four complex) with the eight lanes of
// a line adjacent -- piece (2 j + h) 8 + s holds k2 = 4 h .. 4 h + 3 of row s + 8 j (the last,
// partial group of R = 2A mod 8 rows: h R + s) -- so that a line's store is one 128-byte line of a
// panel tile and no transpose back to natural order is needed.  wl holds the weights in pass
// 2's lane order (k_vhat_lanes).  The next plane's rows are loaded into registers before the
// barrier that frees the work plane.
template <int A>
__global__ void __launch_bounds__(8 * spec_lines(A), spec_min_ctas(A))
    k_spectrum(Geom g, int nq, const Cx<float>* __restrict__ inter, const Cx<float>* __restrict__ tw8,
               const float* __restrict__ wl, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo, int nrb) {
  using S = Split8<float, A, spec_groups(A)>;
  constexpr int NL = spec_lines(A), NB = 8 * A, M = 16 * A, A2 = 2 * A, DP = spec_pitch(A), FROW = 8 * S::FAC;
  constexpr int RF = A2 % 8;   // rows of the last, partial group (0: none)
  static_assert(NB % NL == 0 && NL % 4 == 0, "lines per CTA: whole warps, a divisor of the edge");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cx<float>* scr = reinterpret_cast<Cx<float>*>(smem_raw);
  Cx<float>* D = scr + NL * S::SCR;
  const int lane = threadIdx.x & 31, t = lane & 7, line = threadIdx.x >> 3, l = line & 3;
  const unsigned lmask = 0xFFu << (lane & 24);
  const int lrow = (line | 7) < NL ? (line & ~7) | ((line >> 1) & 3) | ((line & 1) << 2) : line;   // as pass 2
  Cx<float>* sc = scr + line * S::SCR;
  typename S::Tw tw;
  tw.init(tw8, t);
  const int Hy = M / 2 + 1;
  const int nplane = NB * NB;
  const int nwork = nq * g.Hx;
  auto plane_ptr = [&](int w) -> const Cx<float>* {
    if (w >= nwork) return nullptr;
    const int kx = w / nq, ql = w - kx * nq;
    return inter + (size_t)ql * g.inter_elems() + (size_t)kx * nplane;
  };
  Cx<float> v[A];
  auto load_row = [&](const Cx<float>* P, int z) {
#pragma unroll
    for (int a = 0; a < A; ++a) v[a] = P[(size_t)z * NB + t + 8 * a];
  };
  const size_t kb_stride = (size_t)nrb * 8192;
  const Cx<float>* P = plane_ptr(blockIdx.x);
  if (P) load_row(P, lrow);
  for (int w = blockIdx.x; P != nullptr; w += gridDim.x) {
    const int kx = w / nq, ql = w - kx * nq;
    const Cx<float>* Pn = plane_ptr(w + (int)gridDim.x);
    for (int z = lrow; z < NB; z += NL) {
      if (z != lrow) load_row(P, z);
      Cx<float>* row = D + z * DP;
      S::forward(v, t, l, lmask, tw, sc, [&](int k, Cx<float> x) { row[k] = x; });
    }
    __syncthreads();
    // tile-major panel [ld/64][nrb][128][64]: column g of row ql is at
    // ((g / 64) nrb + ql / 128) 8192 + (ql % 128) 64 + g % 64
    const size_t row_off = (size_t)(ql / 128) * 8192 + (size_t)(ql % 128) * 64;
    for (int ky = line; ky < M; ky += NL) {
      const int iy = ky <= M / 2 ? ky : M - ky;
      const float4* wsrc = reinterpret_cast<const float4*>(wl + ((size_t)kx * Hy + iy) * FROW) + t;
      const size_t g0 = ((size_t)kx * M + ky) * (2 * M);
      Cx<float> c[A];
#pragma unroll
      for (int a = 0; a < A; ++a) c[a] = D[(t + 8 * a) * DP + ky];
      S::forward_rows(c, t, l, lmask, tw, sc, [&](int j, int, const Cx<float>(&u)[8]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 m = __ldg(wsrc + (2 * j + h) * 8);
          const float f[4] = {m.x, m.y, m.z, m.w};
          const int piece = (RF != 0 && 8 * j + 8 > A2) ? 16 * j + h * RF + t : (2 * j + h) * 8 + t;
          const size_t gq = g0 + 8 * (size_t)piece;
          const size_t off = (gq / 64) * kb_stride + row_off + (gq % 64);
          uint32_t hv[4], lv[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            // round-to-nearest-even hardware conversions (re in the low half, im in the high)
            const Cx<float> x = cscale(u[4 * h + q], f[q]);
            const __nv_bfloat162 h2 = __float22bfloat162_rn(make_float2(x.x, x.y));
            const float2 hf = __bfloat1622float2(h2);
            const __nv_bfloat162 l2 = __float22bfloat162_rn(make_float2(x.x - hf.x, x.y - hf.y));
            hv[q] = *reinterpret_cast<const uint32_t*>(&h2);
            lv[q] = *reinterpret_cast<const uint32_t*>(&l2);
          }
          *reinterpret_cast<uint4*>(hi + off) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
          *reinterpret_cast<uint4*>(lo + off) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
        }
      });
    }
    P = Pn;
    if (P) load_row(P, lrow);
    __syncthreads();   // every read of D is done
  }
}

}  // namespace rsx
