// Pass 2 of the pair Poisson solve: per (pair, kx) plane, y forward on the nz rows, z
// forward x kernel x z inverse on the My columns, y inverse keeping y < ny; in place on the
// intermediate.  Line transforms on 8 lanes x 2A (poisson_lines.cuh).
#pragma once
#include "poisson_lines.cuh"

namespace rsx {

// Launch shape per precision and edge 8 A: lines per CTA (8 lanes each, 16 for FP32 A = 14; a
// divisor of the edge, so that every line has the same rows and columns), CTAs per SM asked of
// the compiler, and the 8-row groups of a line's scratch held at a time.  FP32, us per pair at
// 128 pairs: several CTAs per SM cover each other's barriers where the planes fit (A = 8: 2.87
// as 2 x 256 threads, 3.10 as 1 x 512; A = 7: 2.21 at 2 x 224, 2.51 at 3 x 224, which spills;
// A = 6 at 3 CTAs spills 44 bytes, A = 4 4 bytes; fewer CTAs were not measured there);
// at A = 12 the plane allows one CTA and 48 lines (12 warps) beat 32 once the scratch holds one
// group (10.08 us; 10.42 at 32 lines, 11.14 with all three groups in scratch).
template <typename R>
__host__ __device__ constexpr int p2_lines(int A) {
  return sizeof(R) == 4 ? (A == 2 ? 16 : A == 3 ? 24 : A == 4 ? 32 : A == 5 ? 20 : A == 6 ? 24 : A == 7 ? 28
                           : A == 8 ? 32 : A == 10 ? 40 : A == 12 ? 48 : 16)
                        : (A == 2 ? 16 : A == 3 ? 24 : A == 4 ? 32 : A == 5 ? 20 : A == 6 ? 24 : A == 7 ? 28
                           : A == 8 ? 32 : A == 10 ? 20 : A == 12 ? 24 : 28);
}
template <typename R>
__host__ __device__ constexpr int p2_min_ctas(int A) {
  return sizeof(R) == 4 ? (A == 2 ? 6 : A == 3 ? 4 : A == 4 ? 3 : A == 5 ? 4 : A == 6 ? 3 : A <= 8 ? 2 : 1)
                        : (A == 2 ? 3 : A <= 5 ? 2 : 1);
}
template <typename R>
__host__ __device__ constexpr int p2_groups(int A) { return sizeof(R) == 4 && A >= 8 ? 1 : line_j(A); }

template <typename R, int A, bool L16 = (sizeof(R) == 4 && A == 14)>
struct P2Split {
  using type = Split8<R, A, p2_groups<R>(A), !(sizeof(R) == 8 && A >= 10)>;
};
template <typename R, int A>
struct P2Split<R, A, true> {
  using type = Split16<A>;
};
template <typename R>
__host__ __device__ constexpr int p2_lanes(int A) { return sizeof(R) == 4 && A == 14 ? 16 : 8; }
template <typename R>   // values of the lane-order kernel table per folded column
__host__ __device__ constexpr int p2_row_factors(int A) { return p2_lanes<R>(A) == 16 ? 256 : 64 * line_j(A); }
template <typename R>
__host__ __device__ constexpr int p2_threads(int A) { return p2_lanes<R>(A) * p2_lines<R>(A); }

// Row pitch of the work plane (complex).  FP32, 8 lanes: M + 2; bank pairs (8-byte units) of
// an access are then 2 row + column mod 16: the two lines of a half-warp take rows 4 apart (the
// 8 consecutive columns of a row access land 8 bank pairs apart) and z columns 1 apart (the
// 8 rows t + 8 a of a column access fall on even bank pairs for one line, odd ones for the
// other).  Otherwise M + 1: rows and columns conflict-free.
template <typename R>
__host__ __device__ constexpr int p2_pitch(int A) { return 16 * A + (sizeof(R) == 4 && A != 14 ? 2 : 1); }

template <typename R, int A>
constexpr size_t p2_scratch_bytes() { return sizeof(Cx<R>) * (size_t)p2_lines<R>(A) * P2Split<R, A>::type::SCR; }
template <typename R, int A>
constexpr size_t p2_plane_bytes() { return sizeof(Cx<R>) * (size_t)(8 * A) * p2_pitch<R>(A); }

// four spectra times four kernel factors
__device__ __forceinline__ void p2_scale4(Cx<float>* u, float4 m) {
  u[0] = cscale(u[0], m.x);
  u[1] = cscale(u[1], m.y);
  u[2] = cscale(u[2], m.z);
  u[3] = cscale(u[3], m.w);
}

// Persistent grid over the work items (pair, kx).  The work plane D lives in shared memory
// (DSMEM) or in a per-CTA slice of global scratch.  A row of D belongs to one line in both y
// loops, so that the y inverse of a plane and the y forward of the CTA's next plane run as one
// loop over rows without a barrier between them: the line loads its next input row into
// registers, inverts the row it holds, and writes the new spectrum over it.  (With the next
// plane staged through shared memory behind the y inverse, its load was exposed once per
// plane and a plane took four barriers instead of two.)
// tw[k1][t] = w_M^{-t k1} (t < 8, k1 < 2A; 16 lanes: t < 16, k1 < A); vl: the kernel table in
// the split's lane order, FAC values per lane and folded column, the lanes' 16-byte pieces
// adjacent (k_vhat_lanes).
// Shared memory: [line scratch] [plane NB x p2_pitch].
template <typename R, int A, bool DSMEM>
__global__ void __launch_bounds__(p2_threads<R>(A), p2_min_ctas<R>(A))
    k_pass2(Geom g, int nq, Cx<R>* inter, const Cx<R>* __restrict__ twg, const R* __restrict__ vl,
            Cx<R>* gscratch) {
  using S = typename P2Split<R, A>::type;
  constexpr int NL = p2_lines<R>(A), LN = S::LANES, NIN = S::NIN;
  constexpr int NB = 8 * A, M = 16 * A, DP = p2_pitch<R>(A), FROW = LN * S::FAC;
  constexpr bool kAhead = !(sizeof(R) == 8 && A >= 10);   // the next input row is loaded before the y inverse (registers permitting)
  static_assert(NB % NL == 0 && NL * LN % 32 == 0, "lines per CTA: whole warps, a divisor of the edge");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cx<R>* scr = reinterpret_cast<Cx<R>*>(smem_raw);
  Cx<R>* D = DSMEM ? scr + NL * S::SCR : gscratch + (size_t)blockIdx.x * NB * DP;
  const int lane = threadIdx.x & 31, t = lane & (LN - 1), line = threadIdx.x / LN, l = line & 3;
  const unsigned lmask = (LN == 8 ? 0xFFu : 0xFFFFu) << (lane & (32 - LN));
  // the two lines of a half-warp (line 2k, 2k + 1) take rows 4 apart and columns 1 apart, see
  // p2_pitch (the last four lines of an odd half block of 8 keep their own rows)
  const int lrow = LN == 8 && (line | 7) < NL ? (line & ~7) | ((line >> 1) & 3) | ((line & 1) << 2) : line;
  Cx<R>* sc = scr + line * S::SCR;
  typename S::Tw tw;
  tw.init(twg, t);   // tables are written once, by rsx_create
  pdl_launch();
  pdl_wait();
  const int Hy = M / 2 + 1;
  const int nplane = NB * NB;
  const int nwork = nq * g.Hx;
  // plane of work item w, null past the last one
  auto plane_ptr = [&](int w) -> Cx<R>* {
    if (w >= nwork) return nullptr;
    const int ql = w / g.Hx, kx = w - ql * g.Hx;
    if (!RSX_IN_RANGE(g, (long long)ql * g.inter_elems() + (long long)(kx + 1) * nplane - 1,
                      (long long)nq * g.inter_elems()))
      return nullptr;
    return inter + (size_t)ql * g.inter_elems() + (size_t)kx * nplane;
  };
  Cx<R> v[NIN];   // this lane's inputs of a y row
  auto load_row = [&](const Cx<R>* P, int z) {
#pragma unroll
    for (int a = 0; a < NIN; ++a) v[a] = P[(size_t)z * NB + t + LN * a];
  };
  auto y_forward = [&](int z) {   // outputs all M columns
    Cx<R>* row = D + z * DP;
    S::forward(v, t, l, lmask, tw, sc, [&](int k, Cx<R> x) { row[k] = x; });
  };
  Cx<R>* P = plane_ptr(blockIdx.x);
  if (P) {
    for (int z = lrow; z < NB; z += NL) {
      load_row(P, z);
      y_forward(z);
    }
  }
  for (int w = blockIdx.x; P != nullptr; w += gridDim.x) {
    const int kx = w % g.Hx;
    Cx<R>* Pn = plane_ptr(w + (int)gridDim.x);
    __syncthreads();
    // ---- z forward, kernel multiply, z inverse on the M columns ky.  Columns ky and M - ky
    // use the same kernel factors (the table is folded in |ky|): a line takes them as one
    // item (item 0: the two unpaired columns 0 and M / 2) and loads the factors once.
    constexpr int E = 16 / (int)sizeof(R);   // values per 16-byte piece
    const R* vrow = vl + (size_t)kx * Hy * FROW + t * E;
    for (int it = line; it < M / 2; it += NL) {
      float4 fac[S::FAC / 4];
#pragma unroll 1
      for (int c = 0; c < 2; ++c) {
        const int ky = c == 0 ? it : (it == 0 ? M / 2 : M - it);
        const R* vsrc = vrow + (size_t)(it == 0 ? ky : it) * FROW;
        if constexpr (sizeof(R) == 4) {
          if (c == 0 || it == 0) {
#pragma unroll
            for (int i = 0; i < S::FAC / 4; ++i) fac[i] = __ldg(reinterpret_cast<const float4*>(vsrc) + i * LN);
          }
        }
        Cx<R>* col = D + ky;
        S::convolve(
            t, l, lmask, tw, sc, [&](int i) { return col[i * DP]; },
            [&](int j, Cx<R>(&u)[S::RAD]) {
              if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int q = 0; q < S::RAD / 4; ++q) p2_scale4(u + 4 * q, fac[j * (S::RAD / 4) + q]);
              } else {
#pragma unroll
                for (int k2 = 0; k2 < S::RAD; k2 += 2) {
                  const double2 m = __ldg(reinterpret_cast<const double2*>(vsrc) + (S::RAD * j + k2) / 2 * LN);
                  u[k2] = cscale(u[k2], m.x);
                  u[k2 + 1] = cscale(u[k2 + 1], m.y);
                }
              }
            },
            [&](int i, Cx<R> x) { col[i * DP] = x; });
      }
    }
    __syncthreads();
    // ---- y inverse of the nz rows, keeping y < ny, from registers straight to the plane in
    // global memory; then the y forward of the next plane's row into the freed row of D
    for (int z = lrow; z < NB; z += NL) {
      if (kAhead && Pn) load_row(Pn, z);
      const Cx<R>* row = D + z * DP;
      Cx<R>* dst = P + (size_t)z * NB;
      S::inverse(t, l, lmask, tw, sc, [&](int k) { return row[k]; }, [&](int i, Cx<R> x) { dst[i] = x; });
      if (Pn) {
        if (!kAhead) load_row(Pn, z);
        y_forward(z);
      }
    }
    P = Pn;
  }
}

}  // namespace rsx
