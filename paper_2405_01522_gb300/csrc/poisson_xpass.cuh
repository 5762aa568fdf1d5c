// Passes 1 and 3 of the pair Poisson solve: the x transforms.
//
// One warp takes an octet of consecutive rows (y, all x) of one plane: four lines of 8 lanes
// (lane 4 t + line), each two real rows packed as one complex line (poisson_lines.cuh).  Octets of a pair are
// independent and rows are contiguous in memory across planes, so a row is addressed by its
// flat index z ny + y (ny = 8 A: whole octets), and a warp needs no barrier wider than itself.
#pragma once
#include "poisson_lines.cuh"

namespace rsx {

constexpr int kXWarps = 4;   // warps (octets) per CTA

// CTAs per SM asked of the compiler.  FP32, us per pair at 128 pairs.  Pass 1 (its work is in L1
// wavefronts): A = 12 1.86 at 5 to 7 CTAs, 2.15 at 8 (spills).  Pass 3 (load latency): A = 12
// 2.38 / 2.00 / 1.77 / 2.65 at 2 / 3 / 4 / 5 (5 spills), A = 14 4.52 / 3.65 / 4.37 at 2 / 3 / 4.
template <typename R>
__host__ __device__ constexpr int p1_min_ctas(int A) {
  return sizeof(R) == 8 ? (A <= 4 ? 6 : A <= 8 ? 4 : 3) : (A <= 4 ? 10 : A <= 7 ? 8 : A == 8 ? 7 : A <= 12 ? 6 : 5);
}
template <typename R>
__host__ __device__ constexpr int p3_min_ctas(int A) {
  return sizeof(R) == 8 ? (A <= 4 ? 4 : A <= 8 ? 3 : 2) : (A <= 4 ? 5 : A <= 12 ? 4 : 3);
}

// per-warp shared memory (complex): the four lines' scratch, or the octet's real rows (pitch
// n + 4 reals: the four lines' rows 2 l and 2 l + 1 fall on distinct banks)
template <typename R, int A>
struct XWarp {
  using S = Split8<R, A, line_j(A), !(sizeof(R) == 8 && A >= 10), true>;
  static constexpr int NB = 8 * A, RP = NB + 4;
  static constexpr int TILE = (8 * RP * (int)sizeof(R) + (int)sizeof(Cx<R>) - 1) / (int)sizeof(Cx<R>);
  static constexpr int SCR = 4 * S::SCR;
};

template <typename R>
__device__ __forceinline__ bool aligned16(const R* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <typename R>
struct Vec16;
template <>
struct Vec16<float> {
  using T = float4;
  static __device__ __forceinline__ T mul(T a, T b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
  static __device__ __forceinline__ T half(T a) { return make_float4(0.5f * a.x, 0.5f * a.y, 0.5f * a.z, 0.5f * a.w); }
};
template <>
struct Vec16<double> {
  using T = double2;
  static __device__ __forceinline__ T mul(T a, T b) { return make_double2(a.x * b.x, a.y * b.y); }
  static __device__ __forceinline__ T half(T a) { return make_double2(0.5 * a.x, 0.5 * a.y); }
};

// two consecutive complex values from / to global memory
__device__ __forceinline__ void ld_pair(const Cx<float>* p, Cx<float>& a, Cx<float>& b) {
  const float4 v = ld_dep(reinterpret_cast<const float4*>(p));
  a = cx<float>(v.x, v.y);
  b = cx<float>(v.z, v.w);
}
__device__ __forceinline__ void ld_pair(const Cx<double>* p, Cx<double>& a, Cx<double>& b) {
  const double2 v = ld_dep(reinterpret_cast<const double2*>(p)), w = ld_dep(reinterpret_cast<const double2*>(p) + 1);
  a = cx<double>(v.x, v.y);
  b = cx<double>(w.x, w.y);
}
__device__ __forceinline__ void st_pair(Cx<float>* p, Cx<float> a, Cx<float> b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_pair(Cx<double>* p, Cx<double> a, Cx<double> b) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a.x, a.y);
  reinterpret_cast<double2*>(p)[1] = make_double2(b.x, b.y);
}

// ---------------------------------------------------------------------------------
// pass 1: pair density and x forward (r2c via row pairs), output I[q][kx][z][y].
// The orbital rows come in as 16-byte loads (the octet is contiguous), their product goes
// through shared memory into the lanes' strided order, and the half spectra X_a(k) =
// (U(k) + conj U(M-k)) / 2, X_b(k) = (U(k) - conj U(M-k)) / 2i leave registers as 16-byte
// stores (rows 2 l, 2 l + 1 of one kx; 64 contiguous bytes per kx and warp).  The partner
// value U(M - k) is one lane exchange.
// Block order: with g.p1_group == 0 a pair's octets are consecutive; with g.p1_group = G > 0
// the pairs are the fastest index in groups of G, so that the CTAs in flight share their rows
// and the orbital rows they multiply are read from HBM once per group and then hit in L2.
template <typename R, int A>
__global__ void __launch_bounds__(32 * kXWarps, p1_min_ctas<R>(A)) k_pass1(Geom g, PairMap<R> pm, int q0, int nq, Cx<R>* inter,
                                                       const Cx<R>* __restrict__ twx) {
  using X = XWarp<R, A>;
  using S = typename X::S;
  using V = Vec16<R>;
  constexpr int NB = X::NB, RP = X::RP, E = 16 / (int)sizeof(R), J = Line<A>::J, A2 = 2 * A;
  constexpr int WS = X::SCR > X::TILE ? X::SCR : X::TILE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane >> 2, line = lane & 3;
  Cx<R>* ws = reinterpret_cast<Cx<R>*>(smem_raw) + warp * WS;
  const int noct = g.nz * (g.ny / 8), nob = (noct + kXWarps - 1) / kXWarps;
  int b = blockIdx.x, ob, ql;
  if (g.p1_group <= 0) {
    ob = b % nob;
    ql = b / nob;
  } else {
    const int lo = b % g.p1_group;
    b /= g.p1_group;
    ob = b % nob;
    ql = (b / nob) * g.p1_group + lo;
  }
  const int oct = ob * kXWarps + warp;
  pdl_launch();
  if (ql >= nq || oct >= noct) return;   // whole warps: the last group, the last block
  pdl_wait();
  const R *f1, *f2;
  pm.pair(q0 + ql, f1, f2);
  const size_t base = (size_t)oct * 8 * NB;
  if (!RSX_IN_RANGE(g, base + 8 * NB - 1, g.N()) || !RSX_IN_RANGE(g, ql, nq)) return;
  f1 += base;
  f2 += base;
  R* tile = reinterpret_cast<R*>(ws);
  if (aligned16(f1) && aligned16(f2)) {
    constexpr int NV = 8 * NB / E, IT = (NV + 31) / 32;
    typename V::T a[IT], c[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i)
      if (NV % 32 == 0 || lane + 32 * i < NV) {
        a[i] = ld_dep(reinterpret_cast<const typename V::T*>(f1) + lane + 32 * i);
        c[i] = ld_dep(reinterpret_cast<const typename V::T*>(f2) + lane + 32 * i);
      }
#pragma unroll
    for (int i = 0; i < IT; ++i)
      if (NV % 32 == 0 || lane + 32 * i < NV) {
        const int e = E * (lane + 32 * i), r = e / NB, x = e - r * NB;
        *reinterpret_cast<typename V::T*>(tile + r * RP + x) = V::half(V::mul(a[i], c[i]));
      }
  } else {   // orbitals off 16-byte boundaries
    for (int e = lane; e < 8 * NB; e += 32) {
      const int r = e / NB, x = e - r * NB;
      tile[r * RP + x] = R(0.5) * (ld_dep(f1 + e) * ld_dep(f2 + e));
    }
  }
  __syncwarp();
  Cx<R> v[A];
#pragma unroll
  for (int a = 0; a < A; ++a) v[a] = cx<R>(tile[2 * line * RP + t + 8 * a], tile[(2 * line + 1) * RP + t + 8 * a]);
  __syncwarp();
  typename S::Tw tw;
  tw.init(twx, t);
  constexpr unsigned lmask = 0xffffffffu;
  Cx<R> U[J][8];   // [j][register k2], see S::reg
  S::forward_rows(v, t, line, lmask, tw, ws + line * S::SCR, [&](int j, int, const Cx<R>(&u)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) U[j][q] = u[q];
  });
  __syncwarp();
  Cx<R>* dst = inter + (size_t)ql * g.inter_elems() + (size_t)oct * 8 + 2 * line;
  const size_t kstride = (size_t)g.nz * g.ny;
  auto store = [&](int kx, Cx<R> u, Cx<R> m) {   // u = U(kx) / 2, m = U(M - kx) / 2
    if (RSX_IN_RANGE(g, (size_t)oct * 8 + 2 * line + (size_t)kx * kstride + 1, g.inter_elems()))
      st_pair(dst + (size_t)kx * kstride, cx<R>(u.x + m.x, u.y - m.y), cx<R>(u.y + m.y, m.x - u.x));
  };
#pragma unroll
  for (int j = 0; j < J; ++j)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
      const Cx<R> u = U[j][S::reg(j, k2)];
      Cx<R> m = S::mirror(j, k2, t, [&](int jj, int q) { return U[jj][S::reg(jj, q)]; });
      if (j == 0 && t == 0) m = U[0][S::reg(0, (8 - k2) & 7)];
      const int k1 = t + 8 * j;
      if (8 * j + 8 <= A2 || k1 < A2) store(k1 + A2 * k2, u, m);
    }
  if (t == 0) store(8 * A, U[0][S::reg(0, 4)], U[0][S::reg(0, 4)]);
}

// ---------------------------------------------------------------------------------
// pass 3: x inverse (c2r via row pairs) of every pair in output p's list, and
// out_p(z, y, x) = - sum_e partner_e(z, y, x) V_e(z, y, x).  With pot != 0 the output p is the
// potential V of pair q = p itself (no partner, no sign).
// A warp's octet of one output: per entry the half spectra of its four lines come in as
// 16-byte loads, Z(k) = X_a(k) + i X_b(k) for k <= M / 2 and the mirrored values of the rest by
// lane exchange, and the partner's rows through shared memory (16-byte cp.async, issued before
// the transform that hides them).  The accumulators stay in registers over the entries.
template <typename R, int A>
__global__ void __launch_bounds__(32 * kXWarps, p3_min_ctas<R>(A)) k_pass3(Geom g, PairMap<R> pm, int q0, int p0, int np, int pot,
                                                       const Cx<R>* inter, const Cx<R>* __restrict__ twx, R* out) {
  using X = XWarp<R, A>;
  using S = typename X::S;
  constexpr int NB = X::NB, RP = X::RP, E = 16 / (int)sizeof(R), J = Line<A>::J, A2 = 2 * A;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane >> 2, line = lane & 3;
  Cx<R>* ws = reinterpret_cast<Cx<R>*>(smem_raw) + warp * (X::SCR + X::TILE);
  R* tile = reinterpret_cast<R*>(ws + X::SCR);   // the partner's octet, [8][RP]
  // outputs are the fastest index: the CTAs in flight share their rows, so the partner rows
  // they multiply come from HBM once and then from L2 for the other outputs
  const int pl = (int)(blockIdx.x % np), oct = (int)(blockIdx.x / np) * kXWarps + warp;
  pdl_launch();
  if (oct >= g.nz * (g.ny / 8)) return;   // whole warps
  pdl_wait();
  const int p = p0 + pl;
  const size_t base = (size_t)oct * 8 * NB;
  if (!RSX_IN_RANGE(g, base + 8 * NB - 1, g.N())) return;
  typename S::Tw tw;
  tw.init(twx, t);
  constexpr unsigned lmask = 0xffffffffu;
  const size_t kstride = (size_t)g.nz * g.ny;
  R acc0[A], acc1[A];
#pragma unroll
  for (int a = 0; a < A; ++a) acc0[a] = acc1[a] = R(0);
  const int ne = pot ? 1 : pm.nentries(p);
  for (int e = 0; e < ne; ++e) {
    int q = p;
    const R* partner = nullptr;
    if (!pot) {
      pm.entry(p, e, q, partner);
      partner += base;
      __syncwarp();   // the tile of the entry before has been read
      if (aligned16(partner)) {
        for (int i = lane; i < 8 * NB / E; i += 32) {
          const int el = E * i, r = el / NB, x = el - r * NB;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(tile + r * RP + x)),
                       "l"(partner + el)
                       : "memory");
        }
      } else {
        for (int el = lane; el < 8 * NB; el += 32) {
          const int r = el / NB, x = el - r * NB;
          asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(tile + r * RP + x)),
                       "l"(partner + el), "n"(sizeof(R))
                       : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const bool slot_ok = RSX_IN_RANGE(g, q - q0, g.dbg_nq > 0 ? g.dbg_nq : 0x7fffffff);
    const Cx<R>* src = inter + (size_t)(q - q0) * g.inter_elems() + (size_t)oct * 8 + 2 * line;
    Cx<R> Z[J][4], C[J][4], zn = cx<R>(R(0), R(0));   // Z(k), Z(M - k) for k2 < 4; Z(M / 2)
    auto load = [&](int kx, Cx<R>& xa, Cx<R>& xb) {
      xa = xb = cx<R>(R(0), R(0));
      if (slot_ok && RSX_IN_RANGE(g, (size_t)oct * 8 + 2 * line + (size_t)kx * kstride + 1, g.inter_elems()))
        ld_pair(src + (size_t)kx * kstride, xa, xb);
    };
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) {
        const int k1 = t + 8 * j;
        Cx<R> xa = cx<R>(R(0), R(0)), xb = xa;
        if (8 * j + 8 <= A2 || k1 < A2) load(k1 + A2 * k2, xa, xb);
        Z[j][k2] = xa;
        C[j][k2] = xb;
      }
    if (t == 0) {
      Cx<R> xa, xb;
      load(8 * A, xa, xb);
      zn = cx<R>(xa.x - xb.y, xa.y + xb.x);
    }
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) {
        const Cx<R> xa = Z[j][k2], xb = C[j][k2];
        Z[j][k2] = cx<R>(xa.x - xb.y, xa.y + xb.x);
        C[j][k2] = cx<R>(xa.x + xb.y, xb.x - xa.y);   // conj(X_a) + i conj(X_b)
      }
    Cx<R> H[J][4];   // Z of k2 = 4 .. 7, from the partner lane
#pragma unroll
    for (int j = 0; j < J; ++j)
#pragma unroll
      for (int k2 = 4; k2 < 8; ++k2) {
        H[j][k2 - 4] = S::mirror(j, k2, t, [&](int jj, int q) { return C[jj][q]; });
        if (j == 0 && t == 0) H[0][k2 - 4] = k2 == 4 ? zn : C[0][8 - k2 < 4 ? 8 - k2 : 0];
      }
    S::inverse_rows(
        t, line, lmask, tw, ws + line * S::SCR,
        [&](int j, int, Cx<R>(&u)[8]) {
#pragma unroll
          for (int k2 = 0; k2 < 4; ++k2) u[S::reg(j, k2)] = Z[j][k2];
#pragma unroll
          for (int k2 = 4; k2 < 8; ++k2) u[S::reg(j, k2)] = H[j][k2 - 4];
        },
        [&](int a, int i, Cx<R> x) {
          if (a == 0 && !pot) {   // the partner rows are in place
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
          }
          if (pot) {
            acc0[a] = x.x;
            acc1[a] = x.y;
          } else {
            acc0[a] -= tile[2 * line * RP + i] * x.x;
            acc1[a] -= tile[(2 * line + 1) * RP + i] * x.y;
          }
        });
  }
  __syncwarp();
#pragma unroll
  for (int a = 0; a < A; ++a) {
    tile[2 * line * RP + t + 8 * a] = acc0[a];
    tile[(2 * line + 1) * RP + t + 8 * a] = acc1[a];
  }
  __syncwarp();
  R* o = pm.out_row(p, out, pl) + base;
  if (aligned16(o)) {
    using T = typename Vec16<R>::T;
    for (int i = lane; i < 8 * NB / E; i += 32) {
      const int el = E * i, r = el / NB, x = el - r * NB;
      reinterpret_cast<T*>(o)[i] = *reinterpret_cast<const T*>(tile + r * RP + x);
    }
  } else {
    for (int el = lane; el < 8 * NB; el += 32) {
      const int r = el / NB, x = el - r * NB;
      o[el] = tile[r * RP + x];
    }
  }
}

}  // namespace rsx
