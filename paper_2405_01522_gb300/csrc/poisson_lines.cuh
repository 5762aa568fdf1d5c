// Line transforms of the pair Poisson passes: a line of M = 16 A points on 8 lanes x 2A.
//
//   stage 1  lane t (< 8) holds x[t + 8 a], does the 2A-point DFT over a in registers,
//            multiplies row k1 of the result by w_M^{-t k1} and stores it in row k1 of the
//            line's scratch (2A rows of 8 complex);
//   stage 2  lane s does the 8-point DFTs over t of rows k1 = s + 8 j (j < ceil(2A / 8)),
//            giving X[k1 + 2A k2].
// The box edge is n = 8 A = M / 2, so half of the inputs of a forward line are zero and half
// of the outputs of an inverse line are dropped: DftHalfIn / DftHalfOut in stage 1.
//
// Rows k1 >= NEG are carried as the negative frequencies k1 - 2A: their twiddle is the
// conjugate of row 2A - k1's, so a lane holds max(NEG - 1, 2A - NEG) twiddles instead of
// 2A - 1 (15 instead of 23 at A = 12; with 23 the y/z pass did not fit 12 warps per SM
// without spills), and output k2 of such a row is X[k1 + 2A ((k2 + 7) mod 8)].  NEG is a
// multiple of 8, so which rows are negative does not depend on the lane.
#pragma once
#include "rsx_internal.cuh"

namespace rsx {

// Programmatic dependent launch: the passes are launched so that a kernel's CTAs may be set up
// while the kernel before it in the stream drains.  Every pass starts with pdl_wait(), before
// its first access to memory that kernel touches (it returns when that kernel is complete
// and its writes are visible), and lets its own successor be set up from its start.
// What the kernel before may still be writing at that time -- the orbitals, the intermediate -- must
// not be read through __ldg or const __restrict__ pointers: those make ld.global.nc, whose data
// may not change while the kernel runs and which the wait's memory clobber does not hold
// back.  It is read by ld_dep, or by plain loads through unqualified pointers.  The tables written by
// rsx_create are constant.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// coherent global loads, in program order with pdl_wait (volatile)
__device__ __forceinline__ float ld_dep(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_dep(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ float4 ld_dep(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 ld_dep(const double2* p) {
  double2 v;
  asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

__host__ __device__ constexpr int line_tw_count(int A, int neg) { return neg - 1 > 2 * A - neg ? neg - 1 : 2 * A - neg; }
__host__ __device__ constexpr int line_neg(int A) {   // 2A: no negative rows
  int best = 2 * A;
  for (int b = 8; b < 2 * A; b += 8)
    if (line_tw_count(A, b) < line_tw_count(A, best)) best = b;
  return best;
}
__host__ __device__ constexpr int line_j(int A) { return (2 * A + 7) / 8; }

template <int A>
struct Line {
  static constexpr int A2 = 2 * A, M = 16 * A, NB = 8 * A, J = line_j(A), NEG = line_neg(A), W = line_tw_count(A, NEG);
  // offset of output k2 of row k1 = s + 8 j from position k1
  __host__ __device__ static constexpr int out(int j, int k2) { return A2 * (8 * j >= NEG ? (k2 + 7) & 7 : k2); }
};

// Scratch rows of 8 complex, element t of row r of line l at off(r, t, l) (l: the line's number
// in its warp, lines' scratch a multiple of 128 bytes apart).  Two lane orders of a warp's
// four lines:
//   t fastest (lane 8 l + t; the y/z pass).  FP32: the row sits at r ^ (l & 1) and its four
//     16-byte chunks are XOR-swizzled by (row >> 1) & 3.  Then (i) the two lines of a half-warp
//     put the same row in opposite halves of the banks, so the 8-byte accesses of stage 1 are
//     conflict-free, and (ii) the eight lanes of a line reading rows s + 8 j as 16-byte
//     chunks hit eight distinct bank groups.  FP64 (128-byte rows): element t at t ^ (r & 7).
//   l fastest (lane 4 t + l; the x passes, whose 16-byte global accesses coalesce over the four
//     lines only if these are consecutive lanes).  FP32: the row sits at r ^ l, its chunks are
//     swizzled by row bit 1 (as 2) and row bit 2 (as 1) and by l & 1: 4 lines x 4 lanes of a
//     half-warp cover the banks once in stage 1, and so do 4 lines x 2 rows of a quarter-warp
//     in stage 2.  FP64: element t at t ^ (r & 7) ^ 2 l.
template <typename R, bool LFAST>
struct LineScr;

template <bool LFAST>
struct LineScr<float, LFAST> {
  static __device__ __forceinline__ int row(int r, int l) { return LFAST ? r ^ l : r ^ (l & 1); }
  static __device__ __forceinline__ int swz(int pr, int l) {
    return LFAST ? ((pr & 2) | ((pr >> 2) & 1)) ^ (l & 1) : (pr >> 1) & 3;
  }
  static __device__ __forceinline__ int off(int r, int t, int l) {
    const int pr = row(r, l);
    return pr * 8 + 2 * ((t >> 1) ^ swz(pr, l)) + (t & 1);
  }
  static __device__ __forceinline__ void load(Cx<float> (&u)[8], const Cx<float>* sc, int r, int l) {
    const int pr = row(r, l), sw = swz(pr, l);
    const float4* rp = reinterpret_cast<const float4*>(sc + pr * 8);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = rp[q ^ sw];
      u[2 * q] = cx<float>(v.x, v.y);
      u[2 * q + 1] = cx<float>(v.z, v.w);
    }
  }
  static __device__ __forceinline__ void store(Cx<float>* sc, int r, int l, const Cx<float> (&u)[8]) {
    const int pr = row(r, l), sw = swz(pr, l);
    float4* rp = reinterpret_cast<float4*>(sc + pr * 8);
#pragma unroll
    for (int q = 0; q < 4; ++q) rp[q ^ sw] = make_float4(u[2 * q].x, u[2 * q].y, u[2 * q + 1].x, u[2 * q + 1].y);
  }
};

template <bool LFAST>
struct LineScr<double, LFAST> {
  static __device__ __forceinline__ int off(int r, int t, int l) { return r * 8 + (t ^ (r & 7) ^ (LFAST ? 2 * l : 0)); }
  static __device__ __forceinline__ void load(Cx<double> (&u)[8], const Cx<double>* sc, int r, int l) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double2 v = *reinterpret_cast<const double2*>(sc + off(r, q, l));
      u[q] = cx<double>(v.x, v.y);
    }
  }
  static __device__ __forceinline__ void store(Cx<double>* sc, int r, int l, const Cx<double> (&u)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) *reinterpret_cast<double2*>(sc + off(r, q, l)) = make_double2(u[q].x, u[q].y);
  }
};

// This lane's twiddles w_M^{-t k}, k <= W, in registers, or (REG = false) read from the
// table tw8[k1][t] where they are used.
template <typename R, int A, bool REG = true>
struct LineTw {
  Cx<R> reg[REG ? Line<A>::W + 1 : 1];
  const Cx<R>* tab;
  __device__ __forceinline__ void init(const Cx<R>* __restrict__ tw8, int t) {
    tab = tw8 + t;
    if constexpr (REG) {
#pragma unroll
      for (int k = 1; k <= Line<A>::W; ++k) reg[k] = tab[8 * k];
    }
  }
  __device__ __forceinline__ Cx<R> get(int k) const {
    if constexpr (REG) return reg[k];
    else return tab[8 * k];
  }
  // row k1 times w^{-t k1} (forward) or w^{+t k1} (inverse), k1 >= 1
  __device__ __forceinline__ Cx<R> fwd(Cx<R> x, int k1) const {
    return k1 < Line<A>::NEG ? cmul(x, get(k1)) : cmul(x, conj(get(Line<A>::A2 - k1)));
  }
  __device__ __forceinline__ Cx<R> inv(Cx<R> x, int k1) const {
    return k1 < Line<A>::NEG ? cmul(x, conj(get(k1))) : cmul(x, get(Line<A>::A2 - k1));
  }
};

// The 8-lane split as used by a kernel: JP groups of 8 rows pass through the line's scratch at
// a time (JP = J: all at once), TWREG: twiddles in registers.
__host__ __device__ constexpr int line_rows(int A, int jp) { return jp >= line_j(A) ? (2 * A + 3) / 4 * 4 : 8 * jp; }

template <typename R, int A, int JP, bool TWREG = true, bool LFAST = false>
struct Split8 {
  using L = Line<A>;
  using Scr = LineScr<R, LFAST>;
  using Tw = LineTw<R, A, TWREG>;
  static constexpr int LANES = 8, NIN = A, RAD = 8, FAC = 8 * L::J, SCR = line_rows(A, JP) * 8;
  __host__ __device__ static constexpr int out(int j, int k2) { return L::out(j, k2); }

  // Forward line: v[a] is input t + 8 a < n = 8 A; `row(j, k1, u)` receives the 8-point spectra
  // u[k2] = X[k1 + out(j, k2)] of this lane's rows k1 = t + 8 j.
  template <class Row>
  static __device__ __forceinline__ void forward_rows(const Cx<R> (&v)[A], int t, int l, unsigned lmask, const Tw& tw,
                                                      Cx<R>* sc, Row row) {
    Cx<R> x[L::A2];
    DftHalfIn<L::A2, -1>::run(v, x);
#pragma unroll
    for (int k1 = 1; k1 < L::A2; ++k1) x[k1] = tw.fwd(x[k1], k1);
#pragma unroll
    for (int p = 0; p < L::J; p += JP) {
#pragma unroll
      for (int k1 = 8 * p; k1 < 8 * (p + JP) && k1 < L::A2; ++k1) sc[Scr::off(k1 - 8 * p, t, l)] = x[k1];
      __syncwarp(lmask);
#pragma unroll
      for (int j = p; j < p + JP && j < L::J; ++j) {
        const int k1 = t + 8 * j;
        if (8 * j + 8 <= L::A2 || k1 < L::A2) {
          Cx<R> u[8];
          Scr::load(u, sc, k1 - 8 * p, l);
          Dft<8, -1>::run(u);
          row(j, k1, u);
        }
      }
      __syncwarp(lmask);
    }
  }
  // the same with `put(k, x)` receiving X[k]
  template <class Put>
  static __device__ __forceinline__ void forward(const Cx<R> (&v)[A], int t, int l, unsigned lmask, const Tw& tw,
                                                 Cx<R>* sc, Put put) {
    forward_rows(v, t, l, lmask, tw, sc, [&](int j, int k1, const Cx<R>(&u)[8]) {
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) put(k1 + out(j, k2), u[k2]);
    });
  }

  // Inverse line: `row(j, k1, u)` fills u[k2] with X[k1 + out(j, k2)] of row k1 = t + 8 j;
  // `put(a, i, x)` receives output i = t + 8 a < n.
  template <class Row, class Put>
  static __device__ __forceinline__ void inverse_rows(int t, int l, unsigned lmask, const Tw& tw, Cx<R>* sc, Row row,
                                                      Put put) {
    Cx<R> r[L::A2], o[A];
#pragma unroll
    for (int p = 0; p < L::J; p += JP) {
#pragma unroll
      for (int j = p; j < p + JP && j < L::J; ++j) {
        const int k1 = t + 8 * j;
        if (8 * j + 8 <= L::A2 || k1 < L::A2) {
          Cx<R> u[8];
          row(j, k1, u);
          Dft<8, 1>::run(u);
          Scr::store(sc, k1 - 8 * p, l, u);
        }
      }
      __syncwarp(lmask);
#pragma unroll
      for (int k1 = 8 * p; k1 < 8 * (p + JP) && k1 < L::A2; ++k1) r[k1] = sc[Scr::off(k1 - 8 * p, t, l)];
      __syncwarp(lmask);
    }
#pragma unroll
    for (int k1 = 1; k1 < L::A2; ++k1) r[k1] = tw.inv(r[k1], k1);
    DftHalfOut<L::A2, 1>::run(r, o);
#pragma unroll
    for (int a = 0; a < A; ++a) put(a, t + 8 * a, o[a]);
  }
  // the same with `in(k)` giving X[k] and `put(i, x)`
  template <class In, class Put>
  static __device__ __forceinline__ void inverse(int t, int l, unsigned lmask, const Tw& tw, Cx<R>* sc, In in, Put put) {
    inverse_rows(
        t, l, lmask, tw, sc,
        [&](int j, int k1, Cx<R>(&u)[8]) {
#pragma unroll
          for (int k2 = 0; k2 < 8; ++k2) u[k2] = in(k1 + out(j, k2));
        },
        [&](int, int i, Cx<R> x) { put(i, x); });
  }

  // Two real rows packed as one complex line have their half spectra in U(k) and U(M - k).  Lane
  // t holds X at (row j, k2): k = t + 8 j + 2A k2; M - k is in lane (2A - t) mod 8 at
  //   row JF - j (lanes t <= 2A mod 8), row JF - 1 - j (the others), JF = floor(2A / 8), and 7 - k2;
  // k1 = 0 (lane 0, row 0) pairs with itself at (8 - k2) mod 8.  mirror(j, k2, get) returns the
  // partner lane's get(row, 7 - k2) for this lane's (j, k2): get reads this lane's own values at
  // compile-time rows.  Valid rows only; lane 0 row 0 takes its own value instead.
  static constexpr int JF = L::A2 / 8, RM = L::A2 % 8;
  template <class Get>
  static __device__ __forceinline__ Cx<R> mirror(int j, int k2, int t, Get get) {
    static_assert(LFAST, "lane order of the x passes");
    const int ja = JF - j < L::J ? JF - j : L::J - 1, jb = JF - 1 - j >= 0 ? JF - 1 - j : 0;
    const Cx<R> va = get(ja, 7 - k2), vb = get(jb, 7 - k2);
    const bool ca = t <= RM;
    const int src = (((RM - t) & 7) << 2) | (threadIdx.x & 3);   // lanes 4 t + l
    return cx<R>(__shfl_sync(0xffffffffu, ca ? va.x : vb.x, src), __shfl_sync(0xffffffffu, ca ? va.y : vb.y, src));
  }
  // register index of logical k2 in row j (negative rows are rotated by one)
  __host__ __device__ static constexpr int reg(int j, int k2) { return 8 * j >= L::NEG ? (k2 + 1) & 7 : k2; }

  // Forward, multiply by the factors, inverse: the spectrum stays in registers and scratch
  // rows; `scale(j, u)` multiplies the 8 spectra of row t + 8 j.
  template <class In, class Scale, class Put>
  static __device__ __forceinline__ void convolve(int t, int l, unsigned lmask, const Tw& tw, Cx<R>* sc, In in,
                                                  Scale scale, Put put) {
    Cx<R> v[A], x[L::A2], o[A];
#pragma unroll
    for (int a = 0; a < A; ++a) v[a] = in(t + 8 * a);
    DftHalfIn<L::A2, -1>::run(v, x);
#pragma unroll
    for (int k1 = 1; k1 < L::A2; ++k1) x[k1] = tw.fwd(x[k1], k1);
#pragma unroll
    for (int p = 0; p < L::J; p += JP) {
#pragma unroll
      for (int k1 = 8 * p; k1 < 8 * (p + JP) && k1 < L::A2; ++k1) sc[Scr::off(k1 - 8 * p, t, l)] = x[k1];
      __syncwarp(lmask);
#pragma unroll
      for (int j = p; j < p + JP && j < L::J; ++j) {
        const int k1 = t + 8 * j;
        if (8 * j + 8 <= L::A2 || k1 < L::A2) {
          Cx<R> u[8];
          Scr::load(u, sc, k1 - 8 * p, l);
          Dft<8, -1>::run(u);
          scale(j, u);
          Dft<8, 1>::run(u);
          Scr::store(sc, k1 - 8 * p, l, u);   // read and written by this lane only
        }
      }
      __syncwarp(lmask);
#pragma unroll
      for (int k1 = 8 * p; k1 < 8 * (p + JP) && k1 < L::A2; ++k1) x[k1] = sc[Scr::off(k1 - 8 * p, t, l)];
      __syncwarp(lmask);
    }
#pragma unroll
    for (int k1 = 1; k1 < L::A2; ++k1) x[k1] = tw.inv(x[k1], k1);
    DftHalfOut<L::A2, 1>::run(x, o);
#pragma unroll
    for (int a = 0; a < A; ++a) put(t + 8 * a, o[a]);
  }
};

// The split on 16 lanes x A (even A): lane t holds x[t + 16 a], A-point DFT, twiddle
// w_M^{-t k1}, and lane k1 < A does the 16-point DFT over t, X[k1 + A k2].  A of 16 lanes work
// in the 16-point stage, but it needs fewer registers: kept for the y/z pass at A = 14 (14 of 16
// lanes), where the 28-point stage leaves 7 warps, or 12 with spills (20.3 us per pair against
// 22.3 on 8 lanes).  FP32.
template <int A>
struct Split16 {
  using R = float;
  static_assert(A % 2 == 0, "even A");
  static constexpr int LANES = 16, NIN = A / 2, RAD = 16, FAC = 16, PITCH = 17, SCR = A * PITCH;
  struct Tw {
    Cx<R> reg[A];
    __device__ __forceinline__ void init(const Cx<R>* __restrict__ tw, int t) {
#pragma unroll
      for (int k = 1; k < A; ++k) reg[k] = tw[16 * k + t];
    }
  };
  static __device__ __forceinline__ void stage1(const Cx<R> (&v)[NIN], int t, const Tw& tw, Cx<R>* sc) {
    Cx<R> x[A];
    DftHalfIn<A, -1>::run(v, x);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) x[k1] = cmul(x[k1], tw.reg[k1]);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) sc[k1 * PITCH + t] = x[k1];
  }
  template <class Put>
  static __device__ __forceinline__ void forward(const Cx<R> (&v)[NIN], int t, int, unsigned lmask, const Tw& tw,
                                                 Cx<R>* sc, Put put) {
    stage1(v, t, tw, sc);
    __syncwarp(lmask);
    if (t < A) {
      Cx<R> u[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) u[q] = sc[t * PITCH + q];
      Dft<16, -1>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) put(t + A * k2, u[k2]);
    }
    __syncwarp(lmask);
  }
  template <class In, class Put>
  static __device__ __forceinline__ void inverse(int t, int, unsigned lmask, const Tw& tw, Cx<R>* sc, In in, Put put) {
    // the same steps as forward with conjugate twiddles: A-point DFTs over X[t + 16 a], then 16-point
    // ones of which outputs y = k1 + A k2 < n = 8 A, k2 < 8, are kept
    Cx<R> x[A];
#pragma unroll
    for (int a = 0; a < A; ++a) x[a] = in(t + 16 * a);
    Dft<A, 1>::run(x);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) x[k1] = cmul(x[k1], conj(tw.reg[k1]));
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) sc[k1 * PITCH + t] = x[k1];
    __syncwarp(lmask);
    if (t < A) {
      Cx<R> u[16], o[8];
#pragma unroll
      for (int q = 0; q < 16; ++q) u[q] = sc[t * PITCH + q];
      DftHalfOut<16, 1>::run(u, o);
#pragma unroll
      for (int k2 = 0; k2 < 8; ++k2) put(t + A * k2, o[k2]);
    }
    __syncwarp(lmask);
  }
  template <class In, class Scale, class Put>
  static __device__ __forceinline__ void convolve(int t, int, unsigned lmask, const Tw& tw, Cx<R>* sc, In in,
                                                  Scale scale, Put put) {
    Cx<R> v[NIN];
#pragma unroll
    for (int a = 0; a < NIN; ++a) v[a] = in(t + 16 * a);
    stage1(v, t, tw, sc);
    __syncwarp(lmask);
    if (t < A) {   // row t is read and written by this lane only
      Cx<R> u[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) u[q] = sc[t * PITCH + q];
      Dft<16, -1>::run(u);
      scale(0, u);
      Dft<16, 1>::run(u);
#pragma unroll
      for (int q = 0; q < 16; ++q) sc[t * PITCH + q] = u[q];
    }
    __syncwarp(lmask);
    Cx<R> r[A], o[NIN];
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) r[k1] = sc[k1 * PITCH + t];
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) r[k1] = cmul(r[k1], conj(tw.reg[k1]));
    DftHalfOut<A, 1>::run(r, o);
#pragma unroll
    for (int a = 0; a < NIN; ++a) put(t + 16 * a, o[a]);
    __syncwarp(lmask);
  }
};

}  // namespace rsx
