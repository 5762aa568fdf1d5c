// Pair Poisson solve by pruned, zero-padded FFT convolution: the three passes.
//
// The potential of a pair density rho = f1 f2 on the box (nz, ny, nx) is
//     V = h^3/N_pad * IDFT( ghat * DFT(rho zero-padded to (2nz, 2ny, 2nx)) )
// restricted to the box (Sec. 3.1: Eq. 2's integral as a Poisson problem at
// O(N log N); padding twice the box makes the periodic convolution the isolated one).
// The solve is split so that only one 1-D transform per pass touches HBM:
//
//   pass 1  x forward, real-to-complex (two rows y, y+1 packed as one complex line),
//           output I[q][kx][z][y], kx in [0, Mx/2]       (Mx/2+1) * nz * ny complex
//   pass 2  per (q, kx): y forward on nz rows, z forward + multiply by vhat + z inverse
//           on My columns, y inverse keeping y < ny; in place on I
//   pass 3  per (output p, z, 32 rows): x inverse complex-to-real of every pair of p's
//           list, keeping x < nx, and  out_p -= partner * V  (Eq. 2's sum over j)
//
// Only nz of the 2nz z-planes and ny of the 2ny rows are non-zero, so the x transforms
// run on nz*ny rows and the y transforms on nz rows per kx; I is 4x smaller than a
// padded half spectrum.  A line of length M = 16 A is transformed by 16 lanes:
// lane t holds x[t + 16 a] (a < A), does an A-point DFT, multiplies by the twiddle
// w_M^{t k1}, and after a shared-memory transpose lane k1 does the 16-point DFT over t,
// giving X[k1 + A k2].  The inverse of that split is the same steps in reverse, so in
// pass 2 the z spectrum never leaves registers between forward, multiply and inverse.
#pragma once
#include <cuda_bf16.h>

#include "rsx_internal.cuh"

namespace rsx {

// round-to-nearest-even f32 -> bf16 bit pattern (finite inputs), and back
__device__ __forceinline__ uint32_t f32_to_bf16_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u + 0x7FFFu + ((u >> 16) & 1u)) >> 16;
}
__device__ __forceinline__ float bf16_bits_to_f32(uint32_t b) { return __uint_as_float(b << 16); }

// ---------------------------------------------------------------------------------
// stage helpers (executed by the 16 lanes t of one half-warp on one line)
// stage 1: v holds x[t + 16 a]; DFT over a, twiddle, store scratch[k1][t]
template <int A, int S, typename R, int PITCH = kScrPitch>
__device__ __forceinline__ void stage1_store(Cx<R> (&v)[A], int t, const Cx<R>* __restrict__ tw,
                                             Cx<R>* sc) {
  Dft<A, S>::run(v);
#pragma unroll
  for (int k1 = 1; k1 < A; ++k1) {
    Cx<R> w = tw[t * A + k1];
    if (S > 0) w.y = -w.y;
    v[k1] = cmul(v[k1], w);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) sc[k1 * PITCH + t] = v[k1];
}

// stage 1 for a forward transform whose inputs t + 16 a >= 8 A are zero (even A, the
// padded half of a line of length 16 A): only v[0 .. A/2) are used
template <int A, int S, typename R, int PITCH = kScrPitch>
__device__ __forceinline__ void stage1_store_halfin(const Cx<R>* v, int t, const Cx<R>* __restrict__ tw, Cx<R>* sc) {
  Cx<R> x[A];
  DftHalfIn<A, S>::run(v, x);
#pragma unroll
  for (int k1 = 1; k1 < A; ++k1) {
    Cx<R> w = tw[t * A + k1];
    if (S > 0) w.y = -w.y;
    x[k1] = cmul(x[k1], w);
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) sc[k1 * PITCH + t] = x[k1];
}

// the same with this lane's twiddles already in registers (w[k1] = w_M^{-t k1}, k1 >= 1)
template <int A, typename R, int PITCH = kScrPitch>
__device__ __forceinline__ void stage1_store_halfin_reg(const Cx<R>* v, int t, const Cx<R> (&w)[A], Cx<R>* sc) {
  Cx<R> x[A];
  DftHalfIn<A, -1>::run(v, x);
#pragma unroll
  for (int k1 = 1; k1 < A; ++k1) x[k1] = cmul(x[k1], w[k1]);
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) sc[k1 * PITCH + t] = x[k1];
}

// stage 2 load: lane s (< A) gathers its 16 values scratch[s][t]; with an even pitch (FP32
// rows on 16-byte boundaries) as eight 16-byte loads
template <typename R, int PITCH = kScrPitch>
__device__ __forceinline__ void stage2_load(Cx<R> (&u)[16], int s, const Cx<R>* sc) {
  if constexpr (sizeof(R) == 4 && PITCH % 2 == 0) {
    const float4* rp = reinterpret_cast<const float4*>(sc + s * PITCH);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 v = rp[j];
      u[2 * j] = cx<R>(v.x, v.y);
      u[2 * j + 1] = cx<R>(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) u[j] = sc[s * PITCH + j];
  }
}
// ---------------------------------------------------------------------------------
// Pieces of the spectrum kernel.  D is the (nz x My) plane of one (pair, kx), row pitch
// DP = My + 1.  Row loops step over pairs of rows per warp so that both half-warps of a warp
// run the same number of iterations (their __syncwarp calls must match).  (Pass 2 itself is
// in poisson_pass2.cuh.)

// forward y transform of rows z < nz (input y < ny, output all My)
template <typename R, int AY, int NT, int PITCH = kScrPitch>
__device__ __forceinline__ void y_forward(Cx<R>* D, int DP, int nz, int ny, const Cx<R>* __restrict__ twy,
                                          Cx<R>* sc, int in_off = 0) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 15;
  for (int z0 = 2 * warp; z0 < nz; z0 += NT / 16) {
    const int z = z0 + (lane >> 4);
    const bool ok = z < nz;
    constexpr int AIN = (AY % 2 == 0) ? AY / 2 : AY;   // inputs y >= ny = 8 AY are zero
    Cx<R> v[AY];
#pragma unroll
    for (int a = 0; a < AIN; ++a) {
      const int y = t + 16 * a;
      v[a] = (ok && y < ny) ? D[z * DP + in_off + y] : cx<R>(R(0), R(0));
    }
    if constexpr (AY % 2 == 0) {
      stage1_store_halfin<AY, -1, R, PITCH>(v, t, twy, sc);
    } else {
      stage1_store<AY, -1, R, PITCH>(v, t, twy, sc);
    }
    __syncwarp();
    Cx<R> u[16];
    if (t < AY) {
      stage2_load<R, PITCH>(u, t, sc);
      Dft<16, -1>::run(u);
    }
    __syncwarp();
    if (ok && t < AY) {
#pragma unroll
      for (int k2 = 0; k2 < 16; ++k2) D[z * DP + t + AY * k2] = u[k2];
    }
    __syncwarp();
  }
}

template <typename R>
__device__ __forceinline__ void prefetch_plane_upper(Cx<R>* D, int DP, const Cx<R>* P, int nz, int ny, int NT) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int z = warp; z < nz; z += NT / 32)
    for (int y = lane; y < ny; y += 32) {
      Cx<R>* dp = D + z * DP + ny + y;
      const Cx<R>* sp = P + z * ny + y;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dp)), "l"(sp)
                   : "memory");
      if (sizeof(R) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dp) + 8u),
                     "l"(reinterpret_cast<const char*>(sp) + 8)
                     : "memory");
    }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Casida pair spectra (panel tile-major, see below): per (transition q, kx) plane, y forward and z forward, then
// S_q(G) = sqrt(w_kx * ghat(G) * h^6 / N_pad) * (Re, Im) R_q(G) with w = 1 at kx = 0, Mx/2
// and 2 otherwise, split into bf16 hi + lo and written to panel row q at column
// 2 * ((kx * My + ky) * Mz + kz) + {0, 1}.  wsq holds the weights sqrt(w * ghat * h^6 /
// N_pad) on the folded half spectrum [kx][|ky|][|kz|] (k_spectrum_weights).
template <int AY, int AZ, int NT>
__global__ void __launch_bounds__(NT) k_spectrum(Geom g, int nq, const Cx<float>* __restrict__ inter,
                                                       const Cx<float>* __restrict__ twy,
                                                       const Cx<float>* __restrict__ twz,
                                                       const float* __restrict__ wsq,
                                                       uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
                                                       size_t ld, int nrb) {
  constexpr int LY = 16 * AY;
  constexpr int LZ = 16 * AZ;
  constexpr int AMAX = AY > AZ ? AY : AZ;
  constexpr int SP = AMAX * kScrPitch;
  constexpr int DP = LY + 1;
  constexpr int LPC = NT / 16;   // lines per CTA (one per half-warp)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cx<float>* scr = reinterpret_cast<Cx<float>*>(smem_raw);
  Cx<float>* D = scr + LPC * SP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = lane & 15, line = warp * 2 + (lane >> 4);
  Cx<float>* sc = scr + line * SP;
  constexpr int Hy = LY / 2 + 1, Hz = LZ / 2 + 1;
  const int nplane = g.nz * g.ny;
  const int nwork = nq * g.Hx;
  // transitions are the fastest index of the work items: the CTAs in flight fill the same
  // 128 x 64 panel tiles (rows = transitions) instead of scattering 128-byte rows
  auto plane_ptr = [&](int w) {
    const int kx = w / nq, ql = w - kx * nq;
    return inter + (size_t)ql * g.inter_elems() + (size_t)kx * nplane;
  };
  // the plane is staged in the upper halves [ny, 2 ny) of the D rows; the next plane is
  // prefetched there once the z transforms of the upper ky columns are done
  if ((int)blockIdx.x < nwork) prefetch_plane_upper<float>(D, DP, plane_ptr(blockIdx.x), g.nz, g.ny, NT);
  for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
    const int kx = w / nq, ql = w - kx * nq;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    y_forward<float, AY, NT>(D, DP, g.nz, g.ny, twy, sc, g.ny);
    __syncthreads();
    const float* vrow = wsq + (size_t)kx * Hy * Hz;
    // tile-major panel [ld/64][nrb][128][64]: column g of row ql is at
    // ((g / 64) * nrb + ql / 128) * 8192 + (ql % 128) * 64 + g % 64
    const size_t row_off = (size_t)(ql / 128) * 8192 + (size_t)(ql % 128) * 64;
    const size_t kb_stride = (size_t)nrb * 8192;
    const int wn = w + (int)gridDim.x;
    // this lane's forward stage-1 twiddles, the same for every column
    Cx<float> twf[AZ];
    if constexpr (AZ % 2 == 0) {
#pragma unroll
      for (int k1 = 1; k1 < AZ; ++k1) twf[k1] = twz[t * AZ + k1];
    }
    // columns ky: the upper half [LY/2, LY) first, then the lower half; slot s of line l
    // takes flat position f = s LPC + l (f < LY/2: upper column LY/2 + f, else lower
    // column f - LY/2), so every line runs the same number of columns, and after slot
    // kPre - 1 (when every upper column is done; possibly the last slot) the next plane is
    // prefetched into the upper halves of the D rows
    constexpr int kSlots = (LY + LPC - 1) / LPC;
    constexpr int kPre = (LY / 2 + LPC - 1) / LPC;
    for (int slot = 0; slot < kSlots; ++slot) {
      const int f = slot * LPC + line;
      if (f < LY) {   // uniform in a warp: LPC is even, a warp's two lines are f, f + 1 with LY even
        const int ky = f < LY / 2 ? LY / 2 + f : f - LY / 2;
        const int iy = ky <= LY / 2 ? ky : LY - ky;
        const float* vcol = vrow + (size_t)iy * Hz;
        constexpr int AIN = (AZ % 2 == 0) ? AZ / 2 : AZ;
        Cx<float> v[AZ];
#pragma unroll
        for (int a = 0; a < AIN; ++a) {
          const int z = t + 16 * a;
          v[a] = (z < g.nz) ? D[z * DP + ky] : cx<float>(0.f, 0.f);
        }
        if constexpr (AZ % 2 == 0) {
          stage1_store_halfin_reg<AZ>(v, t, twf, sc);
        } else {
          stage1_store<AZ, -1>(v, t, twz, sc);
        }
        __syncwarp();
        Cx<float> u[16];
        if (t < AZ) {
          stage2_load(u, t, sc);
          Dft<16, -1>::run(u);
        }
        __syncwarp();
        if (t < AZ) {
#pragma unroll
          for (int k2 = 0; k2 < 16; ++k2) {
            const int kz = t + AZ * k2;
            const float m = __ldg(vcol + (kz <= LZ / 2 ? kz : LZ - kz));
            sc[kz] = cx<float>(u[k2].x * m, u[k2].y * m);
          }
        }
        __syncwarp();
        // 16-byte stores: 4 complex -> 8 bf16 of hi and of lo per lane (never straddle a
        // 64-column block: the line starts at a multiple of 32 columns)
        const size_t g0 = ((size_t)kx * LY + ky) * LZ * 2;
        for (int q = t; q < LZ / 4; q += 16) {
          const size_t gq = g0 + 8 * (size_t)q;
          const size_t off = (gq / 64) * kb_stride + row_off + (gq % 64);
          uint32_t hv[4], lv[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // round-to-nearest-even hardware conversions (re in the low half, im in the high)
            const Cx<float> c = sc[4 * q + j];
            const __nv_bfloat162 h2 = __float22bfloat162_rn(make_float2(c.x, c.y));
            const float2 hf = __bfloat1622float2(h2);
            const __nv_bfloat162 l2 = __float22bfloat162_rn(make_float2(c.x - hf.x, c.y - hf.y));
            hv[j] = *reinterpret_cast<const uint32_t*>(&h2);
            lv[j] = *reinterpret_cast<const uint32_t*>(&l2);
          }
          *reinterpret_cast<uint4*>(hi + off) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
          *reinterpret_cast<uint4*>(lo + off) = make_uint4(lv[0], lv[1], lv[2], lv[3]);
        }
        __syncwarp();
      }
      if (slot == kPre - 1) {
        __syncthreads();   // every read of the upper halves is done
        if (wn < nwork) prefetch_plane_upper<float>(D, DP, plane_ptr(wn), g.nz, g.ny, NT);
      }
    }
  }
}

}  // namespace rsx
