// FP32 Householder tridiagonalisation with the matrix in the registers of one 16-CTA cluster.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "../../include/rsx.h"
#include "tcgen05_util.cuh"

namespace rsx {
// Same reflectors and outputs as k_tridiag_cluster (eig.cu), n <= 16 NL.  Row i lives in CTA
// i % 16 as its local row i / 16 (the trailing block stays dealt evenly as it shrinks), and the
// columns, like every vector of length n, are taken in the order pi(j) = (j % 16) NL + j / 16, in
// which the entries that one CTA computes are contiguous.  A warp holds NR of its CTA's rows
// (rg NR + r) x 128 columns of that order, four adjacent columns per lane, in registers for the
// whole reduction: a step reads only vectors of length n from shared memory.
//
// What bounds it is the dependent chain of a step, not arithmetic (4/3 n^3 flops are 3 us of the
// chip): norm -> tau, v -> p = tau A22 v -> every CTA knows p -> rank-2 update -> next column.
//  - v is never stored: every thread scales the column entries that it needs.
//  - The row sums of a warp's NR rows come from one transposing butterfly (9 shuffles for 8 rows
//    instead of 40).
//  - One message per step goes from each CTA to each CTA: its entries of p, its entries of the
//    column after this one (as they stand before this step's update) and its share of p^T v, as
//    16-byte asynchronous remote stores that complete bytes on the receiver's mbarrier; a warp
//    per receiver.  The receiver waits for 16 messages, which is also all the synchronisation
//    between CTAs.  Scalar stores of every p entry to every CTA and a cluster barrier took more
//    than half of a step.
//  - The rank-2 update of a step is done in the next one, where it covers the latency of the
//    norm -> tau -> v chain; the column that the next message carries is read off after it.
//  - Every CTA forms the next column for itself from the replica minus the rank-2 terms, so the
//    column costs no exchange of its own; all CTAs do the same operations on the same values, so
//    their replicas, and tau, agree to the bit.
// Entries outside the trailing block have v = p = w = 0 and keep their values; the diagonal is
// read off at the end.  Everything a message or the next step reuses is double-buffered: a CTA
// sends its step k + 1 message only after it has read step k's, and nobody can send step k + 2's
// without it.
//
// n = 512: 1761 us (k_tridiag_cluster) -> 720 us; whole solves with 10 roots 1.30 -> 0.87 ms at n = 256,
// 2.80 -> 1.74 at 512, 5.30 -> 3.29 at 768.
template <int NL>
struct TridiagRegs {
  static constexpr int CS = 16;
  static constexpr int RG = NL > 32 ? 2 : 4;      // row groups (warps that share columns)
  static constexpr int CG = NL / 8;               // column groups of 128
  static constexpr int NR = NL / RG;              // rows per thread
  static constexpr int W = RG * CG;               // warps
  static constexpr int NT = 32 * W;
  static constexpr int NC = CS * NL;              // padded columns
  static constexpr uint32_t kBytes = CS * (2 * NL + 1) * sizeof(float);   // of a step's messages
  struct Smem {
    float col[2][NC];        // current column below the diagonal (zero elsewhere), of even / odd steps
    float p[2][NC];          // received: p
    float pre[2][NC];        // received: the next column before this step's update
    float part[2][CS];       // received: shares of p^T v
    float out[NL];           // own entries of the next column before this step's update, to be sent
    float red[CG][NL];       // row sums of the column groups
    float npart[W];          // shares of the next column's squared norm
    float vav[W];            // shares of v^T A22 v
    uint64_t bar[2];
    int abort;
    int last;                // step whose messages this CTA sent last
  };
};

constexpr uint32_t kTridiagWaitLimit = 1u << 22;   // try_wait rounds (each suspends for a while); 0: no waiting at all

__device__ __forceinline__ uint32_t peer_smem(const void* p, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_async4(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async1(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(dst), "f"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 z, {%6, %7};\n"
      " fma.rn.f32x2 z, x, y, z;\n mov.b64 {%0, %1}, z;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n"
      " mul.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;\n}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
// data written by other CTAs of the cluster: acquire at cluster scope
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(tc::smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bytes that no sender will complete any more, taken off the current phase's count
__device__ __forceinline__ void mbar_complete_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes) : "memory");
}

// Sums of N values per lane over the warp's lanes: N = 2^b values leave row (lane >> (5 - b)) in x[0].
template <int N>
__device__ __forceinline__ void warp_row_sums(float (&x)[N], int lane) {
  int m = 16;
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1, m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const float give = up ? x[q] : x[q + h], keep = up ? x[q + h] : x[q];
      x[q] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  }
  for (; m >= 1; m >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], m);
}

template <int NL>
__global__ void __launch_bounds__(TridiagRegs<NL>::NT, 1)
    k_tridiag_regs(float* __restrict__ A, int n, float* __restrict__ d, float* __restrict__ e,
                   float* __restrict__ tau, uint32_t wait_limit, int* __restrict__ status) {
  using T = TridiagRegs<NL>;
  constexpr int CS = T::CS, RG = T::RG, CG = T::CG, NR = T::NR, W = T::W, NT = T::NT, NC = T::NC;
  constexpr int NB = NR < 8 ? NR : 8;   // rows summed together
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ __align__(16) typename T::Smem sm;
  const int me = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // warps that share a scheduler hold different rows: the first row groups run out of work first
  const int cgp = warp / RG, rg = (warp + warp / 4) % RG;
  const int t = lane + 32 * cgp;                       // columns pi = 4 t .. 4 t + 3
  const int cj0 = 4 * t / NL + CS * (4 * t % NL);      // the first one's index j; + 16 per column
  auto perm = [](int j) { return (j % CS) * NL + j / CS; };
  auto row = [&](int r) { return me + CS * (rg * NR + r); };

  float2 a[NR][2];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = row(r), j = cj0 + 2 * CS * c;
      a[r][c].x = i < n && j < n ? A[(size_t)i * n + j] : 0.f;
      a[r][c].y = i < n && j + CS < n ? A[(size_t)i * n + j + CS] : 0.f;
    }
  if (tid == 0) {
    tc::mbar_init(&sm.bar[0], 1);
    tc::mbar_init(&sm.bar[1], 1);
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // column 0 below the diagonal (row 0 of the symmetric matrix) and own rows of column 1
  {
    float s = 0.f;
    for (int q = tid; q < NC; q += NT) {
      const int j = q / NL + CS * (q % NL);
      const float x = j >= 1 && j < n ? A[j] : 0.f;
      sm.col[0][q] = x;
      if (j >= 2) s += x * x;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sm.npart[warp] = s;
    for (int q = tid; q < NL; q += NT) {
      const int i = me + CS * q;
      sm.out[q] = i < n ? A[(size_t)i * n + 1] : 0.f;
    }
  }
  cl.sync();

  bool live = true;
  // of the last step: reflector scale, (tau/2) p^T v, v and w of own columns
  float sc = 0.f, cc = 0.f;
  float2 v[2], w[2];
  // own rows minus v w^T + w v^T of step k (rows of the trailing block only, four at a time)
  auto update = [&](int k) {
    const int b = k & 1;
#pragma unroll
    for (int r0 = 0; r0 < NR; r0 += 4) {
      if (row(r0 + 3) <= k) continue;
      const int q = me * NL + rg * NR + r0;
      const float4 xc = *reinterpret_cast<const float4*>(sm.col[b] + q);
      const float4 xp = *reinterpret_cast<const float4*>(sm.p[b] + q);
      const float cs[4] = {xc.x, xc.y, xc.z, xc.w}, ps[4] = {xp.x, xp.y, xp.z, xp.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float vr = row(r0 + r) == k + 1 ? 1.f : cs[r] * sc, wr = ps[r] - cc * vr;
        const float2 nv = make_float2(-vr, -vr), nw = make_float2(-wr, -wr);
#pragma unroll
        for (int c = 0; c < 2; ++c) a[r0 + r][c] = fma2(nw, v[c], fma2(nv, w[c], a[r0 + r][c]));
      }
    }
  };
  int k = 0;
  for (; k + 2 < n; ++k) {
    const int m0 = k + 1, b = k & 1;
    const float* col = sm.col[b];
    if (tid == 0) tc::mbar_arrive_expect_tx(&sm.bar[b], T::kBytes);
    float s2 = 0.f;
#pragma unroll
    for (int q = 0; q < W; q += 4) {
      const float4 x = *reinterpret_cast<const float4*>(sm.npart + q);
      s2 += (x.x + x.y) + (x.z + x.w);
    }
    const float alpha = col[perm(m0)];
    // ---- the last step's update, whose operations cover the latency of this step's scalars; the
    // updated column m0 goes into this step's message
    if (k > 0) {
      update(k - 1);
      const int pc = perm(m0);
      if (t == pc >> 2) {
        const bool hi = pc & 2, odd = pc & 1;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          const float2 x = hi ? a[r][1] : a[r][0];
          sm.out[rg * NR + r] = odd ? x.y : x.x;
        }
      }
    }
    // ---- the reflector: beta = -sign(alpha) |x|, tau = 1 + |alpha| / |x|, scale 1 / (alpha - beta)
    float tk = 0.f, beta = alpha;
    sc = 0.f;
    if (s2 != 0.f) {
      const float s = alpha * alpha + s2, rs = rsqrtf(s);
      beta = -copysignf(s * rs, alpha);
      tk = 1.f + fabsf(alpha) * rs;
      sc = 1.f / (alpha - beta);
    }
    // v in place: 1 at m0, the scaled column below, 0 above (where the column is 0)
    {
      const float4 x = *reinterpret_cast<const float4*>(col + 4 * t);
      v[0].x = cj0 == m0 ? 1.f : x.x * sc;
      v[0].y = cj0 + CS == m0 ? 1.f : x.y * sc;
      v[1].x = cj0 + 2 * CS == m0 ? 1.f : x.z * sc;
      v[1].y = cj0 + 3 * CS == m0 ? 1.f : x.w * sc;
    }
    // ---- A22 v on own rows, and this warp's share of v^T A22 v
    constexpr int per = 32 / NB;
    float vav = 0.f;
    if (row(NR - 1) >= m0) {
#pragma unroll
      for (int r0 = 0; r0 < NR; r0 += NB) {
        float acc[NB];
#pragma unroll
        for (int r = 0; r < NB; ++r) {
          const float2 x = fma2(a[r0 + r][1], v[1], mul2(a[r0 + r][0], v[0]));
          acc[r] = x.x + x.y;
        }
        warp_row_sums<NB>(acc, lane);
        const int li = rg * NR + r0 + lane / per;
        if (lane % per == 0) sm.red[cgp][li] = acc[0];
        vav += acc[0] * (me + CS * li == m0 ? 1.f : col[me * NL + li] * sc);
      }
#pragma unroll
      for (int o = 16; o >= per; o >>= 1) vav += __shfl_xor_sync(0xffffffffu, vav, o);
    }
    if (lane == 0) sm.vav[warp] = vav;
    __syncthreads();
    float* pb = sm.p[b];
    float* preb = sm.pre[b];
    {
      // p = tau A22 v and the message (a warp per receiver; the receivers go round when there are
      // fewer warps)
      constexpr int H = (NL + 31) / 32, Q = NL / 4;
      float pl[H], pv = 0.f;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int li = lane + 32 * h;
        float x = 0.f;
        if (li < NL)
#pragma unroll
          for (int g = 0; g < CG; ++g) x += sm.red[g][li];
        pl[h] = me + CS * li >= m0 ? tk * x : 0.f;
      }
#pragma unroll
      for (int q = 0; q < W; q += 4) {
        const float4 x = *reinterpret_cast<const float4*>(sm.vav + q);
        pv += (x.x + x.y) + (x.z + x.w);
      }
      float4 msg;
      float* m4 = &msg.x;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        m4[c] = __shfl_sync(0xffffffffu, pl[0], (4 * lane + c) & 31);
        if (H > 1) {
          const float hi = __shfl_sync(0xffffffffu, pl[H - 1], (4 * lane + c) & 31);
          if (lane >= 8) m4[c] = hi;
        }
      }
      if (lane >= Q && lane < 2 * Q) msg = *reinterpret_cast<const float4*>(sm.out + 4 * (lane - Q));
      float* dst = lane < Q ? pb + me * NL + 4 * lane : preb + me * NL + 4 * (lane - Q);
      for (int to = warp; to < CS; to += W) {
        const uint32_t bar = peer_smem(&sm.bar[b], to);
        if (lane < 2 * Q)
          st_async4(peer_smem(dst, to), msg, bar);
        else if (lane == 2 * Q)
          st_async1(peer_smem(&sm.part[b][me], to), tk * pv, bar);
      }
    }
    // while the messages travel: the reflector for the back-transformation, e and tau
    if (warp == W - 1)
      for (int li = lane; li < NL; li += 32) {
        const int i = me + CS * li;
        if (i > m0 && i < n) A[(size_t)i * n + k] = col[me * NL + li] * sc;
      }
    if (me == 0 && tid == 0) {
      e[k] = beta;
      tau[k] = tk;
    }
    const uint32_t phase = (uint32_t)(k >> 1) & 1u;
    {
      uint32_t tries = 0;
      while (live && (wait_limit == 0 || !mbar_try_wait_cluster(&sm.bar[b], phase)))
        if (++tries > wait_limit || *(volatile int*)&sm.abort) {
          sm.abort = 1;
          live = false;
        }
    }
    // ---- w = p - (tau/2)(p^T v) v
    float pvs = 0.f;
#pragma unroll
    for (int q = 0; q < CS; q += 4) {
      const float4 x = *reinterpret_cast<const float4*>(sm.part[b] + q);
      pvs += (x.x + x.y) + (x.z + x.w);
    }
    cc = 0.5f * tk * pvs;
    {
      const float4 x = *reinterpret_cast<const float4*>(pb + 4 * t);
      const float2 ncc = make_float2(-cc, -cc);
      w[0] = fma2(ncc, v[0], make_float2(x.x, x.y));
      w[1] = fma2(ncc, v[1], make_float2(x.z, x.w));
    }
    // ---- the next column (rows beyond m0) and its squared norm below the next subdiagonal
    {
      const float wm = pb[perm(m0)] - cc;   // v_m0 = 1
      float s = 0.f;
#pragma unroll
      for (int q = tid; q < NC; q += NT) {
        const int j = q / NL + CS * (q % NL);
        const float vj = col[q] * sc;
        const float x = j > m0 && j < n ? preb[q] - (vj * wm + (pb[q] - cc * vj)) : 0.f;
        sm.col[b ^ 1][q] = x;
        if (j > m0 + 1) s += x * x;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) sm.npart[warp] = s;
    }
    if (__syncthreads_or(!live)) {   // the whole CTA leaves together
      live = false;
      break;
    }
  }
  if (live && n > 2) update(n - 3);
  const int last = live ? n - 3 : k;
  if (tid == 0) sm.last = last;
  if (!live && tid == 0 && status) atomicMax(status, RSX_ETIMEOUT);
  // diagonal, last subdiagonal
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = row(r), j = cj0 + CS * c;
      const float x = c & 1 ? a[r][c >> 1].y : a[r][c >> 1].x;
      if (i < n && j == i) d[i] = x;
      if (i == n - 1 && j == n - 2) e[n - 2] = x;
    }
  if (me == 0 && tid == 0 && n >= 3) tau[n - 2] = 0.f;
  cl.sync();   // every message has been sent
  // A CTA that gave up at step `last` (n >= 3 then) waits for the messages on their way to it: those
  // of this step from the CTAs that reached it, and of the next from those that passed it (nobody
  // sends step last + 2's without this CTA's of last + 1; everybody sent last - 1's).
  if (!live && warp == 0) {
    const int theirs = lane < CS ? *cl.map_shared_rank(&sm.last, lane) : -1;
    const uint32_t here = __popc(__ballot_sync(0xffffffffu, theirs >= last));
    const uint32_t next = __popc(__ballot_sync(0xffffffffu, theirs > last));
    if (lane == 0) {
      constexpr uint32_t bytes = T::kBytes / CS;   // of one CTA's message
      uint64_t *b0 = &sm.bar[last & 1], *b1 = &sm.bar[(last & 1) ^ 1];
      if (here < CS) mbar_complete_tx(b0, (CS - here) * bytes);
      if (next > 0) tc::mbar_arrive_expect_tx(b1, next * bytes);
      for (uint32_t i = 0; i < kTridiagWaitLimit && !mbar_try_wait_cluster(b0, (uint32_t)(last >> 1) & 1u); ++i) {
      }
      for (uint32_t i = 0; next > 0 && i < kTridiagWaitLimit && !mbar_try_wait_cluster(b1, (uint32_t)((last + 1) >> 1) & 1u); ++i) {
      }
    }
    __syncwarp();
  }
  cl.sync();   // no CTA leaves while others may still address its shared memory
}
}  // namespace rsx
