// Learned preconditioner network: conv3d(2->16) ReLU conv3d(16->16) ReLU conv3d(16->1),
// 3^3 kernels, stride 1, zero padding 1; weights rounded to bf16 for every use (FP32
// masters updated by Adam), FP32 activations and accumulation.  The paper has no
// learned component; this is the eigensolver preconditioner the project adds.
//
// Activations and their gradients between the layers live in a packed form ("planes"): per
// (sample, z, y) four chunks [half][part][x][8] of bf16 -- channels 8 half .. 8 half + 7, part 0
// the value rounded to bf16 (hi), part 1 the rounded remainder (lo), x - hi - lo ~ 2^-18 |x| --
// 64 bytes per voxel, what FP32 channels would take.  They are the operands the tensor cores
// read: a TMA box drops them into shared memory in operand layout with no conversion, and
// every consumer used the same hi + lo split of FP32 values before (ReLU is applied where
// they are written; z > 0 exactly where hi > 0).
//
// Kernels: k_conv (the convolution as an implicit GEMM on the tcgen05 tensor cores; the data
// gradient is the same kernel with flipped, transposed weights and the ReLU mask in its
// epilogue), k_wgrad (the weight gradient as an implicit GEMM, per-CTA partial sums reduced
// in fixed order by k_part_reduce), masked MSE loss and Adam.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>

#include "../../include/rsx.h"
#include "api_internal.cuh"
#include "gemm_tcgen05.cuh"
#include "tcgen05_util.cuh"

namespace {

constexpr int kC1 = 2, kC2 = 16, kC3 = 16, kC4 = 1;   // channels in -> hidden -> hidden -> out
// parameter layout (floats): w1 [16][2][27], b1 [16], w2 [16][16][27], b2 [16], w3 [1][16][27], b3 [1]
constexpr int kW1 = kC2 * kC1 * 27, kW2 = kC3 * kC2 * 27, kW3 = kC4 * kC3 * 27;
constexpr int kOffW1 = 0, kOffB1 = kW1, kOffW2 = kOffB1 + kC2, kOffB2 = kOffW2 + kW2, kOffW3 = kOffB2 + kC3,
              kOffB3 = kOffW3 + kW3, kNParams = kOffB3 + kC4;

// shared-memory matrix descriptor without swizzle, core matrices of 8 rows x 16 B: K-major
// operands take lbo between K-adjacent and sbo between M/N-adjacent core matrices, MN-major
// ones (the idesc transpose bits) lbo between K-adjacent and sbo between MN-adjacent ones
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version for tcgen05; swizzle bits 61-63 stay 0
  return d;
}
// instruction descriptor, kind::f16: D f32, A and B bf16, M = 128; mn: both operands MN-major
constexpr uint32_t idesc_f16(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((128u >> 4) << 24);
}

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }
// eight values as 16-byte hi and lo pieces
__device__ __forceinline__ void split8(const float* v, uint4& hi, uint4& lo) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    const float2 hf = __bfloat1622float2(h2);
    h[j] = bf16x2_bits(h2);
    l[j] = bf16x2_bits(__floats2bfloat162_rn(v[2 * j] - hf.x, v[2 * j + 1] - hf.y));
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}
// 16-byte piece index of chunk c (2 half + part) of voxel (zb, y, x) in packed planes
__device__ __forceinline__ size_t piece(size_t zb, int H, int W, int y, int c, int x) {
  return ((zb * H + y) * 4 + c) * (size_t)W + x;
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2,
                                            int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, "
      "%7}], [%2];" ::"r"(rsx::tc::smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(rsx::tc::smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   rsx::tc::smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(rsx::tc::smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rsx::tc::smem_u32(bar)) : "memory");
}
// one lane of a converged warp (always the same one)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n"
      " .reg .pred q;\n"
      " elect.sync _|q, 0xffffffff;\n"
      " selp.u32 %0, 1, 0, q;\n"
      "}\n"
      : "=r"(p));
  return p != 0;
}
// zeros into 16 consecutive TMEM columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
      "r"(0u)
      : "memory");
}

// ---------------------------------------------------------------------------------
// 3^3 convolution as an implicit GEMM on the tensor cores:
//   out[b][co][v] = bias[co] + sum_{t, ci} w[co][ci][t] in[b][ci][v + t - 1].
// A CTA owns an 8 (x) by 16 (y) block of output voxels over up to kCvZ consecutive z slices;
// slice s accumulates in its own 16 TMEM columns (N = output channels, zero-padded).  An
// input plane contributes to three slices, so one MMA takes rows m = 8 yl + xl (128 voxels),
// K = 16 channels and N = 48 columns: the weights of dz = 2, 1, 0 side by side, onto the
// adjacent accumulators of slices p - 2, p - 1, p.  That is 9 taps x (hi, lo) = 18 MMAs per
// plane; with one MMA per tap and slice (N = 16) the A operand is re-read from shared memory
// 54 times per slice, which bounded the layer (32 cycles per read).  The A operand of tap
// (dy, dx) is the staged halo plane [yh][half][part][xh][8 ch] (18 x 10 voxels, 640 B a row)
// started dy rows and dx voxels in: no im2col copy.
//   IN = kInPlanes: the plane is one TMA box of the packed input (zeros outside).
//   IN = kInRaw:    FP32 input of CI = 2 channels, packed into the same plane by kCvStagers threads.
//                   (Packing the dx taps and both parts into the 16 K slots, 3 MMAs per plane, measured
//                   419 against 506 us at 16 x 96^3, but with 9 instead of 54 accumulations per output
//                   its rounding differs from the other layers' by 4e-6, enough to flip ReLUs.)
// Warps 0-3: epilogue of each finished slice while later planes run (kOutRelu: bias, ReLU, packed
// planes; kOutRaw: channel 0 + bias, FP32; kOutMask: packed planes of a gradient, zeroed where the
// forward activation `act` is zero, and its per-CTA channel sums (FP32) for the bias
// gradient).  Every wait is bounded; a timeout sets RSX_ETIMEOUT in the status word, the CTA
// drains what it issued (bounded), frees its TMEM and returns.
constexpr int kInPlanes = 0, kInRaw = 1;
constexpr int kOutRelu = 0, kOutRaw = 1, kOutMask = 2;
constexpr int kCvX = 8, kCvY = 16, kCvZ = 16, kCvSlots = 4;
constexpr int kCvHX = kCvX + 2, kCvHY = kCvY + 2;
constexpr int kCvPlane = kCvHY * 4 * kCvHX * 16;        // 11520 bytes, kInPlanes
constexpr int kCvTap = 48 * 16 * 2;                     // weights of one (dy, dx): 48 rows x 16 K
constexpr int kCvWBytes = 9 * kCvTap;
constexpr int kCvStagers = 192;                         // staging threads of kInRaw, one halo voxel each
static_assert(kCvStagers >= kCvHX * kCvHY, "one halo voxel per staging thread");
constexpr int kCvCols = 16 * kCvZ;                      // TMEM columns
constexpr int cv_threads(int in) { return in == kInPlanes ? 192 : 160 + kCvStagers; }
// shared memory: weights, slots; at least 76 KB so that two CTAs (256 TMEM columns each) share an SM
constexpr int kCvSmem = 77824;
static_assert(kCvSlots * kCvPlane + kCvWBytes <= kCvSmem, "slots and weights");

// weight image of a layer in B operand layout: [tap][row n][16 K], row n = 16 k + co holds dz = 2 - k;
// element (n, ci) at (n / 8) 256 + (ci / 8) 128 + (n % 8) 16 + (ci % 8) 2 bytes, tap = 3 dy + dx.
// flip: the data gradient's weights wt[co][ci][t] = w[ci][co][26 - t].
struct PackJob {
  const float* w;
  unsigned char* img;
  int ci, co, flip;
};
struct PackJobs {
  PackJob j[5];
};
__global__ void k_pack_weights(PackJobs jobs) {
  const PackJob J = jobs.j[blockIdx.y];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 9 * 48 * 16; i += gridDim.x * blockDim.x) {
    const int tap = i / 768, n = (i / 16) % 48, ci = i & 15;
    const int co = n & 15, t = 9 * (2 - n / 16) + tap;
    float v = 0.f;
    if (ci < J.ci && co < J.co) v = J.flip ? J.w[((size_t)ci * J.co + co) * 27 + 26 - t] : J.w[((size_t)co * J.ci + ci) * 27 + t];
    *reinterpret_cast<__nv_bfloat16*>(J.img + tap * kCvTap + (n >> 3) * 256 + (ci >> 3) * 128 + (n & 7) * 16 + (ci & 7) * 2) =
        __float2bfloat16_rn(v);
  }
}

struct ConvArgs {
  const float* raw;        // kInRaw: [B][CI][D][H][W]
  const unsigned char* wimg;
  const float* bias;       // [16] or [1]; kOutMask: none
  void* out;               // packed planes or FP32 [B][D][H][W]
  const uint4* act;        // kOutMask: forward activation (packed planes)
  float* bpart;            // kOutMask: [CTAs][16] channel sums
  int B, D, H, W;
  int* status;
};

template <int IN, int OUT>
__global__ void __launch_bounds__(cv_threads(IN), 2) k_conv(const __grid_constant__ CUtensorMap map, ConvArgs a) {
  using namespace rsx::tc;
  constexpr int CI = kC1;
  constexpr int kPlane = kCvPlane, kW = kCvWBytes;
  extern __shared__ __align__(1024) unsigned char sm[];
  unsigned char* slots = sm;                       // [kCvSlots][kPlane]
  unsigned char* wsm = sm + kCvSlots * kPlane;
  __shared__ __align__(8) uint64_t full[kCvSlots], empty[kCvSlots], ready[kCvZ + 2], wbar;
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh;
  __shared__ float bred[4][16];
  const int D = a.D, H = a.H, W = a.W;
  const int nbx = (W + kCvX - 1) / kCvX, nby = (H + kCvY - 1) / kCvY;
  int blk = blockIdx.x;
  const int bx = blk % nbx;
  blk /= nbx;
  const int by = blk % nby, bz = blk / nby, b = blockIdx.y;
  const int x0 = bx * kCvX, y0 = by * kCvY, z0 = bz * kCvZ;
  const int nzl = min(kCvZ, D - z0), np = nzl + 2;       // planes z0 - 1 + p, p < np
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  volatile int* abort_flag = &abort_sh;
  if (tid == 0) {
    abort_sh = 0;
    for (int i = 0; i < kCvSlots; ++i) {
      mbar_init(&full[i], IN == kInPlanes ? 1 : kCvStagers);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < np; ++i) mbar_init(&ready[i], 1);
    mbar_init(&wbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                 "n"(kCvCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  if (warp < 4) {
    for (int s = 0; s < nzl; ++s) tmem_zero16(tmem + ((uint32_t)(warp * 32) << 16) + 16 * s);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  const size_t vol = (size_t)D * H * W;
  auto plane_in = [&](int p) { return z0 - 1 + p >= 0 && z0 - 1 + p < D; };

  if (warp == 4) {
    // ---- MMA issue: the whole warp runs the loop, one elected lane issues.  (Issued from a
    // single-lane branch, with descriptors built per MMA in a rolled loop, an MMA took ~100 cycles
    // of issue instead of the 32 of its operand reads.)
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool lead = elect_one();
    if (lead) {
      mbar_arrive_expect_tx(&wbar, kW);
      bulk_load(wsm, a.wimg, kW, &wbar);
    }
    __syncwarp();
    bool ok = mbar_wait_warp(&wbar, 0, abort_flag);
    const uint64_t a_desc = smem_desc(smem_u32(slots), 2 * kCvHX * 16, 4 * kCvHX * 16);
    const uint64_t b_desc = smem_desc(smem_u32(wsm), 128, 256);
    int n = 0, p = 0;
    for (; ok && p < np; ++p) {
      if (plane_in(p)) {
        const int slot = n % kCvSlots;
        ok = mbar_wait_warp(&full[slot], (uint32_t)((n / kCvSlots) & 1), abort_flag);
        if (!ok) break;
        // slices p - 2 + k, k = k0 .. k1 of this plane
        const int k0 = max(0, 2 - p), nk = min(2, nzl - 1 - (p - 2)) - k0 + 1;
        const uint32_t acc = tmem + (uint32_t)(16 * (p - 2 + k0));
        const uint32_t id = nk == 3 ? idesc_f16(48, false) : nk == 2 ? idesc_f16(32, false) : idesc_f16(16, false);
        const uint64_t as = a_desc + (uint64_t)(slot * (kPlane / 16)), bs = b_desc + (uint64_t)(32 * k0);
        if (lead) {
#pragma unroll
          for (int t = 0; t < 9; ++t) {   // descriptor addresses count 16 bytes
            const int off = (t / 3) * (4 * kCvHX) + t % 3;
            mma_f16(acc, as + off, bs + t * (kCvTap / 16), id, 1u);
            mma_f16(acc, as + off + kCvHX, bs + t * (kCvTap / 16), id, 1u);
          }
          mma_commit(&empty[slot]);
        }
        ++n;
      }
      if (lead) mma_commit(&ready[p]);
    }
    // no copy or arrival may land after the CTA exits: the weights, then the last commit of every
    // barrier (bounded waits; after a time-out at plane p, ready[p] closes what came before it)
    int last = np - 1;
    if (!ok) {
      for (uint32_t k = 0; k < kWaitLimit && !mbar_try_wait(&wbar, 0); ++k) {
      }
      last = p > 0 ? p : -1;
      if (last >= 0 && lead) mma_commit(&ready[last]);
    }
    for (int i = max(0, n - kCvSlots); i < n; ++i)
      for (uint32_t k = 0; k < kWaitLimit && !mbar_try_wait(&empty[i % kCvSlots], (uint32_t)((i / kCvSlots) & 1)); ++k) {
      }
    for (uint32_t k = 0; last >= 0 && k < kWaitLimit && !mbar_try_wait(&ready[last], 0); ++k) {
    }
    if (!ok) *abort_flag = 1;
    __syncwarp();
  } else if (IN == kInPlanes && warp == 5) {
    if (lane == 0) {
      // ---- plane loads
      bool ok = true;
      int n = 0;
      for (int p = 0; p < np; ++p) {
        if (!plane_in(p)) continue;
        const int slot = n % kCvSlots;
        if (n >= kCvSlots) ok = mbar_wait(&empty[slot], (uint32_t)((n / kCvSlots - 1) & 1), abort_flag);
        if (!ok) break;
        mbar_arrive_expect_tx(&full[slot], kPlane);
        tma_load_5d(slots + slot * kPlane, &map, &full[slot], 0, x0 - 1, 0, y0 - 1, b * D + z0 - 1 + p);
        ++n;
      }
      for (int i = max(0, n - kCvSlots); i < n; ++i)   // copies still in flight after a timeout (bounded)
        for (uint32_t k = 0; k < kWaitLimit && !mbar_try_wait(&full[i % kCvSlots], (uint32_t)((i / kCvSlots) & 1)); ++k) {
        }
    }
  } else if (IN == kInRaw && warp >= 5) {
    // ---- staging: halo voxel (yh, xh) into chunks 0 and 1 (channels 0 .. 7; the others stay zero)
    const int e = tid - 160, yh = e / kCvHX, xh = e - yh * kCvHX;
    const bool mine = e < kCvHY * kCvHX;
    const int y = y0 - 1 + yh, x = x0 - 1 + xh;
    const bool in = mine && y >= 0 && y < H && x >= 0 && x < W;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float* src = a.raw + (size_t)b * CI * vol + (in ? (size_t)y * W + x : 0);
    if (mine)
      for (int i = 0; i < kCvSlots; ++i)
#pragma unroll
        for (int c = 2; c < 4; ++c)
          *reinterpret_cast<uint4*>(slots + i * kPlane + (yh * 4 + c) * (kCvHX * 16) + xh * 16) = make_uint4(0, 0, 0, 0);
    bool ok = true;
    int n = 0;
    for (int p = 0; ok && p < np; ++p) {
      if (!plane_in(p)) continue;
#pragma unroll
      for (int ci = 0; ci < CI; ++ci) v[ci] = in ? __ldg(src + ci * vol + (size_t)(z0 - 1 + p) * H * W) : 0.f;
      const int slot = n % kCvSlots;
      if (n >= kCvSlots) ok = mbar_wait(&empty[slot], (uint32_t)((n / kCvSlots - 1) & 1), abort_flag);
      if (!ok) break;
      if (mine) {
        uint4 hi, lo;
        split8(v, hi, lo);
        unsigned char* d = slots + slot * kPlane + yh * (4 * kCvHX * 16) + xh * 16;
        *reinterpret_cast<uint4*>(d) = hi;
        *reinterpret_cast<uint4*>(d + kCvHX * 16) = lo;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&full[slot]);
      ++n;
    }
  } else if (warp < 4) {
    // ---- epilogue of slice s once plane s + 2 is done
    const int m = warp * 32 + lane, yl = m >> 3, xl = m & 7;   // TMEM lane = GEMM row
    const int y = y0 + yl, x = x0 + xl;
    const bool inside = y < H && x < W;
    float bias[16], bsum[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      bias[c] = OUT == kOutRelu ? __ldg(a.bias + c) : OUT == kOutRaw && c == 0 ? __ldg(a.bias) : 0.f;
      bsum[c] = 0.f;
    }
    for (int s = 0; s < nzl; ++s) {
      if (!mbar_wait_warp(&ready[s + 2], 0, abort_flag)) break;   // lanes outside the box vote too
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float acc[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(16 * s), acc);
      if (!inside) continue;
      const size_t zb = (size_t)b * D + z0 + s;
      if (OUT == kOutRaw) {
        reinterpret_cast<float*>(a.out)[(zb * H + y) * W + x] = acc[0] + bias[0];
      } else {
        uint4* o = reinterpret_cast<uint4*>(a.out);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[8];
          uint4 av;
          if (OUT == kOutMask) av = __ldg(a.act + piece(zb, H, W, y, 2 * h, x));
          const uint32_t aw[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            if (OUT == kOutRelu) {
              v[c] = fmaxf(acc[8 * h + c] + bias[8 * h + c], 0.f);
            } else {
              const uint32_t bits = (c & 1) ? aw[c / 2] >> 16 : aw[c / 2] & 0xFFFFu;   // hi of the activation, >= 0
              v[c] = bits != 0 ? acc[8 * h + c] : 0.f;
              bsum[8 * h + c] += v[c];
            }
          }
          uint4 hi, lo;
          split8(v, hi, lo);
          o[piece(zb, H, W, y, 2 * h, x)] = hi;
          o[piece(zb, H, W, y, 2 * h + 1, x)] = lo;
        }
      }
    }
    if (OUT == kOutMask) {
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        for (int o = 16; o > 0; o >>= 1) bsum[c] += __shfl_xor_sync(0xffffffffu, bsum[c], o);
        if (lane == 0) bred[warp][c] = bsum[c];
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (OUT == kOutMask && tid < 16)
    a.bpart[((size_t)b * gridDim.x + blockIdx.x) * 16 + tid] = (bred[0][tid] + bred[1][tid]) + (bred[2][tid] + bred[3][tid]);
  if (tid == 0 && *abort_flag && a.status) atomicMax(a.status, RSX_ETIMEOUT);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kCvCols) : "memory");
}

// FP32 channels [B][C][vol], C <= 8, into packed planes (channels C .. 15 zero)
template <int C>
__global__ void k_pack_planes(const float* __restrict__ in, int B, int D, int H, int W, uint4* __restrict__ out) {
  const size_t vol = (size_t)D * H * W;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)B * vol; i += (size_t)gridDim.x * blockDim.x) {
    const size_t b = i / vol, v = i - b * vol, zy = v / W;
    const int x = (int)(v - zy * W), y = (int)(zy % H);
    const size_t zb = b * D + zy / H;
    float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < C; ++c) f[c] = __ldg(in + (b * C + c) * vol + v);
    uint4 hi, lo;
    split8(f, hi, lo);
    out[piece(zb, H, W, y, 0, x)] = hi;
    out[piece(zb, H, W, y, 1, x)] = lo;
    out[piece(zb, H, W, y, 2, x)] = out[piece(zb, H, W, y, 3, x)] = make_uint4(0, 0, 0, 0);
  }
}

// Weight gradient of one layer on the tensor cores, per-CTA partial sums
//   part[cta][t][co][ci] = sum_v g[co][v] in[ci][v + t - 1]
// over the CTA's 16 (x) x 3 (y) columns of up to kWgZ output planes; in and g are packed planes.
// The contraction runs over x: an MMA takes K = 16 consecutive x positions, rows m = 16 y' + ci
// (eight input rows y0 - 1 + y' of one plane, of which the five y' < 5 meet an output row) and
// columns n = 16 y + co (three output rows), both operands MN-major (channels contiguous) as
// the TMA boxes leave them; dx starts the A operand dx voxels in, dz takes another plane.  One
// 48-column accumulator per (dz, dx), 27 MMAs (hi.hi + hi.lo + lo.hi) per plane of 48 voxels.
// The blocks y' = y + dy of each accumulator are summed over y once, at the end.  155 us per
// layer at 32 x 32^3, MMA rate the bound (six output rows and N = 96 per CTA, the taps dealt to
// two CTAs: 156 us).  The kernel before built the 27 shifted copies of the input that a K-major
// operand needs for every 16 voxels: 614-832 us.  Accumulation stays short: at most 3 kWgZ MMAs
// per accumulator.  Waits as in k_conv.
constexpr int kWgX = 16, kWgY = 3, kWgZ = 32, kWgRows = 8;
constexpr int kWgInRow = 4 * (kWgX + 2) * 16;           // 1152 bytes
constexpr int kWgIn = kWgRows * kWgInRow;               // 9216
constexpr int kWgGRow = 4 * kWgX * 16;                  // 1024
constexpr int kWgG = kWgY * kWgGRow;                    // 3072
constexpr int kWgInSlots = 6, kWgGSlots = 3;
constexpr int kWgThreads = 192, kWgCols = 512;
// shared memory: the slots (whose bytes the epilogue's 9 x 256 floats reuse); at least 116 KB, so that a CTA has
// its SM's TMEM to itself
constexpr int kWgSmem = 118784;
static_assert(kWgInSlots * kWgIn + kWgGSlots * kWgG <= kWgSmem, "slots");
static_assert(3 * kWgY * 256 * 4 <= kWgInSlots * kWgIn && 9 * 16 * kWgY <= kWgCols, "epilogue buffer, TMEM");

template <int CI, int CO>
__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad(const __grid_constant__ CUtensorMap map_in,
                                                         const __grid_constant__ CUtensorMap map_g, float* __restrict__ part,
                                                         int D, int H, int W, int* status) {
  using namespace rsx::tc;
  extern __shared__ __align__(1024) unsigned char sm[];
  unsigned char* ins = sm;
  unsigned char* gs = sm + kWgInSlots * kWgIn;
  __shared__ __align__(8) uint64_t fin[kWgInSlots], ein[kWgInSlots], fg[kWgGSlots], eg[kWgGSlots], done;
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh;
  const int nbx = (W + kWgX - 1) / kWgX, nby = (H + kWgY - 1) / kWgY;
  int blk = blockIdx.x;
  const int bx = blk % nbx;
  blk /= nbx;
  const int by = blk % nby, bz = blk / nby, b = blockIdx.y;
  const int x0 = bx * kWgX, y0 = by * kWgY, z0 = bz * kWgZ, nz = min(kWgZ, D - z0);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  volatile int* abort_flag = &abort_sh;
  if (tid == 0) {
    abort_sh = 0;
    for (int i = 0; i < kWgInSlots; ++i) {
      mbar_init(&fin[i], 1);
      mbar_init(&ein[i], 1);
    }
    for (int i = 0; i < kWgGSlots; ++i) {
      mbar_init(&fg[i], 1);
      mbar_init(&eg[i], 1);
    }
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                 "n"(kWgCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  if (warp < 4) {
    for (int c = 0; c < 9 * kWgY; ++c) tmem_zero16(tmem + ((uint32_t)(warp * 32) << 16) + 16 * c);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  // input planes z0 - 1 + i, i < nz + 2 (slot i % kWgInSlots; planes outside the box are signalled
  // without a copy and never read); gradient planes z0 + i, i < nz
  auto plane_in = [&](int i) { return z0 - 1 + i >= 0 && z0 - 1 + i < D; };
  if (warp == 5 && lane == 0) {
    bool ok = true;
    int i = 0, k = 0;
    for (; ok && i < nz + 2; ++i) {
      const int slot = i % kWgInSlots;
      if (i >= kWgInSlots) ok = mbar_wait(&ein[slot], (uint32_t)((i / kWgInSlots - 1) & 1), abort_flag);
      if (!ok) break;
      if (plane_in(i)) {
        mbar_arrive_expect_tx(&fin[slot], kWgIn);
        tma_load_5d(ins + slot * kWgIn, &map_in, &fin[slot], 0, x0 - 1, 0, y0 - 1, b * D + z0 - 1 + i);
      } else {
        mbar_arrive(&fin[slot]);
      }
      if (i >= 2) {   // gradient plane i - 2 is the last one that input plane i completes
        const int gslot = k % kWgGSlots;
        if (k >= kWgGSlots) ok = mbar_wait(&eg[gslot], (uint32_t)((k / kWgGSlots - 1) & 1), abort_flag);
        if (!ok) {
          ++i;
          break;
        }
        mbar_arrive_expect_tx(&fg[gslot], kWgG);
        tma_load_5d(gs + gslot * kWgG, &map_g, &fg[gslot], 0, x0, 0, y0, b * D + z0 + k);
        ++k;
      }
    }
    for (int q = max(0, i - kWgInSlots); q < i; ++q)   // copies still in flight after a timeout (bounded)
      for (uint32_t r = 0; r < kWaitLimit && !mbar_try_wait(&fin[q % kWgInSlots], (uint32_t)((q / kWgInSlots) & 1)); ++r) {
      }
    for (int q = max(0, k - kWgGSlots); q < k; ++q)
      for (uint32_t r = 0; r < kWaitLimit && !mbar_try_wait(&fg[q % kWgGSlots], (uint32_t)((q / kWgGSlots) & 1)); ++r) {
      }
  } else if (warp == 4) {   // MMA issue, as in k_conv
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool lead = elect_one();
    const uint64_t a_desc = smem_desc(smem_u32(ins), 128, 576), b_desc = smem_desc(smem_u32(gs), 128, 512);
    constexpr uint32_t id = idesc_f16(16 * kWgY, true);
    bool ok = true;
    int loaded = 0;   // input planes waited for
    int k = 0;
    for (; k < nz; ++k) {
      for (; ok && loaded < k + 3; ++loaded)
        ok = mbar_wait_warp(&fin[loaded % kWgInSlots], (uint32_t)((loaded / kWgInSlots) & 1), abort_flag);
      const int gslot = k % kWgGSlots;
      if (ok) ok = mbar_wait_warp(&fg[gslot], (uint32_t)((k / kWgGSlots) & 1), abort_flag);
      if (!ok) break;
      const uint64_t bh = b_desc + (uint64_t)(gslot * (kWgG / 16)), bl = bh + kWgX;
#pragma unroll
      for (int dz = 0; dz < 3; ++dz) {
        if (!plane_in(k + dz)) continue;
        const uint64_t as = a_desc + (uint64_t)(((k + dz) % kWgInSlots) * (kWgIn / 16));
        if (lead) {
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {   // descriptor addresses count 16 bytes
            const uint32_t d = tmem + (uint32_t)(16 * kWgY * (3 * dz + dx));
            mma_f16(d, as + dx, bh, id, 1u);
            mma_f16(d, as + dx, bl, id, 1u);
            mma_f16(d, as + (kWgX + 2) + dx, bh, id, 1u);
          }
        }
      }
      if (lead) {
        mma_commit(&eg[gslot]);
        mma_commit(&ein[k % kWgInSlots]);   // input plane k is not read again
      }
    }
    if (lead) mma_commit(&done);
    for (uint32_t r = 0; r < kWaitLimit && !mbar_try_wait(&done, 0); ++r) {
    }
    for (int q = max(0, k - kWgGSlots); q < k; ++q)   // no arrival may land after the CTA exits
      for (uint32_t r = 0; r < kWaitLimit && !mbar_try_wait(&eg[q % kWgGSlots], (uint32_t)((q / kWgGSlots) & 1)); ++r) {
      }
    for (int q = max(0, k - kWgInSlots); q < k; ++q)
      for (uint32_t r = 0; r < kWaitLimit && !mbar_try_wait(&ein[q % kWgInSlots], (uint32_t)((q / kWgInSlots) & 1)); ++r) {
      }
    if (!ok) *abort_flag = 1;
    __syncwarp();
  }
  __syncthreads();   // every MMA is complete
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!*abort_flag) {
    // out[dy][co][ci] = sum_y D[16 (y + dy) + ci][16 y + co]: lane (y', ci) holds the terms
    // 0 <= y' - y < 3; one accumulator at a time through [dy][y][co][ci]
    float* buf = reinterpret_cast<float*>(sm);
    float* dst = part + ((size_t)b * gridDim.x + blockIdx.x) * (CO * CI * 27);
    for (int q = 0; q < 9; ++q) {
      if (warp < 4) {
        const int yp = 2 * warp + (lane >> 4), ci = lane & 15;
#pragma unroll
        for (int y = 0; y < kWgY; ++y) {
          float acc[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(16 * (kWgY * q + y)), acc);
          const int dy = yp - y;
          if (dy >= 0 && dy < 3) {
#pragma unroll
            for (int n = 0; n < 16; ++n) buf[((dy * kWgY + y) * 16 + n) * 16 + ci] = acc[n];
          }
        }
      }
      __syncthreads();
      const int dz = q / 3, dx = q - 3 * dz;
      for (int e = tid; e < 3 * CI * CO; e += kWgThreads) {
        const int dy = e / (CI * CO), r = e - dy * CI * CO, co = r / CI, ci = r - co * CI;
        const float* p = buf + (dy * kWgY * 16 + co) * 16 + ci;
        float sum = p[0];
#pragma unroll
        for (int y = 1; y < kWgY; ++y) sum += p[256 * y];
        dst[(9 * dz + 3 * dy + dx) * (CI * CO) + r] = sum;
      }
      __syncthreads();
    }
  }
  if (tid == 0 && *abort_flag && status) atomicMax(status, RSX_ETIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kWgCols) : "memory");
}

// out[perm(o)] = sum over nparts of part[p][o], FP64 accumulation in a fixed order: a block owns
// 32 consecutive outputs (lane = output, coalesced reads), warp w sums the partials p = w,
// w + 32, ... four at a time, and the 32 warp sums of an output are added by a warp's shuffle
// tree (a serial chain of FP64 additions is ~100 cycles each on this part).  nrow > 0: o = [t][r],
// t < 27, r < nrow, goes to [r][t] (the weight gradients).
constexpr int kRedWarps = 32;
__global__ void __launch_bounds__(32 * kRedWarps) k_part_reduce(const float* __restrict__ part, int nparts, int nout, int nrow,
                                                                float* __restrict__ out) {
  __shared__ double red[kRedWarps][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
  if (o < nout) {
    int p = warp;
    for (; p + 3 * kRedWarps < nparts; p += 4 * kRedWarps) {
      s0 += (double)part[(size_t)p * nout + o];
      s1 += (double)part[(size_t)(p + kRedWarps) * nout + o];
      s2 += (double)part[(size_t)(p + 2 * kRedWarps) * nout + o];
      s3 += (double)part[(size_t)(p + 3 * kRedWarps) * nout + o];
    }
    for (; p < nparts; p += kRedWarps) s0 += (double)part[(size_t)p * nout + o];
  }
  red[warp][lane] = (s0 + s1) + (s2 + s3);
  __syncthreads();
  double t = red[lane][warp];   // output 32 blockIdx.x + warp
  for (int k = 16; k > 0; k >>= 1) t += __shfl_xor_sync(0xffffffffu, t, k);
  const int q = blockIdx.x * 32 + warp;
  if (lane == 0 && q < nout) out[nrow > 0 ? (q % nrow) * 27 + q / nrow : q] = (float)t;
}

// masked mean squared error: loss = sum m (y - t)^2 / sum m over the batch; dy = 2 m (y - t) / sum m
// as packed planes (channel 0), and per block the sum of dy (the last layer's bias gradient).
// The mask excludes `border` voxels at every face of each sample.
constexpr int kMseBlocks = 512;
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, const float* __restrict__ t, uint4* __restrict__ dy, int B,
                                             int D, int H, int W, int border, double* __restrict__ loss_acc,
                                             float* __restrict__ bpart) {
  __shared__ float red[8];
  const size_t vol = (size_t)D * H * W;
  const double cnt = (double)B * (D - 2 * border) * (H - 2 * border) * (W - 2 * border);
  const double scale = 2.0 / cnt;
  double s = 0.0;
  float bs = 0.f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)B * vol;
       i += (size_t)gridDim.x * blockDim.x) {
    const size_t b = i / vol, v = i - b * vol, zy = v / W;
    const int x = (int)(v - zy * W), z = (int)(zy / H), yy = (int)(zy - (size_t)z * H);
    const bool in = x >= border && x < W - border && yy >= border && yy < H - border && z >= border && z < D - border;
    const float d = in ? y[i] - t[i] : 0.f;
    const float f[8] = {(float)(scale * d), 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    bs += f[0];
    uint4 hi, lo;
    split8(f, hi, lo);
    const size_t zb = b * D + z;
    dy[piece(zb, H, W, yy, 0, x)] = hi;
    dy[piece(zb, H, W, yy, 1, x)] = lo;
    dy[piece(zb, H, W, yy, 2, x)] = dy[piece(zb, H, W, yy, 3, x)] = make_uint4(0, 0, 0, 0);
    s += (double)d * d;
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    bs += __shfl_xor_sync(0xffffffffu, bs, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(loss_acc, s / cnt);
    red[threadIdx.x >> 5] = bs;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float q = 0.f;
    for (int w = 0; w < 8; ++w) q += red[w];
    bpart[blockIdx.x] = q;
  }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

}  // namespace

struct rsx_net {
  int device = 0;
  float* params = nullptr;   // FP32 masters
  float* grads = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  unsigned char* wimg = nullptr;   // weight images of the five convolutions (k_pack_weights)
  float* act = nullptr;      // packed planes, 16 floats' bytes per voxel each: relu(z1), relu(z2), and two
  size_t act_elems = 0;      // more for the gradients (backward)
  float* part = nullptr;     // partial sums
  size_t part_elems = 0;
  double* loss = nullptr;
  int* status = nullptr;     // device status word (RSX_ETIMEOUT from a bounded wait)
  long long step = 0;
  char err[256] = {0};
};

namespace {

int nfail(rsx_net* n, int code, const char* msg) {
  snprintf(n->err, sizeof(n->err), "%s", msg);
  return code;
}

int ncuda(rsx_net* n, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return RSX_OK;
  snprintf(n->err, sizeof(n->err), "%s: %s", what, cudaGetErrorString(e));
  return RSX_ECUDA;
}

int ngrow(rsx_net* n, float** p, size_t* have, size_t need) {
  if (need <= *have) return RSX_OK;
  if (*p) cudaFree(*p);
  *p = nullptr;
  *have = 0;
  if (cudaMalloc(p, need * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    return nfail(n, RSX_ENOMEM, "network workspace allocation failed");
  }
  *have = need;
  return RSX_OK;
}

constexpr int kImgBytes = kCvWBytes;   // spacing of the weight images
enum { kImgL1 = 0, kImgL2, kImgL3, kImgD3, kImgD2, kImgCount };

// 5-D map of packed planes [B D][H][4][W][8] bf16 with boxes of bx voxels x by rows of one plane
bool plane_map(CUtensorMap* m, const void* base, int B, int D, int H, int W, int bx, int by) {
  rsx::EncodeTiledFn fn = rsx::encode_fn();
  if (!fn) return false;
  cuuint64_t dims[5] = {8, (cuuint64_t)W, 4, (cuuint64_t)H, (cuuint64_t)B * D};
  cuuint64_t strides[4] = {16, (cuuint64_t)W * 16, (cuuint64_t)W * 64, (cuuint64_t)W * 64 * H};
  cuuint32_t box[5] = {8, (cuuint32_t)bx, 4, (cuuint32_t)by, 1}, es[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// CTAs of a convolution over one sample
int conv_blocks(int D, int H, int W) {
  return ((W + kCvX - 1) / kCvX) * ((H + kCvY - 1) / kCvY) * ((D + kCvZ - 1) / kCvZ);
}

// one 3^3 convolution layer on the tensor cores (k_conv); planes: packed input (kInPlanes)
template <int IN, int OUT>
int conv(rsx_net* n, const void* planes, const ConvArgs& a, const char* what, cudaStream_t s) {
  CUtensorMap m{};
  if (IN == kInPlanes && !plane_map(&m, planes, a.B, a.D, a.H, a.W, kCvHX, kCvHY))
    return nfail(n, RSX_ECUDA, "tensor map of the activation planes");
  auto k = k_conv<IN, OUT>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem);
  if (e != cudaSuccess) return ncuda(n, e, what);
  k<<<dim3((unsigned)conv_blocks(a.D, a.H, a.W), (unsigned)a.B), cv_threads(IN), kCvSmem, s>>>(m, a);
  return ncuda(n, cudaGetLastError(), what);
}

template <int CI, int CO>
int wgrad(rsx_net* n, const void* in, const void* g, float* part, int nblk, int B, int D, int H, int W, float* gw,
          cudaStream_t s) {
  CUtensorMap mi{}, mg{};
  if (!plane_map(&mi, in, B, D, H, W, kWgX + 2, kWgRows) || !plane_map(&mg, g, B, D, H, W, kWgX, kWgY))
    return nfail(n, RSX_ECUDA, "tensor map of the gradient planes");
  auto k = k_wgrad<CI, CO>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem);
  if (e != cudaSuccess) return ncuda(n, e, "weight gradient");
  k<<<dim3((unsigned)nblk, (unsigned)B), kWgThreads, kWgSmem, s>>>(mi, mg, part, D, H, W, n->status);
  constexpr int nw = CO * CI * 27;
  k_part_reduce<<<(nw + 31) / 32, 32 * kRedWarps, 0, s>>>(part, B * nblk, nw, CO * CI, gw);
  return ncuda(n, cudaGetLastError(), "weight gradient");
}

// images of the three layers' weights, and of the two data gradients'
int pack_weights(rsx_net* n, bool backward, cudaStream_t s) {
  const float* P = n->params;
  auto img = [&](int i) { return n->wimg + (size_t)i * kImgBytes; };
  PackJobs j;
  j.j[kImgL1] = {P + kOffW1, img(kImgL1), kC1, kC2, 0};
  j.j[kImgL2] = {P + kOffW2, img(kImgL2), kC2, kC3, 0};
  j.j[kImgL3] = {P + kOffW3, img(kImgL3), kC3, kC4, 0};
  j.j[kImgD3] = {P + kOffW3, img(kImgD3), kC4, kC3, 1};
  j.j[kImgD2] = {P + kOffW2, img(kImgD2), kC3, kC2, 1};
  k_pack_weights<<<dim3(27, backward ? kImgCount : 3), 256, 0, s>>>(j);
  return ncuda(n, cudaGetLastError(), "weight images");
}

int forward_layers(rsx_net* n, const float* x, int B, int D, int H, int W, float* out, cudaStream_t s) {
  const size_t vol = (size_t)D * H * W;
  int rc = ngrow(n, &n->act, &n->act_elems, 2 * (size_t)B * kC2 * vol);
  if (rc) return rc;
  float* a1 = n->act;
  float* a2 = n->act + (size_t)B * kC2 * vol;
  const float* P = n->params;
  auto args = [&](int img, const float* bias, void* o) {
    ConvArgs a{};
    a.wimg = n->wimg + (size_t)img * kImgBytes;
    a.bias = bias;
    a.out = o;
    a.B = B;
    a.D = D;
    a.H = H;
    a.W = W;
    a.status = n->status;
    return a;
  };
  ConvArgs l1 = args(kImgL1, P + kOffB1, a1);
  l1.raw = x;
  rc = conv<kInRaw, kOutRelu>(n, nullptr, l1, "layer 1", s);
  if (!rc) rc = conv<kInPlanes, kOutRelu>(n, a1, args(kImgL2, P + kOffB2, a2), "layer 2", s);
  if (!rc) rc = conv<kInPlanes, kOutRaw>(n, a2, args(kImgL3, P + kOffB3, out), "layer 3", s);
  return rc;
}

int forward(rsx_net* n, const float* x, int B, int D, int H, int W, float* out, cudaStream_t s) {
  const int rc = pack_weights(n, false, s);
  return rc ? rc : forward_layers(n, x, B, D, H, W, out, s);
}

// gradients of the masked MSE loss w.r.t. all parameters into n->grads; loss (device double) += value
int backward(rsx_net* n, const float* x, const float* target, int B, int D, int H, int W, int border, cudaStream_t s) {
  // Device memory is what limits a training batch: four sets of planes, 64 floats a voxel.  Each
  // holds what is alive in turn (in stream order): a2 then the partial sums of layer 2's weight
  // gradient, which may run on into gy's, then d z1; gy then x's planes; y then d z2.
  const size_t vol = (size_t)D * H * W, planes = (size_t)B * kC2 * vol;   // floats' worth of one set of planes
  int rc = ngrow(n, &n->act, &n->act_elems, 4 * planes);
  if (rc) return rc;
  const int nwg = ((W + kWgX - 1) / kWgX) * ((H + kWgY - 1) / kWgY) * ((D + kWgZ - 1) / kWgZ);
  const int ncv = conv_blocks(D, H, W);
  const size_t wpart2 = (size_t)B * nwg * kW2, bpart = std::max((size_t)B * ncv * 16, (size_t)kMseBlocks);
  const bool in_planes = wpart2 <= 2 * planes;   // not so only in boxes of a few voxels
  const size_t wpart = in_planes ? (size_t)B * nwg * std::max(kW1, kW3) : wpart2;
  rc = ngrow(n, &n->part, &n->part_elems, wpart + bpart);
  if (rc) return rc;
  float *a1 = n->act, *a2 = a1 + planes, *gy = a2 + planes, *g2 = gy + planes;
  float *part2 = in_planes ? a2 : n->part, *g1 = a2, *xp = gy, *y = g2;
  float* bp = n->part + wpart;
  rc = pack_weights(n, true, s);
  if (!rc) rc = forward_layers(n, x, B, D, H, W, y, s);
  if (rc) return rc;
  k_mse<<<kMseBlocks, 256, 0, s>>>(y, target, (uint4*)gy, B, D, H, W, border, n->loss, bp);
  k_part_reduce<<<1, 32 * kRedWarps, 0, s>>>(bp, kMseBlocks, kC4, 0, n->grads + kOffB3);
  rc = ncuda(n, cudaGetLastError(), "loss");
  auto dgrad = [&](int img, void* o, const float* act) {
    ConvArgs a{};
    a.wimg = n->wimg + (size_t)img * kImgBytes;
    a.out = o;
    a.act = (const uint4*)act;
    a.bpart = bp;
    a.B = B;
    a.D = D;
    a.H = H;
    a.W = W;
    a.status = n->status;
    return a;
  };
  // layer 3: w3 grads from relu(z2) and gy; d z2 = conv(gy, flip(w3)) * (z2 > 0)
  if (!rc) rc = wgrad<kC3, kC4>(n, a2, gy, n->part, nwg, B, D, H, W, n->grads + kOffW3, s);
  if (!rc) rc = conv<kInPlanes, kOutMask>(n, gy, dgrad(kImgD3, g2, a2), "data gradient 3", s);
  if (!rc) k_part_reduce<<<1, 32 * kRedWarps, 0, s>>>(bp, B * ncv, kC3, 0, n->grads + kOffB2);
  // layer 2
  if (!rc) rc = wgrad<kC2, kC3>(n, a1, g2, part2, nwg, B, D, H, W, n->grads + kOffW2, s);
  if (!rc) rc = conv<kInPlanes, kOutMask>(n, g2, dgrad(kImgD2, g1, a1), "data gradient 2", s);
  if (!rc) k_part_reduce<<<1, 32 * kRedWarps, 0, s>>>(bp, B * ncv, kC2, 0, n->grads + kOffB1);
  // layer 1
  if (!rc) k_pack_planes<kC1><<<1024, 256, 0, s>>>(x, B, D, H, W, (uint4*)xp);
  if (!rc) rc = wgrad<kC1, kC2>(n, xp, g1, n->part, nwg, B, D, H, W, n->grads + kOffW1, s);
  return rc ? rc : ncuda(n, cudaGetLastError(), "network backward");
}

}  // namespace

extern "C" {

int rsx_net_create(rsx_net** out, int device) {
  if (!out) return RSX_EINVAL;
  *out = nullptr;
  if (cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    return RSX_ECUDA;
  }
  rsx_net* n = new rsx_net();
  n->device = device;
  if (cudaMalloc(&n->params, kNParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->grads, kNParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->adam_m, kNParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->adam_v, kNParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->wimg, (size_t)kImgCount * kImgBytes) != cudaSuccess || cudaMalloc(&n->loss, sizeof(double)) != cudaSuccess ||
      cudaMalloc(&n->status, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    rsx_net_destroy(n);
    return RSX_ENOMEM;
  }
  cudaMemset(n->params, 0, kNParams * sizeof(float));
  cudaMemset(n->adam_m, 0, kNParams * sizeof(float));
  cudaMemset(n->adam_v, 0, kNParams * sizeof(float));
  cudaMemset(n->status, 0, sizeof(int));
  *out = n;
  return RSX_OK;
}

int rsx_net_param_count(void) { return kNParams; }

int rsx_net_set_params(rsx_net* n, const float* host, int count) {
  if (!n || !host || count != kNParams) return RSX_EINVAL;
  cudaSetDevice(n->device);
  n->step = 0;
  cudaMemset(n->adam_m, 0, kNParams * sizeof(float));
  cudaMemset(n->adam_v, 0, kNParams * sizeof(float));
  return ncuda(n, cudaMemcpy(n->params, host, kNParams * sizeof(float), cudaMemcpyHostToDevice), "set params");
}

int rsx_net_get_params(rsx_net* n, float* host, int count) {
  if (!n || !host || count != kNParams) return RSX_EINVAL;
  cudaSetDevice(n->device);
  return ncuda(n, cudaMemcpy(host, n->params, kNParams * sizeof(float), cudaMemcpyDeviceToHost), "get params");
}

int rsx_net_forward(rsx_net* n, const float* x, int B, int D, int H, int W, float* out, void* stream) {
  rsx::NvtxRange nvtx_range("rsx_net_forward");
  if (!n || !x || !out || B < 1 || D < 1 || H < 1 || W < 1) return RSX_EINVAL;
  cudaSetDevice(n->device);
  return forward(n, x, B, D, H, W, out, (cudaStream_t)stream);
}

int rsx_net_loss_grad(rsx_net* n, const float* x, const float* target, int B, int D, int H, int W, int border,
                      double* loss_host, float* grad_host, void* stream) {
  rsx::NvtxRange nvtx_range("rsx_net_loss_grad");
  if (!n || !x || !target || B < 1 || D <= 2 * border || H <= 2 * border || W <= 2 * border) return RSX_EINVAL;
  cudaSetDevice(n->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaMemsetAsync(n->loss, 0, sizeof(double), s);
  int rc = backward(n, x, target, B, D, H, W, border, s);
  if (rc) return rc;
  if (loss_host) rc = ncuda(n, cudaMemcpyAsync(loss_host, n->loss, sizeof(double), cudaMemcpyDeviceToHost, s), "loss");
  if (!rc && grad_host)
    rc = ncuda(n, cudaMemcpyAsync(grad_host, n->grads, kNParams * sizeof(float), cudaMemcpyDeviceToHost, s), "grads");
  if (!rc) rc = ncuda(n, cudaStreamSynchronize(s), "sync");
  return rc;
}

int rsx_net_train_step(rsx_net* n, const float* x, const float* target, int B, int D, int H, int W, int border,
                       float lr, double* loss_host, void* stream) {
  rsx::NvtxRange nvtx_range("rsx_net_train_step");
  if (!n || !x || !target || B < 1 || D <= 2 * border || H <= 2 * border || W <= 2 * border || !(lr > 0.f))
    return RSX_EINVAL;
  cudaSetDevice(n->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaMemsetAsync(n->loss, 0, sizeof(double), s);
  int rc = backward(n, x, target, B, D, H, W, border, s);
  if (rc) return rc;
  ++n->step;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
  k_adam<<<(kNParams + 255) / 256, 256, 0, s>>>(n->params, n->grads, n->adam_m, n->adam_v, kNParams, lr, b1, b2, 1e-8f,
                                                 c1, c2);
  rc = ncuda(n, cudaGetLastError(), "adam");
  if (!rc && loss_host)
    rc = ncuda(n, cudaMemcpyAsync(loss_host, n->loss, sizeof(double), cudaMemcpyDeviceToHost, s), "loss");
  return rc;
}

// Synchronises the stream, then reports (and clears) a deferred device error of the
// network kernels: RSX_ETIMEOUT when a tensor-core convolution gave up a bounded wait.
int rsx_net_sync_status(rsx_net* n, void* stream) {
  if (!n) return RSX_EINVAL;
  cudaSetDevice(n->device);
  int rc = ncuda(n, cudaStreamSynchronize((cudaStream_t)stream), "sync");
  if (rc) return rc;
  int st = 0;
  rc = ncuda(n, cudaMemcpy(&st, n->status, sizeof(int), cudaMemcpyDeviceToHost), "status");
  if (rc) return rc;
  if (st != RSX_OK) {
    cudaMemset(n->status, 0, sizeof(int));
    return nfail(n, st, "network kernel gave up a bounded wait (timeout)");
  }
  return RSX_OK;
}

const char* rsx_net_last_error(const rsx_net* n) { return n ? n->err : "null network"; }

int rsx_net_destroy(rsx_net* n) {
  if (!n) return RSX_OK;
  cudaSetDevice(n->device);
  cudaDeviceSynchronize();
  void* bufs[] = {n->params, n->grads, n->adam_m, n->adam_v, n->wimg, n->act, n->part, n->loss, n->status};
  for (void* p : bufs)
    if (p) cudaFree(p);
  delete n;
  return RSX_OK;
}

}  // extern "C"
