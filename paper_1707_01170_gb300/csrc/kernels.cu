// liblrvol kernels for sm_103a.
//
//   k_features, k_mlp_infer, k_labels
//                  learned step multipliers (not in the paper; Eq. 4 stays the
//                  base): per-element features, the network on the tcgen05
//                  tensor cores and training labels (its FP32 training is in
//                  train.cu).
//   k_streamlines, k_streamline_error, k_tube_*
//                  Sec. 5 streamlines (Eq. 4 steps), the Eq. 7 error, tubes.
//   k_trim_raster  Sec. 4.1 trimming: per-pixel interval of a boundary mesh.
//   (k_render, the per-pixel ray casting of Sec. 4, is in render_kernel.cuh, a volume's
//   change of basis in setup.cu, look-up and evaluation at points in points.cu;
//   the device helpers these files share are in device_common.cuh.)
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "device_common.cuh"

namespace lrvol {

// ----------------------------------------------------------------------------
// Learned step sizes: features, BF16 tensor-core inference, fine-step labels.
// The network is 16 -> 64 -> 64 -> 64 -> 1 (ReLU).
// ----------------------------------------------------------------------------
namespace {

// Range of the rendered field on an element: a component's coefficient range
// (convex hull of the Bezier block), or bounds of |v| from the three ranges.
__device__ __forceinline__ void field_range(const FeatureParams &fp, int64_t e, float &lo, float &hi) {
  if (fp.field == LRVOL_FIELD_MAGNITUDE) {
    float s_lo = 0.f, s_hi = 0.f;
    for (int c = 0; c < 3; ++c) {
      const float2 r = fp.range[e * fp.nc + c];
      const float m = fmaxf(fabsf(r.x), fabsf(r.y));
      const float d = r.x > 0.f ? r.x : (r.y < 0.f ? -r.y : 0.f);   // distance of 0 to [r.x, r.y]
      s_hi = fmaf(m, m, s_hi);
      s_lo = fmaf(d, d, s_lo);
    }
    lo = sqrtf(s_lo);
    hi = sqrtf(s_hi);
  } else {
    const float2 r = fp.range[e * fp.nc + (fp.field == LRVOL_FIELD_COMPONENT ? fp.comp : 0)];
    lo = r.x;
    hi = r.y;
  }
}

// The TF in shared memory with aggregates over blocks of kTfBlock bins (the
// largest opacity, the opacity sum, the largest opacity step to the next bin,
// the RGB range), so that an element's bin range [i0, i1] costs at most
// 2 (kTfBlock - 1) single bins plus whole blocks instead of up to 256 bins:
// one element straddling a sharp TF band would otherwise hold its whole warp.
// Maxima and minima are exact in any order; only the opacity sum is added in
// another order.
constexpr int kTfBlock = 16, kTfBlocks = 256 / kTfBlock;

__global__ void k_features(const __grid_constant__ FeatureParams fp, float *__restrict__ out) {
  __shared__ float4 tfs[256];
  __shared__ float b_amax[kTfBlocks], b_asum[kTfBlocks], b_slope[kTfBlocks];
  __shared__ float b_cmin[3][kTfBlocks], b_cmax[3][kTfBlocks];
  for (int q = threadIdx.x; q < 256; q += blockDim.x) tfs[q] = fp.tf[q];
  __syncthreads();
  if (threadIdx.x < kTfBlocks) {
    const int q = threadIdx.x;
    float am = 0.f, as = 0.f, sl = 0.f;
    float mn[3] = {1e30f, 1e30f, 1e30f}, mx[3] = {-1e30f, -1e30f, -1e30f};
    for (int i = q * kTfBlock; i < (q + 1) * kTfBlock; ++i) {
      const float4 t = tfs[i];
      am = fmaxf(am, t.w);
      as += t.w;
      if (i < 255) sl = fmaxf(sl, fabsf(tfs[i + 1].w - t.w));   // the step from bin i to bin i + 1
      mn[0] = fminf(mn[0], t.x); mx[0] = fmaxf(mx[0], t.x);
      mn[1] = fminf(mn[1], t.y); mx[1] = fmaxf(mx[1], t.y);
      mn[2] = fminf(mn[2], t.z); mx[2] = fmaxf(mx[2], t.z);
    }
    b_amax[q] = am;
    b_asum[q] = as;
    b_slope[q] = sl;
    for (int c = 0; c < 3; ++c) {
      b_cmin[c][q] = mn[c];
      b_cmax[c][q] = mx[c];
    }
  }
  __syncthreads();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= fp.n_elem) return;
  {
    // the box as three 16-byte loads (48 bytes per element, so 16-byte aligned)
    const double2 *b2 = reinterpret_cast<const double2 *>(fp.box + 6 * e);
    const double2 q0 = __ldg(b2), q1 = __ldg(b2 + 1), q2 = __ldg(b2 + 2);
    const double b[6] = {q0.x, q0.y, q1.x, q1.y, q2.x, q2.y};
    float w[3], ctr[3];
    for (int a = 0; a < 3; ++a) {
      w[a] = (float)(b[3 + a] - b[a]);
      ctr[a] = (float)(0.5 * (b[a] + b[3 + a]));
    }
    const float ds = __ldg(&fp.elem[e].a.w);
    float lo, hi;
    field_range(fp, e, lo, hi);
    const float xlo = fmaf(lo, fp.tf_scale, fp.tf_bias) * (1.f / 255.f);
    const float xhi = fmaf(hi, fp.tf_scale, fp.tf_bias) * (1.f / 255.f);
    const int i0 = (int)floorf(255.f * fminf(fmaxf(xlo, 0.f), 1.f));
    const int i1 = min(255, (int)ceilf(255.f * fminf(fmaxf(xhi, 0.f), 1.f)));
    float amax = 0.f, asum = 0.f, slope = 0.f;
    float cmin[3] = {1e30f, 1e30f, 1e30f}, cmax[3] = {-1e30f, -1e30f, -1e30f};
    auto bin = [&](int i) {
      const float4 t = tfs[i];
      amax = fmaxf(amax, t.w);
      asum += t.w;
      cmin[0] = fminf(cmin[0], t.x); cmax[0] = fmaxf(cmax[0], t.x);
      cmin[1] = fminf(cmin[1], t.y); cmax[1] = fmaxf(cmax[1], t.y);
      cmin[2] = fminf(cmin[2], t.z); cmax[2] = fmaxf(cmax[2], t.z);
    };
    int i = i0;   // bins i0 .. i1: head to a block boundary, whole blocks, tail
    for (; i <= i1 && (i % kTfBlock) != 0; ++i) bin(i);
    for (; i + kTfBlock - 1 <= i1; i += kTfBlock) {
      const int q = i / kTfBlock;
      amax = fmaxf(amax, b_amax[q]);
      asum += b_asum[q];
      for (int c = 0; c < 3; ++c) {
        cmin[c] = fminf(cmin[c], b_cmin[c][q]);
        cmax[c] = fmaxf(cmax[c], b_cmax[c][q]);
      }
    }
    for (; i <= i1; ++i) bin(i);
    // the largest opacity step between neighbouring bins of the range: steps i -> i + 1 for i0 <= i < i1
    for (i = i0; i < i1 && (i % kTfBlock) != 0; ++i) slope = fmaxf(slope, fabsf(tfs[i + 1].w - tfs[i].w));
    for (; i + kTfBlock - 1 < i1; i += kTfBlock) slope = fmaxf(slope, b_slope[i / kTfBlock]);
    for (; i < i1; ++i) slope = fmaxf(slope, fabsf(tfs[i + 1].w - tfs[i].w));
    float dir[3];
    float nn = 0.f;
    for (int a = 0; a < 3; ++a) {
      dir[a] = ctr[a] - fp.eye[a];
      nn = fmaf(dir[a], dir[a], nn);
    }
    nn = rsqrtf(fmaxf(nn, 1e-30f));
    float proj = 0.f;
    for (int a = 0; a < 3; ++a) {
      dir[a] *= nn;
      proj = fmaf(fabsf(dir[a]), w[a], proj);
    }
    const float f[kIn] = {log2f(64.f * w[0]), log2f(64.f * w[1]), log2f(64.f * w[2]), xlo,
                          xhi, xhi - xlo, amax, asum / (float)(i1 - i0 + 1),
                          255.f * slope, fmaxf(cmax[0] - cmin[0], fmaxf(cmax[1] - cmin[1], cmax[2] - cmin[2])),
                          dir[0], dir[1],
                          dir[2], log2f(2048.f * ds), proj / (8.f * ds), log2f(1.f + 255.f * (xhi - xlo))};
    float *o = out + e * kIn;
    if ((reinterpret_cast<uintptr_t>(out) & 15) == 0) {   // one 64-byte row, four 16-byte stores
      float4 *o4 = reinterpret_cast<float4 *>(o);
#pragma unroll
      for (int c = 0; c < kIn / 4; ++c) o4[c] = make_float4(f[4 * c], f[4 * c + 1], f[4 * c + 2], f[4 * c + 3]);
    } else {                                               // a caller's buffer not 16-byte aligned
#pragma unroll
      for (int c = 0; c < kIn; ++c) o[c] = f[c];
    }
  }
}

// ---- the step network on the 5th-generation tensor cores (tcgen05) ----
// Pack: W1, W2, W3 into the canonical K-major layout of tc_off (B[n][k] =
// W[k][n]), w4 as BF16, biases as FP32.
__global__ void k_mlp_pack(const float *__restrict__ p, uint16_t *__restrict__ out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= kPacked) return;
  if (q < kTcW4) {
    const int K = q < kTcW2 ? kIn : kHid;
    const int base = q < kTcW2 ? kTcW1 : (q < kTcW3 ? kTcW2 : kTcW3);
    const int woff = q < kTcW2 ? kOffW1 : (q < kTcW3 ? kOffW2 : kOffW3);
    const int byte = 2 * (q - base), grp = byte / (K * 16), rem = byte % (K * 16);
    const int n = grp * 8 + (rem % 128) / 16, k = (rem / 128) * 8 + (rem % 16) / 2;
    out[q] = __bfloat16_as_ushort(__float2bfloat16_rn(p[woff + k * kHid + n]));
    return;
  }
  if (q < kTcBias) {
    out[q] = __bfloat16_as_ushort(__float2bfloat16_rn(p[kOffW4 + (q - kTcW4)]));
    return;
  }
  const int r = q - kTcBias, f = r >> 1;
  float bv = 0.f;
  if (f < kHid) bv = p[kOffB1 + f];
  else if (f < 2 * kHid) bv = p[kOffB2 + f - kHid];
  else if (f < 3 * kHid) bv = p[kOffB3 + f - 2 * kHid];
  else if (f == 3 * kHid) bv = p[kOffB4];
  const unsigned bits = __float_as_uint(bv);
  out[q] = q >= kTcEnd ? (uint16_t)0 : ((r & 1) ? (uint16_t)(bits >> 16) : (uint16_t)(bits & 0xffffu));
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (tcgen05): start address, leading byte
// offset (K-adjacent core matrices) and stride byte offset (8-row groups), all
// in 16-byte units; descriptor version 1 at bit 46; no swizzling (bits 61-63 = 0).
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B BF16 (bits 7-9 and 10-12 = 1), both K-major, N >> 3 at bits 17-22,
// M >> 4 at bits 24-28.
constexpr uint32_t kTcM = 128, kTcN = 64;
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((kTcN >> 3) << 17) | ((kTcM >> 4) << 24);
constexpr int kTcSpin = 1 << 20;                 // bound on mbarrier polls per wait ...
constexpr uint64_t kTcWaitNs = 100000000ull;     // ... and on its duration (100 ms)

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :: "r"(tmem), "l"(a), "l"(b), "r"(kTcIdesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(mbar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 16 consecutive FP32 columns of this thread's TMEM lane; the wait is in the
// same statement, so the registers are complete when it returns.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v) {
  uint32_t r[16];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\ttcgen05.wait::ld.sync.aligned;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(mbar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for the mbarrier phase with the given parity; false after kTcSpin polls
// or kTcWaitNs nanoseconds, whichever comes first.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity) {
  if (mbar_try_wait(mbar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (int it = 0; it < kTcSpin; ++it) {
    if (mbar_try_wait(mbar, parity)) return true;
    if (global_ns() - t0 > kTcWaitNs) return false;
  }
  return false;
}

// Synchronisation of the 128 threads of warpgroup g (named barrier 1 + g;
// immediate ids, so only barriers 0-2 are reserved), and the AND of v over them.
__device__ __forceinline__ void wg_sync(int g) {
  if (g == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
  else asm volatile("bar.sync 2, 128;" ::: "memory");
}
__device__ __forceinline__ bool wg_sync_and(int g, bool v) {
  uint32_t r;
  if (g == 0)
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, 1, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(r) : "r"((uint32_t)v) : "memory");
  else
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, 2, 128, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(r) : "r"((uint32_t)v) : "memory");
  return r != 0;
}

// Two BF16 values (round to nearest even) in one word, the first in the low half.
__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&v);
}

constexpr int kTcGroups = 2;                                   // warpgroups (row pipelines) per CTA
constexpr int kTcSmemBytes = 2 * kTcW4 + kTcGroups * 2 * (int)kTcM * kHid;   // weights + operand tiles

// A CTA holds the weights once in shared memory and runs two independent
// pipelines, one per warpgroup, each taking tiles of 128 rows.  Per hidden
// layer the warpgroup's first thread issues the MMAs (M = 128, N = 64, K = 16
// per instruction) from the warpgroup's operand tile and the layer's weights
// into its own 128 x 64 FP32 accumulator in tensor memory, and commits them
// to the warpgroup's mbarrier; every warp then reads its 32 rows back
// (tcgen05.ld), adds the bias, applies ReLU and writes the BF16 activations as
// the next layer's operand tile.  The 64 -> 1 output layer runs on the CUDA
// cores in FP32 on the BF16-rounded operands.  Waits are bounded: a tile
// whose MMAs do not complete gets multiplier 1 (the Eq. 4 step) for its rows
// and for every later tile of that pipeline, and the status word records
// kStatusTimeout.  no_mma (a diagnostic of that path) issues no MMAs and no
// commits, so every pipeline's first wait runs out.
__global__ void __launch_bounds__(128 * kTcGroups, 4) k_mlp_infer(const float *__restrict__ x, int64_t n,
                                                               const uint16_t *__restrict__ packed, float ymin,
                                                               float ymax,
                                                               float *__restrict__ out, uint32_t *__restrict__ status,
                                                               bool no_mma) {
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  uint16_t *sw = reinterpret_cast<uint16_t *>(tc_smem);                         // W1, W2, W3 (18,432 B)
  __shared__ float sb[3 * kHid + 1], sw4[kHid];
  __shared__ __align__(8) unsigned long long mbar[kTcGroups];
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, g = tid >> 7, gt = tid & 127;
  for (int q = tid; q < kTcW4 / 8; q += blockDim.x)
    reinterpret_cast<uint4 *>(sw)[q] = __ldg(reinterpret_cast<const uint4 *>(packed) + q);
  for (int q = tid; q < kHid; q += blockDim.x) sw4[q] = __bfloat162float(__ushort_as_bfloat16(packed[kTcW4 + q]));
  for (int q = tid; q < 3 * kHid + 1; q += blockDim.x)
    sb[q] = __uint_as_float((unsigned)packed[kTcBias + 2 * q] | ((unsigned)packed[kTcBias + 2 * q + 1] << 16));
  if (tid < kTcGroups) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&mbar[tid])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_slot)),
                 "r"(kTcN * kTcGroups) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot + kTcN * g;                               // this pipeline's accumulator
  const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);    // this warp's 32 TMEM lanes
  unsigned char *sa = tc_smem + 2 * kTcW4 + g * 2 * kTcM * kHid;            // this pipeline's operand tile
  const uint32_t a_addr = smem_u32(sa), w_addr = smem_u32(sw), mb = smem_u32(&mbar[g]);
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  uint32_t phase = 0;
  bool ok = true;
  const int64_t tiles = (n + kTcM - 1) / kTcM;
  int64_t tile = (int64_t)blockIdx.x * kTcGroups + g;
  for (; tile < tiles; tile += (int64_t)gridDim.x * kTcGroups) {
    const int64_t row = tile * kTcM + gt;
    {  // layer-1 operand: this thread's feature row in BF16 (K = 16)
      float f[kIn];
      if (row < n && vec) {
        const float4 *xr = reinterpret_cast<const float4 *>(x + row * kIn);
#pragma unroll
        for (int c = 0; c < kIn / 4; ++c) {
          const float4 v = __ldg(xr + c);
          f[4 * c] = v.x; f[4 * c + 1] = v.y; f[4 * c + 2] = v.z; f[4 * c + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < kIn; ++c) f[c] = row < n ? __ldg(x + row * kIn + c) : 0.f;
      }
      unsigned char *dst = sa + tc_off(gt, 0, kIn);
      *reinterpret_cast<uint4 *>(dst) = make_uint4(bf16x2(f[0], f[1]), bf16x2(f[2], f[3]), bf16x2(f[4], f[5]), bf16x2(f[6], f[7]));
      *reinterpret_cast<uint4 *>(dst + 128) =
          make_uint4(bf16x2(f[8], f[9]), bf16x2(f[10], f[11]), bf16x2(f[12], f[13]), bf16x2(f[14], f[15]));
    }
    float y = sb[3 * kHid];
    for (int layer = 0; layer < 3; ++layer) {
      const int K = layer == 0 ? kIn : kHid;
      fence_async_smem();   // the operand tile's generic-proxy stores, visible to the tensor core
      tc_fence_before();
      wg_sync(g);
      if (gt == 0 && !no_mma) {
        tc_fence_after();
        const uint32_t wl = w_addr + 2u * (layer == 0 ? kTcW1 : (layer == 1 ? kTcW2 : kTcW3));
        for (int ks = 0; ks < K / 16; ++ks)
          tc_mma(tmem, tc_desc(a_addr + 256u * ks, 128u, 16u * K), tc_desc(wl + 256u * ks, 128u, 16u * K), ks > 0);
        tc_commit(mb);
      }
      ok = wg_sync_and(g, mbar_wait_bounded(mb, phase));
      phase ^= 1u;
      if (!ok) break;
      tc_fence_after();
      const float *bl = sb + layer * kHid;
      unsigned char *dst = sa + tc_off(gt, 0, kHid);
      float h[16];
#pragma unroll
      for (int c = 0; c < kHid / 8; ++c) {
        if ((c & 1) == 0) tc_ld16(lane_addr + 8 * c, h);   // columns 8c .. 8c + 15
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = 8 * c + 2 * q, i = 8 * (c & 1) + 2 * q;
          w[q] = bf16x2(fmaxf(h[i] + bl[j], 0.f), fmaxf(h[i + 1] + bl[j + 1], 0.f));
        }
        if (layer < 2) {
          *reinterpret_cast<uint4 *>(dst + 128 * c) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int j = 8 * c + 2 * q;
            y = fmaf(__uint_as_float(w[q] << 16), sw4[j], y);
            y = fmaf(__uint_as_float(w[q] & 0xffff0000u), sw4[j + 1], y);
          }
        }
      }
    }
    if (!ok) break;
    if (row < n) out[row] = exp2f(fminf(fmaxf(y, ymin), ymax));
  }
  if (!ok) {
    if (gt == 0) set_status(status, kStatusTimeout);
    for (; tile < tiles; tile += (int64_t)gridDim.x * kTcGroups)
      if (tile * kTcM + gt < n) out[tile * kTcM + gt] = 1.f;
    // one more bounded wait for the MMAs in flight before the accumulator is freed
    if (!no_mma) mbar_wait_bounded(mb, phase ^ 1u);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_slot), "r"(kTcN * kTcGroups)
                 : "memory");
  }
}

// ---- fine-step labels (scalar volumes, FP32 storage) ----
struct SegState {
  uint32_t e;
  float4 ra, rb, rc, rd;
};

template <int P>
__device__ __forceinline__ bool seg_locate(const RenderParams &prm, SegState &st, Block<P, 0, LRVOL_STORE_F32> &blk,
                                           float px, float py, float pz) {
  const bool inside = st.e != kNone && px >= st.ra.x && py >= st.ra.y && pz >= st.ra.z && px < st.rb.x &&
                      py < st.rb.y && pz < st.rb.z;
  if (inside) return true;
  const uint32_t e = forest_lookup(prm.forest, px, py, pz, prm.status);
  if (e >= (uint32_t)prm.n_elem) {   // kNone included
    set_status(prm.status, kStatusBounds);
    return false;
  }
  st.e = e;
  load_record(prm.elem + e, st.ra, st.rb, st.rc, st.rd);
  blk.load(prm.bez + (int64_t)e * blk.BYTES, 0);
  return true;
}

// A lane's sample at parameter t: colour and log2(1 - alpha); false on a failed look-up.
template <int P>
__device__ __forceinline__ bool seg_sample(const RenderParams &prm, const Ray &ray, const float4 *tfb, const float4 *tfd,
                                           float t, SegState &st, Block<P, 0, LRVOL_STORE_F32> &blk, float4 &src) {
  constexpr int N = P + 1;
  const float px = fma_sat(t, ray.d[0], ray.o[0]);
  const float py = fma_sat(t, ray.d[1], ray.o[1]);
  const float pz = fma_sat(t, ray.d[2], ray.o[2]);
  if (!seg_locate<P>(prm, st, blk, px, py, pz)) return false;
  float bx[N], by[N], bz[N];
  monomials<P>(local_u(px, st.ra.x, st.rc.x, st.rd.x), bx);
  monomials<P>(local_u(py, st.ra.y, st.rc.y, st.rd.y), by);
  monomials<P>(local_u(pz, st.ra.z, st.rc.z, st.rd.z), bz);
  src = tf_sample(tfb, tfd, tf_coord(prm, blk.eval(bx, by, bz)));
  return true;
}

// One step of an inclusive scan over the warp: the value o lanes below, where there is one.
__device__ __forceinline__ void scan_mul(float &v, int o) {
  asm volatile("{\n\t.reg .pred p;\n\t.reg .f32 y;\n\tshfl.sync.up.b32 y|p, %0, %1, 0, 0xffffffff;\n\t@p mul.rn.f32 %0, %0, y;\n\t}"
               : "+f"(v) : "r"(o));
}
__device__ __forceinline__ void scan_add(float &v, int o) {
  asm volatile("{\n\t.reg .pred p;\n\t.reg .f32 y;\n\tshfl.sync.up.b32 y|p, %0, %1, 0, 0xffffffff;\n\t@p add.rn.f32 %0, %0, y;\n\t}"
               : "+f"(v) : "r"(o));
}

// Whether the ray at parameter t has left the box [lo, hi) or the cube.
__device__ __forceinline__ bool seg_left(const Ray &ray, const float4 &lo, const float4 &hi, float t) {
  const float px = fma_sat(t, ray.d[0], ray.o[0]);
  const float py = fma_sat(t, ray.d[1], ray.o[1]);
  const float pz = fma_sat(t, ray.d[2], ray.o[2]);
  return !(t < ray.tout) ||
         !(px >= lo.x && py >= lo.y && pz >= lo.z && px < hi.x && py < hi.y && pz < hi.z);
}

// Alg. 2 from transparent over [ta, tb) with samples ta + k*h (each in its element).
template <int P>
__device__ void seg_composite(const RenderParams &prm, const Ray &ray, const float4 *tfb, const float4 *tfd, float ta,
                              float tb, float h, SegState &st, Block<P, 0, LRVOL_STORE_F32> &blk, float &C0, float &C1,
                              float &C2, float &Tr) {
  C0 = C1 = C2 = 0.f;
  Tr = 1.f;
  for (int k = 0; k < kMaxSamplesPerRay; ++k) {
    const float t = __fmaf_rn((float)k, h, ta);
    float4 src;
    if (!(t < tb) || !seg_sample<P>(prm, ray, tfb, tfd, t, st, blk, src)) break;
    const float tn = __fmaf_rn((float)(k + 1), h, ta);
    const float T = ex2_approx(src.w * (__fsub_rn(fminf(tn, tb), t) * prm.inv_xi)), w = fmaf(-Tr, T, Tr);
    C0 = fmaf(w, src.x, C0);
    C1 = fmaf(w, src.y, C1);
    C2 = fmaf(w, src.z, C2);
    Tr *= T;
  }
}

// One lane per ray, one march per composite, candidates until one fails: many
// rays of few samples a visit (rule in launch_labels).
template <int P>
__global__ void __launch_bounds__(128) k_labels_lane(const __grid_constant__ RenderParams prm, float h_fine, float tau,
                                                     const float *__restrict__ cand, int n_cand,
                                                     int32_t *__restrict__ label) {
  __shared__ float4 tfb[kTfEntries], tfd[kTfEntries];
  load_tf(prm, tfb, tfd);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7);
  const int j = prm.row_begin + blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
  if (i >= prm.width || j >= prm.row_end) return;
  Ray ray;
  if (!make_ray(prm.ray, i, j, ray)) return;
  Block<P, 0, LRVOL_STORE_F32> blk;
  SegState st;
  st.e = kNone;
  const float tr_stop = 1.f - prm.alpha_stop;
  float Tfront = 1.f, t = ray.tin;
  for (int visit = 0; visit < kMaxSamplesPerRay && t < ray.tout && Tfront > tr_stop; ++visit) {
    // the visit: element of the heuristic sample at t, up to the first heuristic sample past it
    if (!seg_locate<P>(prm, st, blk, fma_sat(t, ray.d[0], ray.o[0]), fma_sat(t, ray.d[1], ray.o[1]),
                       fma_sat(t, ray.d[2], ray.o[2])))
      return;
    const uint32_t e = st.e;
    const float4 lo = st.ra, hi = st.rb;
    const float ds = lo.w;
    float tb = t;
    for (int q = 0; q < kMaxSamplesPerRay; ++q) {
      tb = __fadd_rn(tb, ds);
      if (seg_left(ray, lo, hi, tb)) break;
    }
    tb = fminf(tb, ray.tout);
    float R0, R1, R2, RT;
    seg_composite<P>(prm, ray, tfb, tfd, t, tb, h_fine, st, blk, R0, R1, R2, RT);
    int best = 0;
    for (int c = 1; c < n_cand; ++c) {
      // the candidate's first sample outside e (or the ray's exit)
      const float sc = __fmul_rn(ds, __ldg(cand + c));
      float tc = t;
      for (int k = 1; k < kMaxSamplesPerRay; ++k) {
        tc = __fmaf_rn((float)k, sc, t);
        if (seg_left(ray, lo, hi, tc)) break;
      }
      tc = fminf(tc, ray.tout);
      float F0, F1, F2, FT, A0, A1, A2, AT;
      seg_composite<P>(prm, ray, tfb, tfd, t, tc, h_fine, st, blk, F0, F1, F2, FT);
      seg_composite<P>(prm, ray, tfb, tfd, t, tc, sc, st, blk, A0, A1, A2, AT);
      const float err = Tfront * fmaxf(fmaxf(fabsf(A0 - F0), fabsf(A1 - F1)), fmaxf(fabsf(A2 - F2), fabsf(AT - FT)));
      if (!(err <= tau)) break;
      best = c;
    }
    atomicMin(label + e, best);
    Tfront *= RT;
    t = tb;
  }
}

// One warp per ray.  A visit's fine samples are independent until they are
// composited, so the lanes take 32 at a time: Alg. 2 over them is a prefix
// product of transmittances and prefix sums of colours.  Lane 0's end is the
// visit's, lane c's that of candidate c; all their fine composites start at
// the visit's first sample, so one march serves them all, and a lane picks its
// composite out of the prefix at its own last sample.  The candidates' own
// samples, a few each, are spread over the lanes as (candidate, sample) slots
// and composited by the candidates' lanes.
//
// A lane per ray with a march per composite (k_labels_lane) evaluates the visit's
// fine samples up to seven times, with 12 of 32 lanes active and a tail of long
// rays: 12.0 ms for a 320x180 camera of a 174,000-element tricubic volume with
// seven candidates, 2.8 ms here.  Held to 128 registers for four CTAs an SM: with the 146 it
// would take, three fit and it is a fifth slower, and five CTAs spill.
// EARLY: longer candidates than one that failed get no end.  The votes and registers
// for it cost up to 3 % of a march, so it is taken where the longest candidate reaches
// past 2.5 chunks (seven candidates, 320x180, h_fine 1/2048: trilinear volume 1.47 ->
// 0.76 ms, tricubic 1.60 -> 1.46; candidates up to 64 steps 4.84 -> 1.96).
template <int P, bool EARLY>
__global__ void __launch_bounds__(128, 4) k_labels(const __grid_constant__ RenderParams prm, float h_fine, float tau,
                                                const float *__restrict__ cand, int n_cand,
                                                int32_t *__restrict__ label) {
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ float4 tfb[kTfEntries], tfd[kTfEntries];
  load_tf(prm, tfb, tfd);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 2 + (warp & 1), j = prm.row_begin + blockIdx.y * 2 + (warp >> 1);
  if (i >= prm.width || j >= prm.row_end) return;
  Ray ray;
  if (!make_ray(prm.ray, i, j, ray)) return;
  Block<P, 0, LRVOL_STORE_F32> blk;
  SegState st;
  st.e = kNone;
  const float tr_stop = 1.f - prm.alpha_stop, inv_h = 1.f / h_fine;
  const bool is_cand = lane > 0 && lane < n_cand;
  const float my_cand = is_cand ? __ldg(cand + lane) : 1.f;
  float Tfront = 1.f, t = ray.tin;
  for (int visit = 0; visit < kMaxSamplesPerRay && t < ray.tout && Tfront > tr_stop; ++visit) {
    // the visit: element of the heuristic sample at t, up to the first heuristic sample past it
    if (!seg_locate<P>(prm, st, blk, fma_sat(t, ray.d[0], ray.o[0]), fma_sat(t, ray.d[1], ray.o[1]),
                       fma_sat(t, ray.d[2], ray.o[2])))
      return;
    const uint32_t e = st.e;
    const float4 lo = st.ra, hi = st.rb;
    const float ds = lo.w;
    float tb = t;
    for (int q = 0; q < kMaxSamplesPerRay; q += 16) {   // 16 steps at a time, a lane each (and its shadow)
      float mine = 0.f;
#pragma unroll
      for (int s = 0; s < 16; ++s) {
        tb = __fadd_rn(tb, ds);
        if (s == (lane & 15)) mine = tb;
      }
      const unsigned left = __ballot_sync(kAll, seg_left(ray, lo, hi, mine));
      if (left) {
        tb = __shfl_sync(kAll, mine, __ffs(left) - 1);
        break;
      }
    }
    tb = fminf(tb, ray.tout);
    // a candidate's end: its first sample outside e (or the ray's exit); nk samples before it
    const float sc = __fmul_rn(ds, my_cand);
    float te = tb;
    int nk = 0;
    bool open = is_cand;
    for (int k = 1; k < kMaxSamplesPerRay && __any_sync(kAll, open); ++k) {
      if (open) {
        const float tc = __fmaf_rn((float)k, sc, t);
        open = !seg_left(ray, lo, hi, tc);
        te = fminf(tc, ray.tout);
        nk = k;
      }
    }
    // the candidates' composites (all their samples lie in e, which every lane
    // holds here): slots off .. off + nk - 1 are candidate `lane`'s samples
    int off = nk;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kAll, off, o);
      if (lane >= o) off += y;
    }
    const int total = __shfl_sync(kAll, off, 31);
    off -= nk;
    float A0 = 0.f, A1 = 0.f, A2 = 0.f, AT = 1.f;
    for (int b = 0; b < total; b += 32) {
      const int slot = b + lane;
      int c = 1;
      for (int q = 2; q < n_cand; ++q)
        if (slot >= __shfl_sync(kAll, off, q)) c = q;
      const float tk = __fmaf_rn((float)(slot - __shfl_sync(kAll, off, c)), __shfl_sync(kAll, sc, c), t);
      float4 src = make_float4(0.f, 0.f, 0.f, 0.f);
      const bool good = slot >= total || seg_sample<P>(prm, ray, tfb, tfd, tk, st, blk, src);
      if (!__all_sync(kAll, good)) return;
      const int k0 = max(b - off, 0), k1 = min(b + 32 - off, nk);   // this lane's samples in these slots
      const int most = (int)__reduce_max_sync(kAll, (unsigned)max(k1 - k0, 0));
      for (int q = 0; q < most; ++q) {
        const int k = k0 + q, from = (off + k - b) & 31;
        const float s0 = __shfl_sync(kAll, src.x, from), s1 = __shfl_sync(kAll, src.y, from);
        const float s2 = __shfl_sync(kAll, src.z, from), lg = __shfl_sync(kAll, src.w, from);
        if (k < k1) {
          const float tq = __fmaf_rn((float)k, sc, t), tn = __fmaf_rn((float)(k + 1), sc, t);
          const float T = ex2_approx(lg * (__fsub_rn(fminf(tn, te), tq) * prm.inv_xi)), w = fmaf(-AT, T, AT);
          A0 = fmaf(w, s0, A0);
          A1 = fmaf(w, s1, A1);
          A2 = fmaf(w, s2, A2);
          AT *= T;
        }
      }
    }
    // fine composites over [t, te)
    float F0 = 0.f, F1 = 0.f, F2 = 0.f, FT = 1.f;
    bool need = lane < n_cand && t < te;
    const float te_max = __uint_as_float(__reduce_max_sync(kAll, need ? __float_as_uint(te) : 0u));   // te >= 0
    // fine samples before te: a quotient, corrected with the samples' own places
    int nf = 0;
    if (need) {
      nf = (int)fminf((te - t) * inv_h, (float)kMaxSamplesPerRay);
      while (nf > 0 && !(__fmaf_rn((float)(nf - 1), h_fine, t) < te)) --nf;
      while (nf < kMaxSamplesPerRay && __fmaf_rn((float)nf, h_fine, t) < te) ++nf;
    }
    float cT = 1.f, cC0 = 0.f, cC1 = 0.f, cC2 = 0.f;   // composite of the earlier chunks
    unsigned open_ends = EARLY ? __ballot_sync(kAll, need) : 0u;
    for (int kb = 0; kb < kMaxSamplesPerRay && (EARLY ? open_ends != 0u : __any_sync(kAll, need)); kb += 32) {
      const float ts = __fmaf_rn((float)(kb + lane), h_fine, t), tn = __fmaf_rn((float)(kb + lane + 1), h_fine, t);
      const bool act = ts < te_max;
      float4 src = make_float4(0.f, 0.f, 0.f, 0.f);
      const bool good = !act || seg_sample<P>(prm, ray, tfb, tfd, ts, st, blk, src);
      if (!__all_sync(kAll, good)) return;
      const float T = act ? ex2_approx(src.w * (__fsub_rn(tn, ts) * prm.inv_xi)) : 1.f;
      float p = T;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) scan_mul(p, o);
      float before = __shfl_up_sync(kAll, p, 1);
      if (lane == 0) before = 1.f;
      const float Tr = cT * before, w = fmaf(-Tr, T, Tr);
      float s0 = w * src.x, s1 = w * src.y, s2 = w * src.z;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        scan_add(s0, o);
        scan_add(s1, o);
        scan_add(s2, o);
      }
      // an end's last sample, clipped there, is in this chunk
      const bool fin = need && nf <= kb + 32;
      const int last = fin ? max(nf - 1 - kb, 0) : 0;
      const float gt = __shfl_sync(kAll, ts, last), gTr = __shfl_sync(kAll, Tr, last), glg = __shfl_sync(kAll, src.w, last);
      const float g0 = __shfl_sync(kAll, src.x, last), g1 = __shfl_sync(kAll, src.y, last), g2 = __shfl_sync(kAll, src.z, last);
      const int prev = last > 0 ? last - 1 : 0;
      float E0 = __shfl_sync(kAll, s0, prev), E1 = __shfl_sync(kAll, s1, prev), E2 = __shfl_sync(kAll, s2, prev);
      if (fin) {
        if (last == 0) E0 = E1 = E2 = 0.f;
        const float Te = ex2_approx(glg * (__fsub_rn(te, gt) * prm.inv_xi)), we = fmaf(-gTr, Te, gTr);
        F0 = fmaf(we, g0, cC0 + E0);
        F1 = fmaf(we, g1, cC1 + E1);
        F2 = fmaf(we, g2, cC2 + E2);
        FT = gTr * Te;
        need = false;
      }
      cT *= __shfl_sync(kAll, p, 31);
      cC0 += __shfl_sync(kAll, s0, 31);
      cC1 += __shfl_sync(kAll, s1, 31);
      cC2 += __shfl_sync(kAll, s2, 31);
      if constexpr (EARLY) {
        // the label is the candidate before the first that fails: those behind one that failed need no end
        open_ends = __ballot_sync(kAll, need);
        if (open_ends > 1u) {
          const float err = Tfront * fmaxf(fmaxf(fabsf(A0 - F0), fabsf(A1 - F1)), fmaxf(fabsf(A2 - F2), fabsf(AT - FT)));
          const unsigned failed = __ballot_sync(kAll, is_cand && fin && !(err <= tau));
          if (failed) {
            need &= lane < __ffs(failed);
            open_ends &= failed ^ (failed - 1u);   // up to the first that failed
          }
        }
      }
    }
    const float err = Tfront * fmaxf(fmaxf(fabsf(A0 - F0), fabsf(A1 - F1)), fmaxf(fabsf(A2 - F2), fabsf(AT - FT)));
    const unsigned bad = __ballot_sync(kAll, is_cand && !(err <= tau));
    if (lane == 0) atomicMin(label + e, bad ? __ffs(bad) - 2 : n_cand - 1);
    Tfront *= __shfl_sync(kAll, FT, 0);
    t = tb;
  }
}

}  // namespace

cudaError_t launch_features(const FeatureParams &fp, float *out, cudaStream_t s) {
  if (fp.n_elem == 0) return cudaSuccess;
  k_features<<<(unsigned)((fp.n_elem + 127) / 128), 128, 0, s>>>(fp, out);
  return cudaGetLastError();
}

cudaError_t launch_mlp_pack(const float *params, uint16_t *packed, cudaStream_t s) {
  k_mlp_pack<<<(kPacked + 255) / 256, 256, 0, s>>>(params, packed);
  return cudaGetLastError();
}

__device__ uint32_t g_mlp_status;

uint32_t *mlp_status_word() {
  void *p = nullptr;
  return cudaGetSymbolAddress(&p, g_mlp_status) == cudaSuccess ? static_cast<uint32_t *>(p) : nullptr;
}

cudaError_t launch_mlp_infer(const float *x, int64_t n, const uint16_t *packed, float ymin, float ymax, float *out,
                             uint32_t *status, cudaStream_t s, bool no_mma) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  static bool smem_set = false;
  if (!smem_set) {
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmemBytes);
    if (e != cudaSuccess) return e;
    smem_set = true;
  }
  // Shared memory (about 52 KB per CTA) allows at most 4 CTAs per SM, so their
  // tensor memory (128 columns each) never exceeds the SM's 512 columns.
  const int64_t tiles = (n + kTcM - 1) / kTcM;
  const int64_t blocks = std::min<int64_t>((tiles + kTcGroups - 1) / kTcGroups, 4 * (int64_t)sms);
  k_mlp_infer<<<(unsigned)std::max<int64_t>(blocks, 1), 128 * kTcGroups, kTcSmemBytes, s>>>(x, n, packed, ymin, ymax,
                                                                                           out, status, no_mma);
  return cudaGetLastError();
}

struct LabelRoute {
  bool by_lane;   // k_labels_lane; else k_labels ...
  bool early;     // ... with EARLY
};

// Whether a lane a ray is faster than a warp a ray.  A warp wastes lanes on a visit
// of few samples, lanes need many rays to fill the GPU and march again for every
// candidate.  Per ray and visit the lane's work is its samples (1 + 0.091 each), the
// warp's a chunk of 32 fine samples up to the longest candidate's end and the steps of
// the candidate with most samples (1 + 0.26 and 0.026 each); rays up to 2,500 (lanes)
// and 85 (warps) per SM are hidden in one another's latency.  An element is crossed
// in `chord` on average, its Eq. 4 step is ds, and a candidate passes the more often the
// larger tau is.  The constants are a fit to 5,271 timings (seven volumes of degree 1 to
// 3, 64x36 to 1280x720 rays, 1 to 16 candidates, h_fine 1/64 to 1/8192, tau 1e-5 to 1e-2),
// in which the choice is within 5 % of the faster kernel for 97 % and 0.5 % on average.
// 174,000 tricubic elements, lane / warp: 640x360 rays, one candidate, h_fine 1/256 0.51 /
// 4.9 ms; 320x180, seven candidates, h_fine 1/2048 12.0 / 2.8 ms.
static LabelRoute label_route(const LabelCost &cost, int64_t rays, int sms, double h_fine, double tau, const float *cand,
                              int n_cand) {
  const double pass = 1 / (1 + std::exp(-2.23 - 0.66 * std::log10(tau / 4e-4)));
  double samples = cost.chord / h_fine, farthest = cost.chord, steps = 0, reached = 1;
  for (int c = 1; c < n_cand; ++c) {
    const double sc = cost.ds * cand[c], length = sc < cost.chord ? cost.chord + 0.5 * sc : sc;
    reached *= pass;
    samples += reached * (length / h_fine + length / sc);
    farthest = std::max(farthest, length);
    steps = std::max(steps, length / sc);
  }
  const double per_sm = (double)rays / sms;
  const double chunks = farthest / (32 * h_fine);
  return {1.29 * (1 + 0.091 * samples) * (1 + per_sm / 2540) <
              1.05 * (1 + 0.257 * chunks + 0.0256 * steps) * (1 + per_sm / 85),
          n_cand > 1 && chunks > 2.5};
}

cudaError_t launch_labels(const RenderParams &prm, int degree, const LabelCost &cost, float h_fine, float tau,
                          const float *cand, const float *cand_host, int n_cand, int32_t *label, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int w = prm.width, h = prm.row_end - prm.row_begin;
  const LabelRoute route = label_route(cost, (int64_t)w * h, sms, h_fine, tau, cand_host, n_cand);
  auto launch = [&](auto degree_c) {
    constexpr int P = decltype(degree_c)::value;
    const dim3 patches((unsigned)((w + 1) / 2), (unsigned)((h + 1) / 2));   // four rays a CTA, a 2x2 patch
    if (route.by_lane)
      k_labels_lane<P><<<dim3((unsigned)((w + 15) / 16), (unsigned)((h + 7) / 8)), 128, 0, s>>>(prm, h_fine, tau, cand,
                                                                                             n_cand, label);
    else if (route.early)
      k_labels<P, true><<<patches, 128, 0, s>>>(prm, h_fine, tau, cand, n_cand, label);
    else
      k_labels<P, false><<<patches, 128, 0, s>>>(prm, h_fine, tau, cand, n_cand, label);
  };
  switch (degree) {
    case 1: launch(std::integral_constant<int, 1>()); break;
    case 2: launch(std::integral_constant<int, 2>()); break;
    case 3: launch(std::integral_constant<int, 3>()); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Trimming (Sec. 4.1).  The paper's z-prepass rasterises the boundary mesh's
// front and back faces into two depth buffers; here each triangle is one
// warp that tests the rays of the pixels in its conservative screen box
// (watertight test, FP32, in the oracle's order of operations) and keeps
// the nearest front-face and farthest back-face distances with atomics on
// the float bits (t > 0, so bit order is value order).
// ----------------------------------------------------------------------------
namespace {

__device__ __forceinline__ float pick3(int k, float x, float y, float z) { return k == 0 ? x : (k == 1 ? y : z); }

// Watertight ray/triangle test (Woop, Benthin and Wald, JCGT 2013), FP32,
// with the oracle's order of operations; component selection by value so
// that nothing goes to local memory.
// v: the triangle's 9 coordinates relative to the ray's origin (in registers).
__device__ __forceinline__ bool tri_hit(const float *d, const float *v, float &t, bool &front) {
  const float d0 = d[0], d1 = d[1], d2 = d[2];
  int kz = 0;
  if (fabsf(d1) > fabsf(pick3(kz, d0, d1, d2))) kz = 1;
  if (fabsf(d2) > fabsf(pick3(kz, d0, d1, d2))) kz = 2;
  int kx = kz == 2 ? 0 : kz + 1, ky = kx == 2 ? 0 : kx + 1;
  const float dz = pick3(kz, d0, d1, d2);
  if (dz < 0.f) {
    const int w = kx;
    kx = ky;
    ky = w;
  }
  const float Sx = __fdiv_rn(pick3(kx, d0, d1, d2), dz), Sy = __fdiv_rn(pick3(ky, d0, d1, d2), dz);
  const float Sz = __fdiv_rn(1.f, dz);
  const float a0 = v[0], a1 = v[1], a2 = v[2], b0 = v[3], b1 = v[4], b2 = v[5], c0 = v[6], c1 = v[7], c2 = v[8];
  const float Akz = pick3(kz, a0, a1, a2), Bkz = pick3(kz, b0, b1, b2), Ckz = pick3(kz, c0, c1, c2);
  const float Ax = __fsub_rn(pick3(kx, a0, a1, a2), __fmul_rn(Sx, Akz));
  const float Ay = __fsub_rn(pick3(ky, a0, a1, a2), __fmul_rn(Sy, Akz));
  const float Bx = __fsub_rn(pick3(kx, b0, b1, b2), __fmul_rn(Sx, Bkz));
  const float By = __fsub_rn(pick3(ky, b0, b1, b2), __fmul_rn(Sy, Bkz));
  const float Cx = __fsub_rn(pick3(kx, c0, c1, c2), __fmul_rn(Sx, Ckz));
  const float Cy = __fsub_rn(pick3(ky, c0, c1, c2), __fmul_rn(Sy, Ckz));
  float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
  float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
  float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
  if (U == 0.f || V == 0.f || W == 0.f) {
    U = __double2float_rn(__dsub_rn(__dmul_rn((double)Cx, (double)By), __dmul_rn((double)Cy, (double)Bx)));
    V = __double2float_rn(__dsub_rn(__dmul_rn((double)Ax, (double)Cy), __dmul_rn((double)Ay, (double)Cx)));
    W = __double2float_rn(__dsub_rn(__dmul_rn((double)Bx, (double)Ay), __dmul_rn((double)By, (double)Ax)));
  }
  if ((U < 0.f || V < 0.f || W < 0.f) && (U > 0.f || V > 0.f || W > 0.f)) return false;
  const float det = __fadd_rn(__fadd_rn(U, V), W);
  if (det == 0.f) return false;
  const float Az = __fmul_rn(Sz, Akz), Bz = __fmul_rn(Sz, Bkz), Cz = __fmul_rn(Sz, Ckz);
  const float T = __fadd_rn(__fadd_rn(__fmul_rn(U, Az), __fmul_rn(V, Bz)), __fmul_rn(W, Cz));
  if (det > 0.f ? !(T > 0.f) : !(T < 0.f)) return false;
  t = __fdiv_rn(T, det);
  front = det > 0.f;
  return true;
}

// The pixels whose centres (i + 1/2, j + 1/2) project into the image-plane
// box [amin, amax] x [bmin, bmax], widened by a margin: 1/4 pixel plus 1e-5
// of the box's coordinates in pixels.  The FP32 projection of a primitive's
// vertices, with approximate reciprocals (2^-22 relative), and the FP32 pixel
// rays of make_ray are each within a few ulps of exact, a few thousandths of a
// pixel even for narrow fields of view, so every pixel whose ray can hit the
// primitive is in the box.  False if the box holds no pixel centre.
struct PixelScale {
  float ax, ay, bx, by;   // pixel = a * image-plane coordinate + b - 1/2
  __device__ __forceinline__ explicit PixelScale(const RayConsts &K)
      : ax(1.f / K.sxs), ay(1.f / K.sys), bx(-K.sxo / K.sxs), by(-K.syo / K.sys) {}
};
__device__ __forceinline__ bool pixel_box(const PixelScale &S, int width, int height, float amin, float amax, float bmin,
                                          float bmax, int &i0, int &i1, int &j0, int &j1) {
  const float ia = fmaf(amin, S.ax, S.bx) - 0.5f, ib = fmaf(amax, S.ax, S.bx) - 0.5f;
  const float ja = fmaf(bmin, S.ay, S.by) - 0.5f, jb = fmaf(bmax, S.ay, S.by) - 0.5f;
  const float mi = 0.25f + 1e-5f * (fabsf(amin) + fabsf(amax) + 1.f) * fabsf(S.ax);
  const float mj = 0.25f + 1e-5f * (fabsf(bmin) + fabsf(bmax) + 1.f) * fabsf(S.ay);
  // clamp before converting (NaN widens to the whole image)
  const float lo_i = fmaxf(fminf(ia, ib) - mi, -1.f), hi_i = fminf(fmaxf(ia, ib) + mi, (float)width);
  const float lo_j = fmaxf(fminf(ja, jb) - mj, -1.f), hi_j = fminf(fmaxf(ja, jb) + mj, (float)height);
  i0 = max(0, (int)ceilf(lo_i));
  i1 = min(width - 1, (int)floorf(hi_i));
  j0 = max(0, (int)ceilf(lo_j));
  j1 = min(height - 1, (int)floorf(hi_j));
  return i0 <= i1 && j0 <= j1;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__global__ void k_trim_init(float2 *__restrict__ out, int64_t n) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) out[q] = make_float2(__int_as_float(0x7f800000), 0.f);
}

// Walks the (primitive, pixel) pairs of a warp's 32 primitives, 32 pairs at a
// time: lane l's primitive has the cnt pairs from exc on.  A lane finds its
// pair's primitive by counting the primitives that start at or before it: a
// mask of the starts within the 32 pairs and the number of earlier ones, kept
// along.  The primitives' data lie in shared memory, those with pairs first, in
// order ("slots").
struct PairWalk {
  long long w0, w1;       // this warp's pairs
  long long rel;          // the lane's first pair, relative to the current 32
  unsigned first;         // exc modulo 2^32: a primitive has < 2^31 pairs
  int slot;               // the lane's slot
  int before;             // primitives that start before the current 32 pairs
  bool has;

  // `split` warps share the pairs, this one is `part`
  __device__ __forceinline__ PairWalk(int lane, int cnt, int split, int part) {
    const unsigned all = 0xffffffffu;
    long long inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(all, inc, o);
      if (lane >= o) inc += y;
    }
    const long long total = __shfl_sync(all, inc, 31), exc = inc - cnt;
    const long long chunk = (((total + split - 1) / split) + 31) & ~31ll;
    w0 = (long long)part * chunk;
    w1 = w0 + chunk < total ? w0 + chunk : total;
    rel = exc - w0;
    first = (unsigned)exc;
    has = cnt > 0;
    const unsigned nonempty = __ballot_sync(all, has);
    slot = __popc(nonempty & ((1u << lane) - 1u));
    before = __popc(__ballot_sync(all, has && rel < 0));
  }
  // slot of pair base + lane, for base = w0, w0 + 32, ...
  __device__ __forceinline__ int next(int lane) {
    const unsigned starts = __reduce_or_sync(0xffffffffu, has && rel >= 0 && rel < 32 ? 1u << (int)rel : 0u);
    const int s = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
    before += __popc(starts);
    rel -= 32;
    return s;
  }
};

// Row of pixel `pix` of a box of width bw.  Below 2^21 pixels the FP32 product
// with 1/bw is within 0.5/bw of (pix + 1/2)/bw, so its floor is exact.
__device__ __forceinline__ unsigned box_row(unsigned pix, unsigned bw, float inv_bw) {
  return pix < (1u << 21) ? (unsigned)(((float)pix + 0.5f) * inv_bw) : pix / bw;
}

// One warp takes 32 consecutive triangles: lane l projects triangle l of the
// group and finds its pixel box, then the warp walks the group's (triangle,
// pixel) pairs.  Small triangles (most of a fine mesh covers a pixel centre or
// none) then cost one lane's set-up instead of a warp's.  `split` warps share a
// group, each taking a contiguous part of its pairs, so a coarse mesh of large
// triangles still spreads over the GPU.  A fine mesh is bound by the set-up of
// its triangles (2.4 M of them at 1280x720: 92 us; 104 with divisions in the
// projection and the pairs searched by shuffles; 99 with the vertices staged
// through shared memory).
__global__ void __launch_bounds__(128) k_trim_raster(const RayConsts K, int width, int height,
                                                     const float *__restrict__ tri, int64_t n_tri, int split,
                                                     float2 *__restrict__ out) {
  // A triangle that has pairs: its vertices (perspective: relative to the eye),
  // 1/width, width, first pair and corner of its box.  80 bytes, so that eight
  // lanes' 16-byte accesses to eight slots touch every bank once.
  struct Slot {
    float4 q[5];
  };
  __shared__ Slot slots[4][32];
  const int lane = threadIdx.x & 31;
  Slot *sl = slots[threadIdx.x >> 5];
  const int64_t wid = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int64_t group = wid / split;
  const int part = (int)(wid - group * split);
  if (group * 32 >= n_tri) return;   // whole warp
  float v[9];
  const int64_t tr = group * 32 + lane;
#pragma unroll
  for (int c = 0; c < 9; ++c) v[c] = tr < n_tri ? __ldg(tri + 9 * tr + c) : 0.f;
  int i0 = 0, j0 = 0, bw = 1, cnt = 0;
  if (tr < n_tri) {
    // conservative pixel box of the projected triangle (whole image when a
    // vertex is at or behind the eye plane; nothing when all three are)
    float amin = __int_as_float(0x7f800000), amax = -amin, bmin = amin, bmax = -amin;
    bool full = false;
    int behind = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float X = v[3 * q] - K.E[0], Y = v[3 * q + 1] - K.E[1], Z = v[3 * q + 2] - K.E[2];
      const float r = X * K.R[0] + Y * K.R[1] + Z * K.R[2];
      const float u = X * K.U[0] + Y * K.U[1] + Z * K.U[2];
      float a = r, b = u;
      if (K.persp) {
        const float z = X * K.F[0] + Y * K.F[1] + Z * K.F[2];
        if (!(z > 1e-6f)) {
          full = true;
          ++behind;
          continue;
        }
        const float iz = rcp_approx(z);
        a = r * iz;
        b = u * iz;
      }
      amin = fminf(amin, a);
      amax = fmaxf(amax, a);
      bmin = fminf(bmin, b);
      bmax = fmaxf(bmax, b);
    }
    int i1 = width - 1, j1 = height - 1;
    if (behind < 3 && (full || pixel_box(PixelScale(K), width, height, amin, amax, bmin, bmax, i0, i1, j0, j1))) {
      if (full) {
        i0 = 0;
        j0 = 0;
        i1 = width - 1;
        j1 = height - 1;
      }
      bw = i1 - i0 + 1;
      cnt = bw * (j1 - j0 + 1);   // <= 32768^2 < 2^31
    }
  }
  PairWalk walk(lane, cnt, split, part);
  if (walk.has) {
    Slot &m = sl[walk.slot];
    if (K.persp) {
#pragma unroll
      for (int c = 0; c < 9; ++c) v[c] = __fsub_rn(v[c], K.E[c % 3]);
    }
    m.q[0] = make_float4(v[0], v[1], v[2], v[3]);
    m.q[1] = make_float4(v[4], v[5], v[6], v[7]);
    m.q[2] = make_float4(v[8], 1.f / (float)bw, __int_as_float(bw), __uint_as_float(walk.first));
    m.q[3] = make_float4(__int_as_float(i0), __int_as_float(j0), 0.f, 0.f);
  }
  __syncwarp();
  for (long long base = walk.w0; base < walk.w1; base += 32) {
    const Slot &m = sl[walk.next(lane)];
    if (base + lane >= walk.w1) continue;
    const float4 q0 = m.q[0], q1 = m.q[1], q2 = m.q[2], q3 = m.q[3];
    const unsigned bw = __float_as_uint(q2.z), pix = (unsigned)(base + lane) - __float_as_uint(q2.w);
    const unsigned row = box_row(pix, bw, q2.y);
    const int i = __float_as_int(q3.x) + (int)(pix - row * bw), j = __float_as_int(q3.y) + (int)row;
    Ray ray;
    make_ray(K, i, j, ray);   // origin and direction; the unit-cube interval is not needed here
    float tv[9] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x};
    if (!K.persp) {
#pragma unroll
      for (int c = 0; c < 9; ++c) tv[c] = __fsub_rn(tv[c], ray.o[c % 3]);
    }
    float t;
    bool front;
    if (!tri_hit(ray.d, tv, t, front)) continue;
    unsigned *slot = reinterpret_cast<unsigned *>(out + (int64_t)j * width + i);
    if (front)
      atomicMin(slot, __float_as_uint(t));
    else
      atomicMax(slot + 1, __float_as_uint(t));
  }
}

}  // namespace

cudaError_t launch_trim(const RayConsts &ray, int width, int height, const float *tri, int64_t n_tri, float *out,
                        cudaStream_t s) {
  const int64_t npix = (int64_t)width * height;
  float2 *o = reinterpret_cast<float2 *>(out);
  k_trim_init<<<(unsigned)((npix + 255) / 256), 256, 0, s>>>(o, npix);
  if (n_tri > 0) {
    // warps per group of 32 triangles: about 512 pairs per warp when the
    // mesh covers the image twice, 1 for fine meshes, at most 256
    const int64_t groups = (n_tri + 31) / 32;
    int64_t split = (2 * npix + groups * 512 - 1) / (groups * 512);
    split = split < 1 ? 1 : (split > 256 ? 256 : split);
    const int64_t warps = groups * split;
    k_trim_raster<<<(unsigned)((warps + 3) / 4), 128, 0, s>>>(ray, width, height, tri, n_tri, (int)split, o);
  }
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Streamlines (Sec. 5): dx/dt = f(x) by explicit Runge-Kutta methods (Eq. 5),
// one thread per seed.  The outer loop keeps x as an unevaluated float pair
// (hi + lo, about 48 significant bits) and t in FP64: on GB300 FP64
// arithmetic runs at a small fraction of the FP32 rate, and compensated
// FP32 sums keep the accumulation exact enough that the steps are not lost
// to rounding (the reason for the paper's double-precision outer loop,
// Sec. 5.5).  Stage increments h * sum a_ij k_j are formed in FP32 (they
// are small against x) and added exactly; the field is evaluated in FP32
// at the FP32 rounding of the stage point, reusing the element (box and
// block in registers) while consecutive points stay in it.
// ----------------------------------------------------------------------------
namespace {

struct __align__(32) SLSample {
  double x, y, z, t;
};

// A sample x = (double)x_hi + (double)x_lo.  With fewer than 32 lines per
// warp the tracing kernel stores the float pairs (x_hi, x_lo, y_hi, y_lo,
// z_hi, z_lo) and t in the same 32 bytes instead, and a second pass widens
// them in place with all 32 lanes of a warp on one line's samples: FP64
// instructions cost the same per warp whatever the number of active lanes.
// With full warps the extra pass over the samples costs more than it saves.
__device__ __forceinline__ void store_sample(SLSample *o, const float *xh, const float *xl, double t, bool pairs) {
  if (pairs) {
    float4 *o4 = reinterpret_cast<float4 *>(o);
    o4[0] = make_float4(xh[0], xl[0], xh[1], xl[1]);
    o4[1] = make_float4(xh[2], xl[2], __int_as_float(__double2loint(t)), __int_as_float(__double2hiint(t)));
  } else {
    *o = SLSample{(double)xh[0] + (double)xl[0], (double)xh[1] + (double)xl[1], (double)xh[2] + (double)xl[2], t};
  }
}

struct SLTab {
  int s, embedded, q_low;
  float a[6][6], b[6], bh[6];
};

// Butcher tableaus in the order of LRVOL_RK1 .. LRVOL_RKF45 (coefficients in FP32).
__constant__ SLTab c_sl_tab[9] = {
    {1, 0, 0, {}, {1.f}, {}},
    {2, 0, 0, {{0.f}, {0.5f}}, {0.f, 1.f}, {}},
    {3, 0, 0, {{0.f}, {0.5f}, {-1.f, 2.f}}, {1.f / 6, 2.f / 3, 1.f / 6}, {}},
    {4, 0, 0, {{0.f}, {0.5f}, {0.f, 0.5f}, {0.f, 0.f, 1.f}}, {1.f / 6, 1.f / 3, 1.f / 3, 1.f / 6}, {}},
    {4, 0, 0, {{0.f}, {1.f / 3}, {-1.f / 3, 1.f}, {1.f, -1.f, 1.f}}, {0.125f, 0.375f, 0.375f, 0.125f}, {}},
    {6, 0, 4,
     {{0.f},
      {0.25f},
      {3.f / 32, 9.f / 32},
      {1932.f / 2197, -7200.f / 2197, 7296.f / 2197},
      {439.f / 216, -8.f, 3680.f / 513, -845.f / 4104},
      {-8.f / 27, 2.f, -3544.f / 2565, 1859.f / 4104, -11.f / 40}},
     {16.f / 135, 0.f, 6656.f / 12825, 28561.f / 56430, -9.f / 50, 2.f / 55},
     {25.f / 216, 0.f, 1408.f / 2565, 2197.f / 4104, -0.2f, 0.f}},
    {2, 1, 1, {{0.f}, {1.f}}, {0.5f, 0.5f}, {1.f, 0.f}},
    {4, 1, 2, {{0.f}, {0.5f}, {0.f, 0.75f}, {2.f / 9, 1.f / 3, 4.f / 9}}, {2.f / 9, 1.f / 3, 4.f / 9, 0.f},
     {7.f / 24, 0.25f, 1.f / 3, 0.125f}},
    {6, 1, 4,
     {{0.f},
      {0.25f},
      {3.f / 32, 9.f / 32},
      {1932.f / 2197, -7200.f / 2197, 7296.f / 2197},
      {439.f / 216, -8.f, 3680.f / 513, -845.f / 4104},
      {-8.f / 27, 2.f, -3544.f / 2565, 1859.f / 4104, -11.f / 40}},
     {16.f / 135, 0.f, 6656.f / 12825, 28561.f / 56430, -9.f / 50, 2.f / 55},
     {25.f / 216, 0.f, 1408.f / 2565, 2197.f / 4104, -0.2f, 0.f}},
};

// x + d for x = hi + lo and a float d, renormalised (two-sum, then fast two-sum)
__device__ __forceinline__ void ff_add(float &hi, float &lo, float d) {
  const float s = __fadd_rn(hi, d);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(d, bb));
  const float t = __fadd_rn(e, lo);
  hi = __fadd_rn(s, t);
  lo = __fsub_rn(t, __fsub_rn(hi, s));
}

// TREES: the forest has trees; else a head word names the element.
template <int P, int STORE, bool TREES>
struct SLField {
  static constexpr int N = P + 1;
  float4 ra, rb, rc, rd;
  uint32_t cur;
  Block<P, 1, STORE> blk;

  // f at the FP32 point p; false outside [0,1]^3 (or on a failed look-up)
  __device__ __forceinline__ bool eval(const SLParams &sp, float px, float py, float pz, float &v0, float &v1,
                                       float &v2) {
    if (!(px >= 0.f && px <= 1.f && py >= 0.f && py <= 1.f && pz >= 0.f && pz <= 1.f)) return false;
    if (!locate(sp, px, py, pz)) return false;
    float bx[N], by[N], bz[N];
    monomials<P>(local_u(px, ra.x, rc.x, rd.x), bx);
    monomials<P>(local_u(py, ra.y, rc.y, rd.y), by);
    monomials<P>(local_u(pz, ra.z, rc.z, rd.z), bz);
    blk.components(bx, by, bz, v0, v1, v2);
    return true;
  }

  __device__ __forceinline__ bool locate(const SLParams &sp, float px, float py, float pz) {
    if (cur != kNone && px >= ra.x && py >= ra.y && pz >= ra.z && px < rb.x && py < rb.y && pz < rb.z) return true;
    const uint32_t e =
        TREES ? forest_lookup(sp.forest, px, py, pz, sp.status) : forest_head(sp.forest, px, py, pz) & ~kLeaf;
    if (e >= (uint32_t)sp.n_elem) {   // kNone included
      set_status(sp.status, kStatusBounds);
      return false;
    }
    cur = e;
    load_record(sp.elem + e, ra, rb, rc, rd);
    blk.load(sp.bez + (int64_t)e * blk.BYTES, 0);
    return true;
  }
};

// One streamline, seed q.
template <int P, int STORE, bool TREES>
__device__ __forceinline__ void trace_line(const SLParams &sp, const double *__restrict__ seeds, int64_t q,
                                           SLSample *__restrict__ out, int32_t *__restrict__ count,
                                           int32_t *__restrict__ status) {
  const SLTab &T = c_sl_tab[sp.method];
  SLField<P, STORE, TREES> F;
  F.cur = kNone;
  float xh[3], xl[3];
  for (int a = 0; a < 3; ++a) {
    const double s = seeds[3 * q + a];
    xh[a] = __double2float_rn(s);
    xl[a] = __double2float_rn(s - (double)xh[a]);
  }
  SLSample *o = out + q * (int64_t)sp.max_samples;
  int nout = 0, st = 0;
  float v0, v1, v2;
  if (!(xh[0] >= 0.f && xh[0] <= 1.f && xh[1] >= 0.f && xh[1] <= 1.f && xh[2] >= 0.f && xh[2] <= 1.f) ||
      !F.locate(sp, xh[0], xh[1], xh[2])) {
    count[q] = 0;
    status[q] = 1;
    return;
  }
  store_sample(o, xh, xl, 0.0, sp.pair_out);
  nout = 1;
  // FP64 runs at a small fraction of the FP32 rate on GB300, so the time
  // bookkeeping keeps to one FP64 add per step: h and fl32(h) change only
  // with the element (Eq. 4 rule) or the controller (adaptive rule); the
  // comparisons with t_end compare bit patterns (t, t_end >= 0 order like
  // their bits); the loop ends on a flag set with the step that reaches t_end.
  double t = 0.0;
  float dsn = F.ra.w;  // Eq. 4 step of the element holding x_n
  double h = sp.rule == 0 ? sp.h : (sp.rule == 1 ? sp.h * (double)dsn : (sp.h > 0.0 ? sp.h : (double)dsn));
  float hf_h = __double2float_rn(h), ds_h = dsn;   // fl32(h); the Eq. 4 step h was formed from
  const long long t_end_bits = __double_as_longlong(sp.t_end);
  bool done = false;   // t >= t_end (t_end > 0 is checked on the host)
  for (;;) {
    if (done) {
      st = 0;
      break;
    }
    if (nout >= sp.max_samples) {
      st = 2;
      break;
    }
    if (sp.rule == 1 && dsn != ds_h) {
      h = sp.h * (double)dsn;
      hf_h = __double2float_rn(h);
      ds_h = dsn;
    }
    bool taken = false, left = false;
    float nh[3], nl[3];
    for (int tries = 0; tries < 64 && !taken; ++tries) {
      const double tn = t + h;
      const bool last = __double_as_longlong(tn) > t_end_bits;
      double hs = h;
      float hf = hf_h;
      if (last) {
        hs = sp.t_end - t;
        hf = __double2float_rn(hs);
      }
      float k[6][3];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        if (i < T.s) {
          float d0 = 0.f, d1 = 0.f, d2 = 0.f;
#pragma unroll
          for (int j = 0; j < i; ++j) {
            const float a = T.a[i][j];
            d0 = fmaf(a, k[j][0], d0);
            d1 = fmaf(a, k[j][1], d1);
            d2 = fmaf(a, k[j][2], d2);
          }
          float yh0 = xh[0], yl0 = xl[0], yh1 = xh[1], yl1 = xl[1], yh2 = xh[2], yl2 = xl[2];
          if (i > 0) {
            ff_add(yh0, yl0, hf * d0);
            ff_add(yh1, yl1, hf * d1);
            ff_add(yh2, yl2, hf * d2);
          }
          if (!left && !F.eval(sp, yh0, yh1, yh2, v0, v1, v2)) left = true;
          k[i][0] = v0;
          k[i][1] = v1;
          k[i][2] = v2;
        }
      }
      if (left) break;
      float D0 = 0.f, D1 = 0.f, D2 = 0.f;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        if (i < T.s) {
          const float b = T.b[i];
          D0 = fmaf(b, k[i][0], D0);
          D1 = fmaf(b, k[i][1], D1);
          D2 = fmaf(b, k[i][2], D2);
        }
      }
      if (sp.rule == 2) {
        float E0 = 0.f, E1 = 0.f, E2 = 0.f;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          if (i < T.s) {
            const float e = T.b[i] - T.bh[i];
            E0 = fmaf(e, k[i][0], E0);
            E1 = fmaf(e, k[i][1], E1);
            E2 = fmaf(e, k[i][2], E2);
          }
        }
        const float err = hf * sqrtf(fmaf(E0, E0, fmaf(E1, E1, E2 * E2)));
        float fac = err > 0.f ? 0.9f * powf(sp.tol_f / err, 1.f / (float)(T.q_low + 1)) : 5.f;
        fac = fminf(fmaxf(fac, 0.2f), 5.f);
        if (err > sp.tol_f) {
          h = hs * (double)fac;
          hf_h = __double2float_rn(h);
          continue;
        }
        if (!last) {
          h = hs * (double)fac;
          hf_h = __double2float_rn(h);
        }
      }
      for (int a = 0; a < 3; ++a) {
        nh[a] = xh[a];
        nl[a] = xl[a];
      }
      ff_add(nh[0], nl[0], hf * D0);
      ff_add(nh[1], nl[1], hf * D1);
      ff_add(nh[2], nl[2], hf * D2);
      if (!(nh[0] >= 0.f && nh[0] <= 1.f && nh[1] >= 0.f && nh[1] <= 1.f && nh[2] >= 0.f && nh[2] <= 1.f) ||
          !F.locate(sp, nh[0], nh[1], nh[2])) {
        left = true;
        break;
      }
      dsn = F.ra.w;
      t = last ? sp.t_end : tn;
      done = last || __double_as_longlong(tn) == t_end_bits;
      taken = true;
    }
    if (left) {
      st = 1;
      break;
    }
    if (!taken) {
      st = 3;
      break;
    }
    for (int a = 0; a < 3; ++a) {
      xh[a] = nh[a];
      xl[a] = nl[a];
    }
    store_sample(o + nout++, xh, xl, t, sp.pair_out);
  }
  count[q] = nout;
  status[q] = st;
}

// Persistent threads: a grid that fits on the GPU at once takes lines from
// a counter until none is left, so lines of very different lengths do not
// leave a partial last wave idle behind the longest one.  Only the first
// `lanes` lanes of each warp trace lines: with fewer lines than the GPU has
// warp slots, one line per warp keeps a line from waiting on its warp-mates'
// element look-ups (a line's steps are a sequential chain, so its latency is
// what a small rake of seeds waits for).  The look-up is inlined at every stage,
// so forests without a tree have a kernel without the walk (24,000 lines of a
// tricubic FP32 volume, RK4: 1,114 us, 1,227 with it, where 292 bytes spill instead
// of 168).  MIN: CTAs on an SM that the registers have to allow, 0 for any (launch_sl).
template <int P, int STORE, bool TREES, int MIN>
__global__ void __launch_bounds__(128, MIN) k_streamlines(
    const __grid_constant__ SLParams sp, const double *__restrict__ seeds, int64_t n, int lanes,
    SLSample *__restrict__ out, int32_t *__restrict__ count, int32_t *__restrict__ status) {
  if ((int)(threadIdx.x & 31) >= lanes) return;
  for (;;) {
    const int64_t q = (int64_t)atomicAdd(sp.queue, 1ull);
    if (q >= n) return;
    trace_line<P, STORE, TREES>(sp, seeds, q, out, count, status);
  }
}

// NaN if any operand is NaN (fminf and fmaxf would drop it)
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float d;
  asm("{\n\t.reg .f32 t;\n\tmin.NaN.f32 t, %1, %2;\n\tmin.NaN.f32 %0, t, %3;\n\t}" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float d;
  asm("{\n\t.reg .f32 t;\n\tmax.NaN.f32 t, %1, %2;\n\tmax.NaN.f32 %0, t, %3;\n\t}" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// ---- one line by four lanes ----
// A small rake waits for the chain of its slowest line, so a line's stage is
// split over a group of four lanes: lane c < 3 holds coordinate c of the point
// and of the stages, evaluates component c of the field (from the plain
// per-component blocks, a third of the coefficients) and adds its coordinate's
// increments; the lanes exchange the stage point by three shuffles, and every
// decision is taken by all lanes on the same values.  Lane 3 shadows lane 2 and
// writes the time.  Each operation is the one trace_line does for that
// coordinate, so the samples are the same bits.
template <int P, int STORE>
__device__ __forceinline__ void trace_line_group(const SLParams &sp, const double *__restrict__ seeds, int64_t q,
                                                 SLSample *__restrict__ out, int32_t *__restrict__ count,
                                                 int32_t *__restrict__ status, unsigned group, int l4) {
  constexpr int N = P + 1;
  const SLTab &T = c_sl_tab[sp.method];
  const int c = l4 < 3 ? l4 : 2;
  float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra, rc = ra, rd = ra;   // an empty box
  Block<P, 2, STORE> blk;
  auto in_cube = [](float x, float y, float z) {
    return x >= 0.f && x <= 1.f && y >= 0.f && y <= 1.f && z >= 0.f && z <= 1.f;
  };
  // The element holding the point, its record and block; false outside the
  // cube.  The signs of the six differences are exact, and the smallest and
  // largest of three take one instruction each, where a chain of six compares
  // waits for each predicate.  A box lies in the cube.
  auto locate = [&](float px, float py, float pz) -> bool {
    const float below = min3_nan(px - ra.x, py - ra.y, pz - ra.z);
    const float above = max3_nan(px - rb.x, py - rb.y, pz - rb.z);
    if (below >= 0.f && above < 0.f) return true;
    if (!in_cube(px, py, pz)) return false;
    const uint32_t e = forest_lookup<true>(sp.forest, px, py, pz, sp.status);
    if (e >= (uint32_t)sp.n_elem) {   // kNone included
      set_status(sp.status, kStatusBounds);
      return false;
    }
    load_record(sp.elem + e, ra, rb, rc, rd);
    blk.load(sp.bezc + (int64_t)e * blk.BYTES, c);
    return true;
  };
  auto field = [&](float px, float py, float pz) -> float {   // component c in the current element
    float bx[N], by[N], bz[N], unused0, unused1, v;
    monomials<P>(local_u(px, ra.x, rc.x, rd.x), bx);
    monomials<P>(local_u(py, ra.y, rc.y, rd.y), by);
    monomials<P>(local_u(pz, ra.z, rc.z, rd.z), bz);
    blk.components(bx, by, bz, unused0, unused1, v);
    return v;
  };
  auto gather = [&](float v, float &x, float &y, float &z) {
    x = __shfl_sync(group, v, 0, 4);
    y = __shfl_sync(group, v, 1, 4);
    z = __shfl_sync(group, v, 2, 4);
  };
  float2 *o = reinterpret_cast<float2 *>(out + q * (int64_t)sp.max_samples) + l4;   // this lane's quarter of sample 0
  auto store = [&](int at, float hi, float lo, double t) {   // as store_sample with pairs
    o[4 * (int64_t)at] = l4 < 3 ? make_float2(hi, lo)
                                : make_float2(__int_as_float(__double2loint(t)), __int_as_float(__double2hiint(t)));
  };
  const double s = seeds[3 * q + c];
  float xh = __double2float_rn(s), xl = __double2float_rn(s - (double)xh);
  float px, py, pz;
  gather(xh, px, py, pz);
  int nout = 0, st = 0;
  if (!locate(px, py, pz)) {
    if (l4 == 0) {
      count[q] = 0;
      status[q] = 1;
    }
    return;
  }
  store(0, xh, xl, 0.0);
  nout = 1;
  double t = 0.0;
  float dsn = ra.w;  // Eq. 4 step of the element holding x_n
  double h = sp.rule == 0 ? sp.h : (sp.rule == 1 ? sp.h * (double)dsn : (sp.h > 0.0 ? sp.h : (double)dsn));
  float hf_h = __double2float_rn(h), ds_h = dsn;   // fl32(h); the Eq. 4 step h was formed from
  const long long t_end_bits = __double_as_longlong(sp.t_end);
  bool done = false;
  for (;;) {
    if (done) {
      st = 0;
      break;
    }
    if (nout >= sp.max_samples) {
      st = 2;
      break;
    }
    if (sp.rule == 1 && dsn != ds_h) {
      h = sp.h * (double)dsn;
      hf_h = __double2float_rn(h);
      ds_h = dsn;
    }
    bool taken = false, left = false;
    float nh = 0.f, nl = 0.f, k[6];
    double tn = t + h;          // its FP64 latency passes under the first stage
    k[0] = field(px, py, pz);   // x_n, which the last step or the seed located: the same for every attempt
    for (int tries = 0; tries < 64 && !taken; ++tries) {
      const bool last = __double_as_longlong(tn) > t_end_bits;
      double hs = h;
      float hf = hf_h;
      if (last) {
        hs = sp.t_end - t;
        hf = __double2float_rn(hs);
      }
#pragma unroll
      for (int i = 1; i < 6; ++i) {
        if (i < T.s) {
          float d = 0.f;
#pragma unroll
          for (int j = 0; j < i; ++j) d = fmaf(T.a[i][j], k[j], d);
          float yh = xh, yl = xl;
          ff_add(yh, yl, hf * d);
          gather(yh, px, py, pz);
          k[i] = 0.f;
          if (!left && locate(px, py, pz))
            k[i] = field(px, py, pz);
          else
            left = true;
        }
      }
      if (left) break;
      float D = 0.f;
#pragma unroll
      for (int i = 0; i < 6; ++i)
        if (i < T.s) D = fmaf(T.b[i], k[i], D);
      if (sp.rule == 2) {
        float E = 0.f, E0, E1, E2;
#pragma unroll
        for (int i = 0; i < 6; ++i)
          if (i < T.s) E = fmaf(T.b[i] - T.bh[i], k[i], E);
        gather(E, E0, E1, E2);
        const float err = hf * sqrtf(fmaf(E0, E0, fmaf(E1, E1, E2 * E2)));
        float fac = err > 0.f ? 0.9f * powf(sp.tol_f / err, 1.f / (float)(T.q_low + 1)) : 5.f;
        fac = fminf(fmaxf(fac, 0.2f), 5.f);
        if (err > sp.tol_f || !last) {
          h = hs * (double)fac;
          hf_h = __double2float_rn(h);
        }
        if (err > sp.tol_f) {
          tn = t + h;
          continue;
        }
      }
      nh = xh;
      nl = xl;
      ff_add(nh, nl, hf * D);
      gather(nh, px, py, pz);
      if (!locate(px, py, pz)) {
        left = true;
        break;
      }
      dsn = ra.w;
      t = last ? sp.t_end : tn;
      done = last || __double_as_longlong(tn) == t_end_bits;
      taken = true;
    }
    if (left) {
      st = 1;
      break;
    }
    if (!taken) {
      st = 3;
      break;
    }
    xh = nh;
    xl = nl;
    store(nout++, xh, xl, t);
  }
  if (l4 == 0) {
    count[q] = nout;
    status[q] = st;
  }
}

// `lines` groups of four lanes a warp (1..8), fed from the counter as k_streamlines.
template <int P, int STORE>
__global__ void __launch_bounds__(128) k_streamlines_group(const __grid_constant__ SLParams sp,
                                                           const double *__restrict__ seeds, int64_t n, int lines,
                                                           SLSample *__restrict__ out, int32_t *__restrict__ count,
                                                           int32_t *__restrict__ status) {
  const int lane = threadIdx.x & 31, l4 = lane & 3;
  if (lane >= 4 * lines) return;
  const unsigned group = 0xfu << (lane & ~3);
  for (;;) {
    unsigned long long q = 0;
    if (l4 == 0) q = atomicAdd(sp.queue, 1ull);
    q = __shfl_sync(group, q, 0, 4);
    if ((int64_t)q >= n) return;
    trace_line_group<P, STORE>(sp, seeds, (int64_t)q, out, count, status, group, l4);
  }
}

// The FP64 samples x = (double)x_hi + (double)x_lo, in place; `split` warps per line.
__global__ void __launch_bounds__(128) k_sl_widen(SLSample *__restrict__ out, const int32_t *__restrict__ count,
                                                  int64_t n, int max_samples, int split) {
  const int64_t w = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5), q = w / split;
  if (q >= n) return;
  SLSample *o = out + q * (int64_t)max_samples;
  const int c = count[q];
  for (int i = 32 * (int)(w - q * split) + (threadIdx.x & 31); i < c; i += 32 * split) {
    const float4 *p4 = reinterpret_cast<const float4 *>(o + i);
    const float4 a = p4[0], b = p4[1];
    o[i] = SLSample{(double)a.x + (double)a.y, (double)a.z + (double)a.w, (double)b.x + (double)b.y,
                    __hiloint2double(__float_as_int(b.w), __float_as_int(b.z))};
  }
}

// Eq. 7 per streamline: sum over the approximation's samples i >= 1 of
// (t_i - t_{i-1}) * |x_ref(t_i) - y_i|, x_ref linear between its samples.
__global__ void __launch_bounds__(128) k_streamline_error(const SLSample *__restrict__ ref,
                                                          const int32_t *__restrict__ rc, int rmax,
                                                          const SLSample *__restrict__ app,
                                                          const int32_t *__restrict__ ac, int amax, int64_t n,
                                                          double *__restrict__ sums) {
  // one warp per line; lane l takes the approximation's samples l+1, l+33, ...
  const int64_t q = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (q >= n) return;
  const int lane = threadIdx.x & 31;
  const SLSample *r = ref + q * (int64_t)rmax, *y = app + q * (int64_t)amax;
  const int nr = rc[q], na = ac[q];
  double acc = 0.0;
  if (nr >= 2 && na >= 2) {
    const double tlast = r[nr - 1].t;
    for (int i = 1 + lane; i < na; i += 32) {
      const SLSample p = y[i];
      if (!(p.t <= tlast)) break;   // the samples after it are later still
      // reference segment [j, j+1]: j = #{m in [1, nr-2] : t_m < t_i}, the
      // first segment that ends at or after t_i (reference times increase)
      int lo = 1, hi = nr - 1;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (r[mid].t < p.t)
          lo = mid + 1;
        else
          hi = mid;
      }
      const SLSample r0 = r[lo - 1], r1 = r[lo];
      const double dt = r1.t - r0.t;
      const double f = dt > 0.0 ? (p.t - r0.t) / dt : 0.0;
      const double ex = fma(f, r1.x - r0.x, r0.x) - p.x;
      const double ey = fma(f, r1.y - r0.y, r0.y) - p.y;
      const double ez = fma(f, r1.z - r0.z, r0.z) - p.z;
      acc = fma(p.t - y[i - 1].t, sqrt(fma(ex, ex, fma(ey, ey, ez * ez))), acc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) sums[q] = acc;
}

}  // namespace

// Lines per warp up to which a line gets four lanes: as many as a warp has
// groups of four.  250 lines of a triquadratic FP32 volume, RK4: 0.79 against
// 1.13 ms with a lane each; 10,000 lines 1.45 against 1.83 (FP16 1.43 against
// 1.76; tricubic 0.60 against 1.03).  Of a trilinear volume a group's exchange of a
// stage's point outweighs a third of its evaluation once lanes are busy: up to
// 5 lines a warp (RKF45 0.90, RK4 0.96 with 5), FP16 blocks 3 (1.02 with 4), and with
// one stage a step 2 (RK1 0.90 with 1, 1.04 to 1.25 with 3), FP16 blocks none (1.10).
template <int P, int STORE>
static int grouped_lines(int method) {
  if (P > 1) return 8;
  if (method == LRVOL_RK1) return STORE == LRVOL_STORE_F16 ? 0 : 2;
  return STORE == LRVOL_STORE_F16 ? 3 : 5;
}

template <int P, int STORE>
cudaError_t launch_sl(const SLParams &sp, const double *seeds, int64_t n, SLSample *o, int32_t *count,
                      int32_t *status, cudaStream_t s) {
  const bool trees = sp.forest.n_nodes > 0 || sp.forest.n_grid_units > 0;
  auto *single = trees ? k_streamlines<P, STORE, true, 0> : k_streamlines<P, STORE, false, 0>;
  int dev = 0, sms = 0, per_sm = 0, per_sm_group = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, single, 128, 0)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_group, k_streamlines_group<P, STORE>, 128, 0)) !=
      cudaSuccess)
    return e;
  // The triquadratic BF16 kernel with trees takes 194 registers, two CTAs an SM; held to
  // the 168 that allow three it spills, and is faster once lines are 1.5 times the two CTAs'
  // lanes (the 388,016-element flow, RK2 / RK4, 100,000 lines: 2,143 / 2,561 us, 2,713 /
  // 3,111 with two; 40,000 lines 1,419 / 1,756, 1,389 / 1,647 with two).
  if constexpr (P == 2 && STORE == LRVOL_STORE_BF16) {
    if (trees && per_sm < 3 && 2 * n > 3 * 128 * (int64_t)sms * std::max(per_sm, 1)) {
      single = k_streamlines<P, STORE, true, 3>;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, single, 128, 0)) != cudaSuccess) return e;
    }
  }
  const int64_t fit = (int64_t)sms * std::max(per_sm, 1);               // resident CTAs of 4 warps
  const int64_t fit_group = (int64_t)sms * std::max(per_sm_group, 1);
  int64_t lanes = std::min<int64_t>(std::max<int64_t>((n + 4 * fit - 1) / (4 * fit), 1), 32);   // lines per warp
  const int64_t groups = (n + 4 * fit_group - 1) / (4 * fit_group);
  if ((e = cudaMemsetAsync(sp.queue, 0, sizeof(unsigned long long), s)) != cudaSuccess) return e;
  SLParams spl = sp;
  const bool grouped = groups <= grouped_lines<P, STORE>(sp.method);
  spl.pair_out = grouped || lanes < 32;
  if (grouped) {
    const int64_t need = (n + 4 * groups - 1) / (4 * groups);
    k_streamlines_group<P, STORE><<<(unsigned)std::min(need, fit_group), 128, 0, s>>>(spl, seeds, n, (int)groups, o,
                                                                                     count, status);
  } else {
    const int64_t need = (n + 4 * lanes - 1) / (4 * lanes);
    single<<<(unsigned)std::min(need, fit), 128, 0, s>>>(spl, seeds, n, (int)lanes, o, count, status);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (spl.pair_out) {
    // warps per line: enough to fill the GPU, each with 32 samples at least
    const int64_t split = std::min<int64_t>(std::max<int64_t>(32 * (int64_t)sms / n, 1), (sp.max_samples + 31) / 32);
    k_sl_widen<<<(unsigned)((n * split + 3) / 4), 128, 0, s>>>(o, count, n, sp.max_samples, (int)split);
  }
  return cudaGetLastError();
}

cudaError_t launch_streamlines(const SLParams &sp, int degree, int storage, const double *seeds, int64_t n,
                               double *out, int32_t *count, int32_t *status, cudaStream_t s) {
  SLSample *o = reinterpret_cast<SLSample *>(out);
#define LRVOL_SL_CASE(P_, S_) return launch_sl<P_, S_>(sp, seeds, n, o, count, status, s)
  switch (degree * 3 + storage) {
    case 3: LRVOL_SL_CASE(1, LRVOL_STORE_F32); break;
    case 4: LRVOL_SL_CASE(1, LRVOL_STORE_F16); break;
    case 5: LRVOL_SL_CASE(1, LRVOL_STORE_BF16); break;
    case 6: LRVOL_SL_CASE(2, LRVOL_STORE_F32); break;
    case 7: LRVOL_SL_CASE(2, LRVOL_STORE_F16); break;
    case 8: LRVOL_SL_CASE(2, LRVOL_STORE_BF16); break;
    case 9: LRVOL_SL_CASE(3, LRVOL_STORE_F32); break;
    case 10: LRVOL_SL_CASE(3, LRVOL_STORE_F16); break;
    case 11: LRVOL_SL_CASE(3, LRVOL_STORE_BF16); break;
    default: return cudaErrorInvalidValue;
  }
#undef LRVOL_SL_CASE
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Streamline tubes (Sec. 5.3): capsules around the polyline segments,
// visibility by a 64-bit atomic minimum of (t bits, segment index) per pixel,
// then one thread per pixel shades the winner.
// ----------------------------------------------------------------------------
namespace {

__device__ __forceinline__ float dot3r(float x0, float x1, float x2, float y0, float y1, float y2) {
  return __fadd_rn(__fadd_rn(__fmul_rn(x0, y0), __fmul_rn(x1, y1)), __fmul_rn(x2, y2));
}

// What the ray/capsule test needs of a segment and the ray's origin: computed
// once per segment when all rays start at the eye.
struct Capsule {
  float ba[3], baba;   // b - a and its square
  float oa[3], baoa;   // origin - a, and its product with b - a
  float ob[3], C;      // origin - b; baba |oa|^2 - baoa^2 - r^2 baba
  float ca, cb;        // |oa|^2 - r^2, |ob|^2 - r^2
  __device__ __forceinline__ void set(const float *o, const float *a, const float *b, float r) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ba[c] = __fsub_rn(b[c], a[c]);
      oa[c] = __fsub_rn(o[c], a[c]);
      ob[c] = __fsub_rn(o[c], b[c]);
    }
    const float rr = __fmul_rn(r, r), oaoa = dot3r(oa[0], oa[1], oa[2], oa[0], oa[1], oa[2]);
    baba = dot3r(ba[0], ba[1], ba[2], ba[0], ba[1], ba[2]);
    baoa = dot3r(ba[0], ba[1], ba[2], oa[0], oa[1], oa[2]);
    C = __fsub_rn(__fsub_rn(__fmul_rn(baba, oaoa), __fmul_rn(baoa, baoa)), __fmul_rn(rr, baba));
    ca = __fsub_rn(oaoa, rr);
    cb = __fsub_rn(dot3r(ob[0], ob[1], ob[2], ob[0], ob[1], ob[2]), rr);
  }
};

// Ray/capsule hit in FP32 with the oracle's order of operations; t > 0 only.
__device__ __forceinline__ bool capsule_hit(const Capsule &S, float d0, float d1, float d2, float &t) {
  const float bard = dot3r(S.ba[0], S.ba[1], S.ba[2], d0, d1, d2), rdoa = dot3r(d0, d1, d2, S.oa[0], S.oa[1], S.oa[2]);
  const float A = __fsub_rn(S.baba, __fmul_rn(bard, bard));
  if (A > 0.f) {
    const float B = __fsub_rn(__fmul_rn(S.baba, rdoa), __fmul_rn(S.baoa, bard));
    const float H = __fsub_rn(__fmul_rn(B, B), __fmul_rn(A, S.C));
    if (H >= 0.f) {
      const float tb = __fdiv_rn(__fsub_rn(-B, __fsqrt_rn(H)), A);
      const float y = __fadd_rn(S.baoa, __fmul_rn(tb, bard));
      if (y > 0.f && y < S.baba) {
        t = tb;
        return tb > 0.f;
      }
    }
  }
  float best = __int_as_float(0x7f800000);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float bb = k == 0 ? rdoa : dot3r(d0, d1, d2, S.ob[0], S.ob[1], S.ob[2]);
    const float h = __fsub_rn(__fmul_rn(bb, bb), k == 0 ? S.ca : S.cb);
    if (h > 0.f) {
      const float tc = __fsub_rn(-bb, __fsqrt_rn(h));
      if (tc > 0.f && tc < best) best = tc;
    }
  }
  t = best;
  return best < __int_as_float(0x7f800000);
}

__device__ __forceinline__ bool tube_segment(const TubeParams &tp, int64_t s, float *a, float *b) {
  const unsigned per = (unsigned)(tp.max_samples - 1), j = (unsigned)s / per, k = (unsigned)s - j * per;   // s < 2^32
  if ((int)k >= tp.count[j] - 1) return false;
  const double *p = tp.samples + ((int64_t)j * tp.max_samples + k) * 4;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    a[c] = __double2float_rn(p[c]);
    b[c] = __double2float_rn(p[4 + c]);
  }
  return true;
}

// No hit anywhere, and with a ray table (rays not null) each pixel's direction in
// the pixel's place of the image (until the resolve overwrites it).
__global__ void __launch_bounds__(256) k_tube_init(const RayConsts K, int width, int height,
                                                   unsigned long long *__restrict__ vis, float4 *__restrict__ rays) {
  const int i = blockIdx.x * 64 + (threadIdx.x & 63), j = blockIdx.y * 4 + (threadIdx.x >> 6);
  if (i >= width || j >= height) return;
  const int64_t q = (int64_t)j * width + i;
  vis[q] = ~0ull;
  if (rays) {
    Ray ray;
    make_ray(K, i, j, ray);
    rays[q] = make_float4(ray.d[0], ray.d[1], ray.d[2], 0.f);
  }
}

__device__ __forceinline__ void tube_dir(const TubeParams &tp, int i, int j, Ray &ray) {
  if (tp.ray_table) {   // perspective: every ray starts at the eye
    const float4 d = reinterpret_cast<const float4 *>(tp.out)[(int64_t)j * tp.width + i];
    ray.d[0] = d.x;
    ray.d[1] = d.y;
    ray.d[2] = d.z;
#pragma unroll
    for (int c = 0; c < 3; ++c) ray.o[c] = tp.ray.E[c];
  } else {
    make_ray(tp.ray, i, j, ray);
  }
}

// A segment that has pairs.  80 bytes, moved 16 at a time: eight lanes' accesses
// to eight slots touch every bank once.
struct __align__(16) TubeSlot {
  Capsule cap;          // perspective; otherwise the end points in cap.ba and cap.ob
  float inv_bw;
  unsigned sid, first;  // segment id, first pair
  int bw, i0, j0;
  __device__ __forceinline__ void put(TubeSlot *to) const {
#pragma unroll
    for (int q = 0; q < 5; ++q) reinterpret_cast<float4 *>(to)[q] = reinterpret_cast<const float4 *>(this)[q];
  }
  __device__ __forceinline__ void get(const TubeSlot *from) {
#pragma unroll
    for (int q = 0; q < 5; ++q) reinterpret_cast<float4 *>(this)[q] = reinterpret_cast<const float4 *>(from)[q];
  }
};
static_assert(sizeof(TubeSlot) == 80, "five 16-byte accesses");

__device__ __forceinline__ void tube_group(const TubeParams &tp, int64_t line, int k0, int nseg, int split, int part,
                                           int lane, TubeSlot *sl);

// A line's segments go in groups of 32: lane l bounds segment l of the group on
// the screen, then the warp walks the group's (segment, pixel) pairs 32 at a
// time, as the trimming raster does.  `strides` warps take a line's groups in
// turn, and `split` warps share each group's pairs, when few long segments
// could cover much of the image.
// Bound by instructions: a segment's share of the test is computed once and
// read from shared memory, a pixel's ray from the table.  4,096 lines of 63
// segments at 1920x1080, in all: 263 us; 335 with both computed for every pair.
constexpr int kTubeWarps = 1;   // an SM takes the next warp when one ends: 4096 lines 263 us, 276 in CTAs of 2 or 4 warps

__global__ void __launch_bounds__(32 * kTubeWarps) k_tube_raster(const __grid_constant__ TubeParams tp, int strides,
                                                                 int split) {
  __shared__ TubeSlot slots[kTubeWarps][32];
  const int lane = threadIdx.x & 31;
  const int64_t wid = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kTubeWarps + (threadIdx.x >> 5);
  const int64_t at = wid / split, line = at / strides;
  const int part = (int)(wid - at * split);
  if (line >= tp.n_lines) return;                      // whole warp
  const int nseg = tp.count[line] - 1;
  for (int k0 = 32 * (int)(at - line * strides); k0 < nseg; k0 += 32 * strides) tube_group(tp, line, k0, nseg, split, part, lane, slots[threadIdx.x >> 5]);
}

// One group of 32 segment slots of a line (see k_tube_raster).
__device__ __forceinline__ void tube_group(const TubeParams &tp, int64_t line, int k0, int nseg, int split, int part,
                                           int lane, TubeSlot *sl) {
  const int per = tp.max_samples - 1;                  // segment slots per line
  const RayConsts &K = tp.ray;
  float a[3] = {0.f, 0.f, 0.f}, b[3] = {0.f, 0.f, 0.f};
  int i0 = 0, j0 = 0, bw = 1, cnt = 0;
  if (k0 + lane < nseg && tube_segment(tp, line * per + k0 + lane, a, b)) {
    // conservative pixel box of the capsule's bounding box
    float amin = __int_as_float(0x7f800000), amax = -amin, bmin = amin, bmax = -amin;
    bool full = false;
    int behind = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float cx = ((q & 1) ? fmaxf(a[0], b[0]) + tp.radius : fminf(a[0], b[0]) - tp.radius) - K.E[0];
      const float cy = ((q & 2) ? fmaxf(a[1], b[1]) + tp.radius : fminf(a[1], b[1]) - tp.radius) - K.E[1];
      const float cz = ((q & 4) ? fmaxf(a[2], b[2]) + tp.radius : fminf(a[2], b[2]) - tp.radius) - K.E[2];
      const float r = cx * K.R[0] + cy * K.R[1] + cz * K.R[2];
      const float u = cx * K.U[0] + cy * K.U[1] + cz * K.U[2];
      float x = r, y = u;
      if (K.persp) {
        const float z = cx * K.F[0] + cy * K.F[1] + cz * K.F[2];
        if (!(z > 1e-6f)) {
          full = true;
          ++behind;
          continue;
        }
        const float iz = rcp_approx(z);
        x = r * iz;
        y = u * iz;
      }
      amin = fminf(amin, x);
      amax = fmaxf(amax, x);
      bmin = fminf(bmin, y);
      bmax = fmaxf(bmax, y);
    }
    int i1 = tp.width - 1, j1 = tp.height - 1;
    if (behind < 8 && (full || pixel_box(PixelScale(K), tp.width, tp.height, amin, amax, bmin, bmax, i0, i1, j0, j1))) {
      if (full) {
        i0 = 0;
        j0 = 0;
        i1 = tp.width - 1;
        j1 = tp.height - 1;
      }
      bw = i1 - i0 + 1;
      cnt = bw * (j1 - j0 + 1);   // <= 32768^2 < 2^31
    }
  }
  PairWalk walk(lane, cnt, split, part);
  if (walk.has) {
    TubeSlot m;
    if (K.persp) {
      m.cap.set(K.E, a, b, tp.radius);
    } else {
      m.cap = Capsule{};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        m.cap.ba[c] = a[c];
        m.cap.ob[c] = b[c];
      }
    }
    m.inv_bw = 1.f / (float)bw;
    m.sid = (uint32_t)(line * per + k0 + lane);
    m.first = walk.first;
    m.bw = bw;
    m.i0 = i0;
    m.j0 = j0;
    m.put(sl + walk.slot);
  }
  __syncwarp();
  for (long long base = walk.w0; base < walk.w1; base += 32) {
    TubeSlot m;
    m.get(sl + walk.next(lane));
    if (base + lane >= walk.w1) continue;
    const unsigned pix = (unsigned)(base + lane) - m.first, row = box_row(pix, (unsigned)m.bw, m.inv_bw);
    const int i = m.i0 + (int)(pix - row * (unsigned)m.bw), j = m.j0 + (int)row;
    Ray ray;
    tube_dir(tp, i, j, ray);
    float t;
    bool hit;
    if (K.persp) {
      hit = capsule_hit(m.cap, ray.d[0], ray.d[1], ray.d[2], t);
    } else {
      Capsule cap;
      cap.set(ray.o, m.cap.ba, m.cap.ob, tp.radius);
      hit = capsule_hit(cap, ray.d[0], ray.d[1], ray.d[2], t);
    }
    if (!hit) continue;
    const unsigned long long key = ((unsigned long long)__float_as_uint(t) << 32) | (unsigned long long)m.sid;
    atomicMin(tp.vis + (int64_t)j * tp.width + i, key);
  }
  __syncwarp();   // the next group overwrites the slots
}

template <int P, int STORE>
__global__ void __launch_bounds__(128) k_tube_resolve(const __grid_constant__ TubeParams tp) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (int64_t)tp.width * tp.height) return;
  float4 *o = reinterpret_cast<float4 *>(tp.out) + q;
  const unsigned long long key = tp.vis[q];
  if (key == ~0ull) {
    *o = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const int64_t s = (int64_t)(key & 0xffffffffull);
  const float t = __uint_as_float((unsigned)(key >> 32));
  float a[3], b[3];
  tube_segment(tp, s, a, b);
  Ray ray;
  tube_dir(tp, (int)((unsigned)q % (unsigned)tp.width), (int)((unsigned)q / (unsigned)tp.width), ray);   // q < 2^30
  float p[3], ba[3], pa[3], qa[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p[c] = __fadd_rn(ray.o[c], __fmul_rn(t, ray.d[c]));
    ba[c] = __fsub_rn(b[c], a[c]);
    pa[c] = __fsub_rn(p[c], a[c]);
  }
  const float baba = dot3r(ba[0], ba[1], ba[2], ba[0], ba[1], ba[2]);
  float hcl = baba > 0.f ? __fdiv_rn(dot3r(pa[0], pa[1], pa[2], ba[0], ba[1], ba[2]), baba) : 0.f;
  hcl = fminf(fmaxf(hcl, 0.f), 1.f);
#pragma unroll
  for (int c = 0; c < 3; ++c) qa[c] = __fadd_rn(a[c], __fmul_rn(hcl, ba[c]));
  SLField<P, STORE, true> F;
  F.cur = kNone;
  float v0 = 0.f, v1 = 0.f, v2 = 0.f;
  F.eval(tp.field, qa[0], qa[1], qa[2], v0, v1, v2);
  const float speed = sqrtf(fmaf(v0, v0, fmaf(v1, v1, v2 * v2)));
  const float x = fminf(fmaxf(fmaf(speed, tp.tf_scale, tp.tf_bias), 0.f), 255.f);
  const int k = min((int)x, 254);
  const float fr = x - (float)k;
  const float4 e0 = tp.cmap[k], e1 = tp.cmap[k + 1];
  const float n0 = p[0] - qa[0], n1 = p[1] - qa[1], n2 = p[2] - qa[2];
  const float nn = fmaf(n0, n0, fmaf(n1, n1, n2 * n2));
  float I = nn > 0.f ? fabsf(fmaf(n0, ray.d[0], fmaf(n1, ray.d[1], n2 * ray.d[2]))) * rsqrtf(nn) : 1.f;
  I = fmaxf(I, 0.4f);
  *o = make_float4(I * fmaf(fr, e1.x - e0.x, e0.x), I * fmaf(fr, e1.y - e0.y, e0.y), I * fmaf(fr, e1.z - e0.z, e0.z),
                   1.f);
}

}  // namespace

// A perspective ray costs a rounded square root and three rounded quotients for
// each of its pairs; with at least a segment to 64 pixels they are computed once
// per pixel instead (4,096 lines of 199 segments at 1920x1080: 0.73 against 0.82
// ms; 40 lines of 99, a segment to 520 pixels: 101 against 97 us).
constexpr int64_t kTubeTablePixels = 64;

cudaError_t launch_tubes(TubeParams tp, int degree, int storage, cudaStream_t s) {
  const int64_t npix = (int64_t)tp.width * tp.height;
  const int64_t nseg = tp.n_lines * (int64_t)(tp.max_samples - 1);
  tp.ray_table = tp.ray.persp && nseg >= npix / kTubeTablePixels;
  k_tube_init<<<dim3((unsigned)((tp.width + 63) / 64), (unsigned)((tp.height + 3) / 4)), 256, 0, s>>>(
      tp.ray, tp.width, tp.height, tp.vis, tp.ray_table ? reinterpret_cast<float4 *>(tp.out) : nullptr);
  if (nseg > 0) {
    // warps per line: its groups spread over warps while there are fewer than
    // 64 warps per SM, and about 512 pairs per warp and group when the lines'
    // first groups cover the image twice, at most 256 in all
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t lines = tp.n_lines, groups = (tp.max_samples - 1 + 31) / 32;
    int64_t split = (2 * npix + lines * 512 - 1) / (lines * 512);
    split = std::min<int64_t>(std::max<int64_t>(split, 1), 256);
    const int64_t strides = std::min<int64_t>(std::max<int64_t>(64 * (int64_t)sms / lines, 1), std::min<int64_t>(groups, 256));
    split = (split + strides - 1) / strides;
    // up to 2^32 lines: in rows of CTAs past what one row holds
    const int64_t ctas = (lines * strides * split + kTubeWarps - 1) / kTubeWarps, row = std::min(ctas, (int64_t)1 << 30);
    const dim3 grid((unsigned)row, (unsigned)((ctas + row - 1) / row));
    k_tube_raster<<<grid, 32 * kTubeWarps, 0, s>>>(tp, (int)strides, (int)split);
  }
  const unsigned blocks = (unsigned)((npix + 127) / 128);
#define LRVOL_TUBE_CASE(P_, S_) k_tube_resolve<P_, S_><<<blocks, 128, 0, s>>>(tp)
  switch (degree * 3 + storage) {
    case 3: LRVOL_TUBE_CASE(1, LRVOL_STORE_F32); break;
    case 4: LRVOL_TUBE_CASE(1, LRVOL_STORE_F16); break;
    case 5: LRVOL_TUBE_CASE(1, LRVOL_STORE_BF16); break;
    case 6: LRVOL_TUBE_CASE(2, LRVOL_STORE_F32); break;
    case 7: LRVOL_TUBE_CASE(2, LRVOL_STORE_F16); break;
    case 8: LRVOL_TUBE_CASE(2, LRVOL_STORE_BF16); break;
    case 9: LRVOL_TUBE_CASE(3, LRVOL_STORE_F32); break;
    case 10: LRVOL_TUBE_CASE(3, LRVOL_STORE_F16); break;
    case 11: LRVOL_TUBE_CASE(3, LRVOL_STORE_BF16); break;
    default: return cudaErrorInvalidValue;
  }
#undef LRVOL_TUBE_CASE
  return cudaGetLastError();
}

cudaError_t launch_streamline_error(const double *ref, const int32_t *rc, int rmax, const double *app,
                                    const int32_t *ac, int amax, int64_t n, double *sums, cudaStream_t s) {
  k_streamline_error<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(reinterpret_cast<const SLSample *>(ref), rc, rmax,
                                                             reinterpret_cast<const SLSample *>(app), ac, amax, n,
                                                             sums);
  return cudaGetLastError();
}

}  // namespace lrvol
