// liblrvol render kernel for sm_103a (Sec. 4, Alg. 2, Eq. 4), compiled once per
// block storage (render_f32.cu, render_f16.cu, render_bf16.cu).
//
//   k_render<P, FIELD, STORE, FIXED, TREES, PAIR, TRACE>
//       per-pixel ray casting with element reuse, Eq. 4 (or fixed, or learned)
//       steps, transfer function and Alg. 2 compositing, and gradient shading
//       (Sec. 4.1).  TRACE = false is the product kernel; TRACE = true is the
//       same template over a pixel list, writing every sample it composites.
#pragma once

#include "device_common.cuh"

static_assert(LRVOL_BAND_ROWS == 8, "a CTA renders 8 rows: one interleaved band");

namespace lrvol {
namespace {

// One CTA of 4 warps renders a 16x8-pixel tile, so the warps sharing an SM's
// L1 march through neighbouring elements; one lane traces one ray.  A warp
// covers an 8x4 patch for scalar fields and a 4x8 patch for 3-vector fields
// (the shapes that measured fastest for each).  The element-change branch
// (look-up and block loads) is kept minimal: a warp runs it whenever any of its
// lanes changes element, which happens almost every iteration.
//
// In the sample loop the Alg. 2 update of sample k comes after the position of
// sample k+1 and, where no block of the forest holds a tree, after the load of
// its head word: the two are independent, so their latencies overlap.  A ray
// that terminates after sample k discards the sample k+1 evaluated with it.
// Sample "-1" is a transfer-function entry of zeros, so the loop has one path.
//
// With PAIR a pass of the loop also evaluates the ray's next sample and keeps it
// where it lies in the box of the pass' element: the wait for an element's loads,
// and their way through L1, then comes once for two samples.  The samples, their
// order and their arithmetic are those of one a pass.
//
// A warp's iteration waits about as long for its instructions as for the loads
// of an element change, so both the sample's and the change's instructions
// count: the position's clamps fused into its multiply-add (.sat), no branch
// besides the element change, block sizes and step rule known to the compiler, a head
// table that needs no clamped index, and without trees (TREES false) no box test.
// 1920x1080 frames of a 174,000-element tricubic volume, Eq. 4 steps, with
// FP32 / BF16 / FP16 blocks: 3.05 / 2.98 / 2.45 ms before these, 2.75 / 2.49 /
// 2.10 with them, 2.60 / 2.34 / 2.08 with two samples a pass as well; FP32
// gradient-shaded 4.51 -> 3.92; learned FP16 at 3840x2160 4.27 -> 3.76; 3-vector
// speed of 388,016 triquadratic elements in a forest with trees, FP32 / FP16:
// 0.93 / 0.79 -> 0.77 / 0.67 (grids for subtrees among it).
//
// TRACE (a compile-time flag; false in every product launch, where the trace
// code compiles out) runs the same march for a list of pixels, one thread per
// listed pixel, and also writes each sample's (t, element id, field value,
// segment length), the composited sample count and the pixel's RGBA.  It is
// the parity hook that compares a kernel's own samples with the oracle.  It takes
// one sample a pass: the kernels that take two are held to its pixels and counts,
// bit for bit, and to those of the untraced kernels that take one.
//
// FIELD 3 renders a scalar volume with gradient shading (Sec. 4.1): each
// sample also evaluates the block's gradient, and C_src is scaled by
// I = max(0.4, |l . g| / max(|g|, eps)).
// CTAs per SM the register budget allows: the tricubic FP32/BF16 block takes
// 64 registers a lane (4 CTAs of 128 threads), 16-bit pairs of an FP16 block
// 32 (5 CTAs); the triquadratic 3-vector FP16 block (42 registers instead of
// 83) also fits 5.  The shaded tricubic kernel keeps the gradient's partial
// sums too: at 4 CTAs it spills (16 bytes without trees, up to 40 with them)
// and still beats 3 CTAs without spills by 5 % (measured); forcing 5 CTAs on the FP32 kernels spills
// inside the sample loop and costs 37-51 %.
template <int P, int FIELD, int STORE>
constexpr int render_min_ctas() {
  if (STORE == LRVOL_STORE_F16) {
    if (P == 3 && FIELD == 0) return 5;
    if (P == 2 && (FIELD == 1 || FIELD == 2)) return 5;
  }
  return 4;
}

template <int P, int FIELD, int STORE, bool FIXED, bool TREES, bool PAIR, bool TRACE>
__global__ void __launch_bounds__(128, (render_min_ctas<P, FIELD, STORE>())) k_render(const __grid_constant__ RenderParams prm) {
  static_assert(!(PAIR && TRACE), "the traced march takes one sample a pass");
  constexpr int N = P + 1;
  constexpr bool SHADE = FIELD == 3;
  // packed colours pay where the blocks are FP32 (1080p Eq. 4 frame 2.81 -> 2.75
  // ms); beside 16-bit blocks or shading they cost up to 1.3 %
  constexpr bool PACKED = STORE == LRVOL_STORE_F32 && !SHADE;
  constexpr int BF = SHADE ? 0 : FIELD;
  __shared__ float4 tfb[kTfEntries], tfd[kTfEntries];
  load_tf(prm, tfb, tfd);
  __syncthreads();

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int i, j;
  bool active;
  int64_t g = 0;               // TRACE: position in the pixel list
  uint32_t cur_e = kNone;      // TRACE: element of the current sample
  if constexpr (TRACE) {
    g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    active = g < prm.trace_n;
    i = active ? __ldg(prm.trace_pix + 2 * g) : 0;
    j = active ? __ldg(prm.trace_pix + 2 * g + 1) : 0;
    if (active && (i < 0 || i >= prm.width || j < 0 || j >= prm.height)) {
      set_status(prm.status, kStatusBounds);
      prm.trace_count[g] = 0;
      prm.trace_rgba[g] = make_float4(0.f, 0.f, 0.f, 0.f);
      active = false;
    }
  } else {
    if constexpr (BF == 1 || BF == 2) {   // 3-vector fields: four 4x8 patches side by side
      i = blockIdx.x * 16 + warp * 4 + (lane & 3);
      j = prm.row_begin + (blockIdx.y * prm.band_count + prm.band_index) * 8 + (lane >> 2);
    } else {                              // scalar fields: 2x2 patches of 8x4
      i = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7);
      j = prm.row_begin + (blockIdx.y * prm.band_count + prm.band_index) * 8 + (warp >> 1) * 4 + (lane >> 3);
    }
    active = i < prm.width && j < prm.row_end;
  }
  unsigned nsamp = 0, nlook = 0, nhit = 0;

  Ray ray;
  if (active) {
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, Tr = 1.f;
    if (make_ray(prm.ray, i, j, ray) &&
        (prm.trim == nullptr || trim_cut(__ldg(prm.trim + (int64_t)j * prm.width + i), ray.tin, ray.tout))) {
      ++nhit;
      const float tr_stop = 1.f - prm.alpha_stop;
      float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra, rc = ra, rd = ra;
      float dsv = 0.f;       // step inside the current element (Eq. 4, or Eq. 4 x learned multiplier)
      Block<P, BF, STORE> blk;
      float t = ray.tin + 0.f;   // not -0
      float kf = 0.f;        // FIXED: k + 1 (exact up to kMaxSamplesPerRay)
      int k = 0;             // samples evaluated; the last pass' are not yet composited
      int pending = 0;       // how many those are
      // their TF coordinates, segments, shading; kTfNothing: a sample of no opacity
      float pcoord = kTfNothing, pseg = 0.f, psh = 1.f;
      float qcoord = kTfNothing, qseg = 0.f, qsh = 1.f;
      float lx = 0.f, ly = 0.f, lz = 0.f;   // towards the light (shading)
      if constexpr (SHADE) {
        lx = prm.light_set ? prm.light[0] : -ray.d[0];
        ly = prm.light_set ? prm.light[1] : -ray.d[1];
        lz = prm.light_set ? prm.light[2] : -ray.d[2];
      }
      uint32_t word = kNone;  // !TREES: head word of the current element
      bool stopped = false;  // opaque: sample k is not composited
      do {
        const float px = fma_sat(t, ray.d[0], ray.o[0]);
        const float py = fma_sat(t, ray.d[1], ray.o[1]);
        const float pz = fma_sat(t, ray.d[2], ray.o[2]);
        // without trees the head word names the element, so a new word is the
        // test of having left the box; its load is under way while sample k - 1
        // is composited
        uint32_t head = 0;
        bool changed = false;
        if constexpr (TREES)
          changed = !(px >= ra.x && py >= ra.y && pz >= ra.z && px < rb.x && py < rb.y && pz < rb.z);
        else
          head = forest_head(prm.forest, px, py, pz);
        composite<SHADE, PACKED>(tfb, tfd, pcoord, pseg, psh, prm, C0, C1, C2, Tr);
        stopped = Tr <= tr_stop && k > 0;
        bool first = false;   // stopped at the first of two
        if constexpr (PAIR) {
          first = stopped && pending == 2;
          composite<SHADE, PACKED>(tfb, tfd, first ? kTfNothing : qcoord, qseg, qsh, prm, C0, C1, C2, Tr);
          stopped = Tr <= tr_stop && k > 0;
          k -= first;
        }
        if constexpr (!TREES) changed = head != word;
        if (changed) {
          uint32_t cur;
          if constexpr (TREES) {
            cur = forest_lookup(prm.forest, px, py, pz, prm.status);
          } else {
            cur = head & ~kLeaf;
            word = head;
          }
          if (cur >= (uint32_t)prm.n_elem) {   // kNone included: the ray ends, its pixel means nothing
            set_status(prm.status, kStatusBounds);
            ray.tout = 0.f;
            cur = 0;
          }
          nlook += !first;
          if constexpr (TRACE) cur_e = cur;
          load_record(prm.elem + cur, ra, rb, rc, rd);
          if constexpr (!FIXED)
            dsv = prm.mode == LRVOL_STEP_LEARNED ? __fmul_rn(ra.w, __ldg(prm.mult + cur)) : ra.w;
          if constexpr (BF == 2)
            blk.load(prm.bezc + (int64_t)cur * blk.BYTES, prm.comp);
          else
            blk.load(prm.bez + (int64_t)cur * blk.BYTES, 0);
        }
        // the next float where a step does not advance (t >= 0, so its bits order like it)
        auto advance = [&](float from, float steps) -> float {
          const float to = FIXED ? __fmaf_rn(steps, prm.h, ray.tin) : __fadd_rn(from, dsv);
          return to > from ? to : __int_as_float(__float_as_int(from) + 1);
        };
        auto evaluate = [&](float x, float y, float z, float &sh) -> float {
          float bx[N], by[N], bz[N];
          const float ux = local_u(x, ra.x, rc.x, rd.x);
          const float uy = local_u(y, ra.y, rc.y, rd.y);
          const float uz = local_u(z, ra.z, rc.z, rd.z);
          monomials<P>(ux, bx);
          monomials<P>(uy, by);
          monomials<P>(uz, bz);
          sh = 1.f;
          if constexpr (SHADE) {
            float dx[N], dy[N], dz[N], gu, gv, gw;
            dmonomials<P>(ux, dx);
            dmonomials<P>(uy, dy);
            dmonomials<P>(uz, dz);
            const float v = blk.eval_grad(bx, by, bz, dx, dy, dz, gu, gv, gw);
            const float gx = gu * rd.x, gy = gv * rd.y, gz = gw * rd.z;   // world gradient: d/dx = iw d/du
            const float gl = fmaf(gx, lx, fmaf(gy, ly, gz * lz));
            const float gn = fmaxf(sqrtf(fmaf(gx, gx, fmaf(gy, gy, gz * gz))), prm.grad_eps);
            sh = fmaxf(0.4f, fabsf(gl) / gn);
            return v;
          } else {
            return blk.eval(bx, by, bz);
          }
        };
        float tn = advance(t, kf + 1.f);
        const float te = fminf(tn, ray.tout);
        pseg = __fsub_rn(te, t);
        const float v = evaluate(px, py, pz, psh);
        if constexpr (TRACE) {
          if (k < prm.trace_max) prm.trace_rec[g * prm.trace_max + k] = make_float4(t, __uint_as_float(cur_e), v, pseg);
        }
        pcoord = tf_coord(prm, v);
        bool two = false;
        if constexpr (PAIR) {
          const float qx = fma_sat(tn, ray.d[0], ray.o[0]);
          const float qy = fma_sat(tn, ray.d[1], ray.o[1]);
          const float qz = fma_sat(tn, ray.d[2], ray.o[2]);
          two = qx >= ra.x && qy >= ra.y && qz >= ra.z && qx < rb.x && qy < rb.y && qz < rb.z && tn < ray.tout &&
                k + 2 < kMaxSamplesPerRay;
          const float t2 = advance(tn, kf + 2.f);
          qseg = __fsub_rn(fminf(t2, ray.tout), te);   // finite also where the sample is dropped
          const float v2 = evaluate(qx, qy, qz, qsh);
          qcoord = two ? tf_coord(prm, v2) : kTfNothing;
          tn = two ? t2 : tn;
        }
        pending = two ? 2 : 1;
        if constexpr (FIXED) kf += two ? 2.f : 1.f;
        t = tn;
        k += pending;
      } while (!stopped && t < ray.tout && k < kMaxSamplesPerRay);
      if (stopped || k >= kMaxSamplesPerRay) {
        if (!stopped) set_status(prm.status, kStatusTimeout);
        nsamp = k - pending;
      } else {
        composite<SHADE, PACKED>(tfb, tfd, pcoord, pseg, psh, prm, C0, C1, C2, Tr);
        if constexpr (PAIR) {
          if (pending == 2) {
            if (Tr <= tr_stop)
              --k;
            else
              composite<SHADE, PACKED>(tfb, tfd, qcoord, qseg, qsh, prm, C0, C1, C2, Tr);
          }
        }
        nsamp = k;
      }
    }
    if constexpr (TRACE) {
      prm.trace_rgba[g] = make_float4(C0, C1, C2, 1.f - Tr);
      prm.trace_count[g] = (int32_t)nsamp;
    } else {
      reinterpret_cast<float4 *>(prm.out)[(int64_t)j * prm.width + i] = make_float4(C0, C1, C2, 1.f - Tr);
    }
  }
  // per-warp counters
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    nsamp += __shfl_down_sync(0xffffffffu, nsamp, o);
    nlook += __shfl_down_sync(0xffffffffu, nlook, o);
    nhit += __shfl_down_sync(0xffffffffu, nhit, o);
  }
  if (lane == 0) {
    atomicAdd(prm.counters + kCntSamples, (unsigned long long)nsamp);
    atomicAdd(prm.counters + kCntLookups, (unsigned long long)nlook);
    atomicAdd(prm.counters + kCntRays, (unsigned long long)nhit);
  }
}

// This call's 8-row bands: band_index, band_index + band_count, ...
inline dim3 render_grid(const RenderParams &prm) {
  const int n_bands = (prm.row_end - prm.row_begin + 7) / 8;
  const int mine = (n_bands - prm.band_index + prm.band_count - 1) / prm.band_count;
  return dim3((unsigned)((prm.width + 15) / 16), (unsigned)mine);
}

template <int P, int FIELD, int STORE, bool FIXED, bool TREES, bool PAIR, bool TRACE>
cudaError_t launch_render_f(const RenderParams &prm, cudaStream_t s) {
  if constexpr (TRACE) {
    k_render<P, FIELD, STORE, FIXED, TREES, PAIR, true><<<(unsigned)((prm.trace_n + 127) / 128), 128, 0, s>>>(prm);
  } else {
    const dim3 grid = render_grid(prm);
    k_render<P, FIELD, STORE, FIXED, TREES, PAIR, false><<<grid, 128, 0, s>>>(prm);
  }
  return cudaGetLastError();
}

// Two samples a pass (PAIR) or one.  Two cost their instructions also where the
// second lies in another element, one waits for an element's loads once a sample.
// Two / one a pass, time of the frame (a 174,000-element volume with scalar and
// 3-vector blocks of degree 3, the 388,016-element flow of degree 2, and two small
// volumes of degree 3 and 2 behind the comma; FP32, FP16 and BF16 blocks):
//   Eq. 4, tricubic scalar      0.89..0.95 at 256x256, 0.95..1.00 at 960x540, 0.94..0.98
//                               at 1080p, 0.91..1.04: always two
//   other frames                one above 12 CTAs an SM (640x360): 1.04 (learned scalar),
//                               1.06 (FP16 speed) at 1080p
//   learned                     0.82..0.92 at 256x256, 0.78..0.94 at 640x360: two
//   Eq. 4, 3-vectors            0.81..1.01 and 0.84..1.05, 0.85..1.06: two, but the speed of a
//                               degree-2 volume that caches hold 1.03..1.12: one
//   fixed, scalar or component  0.91..1.06 at 256x256; 0.96..1.16 at 640x360, BF16
//                               0.89..1.03: two up to 4 CTAs an SM, BF16 12
//   fixed, speed                0.99..1.14 at 256x256: one, but tricubic BF16 0.90..0.99
// Never: shaded frames (1.03 at 256x256, 1.11 at 1080p), and scalar volumes of degree 2
// and 1, whose elements hold fewer samples and load less (0.95..1.06).
constexpr int64_t kPairBytes = (int64_t)16 << 20;

template <int P, int FIELD, int STORE, bool FIXED>
constexpr bool pairs_exist() {
  if (FIXED && FIELD == 1) return P == 3 && STORE == LRVOL_STORE_BF16;
  return (P == 3 || (P == 2 && FIELD != 0)) && FIELD != 3;
}

template <int P, int FIELD, int STORE, bool FIXED>
bool take_pairs(const RenderParams &prm, int64_t ctas, int sms) {
  if (P == 3 && FIELD == 0 && prm.mode == LRVOL_STEP_HEURISTIC) return true;
  if (ctas > (FIXED && STORE != LRVOL_STORE_BF16 ? 4 : 12) * (int64_t)sms) return false;
  return !(P == 2 && FIELD == 1 && prm.mode == LRVOL_STEP_HEURISTIC && prm.n_elem * Block<P, FIELD, STORE>::BYTES < kPairBytes);
}

template <int P, int FIELD, int STORE, bool FIXED, bool TREES, bool TRACE>
cudaError_t launch_render_p(const RenderParams &prm, cudaStream_t s) {
  if constexpr (pairs_exist<P, FIELD, STORE, FIXED>() && !TRACE) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const dim3 grid = render_grid(prm);
    if (take_pairs<P, FIELD, STORE, FIXED>(prm, (int64_t)grid.x * grid.y, sms))
      return launch_render_f<P, FIELD, STORE, FIXED, TREES, true, TRACE>(prm, s);
  }
  return launch_render_f<P, FIELD, STORE, FIXED, TREES, false, TRACE>(prm, s);
}

// Fixed steps, and forests without a tree, have kernels of their own: which step
// rule a frame takes is the same for every sample, and a test of it costs a
// sample two instructions and the registers of both rules; without trees the
// box test goes (1080p Eq. 4 frame of a tricubic FP32 volume: 2.95 -> 2.85 ms, and
// 2.81 with the composite under the head load).
template <int P, int FIELD, int STORE, bool TRACE>
cudaError_t launch_render_t(const RenderParams &prm, cudaStream_t s) {
  const bool trees = prm.forest.n_nodes > 0 || prm.forest.n_grid_units > 0;
  if (prm.mode == LRVOL_STEP_FIXED)
    return trees ? launch_render_p<P, FIELD, STORE, true, true, TRACE>(prm, s)
                 : launch_render_p<P, FIELD, STORE, true, false, TRACE>(prm, s);
  return trees ? launch_render_p<P, FIELD, STORE, false, true, TRACE>(prm, s)
               : launch_render_p<P, FIELD, STORE, false, false, TRACE>(prm, s);
}

template <int STORE, bool TRACE>
cudaError_t launch_render_s(const RenderParams &prm, int degree, int f, cudaStream_t s) {
  if (f == 3) {  // scalar with gradient shading
    switch (degree) {
      case 1: return launch_render_t<1, 3, STORE, TRACE>(prm, s);
      case 2: return launch_render_t<2, 3, STORE, TRACE>(prm, s);
      case 3: return launch_render_t<3, 3, STORE, TRACE>(prm, s);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (degree * 3 + f) {
    case 3: return launch_render_t<1, 0, STORE, TRACE>(prm, s);
    case 4: return launch_render_t<1, 1, STORE, TRACE>(prm, s);
    case 5: return launch_render_t<1, 2, STORE, TRACE>(prm, s);
    case 6: return launch_render_t<2, 0, STORE, TRACE>(prm, s);
    case 7: return launch_render_t<2, 1, STORE, TRACE>(prm, s);
    case 8: return launch_render_t<2, 2, STORE, TRACE>(prm, s);
    case 9: return launch_render_t<3, 0, STORE, TRACE>(prm, s);
    case 10: return launch_render_t<3, 1, STORE, TRACE>(prm, s);
    case 11: return launch_render_t<3, 2, STORE, TRACE>(prm, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace lrvol
