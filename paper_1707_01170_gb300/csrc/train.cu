// liblrvol: FP32 training of the step network (16 -> 64 -> 64 -> 64 -> 1, ReLU)
// for sm_103a.
//
//   k_mlp_tiles    forward, loss and backward of whole row tiles in shared
//                  memory; one partial gradient per CTA.
//   k_mlp_reduce   sum of the partial gradients in a fixed order, the loss and
//                  (for a training step) Adam.
#include <algorithm>

#include "device_common.cuh"

namespace lrvol {
namespace {

constexpr int kTrainWarps = 8;
constexpr int kTrainThreads = 32 * kTrainWarps;
// Row strides in floats.  Multiples of 4 (float4 rows) that step the banks by
// 4 or 20 words a row, so eight lanes reading 16 bytes each of eight
// consecutive rows touch every bank once.
constexpr int kHS = kHid + 4;
constexpr int kXS = kIn + 4;

template <int R>
struct TrainSmem {
  float x[R * kXS];
  float h[3][R * kHS];     // activations h1, h2, h3; each turns into its own gradient on the way back
  float w1[kIn * kHid];
  float w2[kHid * kHid], w3[kHid * kHid];      // [in][out]: forward
  float w2t[kHid * kHS], w3t[kHid * kHS];      // [out][in]: backward
  float w4[kHid];
  float b[3 * kHid];
  float dy[R];
  float red[3][kTrainThreads / kHid][kHid];    // the column sums' row groups
  double loss[R / 32];
};

// acc[r][q] = sum_k a[lane + 32 r][k] * w[k][j0 + 2q .. 2q + 1]: a row a lane,
// so the weights are the same address for a whole warp (one wavefront per 16
// bytes) and a row's values are read 16 bytes at a time.
template <int R, int K, int AS, int WS>
__device__ __forceinline__ void rows_times_weights(const float *a, const float *w, int j0, int lane, f2 (&acc)[R / 32][4]) {
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 x[R / 32];
#pragma unroll
    for (int r = 0; r < R / 32; ++r) x[r] = *reinterpret_cast<const float4 *>(a + (lane + 32 * r) * AS + k);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(w + (k + kk) * WS + j0);
      const ulonglong2 wb = *reinterpret_cast<const ulonglong2 *>(w + (k + kk) * WS + j0 + 4);
#pragma unroll
      for (int r = 0; r < R / 32; ++r) {
        const float xv = kk == 0 ? x[r].x : (kk == 1 ? x[r].y : (kk == 2 ? x[r].z : x[r].w));
        const f2 xx = f2_pack(xv, xv);
        acc[r][0] = f2_fma(wa.x, xx, acc[r][0]);
        acc[r][1] = f2_fma(wa.y, xx, acc[r][1]);
        acc[r][2] = f2_fma(wb.x, xx, acc[r][2]);
        acc[r][3] = f2_fma(wb.y, xx, acc[r][3]);
      }
    }
  }
}

// One hidden layer: out = relu(in W + b), this warp's 8 columns.
template <int R, int K, int AS>
__device__ __forceinline__ void layer_forward(const float *in, const float *w, const float *bias, float *out, int warp,
                                              int lane) {
  const int j0 = 8 * warp;
  f2 acc[R / 32][4];
#pragma unroll
  for (int r = 0; r < R / 32; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = f2_pack(bias[j0 + 2 * q], bias[j0 + 2 * q + 1]);
  rows_times_weights<R, K, AS, kHid>(in, w, j0, lane, acc);
#pragma unroll
  for (int r = 0; r < R / 32; ++r) {
    float4 *o = reinterpret_cast<float4 *>(out + (lane + 32 * r) * kHS + j0);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 v = f2x2_to_float4(acc[r][2 * h], acc[r][2 * h + 1]);
      v.x = fmaxf(v.x, 0.f);
      v.y = fmaxf(v.y, 0.f);
      v.z = fmaxf(v.z, 0.f);
      v.w = fmaxf(v.w, 0.f);
      o[h] = v;
    }
  }
}

// g[p][c] += sum_b in[b][k0 + 2p .. 2p + 1] * d[b][lane + 32 c]: lanes are
// columns here, the inputs the same address for a whole warp.
template <int R, int NP, int AS>
__device__ __forceinline__ void weight_grad(const float *in, const float *d, int k0, int lane, f2 (&g)[NP][2]) {
#pragma unroll 4
  for (int b = 0; b < R; ++b) {
    const float d0 = d[b * kHS + lane], d1 = d[b * kHS + lane + 32];
    const f2 dd0 = f2_pack(d0, d0), dd1 = f2_pack(d1, d1);
    f2 v[NP];
    if constexpr (NP % 2 == 0) {
#pragma unroll
      for (int p = 0; p < NP; p += 2) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(in + b * AS + k0 + 2 * p);
        v[p] = w.x;
        v[p + 1] = w.y;
      }
    } else {
#pragma unroll
      for (int p = 0; p < NP; ++p) v[p] = *reinterpret_cast<const f2 *>(in + b * AS + k0 + 2 * p);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      g[p][0] = f2_fma(v[p], dd0, g[p][0]);
      g[p][1] = f2_fma(v[p], dd1, g[p][1]);
    }
  }
}

template <int NP>
__device__ __forceinline__ void store_weight_grad(float *out, const f2 (&g)[NP][2], int k0, int lane) {
#pragma unroll
  for (int p = 0; p < NP; ++p)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float lo, hi;
      f2_unpack(g[p][c], lo, hi);
      out[(k0 + 2 * p) * kHid + lane + 32 * c] = lo;
      out[(k0 + 2 * p + 1) * kHid + lane + 32 * c] = hi;
    }
}

// Gradient of the inputs of a layer, where the inputs' ReLU is open: acc =
// (d W^T), kept until every warp has read what it overwrites.
template <int R>
__device__ __forceinline__ void input_grad(const float *d, const float *wt, int warp, int lane, f2 (&acc)[R / 32][4]) {
#pragma unroll
  for (int r = 0; r < R / 32; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[r][q] = 0;
  rows_times_weights<R, kHid, kHS, kHS>(d, wt, 8 * warp, lane, acc);
}
template <int R>
__device__ __forceinline__ void store_input_grad(float *h, const f2 (&acc)[R / 32][4], int warp, int lane) {
#pragma unroll
  for (int r = 0; r < R / 32; ++r) {
    float4 *o = reinterpret_cast<float4 *>(h + (lane + 32 * r) * kHS + 8 * warp);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float4 a = o[q], v = f2x2_to_float4(acc[r][2 * q], acc[r][2 * q + 1]);
      o[q] = make_float4(a.x > 0.f ? v.x : 0.f, a.y > 0.f ? v.y : 0.f, a.z > 0.f ? v.z : 0.f, a.w > 0.f ? v.w : 0.f);
    }
  }
}

// A CTA takes row tiles of R rows in turn (grid stride): the three layers
// forward, the loss, and the backward pass all stay in shared memory, and the
// gradient of the CTA's rows stays in registers until its last tile.  Each
// CTA then writes one partial gradient; k_mlp_reduce adds them.  Per tile a
// layer is a (R x 64) x (64 x 64) product on packed FP32 FMAs; a lane's
// operand is 16 bytes of its own row (4 wavefronts) and the other operand is
// uniform over the warp (1 wavefront per 16 bytes), so a 64-row tile costs
// 0.25 shared-memory wavefronts per FMA instruction of the four schedulers.
// With every SM on one tile the step is bound by the chain of twelve phases
// between barriers, not by the FMA rate (8,192 rows: 456 MFLOP, 6 us at the
// FP32 peak): 29 us a step through the binding, against 3,558 us for a launch
// per layer and direction whose weight-gradient threads walked all rows alone.
// (One CTA an SM is stated: left open, the registers are cut to 80 and 100 of 169
// and 145, and a step takes 2 us more.)
template <int R>
__global__ void __launch_bounds__(kTrainThreads, 1) k_mlp_tiles(const float *__restrict__ x, const float *__restrict__ tgt,
                                                                int64_t n, const float *__restrict__ p,
                                                                float *__restrict__ part, float *__restrict__ loss_part) {
  extern __shared__ __align__(16) unsigned char train_smem[];
  TrainSmem<R> &S = *reinterpret_cast<TrainSmem<R> *>(train_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int q = tid; q < kIn * kHid; q += kTrainThreads) S.w1[q] = __ldg(p + kOffW1 + q);
  for (int q = tid; q < kHid * kHid; q += kTrainThreads) {
    const float a = __ldg(p + kOffW2 + q), b = __ldg(p + kOffW3 + q);
    S.w2[q] = a;
    S.w3[q] = b;
    S.w2t[(q % kHid) * kHS + q / kHid] = a;
    S.w3t[(q % kHid) * kHS + q / kHid] = b;
  }
  if (tid < kHid) {
    S.w4[tid] = __ldg(p + kOffW4 + tid);
    S.b[tid] = __ldg(p + kOffB1 + tid);
    S.b[kHid + tid] = __ldg(p + kOffB2 + tid);
    S.b[2 * kHid + tid] = __ldg(p + kOffB3 + tid);
  }
  const float b4 = __ldg(p + kOffB4), nf = (float)n;
  f2 g1[1][2] = {}, g2[4][2] = {}, g3[4][2] = {};
  float gw4 = 0.f, gb3 = 0.f, gb2 = 0.f, gb1 = 0.f, gb4 = 0.f;
  double loss = 0.0;
  const int col = tid % kHid, grp = tid / kHid;        // column sums: a column and a quarter of the rows a thread
  constexpr int GR = R * kHid / kTrainThreads;         // rows of a quarter
  const int64_t tiles = (n + R - 1) / R;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t row0 = tile * R;
    const int rows = (int)min((int64_t)R, n - row0);
    __syncthreads();   // the weights are staged; the last tile's readers are done
    for (int q = tid; q < R * kIn; q += kTrainThreads)
      S.x[(q / kIn) * kXS + q % kIn] = q < rows * kIn ? __ldg(x + row0 * kIn + q) : 0.f;
    __syncthreads();
    layer_forward<R, kIn, kXS>(S.x, S.w1, S.b, S.h[0], warp, lane);
    __syncthreads();
    layer_forward<R, kHid, kHS>(S.h[0], S.w2, S.b + kHid, S.h[1], warp, lane);
    __syncthreads();
    layer_forward<R, kHid, kHS>(S.h[1], S.w3, S.b + 2 * kHid, S.h[2], warp, lane);
    __syncthreads();
    if (tid < R) {     // output, loss and its derivative: a row a thread
      float y = b4;
#pragma unroll 4
      for (int k = 0; k < kHid; k += 4) {
        const float4 v = *reinterpret_cast<const float4 *>(S.h[2] + tid * kHS + k);
        y = fmaf(v.x, S.w4[k], y);
        y = fmaf(v.y, S.w4[k + 1], y);
        y = fmaf(v.z, S.w4[k + 2], y);
        y = fmaf(v.w, S.w4[k + 3], y);
      }
      const float r = tid < rows ? y - __ldg(tgt + row0 + tid) : 0.f;
      const float dy = r / nf;
      S.dy[tid] = dy;
      gb4 += dy;
      loss += 0.5 * (double)r * (double)r;
    }
    __syncthreads();
    {                  // h3 -> its gradient; sums over the rows for w4 and b3
      const float w4 = S.w4[col];
#pragma unroll 8
      for (int b = grp * GR; b < (grp + 1) * GR; ++b) {
        const float h = S.h[2][b * kHS + col], dy = S.dy[b];
        gw4 = fmaf(h, dy, gw4);
        const float d = h > 0.f ? dy * w4 : 0.f;
        gb3 += d;
        S.h[2][b * kHS + col] = d;
      }
    }
    __syncthreads();
    f2 acc[R / 32][4];
    weight_grad<R, 4, kHS>(S.h[1], S.h[2], 8 * warp, lane, g3);
    input_grad<R>(S.h[2], S.w3t, warp, lane, acc);
    __syncthreads();
    store_input_grad<R>(S.h[1], acc, warp, lane);
    __syncthreads();
    weight_grad<R, 4, kHS>(S.h[0], S.h[1], 8 * warp, lane, g2);
    input_grad<R>(S.h[1], S.w2t, warp, lane, acc);
#pragma unroll 8
    for (int b = grp * GR; b < (grp + 1) * GR; ++b) gb2 += S.h[1][b * kHS + col];
    __syncthreads();
    store_input_grad<R>(S.h[0], acc, warp, lane);
    __syncthreads();
    weight_grad<R, 1, kXS>(S.x, S.h[0], 2 * warp, lane, g1);
#pragma unroll 8
    for (int b = grp * GR; b < (grp + 1) * GR; ++b) gb1 += S.h[0][b * kHS + col];
  }
  // this CTA's partial gradient
  float *out = part + (int64_t)blockIdx.x * kParams;
  store_weight_grad(out + kOffW1, g1, 2 * warp, lane);
  store_weight_grad(out + kOffW2, g2, 8 * warp, lane);
  store_weight_grad(out + kOffW3, g3, 8 * warp, lane);
  float(*red)[kHid] = &S.red[0][0];
  __syncthreads();
  S.red[0][grp][col] = gb1;
  S.red[1][grp][col] = gb2;
  S.red[2][grp][col] = gb3;
  __syncthreads();
  if (tid < 3 * kHid) {
    const int l = tid / kHid, c = tid % kHid;
    float s = S.red[l][0][c];
    for (int q = 1; q < kTrainThreads / kHid; ++q) s += S.red[l][q][c];
    out[(l == 0 ? kOffB1 : (l == 1 ? kOffB2 : kOffB3)) + c] = s;
  }
  __syncthreads();
  red[grp][col] = gw4;
  // b4 and the loss: rows sit in the first R / 32 warps
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gb4 += __shfl_down_sync(0xffffffffu, gb4, o);
    loss += __shfl_down_sync(0xffffffffu, loss, o);
  }
  if (lane == 0 && warp < R / 32) {
    S.dy[warp] = gb4;
    S.loss[warp] = loss;
  }
  __syncthreads();
  if (tid < kHid) {
    float s = red[0][tid];
    for (int q = 1; q < kTrainThreads / kHid; ++q) s += red[q][tid];
    out[kOffW4 + tid] = s;
  }
  if (tid == 0) {
    float s = S.dy[0];
    double l = S.loss[0];
    for (int q = 1; q < R / 32; ++q) {
      s += S.dy[q];
      l += S.loss[q];
    }
    out[kOffB4] = s;
    loss_part[2 * blockIdx.x] = __int_as_float(__double2loint(l));
    loss_part[2 * blockIdx.x + 1] = __int_as_float(__double2hiint(l));
  }
}

struct AdamParams {
  float *p, *m, *v;   // null for a gradient only
  float lr, c1, c2;   // c = 1 - beta^t
};

constexpr int kRedParams = 32, kRedGroups = 8;

// grad[q] = the sum over the CTAs' partials: 32 parameters a CTA, one per
// lane, every warp an eighth of the partials, the eighths added in order; then
// Adam on the parameter.  The first CTA adds the losses.  (part may be grad
// itself when there is one partial.)
__global__ void __launch_bounds__(kRedParams *kRedGroups) k_mlp_reduce(const float *part, int parts,
                                                                      const float *__restrict__ loss_part, int64_t n,
                                                                      float *grad, float *__restrict__ loss,
                                                                      AdamParams ad) {
  __shared__ float red[kRedGroups][kRedParams];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int q = blockIdx.x * kRedParams + lane;
  const int per = (parts + kRedGroups - 1) / kRedGroups;
  const int g1 = min(parts, (grp + 1) * per);
  float s = 0.f;
  if (q < kParams) {
#pragma unroll 8
    for (int g = grp * per; g < g1; ++g) s += part[(int64_t)g * kParams + q];
  }
  red[grp][lane] = s;
  __syncthreads();
  if (grp == 0 && q < kParams) {
    for (int g = 1; g < kRedGroups; ++g) s += red[g][lane];
    grad[q] = s;
    if (ad.p) {
      const float mq = 0.9f * ad.m[q] + 0.1f * s;
      const float vq = 0.999f * ad.v[q] + 0.001f * s * s;
      ad.m[q] = mq;
      ad.v[q] = vq;
      ad.p[q] -= ad.lr * (mq / ad.c1) / (sqrtf(vq / ad.c2) + 1e-8f);
    }
  }
  if (blockIdx.x == 0 && grp == 1 && loss) {
    double l = 0.0;
    for (int g = lane; g < parts; g += 32)
      l += __hiloint2double(__float_as_int(loss_part[2 * g + 1]), __float_as_int(loss_part[2 * g]));
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if (lane == 0) *loss = (float)(l / (double)n);
  }
}

template <int R>
cudaError_t launch_tiles(const float *x, const float *target, int64_t n, const float *p, float *part, float *loss_part,
                         unsigned ctas, cudaStream_t s) {
  const int bytes = (int)sizeof(TrainSmem<R>);
  const cudaError_t e = cudaFuncSetAttribute(k_mlp_tiles<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  k_mlp_tiles<R><<<ctas, kTrainThreads, bytes, s>>>(x, target, n, p, part, loss_part);
  return cudaGetLastError();
}

}  // namespace

// Scratch (floats): the CTAs' losses (a double each, as two floats), then
// their partial gradients.  The scratch holds n * (6 * 64 + 2) floats before
// its gradient vector, which bounds the CTAs of a small batch; one CTA's
// partial is the gradient itself.  Batches of up to 32 rows per SM take 32-row
// tiles: half the work between two barriers (23 against 28 us at 64 to 4,096
// rows, 26.8 against 30.9 us at 4,864).  Past that a CTA would take a second
// 32-row tile, and 64-row tiles, with half the weight reads per row, are
// faster (6,000 rows: 30 against 35 us; 65,536: 115 against 148 us).
cudaError_t launch_mlp_grad(const float *x, const float *target, int64_t n, float *p, float *grad, float *loss,
                            float *scratch, const AdamStep *adam, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t room = n * (6 * (int64_t)kHid + 2) / (kParams + 2);
  const bool small = n <= 32 * (int64_t)sms;
  const int64_t tiles = (n + (small ? 31 : 63)) / (small ? 32 : 64);
  const int64_t ctas = std::max<int64_t>(1, std::min(std::min<int64_t>(tiles, sms), room));
  float *loss_part = scratch, *part = ctas == 1 ? grad : scratch + 2 * ctas;
  e = small ? launch_tiles<32>(x, target, n, p, part, loss_part, (unsigned)ctas, s)
            : launch_tiles<64>(x, target, n, p, part, loss_part, (unsigned)ctas, s);
  if (e != cudaSuccess) return e;
  AdamParams ad = {nullptr, nullptr, nullptr, 0.f, 1.f, 1.f};
  if (adam)
    ad = {p, adam->m, adam->v, adam->lr, 1.f - powf(0.9f, (float)adam->t), 1.f - powf(0.999f, (float)adam->t)};
  k_mlp_reduce<<<(kParams + kRedParams - 1) / kRedParams, kRedParams * kRedGroups, 0, s>>>(part, (int)ctas, loss_part, n,
                                                                                         grad, loss, ad);
  return cudaGetLastError();
}

}  // namespace lrvol
