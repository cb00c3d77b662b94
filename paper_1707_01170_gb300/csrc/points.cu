// liblrvol point kernels for sm_103a: look-up, value and gradient at points.
//
//   k_lookup         Alg. 1 element look-up through the k-d forest.
//   k_eval_points    look-up + Bezier block evaluation (values, or value and
//                    gradient of a scalar volume) at equal degrees 1..3.
//   k_eval_any, k_eval_grad_any   the same at any degrees up to 4.
#include "device_common.cuh"

namespace lrvol {
namespace {

__global__ void k_lookup(ForestView f, int64_t n_elem, const float *__restrict__ pts, int64_t n,
                         uint32_t *__restrict__ out, uint32_t *status) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float x = pts[3 * q], y = pts[3 * q + 1], z = pts[3 * q + 2];
  uint32_t e = kNone;
  if (x >= 0.f && x <= 1.f && y >= 0.f && y <= 1.f && z >= 0.f && z <= 1.f) {
    e = forest_lookup(f, x, y, z, status);
    if (e != kNone && (int64_t)e >= n_elem) {
      set_status(status, kStatusBounds);
      e = kNone;
    }
  }
  out[q] = e;
}


// The element holding point q, or kNone outside [0,1]^3.
__device__ __forceinline__ uint32_t find_element(const ForestView &f, int64_t n_elem, float x, float y, float z,
                                                 uint32_t *status) {
  if (!(x >= 0.f && x <= 1.f && y >= 0.f && y <= 1.f && z >= 0.f && z <= 1.f)) return kNone;
  const uint32_t e = forest_lookup(f, x, y, z, status);
  return (int64_t)e < n_elem ? e : kNone;
}

// One point a thread, with the renderer's block code (256-bit loads, packed
// FP32 contraction): a dependent head load, then the record and the block.
// Scattered points are bound by L1's data path, 86 % busy (a scattered 256-bit
// load is eight wavefronts), with the L2 at 58 % of its rate: 1,000,003 gradients of
// a tricubic FP32 volume read 336 bytes each and take 52 us (350 us when the block
// went through a local array, a scalar load a coefficient, under loops over
// any degree); points in grid order share blocks and take 29 us (190).
// Gathering a warp's blocks to shared memory with neighbouring lanes on one
// block took 52 to 56 us, and more registers a thread 52 us.
template <int P, int NC, int STORE, bool GRAD>
__global__ void __launch_bounds__(128) k_eval_points(const ForestView f, const ElemRec *__restrict__ elem, int64_t n_elem,
                                                     const unsigned char *__restrict__ bez, const float *__restrict__ pts, int64_t n, float *__restrict__ out,
                                                     uint32_t *status) {
  constexpr int N = P + 1;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float x = __ldg(pts + 3 * q), y = __ldg(pts + 3 * q + 1), z = __ldg(pts + 3 * q + 2);
  const uint32_t e = find_element(f, n_elem, x, y, z, status);
  float v[NC], g[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int c = 0; c < NC; ++c) v[c] = 0.f;
  if (e != kNone) {
    float4 ra, rb, rc, rd;
    Block<P, NC == 3 ? 1 : 0, STORE, false> blk;
    load_record(elem + e, ra, rb, rc, rd);
    blk.load(bez + (int64_t)e * blk.BYTES, 0);
    const float ux = local_u(x, ra.x, rc.x, rd.x), uy = local_u(y, ra.y, rc.y, rd.y), uz = local_u(z, ra.z, rc.z, rd.z);
    float bx[N], by[N], bz[N];
    monomials<P>(ux, bx);
    monomials<P>(uy, by);
    monomials<P>(uz, bz);
    if constexpr (GRAD) {
      float dx[N], dy[N], dz[N];
      dmonomials<P>(ux, dx);
      dmonomials<P>(uy, dy);
      dmonomials<P>(uz, dz);
      v[0] = blk.eval_grad(bx, by, bz, dx, dy, dz, g[0], g[1], g[2]);
      g[0] *= rd.x;
      g[1] *= rd.y;
      g[2] *= rd.z;
    } else if constexpr (NC == 3) {
      blk.components(bx, by, bz, v[0], v[1], v[2]);
    } else {
      v[0] = blk.eval(bx, by, bz);
    }
  }
  if constexpr (GRAD) {
    reinterpret_cast<float4 *>(out)[q] = make_float4(v[0], g[0], g[1], g[2]);
  } else {
#pragma unroll
    for (int c = 0; c < NC; ++c) out[NC * q + c] = v[c];
  }
}

// Evaluation at any degrees p0, p1, p2 <= 4: degree 4 and unequal degrees.
__device__ float eval_generic(const float *c, const int *deg, float ux, float uy, float uz) {
  float b[3][kMaxDeg + 1];
  const float u[3] = {ux, uy, uz};
  for (int a = 0; a < 3; ++a) {
    const int p = deg[a];
    const float v = 1.f - u[a];
    for (int i = 0; i <= p; ++i) {
      float m = 1.f;
      for (int q = 0; q < i; ++q) m *= u[a];
      for (int q = i; q < p; ++q) m *= v;
      b[a][i] = m;
    }
  }
  const int n0 = deg[0] + 1, n1 = deg[1] + 1, n2 = deg[2] + 1;
  float f = 0.f;
  for (int k = 0; k < n2; ++k) {
    float t = 0.f;
    for (int j = 0; j < n1; ++j) {
      float s = 0.f;
      for (int i = 0; i < n0; ++i) s = fmaf(c[(k * n1 + j) * n0 + i], b[0][i], s);
      t = fmaf(s, b[1][j], t);
    }
    f = fmaf(t, b[2][k], f);
  }
  return f;
}

// Value and derivatives in local coordinates (d/du, d/dv, d/dw) of the same block.
__device__ float eval_generic_grad(const float *c, const int *deg, float ux, float uy, float uz, float *g) {
  float b[3][kMaxDeg + 1], db[3][kMaxDeg + 1];
  const float u[3] = {ux, uy, uz};
  for (int a = 0; a < 3; ++a) {
    const int p = deg[a];
    const float v = 1.f - u[a];
    for (int i = 0; i <= p; ++i) {
      float m = 1.f, d1 = 0.f, d2 = 0.f;
      for (int q = 0; q < i; ++q) m *= u[a];
      for (int q = i; q < p; ++q) m *= v;
      if (i > 0) {  // i u^(i-1) v^(p-i)
        d1 = (float)i;
        for (int q = 0; q < i - 1; ++q) d1 *= u[a];
        for (int q = i; q < p; ++q) d1 *= v;
      }
      if (i < p) {  // (p-i) u^i v^(p-i-1)
        d2 = (float)(p - i);
        for (int q = 0; q < i; ++q) d2 *= u[a];
        for (int q = i + 1; q < p; ++q) d2 *= v;
      }
      b[a][i] = m;
      db[a][i] = d1 - d2;
    }
  }
  const int n0 = deg[0] + 1, n1 = deg[1] + 1, n2 = deg[2] + 1;
  float f = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
  for (int k = 0; k < n2; ++k) {
    float t = 0.f, tx = 0.f, ty = 0.f;
    for (int j = 0; j < n1; ++j) {
      float s = 0.f, sx = 0.f;
      for (int i = 0; i < n0; ++i) {
        const float cc = c[(k * n1 + j) * n0 + i];
        s = fmaf(cc, b[0][i], s);
        sx = fmaf(cc, db[0][i], sx);
      }
      t = fmaf(s, b[1][j], t);
      tx = fmaf(sx, b[1][j], tx);
      ty = fmaf(s, db[1][j], ty);
    }
    f = fmaf(t, b[2][k], f);
    gx = fmaf(tx, b[2][k], gx);
    gy = fmaf(ty, b[2][k], gy);
    gz = fmaf(t, db[2][k], gz);
  }
  g[0] = gx;
  g[1] = gy;
  g[2] = gz;
  return f;
}

__device__ __forceinline__ float load_slot(const unsigned char *eb, int storage, int slot) {
  if (storage == LRVOL_STORE_F32) return __ldg(reinterpret_cast<const float *>(eb) + slot);
  const unsigned short h = __ldg(reinterpret_cast<const unsigned short *>(eb + kHeaderBytes) + slot);
  if (storage == LRVOL_STORE_F16) return __half2float(__ushort_as_half(h));
  return __uint_as_float((unsigned)h << 16);
}

__global__ void k_eval_any(ForestView f, const ElemRec *__restrict__ elem, int64_t n_elem,
                       const unsigned char *__restrict__ bez, int ebytes, int storage, int p0, int p1, int p2, int nc,
                       const float *__restrict__ pts, int64_t n, float *__restrict__ out, uint32_t *status) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float x = pts[3 * q], y = pts[3 * q + 1], z = pts[3 * q + 2];
  uint32_t e = kNone;
  if (x >= 0.f && x <= 1.f && y >= 0.f && y <= 1.f && z >= 0.f && z <= 1.f) e = forest_lookup(f, x, y, z, status);
  if (e == kNone || (int64_t)e >= n_elem) {
    for (int c = 0; c < nc; ++c) out[q * nc + c] = 0.f;
    return;
  }
  const ElemRec r = elem[e];
  const float ux = local_u(x, r.a.x, r.c.x, r.d.x);
  const float uy = local_u(y, r.a.y, r.c.y, r.d.y);
  const float uz = local_u(z, r.a.z, r.c.z, r.d.z);
  const int deg[3] = {p0, p1, p2};
  const int n0 = p0 + 1, n1 = p1 + 1, nb = n0 * n1 * (p2 + 1);
  const unsigned char *eb = bez + (int64_t)e * ebytes;
  for (int c = 0; c < nc; ++c) {
    float cl[(kMaxDeg + 1) * (kMaxDeg + 1) * (kMaxDeg + 1)];
    for (int t = 0; t < nb; ++t) cl[t] = load_slot(eb, storage, render_slot(nc, n0, nb, t / n0, t % n0, c));
    const float v = eval_generic(cl, deg, ux, uy, uz);
    if (storage == LRVOL_STORE_F32) {
      out[q * nc + c] = v;
    } else {
      const float *hdr = reinterpret_cast<const float *>(eb);
      out[q * nc + c] = fmaf(__ldg(hdr + 3 + c), v, __ldg(hdr + c));
    }
  }
}

// Value and world-space gradient of a scalar volume at points (n x 4 out).
__global__ void k_eval_grad_any(ForestView f, const ElemRec *__restrict__ elem, int64_t n_elem,
                            const unsigned char *__restrict__ bez, int ebytes, int storage, int p0, int p1, int p2,
                            const float *__restrict__ pts, int64_t n, float *__restrict__ out, uint32_t *status) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const float x = pts[3 * q], y = pts[3 * q + 1], z = pts[3 * q + 2];
  uint32_t e = kNone;
  if (x >= 0.f && x <= 1.f && y >= 0.f && y <= 1.f && z >= 0.f && z <= 1.f) e = forest_lookup(f, x, y, z, status);
  float4 *o = reinterpret_cast<float4 *>(out) + q;
  if (e == kNone || (int64_t)e >= n_elem) {
    *o = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const ElemRec r = elem[e];
  const int deg[3] = {p0, p1, p2};
  const int n0 = p0 + 1, nb = n0 * (p1 + 1) * (p2 + 1);
  const unsigned char *eb = bez + (int64_t)e * ebytes;
  float cl[(kMaxDeg + 1) * (kMaxDeg + 1) * (kMaxDeg + 1)];
  for (int t = 0; t < nb; ++t) cl[t] = load_slot(eb, storage, render_slot(1, n0, nb, t / n0, t % n0, 0));
  float g[3];
  float v = eval_generic_grad(cl, deg, local_u(x, r.a.x, r.c.x, r.d.x), local_u(y, r.a.y, r.c.y, r.d.y),
                              local_u(z, r.a.z, r.c.z, r.d.z), g);
  float sc = 1.f;
  if (storage != LRVOL_STORE_F32) {
    const float *hdr = reinterpret_cast<const float *>(eb);
    sc = __ldg(hdr + 3);
    v = fmaf(sc, v, __ldg(hdr));
  }
  *o = make_float4(v, sc * g[0] * r.d.x, sc * g[1] * r.d.y, sc * g[2] * r.d.z);
}

template <int NC, bool GRAD, int P>
cudaError_t launch_points_p(const lrvol_s *v, const float *pts, int64_t n, float *out, cudaStream_t s) {
  const unsigned blocks = (unsigned)((n + 127) / 128);
  const ForestView f = forest_view(v);
  switch (v->storage) {
#define LRVOL_PTS(S_)                                                                                             \
  k_eval_points<P, NC, S_, GRAD><<<blocks, 128, 0, s>>>(f, v->d_elem, v->n_elem, v->d_bez, pts, n, out, \
                                                        v->d_status);                                             \
  break
    case LRVOL_STORE_F32: LRVOL_PTS(LRVOL_STORE_F32);
    case LRVOL_STORE_F16: LRVOL_PTS(LRVOL_STORE_F16);
    case LRVOL_STORE_BF16: LRVOL_PTS(LRVOL_STORE_BF16);
    default: return cudaErrorInvalidValue;
#undef LRVOL_PTS
  }
  return cudaGetLastError();
}

template <int NC, bool GRAD>
cudaError_t launch_points(const lrvol_s *v, const float *pts, int64_t n, float *out, cudaStream_t s) {
  switch (v->p[0]) {
    case 1: return launch_points_p<NC, GRAD, 1>(v, pts, n, out, s);
    case 2: return launch_points_p<NC, GRAD, 2>(v, pts, n, out, s);
    default: return launch_points_p<NC, GRAD, 3>(v, pts, n, out, s);
  }
}

// Equal degrees 1..3 have kernels with the degree known (6.8 times as fast at
// degree 3, see k_eval_points); other volumes go through the loops over any
// degree.
bool has_point_kernel(const lrvol_s *v) { return v->p[0] == v->p[1] && v->p[0] == v->p[2] && v->p[0] <= 3; }

}  // namespace

cudaError_t launch_lookup(const lrvol_s *v, const float *pts, int64_t n, uint32_t *out, cudaStream_t s) {
  k_lookup<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(forest_view(v), v->n_elem, pts, n, out, v->d_status);
  return cudaGetLastError();
}

cudaError_t launch_eval(const lrvol_s *v, const float *pts, int64_t n, float *out, cudaStream_t s) {
  if (has_point_kernel(v))
    return v->nc == 3 ? launch_points<3, false>(v, pts, n, out, s) : launch_points<1, false>(v, pts, n, out, s);
  k_eval_any<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(forest_view(v), v->d_elem, v->n_elem, v->d_bez,
                                                    v->elem_bytes, v->storage, v->p[0], v->p[1], v->p[2],
                                                    v->nc, pts, n, out, v->d_status);
  return cudaGetLastError();
}

cudaError_t launch_eval_grad(const lrvol_s *v, const float *pts, int64_t n, float *out, cudaStream_t s) {
  if (has_point_kernel(v)) return launch_points<1, true>(v, pts, n, out, s);
  k_eval_grad_any<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(forest_view(v), v->d_elem, v->n_elem, v->d_bez,
                                                         v->elem_bytes, v->storage, v->p[0], v->p[1], v->p[2], pts,
                                                         n, out, v->d_status);
  return cudaGetLastError();
}

}  // namespace lrvol
