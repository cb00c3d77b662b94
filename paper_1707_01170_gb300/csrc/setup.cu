// liblrvol set-up kernels for sm_103a: what lrvol_to_bezier does once per volume.
//
//   k_cell_*, k_incident, k_sort_lists, k_scan_*, k_incident_direct, k_incident_small
//                  element -> B-spline incidence: the B-splines whose support
//                  contains the element, in ascending order.
//   k_to_bezier    Sec. 3.2.3 change of basis, FP64: per element, the Bernstein
//                  coefficients of every incident B-spline's univariate factors
//                  over the element, by blossoming, accumulated with gamma*c.
//   k_pack         the render copy of the blocks in its storage, and their ranges.
//   k_elem_records element boxes -> FP32 records (rounded-up corners, Eq. 4 step).
#include <algorithm>
#include <cmath>

#include "device_common.cuh"

namespace lrvol {
namespace {

// ----------------------------------------------------------------------------
// incidence.  Elements are bucketed by their centres on a grid of R^3 cells, so
// a B-spline's candidates are the buckets its support meets: for each (y, z)
// one contiguous run of elements.  A warp takes a B-spline and its lanes the
// run's elements, 16 to a run (about 16 elements); a pass counts the elements'
// B-splines, the other fills their lists.  The lists are filled in no fixed order
// and sorted afterwards, since k_to_bezier adds in the list's order.  An FP64
// comparison occupies an SM for 16 cycles whatever lanes take part, so FP64 values
// are compared by their bits as integers, and the support's six cells are
// computed by six lanes at once; the boxes are copied into the buckets' order,
// so that a run is read in whole lines.  179,768 elements and 11.8 M entries: 240 us
// to count and 325 to fill; 677 each with the boxes read where they are, 865 with
// FP64 comparisons and a warp to a run.  (One host thread took 145 ms for it all.)
// ----------------------------------------------------------------------------
struct CellGrid {
  int R;
  __host__ __device__ int64_t cells() const { return (int64_t)R * R * R; }
  __device__ __forceinline__ int coord(double x) const { return min(R - 1, max(0, (int)(x * R))); }
};

__global__ void __launch_bounds__(256) k_cell_count(const double *__restrict__ box, int64_t n_elem, CellGrid g,
                                                    int32_t *__restrict__ cell_of, uint32_t *__restrict__ count) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_elem) return;
  const double *b = box + 6 * e;
  const int cx = g.coord(0.5 * (b[0] + b[3])), cy = g.coord(0.5 * (b[1] + b[4])), cz = g.coord(0.5 * (b[2] + b[5]));
  const int32_t c = (cz * g.R + cy) * g.R + cx;
  cell_of[e] = c;
  atomicAdd(count + c, 1u);
}

// Integers in the order of the numbers (no NaN; both zeros are 0).
__device__ __forceinline__ int64_t order_key(double x) {
  const int64_t b = __double_as_longlong(x);
  return b >= 0 ? b : (b == INT64_MIN ? 0 : b ^ INT64_MAX);
}
__device__ __forceinline__ double from_order_key(int64_t k) { return __longlong_as_double(k >= 0 ? k : k ^ INT64_MAX); }
__device__ __forceinline__ int64_t order_key_01(double x) { return __double_as_longlong(x) & INT64_MAX; }   // x >= 0 or -0

// The elements of a cell side by side: their numbers, and for each axis the keys of
// their lower and upper ends.
__global__ void __launch_bounds__(256) k_cell_fill(const double *__restrict__ box, const int32_t *__restrict__ cell_of, int64_t n_elem,
                                                   const int64_t *__restrict__ cell_ptr, uint32_t *__restrict__ cursor,
                                                   int32_t *__restrict__ cell_el, longlong2 *__restrict__ ends) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_elem) return;
  const int32_t c = cell_of[e];
  const int64_t slot = cell_ptr[c] + atomicAdd(cursor + c, 1u);
  cell_el[slot] = (int32_t)e;
  const double *b = box + 6 * e;
#pragma unroll
  for (int a = 0; a < 3; ++a) ends[a * n_elem + slot] = make_longlong2(order_key_01(b[a]), order_key_01(b[3 + a]));
}

constexpr int kSetupWarps = 8;

// FILL false: count[e] = B-splines whose support contains element e.  FILL
// true: their indices from list[ptr[e]] on, count as the cursors (zeroed).
template <bool FILL>
__global__ void __launch_bounds__(32 * kSetupWarps) k_incident(
    const longlong2 *__restrict__ ends, int64_t n_elem, const double *__restrict__ knots, int64_t n_basis, int p0,
    int p1, int p2, int kw, CellGrid g, const int64_t *__restrict__ cell_ptr, const int32_t *__restrict__ cell_el,
    uint32_t *__restrict__ count, const int64_t *__restrict__ ptr, int32_t *__restrict__ list) {
  const int64_t i = (int64_t)blockIdx.x * kSetupWarps + (threadIdx.x >> 5);
  if (i >= n_basis) return;
  const int lane = threadIdx.x & 31;
  // lane 2a: lower end of the support on axis a, lane 2a + 1: its upper end
  const int axis = (lane >> 1) % 3;
  const int at = (axis > 0 ? p0 + 2 : 0) + (axis > 1 ? p1 + 2 : 0) + (lane & 1) * ((axis == 0 ? p0 : axis == 1 ? p1 : p2) + 1);
  const double knot = knots[i * kw + at];
  const int64_t key = order_key(knot);
  const int cell = g.coord(knot);
  int64_t end[6];
  int c[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    end[t] = __shfl_sync(0xffffffffu, key, t);
    c[t] = __shfl_sync(0xffffffffu, cell, t);
  }
  const int ny = c[3] - c[2] + 1, rows = ny * (c[5] - c[4] + 1);
  for (int r = lane >> 4; r < rows; r += 2) {
    const int64_t row = ((int64_t)(c[4] + r / ny) * g.R + c[2] + r % ny) * g.R;
    const int64_t stop = cell_ptr[row + c[1] + 1];
    for (int64_t q = cell_ptr[row + c[0]] + (lane & 15); q < stop; q += 16) {
      const longlong2 x = __ldg(ends + q), y = __ldg(ends + n_elem + q), z = __ldg(ends + 2 * n_elem + q);
      if (end[0] <= x.x && end[2] <= y.x && end[4] <= z.x && x.y <= end[1] && y.y <= end[3] && z.y <= end[5]) {
        const int32_t e = cell_el[q];
        const uint32_t n = atomicAdd(count + e, 1u);
        if constexpr (FILL) list[ptr[e] + n] = (int32_t)i;
      }
    }
  }
}

// out = the lists of `in` in ascending order (`in` is lost): a warp per element,
// every entry placed at the number of smaller ones (the entries are distinct).
// That is quadratic, and a list may hold every B-spline: past kSortLong entries
// the warp sorts by one bit after the other instead (n_bits of them hold an
// entry).  One element with 350,000 entries, the whole conversion: 0.24 s, 60 s
// by counting.
constexpr int64_t kSortLong = 4096;

__global__ void __launch_bounds__(32 * kSetupWarps) k_sort_lists(const int64_t *__restrict__ ptr, int64_t n_elem,
                                                                int n_bits, int32_t *in, int32_t *out) {
  const int64_t e = (int64_t)blockIdx.x * kSetupWarps + (threadIdx.x >> 5);
  if (e >= n_elem) return;
  const int lane = threadIdx.x & 31;
  const int64_t beg = ptr[e], end = ptr[e + 1];
  if (end - beg > kSortLong) {
    int32_t *from = in, *to = out;
    for (int bit = 0; bit < (n_bits | 1); ++bit) {   // an odd number of passes ends in `out`
      int64_t zeros = 0;
      for (int64_t q = beg + lane; q < end; q += 32) zeros += !(from[q] >> bit & 1);
      for (int o = 16; o > 0; o >>= 1) zeros += __shfl_xor_sync(0xffffffffu, zeros, o);
      int64_t at[2] = {beg, beg + zeros};
      int32_t next = beg + lane < end ? from[beg + lane] : 0;
      for (int64_t q0 = beg; q0 < end; q0 += 32) {
        const int32_t v = next;
        if (q0 + 32 + lane < end) next = from[q0 + 32 + lane];
        const bool valid = q0 + lane < end, one = v >> bit & 1;
        const unsigned m1 = __ballot_sync(0xffffffffu, valid && one), m0 = __ballot_sync(0xffffffffu, valid && !one);
        if (valid) to[(one ? at[1] : at[0]) + __popc((one ? m1 : m0) & ((1u << lane) - 1u))] = v;
        at[0] += __popc(m0);
        at[1] += __popc(m1);
      }
      __syncwarp();
      int32_t *const t = from;
      from = to;
      to = t;
    }
    return;
  }
  for (int64_t q0 = beg; q0 < end; q0 += 32) {
    const int32_t v = q0 + lane < end ? in[q0 + lane] : INT32_MAX;
    int rank = 0;
    for (int64_t t0 = beg; t0 < end; t0 += 32) {
      const int32_t w = t0 + lane < end ? in[t0 + lane] : INT32_MAX;
      const int n = (int)min((int64_t)32, end - t0);
      for (int s = 0; s < n; ++s) rank += __shfl_sync(0xffffffffu, w, s) < v;
    }
    if (q0 + lane < end) out[beg + rank] = v;
  }
}

// Exclusive prefix sums of n counts into out[0 .. n], three launches: tiles of
// 2,048 counts, the tiles' totals by one CTA, and the tiles' offsets added.
// `empty` is set when a count is 0.
constexpr int kScanThreads = 256, kScanItems = 8, kScanTile = kScanThreads * kScanItems;

// Exclusive prefix of v over the CTA's 256 threads, and the total.
__device__ __forceinline__ int64_t cta_exclusive(int64_t v, int64_t &total) {
  __shared__ int64_t warp_sum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();
  int64_t before = 0;
  total = 0;
  for (int w = 0; w < kScanThreads / 32; ++w) {
    if (w == warp) before = total;
    total += warp_sum[w];
  }
  __syncthreads();
  return before + inc - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(const uint32_t *__restrict__ count, int64_t n,
                                                             int64_t *__restrict__ out, int64_t *__restrict__ sums,
                                                             uint32_t *__restrict__ empty) {
  const int64_t q0 = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t c[kScanItems];
  int64_t sum = 0, total;
  bool zero = false;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    c[i] = q0 + i < n ? count[q0 + i] : 0u;
    zero |= q0 + i < n && c[i] == 0u;
    sum += c[i];
  }
  int64_t at = cta_exclusive(sum, total);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (q0 + i < n) out[q0 + i] = at;
    at += c[i];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
  if (empty && zero) *empty = 1u;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(int64_t *__restrict__ sums, int64_t tiles,
                                                            int64_t *__restrict__ grand) {
  int64_t carry = 0;
  for (int64_t base = 0; base < tiles; base += kScanThreads) {
    const int64_t q = base + threadIdx.x;
    int64_t total;
    const int64_t v = q < tiles ? sums[q] : 0;
    const int64_t at = cta_exclusive(v, total);
    if (q < tiles) sums[q] = carry + at;
    carry += total;
  }
  if (threadIdx.x == 0) *grand = carry;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(int64_t *__restrict__ out, int64_t n,
                                                           const int64_t *__restrict__ sums) {
  const int64_t q0 = (int64_t)blockIdx.x * kScanTile, add = sums[blockIdx.x];
  for (int64_t q = q0 + threadIdx.x; q < min(n, q0 + kScanTile); q += kScanThreads) out[q] += add;
}

// The B-splines over element e out of all of them, by a warp: their number, and
// with FILL their indices from list[0] on, in ascending order.
template <bool FILL>
__device__ __forceinline__ int64_t pairs_of_element(const double *__restrict__ box, int64_t e,
                                                    const double *__restrict__ knots, int64_t n_basis, int p0, int p1,
                                                    int p2, int kw, int32_t *__restrict__ list) {
  const int lane = threadIdx.x & 31, off[3] = {0, p0 + 2, p0 + p1 + 4}, deg[3] = {p0, p1, p2};
  int64_t lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = order_key_01(box[6 * e + a]);
    hi[a] = order_key_01(box[6 * e + 3 + a]);
  }
  constexpr int U = 4;   // B-splines a lane has under way
  int64_t n = 0;
  for (int64_t i0 = 0; i0 < n_basis; i0 += 32 * U) {
    bool in[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + 32 * u + lane;
      const double *k = knots + min(i, n_basis - 1) * kw;
      in[u] = i < n_basis;
#pragma unroll
      for (int a = 0; a < 3; ++a)
        in[u] &= order_key(__ldg(k + off[a])) <= lo[a] && hi[a] <= order_key(__ldg(k + off[a] + deg[a] + 1));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned m = __ballot_sync(0xffffffffu, in[u]);
      if constexpr (FILL) {
        if (in[u]) list[n + __popc(m & ((1u << lane) - 1u))] = (int32_t)(i0 + 32 * u + lane);
      }
      n += __popc(m);
    }
  }
  return n;
}

// Incidence of a small volume, a warp an element.  FILL false: ptr[e] = the
// length of e's list; FILL true: the lists from ptr[e] on.
template <bool FILL>
__global__ void __launch_bounds__(32 * kSetupWarps) k_incident_direct(const double *__restrict__ box, int64_t n_elem,
                                                                     const double *__restrict__ knots, int64_t n_basis,
                                                                     int p0, int p1, int p2, int kw,
                                                                     int64_t *__restrict__ ptr, int32_t *__restrict__ list) {
  const int64_t e = (int64_t)blockIdx.x * kSetupWarps + (threadIdx.x >> 5);
  if (e >= n_elem) return;
  const int64_t n = pairs_of_element<FILL>(box, e, knots, n_basis, p0, p1, p2, kw, FILL ? list + ptr[e] : nullptr);
  if (!FILL && (threadIdx.x & 31) == 0) ptr[e] = n;
}

// ptr: lengths to offsets in place, the total in ptr[n] and in ptr[n + 1]
// whether a length is 0.  One CTA.
__global__ void __launch_bounds__(kScanThreads) k_scan_direct(int64_t *__restrict__ ptr, int64_t n) {
  int64_t carry = 0;
  int empty = 0;
  for (int64_t base = 0; base < n; base += kScanThreads) {
    const int64_t q = base + threadIdx.x, v = q < n ? ptr[q] : 0;
    int64_t total;
    const int64_t at = cta_exclusive(v, total);
    empty |= q < n && v == 0;
    if (q < n) ptr[q] = carry + at;
    carry += total;
  }
  empty = __syncthreads_or(empty);
  if (threadIdx.x == 0) {
    ptr[n] = carry;
    ptr[n + 1] = empty;
  }
}

// The same three steps in one CTA, for at most kSmallElems elements.
constexpr int kSmallElems = 64;

__global__ void __launch_bounds__(1024) k_incident_small(const double *__restrict__ box, int n_elem,
                                                         const double *__restrict__ knots, int n_basis, int p0, int p1,
                                                         int p2, int kw, int64_t *__restrict__ ptr,
                                                         int32_t *__restrict__ list) {
  __shared__ int at[kSmallElems];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int e = w; e < n_elem; e += 32) {
    const int n = (int)pairs_of_element<false>(box, e, knots, n_basis, p0, p1, p2, kw, nullptr);
    if (lane == 0) at[e] = n;
  }
  __syncthreads();
  if (w == 0) {
    int before = 0;
    bool empty = false;
    for (int q = lane; q < kSmallElems; q += 32) {   // every lane takes both turns
      const int v = q < n_elem ? at[q] : 0;
      int inc = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      empty |= q < n_elem && v == 0;
      if (q < n_elem) ptr[q] = at[q] = before + inc - v;
      before += __shfl_sync(0xffffffffu, inc, 31);
    }
    empty = __any_sync(0xffffffffu, empty);
    if (lane == 0) {
      ptr[n_elem] = before;
      ptr[n_elem + 1] = empty;
    }
  }
  __syncthreads();
  for (int e = w; e < n_elem; e += 32) pairs_of_element<true>(box, e, knots, n_basis, p0, p1, p2, kw, list + at[e]);
}

cudaError_t exclusive_scan(const uint32_t *count, int64_t n, int64_t *out, int64_t *sums, uint32_t *empty,
                           cudaStream_t s) {
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  k_scan_tiles<<<(unsigned)tiles, kScanThreads, 0, s>>>(count, n, out, sums, empty);
  k_scan_sums<<<1, kScanThreads, 0, s>>>(sums, tiles, out + n);
  k_scan_add<<<(unsigned)tiles, kScanThreads, 0, s>>>(out, n, sums);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// change of basis (FP64)
// ----------------------------------------------------------------------------

// Bernstein coefficients over [a, b] of the univariate B-spline on knots
// xi[0..p+1], where [a, b] lies in one knot span.  beta_j is the blossom
// B(a,..,a, b,..,b) with j arguments b, evaluated by the de Boor triangle of
// the span restricted to its non-zero entries (only the B-spline itself has
// coefficient 1), so every denominator is a positive knot difference.
__device__ void bernstein_of_bspline(const double *xi, int p, double a, double b, double *beta) {
  int m = 0;
  for (int q = 1; q <= p; ++q)
    if (xi[q] <= a) m = q;
  // the triangle's denominators depend on (r, k) only: one FP64 division
  // each (FP64 division is a long instruction sequence on GB300), reused for
  // all p + 1 blossoms
  double inv[kMaxDeg + 1][kMaxDeg + 1];
  for (int r = 1; r <= p; ++r) {
    const int khi = m < r ? m : r;
    const int klo = (m - p + r) > 0 ? (m - p + r) : 0;
    for (int k = khi; k >= klo; --k) inv[r][k] = 1.0 / (xi[k + p + 1 - r] - xi[k]);
  }
  for (int j = 0; j <= p; ++j) {
    double D[kMaxDeg + 1];
    D[0] = 1.0;
    for (int q = 1; q <= p; ++q) D[q] = 0.0;
    for (int r = 1; r <= p; ++r) {
      const double t = (r <= p - j) ? a : b;
      const int khi = m < r ? m : r;
      const int klo = (m - p + r) > 0 ? (m - p + r) : 0;
      for (int k = khi; k >= klo; --k) {
        const double alpha = (t - xi[k]) * inv[r][k];
        const double prev = k > 0 ? D[k - 1] : 0.0;
        D[k] = (1.0 - alpha) * prev + alpha * D[k];
      }
    }
    beta[j] = D[m];
  }
}

// C(n, k) in integer arithmetic (each partial product is itself a binomial,
// so every division is exact)
__device__ __forceinline__ int binomial(int n, int k) {
  int b = 1;
  for (int i = 1; i <= k; ++i) b = b * (n - k + i) / i;
  return b;
}

constexpr int kBezWarps = 4;
constexpr int kChunk = 32;

// Any degrees; one warp per element (of the n_list listed ones, or of all with
// no list); lane l owns coefficients q = l, l+32, ... of the (p0+1)(p1+1)(p2+1)
// block, for every component.
__global__ void __launch_bounds__(32 * kBezWarps) k_to_bezier(
    const double *__restrict__ box, const double *__restrict__ knots, const double *__restrict__ coef,
    const double *__restrict__ weight, const int64_t *__restrict__ inc_ptr, const int32_t *__restrict__ inc_idx,
    int p0, int p1, int p2, int nc, int kw, int64_t n_elem, double *__restrict__ out64,
    const int32_t *__restrict__ list, const uint32_t *__restrict__ n_list) {
  __shared__ double sb[kBezWarps][kChunk][3 * (kMaxDeg + 1)];
  __shared__ double sg[kBezWarps][kChunk][3];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t at = (int64_t)blockIdx.x * kBezWarps + w; at < (list ? (int64_t)*n_list : n_elem);
       at += (int64_t)gridDim.x * kBezWarps) {
    const int64_t e = list ? list[at] : at;
    const int n0 = p0 + 1, n1 = p1 + 1, n2 = p2 + 1;
    const int nb = n0 * n1 * n2;
    const int deg[3] = {p0, p1, p2};
    const int off[3] = {0, p0 + 2, p0 + p1 + 4};
    double acc[4][3];
    for (int r = 0; r < 4; ++r)
      for (int c = 0; c < 3; ++c) acc[r][c] = 0.0;
    const double *eb = box + 6 * e;
    const int64_t beg = inc_ptr[e], end = inc_ptr[e + 1];
    for (int64_t base = beg; base < end; base += kChunk) {
      const int cnt = (int)min((int64_t)kChunk, end - base);
      if (lane < cnt) {
        const int32_t i = inc_idx[base + lane];
        for (int a = 0; a < 3; ++a) {
          double xi[kMaxDeg + 2];
          for (int q = 0; q <= deg[a] + 1; ++q) xi[q] = knots[(int64_t)i * kw + off[a] + q];
          bernstein_of_bspline(xi, deg[a], eb[a], eb[3 + a], &sb[w][lane][a * (kMaxDeg + 1)]);
        }
        for (int c = 0; c < nc; ++c) sg[w][lane][c] = weight[i] * coef[(int64_t)i * nc + c];
      }
      __syncwarp();
      for (int s = 0; s < cnt; ++s) {
        const double *bs = sb[w][s];
        for (int r = 0; r < 4; ++r) {
          const int q = lane + 32 * r;
          if (q < nb) {
            const int ix = q % n0, iy = (q / n0) % n1, iz = q / (n0 * n1);
            const double prod = bs[ix] * bs[(kMaxDeg + 1) + iy] * bs[2 * (kMaxDeg + 1) + iz];
            for (int c = 0; c < nc; ++c) acc[r][c] += sg[w][s][c] * prod;
          }
        }
      }
      __syncwarp();
    }
    for (int r = 0; r < 4; ++r) {
      const int q = lane + 32 * r;
      if (q < nb)
        for (int c = 0; c < nc; ++c) out64[(e * nc + c) * nb + q] = acc[r][c];
    }
  }
}

// The same factor with the degree known.  With i = m - k the triangle's level r
// has entries i = 0 .. P - r, whatever m; entries outside the B-spline stay 0,
// so their knots only have to be finite and distinct.  The P + 1 blossoms share
// their leading levels at a: 16 instead of 24 entries for P = 3.
template <int P>
__device__ __forceinline__ void factor(const double *__restrict__ xi, double a, double b, double *beta) {
  int m = 0;
#pragma unroll
  for (int q = 1; q <= P; ++q)
    if (xi[q] <= a) m = q;
  double tau[2 * P];   // xi[m - P + 1 .. m + P]
#pragma unroll
  for (int s = 0; s < 2 * P; ++s) {
    const int q = m - P + 1 + s;
    const double x = xi[min(max(q, 0), P + 1)];
    tau[s] = q < 0 ? x + (double)(q - 1) : (q > P + 1 ? x + (double)q : x);
  }
  double inv[P + 1][P];
#pragma unroll
  for (int r = 1; r <= P; ++r)
#pragma unroll
    for (int i = 0; i <= P - r; ++i) inv[r][i] = 1.0 / (tau[2 * P - i - r] - tau[P - 1 - i]);
  double A[P + 1];     // the triangle after j levels at a
#pragma unroll
  for (int i = 0; i <= P; ++i) A[i] = i == m ? 1.0 : 0.0;
#pragma unroll
  for (int j = 0; j <= P; ++j) {   // A holds j levels at a: the other P - j at b give the blossom with P - j arguments b
    double D[P + 1];
#pragma unroll
    for (int i = 0; i <= P - j; ++i) D[i] = A[i];
#pragma unroll
    for (int r = j + 1; r <= P; ++r)
#pragma unroll
      for (int i = 0; i <= P - r; ++i) {
        const double alpha = (b - tau[P - 1 - i]) * inv[r][i];
        D[i] = (1.0 - alpha) * D[i + 1] + alpha * D[i];
      }
    beta[P - j] = D[0];
    if (j < P) {
#pragma unroll
      for (int i = 0; i <= P - j - 1; ++i) {
        const double alpha = (a - tau[P - 1 - i]) * inv[j + 1][i];
        A[i] = (1.0 - alpha) * A[i + 1] + alpha * A[i];
      }
    }
  }
}

// k_to_bezier for equal degrees.  FP64 runs at 1/64 of the FP32 rate here, an
// instruction costing the same whatever number of lanes is active, and the
// B-splines over an element share their univariate factors (about 20 different
// ones over the three axes among 66 B-splines).  So the warp first finds the
// different local knot vectors of each axis, by bits, computes each factor
// once, a lane a factor, and then adds the products of the listed factors.
// A list of more than kListMax B-splines, or with more than 32 different knot
// vectors on an axis, is left to the general kernel (todo, n_todo).
// 179,768 tricubic elements (11.8 M pairs) take 4.74 ms, 13.8 with a factor of
// every pair and axis computed anew; 388,016 triquadratic 3-vector elements 4.20.
// The products and sums keep the general kernel's order: contracting a table of
// the coefficients one axis after the other takes 2.49 and 2.39 ms, but moves the
// blocks' last bits, and where |v| is constant over an element those decide the
// bins of its features.
constexpr int kListMax = 128;

template <int P, int NC>
__global__ void __launch_bounds__(32 * kBezWarps) k_to_bezier_shared(
    const double *__restrict__ box, const double *__restrict__ knots, const double *__restrict__ coef,
    const double *__restrict__ weight, const int64_t *__restrict__ inc_ptr, const int32_t *__restrict__ inc_idx,
    int64_t n_elem, double *__restrict__ out64, int32_t *__restrict__ todo, uint32_t *__restrict__ n_todo) {
  constexpr int N = P + 1, NB = N * N * N, R = (NB + 31) / 32, K = P + 2, KW = 3 * K;
  constexpr unsigned kAll = 0xffffffffu;
  __shared__ double s_fac[kBezWarps][3][32][N];
  __shared__ double s_g[kBezWarps][NC][kListMax];
  __shared__ uint32_t s_ids[kBezWarps][kListMax];
  __shared__ int32_t s_rep[kBezWarps][3][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t e = (int64_t)blockIdx.x * kBezWarps + w;
  if (e >= n_elem) return;
  const int64_t beg = inc_ptr[e];
  const int L = (int)min(inc_ptr[e + 1] - beg, (int64_t)kListMax + 1);
  int nd[3] = {0, 0, 0};
  bool fits = L <= kListMax;
  for (int c = 0; c < L && fits; c += 32) {
    const bool valid = c + lane < L;
    const int32_t i = valid ? inc_idx[beg + c + lane] : 0;
    uint32_t ids = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const long long *mine = reinterpret_cast<const long long *>(knots + (int64_t)i * KW + a * K);
      long long x[K];
#pragma unroll
      for (int q = 0; q < K; ++q) x[q] = __ldg(mine + q);
      auto equals = [&](int32_t other) {
        const long long *o = reinterpret_cast<const long long *>(knots + (int64_t)other * KW + a * K);
        bool same = true;
#pragma unroll
        for (int q = 0; q < K; ++q) same &= x[q] == __ldg(o + q);
        return same;
      };
      int id = -1;
      for (int t = 0; t < nd[a]; ++t) {
        if (equals(s_rep[w][a][t])) id = t;
        if (__all_sync(kAll, id >= 0 || !valid)) break;
      }
      for (unsigned open = __ballot_sync(kAll, valid && id < 0); open && fits; open = __ballot_sync(kAll, valid && id < 0)) {
        if (nd[a] == 32) {
          fits = false;
          break;
        }
        const int32_t rep = __shfl_sync(kAll, i, __ffs(open) - 1);
        if (id < 0 && equals(rep)) id = nd[a];
        if (lane == 0) s_rep[w][a][nd[a]] = rep;
        ++nd[a];
      }
      ids |= (uint32_t)(id & 31) << (8 * a);
      __syncwarp();
    }
    if (valid && fits) {
      s_ids[w][c + lane] = ids;
      const double wt = weight[i];
#pragma unroll
      for (int q = 0; q < NC; ++q) s_g[w][q][c + lane] = wt * coef[(int64_t)i * NC + q];
    }
  }
  if (!fits) {
    if (lane == 0) todo[atomicAdd(n_todo, 1u)] = (int32_t)e;
    return;
  }
  const double *eb = box + 6 * e;
  for (int d = lane; d < nd[0] + nd[1] + nd[2]; d += 32) {
    const int a = d < nd[0] ? 0 : (d < nd[0] + nd[1] ? 1 : 2);
    const int t = d - (a > 0 ? nd[0] : 0) - (a > 1 ? nd[1] : 0);
    double beta[N];
    factor<P>(knots + (int64_t)s_rep[w][a][t] * KW + a * K, eb[a], eb[3 + a], beta);
#pragma unroll
    for (int q = 0; q < N; ++q) s_fac[w][a][t][q] = beta[q];
  }
  __syncwarp();
  double acc[R][NC];
  int ix[R], iy[R], iz[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int q = min(lane + 32 * r, NB - 1);
    ix[r] = q % N;
    iy[r] = (q / N) % N;
    iz[r] = q / (N * N);
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[r][c] = 0.0;
  }
#pragma unroll 2
  for (int s = 0; s < L; ++s) {
    const uint32_t ids = s_ids[w][s];
    const double *fx = s_fac[w][0][ids & 255u], *fy = s_fac[w][1][(ids >> 8) & 255u], *fz = s_fac[w][2][ids >> 16];
    double xy = fx[ix[0]] * fy[iy[0]];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (N != 4 && r > 0) xy = fx[ix[r]] * fy[iy[r]];   // N = 4: the lane's coefficients differ in z only
      const double prod = xy * fz[iz[r]];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[r][c] = fma(s_g[w][c][s], prod, acc[r][c]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (lane + 32 * r < NB)
#pragma unroll
      for (int c = 0; c < NC; ++c) out64[(e * NC + c) * NB + lane + 32 * r] = acc[r][c];
}

// Render copy of the FP64 blocks (layout and storage in lrvol_internal.h):
// binomials folded in; for 16-bit storage a per-element, per-component offset
// o = (max+min)/2 and scale s = (max-min)/2 of the FP64 coefficients, and
// q' = binomial*(c - o)/s rounded once from FP64.  One warp per element.  Bound by
// FP64 operations (16 cycles of an SM each), so the range is found on integers:
// 179,768 tricubic elements, FP32 187 us (291 with FP64 minima and maxima),
// FP16 378 (549), of which the division is most.
__device__ __forceinline__ void store_slot(unsigned char *base, int storage, int slot, double x) {
  if (storage == LRVOL_STORE_F32) {
    reinterpret_cast<float *>(base)[slot] = (float)x;
  } else if (storage == LRVOL_STORE_F16) {
    reinterpret_cast<__half *>(base + kHeaderBytes)[slot] = __double2half(x);
  } else {
    reinterpret_cast<__nv_bfloat16 *>(base + kHeaderBytes)[slot] = __double2bfloat16(x);
  }
}

__global__ void __launch_bounds__(32 * kBezWarps) k_pack(const double *__restrict__ b64, int p0, int p1, int p2, int nc,
                                                        int64_t n_elem, int storage, unsigned char *__restrict__ out,
                                                        int ebytes, unsigned char *__restrict__ outc, int ecbytes,
                                                        float2 *__restrict__ range) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t e = (int64_t)blockIdx.x * kBezWarps + w;
  if (e >= n_elem) return;
  const int n0 = p0 + 1, n1 = p1 + 1, nb = n0 * n1 * (p2 + 1);
  const double *be = b64 + e * nc * nb;
  double o[3] = {0.0, 0.0, 0.0}, sc[3] = {1.0, 1.0, 1.0};
  for (int c = 0; c < nc; ++c) {
    // coefficient range (the block's convex hull bounds the field on the element)
    constexpr int64_t kInf = 0x7ff0000000000000ll;
    int64_t kmn = kInf, kmx = kInf ^ INT64_MIN ^ INT64_MAX;   // inf and -inf
    for (int q = lane; q < nb; q += 32) {
      const double x = be[c * nb + q];
      if (order_key_01(x) <= kInf) {   // no NaN
        kmn = min(kmn, order_key(x));
        kmx = max(kmx, order_key(x));
      }
    }
    for (int off = 16; off > 0; off >>= 1) {
      kmn = min(kmn, __shfl_xor_sync(0xffffffffu, kmn, off));
      kmx = max(kmx, __shfl_xor_sync(0xffffffffu, kmx, off));
    }
    const double mn = from_order_key(kmn), mx = from_order_key(kmx);
    if (lane == 0) range[e * nc + c] = make_float2(__double2float_rd(mn), __double2float_ru(mx));
    if (storage != LRVOL_STORE_F32) {
      o[c] = 0.5 * (mx + mn);
      sc[c] = 0.5 * (mx - mn);
      if (!(sc[c] > 0.0)) sc[c] = 1.0;
    }
  }
  if (storage != LRVOL_STORE_F32) {
    if (lane < 8) {
      const float hv = lane < 3 ? (float)o[lane] : (lane < 6 ? (float)sc[lane - 3] : 0.f);
      reinterpret_cast<float *>(out + e * ebytes)[lane] = hv;
      if (outc) reinterpret_cast<float *>(outc + e * ecbytes)[lane] = hv;
    }
  }
  for (int q = lane; q < nb; q += 32) {
    const int ix = q % n0, iy = (q / n0) % n1, iz = q / (n0 * n1);
    const double binom = (double)(binomial(p0, ix) * binomial(p1, iy) * binomial(p2, iz));
    for (int c = 0; c < nc; ++c) {
      const double b = be[c * nb + q];
      const double x = storage == LRVOL_STORE_F32 ? binom * b : binom * (b - o[c]) / sc[c];
      store_slot(out + e * ebytes, storage, render_slot(nc, n0, nb, iz * n1 + iy, ix, c), x);
      if (outc) store_slot(outc + e * ecbytes, storage, c * roundup8(nb) + q, x);
    }
  }
}

__global__ void k_elem_records(const double *__restrict__ box, int64_t n_elem, int d, ElemRec *__restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_elem) return;
  const double *b = box + 6 * e;
  float lo[3], hi[3], off[3], iw[3];
  double m = b[3] - b[0];
  if (b[4] - b[1] < m) m = b[4] - b[1];
  if (b[5] - b[2] < m) m = b[5] - b[2];
  for (int a = 0; a < 3; ++a) {
    lo[a] = __double2float_ru(b[a]);
    hi[a] = b[3 + a] == 1.0 ? __int_as_float(0x3f800001) : __double2float_ru(b[3 + a]);   // the float after 1
    const double inv = 1.0 / (b[3 + a] - b[a]);
    off[a] = (float)(((double)lo[a] - b[a]) * inv);   // (lo_RU - lo) / (hi - lo), in FP64
    iw[a] = (float)inv;
  }
  ElemRec r;
  r.a = make_float4(lo[0], lo[1], lo[2], __double2float_rn(ldexp(m, -d)));
  r.b = make_float4(hi[0], hi[1], hi[2], 0.f);
  r.c = make_float4(off[0], off[1], off[2], 0.f);
  r.d = make_float4(iw[0], iw[1], iw[2], 0.f);
  out[e] = r;
}

}  // namespace

// Scratch of the incidence: one allocation, carved up here.
int64_t Incidence::plan(int64_t n_elem_) {
  n_elem = n_elem_;
  R = std::max(1, std::min((int)std::cbrt((double)n_elem / 4.0), 96));
  const int64_t cells = (int64_t)R * R * R, most = std::max(cells, n_elem);
  int64_t at = 0;
  auto take = [&](int64_t bytes) {
    const int64_t off = at;
    at += (bytes + 255) & ~int64_t(255);
    return off;
  };
  o_ptr = take(8 * (n_elem + 1));
  o_cell_ptr = take(8 * (cells + 1));
  o_sums = take(8 * ((most + kScanTile - 1) / kScanTile));
  o_cell_count = take(4 * cells);
  o_cell_of = take(4 * n_elem);
  o_cell_el = take(4 * n_elem);
  o_cell_ends = take(48 * n_elem);
  o_count = take(4 * n_elem);
  o_empty = take(4);
  return at;
}

cudaError_t Incidence::count(const lrvol_s *v, unsigned char *scratch, cudaStream_t s) {
  base = scratch;
  const CellGrid g = {R};
  const int64_t cells = g.cells();
  cudaError_t e;
  if ((e = cudaMemsetAsync(cell_count(), 0, 4 * cells, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(counts(), 0, 4 * n_elem, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(empty(), 0, 4, s)) != cudaSuccess) return e;
  const unsigned eb = (unsigned)((n_elem + 255) / 256), wb = (unsigned)((v->n_basis + kSetupWarps - 1) / kSetupWarps);
  k_cell_count<<<eb, 256, 0, s>>>(v->d_box, n_elem, g, cell_of(), cell_count());
  if ((e = exclusive_scan(cell_count(), cells, cell_ptr(), sums(), nullptr, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(cell_count(), 0, 4 * cells, s)) != cudaSuccess) return e;
  k_cell_fill<<<eb, 256, 0, s>>>(v->d_box, cell_of(), n_elem, cell_ptr(), cell_count(), cell_el(), cell_ends());
  k_incident<false><<<wb, 32 * kSetupWarps, 0, s>>>(cell_ends(), n_elem, v->d_knots, v->n_basis, v->p[0], v->p[1],
                                                   v->p[2], v->kw, g, cell_ptr(), cell_el(), counts(), nullptr, nullptr);
  if ((e = exclusive_scan(counts(), n_elem, ptr(), sums(), empty(), s)) != cudaSuccess) return e;
  return cudaMemsetAsync(counts(), 0, 4 * n_elem, s);   // from here the fill's cursors
}

cudaError_t Incidence::fill(const lrvol_s *v, int32_t *unsorted, int32_t *list, cudaStream_t s) {
  const unsigned wb = (unsigned)((v->n_basis + kSetupWarps - 1) / kSetupWarps);
  k_incident<true><<<wb, 32 * kSetupWarps, 0, s>>>(cell_ends(), n_elem, v->d_knots, v->n_basis, v->p[0], v->p[1],
                                                  v->p[2], v->kw, CellGrid{R}, cell_ptr(), cell_el(), counts(), ptr(), unsorted);
  int n_bits = 1;
  while (v->n_basis > (int64_t)1 << n_bits) ++n_bits;
  k_sort_lists<<<(unsigned)((n_elem + kSetupWarps - 1) / kSetupWarps), 32 * kSetupWarps, 0, s>>>(ptr(), n_elem, n_bits,
                                                                                              unsorted, list);
  return cudaGetLastError();
}

// Pair by pair: one CTA's kernel while a warp has one or two elements and a load
// round for each, then a warp an element over the GPU, counted (fill false) and filled.
bool incidence_small(const lrvol_s *v) { return v->n_elem <= kSmallElems && v->n_basis <= 8192 / v->n_elem; }

cudaError_t launch_incidence_direct(const lrvol_s *v, bool fill, cudaStream_t s) {
  const unsigned blocks = (unsigned)((v->n_elem + kSetupWarps - 1) / kSetupWarps);
  if (fill) {
    if (incidence_small(v))
      k_incident_small<<<1, 1024, 0, s>>>(v->d_box, (int)v->n_elem, v->d_knots, (int)v->n_basis, v->p[0], v->p[1],
                                          v->p[2], v->kw, v->d_inc_ptr, v->d_inc_idx);
    else
      k_incident_direct<true><<<blocks, 32 * kSetupWarps, 0, s>>>(v->d_box, v->n_elem, v->d_knots, v->n_basis, v->p[0],
                                                                 v->p[1], v->p[2], v->kw, v->d_inc_ptr, v->d_inc_idx);
  } else if (!incidence_small(v)) {
    k_incident_direct<false><<<blocks, 32 * kSetupWarps, 0, s>>>(v->d_box, v->n_elem, v->d_knots, v->n_basis, v->p[0],
                                                                v->p[1], v->p[2], v->kw, v->d_inc_ptr, nullptr);
    k_scan_direct<<<1, kScanThreads, 0, s>>>(v->d_inc_ptr, v->n_elem);
  }
  return cudaGetLastError();
}

template <int P, int NC>
static void launch_shared(const lrvol_s *v, int32_t *todo, uint32_t *n_todo, cudaStream_t s) {
  k_to_bezier_shared<P, NC><<<(unsigned)((v->n_elem + kBezWarps - 1) / kBezWarps), 32 * kBezWarps, 0, s>>>(
      v->d_box, v->d_knots, v->d_coef, v->d_weight, v->d_inc_ptr, v->d_inc_idx, v->n_elem, v->d_bez64, todo, n_todo);
}

// Equal degrees share factors; what that kernel leaves over, and unequal
// degrees, go through the general one.  todo: room for n_elem elements.
cudaError_t launch_to_bezier(const lrvol_s *v, int32_t *todo, uint32_t *n_todo, cudaStream_t s) {
  const bool equal = v->p[0] == v->p[1] && v->p[0] == v->p[2];
  int64_t blocks = (v->n_elem + kBezWarps - 1) / kBezWarps;
  if (equal) {
    cudaError_t e = cudaMemsetAsync(n_todo, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    switch (v->p[0] * 2 + (v->nc == 3)) {
      case 2: launch_shared<1, 1>(v, todo, n_todo, s); break;
      case 3: launch_shared<1, 3>(v, todo, n_todo, s); break;
      case 4: launch_shared<2, 1>(v, todo, n_todo, s); break;
      case 5: launch_shared<2, 3>(v, todo, n_todo, s); break;
      case 6: launch_shared<3, 1>(v, todo, n_todo, s); break;
      case 7: launch_shared<3, 3>(v, todo, n_todo, s); break;
      case 8: launch_shared<4, 1>(v, todo, n_todo, s); break;
      case 9: launch_shared<4, 3>(v, todo, n_todo, s); break;
      default: return cudaErrorInvalidValue;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (v->n_basis <= 32) return e;   // no list that the kernel leaves over
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    blocks = std::min<int64_t>(blocks, 8 * sms);   // usually nothing is left: a grid that strides over the list
  }
  k_to_bezier<<<(unsigned)blocks, 32 * kBezWarps, 0, s>>>(v->d_box, v->d_knots, v->d_coef, v->d_weight, v->d_inc_ptr,
                                                         v->d_inc_idx, v->p[0], v->p[1], v->p[2], v->nc, v->kw,
                                                         v->n_elem, v->d_bez64, equal ? todo : nullptr, n_todo);
  return cudaGetLastError();
}

cudaError_t launch_pack(const lrvol_s *v, cudaStream_t s) {
  const int64_t blocks = (v->n_elem + kBezWarps - 1) / kBezWarps;
  k_pack<<<(unsigned)blocks, 32 * kBezWarps, 0, s>>>(v->d_bez64, v->p[0], v->p[1], v->p[2], v->nc, v->n_elem,
                                                    v->storage, v->d_bez, v->elem_bytes, v->d_bezc, v->elemc_bytes,
                                                    v->d_range);
  return cudaGetLastError();
}

cudaError_t launch_elem_records(const lrvol_s *v, cudaStream_t s) {
  int d = v->p[0];
  if (v->p[1] > d) d = v->p[1];
  if (v->p[2] > d) d = v->p[2];
  k_elem_records<<<(unsigned)((v->n_elem + 255) / 256), 256, 0, s>>>(v->d_box, v->n_elem, d, v->d_elem);
  return cudaGetLastError();
}

}  // namespace lrvol
