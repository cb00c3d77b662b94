// liblrvol host side: the C ABI of lrvol.h, input validation and the k-d forest
// build (Sec. 3.2.1).  Everything else runs in the kernels.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <thread>
#include <vector>

#include "lrvol_internal.h"

using namespace lrvol;

namespace {
thread_local std::string g_last_error;
}  // namespace

namespace lrvol {

int fail(int status, const std::string &msg) {
  g_last_error = msg;
  return status;
}

int cuda_fail(cudaError_t e, const char *what) {
  g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? LRVOL_ERR_OOM : LRVOL_ERR_CUDA;
}

}  // namespace lrvol

namespace {

template <class T>
int dev_alloc(lrvol_s *v, T **p, size_t count, const char *what) {
  if (*p) {   // a rebuild replaces the buffer
    auto it = v->alloc_bytes.find(*p);
    if (it != v->alloc_bytes.end()) {
      v->bytes_device -= it->second;
      v->alloc_bytes.erase(it);
    }
    cudaFree(*p);
    *p = nullptr;
  }
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc((void **)p, count * sizeof(T));
  if (e != cudaSuccess) {
    *p = nullptr;
    return cuda_fail(e, what);
  }
  v->bytes_device += (int64_t)(count * sizeof(T));
  v->alloc_bytes[*p] = (int64_t)(count * sizeof(T));
  return LRVOL_OK;
}

// Scratch of one call.  cudaFree waits for the device, so kernels in flight
// (after an error between launches) are done with it.
struct DeviceBuffer {
  unsigned char *p = nullptr;
  int alloc(int64_t bytes, const char *what) {
    const cudaError_t e = cudaMalloc((void **)&p, (size_t)std::max<int64_t>(bytes, 1));
    if (e == cudaSuccess) return LRVOL_OK;
    p = nullptr;
    return cuda_fail(e, what);
  }
  ~DeviceBuffer() {
    if (p) cudaFree(p);
  }
};

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

// ----------------------------------------------------------------------------
// k-d forest (Sec. 3.2.1).  Split rule (the paper balances depth by counting,
// per direction, the elements on either side of a mean split plane): candidates are the
// element faces strictly inside the node region; per axis the candidate
// nearest to the mean of the candidates; score = max(#left, #right) with
// straddling elements counted on both sides; lowest score wins, ties x<y<z.
// ----------------------------------------------------------------------------
float round_up_f32(double x) {
  float f = (float)x;
  if ((double)f < x) f = std::nextafter(f, INFINITY);
  return f;
}

struct TreeBuilder {
  const lrvol_s *v = nullptr;
  std::vector<Node> nodes;
  bool midpoint = false;       // octree-style splits (LRVOL_SPLIT_MIDPOINT)
  bool unresolved = false;     // a midpoint tree reached kMaxDepth

  const double *box(int32_t e) const { return &v->box[6 * (size_t)e]; }

  // Build a tree over `els` inside region [rlo, rhi); returns a reference.
  uint32_t build(const int32_t *els, size_t n, const double *rlo, const double *rhi, int *maxd) {
    pool.assign(els, els + n);
    return subtree(0, n, rlo, rhi, 0, maxd);
  }

 private:
  // Element lists of the subtrees under way, on one stack: a node puts its
  // children's lists on top and takes them off when both are built.  (4,096
  // elements in one tree, the whole call: 583 us by midpoints and 2,148 balanced
  // with a vector for each list, 349 and 1,698 so.)
  std::vector<int32_t> pool;
  std::vector<double> cand;

  // The elements of pool[beg, end) on either side of the plane t, on top of the
  // pool: the low ones, and from the returned place on the high ones.
  size_t divide(size_t beg, size_t end, int a, double t) {
    size_t to = pool.size();
    pool.resize(to + 2 * (end - beg));
    for (size_t q = beg; q < end; ++q) {
      pool[to] = pool[q];
      to += box(pool[q])[a] < t;
    }
    const size_t mid = to;
    for (size_t q = beg; q < end; ++q) {
      pool[to] = pool[q];
      to += box(pool[q])[3 + a] > t;
    }
    pool.resize(to);
    return mid;
  }

  // The node that splits region [rlo, rhi) at t, its children from the lists on top of the pool.
  uint32_t node(size_t low, size_t mid, int a, double t, const double *rlo, const double *rhi, int d, int *maxd) {
    const uint32_t me = (uint32_t)nodes.size();
    nodes.push_back(Node{0, 0, {0, 0}});
    Node nd;
    const float s = round_up_f32(t);
    std::memcpy(&nd.split_bits, &s, 4);
    nd.axis = (uint32_t)a;
    double lhi[3], hlo[3];
    for (int c = 0; c < 3; ++c) {
      lhi[c] = c == a ? t : rhi[c];
      hlo[c] = c == a ? t : rlo[c];
    }
    const size_t top = pool.size();
    nd.child[0] = subtree(low, mid, rlo, lhi, d + 1, maxd);
    if (nd.child[0] == kNone) return kNone;
    nd.child[1] = subtree(mid, top, hlo, rhi, d + 1, maxd);
    if (nd.child[1] == kNone) return kNone;
    pool.resize(low);
    nodes[me] = nd;
    return me;
  }

  uint32_t subtree(size_t beg, size_t end, const double *rlo, const double *rhi, int d, int *maxd) {
    *maxd = std::max(*maxd, d);
    const size_t n = end - beg;
    if (n == 1) return kLeaf | (uint32_t)pool[beg];
    if (midpoint) return subtree_mid(beg, end, rlo, rhi, d, maxd);
    int best_axis = -1;
    double best_t = 0;
    size_t best_score = SIZE_MAX;
    for (int a = 0; a < 3; ++a) {
      cand.clear();
      for (size_t q = beg; q < end; ++q) {
        const double *b = box(pool[q]);
        if (b[a] > rlo[a] && b[a] < rhi[a]) cand.push_back(b[a]);
        if (b[3 + a] > rlo[a] && b[3 + a] < rhi[a]) cand.push_back(b[3 + a]);
      }
      if (cand.empty()) continue;
      std::sort(cand.begin(), cand.end());
      cand.erase(std::unique(cand.begin(), cand.end()), cand.end());
      double mean = 0;
      for (double c : cand) mean += c;
      mean /= (double)cand.size();
      double t = cand[0];
      for (double c : cand)
        if (std::fabs(c - mean) < std::fabs(t - mean)) t = c;
      size_t nl = 0, nr = 0;
      for (size_t q = beg; q < end; ++q) {
        const double *b = box(pool[q]);
        nl += b[a] < t;
        nr += b[3 + a] > t;
      }
      size_t score = std::max(nl, nr);
      if (score < best_score) {
        best_score = score;
        best_axis = a;
        best_t = t;
      }
    }
    if (best_axis < 0) return kNone;  // cannot happen for a valid box partition
    const size_t low = pool.size(), mid = divide(beg, end, best_axis, best_t), nl = mid - low, nr = pool.size() - mid;
    if (nl >= n || nr >= n || nl == 0 || nr == 0) return kNone;
    return node(low, mid, best_axis, best_t, rlo, rhi, d, maxd);
  }

  // Octree-style tree: the region's midpoint on axes x, y, z in turn (three
  // binary levels make one octree level).  An element straddling the plane
  // goes to both sides; a leaf is a region that one element covers.  Dyadic
  // faces are reached exactly (midpoints of dyadic regions are dyadic, and
  // exact in FP32 down to 2^-149); a face at a non-dyadic coordinate never
  // is, and the tree is abandoned at kMaxDepth.
  uint32_t subtree_mid(size_t beg, size_t end, const double *rlo, const double *rhi, int d, int *maxd) {
    if (d >= kMaxDepth - 1) {
      unresolved = true;
      return kNone;
    }
    const int a = d % 3;
    const double t = 0.5 * (rlo[a] + rhi[a]);
    const size_t low = pool.size(), mid = divide(beg, end, a, t);
    if (mid == low || mid == pool.size()) return kNone;   // not a box partition
    return node(low, mid, a, t, rlo, rhi, d, maxd);
  }
};

// The trees as the device walks them.  A look-up waits for every node on its
// way, so a subtree whose splits lie on at most three planes per axis, and that
// is at least kGridDepth levels deep, becomes a grid: its planes and the element
// of each of its cells, two dependent reads whatever its depth.  A point is in
// cell c of an axis if it is on the >= side of c planes, which decides every
// split of the subtree as the walk does.
// References while compiling: kLeaf | element; kGridRef | offset into grids;
// else an index into nodes.
constexpr uint32_t kGridRef = 0x40000000u;
constexpr int kGridDepth = 3, kGridPlanes = 3;

struct Compiled {
  std::vector<Node> nodes;
  std::vector<GridUnit> grids;   // per grid three units of planes, then its cells, four to a unit

  // A subtree not yet emitted: its planes and depth (wide: more than kGridPlanes on an axis).
  struct Sub {
    float plane[3][kGridPlanes];
    int n[3], depth;
    bool wide;
    uint32_t ref;                // in the source tree; once wide, in this one
  };

  static void add_plane(Sub &s, int a, float x) {
    if (s.wide) return;
    int k = 0;
    while (k < s.n[a] && s.plane[a][k] < x) ++k;
    if (k < s.n[a] && s.plane[a][k] == x) return;
    if (s.n[a] == kGridPlanes) {
      s.wide = true;
      return;
    }
    for (int q = s.n[a]++; q > k; --q) s.plane[a][q] = s.plane[a][q - 1];
    s.plane[a][k] = x;
  }

  Sub scan(const std::vector<Node> &src, uint32_t ref) {
    Sub s{};
    s.ref = ref;
    if (ref & kLeaf) return s;
    const Node &nd = src[ref];
    Sub c[2] = {scan(src, nd.child[0]), scan(src, nd.child[1])};
    s.wide = c[0].wide || c[1].wide;
    s.depth = 1 + std::max(c[0].depth, c[1].depth);
    float x;
    std::memcpy(&x, &nd.split_bits, 4);
    add_plane(s, (int)nd.axis, x);
    for (const Sub &k : c)
      for (int a = 0; a < 3; ++a)
        for (int q = 0; q < k.n[a]; ++q) add_plane(s, a, k.plane[a][q]);
    if (!s.wide) return s;
    Node out = nd;
    for (int k = 0; k < 2; ++k) out.child[k] = c[k].wide ? c[k].ref : emit(src, c[k]);
    s.ref = (uint32_t)nodes.size();
    nodes.push_back(out);
    return s;
  }

  uint32_t copy(const std::vector<Node> &src, uint32_t ref) {
    if (ref & kLeaf) return ref;
    const uint32_t me = (uint32_t)nodes.size();
    nodes.push_back(src[ref]);
    const uint32_t a = copy(src, src[ref].child[0]), b = copy(src, src[ref].child[1]);
    nodes[me].child[0] = a;
    nodes[me].child[1] = b;
    return me;
  }

  void fill(const std::vector<Node> &src, uint32_t ref, const Sub &s, uint32_t *cells, const int *lo, const int *hi) {
    const int sy = s.n[0] + 1, sz = sy * (s.n[1] + 1);
    if (ref & kLeaf) {
      for (int z = lo[2]; z < hi[2]; ++z)
        for (int y = lo[1]; y < hi[1]; ++y)
          for (int x = lo[0]; x < hi[0]; ++x) cells[z * sz + y * sy + x] = ref;
      return;
    }
    const Node &nd = src[ref];
    const int a = (int)nd.axis;
    float x;
    std::memcpy(&x, &nd.split_bits, 4);
    int k = 0;
    while (s.plane[a][k] != x) ++k;
    int mid[3] = {hi[0], hi[1], hi[2]};
    mid[a] = k + 1;
    fill(src, nd.child[0], s, cells, lo, mid);
    for (int c = 0; c < 3; ++c) mid[c] = lo[c];
    mid[a] = k + 1;
    fill(src, nd.child[1], s, cells, mid, hi);
  }

  uint32_t emit(const std::vector<Node> &src, const Sub &s) {
    if (s.depth < kGridDepth) return copy(src, s.ref);
    const int dim[3] = {s.n[0] + 1, s.n[1] + 1, s.n[2] + 1}, zero[3] = {0, 0, 0};
    const size_t at = grids.size();
    grids.resize(at + 3 + (dim[0] * dim[1] * dim[2] + 3) / 4, GridUnit{{kLeaf, kLeaf, kLeaf, kLeaf}});
    for (int a = 0; a < 3; ++a) {
      for (int q = 0; q < kGridPlanes; ++q) {
        const float x = q < s.n[a] ? s.plane[a][q] : INFINITY;
        std::memcpy(&grids[at + a].w[q], &x, 4);
      }
      grids[at + a].w[3] = a == 0 ? 1 : (a == 1 ? dim[0] : dim[0] * dim[1]);
    }
    fill(src, s.ref, s, grids[at + 3].w, zero, dim);
    return kGridRef | (uint32_t)at;
  }

  // The tree at `ref` of src, compiled; its new reference.
  uint32_t add(const std::vector<Node> &src, uint32_t ref) {
    const Sub s = scan(src, ref);
    return s.wide ? s.ref : emit(src, s);
  }
};

// Threads for work of about `ns` nanoseconds on one.  Starting a thread takes
// the caller 50 us, so k threads finish after ns / k + 50 us (k - 1).  (8 elements
// in 16^3 blocks: 780 us with 15 threads started, 37 with none.)
int threads_for(double ns) {
  const double k = std::sqrt(ns / 50e3);
  if (k < 2) return 1;
  return (int)std::min<double>(k, std::min(16u, std::max(1u, std::thread::hardware_concurrency())));
}

// fn(k) for k = 0 .. n - 1 on up to `n_threads` threads, the caller's among them;
// false if a call returned false or threw.
template <class Fn>
bool parallel_for(int n, int n_threads, Fn fn) {
  std::atomic<int> next{0};
  std::atomic<bool> ok{true};
  auto work = [&]() {
    try {
      for (int k; (k = next.fetch_add(1)) < n;)
        if (!fn(k)) ok = false;
    } catch (...) {
      ok = false;
    }
  };
  std::vector<std::thread> threads;
  const int extra = std::min(n, n_threads) - 1;
  try {
    for (int t = 0; t < extra; ++t) threads.emplace_back(work);
  } catch (...) {   // fewer threads than wanted
  }
  work();
  for (auto &t : threads) t.join();
  return ok;
}

struct ForestBuilder : TreeBuilder {
  std::vector<uint32_t> head;  // as ForestView::head
  std::vector<GridUnit> grids;
  int64_t n_tree_nodes = 0;    // nodes of the trees before subtrees became grids
  std::vector<int32_t> depth;  // per block
  LabelCost cost;              // from the boxes (layers())
  int B[3];

  size_t head_at(int x, int y, int z) const { return ((size_t)z * (B[1] + 1) + y) * (B[0] + 1) + x; }

  // The repeated last layer of each axis.
  void pad_head() {
    for (int z = 0; z < B[2]; ++z)
      for (int y = 0; y < B[1]; ++y) head[head_at(B[0], y, z)] = head[head_at(B[0] - 1, y, z)];
    for (int z = 0; z < B[2]; ++z)
      std::copy_n(head.begin() + head_at(0, B[1] - 1, z), B[0] + 1, head.begin() + head_at(0, B[1], z));
    std::copy_n(head.begin() + head_at(0, 0, B[2] - 1), head_at(0, 0, 1), head.begin() + head_at(0, 0, B[2]));
  }

  // The forest by layers of blocks: each element is painted over the blocks it
  // meets, a block that one element meets names it, and the others get their
  // trees.  Layers (runs of consecutive blocks) are independent and run on
  // several threads where the work is worth their start; their nodes follow one
  // another in the blocks' order, however many layers there are.  Gives the trees of region(), and false
  // wherever a block meets no element or a tree fails: region() then decides
  // (it accepts some meshes with gaps, and names the error).  Also false, before
  // anything is painted, where the boxes' volumes add up to more than the cube's
  // or the elements meet far more blocks than a partition has reason to: region()
  // goes depth first and finds the fault of overlapping boxes in its first block
  // (8,000 boxes that all cover the cube, 64^3 blocks: 1 ms; painted, 4.4 s and
  // 1.2 GB), and what layers() keeps stays within 64 MB and 64 bytes a block and
  // element.  (1,000 sheets across 64^3 blocks are 4.4 M meetings, 16 a block.)
  // The whole call, 174,000 elements in 64^3 blocks (no trees): 18.8 ms by region(),
  // 1.9 ms so; 388,016 elements and 562,882 nodes: 144 and 11.3 ms.
  bool layers() {
    const int64_t N = v->n_elem;
    struct Range {
      uint16_t lo[3], hi[3];   // blocks the element meets, [lo, hi)
    };
    std::vector<Range> range((size_t)N);
    const int64_t part = 16384;
    const int n_parts = (int)((N + part - 1) / part);
    struct Sums {
      double volume = 0, visits = 0;   // of the boxes; blocks that their elements meet
      double surface = 0, steps = 0;   // of the boxes; volume / smallest side
    };
    std::vector<Sums> sums(n_parts);
    if (!parallel_for(n_parts, threads_for(10. * N), [&](int k) {
          for (int64_t e = k * part; e < std::min(N, (k + 1) * part); ++e) {
            const double *b = box((int32_t)e);
            double visits = 1, s[3];
            for (int a = 0; a < 3; ++a) {   // exact: B is a power of two
              range[e].lo[a] = (uint16_t)(int)(b[a] * B[a]);
              range[e].hi[a] = (uint16_t)(int)std::ceil(b[3 + a] * B[a]);
              s[a] = b[3 + a] - b[a];
              visits *= range[e].hi[a] - range[e].lo[a];
            }
            sums[k].volume += s[0] * s[1] * s[2];
            sums[k].surface += 2 * (s[0] * s[1] + s[1] * s[2] + s[0] * s[2]);
            sums[k].steps += std::max({s[1] * s[2], s[0] * s[2], s[0] * s[1]});
            sums[k].visits += visits;
          }
          return true;
        }))
      return false;
    Sums all;
    for (const Sums &k : sums) {
      all.volume += k.volume;
      all.visits += k.visits;
      all.surface += k.surface;
      all.steps += k.steps;
    }
    cost.chord = 4 * all.volume / all.surface;   // a random line's mean chord of a convex body is 4 V / S
    cost.ds = std::ldexp(all.volume / all.steps, -std::max({v->p[0], v->p[1], v->p[2]}));
    // a partition's volumes add up to 1, rounded five times each and once a sum (2^-53 relative)
    if (all.volume > 1 + (N + 8) * 0x1p-52 || all.visits > 0x1p24 + 16. * ((double)N + (double)depth.size()))
      return false;
    // about: 1 ns a block, 1.5 a meeting, and 400 (or 100, by midpoints) for an element in a tree
    const int64_t n_blocks = (int64_t)depth.size(), plane = (int64_t)B[0] * B[1];
    const int n_threads = threads_for(1. * n_blocks + 1.5 * all.visits +
                                      std::max(0., all.visits - (double)n_blocks) * (midpoint ? 100. : 400.));
    const int n_slabs = n_threads == 1 ? 1 : (int)std::min<int64_t>(n_blocks, 4 * n_threads);
    std::vector<Compiled> slab(n_slabs);
    std::vector<int64_t> slab_nodes(n_slabs, 0);                      // of the trees as built
    std::vector<std::vector<int64_t>> slab_trees(n_slabs);            // blocks with a tree, as offsets into `depth`
    auto at = [&](int64_t q) { return head_at((int)(q % B[0]), (int)(q / B[0] % B[1]), (int)(q / plane)); };
    if (!parallel_for(n_slabs, n_threads, [&](int s) {
          const int64_t q0 = n_blocks * s / n_slabs, q1 = n_blocks * (s + 1) / n_slabs;
          const int64_t r0 = q0 / B[0], r1 = (q1 - 1) / B[0] + 1;        // its rows of blocks along x
          const int z0 = (int)(q0 / plane), z1 = (int)((q1 - 1) / plane) + 1;
          auto paint = [&](auto block) {   // block(element, offset into depth, into head) for every block of the slab it meets
            for (int64_t e = 0; e < N; ++e) {
              const Range &r = range[e];
              for (int z = std::max<int>(z0, r.lo[2]); z < std::min<int>(z1, r.hi[2]); ++z) {
                const int64_t row = (int64_t)z * B[1], y1 = std::min<int64_t>(r.hi[1], r1 - row);
                for (int64_t y = std::max<int64_t>(r.lo[1], r0 - row); y < y1; ++y) {
                  const int64_t q = (row + y) * B[0], h = (int64_t)head_at(0, (int)y, z);
                  const int64_t x1 = std::min<int64_t>(r.hi[0], q1 - q);
                  for (int64_t x = std::max<int64_t>(r.lo[0], q0 - q); x < x1; ++x) block((int32_t)e, q + x, h + x);
                }
              }
            }
          };
          paint([&](int32_t e, int64_t q, int64_t h) {   // depth counts the elements here
            if (depth[q]++ == 0) head[h] = kLeaf | (uint32_t)e;
          });
          std::vector<int64_t> &trees = slab_trees[s];
          std::vector<size_t> off(1, 0);
          for (int64_t q = q0; q < q1; ++q) {
            if (depth[q] == 0) return false;
            if (depth[q] == 1) {
              depth[q] = 0;
              continue;
            }
            head[at(q)] = (uint32_t)trees.size();
            trees.push_back(q);
            off.push_back(off.back() + depth[q]);
          }
          if (trees.empty()) return true;
          std::vector<int32_t> els(off.back());
          std::vector<size_t> cur(off.begin(), off.end() - 1);
          paint([&](int32_t e, int64_t q, int64_t h) {
            if (depth[q] > 0) els[cur[head[h]]++] = e;
          });
          TreeBuilder tb;
          tb.v = v;
          tb.midpoint = midpoint;
          for (size_t k = 0; k < trees.size(); ++k) {
            tb.nodes.clear();
            const int64_t q = trees[k];
            const int b[3] = {(int)(q % B[0]), (int)(q / B[0] % B[1]), (int)(q / plane)};
            double lo[3], hi[3];
            for (int a = 0; a < 3; ++a) {
              lo[a] = (double)b[a] / B[a];
              hi[a] = (double)(b[a] + 1) / B[a];
            }
            int maxd = 0;
            const uint32_t r = tb.build(&els[off[k]], off[k + 1] - off[k], lo, hi, &maxd);
            if (r == kNone) return false;
            slab_nodes[s] += (int64_t)tb.nodes.size();
            if (slab[s].nodes.size() + tb.nodes.size() >= kGridRef || slab[s].grids.size() >= kGridRef / 2) return false;
            head[at(q)] = slab[s].add(tb.nodes, r);
            depth[q] = maxd;
          }
          return true;
        }))
      return false;
    // the slabs one after the other: nodes, then grids
    size_t n_split = 0, n_units = 0;
    n_tree_nodes = 0;
    for (int s = 0; s < n_slabs; ++s) {
      n_split += slab[s].nodes.size();
      n_units += slab[s].grids.size();
      n_tree_nodes += slab_nodes[s];
    }
    if (n_split + n_units >= kLeaf || n_tree_nodes >= (int64_t)kLeaf) return false;
    nodes.clear();
    nodes.reserve(n_split);
    grids.clear();
    grids.reserve(n_units);
    for (int s = 0; s < n_slabs; ++s) {
      const uint32_t base = (uint32_t)nodes.size(), grid_base = (uint32_t)(n_split + grids.size());
      auto shift = [&](uint32_t r) { return r & kLeaf ? r : (r & kGridRef ? (r & ~kGridRef) + grid_base : r + base); };
      for (Node n : slab[s].nodes) {
        n.child[0] = shift(n.child[0]);
        n.child[1] = shift(n.child[1]);
        nodes.push_back(n);
      }
      for (int64_t q : slab_trees[s]) head[at(q)] = shift(head[at(q)]);
      grids.insert(grids.end(), slab[s].grids.begin(), slab[s].grids.end());
      slab[s] = Compiled();
    }
    return true;
  }

  // region()'s trees as layers() leaves its own (too large a forest stays as
  // built; blocks without an element, kNone, read as leaves here).
  void compile() {
    n_tree_nodes = (int64_t)nodes.size();
    Compiled c;
    std::vector<uint32_t> refs(head.size());
    for (size_t q = 0; q < head.size(); ++q) {
      if (c.nodes.size() + nodes.size() >= kGridRef || c.grids.size() >= kGridRef / 2) return;
      refs[q] = head[q] & kLeaf ? head[q] : c.add(nodes, head[q]);
    }
    const uint32_t base = (uint32_t)c.nodes.size();
    auto shift = [&](uint32_t r) { return !(r & kLeaf) && (r & kGridRef) ? (r & ~kGridRef) + base : r; };
    for (Node &n : c.nodes)
      for (uint32_t &r : n.child) r = shift(r);
    for (size_t q = 0; q < head.size(); ++q) head[q] = shift(refs[q]);
    nodes = std::move(c.nodes);
    grids = std::move(c.grids);
  }

  // Recursive region subdivision over blocks [b0, b1) with the elements meeting it.
  bool region(std::vector<int32_t> &els, const int *b0, const int *b1) {
    if (els.empty()) return false;
    if (els.size() == 1) {
      for (int z = b0[2]; z < b1[2]; ++z)
        for (int y = b0[1]; y < b1[1]; ++y)
          for (int x = b0[0]; x < b1[0]; ++x) {
            head[head_at(x, y, z)] = kLeaf | (uint32_t)els[0];
            depth[((size_t)z * B[1] + y) * B[0] + x] = 0;
          }
      return true;
    }
    int ext[3] = {b1[0] - b0[0], b1[1] - b0[1], b1[2] - b0[2]};
    if (ext[0] == 1 && ext[1] == 1 && ext[2] == 1) {
      double lo[3], hi[3];
      for (int a = 0; a < 3; ++a) {
        lo[a] = (double)b0[a] / B[a];
        hi[a] = (double)b1[a] / B[a];
      }
      int maxd = 0;
      uint32_t r = build(els.data(), els.size(), lo, hi, &maxd);
      if (r == kNone) return false;
      head[head_at(b0[0], b0[1], b0[2])] = r;
      depth[((size_t)b0[2] * B[1] + b0[1]) * B[0] + b0[0]] = maxd;
      return true;
    }
    int a = 0;
    for (int c = 1; c < 3; ++c)
      if (ext[c] > ext[a]) a = c;
    int mid = b0[a] + ext[a] / 2;
    double m = (double)mid / B[a];
    std::vector<int32_t> L, R;
    for (int32_t e : els) {
      const double *b = box(e);
      if (b[a] < m) L.push_back(e);
      if (b[3 + a] > m) R.push_back(e);
    }
    els.clear();
    els.shrink_to_fit();
    int l1[3] = {b1[0], b1[1], b1[2]}, r0[3] = {b0[0], b0[1], b0[2]};
    l1[a] = mid;
    r0[a] = mid;
    return region(L, b0, l1) && region(R, r0, b1);
  }
};

}  // namespace

namespace lrvol {

void camera_consts(const lrvol_camera *c, RayConsts *k) {
  // FP64 camera algebra rounded once to FP32; the order of operations is part
  // of the ray definition in lrvol.h.
  double F[3], R[3], U[3], n;
  for (int a = 0; a < 3; ++a) F[a] = c->target[a] - c->eye[a];
  n = std::sqrt(F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
  for (int a = 0; a < 3; ++a) F[a] = F[a] / n;
  R[0] = F[1] * c->up[2] - F[2] * c->up[1];
  R[1] = F[2] * c->up[0] - F[0] * c->up[2];
  R[2] = F[0] * c->up[1] - F[1] * c->up[0];
  n = std::sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
  for (int a = 0; a < 3; ++a) R[a] = R[a] / n;
  U[0] = R[1] * F[2] - R[2] * F[1];
  U[1] = R[2] * F[0] - R[0] * F[2];
  U[2] = R[0] * F[1] - R[1] * F[0];
  double ty = c->projection == LRVOL_PERSP ? std::tan(0.5 * c->fovy) : 0.5 * c->extent;
  double tx = ty * (double)c->width / (double)c->height;
  for (int a = 0; a < 3; ++a) {
    k->E[a] = (float)c->eye[a];
    k->F[a] = (float)F[a];
    k->R[a] = (float)R[a];
    k->U[a] = (float)U[a];
  }
  k->sxs = (float)(2.0 * tx / (double)c->width);
  k->sxo = (float)(-tx);
  k->sys = (float)(-2.0 * ty / (double)c->height);
  k->syo = (float)ty;
  k->persp = c->projection == LRVOL_PERSP;
}

ForestView forest_view(const lrvol_s *v) {
  ForestView f;
  f.head = v->d_head;
  f.nodes = v->d_nodes;
  f.n_nodes = (uint32_t)v->n_nodes;
  f.grids = reinterpret_cast<const float4 *>(v->d_nodes + v->n_nodes);
  f.n_grid_units = (uint32_t)v->n_grid_units;
  f.head_sy = (uint32_t)v->blocks[0] + 1;
  f.head_sz = f.head_sy * ((uint32_t)v->blocks[1] + 1);
  f.head_bias = 0x4b000000u * (1u + f.head_sy + f.head_sz);
  f.fbx = (float)v->blocks[0];
  f.fby = (float)v->blocks[1];
  f.fbz = (float)v->blocks[2];
  return f;
}

}  // namespace lrvol

namespace lrvol {

// Checks of lrvol_render and the kernel parameters of a frame, except the
// scratch pointers (counters, status), which the caller sets.
int prepare_render(const lrvol_s *v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step,
                   float *rgba_dev, RenderParams *prm, int *field_out) {
  if (!v || !cam || !tf || !step || !rgba_dev) return fail(LRVOL_ERR_ARG, "null pointer");
  if (!v->have_bezier || !v->have_accel) return fail(LRVOL_ERR_STATE, "render needs to_bezier and build_accel");
  if (cam->width < 1 || cam->height < 1 || cam->width > 32768 || cam->height > 32768)
    return fail(LRVOL_ERR_ARG, "bad image size");
  if (cam->projection != LRVOL_ORTHO && cam->projection != LRVOL_PERSP) return fail(LRVOL_ERR_ARG, "bad projection");
  int r0 = cam->row_begin, r1 = cam->row_end;
  if (r0 == 0 && r1 == 0) r1 = cam->height;
  if (r0 < 0 || r1 > cam->height || r0 > r1) return fail(LRVOL_ERR_ARG, "bad row range");
  const int nb = cam->band_count < 1 ? 1 : cam->band_count;
  if (cam->band_count < 0 || cam->band_index < 0 || cam->band_index >= nb)
    return fail(LRVOL_ERR_ARG, "bad interleaved band (need 0 <= band_index < band_count)");
  // rows of this call's first band to the end: none when band_index is past the last band
  const int n_bands = (r1 - r0 + LRVOL_BAND_ROWS - 1) / LRVOL_BAND_ROWS;
  if (cam->band_index >= n_bands) r1 = r0;
  if (step->mode != LRVOL_STEP_FIXED && step->mode != LRVOL_STEP_HEURISTIC && step->mode != LRVOL_STEP_LEARNED)
    return fail(LRVOL_ERR_ARG, "bad step mode");
  if (step->mode == LRVOL_STEP_LEARNED && !step->mult) return fail(LRVOL_ERR_ARG, "learned steps need multipliers");
  if (step->mode == LRVOL_STEP_FIXED && !(step->h > 0)) return fail(LRVOL_ERR_ARG, "fixed step must be > 0");
  if (!(step->xi > 0) || !(tf->vmax > tf->vmin)) return fail(LRVOL_ERR_ARG, "xi and vmax - vmin must be > 0");
  int field = step->field;
  if (field == LRVOL_FIELD_SCALAR && v->nc != 1) return fail(LRVOL_ERR_ARG, "scalar field needs ncomp = 1");
  if (field == LRVOL_FIELD_MAGNITUDE && v->nc != 3) return fail(LRVOL_ERR_ARG, "magnitude needs ncomp = 3");
  if (field == LRVOL_FIELD_COMPONENT && (step->component < 0 || step->component >= v->nc))
    return fail(LRVOL_ERR_ARG, "bad component");
  if (field < 0 || field > 2) return fail(LRVOL_ERR_ARG, "bad field");
  if (v->p[0] != v->p[1] || v->p[0] != v->p[2] || v->p[0] > 3)
    return fail(LRVOL_ERR_UNSUPPORTED, "render needs equal degrees 1..3");
  if (step->shading != LRVOL_SHADE_NONE && step->shading != LRVOL_SHADE_GRADIENT)
    return fail(LRVOL_ERR_ARG, "bad shading");
  if (step->shading == LRVOL_SHADE_GRADIENT && field != LRVOL_FIELD_SCALAR)
    return fail(LRVOL_ERR_UNSUPPORTED, "gradient shading needs a scalar field");
  const double ll = step->light[0] * step->light[0] + step->light[1] * step->light[1] +
                    step->light[2] * step->light[2];
  if (!(ll < INFINITY)) return fail(LRVOL_ERR_ARG, "light must be finite");
  std::memset(prm, 0, sizeof(*prm));
  prm->elem = v->d_elem;
  prm->n_elem = v->n_elem;
  prm->bez = v->d_bez;
  prm->bezc = v->d_bezc;
  prm->comp = field == LRVOL_FIELD_COMPONENT ? step->component : 0;
  prm->forest = forest_view(v);
  prm->out = rgba_dev;
  prm->width = cam->width;
  prm->height = cam->height;
  prm->row_begin = r0;
  prm->row_end = r1;
  prm->band_count = nb;
  prm->band_index = r1 > r0 ? cam->band_index : 0;
  camera_consts(cam, &prm->ray);
  prm->mode = step->mode;
  prm->mult = step->mult;
  prm->h = (float)step->h;
  prm->inv_xi = (float)(1.0 / step->xi);
  prm->alpha_stop = (float)step->alpha_stop;
  prm->tf_scale = (float)(255.0 / (tf->vmax - tf->vmin));
  prm->tf_bias = (float)(-tf->vmin * 255.0 / (tf->vmax - tf->vmin));
  for (int q = 0; q < 256; ++q) prm->tf[q] = make_float4(tf->rgba[q][0], tf->rgba[q][1], tf->rgba[q][2], tf->rgba[q][3]);
  prm->trim = reinterpret_cast<const float2 *>(step->trim);
  if (step->shading == LRVOL_SHADE_GRADIENT) {
    field = kFieldShaded;
    prm->light_set = ll > 0.0;
    for (int a = 0; a < 3; ++a) prm->light[a] = ll > 0.0 ? (float)(step->light[a] / std::sqrt(ll)) : 0.f;
    prm->grad_eps = (float)(1e-3 * (tf->vmax - tf->vmin));
  }
  *field_out = field;
  return LRVOL_OK;
}

// Checks of lrvol_features and its kernel parameters.
int prepare_features(const lrvol_s *v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step,
                     FeatureParams *fp) {
  if (!v || !cam || !tf || !step) return fail(LRVOL_ERR_ARG, "null pointer");
  if (!v->have_bezier) return fail(LRVOL_ERR_STATE, "features need to_bezier");
  if (!(tf->vmax > tf->vmin)) return fail(LRVOL_ERR_ARG, "vmax - vmin must be > 0");
  const int field = step->field;
  if (field < 0 || field > 2 || (field == LRVOL_FIELD_SCALAR && v->nc != 1) ||
      (field == LRVOL_FIELD_MAGNITUDE && v->nc != 3) ||
      (field == LRVOL_FIELD_COMPONENT && (step->component < 0 || step->component >= v->nc)))
    return fail(LRVOL_ERR_ARG, "bad field/component for this volume");
  std::memset(fp, 0, sizeof(*fp));
  fp->box = v->d_box;
  fp->elem = v->d_elem;
  fp->range = v->d_range;
  fp->n_elem = v->n_elem;
  fp->nc = v->nc;
  fp->field = field;
  fp->comp = step->component;
  for (int a = 0; a < 3; ++a) fp->eye[a] = (float)cam->eye[a];
  fp->tf_scale = (float)(255.0 / (tf->vmax - tf->vmin));
  fp->tf_bias = (float)(-tf->vmin * 255.0 / (tf->vmax - tf->vmin));
  for (int q = 0; q < 256; ++q) fp->tf[q] = make_float4(tf->rgba[q][0], tf->rgba[q][1], tf->rgba[q][2], tf->rgba[q][3]);
  return LRVOL_OK;
}

}  // namespace lrvol

extern "C" {

const char *lrvol_status_string(int s) {
  switch (s) {
    case LRVOL_OK: return "ok";
    case LRVOL_ERR_ARG: return "invalid argument";
    case LRVOL_ERR_OOM: return "out of memory";
    case LRVOL_ERR_CUDA: return "CUDA error";
    case LRVOL_ERR_STATE: return "call out of order";
    case LRVOL_ERR_BOUNDS: return "device bounds check failed";
    case LRVOL_ERR_TIMEOUT: return "device wait timed out";
    case LRVOL_ERR_UNSUPPORTED: return "unsupported by this build";
    default: return "unknown status";
  }
}

const char *lrvol_last_error(void) { return g_last_error.c_str(); }

int lrvol_create(const int32_t deg[3], int32_t ncomp, int64_t n_elem, const double *elem_box,
                 int64_t n_basis, const double *knots, const double *coef, const double *weight,
                 lrvol_t *out) {
  if (!deg || !elem_box || !knots || !coef || !weight || !out) return fail(LRVOL_ERR_ARG, "null pointer");
  *out = nullptr;
  if (ncomp != 1 && ncomp != 3) return fail(LRVOL_ERR_ARG, "ncomp must be 1 or 3");
  if (n_elem < 1 || n_elem >= (int64_t)kLeaf || n_basis < 1 || n_basis >= (int64_t)INT32_MAX)
    return fail(LRVOL_ERR_ARG, "bad element or basis count");
  for (int a = 0; a < 3; ++a)
    if (deg[a] < 1 || deg[a] > kMaxDeg) return fail(LRVOL_ERR_ARG, "degree out of range 1..4");
  int kw = deg[0] + deg[1] + deg[2] + 6;
  for (int64_t e = 0; e < n_elem; ++e)
    for (int a = 0; a < 3; ++a) {
      double lo = elem_box[6 * e + a], hi = elem_box[6 * e + 3 + a];
      if (!(lo >= 0.0 && hi <= 1.0 && lo < hi)) return fail(LRVOL_ERR_ARG, "element box outside [0,1] or empty");
    }
  for (int64_t i = 0; i < n_basis; ++i) {
    const double *k = knots + i * kw;
    for (int j = 1; j < kw; ++j) {
      bool axis_start = (j == deg[0] + 2) || (j == deg[0] + deg[1] + 4);
      if (!axis_start && !(k[j] >= k[j - 1])) return fail(LRVOL_ERR_ARG, "knots must be non-decreasing");
    }
    if (!std::isfinite(weight[i])) return fail(LRVOL_ERR_ARG, "non-finite weight");
  }
  int dev = 0;
  CU(cudaGetDevice(&dev), "cudaGetDevice");
  lrvol_s *v = new lrvol_s();
  v->device = dev;
  for (int a = 0; a < 3; ++a) v->p[a] = deg[a];
  v->nc = ncomp;
  v->n_elem = n_elem;
  v->n_basis = n_basis;
  v->kw = kw;
  v->box.assign(elem_box, elem_box + 6 * n_elem);
  int rc;
  if ((rc = dev_alloc(v, &v->d_box, 6 * n_elem, "alloc boxes")) ||
      (rc = dev_alloc(v, &v->d_knots, (size_t)kw * n_basis, "alloc knots")) ||
      (rc = dev_alloc(v, &v->d_coef, (size_t)ncomp * n_basis, "alloc coef")) ||
      (rc = dev_alloc(v, &v->d_weight, n_basis, "alloc weight")) ||
      (rc = dev_alloc(v, &v->d_counters, kNumCounters, "alloc counters")) ||
      (rc = dev_alloc(v, &v->d_status, 1, "alloc status"))) {
    lrvol_destroy(v);
    return rc;
  }
  cudaError_t e = cudaSuccess;
  if (!e) e = cudaMemcpy(v->d_box, elem_box, sizeof(double) * 6 * n_elem, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(v->d_knots, knots, sizeof(double) * kw * n_basis, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(v->d_coef, coef, sizeof(double) * ncomp * n_basis, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemcpy(v->d_weight, weight, sizeof(double) * n_basis, cudaMemcpyHostToDevice);
  if (!e) e = cudaMemset(v->d_counters, 0, sizeof(unsigned long long) * kNumCounters);
  if (!e) e = cudaMemset(v->d_status, 0, sizeof(uint32_t));
  if (e) {
    lrvol_destroy(v);
    return cuda_fail(e, "upload volume");
  }
  *out = v;
  return LRVOL_OK;
}

int lrvol_build_accel(lrvol_t v, const int32_t blocks[3], void *stream) {
  return lrvol_build_accel_split(v, blocks, LRVOL_SPLIT_BALANCED, stream);
}

int lrvol_build_accel_split(lrvol_t v, const int32_t blocks[3], int32_t split, void *stream) {
  if (!v || !blocks) return fail(LRVOL_ERR_ARG, "null pointer");
  if (split != LRVOL_SPLIT_BALANCED && split != LRVOL_SPLIT_MIDPOINT) return fail(LRVOL_ERR_ARG, "bad split rule");
  for (int a = 0; a < 3; ++a)
    if (!is_pow2(blocks[a]) || blocks[a] > 1024) return fail(LRVOL_ERR_ARG, "blocks must be powers of two <= 1024");
  if ((int64_t)blocks[0] * blocks[1] * blocks[2] > (int64_t)1 << 28) return fail(LRVOL_ERR_ARG, "too many blocks");
  ForestBuilder fb;
  fb.v = v;
  fb.midpoint = split == LRVOL_SPLIT_MIDPOINT;
  for (int a = 0; a < 3; ++a) fb.B[a] = blocks[a];
  size_t nblk = (size_t)blocks[0] * blocks[1] * blocks[2];
  fb.head.assign(fb.head_at(0, 0, blocks[2] + 1), kNone);
  fb.depth.assign(nblk, 0);
  if (!fb.layers()) {
    fb.nodes.clear();
    fb.head.assign(fb.head.size(), kNone);
    fb.depth.assign(nblk, 0);
    std::vector<int32_t> all(v->n_elem);
    std::iota(all.begin(), all.end(), 0);
    int b0[3] = {0, 0, 0}, b1[3] = {blocks[0], blocks[1], blocks[2]};
    if (!fb.region(all, b0, b1)) {
      if (fb.unresolved)
        return fail(LRVOL_ERR_UNSUPPORTED, "midpoint splits do not resolve this mesh (faces at non-dyadic coordinates)");
      return fail(LRVOL_ERR_ARG, "elements do not form a box partition of [0,1]^3");
    }
    fb.compile();
  }
  fb.pad_head();
  for (uint32_t h : fb.head)
    if (h == kNone) return fail(LRVOL_ERR_ARG, "a forest block holds no element");
  if (fb.nodes.size() >= kLeaf) return fail(LRVOL_ERR_ARG, "forest too large");
  // depth statistics over blocks
  int64_t s = 0, s2 = 0;
  int dmin = INT32_MAX, dmax = 0;
  for (int32_t d : fb.depth) {
    s += d;
    s2 += (int64_t)d * d;
    dmin = std::min(dmin, d);
    dmax = std::max(dmax, d);
  }
  cudaStream_t st = (cudaStream_t)stream;
  int rc;
  // from here the previous forest is replaced: until the new one is complete
  // the handle has none (a failed host build above left the previous one)
  v->have_accel = false;
  if ((rc = dev_alloc(v, &v->d_head, fb.head.size(), "alloc forest head")) ||
      (rc = dev_alloc(v, &v->d_nodes, fb.nodes.size() + fb.grids.size(), "alloc forest nodes")))
    return rc;
  CU(cudaMemcpyAsync(v->d_head, fb.head.data(), sizeof(uint32_t) * fb.head.size(), cudaMemcpyHostToDevice, st), "upload head");
  if (!fb.nodes.empty())
    CU(cudaMemcpyAsync(v->d_nodes, fb.nodes.data(), sizeof(Node) * fb.nodes.size(), cudaMemcpyHostToDevice, st),
       "upload nodes");
  if (!fb.grids.empty())
    CU(cudaMemcpyAsync(v->d_nodes + fb.nodes.size(), fb.grids.data(), sizeof(GridUnit) * fb.grids.size(),
                       cudaMemcpyHostToDevice, st), "upload grids");
  CU(cudaStreamSynchronize(st), "build_accel sync");  // host vectors go out of scope
  v->label_cost = fb.cost;
  v->n_tree_nodes = fb.n_tree_nodes;
  v->n_nodes = (int64_t)fb.nodes.size();
  v->n_grid_units = (int64_t)fb.grids.size();
  for (int a = 0; a < 3; ++a) v->blocks[a] = blocks[a];
  v->depth_min = dmin;
  v->depth_max = dmax;
  v->depth_mean = (double)s / (double)nblk;
  v->depth_var = std::max(0.0, (double)s2 / (double)nblk - v->depth_mean * v->depth_mean);
  v->have_accel = true;
  return LRVOL_OK;
}

// Pairs of an element and a B-spline up to which lrvol_to_bezier's incidence goes
// pair by pair, and up to which its lists get room for every pair (2^17 integers,
// 512 KB: larger allocations cost more than the wait for the lists' size).
constexpr int64_t kDirectPairs = (int64_t)1 << 20, kRoomPairs = (int64_t)1 << 17;

int lrvol_to_bezier(lrvol_t v, int32_t storage, void *stream) {
  if (!v) return fail(LRVOL_ERR_ARG, "null handle");
  if (storage != LRVOL_STORE_F32 && storage != LRVOL_STORE_F16 && storage != LRVOL_STORE_BF16)
    return fail(LRVOL_ERR_ARG, "bad storage");
  cudaStream_t st = (cudaStream_t)stream;
  int rc;
  // Small volumes go pair by pair of an element and a B-spline: the buckets' scratch
  // and launches take longer (a volume made, with its forest, converted and closed:
  // 8 trilinear elements 251 us through the buckets, 135 so; 512 tricubic ones 384 and
  // 316).  With few pairs the lists get room for all of them and nothing waits for
  // their size.
  const bool direct = v->n_basis <= kDirectPairs / v->n_elem, room = v->n_basis <= kRoomPairs / v->n_elem;
  int64_t size[2] = {0, 0};   // entries of all lists, whether one is empty
  Incidence inc;
  DeviceBuffer scratch, unsorted;
  if (!direct) {
    if ((rc = scratch.alloc(inc.plan(v->n_elem), "alloc incidence scratch"))) return rc;
    CU(inc.count(v, scratch.p, st), "incidence count kernels");
    uint32_t empty = 0;
    CU(cudaMemcpyAsync(size, inc.ptr() + v->n_elem, sizeof size[0], cudaMemcpyDeviceToHost, st), "read incidence size");
    CU(cudaMemcpyAsync(&empty, inc.empty(), sizeof empty, cudaMemcpyDeviceToHost, st), "read incidence check");
    CU(cudaStreamSynchronize(st), "incidence sync");
    if (empty) return fail(LRVOL_ERR_ARG, "an element lies in no B-spline support");
    if ((rc = unsorted.alloc(4 * size[0], "alloc incidence lists"))) return rc;
  }
  const int n0 = v->p[0] + 1, n1 = v->p[1] + 1, n2 = v->p[2] + 1, nb = n0 * n1 * n2;
  v->have_bezier = false;   // the blocks are replaced: none until the new ones are complete
  v->storage = storage;
  v->elem_bytes = elem_bytes(storage, render_slots(v->nc, n0, n1, n2));
  v->elemc_bytes = v->nc == 3 ? elem_bytes(storage, 3 * roundup8(nb)) : 0;
  if ((rc = dev_alloc(v, &v->d_inc_ptr, (size_t)v->n_elem + 2, "alloc incidence ptr"))) return rc;
  if (direct) {
    CU(launch_incidence_direct(v, false, st), "incidence count kernels");
    if (!room) {
      CU(cudaMemcpyAsync(size, v->d_inc_ptr + v->n_elem, sizeof size, cudaMemcpyDeviceToHost, st), "read incidence size");
      CU(cudaStreamSynchronize(st), "incidence sync");
    }
  }
  // the lists, and behind them what k_to_bezier needs besides (the buckets' scratch has that)
  const int64_t entries = room ? v->n_elem * v->n_basis : size[0];
  if ((rc = dev_alloc(v, &v->d_inc_idx, (size_t)(entries + (direct ? v->n_elem + 1 : 0)), "alloc incidence")) ||
      (rc = dev_alloc(v, &v->d_bez64, (size_t)v->n_elem * v->nc * nb, "alloc bezier64")) ||
      (rc = dev_alloc(v, &v->d_bez, (size_t)v->n_elem * v->elem_bytes, "alloc render blocks")) ||
      (v->nc == 3 && (rc = dev_alloc(v, &v->d_bezc, (size_t)v->n_elem * v->elemc_bytes, "alloc render copy"))) ||
      (rc = dev_alloc(v, &v->d_elem, (size_t)v->n_elem, "alloc element records")) ||
      (rc = dev_alloc(v, &v->d_range, (size_t)v->n_elem * v->nc, "alloc coefficient ranges")))
    return rc;
  int32_t *todo = direct ? v->d_inc_idx + entries : inc.cell_of();
  uint32_t *n_todo = direct ? reinterpret_cast<uint32_t *>(todo + v->n_elem) : inc.empty();
  if (direct) {
    CU(launch_incidence_direct(v, true, st), "incidence list kernels");
  } else {
    CU(cudaMemcpyAsync(v->d_inc_ptr, inc.ptr(), sizeof(int64_t) * (v->n_elem + 1), cudaMemcpyDeviceToDevice, st),
       "keep incidence ptr");
    CU(inc.fill(v, reinterpret_cast<int32_t *>(unsorted.p), v->d_inc_idx, st), "incidence list kernels");
  }
  CU(cudaMemsetAsync(v->d_bez, 0, (size_t)v->n_elem * v->elem_bytes, st), "clear render blocks");
  if (v->d_bezc) CU(cudaMemsetAsync(v->d_bezc, 0, (size_t)v->n_elem * v->elemc_bytes, st), "clear render copy");
  CU(launch_to_bezier(v, todo, n_todo, st), "to_bezier kernels");
  CU(launch_pack(v, st), "pack kernel");
  CU(launch_elem_records(v, st), "element record kernel");
  if (room)
    CU(cudaMemcpyAsync(size, v->d_inc_ptr + v->n_elem, sizeof size, cudaMemcpyDeviceToHost, st), "read incidence size");
  CU(cudaStreamSynchronize(st), "to_bezier sync");  // the scratch goes out of scope
  if (size[1]) return fail(LRVOL_ERR_ARG, "an element lies in no B-spline support");
  v->inc_entries = size[0];
  v->have_bezier = true;
  return LRVOL_OK;
}

int lrvol_render(lrvol_t v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step,
                 float *rgba_dev, void *stream) {
  RenderParams prm;
  int field = 0;
  int rc = prepare_render(v, cam, tf, step, rgba_dev, &prm, &field);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  prm.counters = v->d_counters;
  prm.status = v->d_status;
  CU(cudaMemsetAsync(v->d_counters, 0, sizeof(unsigned long long) * kNumCounters, st), "clear counters");
  if (prm.row_end > prm.row_begin) CU(launch_render(prm, v->p[0], field, v->storage, st), "render kernel");
  return LRVOL_OK;
}

// The render kernel's own samples for a list of pixels (parity diagnostic):
// same checks and kernel template as lrvol_render, with the trace compiled in.
int lrvol_render_trace(lrvol_t v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step,
                       const int32_t *pix_dev, int64_t n_pix, int32_t max_samples, float *trace_dev,
                       int32_t *count_dev, float *rgba_dev, void *stream) {
  if (n_pix < 0 || max_samples < 0) return fail(LRVOL_ERR_ARG, "n_pix and max_samples must be >= 0");
  if (n_pix > ((int64_t)1 << 37)) return fail(LRVOL_ERR_ARG, "more than 2^37 pixels");
  if (n_pix > 0 && (!pix_dev || !count_dev || !rgba_dev || (max_samples > 0 && !trace_dev)))
    return fail(LRVOL_ERR_ARG, "null pointer");
  RenderParams prm;
  int field = 0;
  float unused = 0.f;   // prepare_render wants an image pointer; the traced kernel writes none
  int rc = prepare_render(v, cam, tf, step, &unused, &prm, &field);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  prm.counters = v->d_counters;
  prm.status = v->d_status;
  prm.out = nullptr;
  prm.trace_pix = pix_dev;
  prm.trace_n = n_pix;
  prm.trace_max = max_samples;
  prm.trace_rec = reinterpret_cast<float4 *>(trace_dev);
  prm.trace_count = count_dev;
  prm.trace_rgba = reinterpret_cast<float4 *>(rgba_dev);
  CU(cudaMemsetAsync(v->d_counters, 0, sizeof(unsigned long long) * kNumCounters, st), "clear counters");
  CU(launch_render_trace(prm, v->p[0], field, v->storage, st), "render trace kernel");
  return LRVOL_OK;
}

// The allocation-free render: same checks and kernel as lrvol_render, but the
// kernel's scratch (statistics counters, status word) is the library's
// static device array instead of memory of the handle, and nothing is allocated.
int lrvol_render_noalloc(lrvol_t v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step,
                         float *rgba_dev, uint64_t *counters_dev, void *stream) {
  if (cam && (cam->width > kMaxImageSide || cam->height > kMaxImageSide))
    return fail(LRVOL_ERR_ARG, "image size outside 1..32768 x 1..32768, the maximum of lrvol_render_noalloc");
  RenderParams prm;
  int field = 0;
  int rc = prepare_render(v, cam, tf, step, rgba_dev, &prm, &field);
  if (rc) return rc;
  cudaError_t e = launch_render_static(prm, v->p[0], field, v->storage, (cudaStream_t)stream,
                                       reinterpret_cast<unsigned long long *>(counters_dev));
  if (e != cudaSuccess) return cuda_fail(e, "render_noalloc");
  return LRVOL_OK;
}

// ---- learned step sizes ----------------------------------------------------

int lrvol_features(lrvol_t v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step, float *feat,
                   void *stream) {
  if (!feat) return fail(LRVOL_ERR_ARG, "null pointer");
  FeatureParams fp;
  int rc = prepare_features(v, cam, tf, step, &fp);
  if (rc) return rc;
  CU(launch_features(fp, feat, (cudaStream_t)stream), "features kernel");
  return LRVOL_OK;
}

int lrvol_mlp_pack(const float *params, uint16_t *packed, void *stream) {
  if (!params || !packed) return fail(LRVOL_ERR_ARG, "null pointer");
  CU(launch_mlp_pack(params, packed, (cudaStream_t)stream), "mlp pack kernel");
  return LRVOL_OK;
}

int lrvol_mlp_infer(const float *x, int64_t n, const uint16_t *packed, float ymin, float ymax, float *out,
                    void *stream) {
  if (n < 0 || (n > 0 && (!x || !packed || !out))) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!(ymax >= 0.f && ymax <= 8.f)) return fail(LRVOL_ERR_ARG, "ymax must be in [0, 8]");
  if (!(ymin >= -8.f && ymin <= 0.f)) return fail(LRVOL_ERR_ARG, "ymin must be in [-8, 0]");
  if (n == 0) return LRVOL_OK;
  if (reinterpret_cast<uintptr_t>(packed) & 15) return fail(LRVOL_ERR_ARG, "packed weights must be 16-byte aligned");
  uint32_t *status = mlp_status_word();
  if (!status) return fail(LRVOL_ERR_CUDA, "network status word unavailable");
  CU(launch_mlp_infer(x, n, packed, ymin, ymax, out, status, (cudaStream_t)stream), "mlp infer kernel");
  return LRVOL_OK;
}

int lrvol_mlp_infer_timeout_test(const float *x, int64_t n, const uint16_t *packed, float ymin, float ymax,
                                 float *out, void *stream) {
  if (n < 1 || n > ((int64_t)1 << 20) || !x || !packed || !out) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!(ymax >= 0.f && ymax <= 8.f)) return fail(LRVOL_ERR_ARG, "ymax must be in [0, 8]");
  if (!(ymin >= -8.f && ymin <= 0.f)) return fail(LRVOL_ERR_ARG, "ymin must be in [-8, 0]");
  if (reinterpret_cast<uintptr_t>(packed) & 15) return fail(LRVOL_ERR_ARG, "packed weights must be 16-byte aligned");
  uint32_t *status = mlp_status_word();
  if (!status) return fail(LRVOL_ERR_CUDA, "network status word unavailable");
  CU(launch_mlp_infer(x, n, packed, ymin, ymax, out, status, (cudaStream_t)stream, true),
     "mlp infer kernel (timeout test)");
  return LRVOL_OK;
}

int lrvol_mlp_check(void) {
  uint32_t *status = mlp_status_word();
  if (!status) return fail(LRVOL_ERR_CUDA, "network status word unavailable");
  uint32_t h = 0;
  CU(cudaDeviceSynchronize(), "synchronise before the network status");
  CU(cudaMemcpy(&h, status, sizeof h, cudaMemcpyDeviceToHost), "read the network status");
  if (h == 0) return LRVOL_OK;
  CU(cudaMemset(status, 0, sizeof h), "clear the network status");
  return fail(LRVOL_ERR_TIMEOUT, "a tensor-core wait of lrvol_mlp_infer ran out; its rows got multiplier 1");
}

// room for the partial gradients (n x (6*64 + 2)), then one gradient vector
int64_t lrvol_mlp_scratch_floats(int64_t n) { return n < 0 ? 0 : n * (6 * (int64_t)kHid + 2) + kParams; }

static int mlp_gradient(const float *x, const float *target, int64_t n, float *params, float *grad, float *loss,
                        float *scratch, const AdamStep *adam, void *stream) {
  if (!x || !target || !params || !grad || !scratch) return fail(LRVOL_ERR_ARG, "null pointer");
  if (n < 1 || n > ((int64_t)1 << 20)) return fail(LRVOL_ERR_ARG, "batch must be 1 .. 2^20 rows");
  CU(launch_mlp_grad(x, target, n, params, grad, loss, scratch, adam, (cudaStream_t)stream), "mlp training kernels");
  return LRVOL_OK;
}

int lrvol_mlp_grad(const float *x, const float *target, int64_t n, const float *params, float *grad, float *loss,
                   float *scratch, void *stream) {
  // without an Adam step the parameters are only read
  return mlp_gradient(x, target, n, const_cast<float *>(params), grad, loss, scratch, nullptr, stream);
}

int lrvol_mlp_train_step(const float *x, const float *target, int64_t n, float *params, float *m, float *vv,
                         int64_t t, float lr, float *loss, float *scratch, void *stream) {
  if (!m || !vv || t < 1 || !(lr > 0.f)) return fail(LRVOL_ERR_ARG, "bad optimiser arguments");
  if (!scratch) return fail(LRVOL_ERR_ARG, "null pointer");
  // the gradient lands in the last kParams floats of the scratch
  float *grad = scratch + lrvol_mlp_scratch_floats(n) - kParams;
  const AdamStep adam = {m, vv, t, lr};
  return mlp_gradient(x, target, n, params, grad, loss, scratch, &adam, stream);
}

int lrvol_labels(lrvol_t v, const lrvol_camera *cam, const lrvol_tf *tf, const lrvol_step *step, double h_fine,
                 double tau, const float *cand, int32_t n_cand, int32_t *label, void *stream) {
  if (!v || !cam || !tf || !step || !cand || !label) return fail(LRVOL_ERR_ARG, "null pointer");
  if (!v->have_bezier || !v->have_accel) return fail(LRVOL_ERR_STATE, "labels need to_bezier and build_accel");
  if (v->nc != 1 || v->storage != LRVOL_STORE_F32) return fail(LRVOL_ERR_UNSUPPORTED, "labels need a scalar FP32 volume");
  if (v->p[0] != v->p[1] || v->p[0] != v->p[2] || v->p[0] > 3)
    return fail(LRVOL_ERR_UNSUPPORTED, "labels need equal degrees 1..3");
  if (n_cand < 1 || n_cand > 16 || !(h_fine > 0) || !(tau >= 0)) return fail(LRVOL_ERR_ARG, "bad label arguments");
  if (cam->width < 1 || cam->height < 1 || cam->width > 32768 || cam->height > 32768)
    return fail(LRVOL_ERR_ARG, "bad image size");
  if (!(step->xi > 0) || !(tf->vmax > tf->vmin)) return fail(LRVOL_ERR_ARG, "xi and vmax - vmin must be > 0");
  float hc[16];
  static_assert(sizeof(hc) / sizeof(hc[0]) >= 16, "room for the largest candidate list");
  CU(cudaMemcpy(hc, cand, sizeof(float) * n_cand, cudaMemcpyDeviceToHost), "read candidates");
  if (!(hc[0] > 0.f)) return fail(LRVOL_ERR_ARG, "candidates must be positive");
  for (int q = 1; q < n_cand; ++q)
    if (!(hc[q] > hc[q - 1])) return fail(LRVOL_ERR_ARG, "candidates must increase");
  RenderParams prm;
  std::memset(&prm, 0, sizeof(prm));
  prm.elem = v->d_elem;
  prm.n_elem = v->n_elem;
  prm.bez = v->d_bez;
  prm.forest = forest_view(v);
  prm.width = cam->width;
  prm.height = cam->height;
  prm.row_begin = 0;
  prm.row_end = cam->height;
  prm.band_count = 1;
  prm.band_index = 0;
  camera_consts(cam, &prm.ray);
  prm.mode = LRVOL_STEP_HEURISTIC;
  prm.inv_xi = (float)(1.0 / step->xi);
  prm.alpha_stop = (float)step->alpha_stop;
  prm.tf_scale = (float)(255.0 / (tf->vmax - tf->vmin));
  prm.tf_bias = (float)(-tf->vmin * 255.0 / (tf->vmax - tf->vmin));
  prm.counters = v->d_counters;
  prm.status = v->d_status;
  for (int q = 0; q < 256; ++q) prm.tf[q] = make_float4(tf->rgba[q][0], tf->rgba[q][1], tf->rgba[q][2], tf->rgba[q][3]);
  CU(launch_labels(prm, v->p[0], v->label_cost, (float)h_fine, (float)tau, cand, hc, n_cand, label, (cudaStream_t)stream),
     "labels kernel");
  return LRVOL_OK;
}

int lrvol_lookup(lrvol_t v, const float *pts, int64_t n, uint32_t *elem, void *stream) {
  if (!v || (n > 0 && (!pts || !elem)) || n < 0) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!v->have_accel) return fail(LRVOL_ERR_STATE, "lookup needs build_accel");
  if (n == 0) return LRVOL_OK;
  CU(launch_lookup(v, pts, n, elem, (cudaStream_t)stream), "lookup kernel");
  return LRVOL_OK;
}

int lrvol_eval(lrvol_t v, const float *pts, int64_t n, float *val, void *stream) {
  if (!v || (n > 0 && (!pts || !val)) || n < 0) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!v->have_accel || !v->have_bezier) return fail(LRVOL_ERR_STATE, "eval needs build_accel and to_bezier");
  if (n == 0) return LRVOL_OK;
  CU(launch_eval(v, pts, n, val, (cudaStream_t)stream), "eval kernel");
  return LRVOL_OK;
}

int lrvol_eval_grad(lrvol_t v, const float *pts, int64_t n, float *out, void *stream) {
  if (!v || (n > 0 && (!pts || !out)) || n < 0) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!v->have_bezier || !v->have_accel) return fail(LRVOL_ERR_STATE, "eval_grad needs to_bezier and build_accel");
  if (v->nc != 1) return fail(LRVOL_ERR_UNSUPPORTED, "eval_grad needs a scalar volume");
  if (n == 0) return LRVOL_OK;
  CU(launch_eval_grad(v, pts, n, out, (cudaStream_t)stream), "eval_grad kernel");
  return LRVOL_OK;
}

int lrvol_trim(const lrvol_camera *cam, const float *tri, int64_t n_tri, float *out, void *stream) {
  if (!cam || !out || n_tri < 0 || (n_tri > 0 && !tri)) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (cam->width < 1 || cam->height < 1 || cam->width > 32768 || cam->height > 32768)
    return fail(LRVOL_ERR_ARG, "bad image size");
  if (cam->projection != LRVOL_ORTHO && cam->projection != LRVOL_PERSP) return fail(LRVOL_ERR_ARG, "bad projection");
  RayConsts K;
  camera_consts(cam, &K);
  CU(launch_trim(K, cam->width, cam->height, tri, n_tri, out, (cudaStream_t)stream), "trim kernels");
  return LRVOL_OK;
}

int lrvol_streamlines(lrvol_t v, const lrvol_streamline_params *P, const double *seeds, int64_t n, double *out,
                      int32_t *count, int32_t *status, void *stream) {
  if (!v || !P || n < 0 || (n > 0 && (!seeds || !out || !count || !status))) return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!v->have_bezier || !v->have_accel) return fail(LRVOL_ERR_STATE, "streamlines need to_bezier and build_accel");
  if (v->nc != 3) return fail(LRVOL_ERR_UNSUPPORTED, "streamlines need a 3-vector volume");
  if (v->p[0] != v->p[1] || v->p[0] != v->p[2] || v->p[0] > 3)
    return fail(LRVOL_ERR_UNSUPPORTED, "streamlines need equal degrees 1..3");
  if (P->method < LRVOL_RK1 || P->method > LRVOL_RKF45) return fail(LRVOL_ERR_ARG, "bad method");
  if (P->step_rule < LRVOL_SL_FIXED || P->step_rule > LRVOL_SL_ADAPTIVE) return fail(LRVOL_ERR_ARG, "bad step rule");
  if (P->step_rule == LRVOL_SL_ADAPTIVE && P->method < LRVOL_HE)
    return fail(LRVOL_ERR_ARG, "adaptive steps need an embedded pair (HE, BS, RKF45)");
  if (P->step_rule != LRVOL_SL_ADAPTIVE ? !(P->h > 0) : !(P->h >= 0)) return fail(LRVOL_ERR_ARG, "bad step");
  if (!(P->t_end > 0 && P->t_end < INFINITY)) return fail(LRVOL_ERR_ARG, "t_end must be positive and finite");
  if (P->step_rule == LRVOL_SL_ADAPTIVE && !(P->tol > 0)) return fail(LRVOL_ERR_ARG, "tol must be > 0");
  if (P->max_samples < 1) return fail(LRVOL_ERR_ARG, "max_samples must be >= 1");
  if (n == 0) return LRVOL_OK;
  SLParams sp;
  std::memset(&sp, 0, sizeof(sp));
  sp.elem = v->d_elem;
  sp.n_elem = v->n_elem;
  sp.bez = v->d_bez;
  sp.bezc = v->d_bezc;
  sp.forest = forest_view(v);
  sp.status = v->d_status;
  sp.queue = v->d_counters + kCntQueue;
  sp.method = P->method;
  sp.rule = P->step_rule;
  sp.max_samples = P->max_samples;
  sp.h = P->h;
  sp.t_end = P->t_end;
  sp.tol_f = (float)P->tol;
  CU(launch_streamlines(sp, v->p[0], v->storage, seeds, n, out, count, status, (cudaStream_t)stream),
     "streamline kernel");
  return LRVOL_OK;
}

int lrvol_tubes(lrvol_t v, const lrvol_camera *cam, const double *samples, const int32_t *count, int64_t n_lines,
                int32_t max_samples, float radius, const lrvol_tf *cmap, uint64_t *vis, float *rgba, void *stream) {
  if (!v || !cam || !cmap || !vis || !rgba || n_lines < 0 || (n_lines > 0 && (!samples || !count)))
    return fail(LRVOL_ERR_ARG, "bad arguments");
  if (!v->have_bezier || !v->have_accel) return fail(LRVOL_ERR_STATE, "tubes need to_bezier and build_accel");
  if (v->nc != 3) return fail(LRVOL_ERR_UNSUPPORTED, "tubes need a 3-vector volume (speed colouring)");
  if (v->p[0] != v->p[1] || v->p[0] != v->p[2] || v->p[0] > 3)
    return fail(LRVOL_ERR_UNSUPPORTED, "tubes need equal degrees 1..3");
  if (max_samples < 2 || !(radius > 0.f && radius < INFINITY)) return fail(LRVOL_ERR_ARG, "bad max_samples or radius");
  if (n_lines * (int64_t)(max_samples - 1) >= ((int64_t)1 << 32)) return fail(LRVOL_ERR_ARG, "too many segments");
  if (cam->width < 1 || cam->height < 1 || cam->width > 32768 || cam->height > 32768)
    return fail(LRVOL_ERR_ARG, "bad image size");
  if (cam->projection != LRVOL_ORTHO && cam->projection != LRVOL_PERSP) return fail(LRVOL_ERR_ARG, "bad projection");
  if (!(cmap->vmax > cmap->vmin)) return fail(LRVOL_ERR_ARG, "colour map needs vmax > vmin");
  TubeParams tp;
  std::memset(&tp, 0, sizeof(tp));
  tp.field.elem = v->d_elem;
  tp.field.n_elem = v->n_elem;
  tp.field.bez = v->d_bez;
  tp.field.forest = forest_view(v);
  tp.field.status = v->d_status;
  camera_consts(cam, &tp.ray);
  tp.width = cam->width;
  tp.height = cam->height;
  tp.radius = radius;
  tp.samples = samples;
  tp.count = count;
  tp.n_lines = n_lines;
  tp.max_samples = max_samples;
  tp.vis = reinterpret_cast<unsigned long long *>(vis);
  tp.out = rgba;
  tp.tf_scale = (float)(255.0 / (cmap->vmax - cmap->vmin));
  tp.tf_bias = (float)(-cmap->vmin * 255.0 / (cmap->vmax - cmap->vmin));
  for (int q = 0; q < 256; ++q)
    tp.cmap[q] = make_float4(cmap->rgba[q][0], cmap->rgba[q][1], cmap->rgba[q][2], cmap->rgba[q][3]);
  CU(launch_tubes(tp, v->p[0], v->storage, (cudaStream_t)stream), "tube kernels");
  return LRVOL_OK;
}

int lrvol_streamline_error(const double *ref, const int32_t *rc, int32_t rmax, const double *app, const int32_t *ac,
                           int32_t amax, int64_t n, double *sums, void *stream) {
  if (n < 0 || rmax < 1 || amax < 1 || (n > 0 && (!ref || !rc || !app || !ac || !sums)))
    return fail(LRVOL_ERR_ARG, "bad arguments");
  if (n == 0) return LRVOL_OK;
  CU(launch_streamline_error(ref, rc, rmax, app, ac, amax, n, sums, (cudaStream_t)stream), "streamline error kernel");
  return LRVOL_OK;
}

int lrvol_get_bezier(lrvol_t v, double *host_out) {
  if (!v || !host_out) return fail(LRVOL_ERR_ARG, "null pointer");
  if (!v->have_bezier) return fail(LRVOL_ERR_STATE, "get_bezier needs to_bezier");
  size_t nb = (size_t)(v->p[0] + 1) * (v->p[1] + 1) * (v->p[2] + 1);
  CU(cudaDeviceSynchronize(), "sync");
  CU(cudaMemcpy(host_out, v->d_bez64, sizeof(double) * nb * v->nc * v->n_elem, cudaMemcpyDeviceToHost),
     "download bezier");
  return LRVOL_OK;
}

int lrvol_stats(lrvol_t v, lrvol_stats_t *out) {
  if (!v || !out) return fail(LRVOL_ERR_ARG, "null pointer");
  std::memset(out, 0, sizeof(*out));
  out->n_elem = v->n_elem;
  out->n_basis = v->n_basis;
  out->n_nodes = v->n_tree_nodes;
  for (int a = 0; a < 3; ++a) out->blocks[a] = v->blocks[a];
  out->depth_min = v->depth_min;
  out->depth_max = v->depth_max;
  out->depth_mean = v->depth_mean;
  out->depth_var = v->depth_var;
  out->incidence_entries = v->inc_entries;
  out->bytes_device = v->bytes_device;
  CU(cudaDeviceSynchronize(), "sync");
  unsigned long long c[kNumCounters];
  uint32_t status = 0;
  CU(cudaMemcpy(c, v->d_counters, sizeof(c), cudaMemcpyDeviceToHost), "read counters");
  CU(cudaMemcpy(&status, v->d_status, sizeof(status), cudaMemcpyDeviceToHost), "read status");
  out->samples = (int64_t)c[kCntSamples];
  out->lookups = (int64_t)c[kCntLookups];
  out->rays_hit = (int64_t)c[kCntRays];
  if (status == kStatusBounds) return fail(LRVOL_ERR_BOUNDS, "a kernel bounds check tripped");
  if (status == kStatusTimeout) return fail(LRVOL_ERR_TIMEOUT, "a device wait timed out");
  return LRVOL_OK;
}

void lrvol_destroy(lrvol_t v) {
  if (!v) return;
  cudaDeviceSynchronize();
  void *ptrs[] = {v->d_box,   v->d_knots, v->d_coef,  v->d_weight, v->d_inc_ptr,  v->d_inc_idx, v->d_bez64,
                  v->d_bez,   v->d_bezc,  v->d_elem,  v->d_head,  v->d_nodes, v->d_counters, v->d_status,
                  v->d_range};
  for (void *p : ptrs)
    if (p) cudaFree(p);
  delete v;
}

}  // extern "C"
