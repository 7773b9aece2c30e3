// Step III and the on-line phase: hierarchical surpluses and evaluation of the
// sparse-grid interpolant (Section 3.3, Eq. interpo).
//
// The 1-D hierarchical basis a^i_j is the Lagrange polynomial on the CGL set
// X^i that is 1 at its point of dX^i.  It is evaluated in barycentric form
// with the Chebyshev-Lobatto weights w_m = (-1)^m delta_m (delta = 1/2 at the
// two ends), which needs the reciprocals 1/(x - x_m) of the finest set only:
// every coarser X^i is a subset of it.
//
// Distinct 1-D functions are numbered per dimension: id 0 = a^1 (constant),
// then level 2 (points 0 and 1), level 3 (2 points), level 4 (4), ..., so a
// node is a tuple of d ids and its basis function is the product of d table
// entries.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <cstring>
#include <memory>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "diag.cuh"
#include "grid.cuh"
#include "basis.cuh"
#include "interp.cuh"

namespace sg {

// Number of 1-D functions for levels 1..L+1.
int n_functions(int level) {
  int nf = 0;
  for (int l = 1; l <= level + 1; ++l) nf += delta_count(l);
  return nf;
}

int function_id(int l, int kidx) {
  int off = 0;
  for (int m = 1; m < l; ++m) off += delta_count(m);
  const int j = l == 1 ? 0 : (l == 2 ? kidx / 2 : (kidx - 1) / 2);
  return off + j;
}

// The grid's box (lo, then hi - lo), passed by value so that no host copy
// waits for the stream.
struct SurplusBox {
  double v[2 * kMaxDim];
};

// Points of the finest set X^{L+1} on [0, 1]: x_p = (1 - cos(p pi / 2^L)) / 2
// = sin^2(p pi / 2^(L+1)) (Eq. CGL).  The first 2d threads also store the box.
__global__ void k_fine_coords(int level, double* xf, SurplusBox box, int nbox, double* dbox) {
  const int fine_n = 1 << level;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < nbox) dbox[p] = box.v[p];
  if (p > fine_n) return;
  if (level == 0) {
    xf[p] = 0.5;
    return;
  }
  if (p == 0 || p == fine_n || 2 * p == fine_n) {
    xf[p] = p == 0 ? 0.0 : (p == fine_n ? 1.0 : 0.5);   // exact ends and middle
    return;
  }
  const double s = sinpi(static_cast<double>(p) / static_cast<double>(2 * fine_n));
  xf[p] = s * s;
}

// Basis values of every 1-D function at every point of the finest set:
// tab1[id * (fine_n+1) + p].  Used by the surplus build, whose nodes sit on it.
__global__ void k_fine_table(int level, const double* xf, double* tab1) {
  const int fine_n = 1 << level;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p > fine_n) return;
  basis_row(level == 0 ? 0.5 : xf[p], level, xf, tab1 + p, fine_n + 1);
}

// One level of Eq. interpo: for the nodes n in [n0, n1) (all with |i| = s),
// w_n = f_n - sum over coarser nodes m < n0 of phi_m(x_n) w_m.  A warp per
// node n: lane l takes the coarser nodes m = l (mod 32), then the 32 partial
// sums are added by a fixed shuffle tree (the result does not depend on the
// launch).
constexpr int kSurpWarps = 4;
template <int KM>   // compile-time bound on the outputs k (so the sums stay in registers)
__global__ void __launch_bounds__(32 * kSurpWarps)
    k_surplus_level(int64_t n0, int64_t n1, int d, int k, int fine_n, const uint16_t* __restrict__ fid,
                    const int16_t* __restrict__ fpt, const double* __restrict__ tab1,
                    const double* __restrict__ f, double* __restrict__ W) {
  const int lane = threadIdx.x & 31;
  const int64_t n = n0 + blockIdx.x * int64_t(kSurpWarps) + (threadIdx.x >> 5);
  if (n >= n1) return;
  double acc[KM];
#pragma unroll
  for (int c = 0; c < KM; ++c) acc[c] = 0.0;
  int pts[kMaxDim];
#pragma unroll
  for (int dim = 0; dim < kMaxDim; ++dim) pts[dim] = dim < d ? fpt[n * d + dim] : 0;
  for (int64_t m = lane; m < n0; m += 32) {
    double phi = 1.0;
#pragma unroll
    for (int dim = 0; dim < kMaxDim; ++dim)
      if (dim < d && phi != 0.0) phi *= tab1[int(fid[m * d + dim]) * (fine_n + 1) + pts[dim]];
    if (phi != 0.0) {
#pragma unroll
      for (int c = 0; c < KM; ++c)
        if (c < k) acc[c] = fma(phi, W[m * k + c], acc[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < KM; ++c) {
    if (c < k) {
      double v = acc[c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) W[n * k + c] = f[n * k + c] - v;
    }
  }
}

// Gathers rows of W into the evaluation order (M) and into the nested order (nrows;
// rows that stand for no node, nested < 0, are zero).
__global__ void k_gather_rows(int64_t M, int nrows, int k, const int32_t* __restrict__ order,
                              const int32_t* __restrict__ nested, const double* __restrict__ W,
                              double* __restrict__ Ws, double* __restrict__ Wt) {
  const int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const int64_t r = e / k, c = e % k;
  if (r < M) Ws[e] = W[int64_t(order[r]) * k + c];
  if (r < nrows) Wt[e] = nested[r] < 0 ? 0.0 : W[int64_t(nested[r]) * k + c];
}

// ---------------------------------------------------------------- FP64 evaluation
// Both kernels are bound by the FP64 pipe, which a warp's instruction holds for
// 20 cycles whatever its active lanes.
//
// In lexicographic order of the function ids the nodes are the preorder of a
// tree: a node's parent is the node with its last active dimension set to
// level 1 (in the grid, which is downward closed), and
//   u = value(root),  value(n) = W_n + sum over the children c of phi_c value(c)
// with phi_c the one 1-D basis value of c's last active dimension.  That is K
// multiply-adds per node and no products (the sum over nodes of products of
// their active factors takes A - 1 products more per node: 7.7 FP64 operations
// per node against 4.4 on the level-4 6-D grid).
//
// The order of the sum: the preorder is cut into ranges (four groups of one, two
// or four, by the grid's size), each is summed by itself, and the ranges' sums
// are added by groups (range_sum).  Both kernels perform exactly these
// operations, so a query's result is the same to the last bit whatever the
// number of queries in the call.
// A range is a tree of its own: rows of the nested order, first its start (the
// root's surplus in the range that has the root, else 0), then copies with
// surplus 0 of its first node's ancestors, then its nodes.
constexpr int kNestGroups = 4, kNestGroup = kNestRanges / kNestGroups;
__device__ __forceinline__ double group_sum(const double (&g)[kNestGroups]) {
  return __dadd_rn(__dadd_rn(g[0], g[1]), __dadd_rn(g[2], g[3]));
}
// v(i): the sum of range i; per: ranges of a group
template <typename V>
__device__ __forceinline__ double range_sum(V v, int per) {
  double g[kNestGroups];
#pragma unroll
  for (int i = 0; i < kNestGroups; ++i) {
    g[i] = v(i * per);
#pragma unroll
    for (int j = 1; j < kNestGroup; ++j)
      if (j < per) g[i] = __dadd_rn(g[i], v(i * per + j));
  }
  return group_sum(g);
}

// Grids whose 1-D tables are too large (128 queries' in 200 KB)
static bool fp64_eval_refused(int d, int nf) { return sizeof(double) * d * nf * kEvalThreads > 200 * 1024; }

// Nested form (many queries).  A lane per query, 32 queries per block, a warp
// per range or per group of ranges, so that every warp's control flow is
// uniform.
// Measured (K = 3, d = 6) against a thread per query over the products: 1e6
// queries 20.2 -> 8.76 ms on the level-4 grid (the FP64 pipe's time for the
// multiply-adds and the tables) and 114 -> 26.5 ms on the level-5 grid.
constexpr int kNestQ = 32;

// prog of a row: table offset of its last active dimension (12 bits), its
// depth (active dimensions, 4 bits; 0: a range's start or the end of the last),
// and for a row without children the number of rows from it on that are such
// rows at its depth (16 bits): three quarters of the nodes are taken in runs, by
// a short loop.
__host__ __device__ constexpr uint32_t nested_entry(uint32_t off, uint32_t depth, uint32_t run) {
  return off | depth << 12 | run << 16;
}

template <int K>
struct Nested {
  const uint32_t* prog;
  const double* W;         // K columns of the surpluses in nested order, row stride k
  const double* tab;       // this query's table column
  int k, kc, mend;         // kc: columns that exist (<= K)
  // rows base .. base + 31 of the warp's (they end before mend), staged in
  // shared memory (a row steers the walk, so a load from L2 would stand in
  // its path); lp, lw: the 32 after them, one per lane, on their way
  uint32_t* sp;            // [32]
  double* sw;              // [32][K]
  int lane, base, pos;
  uint32_t lp;
  double lw[K];
  __device__ __forceinline__ void load(int m0) {
    const int i = m0 + lane;
    lp = i < mend ? prog[i] : 0u;
#pragma unroll
    for (int c = 0; c < K; ++c) lw[c] = i < mend && c < kc ? W[int64_t(i) * k + c] : 0.0;
  }
  __device__ __forceinline__ void refill() {
    __syncwarp();
    sp[lane] = lp;
#pragma unroll
    for (int c = 0; c < K; ++c) sw[lane * K + c] = lw[c];
    __syncwarp();
    base += 32;
    pos = 0;
    load(base + 32);
  }
};
constexpr int nested_stage_bytes(int K) { return 32 * (8 * K + 4); }   // per warp

// Adds the children (and theirs) at depth D from the current row on to acc.
template <int K, int D>
__device__ __forceinline__ void nested_children(Nested<K>& t, double (&acc)[K]) {
  if constexpr (D <= kMaxDim) {
    while (true) {
      if (t.pos == 32) t.refill();
      const uint32_t p = t.sp[t.pos];
      if (((p >> 12) & 15u) != uint32_t(D)) break;   // (depth 0 ends every loop)
      int run = static_cast<int>(p >> 16);
      if (run != 0) {
        run = min(run, 32 - t.pos);
        const uint32_t* sp = t.sp + t.pos;
        const double* sw = t.sw + t.pos * K;
        t.pos += run;
#pragma unroll 2
        for (; run > 0; --run, ++sp, sw += K) {
          const double phi = t.tab[(*sp & 0xFFFu) * kNestQ];
#pragma unroll
          for (int c = 0; c < K; ++c) acc[c] = fma(phi, sw[c], acc[c]);
        }
        continue;
      }
      double v[K];
#pragma unroll
      for (int c = 0; c < K; ++c) v[c] = t.sw[t.pos * K + c];
      ++t.pos;
      const double phi = t.tab[(p & 0xFFFu) * kNestQ];
      nested_children<K, D + 1>(t, v);
#pragma unroll
      for (int c = 0; c < K; ++c) acc[c] = fma(phi, v[c], acc[c]);
    }
  }
}

template <int K>
__global__ void __launch_bounds__(32 * kNestRanges, 1) k_eval_fp64_nested(EvalArgs e, int d, int c0, size_t stage0) {
  extern __shared__ double tabs_s[];   // [d * nf][kNestQ] (then the warps' sums), the warps' stages
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t q = blockIdx.x * int64_t(kNestQ) + lane;
  const bool live = q < e.Q;
  for (int dim = warp; dim < d; dim += nw) {
    const double u = live ? (e.xq[q * d + dim] - e.lo[dim]) / e.width[dim] : 0.5;
    basis_row_fast(u, e.level, e.xf, tabs_s + (dim * e.nf) * kNestQ + lane, kNestQ);
  }
  __syncthreads();
  Nested<K> t;
  t.prog = e.prog;
  t.W = e.Wt + c0;
  t.tab = tabs_s + lane;
  t.k = e.k;
  t.kc = e.k - c0 < K ? e.k - c0 : K;
  t.lane = lane;
  t.sw = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(tabs_s) + stage0 + warp * nested_stage_bytes(K));
  t.sp = reinterpret_cast<uint32_t*>(t.sw + 32 * K);
  const int per = nw == kNestGroups ? e.per : 1;   // ranges of this warp
  // (a warp's number is its quarter of the SM: the groups, a few per cent
  // apart, go round the quarters from block to block)
  const int part = (warp + blockIdx.x) & (nw - 1), r0 = part * per;
  double total[K];
  t.mend = e.range[r0 + per] + 1;   // (the next range's start ends the last)
  t.base = e.range[r0] - 32;
  t.load(t.base + 32);
  t.refill();
#pragma unroll 1
  for (int j = 0; j < per; ++j) {
    if (t.pos == 32) t.refill();
    double acc[K];
#pragma unroll
    for (int c = 0; c < K; ++c) acc[c] = t.sw[t.pos * K + c];   // the range's start
    ++t.pos;
    nested_children<K, 1>(t, acc);
#pragma unroll
    for (int c = 0; c < K; ++c) total[c] = j == 0 ? acc[c] : __dadd_rn(total[c], acc[c]);
  }
  __syncthreads();   // the tables are read; their space takes the sums
  double* sum = tabs_s;
#pragma unroll
  for (int c = 0; c < K; ++c) sum[(part * K + c) * 32 + lane] = total[c];
  __syncthreads();
  for (int c = warp; c < t.kc; c += nw) {
    double u;
    if (nw == kNestGroups) {
      double g[kNestGroups];
#pragma unroll
      for (int s = 0; s < kNestGroups; ++s) g[s] = sum[(s * K + c) * 32 + lane];
      u = group_sum(g);
    } else {
      u = range_sum([&](int r) { return sum[(r * K + c) * 32 + lane]; }, e.per);
    }
    if (live) e.out[q * e.k + c0 + c] = u;
  }
}

// Few queries: the same sums with the nodes over the lanes.  Only rows with
// children (entries) need work: an entry's value is one chain of
// multiply-adds over its children, whose values are surpluses (leaves) or
// entries of smaller height.  Entries go by height, a block barrier between
// heights; a thread per query, entry and output; within a height the entries
// are sorted by their number of children, so that a warp's chains are about
// equally long.  The chains are latency, so the node data is copied to shared
// memory beside the tables (kStaged, where it fits), and a batch of four
// children (lists are padded) is loaded while the one before is summed.
constexpr int kFewBatch = 4, kFewThreads = 512;   // (or 256 threads)

constexpr size_t kFewSmem = 220 * 1024;
struct FewLayout {   // byte offsets in shared memory after the tables
  size_t val, W, child, ent, total;
};
// kv columns at a time
__host__ __device__ inline FewLayout few_layout(const EvalArgs& e, int d, int kv, int QB, bool staged) {
  auto up = [](size_t x) { return (x + 15) & ~size_t(15); };
  FewLayout L;
  L.val = up(sizeof(double) * d * e.nf * QB);
  // (first the rows' reciprocals, factors, coordinates and hits)
  const size_t rows = (sizeof(double) * ((size_t(1) << e.level) + 1 + e.level + 1) + sizeof(int)) * d * QB;
  const size_t vals = sizeof(double) * (e.fheight[kMaxDim + 1] + 1) * kv * QB;
  L.W = L.val + up(rows > vals ? rows : vals);
  L.child = L.W + (staged ? up(sizeof(double) * e.nrows * kv) : 0);
  L.ent = L.child + (staged ? up(sizeof(uint32_t) * e.nchild) : 0);
  L.total = L.ent + (staged ? sizeof(int4) * e.fheight[kMaxDim + 1] : 0);
  return L;
}

template <int QB, bool kStaged>
__global__ void __launch_bounds__(kFewThreads, 1) k_eval_fp64_few(EvalArgs e, int d, int c0, int kc, int kv) {
  extern __shared__ __align__(16) double tabs_s[];   // [d * nf][QB], values of the entries [entry][kv][QB], node data
  char* sm = reinterpret_cast<char*>(tabs_s);
  const FewLayout at = few_layout(e, d, kv, QB, kStaged);
  double* val = reinterpret_cast<double*>(sm + at.val);
  const int tid = threadIdx.x, nt = blockDim.x;
  const int64_t q0 = blockIdx.x * int64_t(QB);
  const int nent = e.fheight[kMaxDim + 1];
  const double* W = e.Wt + c0;
  const uint4* child = reinterpret_cast<const uint4*>(e.fchild);
  const int4* ent = e.fent;
  int ldw = e.k;
  if constexpr (kStaged) {
    auto copy16 = [&](size_t dst, const void* src, int n) {   // n 16-byte words
      for (int i = tid; i < n; i += nt) {
        const unsigned to = static_cast<unsigned>(__cvta_generic_to_shared(sm + dst + size_t(i) * 16));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(static_cast<const char*>(src) + size_t(i) * 16));
      }
    };
    copy16(at.child, e.fchild, e.nchild / 4);
    copy16(at.ent, e.fent, nent);
    if (kv == e.k) copy16(at.W, e.Wt, (e.nrows * kv + 1) / 2);   // (the array is padded to whole words)
    W = reinterpret_cast<const double*>(sm + at.W);
    ldw = kv;
    child = reinterpret_cast<const uint4*>(sm + at.child);
    ent = reinterpret_cast<const int4*>(sm + at.ent);
  }
  // tables: row (dim, query) = task, spread over the threads at the levels that
  // basis_row_fast unrolls (12,000 cycles with a thread per row at level 4, 9,300 now)
  const int rows = QB * d;
  const bool spread = e.level >= 1 && e.level <= 5;
  const int np = (1 << e.level) + 1;
  double* rinv = val;                     // [np][rows]
  double* wi = rinv + np * rows;          // [level][rows]
  double* us = wi + e.level * rows;       // [rows]
  int* hits = reinterpret_cast<int*>(us + rows);
  for (int task = tid; task < rows; task += nt) {
    const int tq = task % QB, dim = task / QB;
    const int64_t q = q0 + tq;
    const double u = q < e.Q ? (e.xq[q * d + dim] - e.lo[dim]) / e.width[dim] : 0.5;
    us[task] = u;
    hits[task] = -1;
    if (!spread || !basis_in_range(u)) {
      hits[task] = -2;   // done
      basis_row(u, e.level, e.xf, tabs_s + (dim * e.nf) * QB + tq, QB);
    }
  }
  if (spread) {
    __syncthreads();
    for (int i = tid; i < np * rows; i += nt) {
      const int task = i % rows, pt = i / rows;
      bool zero;
      rinv[i] = basis_reciprocal(us[task], e.xf[pt], zero);
      if (zero && hits[task] != -2) hits[task] = pt;
    }
    __syncthreads();
    for (int task = tid; task < rows; task += nt) basis_factors(rinv + task, rows, e.level, wi + task);
    __syncthreads();
    for (int i = tid; i < e.nf * rows; i += nt) {
      const int task = i % rows, id = i / rows, tq = task % QB, dim = task / QB;
      if (hits[task] == -2) continue;
      tabs_s[(dim * e.nf + id) * QB + tq] =
          id == 0 ? 1.0 : basis_value(rinv + task, wi + task, rows, e.level, id, hits[task]);
    }
  }
  __syncthreads();
  // a list's padding: entry nent with factor 1, v + 1 * -0 = v for every v
  for (int i = tid; i < kv * QB; i += nt) val[nent * kv * QB + i] = -0.0;
  if constexpr (kStaged) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int b = 0; b < kc; b += kv) {
    const int kn = min(kv, kc - b);
    if constexpr (kStaged) {
      if (kv != e.k) {   // this pass's columns
        double* Ws = reinterpret_cast<double*>(sm + at.W);
        for (int i = tid; i < e.nrows * kn; i += nt) Ws[i / kn * kv + i % kn] = e.Wt[int64_t(i / kn) * e.k + c0 + b + i % kn];
        __syncthreads();
      }
    }
    const double* Wb = kStaged ? W : W + b;
    for (int h = 0; h < kMaxDim + 1; ++h) {
      const int n = (e.fheight[h + 1] - e.fheight[h]) * kn * QB;
      if (n == 0) continue;
      for (int item = tid; item < n; item += nt) {
        const int t = item / QB, q = item % QB, c = t % kn, en = e.fheight[h] + t / kn;
        const int4 E = ent[en];
        double v = Wb[E.z * ldw + c];
        const uint4* ch = child + E.x / 4;
        double p[kFewBatch], w[kFewBatch];
        uint4 x4 = ch[0];
        auto load = [&]() {
          const uint32_t x[kFewBatch] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
          for (int j = 0; j < kFewBatch; ++j) {
            p[j] = tabs_s[(x[j] & 0xFFFu) * QB + q];
            w[j] = *((x[j] & 0x1000u) ? val + ((x[j] >> 13) * kv + c) * QB + q : Wb + (x[j] >> 13) * ldw + c);
          }
        };
        if (E.y > 0) load();
        x4 = ch[1];   // (past the last list: padding)
        for (int i = 0; i < E.y; i += kFewBatch) {
          double p0[kFewBatch], w0[kFewBatch];
#pragma unroll
          for (int j = 0; j < kFewBatch; ++j) {
            p0[j] = p[j];
            w0[j] = w[j];
          }
          if (i + kFewBatch < E.y) {
            load();
            x4 = ch[i / 4 + 2];
          }
#pragma unroll
          for (int j = 0; j < kFewBatch; ++j)
            v = fma(p0[j], w0[j], v);
        }
        val[(en * kv + c) * QB + q] = v;
      }
      __syncthreads();
    }
    for (int t = tid; t < QB * kn; t += nt) {
      const int q = t / kn, c = t % kn;
      if (q0 + q >= e.Q) break;
      e.out[(q0 + q) * e.k + c0 + b + c] =
          range_sum([&](int r) { return val[(e.froot[r] * kv + c) * QB + q]; }, e.per);
    }
    if (b + kv < kc) __syncthreads();   // the entries' values are read
  }
}

template <int K>
static int launch_eval_fp64_nested(const EvalArgs& e, int d, int c0, cudaStream_t st) {
  const int64_t blocks = ceil_div(e.Q, kNestQ);
  // A warp per range leaves room for one or two blocks per SM, a warp per group
  // for four: taken where the last wave of those would be nearly empty (level 4,
  // 20,000 queries: 224 us against 262; 1e6: 9.2 ms against 8.8).
  const int64_t waves = ceil_div(blocks, kNumSMs);
  const int nw = waves <= 2 || (waves < 24 && waves % 4 == 1) ? kNestGroups * e.per : kNestGroups;
  const size_t tab = sizeof(double) * d * e.nf * kNestQ, sum = sizeof(double) * nw * K * 32;
  const size_t stage0 = tab > sum ? tab : sum, smem = stage0 + nw * nested_stage_bytes(K);
  SG_CUDA_TRY(ensure_dynamic_smem(k_eval_fp64_nested<K>, smem));
  SG_TIMED("k_eval_fp64_nested", st,
           (k_eval_fp64_nested<K><<<static_cast<unsigned>(blocks), 32 * nw, smem, st>>>(e, d, c0, stage0)));
  SG_LAUNCH_CHECK("k_eval_fp64_nested");
  return SG_OK;
}

template <int QB>
static int launch_eval_fp64_few(const EvalArgs& e, int d, int c0, int kc, int nt, cudaStream_t st, int kv = 0) {
  if (kv == 0) kv = kc;
  const bool staged = few_layout(e, d, kv, QB, true).total <= kFewSmem;
  const size_t smem = few_layout(e, d, kv, QB, staged).total;
  auto* kern = staged ? k_eval_fp64_few<QB, true> : k_eval_fp64_few<QB, false>;
  SG_CUDA_TRY(ensure_dynamic_smem(kern, smem));
  SG_TIMED("k_eval_fp64_few", st, (kern<<<static_cast<unsigned>(ceil_div(e.Q, QB)), nt, smem, st>>>(e, d, c0, kc, kv)));
  SG_LAUNCH_CHECK("k_eval_fp64_few");
  return SG_OK;
}

// K columns from c0 on.  The nested form comes in blocks of 32 queries, one SM's
// work at least.  Below a wave of them, the fewest queries per block that fill one
// wave: two blocks of 256 threads or one of 512 per SM, by what fits in shared
// memory (16 queries: a column at a time where the entries' values of all do
// not).  Measured (K = 3, d = 6, us on the level-4 and level-5 grid): 1 query 13.6 /
// 22.4, 304: 16.3 / 26.2, 608: 17.1 / 43.9, 1,216: 23.2 / 68.5, 2,432: 33.7 / 108;
// nested, up to a wave: 51.0 / 134.
template <int K>
static int launch_eval_fp64(const EvalArgs& e, int d, int c0, cudaStream_t st) {
  const int kc = e.k - c0 < K ? e.k - c0 : K;
  auto fits16 = [&](int kv) { return few_layout(e, d, kv, 16, false).total <= kFewSmem; };
  const size_t one = few_layout(e, d, kc, 1, true).total;   // two staged blocks per SM, or one
  const bool two = one <= kFewSmem / 2 || one > kFewSmem;
  if (e.Q <= (two ? 2 : 1) * kNumSMs) return launch_eval_fp64_few<1>(e, d, c0, kc, 256, st);
  if (e.Q <= 2 * kNumSMs) return launch_eval_fp64_few<2>(e, d, c0, kc, 512, st);
  if (e.Q <= 4 * kNumSMs) return launch_eval_fp64_few<4>(e, d, c0, kc, 512, st);
  if (e.Q <= 8 * kNumSMs) return launch_eval_fp64_few<4>(e, d, c0, kc, 256, st);
  if (e.Q <= 16 * kNumSMs && fits16(kc)) return launch_eval_fp64_few<16>(e, d, c0, kc, 512, st);
  if (e.Q <= 16 * kNumSMs && fits16(1)) return launch_eval_fp64_few<16>(e, d, c0, kc, 512, st, 1);
  return launch_eval_fp64_nested<K>(e, d, c0, st);
}

int eval_fp64(const EvalArgs& e, int d, cudaStream_t st) {
  if (d < 1 || d > kMaxDim) return fail(SG_EUNSUPPORTED, "sg_eval_feedback: d must be 1..8");
  if (fp64_eval_refused(d, e.nf))
    return fail(SG_EUNSUPPORTED, "sg_eval_feedback: grid level too high for the FP64 kernel");
  switch (e.k) {
    case 1: return launch_eval_fp64<1>(e, d, 0, st);
    case 2: return launch_eval_fp64<2>(e, d, 0, st);
    case 3: return launch_eval_fp64<3>(e, d, 0, st);
    case 4: return launch_eval_fp64<4>(e, d, 0, st);
    case 6: return launch_eval_fp64<6>(e, d, 0, st);
    default:   // any output count, four columns at a time (rarely used shapes)
      for (int c0 = 0; c0 < e.k; c0 += 4) {
        const int rc = launch_eval_fp64<4>(e, d, c0, st);
        if (rc != SG_OK) return rc;
      }
      return SG_OK;
  }
}

}  // namespace sg

using namespace sg;

namespace sg {
namespace {
// The host-made part of a surplus build: the integer structure of the grid's
// nodes (function ids, fine positions, level ranges, evaluation order, active
// dimensions and table offsets, the sum-factorised plan), the layout of the
// surplus's one device allocation, and the bytes of it that the host fills
// (all but the box).  It depends on the grid's node structure and on k only,
// so builds on grids of the same structure (a grid rebuilt every step) reuse
// it: a small cache keyed by (d, L, k) and checked against the grid's levels
// and indices.
struct SurplusHost {
  int d = 0, L = 0, k = 0, nf = 0, amax = 0;
  int64_t M = 0;
  std::vector<int8_t> lev;      // the key: the grid's integer structure
  std::vector<int16_t> kidx;
  std::vector<int64_t> level_start;
  int64_t grp[kMaxDim + 2] = {};
  bool sf_ok = false, tcoff_ok = false;
  SfPlan sf;                    // scalar fields (its tables are in the staged bytes)
  size_t npack = 0, off = 0, ohost = 0;
  size_t oW = 0, oWs = 0, oWdf = 0, oxf = 0, oxfdf = 0, otab1 = 0, obp = 0, oerr = 0, osfb = 0;
  size_t oWt = 0, oprog = 0, onested = 0;   // nested order (FP64 evaluation)
  size_t ofent = 0, ofchild = 0;                       // ... and its ranges' inner entries
  int nrows = 0, per = 0, range[kNestRanges + 1] = {}, fheight[kMaxDim + 2] = {}, froot[kNestRanges] = {}, nchild = 0;
  size_t obox = 0, onact = 0, oops = 0, otcoff = 0, ofid = 0, ofpt = 0, oorder = 0, ometa = 0, obmap = 0;
  std::vector<unsigned char> staging;   // bytes [ohost, off) of the allocation, box zero
  // The same bytes in page-locked memory when it could be had (then
  // `staging` is emptied): a copy from it is queued without waiting for the
  // stream, where a copy from pageable memory first synchronises it.
  unsigned char* pinned = nullptr;
  const unsigned char* bytes() const { return pinned ? pinned : staging.data(); }
  SurplusHost() = default;
  SurplusHost(const SurplusHost&) = delete;
  SurplusHost& operator=(const SurplusHost&) = delete;
  ~SurplusHost() {
    if (pinned) {
      cudaDeviceSynchronize();   // a build may still be copying from it
      cudaFreeHost(pinned);
    }
  }
};

// The rows of the nested order (see k_eval_fp64_nested) from its nodes' depths and
// table offsets.
struct NestedRows {
  std::vector<int32_t> node;      // place of the row's node in the nested order, or -1
  std::vector<uint32_t> prog;     // nested_entry
  int per;                        // ranges of a group
  int range[kNestRanges + 1] = {};   // first rows of the ranges; the last row (an end)
};
NestedRows nested_rows(const std::vector<uint32_t>& depth, const std::vector<uint16_t>& path) {
  const int64_t M = static_cast<int64_t>(depth.size());
  // about equal ranges (within a tenth of one), cut where few ancestors have to
  // be entered again; a range costs each query about six FP64 operations, so
  // small grids have fewer
  NestedRows rows;
  rows.per = M < 150 ? 1 : (M < 2500 ? 2 : kNestGroup);
  const int n = rows.per * kNestGroups;
  const int64_t slack = M / (10 * n);
  auto begin = [&](int r) {
    const int64_t at = M * r / n;
    int64_t best = at;
    for (int64_t o = 1; r > 0 && r < n && o <= slack; ++o) {
      if (depth[at - o] < depth[best]) best = at - o;
      if (depth[at + o] < depth[best]) best = at + o;
    }
    return best;
  };
  std::vector<uint32_t> dep, off;
  auto add = [&](int64_t node, uint32_t D, uint32_t o) {
    rows.node.push_back(static_cast<int32_t>(node));
    dep.push_back(D);
    off.push_back(o);
  };
  for (int r = 0; r < n; ++r) {
    const int64_t m0 = begin(r), m1 = begin(r + 1);
    rows.range[r] = static_cast<int>(dep.size());
    add(m0 == 0 && m1 > 0 ? 0 : -1, 0, 0);
    if (m0 < m1)
      for (uint32_t D = 1; D < depth[m0]; ++D) add(-1, D, path[m0 * kMaxDim + D - 1]);
    for (int64_t m = std::max<int64_t>(m0, 1); m < m1; ++m) add(m, depth[m], path[m * kMaxDim + depth[m] - 1]);
  }
  rows.range[n] = static_cast<int>(dep.size());
  add(-1, 0, 0);
  rows.prog.resize(dep.size());
  uint32_t run = 0;
  for (size_t i = dep.size(); i-- > 0;) {   // a row's first child, if any, is the row after it
    const bool leaf = dep[i] > 0 && dep[i + 1] <= dep[i];
    run = leaf ? (run != 0 && dep[i + 1] == dep[i] && run < 0xFFFFu ? run + 1 : 1) : 0;
    rows.prog[i] = nested_entry(off[i], dep[i], run);
  }
  return rows;
}

// The rows with children for k_eval_fp64_few (and the starts of empty ranges): by
// height (fheight[h]: the first of height h + 1), within a height by falling
// number of children; froot: the ranges' starts.
void nested_entries(const NestedRows& rows, std::vector<int32_t>& fent, std::vector<uint32_t>& fchild,
                    int (&fheight)[kMaxDim + 2], int (&froot)[kNestRanges]) {
  struct Entry {
    int32_t row;
    int height;
    std::vector<uint32_t> kids;   // as fchild
  };
  std::vector<Entry> es;
  int open[kMaxDim + 1] = {};     // the entry at each depth on the current path
  auto depth = [&](size_t i) { return (rows.prog[i] >> 12) & 15u; };
  for (size_t i = 0; i + 1 < rows.prog.size(); ++i) {
    const uint32_t D = depth(i), off = rows.prog[i] & 0xFFFu;
    const bool entry = D == 0 || depth(i + 1) > D;
    if (D > 0)
      es[open[D - 1]].kids.push_back(entry ? off | 0x1000u | uint32_t(es.size()) << 13 : off | uint32_t(i) << 13);
    if (entry) {
      open[D] = static_cast<int>(es.size());
      es.push_back({static_cast<int32_t>(i), 1, {}});
    }
  }
  for (size_t i = es.size(); i-- > 0;)   // (an entry comes before its children)
    for (uint32_t x : es[i].kids)
      if (x & 0x1000u) es[i].height = std::max(es[i].height, es[x >> 13].height + 1);
  std::vector<int32_t> by(es.size()), at(es.size());
  std::iota(by.begin(), by.end(), 0);
  std::stable_sort(by.begin(), by.end(), [&](int32_t a, int32_t b) {
    return es[a].height != es[b].height ? es[a].height < es[b].height : es[a].kids.size() > es[b].kids.size();
  });
  for (size_t i = 0; i < by.size(); ++i) at[by[i]] = static_cast<int32_t>(i);
  for (int h = 0; h < kMaxDim + 2; ++h)
    fheight[h] = static_cast<int>(std::count_if(es.begin(), es.end(), [&](const Entry& x) { return x.height <= h; }));
  int r = 0;
  for (size_t i = 0; i < es.size(); ++i)
    if (depth(es[i].row) == 0) froot[r++] = at[i];
  const uint32_t pad = 0x1000u | uint32_t(es.size()) << 13;
  for (int32_t i : by) {
    const Entry& x = es[i];
    fent.insert(fent.end(), {static_cast<int32_t>(fchild.size()), static_cast<int32_t>(x.kids.size()), x.row, 0});
    for (uint32_t kid : x.kids) fchild.push_back(kid & 0x1000u ? (kid & 0x1FFFu) | uint32_t(at[kid >> 13]) << 13 : kid);
    fchild.resize((fchild.size() + kFewBatch - 1) / kFewBatch * kFewBatch, pad);   // whole batches
  }
  fchild.resize(fchild.size() + 2 * kFewBatch, pad);   // read ahead, not used
}

std::shared_ptr<const SurplusHost> make_surplus_host(const sg_grid* g, int k) {
  auto h = std::make_shared<SurplusHost>();
  const int d = g->d, L = g->level, fine_n = 1 << L;
  const int64_t M = g->M;
  h->d = d;
  h->L = L;
  h->k = k;
  h->M = M;
  h->nf = n_functions(L);
  h->lev = g->h_lev;
  h->kidx = g->h_kidx;
  // integer structure (function ids, fine positions, level ranges, order)
  std::vector<uint16_t> fid(M * d);
  std::vector<int16_t> fpt(M * d);
  int prev_sum = -1;
  for (int64_t n = 0; n < M; ++n) {
    int sum = 0;
    for (int dim = 0; dim < d; ++dim) {
      const int l = g->h_lev[n * d + dim], kk = g->h_kidx[n * d + dim];
      sum += l;
      fid[n * d + dim] = static_cast<uint16_t>(function_id(l, kk));
      fpt[n * d + dim] = static_cast<int16_t>(l == 1 ? fine_n / 2 : kk * (fine_n >> (l - 1)));
    }
    if (sum != prev_sum) {
      h->level_start.push_back(n);
      prev_sum = sum;
    }
  }
  h->level_start.push_back(M);
  // evaluation order: by the number of active dimensions (so that a kernel
  // can take each group with a fixed-length basis product), then the
  // function ids lexicographically
  std::vector<int> na_of(M, 0);
  for (int64_t n = 0; n < M; ++n)
    for (int dim = 0; dim < d; ++dim) na_of[n] += fid[n * d + dim] != 0;
  std::vector<int32_t> order(M);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    if (na_of[a] != na_of[b]) return na_of[a] < na_of[b];
    for (int dim = 0; dim < d; ++dim) {
      if (fid[a * d + dim] != fid[b * d + dim]) return fid[a * d + dim] < fid[b * d + dim];
    }
    return false;
  });
  std::vector<uint8_t> nact(M, 0);
  std::vector<uint16_t> ops(M * kMaxDim, 0);
  for (int a = 0; a <= kMaxDim + 1; ++a) h->grp[a] = M;
  for (int64_t r = M - 1; r >= 0; --r) {
    const int32_t n = order[r];
    int na = 0;
    for (int dim = 0; dim < d; ++dim) {
      const int id = fid[int64_t(n) * d + dim];
      if (id != 0) ops[r * kMaxDim + na++] = static_cast<uint16_t>(dim * h->nf + id);
    }
    nact[r] = static_cast<uint8_t>(na);
    if (na > h->amax) h->amax = na;
    for (int a = 0; a <= na; ++a) h->grp[a] = r < h->grp[a] ? r : h->grp[a];
  }
  // grp[a] = first node with at least a active dimensions (non-decreasing)
  for (int a = kMaxDim; a >= 0; --a) h->grp[a] = h->grp[a] < h->grp[a + 1] ? h->grp[a] : h->grp[a + 1];

  // the nested order (preorder of the tree of active dimensions): function
  // ids lexicographically; per node its depth and last table offset, and the
  // offsets of its whole path
  std::vector<int32_t> nested(M);
  std::iota(nested.begin(), nested.end(), 0);
  std::stable_sort(nested.begin(), nested.end(), [&](int32_t a, int32_t b) {
    return std::lexicographical_compare(&fid[int64_t(a) * d], &fid[int64_t(a) * d] + d, &fid[int64_t(b) * d],
                                        &fid[int64_t(b) * d] + d);
  });
  std::vector<uint32_t> depth(M, 0);
  std::vector<uint16_t> path(M * kMaxDim, 0);
  for (int64_t r = 0; r < M; ++r) {
    int na = 0;
    for (int dim = 0; dim < d; ++dim) {
      const int id = fid[int64_t(nested[r]) * d + dim];
      if (id != 0) path[r * kMaxDim + na++] = static_cast<uint16_t>(dim * h->nf + id);
    }
    depth[r] = na;
  }
  const NestedRows rows = nested_rows(depth, path);
  const size_t nrows = rows.prog.size();
  h->nrows = static_cast<int>(nrows);
  h->per = rows.per;
  std::copy(std::begin(rows.range), std::end(rows.range), h->range);
  std::vector<int32_t> row_node(nrows, -1);
  for (size_t i = 0; i < nrows; ++i)
    if (rows.node[i] >= 0) row_node[i] = nested[rows.node[i]];
  // the rows with children, and those (few queries)
  std::vector<int32_t> fent;      // per entry: first child, children, row, unused
  std::vector<uint32_t> fchild;   // per child: table offset (12 bits), whether an entry (1), entry or row
  if (!fp64_eval_refused(d, h->nf)) nested_entries(rows, fent, fchild, h->fheight, h->froot);

  // one device allocation: the surplus's arrays and the build's tables; the
  // device-computed ones first, then the host-made ones (one copy)
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~size_t(255);
    return o;
  };
  h->oW = take(M * k * sizeof(double));
  h->oWs = take(M * k * sizeof(double));
  h->oWt = take(nrows * k * sizeof(double));
  h->oWdf = take(M * k * sizeof(float2));
  h->oxf = take((fine_n + 1) * sizeof(double));
  h->oxfdf = take((fine_n + 1) * sizeof(float2));
  h->otab1 = take(size_t(h->nf) * (fine_n + 1) * sizeof(double));
  // the sum-factorised tensor-core plan; the per-node tensor-core pack only
  // where that plan does not fit
  h->sf_ok = sf_plan(d, L, h->nf, k, M, fid, h->sf);
  h->npack = h->sf_ok ? 0 : tf32_pack_floats(M, k);
  h->obp = take(h->npack * sizeof(float));
  h->oerr = take(sizeof(int));
  h->osfb = take(h->sf_ok ? h->sf.bbytes : 0);   // filled on the device (k_pack_sf)
  h->ohost = off;
  h->obox = take(2 * d * sizeof(double));
  h->onact = take(M);
  h->oops = take(M * kMaxDim * sizeof(uint16_t));
  // the tensor-core kernel's table offsets: ops scaled by its 128 table rows
  // (uint16, so the tables must have at most 511 entries per query)
  h->tcoff_ok = h->npack && size_t(d) * h->nf <= 511;
  h->otcoff = take(h->tcoff_ok ? M * kMaxDim * sizeof(uint16_t) : 0);
  h->ofid = take(M * d * sizeof(uint16_t));
  h->ofpt = take(M * d * sizeof(int16_t));
  h->oorder = take(M * sizeof(int32_t));
  h->onested = take(nrows * sizeof(int32_t));
  h->oprog = take(nrows * sizeof(uint32_t));
  h->ofent = take(fent.size() * sizeof(int32_t));
  h->nchild = static_cast<int>(fchild.size());
  h->ofchild = take(fchild.size() * sizeof(uint32_t));
  h->ometa = take(h->sf_ok ? h->sf.meta.size() : 0);
  h->obmap = take(h->sf_ok ? h->sf.bmap.size() * sizeof(int32_t) : 0);
  h->off = off;
  const size_t oh = h->ohost;
  auto& st = h->staging;
  st.assign(off - oh, 0);
  std::memcpy(st.data() + (h->onact - oh), nact.data(), M);
  std::memcpy(st.data() + (h->oops - oh), ops.data(), M * kMaxDim * sizeof(uint16_t));
  if (h->tcoff_ok) {
    std::vector<uint16_t> tco(M * kMaxDim);
    for (size_t x = 0; x < tco.size(); ++x) tco[x] = static_cast<uint16_t>(ops[x] * 128u);
    std::memcpy(st.data() + (h->otcoff - oh), tco.data(), M * kMaxDim * sizeof(uint16_t));
  }
  std::memcpy(st.data() + (h->ofid - oh), fid.data(), M * d * sizeof(uint16_t));
  std::memcpy(st.data() + (h->ofpt - oh), fpt.data(), M * d * sizeof(int16_t));
  std::memcpy(st.data() + (h->oorder - oh), order.data(), M * sizeof(int32_t));
  std::memcpy(st.data() + (h->onested - oh), row_node.data(), nrows * sizeof(int32_t));
  std::memcpy(st.data() + (h->oprog - oh), rows.prog.data(), nrows * sizeof(uint32_t));
  if (!fent.empty()) {
    std::memcpy(st.data() + (h->ofent - oh), fent.data(), fent.size() * sizeof(int32_t));
    if (!fchild.empty()) std::memcpy(st.data() + (h->ofchild - oh), fchild.data(), fchild.size() * sizeof(uint32_t));
  }
  if (h->sf_ok) {
    std::memcpy(st.data() + (h->ometa - oh), h->sf.meta.data(), h->sf.meta.size());
    std::memcpy(st.data() + (h->obmap - oh), h->sf.bmap.data(), h->sf.bmap.size() * sizeof(int32_t));
    h->sf.bfloats_ = h->sf.bmap.size();
    h->sf.meta_bytes_ = h->sf.meta.size();
    h->sf.meta.clear();
    h->sf.meta.shrink_to_fit();
    h->sf.bmap.clear();
    h->sf.bmap.shrink_to_fit();
  }
  if (cudaHostAlloc(reinterpret_cast<void**>(&h->pinned), st.size(), cudaHostAllocDefault) == cudaSuccess) {
    std::memcpy(h->pinned, st.data(), st.size());
    st.clear();
    st.shrink_to_fit();
  } else {
    h->pinned = nullptr;
    (void)cudaGetLastError();   // pageable staging still works, the copy then waits
  }
  return h;
}

std::shared_ptr<const SurplusHost> surplus_host(const sg_grid* g, int k) {
  static std::mutex mu;
  // most recent last; never destroyed (its entries' page-locked memory is not
  // handed back to a CUDA runtime that may already be shut down at exit)
  static auto* cache = new std::vector<std::shared_ptr<const SurplusHost>>();
  {
    std::lock_guard<std::mutex> lk(mu);
    for (auto& c : *cache)
      if (c->d == g->d && c->L == g->level && c->k == k && c->M == g->M && c->lev == g->h_lev && c->kidx == g->h_kidx)
        return c;
  }
  auto h = make_surplus_host(g, k);
  std::lock_guard<std::mutex> lk(mu);
  if (cache->size() >= 8) cache->erase(cache->begin());
  cache->push_back(h);
  return h;
}
}  // namespace
}  // namespace sg

extern "C" int sg_build_surpluses(const sg_grid* g, const double* d_values, int k, sg_surplus** out,
                                  void* stream) {
  clear_error();
  if (!g || !d_values || !out) return fail(SG_EINVAL, "sg_build_surpluses: null pointer");
  *out = nullptr;
  if (k < 1 || k > kMaxOut) return fail(SG_EINVAL, "sg_build_surpluses: k must be 1..16");
  if (g->level > kMaxLevel) return fail(SG_EUNSUPPORTED, "sg_build_surpluses: level above 8");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int d = g->d, L = g->level, fine_n = 1 << L;
  const int64_t M = g->M;
  std::shared_ptr<const SurplusHost> hp;
  try {
    hp = surplus_host(g, k);
  } catch (const std::bad_alloc&) {
    return fail(SG_ENOMEM, "sg_build_surpluses: host memory");
  }
  const SurplusHost& h = *hp;
  auto* s = new sg_surplus();
  s->d = d;
  s->level = L;
  s->k = k;
  s->M = M;
  s->nf = h.nf;
  s->amax = h.amax;
  for (int a = 0; a <= kMaxDim + 1; ++a) s->grp[a] = h.grp[a];
  cudaError_t e = block_alloc(&s->block, h.off, st);
  if (e != cudaSuccess) {
    delete s;
    return e == cudaErrorMemoryAllocation ? fail(SG_ENOMEM, "sg_build_surpluses: device allocation") : cuda_fail(e, "sg_build_surpluses: device allocation");
  }
  char* base = static_cast<char*>(s->block);
  s->W = reinterpret_cast<double*>(base + h.oW);
  s->Ws = reinterpret_cast<double*>(base + h.oWs);
  s->Wt = reinterpret_cast<double*>(base + h.oWt);
  s->prog = reinterpret_cast<uint32_t*>(base + h.oprog);
  s->nrows = h.nrows;
  s->per = h.per;
  s->fent = reinterpret_cast<int4*>(base + h.ofent);
  s->fchild = reinterpret_cast<uint32_t*>(base + h.ofchild);
  s->nchild = h.nchild;
  std::copy(std::begin(h.range), std::end(h.range), s->range);
  std::copy(std::begin(h.fheight), std::end(h.fheight), s->fheight);
  std::copy(std::begin(h.froot), std::end(h.froot), s->froot);
  s->Wdf = reinterpret_cast<float2*>(base + h.oWdf);
  s->xf = reinterpret_cast<double*>(base + h.oxf);
  s->xfdf = reinterpret_cast<float2*>(base + h.oxfdf);
  s->bpack = h.npack ? reinterpret_cast<float*>(base + h.obp) : nullptr;
  s->tc_err = reinterpret_cast<int*>(base + h.oerr);
  s->box = reinterpret_cast<double*>(base + h.obox);
  s->nact = reinterpret_cast<uint8_t*>(base + h.onact);
  s->ops = reinterpret_cast<uint16_t*>(base + h.oops);
  s->tcoff = h.tcoff_ok ? reinterpret_cast<uint16_t*>(base + h.otcoff) : nullptr;
  auto* d_fid = reinterpret_cast<uint16_t*>(base + h.ofid);
  auto* d_fpt = reinterpret_cast<int16_t*>(base + h.ofpt);
  auto* d_tab1 = reinterpret_cast<double*>(base + h.otab1);
  auto* d_order = reinterpret_cast<int32_t*>(base + h.oorder);
  auto* d_nested = reinterpret_cast<int32_t*>(base + h.onested);
  if (h.sf_ok) {
    const SfPlan& sf = h.sf;
    s->sf_ok = 1;
    s->sf_side = sf.side;
    s->sf_nks = sf.nks;
    s->sf_ngemv = sf.ngemv;
    for (int i = 0; i < 5; ++i) s->sf_gseg[i] = sf.gseg[i];
    s->sf_kw = sf.kw;
    s->sf_o_gw = sf.o_gw;
    s->sf_o_gops = sf.o_gops;
    s->sf_nepi = sf.nepi;
    s->sf_tmem = sf.tmem_cols;
    s->sf_bbytes = sf.bbytes;
    s->sf_smem = sf.smem;
    s->sf_bfloats = sf.bfloats_;
    s->sf_meta_bytes = sf.meta_bytes_;
    s->sf_o_aops = sf.o_aops;
    s->sf_o_epi = sf.o_epi;
    s->sf_o_prog = sf.o_prog;
    s->sf_o_pstart = sf.o_pstart;
    s->sf_meta = reinterpret_cast<unsigned char*>(base + h.ometa);
    s->sf_bmap = reinterpret_cast<int32_t*>(base + h.obmap);
    s->sf_b = reinterpret_cast<float*>(base + h.osfb);
  }
  auto cleanup = [&](cudaError_t err, const char* what) {
    sg_surplus_free(s);
    return err == cudaErrorMemoryAllocation ? fail(SG_ENOMEM, what) : cuda_fail(err, what);
  };
#define SG_TRY_CLEAN(expr)                                  \
  if ((e = (expr)) != cudaSuccess) return cleanup(e, #expr);
  // the host-made tables (cached), then this grid's box over their zero
  // bytes (written by k_fine_coords from its arguments)
  SurplusBox box{};
  for (int dim = 0; dim < d; ++dim) {
    box.v[dim] = g->h_lo[dim];
    box.v[d + dim] = g->h_hi[dim] - g->h_lo[dim];
  }
  SG_TRY_CLEAN(cudaMemcpyAsync(base + h.ohost, h.bytes(), h.off - h.ohost, cudaMemcpyHostToDevice, st));
  SG_TIMED("k_fine_coords", st,
           (k_fine_coords<<<static_cast<unsigned>(ceil_div(fine_n + 1 > 2 * d ? fine_n + 1 : 2 * d, 64)), 64, 0, st>>>(
               L, s->xf, box, 2 * d, s->box)));
  SG_TIMED("k_fine_table", st, (k_fine_table<<<static_cast<unsigned>(ceil_div(fine_n + 1, 64)), 64, 0, st>>>(L, s->xf, d_tab1)));
  SG_TRY_CLEAN(cudaGetLastError());
  for (size_t lv = 0; lv + 1 < h.level_start.size(); ++lv) {
    const int64_t n0 = h.level_start[lv], n1 = h.level_start[lv + 1];
    auto* kern = k <= 4 ? k_surplus_level<4> : k_surplus_level<kMaxOut>;
    SG_TIMED("k_surplus_level", st,
             (kern<<<static_cast<unsigned>(ceil_div(n1 - n0, kSurpWarps)), 32 * kSurpWarps, 0, st>>>(
                 n0, n1, d, k, fine_n, d_fid, d_fpt, d_tab1, d_values, s->W)));
    SG_TRY_CLEAN(cudaGetLastError());
  }
  SG_TIMED("k_gather_rows", st, (k_gather_rows<<<static_cast<unsigned>(ceil_div(std::max<int64_t>(M, h.nrows) * k, 256)), 256, 0, st>>>(M, h.nrows, k, d_order, d_nested, s->W, s->Ws, s->Wt)));
  SG_TRY_CLEAN(cudaGetLastError());
  if (split_df(fine_n + 1, s->xf, s->xfdf, st) != SG_OK || split_df(M * k, s->Ws, s->Wdf, st) != SG_OK)
    return cleanup(cudaGetLastError(), "split_df");
  SG_TRY_CLEAN(cudaMemsetAsync(s->tc_err, 0, sizeof(int), st));
  if (pack_tf32(s, st) != SG_OK) return cleanup(cudaGetLastError(), "pack_tf32");
  if (sf_pack(s, st) != SG_OK) return cleanup(cudaGetLastError(), "sf_pack");
#undef SG_TRY_CLEAN
  *out = s;
  return SG_OK;
}

extern "C" int sg_surplus_info(const sg_surplus* s, int64_t* n_nodes, int* k, const double** d_W) {
  clear_error();
  if (!s) return fail(SG_EINVAL, "sg_surplus_info: null handle");
  if (n_nodes) *n_nodes = s->M;
  if (k) *k = s->k;
  if (d_W) *d_W = s->W;
  return SG_OK;
}

extern "C" void sg_surplus_free(sg_surplus* s) {
  if (!s) return;
  block_free(s->block);
  delete s;
}

extern "C" int sg_eval_feedback(const sg_surplus* s, const double* d_xq, int64_t Q, int mode, double* d_out,
                                void* stream) {
  clear_error();
  if (!s) return fail(SG_EINVAL, "sg_eval_feedback: null handle");
  if (Q < 0) return fail(SG_EINVAL, "sg_eval_feedback: Q < 0");
  if (Q == 0) return SG_OK;
  if (!d_xq || !d_out) return fail(SG_EINVAL, "sg_eval_feedback: null device pointer");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  EvalArgs e{};
  e.xq = d_xq;
  e.Q = Q;
  e.M = s->M;
  e.k = s->k;
  e.nf = s->nf;
  e.level = s->level;
  e.amax = s->amax;
  e.nact = s->nact;
  e.ops = s->ops;
  e.W = s->Ws;
  e.Wt = s->Wt;
  e.prog = s->prog;
  e.nrows = s->nrows;
  e.per = s->per;
  e.fent = s->fent;
  e.fchild = s->fchild;
  e.nchild = s->nchild;
  std::copy(std::begin(s->range), std::end(s->range), e.range);
  std::copy(std::begin(s->fheight), std::end(s->fheight), e.fheight);
  std::copy(std::begin(s->froot), std::end(s->froot), e.froot);
  e.lo = s->box;
  e.width = s->box + s->d;
  e.xf = s->xf;
  e.xfdf = s->xfdf;
  e.Wdf = s->Wdf;
  for (int a = 0; a <= kMaxDim + 1; ++a) e.grp[a] = s->grp[a];
  e.out = d_out;
  if (mode == SG_EVAL_FP64) return eval_fp64(e, s->d, st);
  if (mode == SG_EVAL_TF32X3) return s->sf_ok ? eval_sf_tf32x3(e, s, st) : eval_tf32x3(e, s, st);
  if (mode == SG_EVAL_DF32) return eval_df32(e, s->d, st);
  return fail(SG_EINVAL, "sg_eval_feedback: unknown mode");
}
