// The FP64 Newton direction of the launch-per-phase and graph forms: stage
// condensation, elimination over the intervals and stage recovery.  All three
// are bound by the FP64 pipe (a warp's FP64 instruction holds it for 20
// cycles, whatever its active lanes), so the formulation is the one with the
// fewest FP64 operations, and rows are packed onto all 32 lanes.
//
// Condensation.  With the 2 x 2 inverse B of the interior block of the
// Lobatto IIIA matrix, B [[a22, a23], [a32, a33]] = I, the two interior stage
// rows of an interval become
//   (hJ2 - B11 I) dY2 - B12 dY3 = g1,    -B21 dY2 + (hJ3 - B22 I) dY3 = g2,
//   g_i = -s_i dy_i - alpha_i hJ1 dy_i - gamma_i hJ4 dy_{i+1} + rho_i
// (points 1..4 of the interval; s, alpha, gamma: scalars; rho: combinations
// of the residual rows): the blocks off the diagonal are multiples of the
// identity, so one 12 x 12 system is left of the 24 x 24 one,
//   C dY3 = G = (hJ2 - B11 I) g2 + B21 g1,  C = (hJ2 - B11 I)(hJ3 - B22 I) - B12 B21 I,
//   dY2 = ((hJ3 - B22 I) dY3 - g2) / B21,
// and the last stage row, in which hJ2 dY2 and hJ3 dY3 are replaced by the
// same combinations, needs only L G with L = E C^-1, E = c (hJ3 - B22 I) + d I.
// G is not formed: L G is the product of hJ1 and of hJ4 with a combination of
// L and L hJ2 each, two 12 x 12 products less.  That is 11,800 multiply-adds
// per interval (five 12 x 12 products 8,640, one 12 x 12 inversion with partial
// pivoting 1,584, the combinations 1,584; 9,360 without the attitude family's
// structural zeros) instead of the 23,000 of the elimination of the 24 interior
// columns, and what the recovery needs is C^-1 (144 numbers) instead of 24
// pivot rows (1,248).  The FP32 forms keep the
// elimination: a direction rounded otherwise moves their residuals near the
// tolerance by about a thousandth, and with them the iteration counts of one
// node in 5,000.
//
// Measured on the level-4 batch (1,457 nodes, horizons 10 / 20 / 40, six
// iterations): condensation 74.8 -> 21.7 ms (FP64 pipe 95 % busy), elimination
// and back substitution over the intervals 23.9 -> 8.5 ms, recovery 4.3 -> 1.8
// ms; the solve (a graph per mesh size) 112.0 -> 37.0 ms; 85 nodes at 128
// intervals 8.09 -> 2.92 ms.
//
// Elimination over the intervals.  An interval's condensed row
// S dy_i + double dy_{i+1} = r is solved for (dx_{i+1}, dlambda_i) in terms of
// (dx_i, dlambda_{i+1}): the scattering form of the two-point relation, whose
// composition (Redheffer's star product) does not grow along the mesh as
// products of transition matrices do.  Composing [a, m] and [m, b] solves one
// 6 x 6 system I - B_1 C_2 for (dx_m, dlambda_m) in terms of (dx_a,
// dlambda_b); a binary tree of compositions over the N intervals (depth
// log2 N) leaves the relation over [0, T], the boundary rows close it, and
// the tree is walked down for the mesh-point corrections.  Its rounding is that of
// the elimination: over eight linear-quadratic problems (64 intervals, |h J| up to
// 25), where one direction is the whole solve, lambda(0) is 1.5e-15 to 5.8e-15 off
// (the elimination's 1.7e-15 to 3.6e-15; either is the better one in four of them).
//
// A node with a pivot too small for the arithmetic, and a node whose full step
// does not pass the Armijo test (ls_node), take the direction of the elimination
// with full partial pivoting instead (the FP32 forms' algorithm in FP64).  The first
// has no scattering form; the second is far from its root, where the path of
// Newton's iteration depends on the last bits of the direction and whether it
// arrives is found out by following it.
#pragma once

#include "bvp_kernels.cuh"
#include "bvp_persistent.cuh"

namespace sg {

// Scalars of the combined stage rows, from a = A of Lobatto IIIA (closed
// forms in sqrt 5).
namespace lob {
constexpr double s5 = SG_S5;
constexpr double B11 = (25.0 + s5) / 7.0, B21 = -(25.0 + 13.0 * s5) / 7.0, B22 = (25.0 - s5) / 7.0;
constexpr double P12 = -220.0 / 49.0;                                              // B12 B21
constexpr double R2 = -120.0 / 7.0;                                                // B12 B21 - B11 B22
constexpr double S1 = 2.0 * s5;                                                    // s_1; s_2 = -s_1
constexpr double A1 = (17.0 * s5 - 5.0) / 70.0, A2 = -(17.0 * s5 + 5.0) / 70.0;    // alpha
constexpr double G1 = (3.0 * s5 - 5.0) / 70.0, G2 = -(3.0 * s5 + 5.0) / 70.0;      // gamma
constexpr double B12 = (13.0 * s5 - 25.0) / 7.0;
constexpr double CE = 5.0 * s5 / (25.0 + 13.0 * s5);                               // E = CE (hJ3 - B22 I) + C2 I
constexpr double C2 = 5.0 * s5 / 7.0;
constexpr double W1 = 5.0 / 12.0, W2 = 5.0 / 12.0 - CE;                            // factors of g1, g2 in the last row
constexpr double KD = -1.0 + W1 * S1 - W2 * S1;                                    // dy_i, hJ1 dy_i and hJ4 dy_{i+1}
constexpr double K0 = -1.0 / 12.0 + W1 * A1 + W2 * A2;
constexpr double K3 = -1.0 / 12.0 + W1 * G1 + W2 * G2;
}  // namespace lob

constexpr int kOp = 13 * 12;   // a scattering relation: columns (dx_a 6 | dlambda_b 6 | 1), rows (dx_b 6 | dlambda_a 6)
constexpr int kCi = 144;       // C^-1 of an interval, row-major

// n x Nmax x kCi inverses and n x Nmax x kOp relations share the region that
// holds the segments' pivot rows in the FP32 forms.
__host__ __device__ __forceinline__ double* dir_ci(const Workspace& w) { return static_cast<double*>(w.Seg); }
__host__ __device__ __forceinline__ double* dir_op(const SolveArgs& a, const Workspace& w) {
  return static_cast<double*>(w.Seg) + a.n * a.Nmax * int64_t(kCi);
}
static_assert(kCi + kOp <= kSegBlk, "the direction's arrays fit the region");

// 1/p for the pivots of the direction: Newton's iteration (one cubic step)
// from the approximate reciprocal instruction, which is good to about 20
// bits.  `good` is false for a small pivot or one that is not finite (the result
// is then 0).  The rows are of order one, and so are the pivots unless an
// interval or a composition is close to having no scattering form; the
// direction's error grows with the square of a pivot's reciprocal, to 1e-10 at
// the line drawn here.
__device__ __forceinline__ double dir_recip(double p, bool& good) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
  const double e = fma(-p, r, 1.0);
  r = fma(r, fma(e, e, e), r);
  const unsigned hi = static_cast<unsigned>(__double_as_longlong(p) >> 32) & 0x7FFFFFFFu;
  good = hi >= 0x3F500000u && hi < 0x7E300000u;   // 2^-10 .. 2^996
  return good ? r : 0.0;
}

__device__ __forceinline__ void mark_elim(const Workspace& w, int64_t node) {
  atomicOr(&w.ns[node].singular, kElimNode);
}
// Whether the tree forms the node's direction.  (kElimFirst, unlike kElimNode,
// does not change while these kernels run: the answer is the block's.)
__device__ __forceinline__ bool tree_node(const Workspace& w, int64_t node) {
  return w.ns[node].active && !(w.ns[node].singular & kElimFirst);
}

// n contiguous entries (16-byte vectors) from or to shared or global memory
template <int n>
__device__ __forceinline__ void ld_vec(const double* src, double (&r)[n]) {
  static_assert(n % 2 == 0, "whole vectors");
#pragma unroll
  for (int q = 0; q < n / 2; ++q) {
    const double2 v = reinterpret_cast<const double2*>(src)[q];
    r[2 * q] = v.x; r[2 * q + 1] = v.y;
  }
}
// vectors q0 .. of n entries
template <int n>
__device__ __forceinline__ void st_vec(double* dst, const double (&r)[n], int q0 = 0) {
  static_assert(n % 2 == 0, "whole vectors");
#pragma unroll
  for (int q = 0; q < n / 2; ++q)
    if (q >= q0) reinterpret_cast<double2*>(dst)[q] = make_double2(r[2 * q], r[2 * q + 1]);
}

// ---------------------------------------------------------------- condensation
// Eight intervals per block of 96 threads, a thread per row of an interval's
// 12-row matrices (every lane of the three warps a row; two intervals per
// warp would leave a quarter of the FP64 pipe's lanes idle); the other operand
// of every product is broadcast from shared memory.  Block barriers hide
// behind the FP64 pipe.
constexpr int kCondIv = 8;                       // intervals per block
constexpr int kCondThreads = 12 * kCondIv;
constexpr int kCondU = 28;                       // a published pivot row
// J (4 x 144), C^-1 (144), U (2), the residuals' two vectors (24), pivot keys and pivot rows (24 words)
constexpr int kCondElems = 576 + 144 + 2 * kCondU + 24 + 12;
constexpr int kCondSmem = kCondIv * kCondElems * 8;
__host__ __device__ __forceinline__ int cond_chunks(int Nmax) { return (Nmax + kCondIv - 1) / kCondIv; }

// Whether this thread's row holds the pivot: the largest |v| among the
// interval's candidate rows, ties to the lower row (the low four bits of the
// magnitude key are replaced by a row tag).  A block barrier.
__device__ __forceinline__ bool row_pivot(double v, bool cand, int row, unsigned* keys) {
  const unsigned key = cand ? ((mag_key(v) & ~15u) | unsigned(15 - row)) : 0u;
  keys[row] = key;
  __syncthreads();
  unsigned best = 0u;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const uint4 k = reinterpret_cast<const uint4*>(keys)[q];
    best = max(best, max(max(k.x, k.y), max(k.z, k.w)));
  }
  return cand && key == best;
}

// Entries (m, j) of the attitude family's Jacobian that are zero at every point:
// of f0_x (x' = E(v) w, w' = J^-1 (g(v) x w)), of -K (the controls enter the
// rates only), of the Hessian in the rates (lambda' f0 is linear in w) and of
// -f0_x'; 51 of 144.
__host__ __device__ constexpr bool attitude_zero(int m, int j) {
  if (m >= 6 && j >= 6) {   // -f0_x'
    const int t = m - 6;
    m = j - 6;
    j = t;
  }
  if (m < 6 && j < 6) {
    if (m >= 3) return j == m;
    return j == 2 || (m >= 1 && j == 3) || (m == 1 && j == 1);
  }
  if (m < 6) return m < 3 || j < 9;            // -K
  return m >= 9 && j >= 3 && m - 6 != j;       // l_ww + (lambda' f0)_ww
}

// kAtt: the attitude family, whose structural zeros are left out of the four
// products with the Jacobians (204 of 1,380 FP64 instructions; a term that is
// left out adds an exact zero).  Level-4 batch 42.8 -> 38.9 ms.
template <bool kAtt>
__global__ void __launch_bounds__(kCondThreads, 4) k_condense_fp64(SolveArgs a, Workspace w) {
  extern __shared__ __align__(16) unsigned char cond_smem[];
  const int chunks = cond_chunks(a.Nmax);
  const int64_t node = blockIdx.x / chunks;
  int i = static_cast<int>(blockIdx.x % chunks) * kCondIv;
  if (!tree_node(w, node)) return;
  const int N = a.N[node];
  if (i >= N) return;
  const int slot = threadIdx.x / 12, r = threadIdx.x % 12;
  // intervals past the mesh repeat the last one and store nothing
  const bool valid = i + slot < N;
  i = valid ? i + slot : N - 1;

  double* sm = reinterpret_cast<double*>(cond_smem) + slot * kCondElems;
  double* J_s = sm;                 // J of the four points
  double* Ci_s = sm + 576;
  double* U_s = Ci_s + 144;         // [2][28]
  double* rho_s = U_s + 2 * kCondU;
  unsigned* keys = reinterpret_cast<unsigned*>(rho_s + 24);
  int* perm_s = reinterpret_cast<int*>(keys + 12);

  const int64_t wid = node * a.Nmax + i;
  const double h = a.T[node] / N;
  {
    const double* J = static_cast<const double*>(w.Jm) + (node * npts(a.Nmax) + 3 * int64_t(i)) * 144;
#pragma unroll
    for (int e = 0; e < 576 / 2 / 12; ++e) cp_async16(J_s + (r + e * 12) * 2, J + (r + e * 12) * 2);
    cp_async_commit();
  }
  double res_c;   // the stage residuals' part that needs no product
  {
    const double* res = static_cast<const double*>(w.Res) + wid * kResRows;
    const double r1 = res[r], r2 = res[12 + r], r3 = res[24 + r];
    const double rho1 = lob::B11 * r1 + lob::B12 * r2, rho2 = lob::B21 * r1 + lob::B22 * r2;
    res_c = lob::W1 * rho1 + lob::W2 * rho2 - r3;
    rho_s[r] = h * rho2;
    rho_s[12 + r] = lob::R2 * r2;   // B21 rho_1 - B11 rho_2
  }
  cp_async_wait_all();
  __syncthreads();

  bool bad = false;
  // ---- C and its inverse (Gauss-Jordan in place, partial pivoting, rows
  // stay where they are)
  {
    double c[12];
    {
      double e1[12];
      ld_vec<12>(J_s + 144 + r * 12, e1);
#pragma unroll
      for (int j = 0; j < 12; ++j) {
        e1[j] = fma(h, e1[j], j == r ? -lob::B11 : 0.0);
        c[j] = fma(-lob::B22, e1[j], j == r ? -lob::P12 : 0.0);
        e1[j] *= h;
      }
#pragma unroll
      for (int m = 0; m < 12; ++m) {
        double u[12];
        ld_vec<12>(J_s + 288 + m * 12, u);
#pragma unroll
        for (int j = 0; j < 12; ++j)
          if (!(kAtt && attitude_zero(m, j))) c[j] = fma(e1[m], u[j], c[j]);
      }
    }
    bool cand = true;
    int my = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      double* U = U_s + (k & 1) * kCondU;
      const bool is_p = row_pivot(c[k], cand, r, keys);
      if (is_p) {
        st_vec<12>(U, c);
        perm_s[k] = r;
        my = k;
        cand = false;
#pragma unroll
        for (int j = 0; j < 12; ++j) c[j] = 0.0;
      }
      __syncthreads();
      bool good;
      double u[12];
      ld_vec<12>(U, u);
      const double inv = dir_recip(u[k], good);
      bad = bad || !good;
      // row r: c -= (c_k / p) u, c_k = -c_k / p; the pivot row: u / p, 1 / p
      const double l = is_p ? -inv : c[k] * inv;
#pragma unroll
      for (int j = 0; j < 12; ++j)
        if (j != k) c[j] = fma(-l, u[j], c[j]);
      c[k] = -l;
    }
    // register j of the row of step k is entry (k, pivot row of step j) of the inverse
#pragma unroll
    for (int j = 0; j < 12; ++j) Ci_s[my * 12 + perm_s[j]] = c[j];
  }
  __syncthreads();
  if (valid) {
    double* dst = dir_ci(w) + wid * kCi;
    for (int e = r; e < kCi / 2; e += 12) {
      double v[2];
      ld_vec<2>(Ci_s + e * 2, v);
      st_vec<2>(dst + e * 2, v);
    }
  }

  // ---- L = E C^-1 and L J2
  double L[12], M[12];
  {
    double e[12];
    ld_vec<12>(J_s + 288 + r * 12, e);
    const double ce = lob::CE * h;
#pragma unroll
    for (int j = 0; j < 12; ++j) {
      e[j] = fma(ce, e[j], j == r ? lob::C2 - lob::CE * lob::B22 : 0.0);
      L[j] = M[j] = 0.0;
    }
#pragma unroll
    for (int m = 0; m < 12; ++m) {
      double u[12];
      ld_vec<12>(Ci_s + m * 12, u);
#pragma unroll
      for (int j = 0; j < 12; ++j) L[j] = fma(e[m], u[j], L[j]);
    }
#pragma unroll
    for (int m = 0; m < 12; ++m) {
      double u[12];
      ld_vec<12>(J_s + 144 + m * 12, u);
#pragma unroll
      for (int j = 0; j < 12; ++j)
        if (!(kAtt && attitude_zero(m, j))) M[j] = fma(L[m], u[j], M[j]);
    }
  }

  // ---- the condensed row [S | T | r] as [T_x | S_lambda | -S_x | -T_lambda | r]:
  // with M = L (hJ2 - B11 I),
  //   S = (K0 I + alpha_2 M + B21 alpha_1 L) hJ1 + KD I - s_1 M + B21 s_1 L,
  //   T = (K3 I + gamma_2 M + B21 gamma_1 L) hJ4 + I
  double v[28];
  {
    const double cm = -lob::S1 * h, hK0 = lob::K0 * h, hK3 = lob::K3 * h, h2 = h * h;
    const double am = lob::A2 * h2, al = (lob::B21 * lob::A1 - lob::A2 * lob::B11) * h;
    const double gm = lob::G2 * h2, gl = (lob::B21 * lob::G1 - lob::G2 * lob::B11) * h;
    double t[12];
#pragma unroll
    for (int j = 0; j < 12; ++j)
      t[j] = fma(cm, M[j], fma(lob::S1 * (lob::B11 + lob::B21), L[j], j == r ? lob::KD : 0.0));
#pragma unroll
    for (int m = 0; m < 12; ++m) {
      double u[12];
      ld_vec<12>(J_s + m * 12, u);
      const double x = fma(am, M[m], fma(al, L[m], m == r ? hK0 : 0.0));
#pragma unroll
      for (int j = 0; j < 12; ++j)
        if (!(kAtt && attitude_zero(m, j))) t[j] = fma(x, u[j], t[j]);
    }
#pragma unroll
    for (int j = 0; j < 12; ++j) {
      if (j < 6) v[12 + j] = -t[j];
      else v[j] = t[j];
      t[j] = j == r ? 1.0 : 0.0;
    }
    double rr = res_c;
#pragma unroll
    for (int m = 0; m < 12; ++m) {
      double u[12];
      ld_vec<12>(J_s + 432 + m * 12, u);
      const double x = fma(gm, M[m], fma(gl, L[m], m == r ? hK3 : 0.0));
#pragma unroll
      for (int j = 0; j < 12; ++j)
        if (!(kAtt && attitude_zero(m, j))) t[j] = fma(x, u[j], t[j]);
      rr = fma(M[m], rho_s[m], fma(L[m], rho_s[12 + m], rr));
    }
#pragma unroll
    for (int j = 0; j < 12; ++j) {
      if (j < 6) v[j] = t[j];
      else v[12 + j] = -t[j];
    }
    v[24] = rr;
    v[25] = v[26] = v[27] = 0.0;
  }

  // ---- (dx_{i+1}, dlambda_i) from (dx_i, dlambda_{i+1}): Gauss-Jordan with
  // partial pivoting on the first 12 columns
  {
    bool cand = true;
    int my = 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      double* U = U_s + (k & 1) * kCondU;
      const bool is_p = row_pivot(v[k], cand, r, keys);
      if (is_p) {
        st_vec<28>(U, v, k / 2);
        my = k;
        cand = false;
#pragma unroll
        for (int j = k; j < 25; ++j) v[j] = 0.0;
      }
      __syncthreads();
      bool good;
      const double inv = dir_recip(U[k], good);
      bad = bad || !good;
      const double l = is_p ? -inv : v[k] * inv;
#pragma unroll
      for (int q = k / 2; q < (25 + 2 - 1) / 2; ++q) {
        double u[2];
        ld_vec<2>(U + q * 2, u);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int j = q * 2 + t;
          if (j > k && j < 25) v[j] = fma(-l, u[t], v[j]);
        }
      }
    }
    // column-major relation through shared memory (J is no longer read)
#pragma unroll
    for (int j = 0; j < 13; ++j) J_s[j * 12 + my] = v[12 + j];
    __syncthreads();
    if (valid) {
      double* dst = dir_op(a, w) + wid * kOp;
      for (int e = r; e < kOp / 2; e += 12) {
        double x[2];
        ld_vec<2>(J_s + e * 2, x);
        st_vec<2>(dst + e * 2, x);
      }
    }
  }
  if (bad && valid && r == 0) mark_elim(w, node);
}

// ---------------------------------------------------------------- tree
// Composition of o1 over [a, m] with o2 over [m, b] by 16 lanes, lane c < 13 a
// column (dx_a | dlambda_b | 1): km = (dx_m, dlambda_m), nw = the relation over
// [a, b].  The 6 x 6 matrix I - B_1 C_2 has its columns on lanes 0..5;
// elimination with partial pivoting, the pivot column (above it a column of the
// unit upper triangle, kept for the back substitution) passed through `pub`.
// All 32 lanes of the warp call it.  (FP64 instructions are its time: 219, with
// Gauss-Jordan and the identity and the right-hand side added apart 246.)
__device__ __forceinline__ void compose(const double* o1, const double* o2, double* pub, int c, double (&km)[12],
                                        double (&nw)[12], bool& bad) {
  double c2[12], c1[12], q[6], b[6];
  ld_vec<12>(o2 + c * 12, c2);   // A2 | B2 | f2 above C2 | D2 | e2
  ld_vec<12>(o1 + c * 12, c1);
  const bool left = c < 6, one = c == 12;
  // -I + B1 C2, B1 D2, f1 + B1 e2
#pragma unroll
  for (int t = 0; t < 6; ++t) q[t] = one ? c1[t] : (t == c ? -1.0 : 0.0);
#pragma unroll
  for (int m = 0; m < 6; ++m) {     // B1 times (C2 | D2 | e2)
    const double* col = o1 + (6 + m) * 12;
#pragma unroll
    for (int t = 0; t < 6; ++t) q[t] = fma(col[t], c2[6 + m], q[t]);
  }
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    b[t] = left ? c1[t] : q[t];
    q[t] = -q[t];
  }
  double up[6][6];   // up[k][t], t < k: the unit upper triangle
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double* p_s = pub + (k & 1) * 8;
    int p = k;
    unsigned best = mag_key(q[k]);
#pragma unroll
    for (int t = k + 1; t < 6; ++t) {
      const unsigned x = mag_key(q[t]);
      if (x > best) {
        best = x;
        p = t;
      }
    }
    if (c == k) {
#pragma unroll
      for (int t = 0; t < 6; ++t) p_s[t] = q[t];
      *reinterpret_cast<int*>(p_s + 6) = p;
    }
    __syncwarp();
    double l[6];
#pragma unroll
    for (int t = 0; t < 6; ++t) l[t] = p_s[t];
    p = *reinterpret_cast<const int*>(p_s + 6);
    double piv = l[k];
#pragma unroll
    for (int t = k + 1; t < 6; ++t) {
      if (p == t) {
        piv = l[t];
        l[t] = l[k];
        const double x = q[k], y = b[k];
        q[k] = q[t];
        q[t] = x;
        b[k] = b[t];
        b[t] = y;
      }
    }
    bool good;
    const double inv = dir_recip(piv, good);
    bad = bad || !good;
    q[k] *= inv;
    b[k] *= inv;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      if (t < k) up[k][t] = l[t];
      if (t > k) {
        q[t] = fma(-l[t], q[k], q[t]);
        b[t] = fma(-l[t], b[k], b[t]);
      }
    }
  }
#pragma unroll
  for (int k = 5; k > 0; --k)
#pragma unroll
    for (int t = 0; t < k; ++t) b[t] = fma(-up[k][t], b[k], b[t]);
  double y[12];
#pragma unroll
  for (int t = 0; t < 12; ++t) y[t] = left ? 0.0 : c2[t];
#pragma unroll
  for (int m = 0; m < 6; ++m) {     // (A2 | C2) dx_m
    double u[12];
    ld_vec<12>(o2 + m * 12, u);
#pragma unroll
    for (int t = 0; t < 12; ++t) y[t] = fma(u[t], b[m], y[t]);
  }
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    km[t] = b[t];
    km[6 + t] = y[6 + t];
    nw[t] = y[t];
    nw[6 + t] = (left || one) ? c1[6 + t] : 0.0;
  }
#pragma unroll
  for (int m = 0; m < 6; ++m) {     // D1 dlambda_m
    const double* col = o1 + (6 + m) * 12 + 6;
#pragma unroll
    for (int t = 0; t < 6; ++t) nw[6 + t] = fma(col[t], km[6 + m], nw[6 + t]);
  }
}

constexpr int kTreeMaxThreads = 512;
constexpr int kTreeGroupElems = 4 * kOp + 16;   // two pairs of relations in flight, pivot columns
constexpr int tree_smem(int threads) { return threads / 16 * kTreeGroupElems * 8; }
// Threads per block: many nodes fill the chip with small blocks; few nodes
// take the levels of their trees in fewer rounds.
inline int tree_threads(int64_t n, int Nmax) {
  int t = n >= 4 * kNumSMs ? 128 : (n >= kNumSMs ? 256 : kTreeMaxThreads);
  while (t > 32 && t / 16 >= Nmax) t /= 2;
  return t;
}

// The compositions of the relations [i0, i1) at strides st0, 2 st0, .. below
// st1, by the block's groups of 16 lanes.  A block barrier per stride.
__device__ __forceinline__ bool tree_up(double* ops, int i0, int i1, int st0, int st1, double* buf, double* pub, int c,
                                        int lane16, int g, int ng) {
  bool bad = false;
  auto fetch = [&](int i, int st, int b) {   // relations i and i + st to buffer b
    double* dst = buf + b * 2 * kOp;
    for (int e = lane16; e < 2 * kOp / 2; e += 16) {
      const double* src = ops + (e < kOp / 2 ? int64_t(i) * kOp + e * 2 : int64_t(i + st) * kOp + (e - kOp / 2) * 2);
      cp_async16(dst + e * 2, src);
    }
    cp_async_commit();
  };
  const int n = i1 - i0;
  for (int st = st0; st < n && st < st1; st *= 2) {
    const int pairs = (n - st + 2 * st - 1) / (2 * st);   // left ends i0 + 2 st j with 2 st j + st < n
    int b = 0;
    if (g < pairs) fetch(i0 + 2 * st * g, st, 0);
    for (int j0 = 0; j0 < pairs; j0 += ng, b ^= 1) {
      const int j = j0 + g;
      cp_async_wait_all();
      __syncwarp();
      if (j + ng < pairs) fetch(i0 + 2 * st * (j + ng), st, b ^ 1);
      if (j0 + (g & ~1) >= pairs) continue;   // the whole warp
      double km[12], nw[12];
      bool bd = false;
      compose(buf + b * 2 * kOp, buf + b * 2 * kOp + kOp, pub, c, km, nw, bd);
      if (j < pairs) {
        bad = bad || bd;
        if (lane16 < 13) {
          st_vec<12>(ops + int64_t(i0 + 2 * st * j) * kOp + c * 12, nw);
          st_vec<12>(ops + int64_t(i0 + 2 * st * j + st) * kOp + c * 12, km);
        }
      }
      __syncwarp();   // buffer b is fetched again in the next round
    }
    __syncthreads();
  }
  return bad;
}

// With fewer than two nodes per SM a block per node leaves SMs idle or unevenly
// loaded through the tree's lowest levels, which hold most of its work: then a
// block per kLeafIv intervals runs those first.  (85 nodes at 128 intervals: the
// tree 0.92 -> 0.72 ms, the solve 3.52 -> 3.31 ms; five blocks per SM, which
// the shared memory allows, with a few spills: 0.45 ms against 0.52; at 389 nodes of 64 intervals
// the solve would go from 1.29 to 1.31 ms, at 486 per graph from 41.9 to 43.3.)
constexpr int kLeafIv = 16;
__host__ __device__ __forceinline__ bool tree_leaves(int64_t n, int Nmax) {
  return n < 2 * kNumSMs && Nmax >= 2 * kLeafIv;
}
constexpr int kLeafThreads = kLeafIv / 2 * 16;   // a group per pair of intervals
__global__ void __launch_bounds__(kLeafThreads, 5) k_tree_leaf_fp64(SolveArgs a, Workspace w) {
  extern __shared__ __align__(16) unsigned char tree_smem_raw[];
  const int chunks = (a.Nmax + kLeafIv - 1) / kLeafIv;
  const int64_t node = blockIdx.x / chunks;
  const int i0 = static_cast<int>(blockIdx.x % chunks) * kLeafIv;
  if (!tree_node(w, node)) return;
  const int N = a.N[node];
  if (i0 >= N) return;
  const int tid = threadIdx.x, lane16 = tid & 15, g = tid >> 4;
  double* buf = reinterpret_cast<double*>(tree_smem_raw) + g * kTreeGroupElems;
  const bool bad = tree_up(dir_op(a, w) + node * a.Nmax * int64_t(kOp), i0, i0 + kLeafIv < N ? i0 + kLeafIv : N, 1,
                           kLeafIv, buf, buf + 4 * kOp, lane16 < 13 ? lane16 : 12, lane16, g, kLeafThreads / 16);
  if (__syncthreads_or(bad) && tid == 0) mark_elim(w, node);
}

// The node's line search starts: at the full step, or (marked here or before)
// after the first trial of the others with its elimination.
__device__ __forceinline__ void tree_ls_start(const Workspace& w, int64_t node, bool bad) {
  NodeState s = w.ns[node];
  if (!s.active) return;
  if (bad) s.singular |= kElimNode;
  s.searching = s.singular & (kElimNode | kElimFirst) ? 2 : 1;
  s.alpha = 1.0;
  w.ns[node] = s;
}

// Block per node.  Relations are composed in place: the result over [a, b)
// replaces the left operand, and the interior solution (dx_m, dlambda_m) of
// the composition takes the right operand's place, to be used on the way
// down.  The boundary rows x(0), lambda(T) close the tree as one more
// composition, with the relation (dlambda_N = H dx_N + eta).
__global__ void __launch_bounds__(kTreeMaxThreads, 1) k_tree_fp64(SolveArgs a, Workspace w) {
  extern __shared__ __align__(16) unsigned char tree_smem_raw[];
  const int64_t node = blockIdx.x;
  if (!tree_node(w, node)) {
    if (threadIdx.x == 0) tree_ls_start(w, node, false);
    return;
  }
  const int N = a.N[node];
  const int tid = threadIdx.x, lane16 = tid & 15, g = tid >> 4, ng = blockDim.x >> 4;
  const int c = lane16 < 13 ? lane16 : 12;
  double* buf = reinterpret_cast<double*>(tree_smem_raw) + g * kTreeGroupElems;   // [2][o1 | o2]
  double* pub = buf + 4 * kOp;
  double* ops = dir_op(a, w) + node * a.Nmax * int64_t(kOp);
  bool bad = tree_up(ops, 0, N, tree_leaves(a.n, a.Nmax) ? kLeafIv : 1, N, buf, pub, c, lane16, g, ng);

  // boundary rows
  const int64_t pb = node * npts(a.Nmax);
  double* D = w.D + pb * 12;
  if (tid < 32) {
    const double* Y = (w.ns[node].ybuf ? w.Y2 : w.Y) + pb * 12;
    const double* yN = Y + 3 * int64_t(N) * 12;
    double* o1 = reinterpret_cast<double*>(tree_smem_raw);
    double* o2 = o1 + kOp;
    for (int e = tid; e < kOp; e += 32) {
      o1[e] = ops[e];
      const int cc = e / 12, rr = e % 12 - 6;
      double x = 0.0;
      if (rr >= 0 && cc < 6) x = terminal_hess(a.P, rr, cc);
      if (rr >= 0 && cc == 12) x = -(yN[6 + rr] - terminal_grad(a.P, yN, rr));
      o2[e] = x;
    }
    __syncwarp();
    double km[12], nw[12];
    compose(o1, o2, o1 + 4 * kOp, c, km, nw, bad);
    __syncwarp();
    if (tid < 13) {
      st_vec<12>(o1 + c * 12, km);
      st_vec<12>(o2 + c * 12, nw);
    }
    __syncwarp();
    if (tid < 12) {
      const double* x0 = a.x0 + node * 6;
      double xi[6];
#pragma unroll
      for (int m = 0; m < 6; ++m) xi[m] = -(Y[m] - x0[m]);
      double yn = o1[144 + tid], y0 = o2[144 + tid];
#pragma unroll
      for (int m = 0; m < 6; ++m) {
        yn = fma(o1[m * 12 + tid], xi[m], yn);
        y0 = fma(o2[m * 12 + tid], xi[m], y0);
      }
#pragma unroll
      for (int m = 0; m < 6; ++m)
        if (m == tid) y0 = xi[m];
      D[3 * int64_t(N) * 12 + tid] = yn;
      D[tid] = y0;
    }
  }
  bad = __syncthreads_or(bad);
  if (tid == 0) tree_ls_start(w, node, bad);
  if (bad) return;   // the elimination solves it

  // down the tree: the corrections at the middle of [i, e) from those at its ends
  int top = 1;
  while (2 * top < N) top *= 2;
  if (N < 2) return;
  for (int st = top; st >= 1; st /= 2) {
    for (int j = g; 2 * st * j + st < N; j += ng) {
      const int i = 2 * st * j, m = i + st, e = i + 2 * st < N ? i + 2 * st : N;
      const double* K = ops + int64_t(m) * kOp;
      const int r = lane16 < 12 ? lane16 : 11;
      double k[13];
#pragma unroll
      for (int cc = 0; cc < 13; ++cc) k[cc] = K[cc * 12 + r];
      const double* ya = D + 3 * int64_t(i) * 12;
      const double* yb = D + 3 * int64_t(e) * 12;
      double y = k[12];
#pragma unroll
      for (int cc = 0; cc < 12; ++cc) y = fma(k[cc], cc < 6 ? ya[cc] : yb[cc], y);
      if (lane16 < 12) D[3 * int64_t(m) * 12 + r] = y;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- elimination
// Condensation by elimination of the 24 interior columns, segmented staircase,
// back substitution and recovery of the nodes that take the elimination's
// direction; launched only when there are some (in a graph, under h_elim).  A
// warp per interval, segment or node, in strides of a grid that fills the chip,
// so that one node's intervals are spread over it as well as many nodes'.  (The
// relations and inverses in the segments' region are no longer read when they
// run.)  Against a block of four warps per node: 85 nodes from states twice
// the box, twelve of them damped for 50 iterations, 215 -> 60 ms; 1,457 nodes of
// Example II's box 400 -> 136 ms.
__device__ __forceinline__ bool elim_node(const Workspace& w, int64_t node) {
  const NodeState& s = w.ns[node];
  return s.active && s.searching == 1 && (s.singular & (kElimNode | kElimDone)) == kElimNode;
}

constexpr int kElimCondWarps = 4, kElimSegWarps = 2, kElimRedWarps = 2, kElimBackWarps = 4, kElimRecWarps = 4;
constexpr int kElimCondSmem = kElimCondWarps * 36 * kCols * 8;
__global__ void __launch_bounds__(32 * kElimCondWarps) k_elim_condense_fp64(SolveArgs a, Workspace w) {
  extern __shared__ __align__(16) unsigned char elim_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* sm = reinterpret_cast<double*>(elim_smem) + warp * (36 * kCols);
  for (int64_t wid = blockIdx.x * int64_t(kElimCondWarps) + warp; wid < a.n * a.Nmax;
       wid += int64_t(gridDim.x) * kElimCondWarps) {
    const int64_t node = wid / a.Nmax;
    const int i = static_cast<int>(wid % a.Nmax);
    if (!elim_node(w, node) || i >= a.N[node]) continue;
    condense_interval_smem(a, w, node, i, a.N[node], lane, sm);
    __syncwarp();
  }
}

__global__ void __launch_bounds__(32 * kElimSegWarps) k_elim_seg_fp64(SolveArgs a, Workspace w) {
  __shared__ __align__(16) double sm[kElimSegWarps][seg_smem_elems<double>()];
  const int warp = threadIdx.x >> 5, smax = seg_count(a.Nmax);
  for (int64_t wid = blockIdx.x * int64_t(kElimSegWarps) + warp; wid < a.n * smax;
       wid += int64_t(gridDim.x) * kElimSegWarps) {
    const int64_t node = wid / smax;
    const int s = static_cast<int>(wid % smax);
    if (!elim_node(w, node) || s >= seg_count(a.N[node])) continue;
    abd_segment<double>(a, w, node, s, a.N[node], threadIdx.x & 31, sm[warp]);
    __syncwarp();
  }
}

__global__ void __launch_bounds__(32 * kElimRedWarps) k_elim_red_fp64(SolveArgs a, Workspace w) {
  __shared__ __align__(16) double sm[kElimRedWarps][stair_smem_elems<double>()];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t node = blockIdx.x * int64_t(kElimRedWarps) + warp; node < a.n;
       node += int64_t(gridDim.x) * kElimRedWarps) {
    if (!elim_node(w, node)) continue;
    abd_reduced<double>(a, w, node, a.N[node], lane, sm[warp]);
    __syncwarp();
    if (lane == 0 && (w.ns[node].singular & 1)) {
      w.ns[node].status = SG_SINGULAR;
      w.ns[node].active = 0;
      w.ns[node].searching = 0;
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(32 * kElimBackWarps) k_elim_segback_fp64(SolveArgs a, Workspace w) {
  __shared__ __align__(16) double sm[kElimBackWarps][kSegBackStages<double>][12 * kSegLd];
  const int warp = threadIdx.x >> 5, smax = seg_count(a.Nmax);
  for (int64_t wid = blockIdx.x * int64_t(kElimBackWarps) + warp; wid < a.n * smax;
       wid += int64_t(gridDim.x) * kElimBackWarps) {
    const int64_t node = wid / smax;
    const int s = static_cast<int>(wid % smax);
    if (!elim_node(w, node) || s >= seg_count(a.N[node])) continue;
    abd_segment_back<double>(a, w, node, s, a.N[node], threadIdx.x & 31, sm[warp]);
    __syncwarp();
  }
}

__global__ void __launch_bounds__(32 * kElimRecWarps) k_elim_recover_fp64(SolveArgs a, Workspace w) {
  for (int64_t wid = blockIdx.x * int64_t(kElimRecWarps) + (threadIdx.x >> 5); wid < a.n * a.Nmax;
       wid += int64_t(gridDim.x) * kElimRecWarps) {
    const int64_t node = wid / a.Nmax;
    const int i = static_cast<int>(wid % a.Nmax);
    if (!elim_node(w, node) || i >= a.N[node]) continue;
    recover_interval<double>(a, w, node, i, threadIdx.x & 31);
  }
}

// ---------------------------------------------------------------- recovery
// Interior-stage corrections from the mesh-point corrections: eight intervals
// per block of 96 threads, a thread per row (every lane of the three warps, as
// in the condensation: the FP64 pipe is its time); the Jacobians and C^-1 are
// staged in shared memory by asynchronous copies, the vectors pass through it.
// J dy at a mesh point serves the intervals on both sides.  (Two intervals per
// warp, 16 lanes each, both products per interval: 2.6 ms of the level-4 batch
// against 1.8.)
constexpr int kRecIv = kCondIv;
// J of the 3 kRecIv + 1 points, C^-1, dy and J dy at the kRecIv + 1 mesh points, three vectors per interval
constexpr int kRecElems = (3 * kRecIv + 1) * 144 + kRecIv * kCi + 2 * (kRecIv + 1) * 12 + 3 * kRecIv * 12;
constexpr int kRecSmem = kRecElems * 8;

__device__ __forceinline__ double dot12(const double* row, const double* vec) {
  double x[12], y[12];
  ld_vec<12>(row, x);
  ld_vec<12>(vec, y);
  double s = x[0] * y[0], t = x[1] * y[1];
#pragma unroll
  for (int m = 2; m < 12; m += 2) {
    s = fma(x[m], y[m], s);
    t = fma(x[m + 1], y[m + 1], t);
  }
  return s + t;
}

__global__ void __launch_bounds__(12 * kRecIv) k_recover_fp64(SolveArgs a, Workspace w) {
  extern __shared__ __align__(16) unsigned char rec_smem[];
  const int chunks = cond_chunks(a.Nmax);
  const int64_t node = blockIdx.x / chunks;
  const int i0 = static_cast<int>(blockIdx.x % chunks) * kRecIv;
  if (!w.ns[node].active || (w.ns[node].singular & (kElimNode | kElimFirst))) return;
  const int N = a.N[node];
  if (i0 >= N) return;
  const int nv = N - i0 < kRecIv ? N - i0 : kRecIv;
  const int tid = threadIdx.x, slot = tid / 12, r = tid % 12;
  const bool valid = slot < nv;
  const int q = valid ? slot : nv - 1;   // slots past the mesh repeat the last one and store nothing
  double* J_s = reinterpret_cast<double*>(rec_smem);
  double* Ci_s = J_s + (3 * kRecIv + 1) * 144;
  double* dy_s = Ci_s + kRecIv * kCi;            // [kRecIv + 1][12]
  double* u_s = dy_s + (kRecIv + 1) * 12;        // [kRecIv + 1][12] J dy
  double* g2_s = u_s + (kRecIv + 1) * 12;        // [kRecIv][12] each
  double* G_s = g2_s + kRecIv * 12;
  double* x_s = G_s + kRecIv * 12;
  const int64_t wid = node * a.Nmax + i0;
  const double* J = static_cast<const double*>(w.Jm) + (node * npts(a.Nmax) + 3 * int64_t(i0)) * 144;
  const double* Ci = dir_ci(w) + wid * kCi;
  for (int e = tid; e < (3 * nv + 1) * 72; e += 12 * kRecIv) cp_async16(J_s + e * 2, J + e * 2);
  for (int e = tid; e < nv * (kCi / 2); e += 12 * kRecIv) cp_async16(Ci_s + e * 2, Ci + e * 2);
  cp_async_commit();
  double* D = w.D + (node * npts(a.Nmax) + 3 * int64_t(i0)) * 12;
  const double d0 = D[36 * q + r];
  dy_s[q * 12 + r] = d0;
  if (q == nv - 1) dy_s[nv * 12 + r] = D[36 * nv + r];
  const double* res = static_cast<const double*>(w.Res) + (wid + q) * kResRows;
  const double r1 = res[r], r2 = res[12 + r];
  const double h = a.T[node] / N;
  cp_async_wait_all();
  __syncthreads();
  u_s[q * 12 + r] = h * dot12(J_s + 3 * q * 144 + r * 12, dy_s + q * 12);
  if (q == nv - 1) u_s[nv * 12 + r] = h * dot12(J_s + 3 * nv * 144 + r * 12, dy_s + nv * 12);
  __syncthreads();
  const double u0 = u_s[q * 12 + r], u3 = u_s[(q + 1) * 12 + r];
  const double g1 = lob::B11 * r1 + lob::B12 * r2 - lob::S1 * d0 - lob::A1 * u0 - lob::G1 * u3;
  const double g2 = lob::B21 * r1 + lob::B22 * r2 + lob::S1 * d0 - lob::A2 * u0 - lob::G2 * u3;
  g2_s[q * 12 + r] = g2;
  __syncthreads();
  const double G = h * dot12(J_s + (3 * q + 1) * 144 + r * 12, g2_s + q * 12) - lob::B11 * g2 + lob::B21 * g1;
  G_s[q * 12 + r] = G;
  __syncthreads();
  const double x = dot12(Ci_s + q * kCi + r * 12, G_s + q * 12);   // dY3
  x_s[q * 12 + r] = x;
  __syncthreads();
  const double y =
      (h * dot12(J_s + (3 * q + 2) * 144 + r * 12, x_s + q * 12) - lob::B22 * x - g2) * (1.0 / lob::B21);
  if (valid) {
    D[36 * q + 12 + r] = y;
    D[36 * q + 24 + r] = x;
  }
}

// The launches of a Newton direction (after the Jacobians): kernel, grid,
// block and shared memory of each, in order, for the host loop and the graphs
// (none where the grid is 0).
struct DirLaunch {
  const char* name;
  void (*fn)(SolveArgs, Workspace);
  int64_t grid;
  int block, smem;
};
template <typename T>
constexpr int kDirLaunches = sizeof(T) == sizeof(float) ? 5 : 4;

template <typename T>
inline void direction_launches(const SolveArgs& a, DirLaunch (&out)[kDirLaunches<T>]) {
  const int64_t nint = a.n * a.Nmax;
  if constexpr (sizeof(T) == sizeof(float)) {
    const int64_t nseg = a.n * seg_count(a.Nmax);
    const int cw = condense_reg_warps(a.cond_warps);
    out[0] = {"k_condense_reg_fp32", condense_reg_kernel(cw), ceil_div(nint, cw), 32 * cw, 0};
    out[1] = {"k_abd_seg_fp32", k_abd_seg, ceil_div(nseg, seg_warps<float>()), 32 * seg_warps<float>(), 0};
    out[2] = {"k_abd_red_fp32", k_abd_red, ceil_div(a.n, 4), 128, 0};
    out[3] = {"k_abd_segback_fp32", k_abd_segback, ceil_div(nseg, 4), 128, 0};
    out[4] = {"k_recover_fp32", k_recover_fp32, ceil_div(nint, 4), 128, 0};
  } else {
    const int tt = tree_threads(a.n, a.Nmax);
    out[0] = {"k_condense_fp64", a.P.kind == SG_PROBLEM_ATTITUDE ? k_condense_fp64<true> : k_condense_fp64<false>,
              a.n * cond_chunks(a.Nmax), kCondThreads, kCondSmem};
    out[1] = {"k_tree_leaf_fp64", k_tree_leaf_fp64,
              tree_leaves(a.n, a.Nmax) ? a.n * ((a.Nmax + kLeafIv - 1) / kLeafIv) : 0, kLeafThreads,
              tree_smem(kLeafThreads)};
    out[2] = {"k_tree_fp64", k_tree_fp64, a.n, tt, tree_smem(tt)};
    out[3] = {"k_recover_fp64", k_recover_fp64, a.n * cond_chunks(a.Nmax), 12 * kRecIv, kRecSmem};
  }
}

// The elimination's launches, for the trials of a line search that follow a
// reduction which counted nodes for it.
constexpr int kElimLaunches = 5;
inline void elim_launches(const SolveArgs& a, DirLaunch (&out)[kElimLaunches]) {
  const int64_t nint = a.n * a.Nmax, nseg = a.n * seg_count(a.Nmax);
  auto fill = [](int64_t warps, int per, int blocks_per_sm) {
    const int64_t all = ceil_div(warps, per), cap = int64_t(kNumSMs) * blocks_per_sm;
    return all < cap ? all : cap;
  };
  out[0] = {"k_elim_condense_fp64", k_elim_condense_fp64, fill(nint, kElimCondWarps, 4), 32 * kElimCondWarps,
            kElimCondSmem};
  out[1] = {"k_elim_seg_fp64", k_elim_seg_fp64, fill(nseg, kElimSegWarps, 8), 32 * kElimSegWarps, 0};
  out[2] = {"k_elim_red_fp64", k_elim_red_fp64, fill(a.n, kElimRedWarps, 8), 32 * kElimRedWarps, 0};
  out[3] = {"k_elim_segback_fp64", k_elim_segback_fp64, fill(nseg, kElimBackWarps, 7), 32 * kElimBackWarps, 0};
  out[4] = {"k_elim_recover_fp64", k_elim_recover_fp64, fill(nint, kElimRecWarps, 16), 32 * kElimRecWarps, 0};
}

// Raises the dynamic shared-memory caps of a direction's kernels.
template <typename T>
inline cudaError_t direction_setup(const SolveArgs& a) {
  DirLaunch d[kDirLaunches<T>];
  direction_launches<T>(a, d);
  for (auto& x : d) {
    const cudaError_t e = ensure_dynamic_smem(x.fn, x.smem);
    if (e != cudaSuccess) return e;
  }
  if constexpr (sizeof(T) == sizeof(double)) return ensure_dynamic_smem(k_elim_condense_fp64, kElimCondSmem);
  return cudaSuccess;
}

}  // namespace sg
