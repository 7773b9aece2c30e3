// One-dimensional hierarchical basis on nested Chebyshev-Gauss-Lobatto sets
// (Section 3.3): a^i_j is the Lagrange polynomial on X^i that is 1 at its
// point of dX^i, evaluated in barycentric form with the Chebyshev-Lobatto
// weights w_m = (-1)^m delta_m (delta = 1/2 at the ends) from the reciprocals
// 1/(u - x_p) of the finest set (every coarser set is a subset of it).
// FP64 form and pair-of-floats form (about 48 significant bits on the FP32
// pipe: exact products by FMA, Knuth's two_sum, corrected reciprocal).
#pragma once

#include "common.cuh"
#include "interp.cuh"

namespace sg {

// All 1-D basis values at one coordinate u in [0, 1] for levels 1..L+1,
// written to tab[id * stride].  xf holds the fine_n + 1 = 2^L + 1 points of
// the finest set X^{L+1}.  Exact Kronecker values when u coincides with a
// point of the level's set.
__device__ inline void basis_row(double u, int level, const double* __restrict__ xf, double* tab, int stride) {
  tab[0] = 1.0;   // a^1 = 1
  if (level == 0) return;
  const int fine_n = 1 << level;
  double rinv[kMaxFine + 1];
  int hit = -1;
  for (int p = 0; p <= fine_n; ++p) {
    const double diff = u - xf[p];
    if (diff == 0.0) hit = p;
    rinv[p] = diff == 0.0 ? 0.0 : 1.0 / diff;
  }
  int id = 1;
  for (int l = 2; l <= level + 1; ++l) {
    const int n = 1 << (l - 1);            // X^l has n + 1 points
    const int sf = fine_n / n;             // point m of X^l is fine point m * sf
    const bool exact = hit >= 0 && (hit % sf) == 0;
    double denom = 0.0;
    if (!exact) {
      for (int m = 0; m <= n; ++m) {
        double wm = (m & 1) ? -1.0 : 1.0;
        if (m == 0 || m == n) wm *= 0.5;
        denom += wm * rinv[m * sf];
      }
    }
    const double inv_denom = exact ? 0.0 : 1.0 / denom;
    // increment points of X^l: level 2 -> m = 0, n; level >= 3 -> odd m
    const int cnt = l == 2 ? 2 : (n >> 1);
    for (int j = 0; j < cnt; ++j) {
      const int m = l == 2 ? j * n : 2 * j + 1;
      double v;
      if (exact) {
        v = (m * sf == hit) ? 1.0 : 0.0;
      } else {
        double wm = (m & 1) ? -1.0 : 1.0;
        if (m == 0 || m == n) wm *= 0.5;
        v = wm * rinv[m * sf] * inv_denom;
      }
      tab[(id + j) * stride] = v;
    }
    id += cnt;
  }
}


// 1/x by Newton's iteration (one cubic step) from the approximate reciprocal
// instruction, which is good to about 20 bits: three FP64 operations and
// within one unit in the last place, where the correctly rounded reciprocal
// takes about seven.
__device__ __forceinline__ double recip_newton(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Whether the forms built on recip_newton hold at u: they need differences and
// reciprocals in the normal range, and denominators away from zero (far outside
// the box they are rounding noise, and an exact 0 would give NaN).  Elsewhere,
// and for NaN, basis_row.  On the integer pipe: u in (-1/4, 5/4), and 0 or at
// least 2^-1000 in size.
__device__ __forceinline__ bool basis_in_range(double u) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(u)), a = hi & 0x7FFFFFFFu;
  const bool inside = a < ((hi >> 31) ? 0x3FD00000u : 0x3FF40000u);
  return inside && (a >= 0x01700000u || (a | static_cast<unsigned>(__double2loint(u))) == 0u);
}

// The FP64 basis for a level fixed at compile time (every loop unrolls, the
// reciprocals stay in registers).  The denominators of the nested sets follow
// from one another: the points of X^l are the even points of X^{l+1}, so with P
// the sum of |w_m| / (u - x_m) over X^l and N the sum over the new points, the
// denominator of X^{l+1} is P - N and its own P is P + N.  Written out(id, v).
template <int L, typename Out>
__device__ __forceinline__ void basis_row_t(double u, const double* __restrict__ xf, Out out) {
  constexpr int fine_n = 1 << L;
  out(0, 1.0);
  double rinv[fine_n + 1];
  int hit = -1;
#pragma unroll
  for (int p = 0; p <= fine_n; ++p) {
    const double diff = u - xf[p];
    const bool zero = (static_cast<unsigned long long>(__double_as_longlong(diff)) << 1) == 0ull;
    if (zero) hit = p;
    const double r = recip_newton(diff);
    rinv[p] = zero ? 0.0 : r;
  }
  double P = 0.0;
  int id = 1;
#pragma unroll
  for (int l = 2; l <= L + 1; ++l) {
    const int n = 1 << (l - 1);
    const int sf = fine_n / n;
    const bool exact = hit >= 0 && (hit % sf) == 0;
    double nw, ends = 0.0;
    if (l == 2) {
      ends = 0.5 * (rinv[0] + rinv[fine_n]);
      nw = rinv[sf];
      P = ends;
    } else {
      nw = rinv[sf];
#pragma unroll
      for (int m = 3; m < n; m += 2) nw += rinv[m * sf];
    }
    const double inv = recip_newton(P - nw);
    P += nw;
    const int cnt = l == 2 ? 2 : (n >> 1);
    // increment points: l = 2 the two ends (weight +1/2), l >= 3 the odd points (weight -1)
    const double wi = l == 2 ? 0.5 * inv : -inv;
#pragma unroll
    for (int j = 0; j < cnt; ++j) {
      const int m = l == 2 ? j * n : 2 * j + 1;
      const double v = wi * rinv[m * sf];
      out(id + j, exact ? ((m * sf == hit) ? 1.0 : 0.0) : v);
    }
    id += cnt;
  }
}

// basis_row_t in three steps for a row spread over threads, the same operations
// in the same order: the reciprocals (zero at a hit), the factor of each level's
// values, the values.
__device__ __forceinline__ double basis_reciprocal(double u, double x, bool& zero) {
  const double diff = u - x;
  zero = diff == 0.0;
  const double r = recip_newton(diff);
  return zero ? 0.0 : r;
}
// rinv[p * stride], p = 0 .. 2^level, to wi[(l - 2) * stride], l = 2 .. level + 1
__device__ __forceinline__ void basis_factors(const double* rinv, int stride, int level, double* wi) {
  const int fine_n = 1 << level;
  double P = 0.5 * (rinv[0] + rinv[fine_n * stride]);
  for (int l = 2; l <= level + 1; ++l) {
    const int n = 1 << (l - 1), sf = fine_n / n;
    double nw = rinv[sf * stride];
    for (int m = 3; m < n; m += 2) nw += rinv[m * sf * stride];
    const double inv = recip_newton(P - nw);
    P += nw;
    wi[(l - 2) * stride] = l == 2 ? 0.5 * inv : -inv;
  }
}
// the value of function id >= 1; hit: the point that u coincides with, or -1
__device__ __forceinline__ double basis_value(const double* rinv, const double* wi, int stride, int level, int id,
                                              int hit) {
  const int fine_n = 1 << level;
  const int l = id <= 2 ? 2 : 33 - __clz(id - 1);                       // id - 1 = 2^(l - 2) + j
  const int sf = fine_n >> (l - 1);
  const int p = id <= 2 ? (id - 1) * fine_n : (2 * (id - 1 - (1 << (l - 2))) + 1) * sf;
  if (hit >= 0 && (hit & (sf - 1)) == 0) return p == hit ? 1.0 : 0.0;
  return wi[(l - 2) * stride] * rinv[p * stride];
}

// All 1-D basis values at u to tab[id * stride]: levels 1..5 in range unrolled,
// the others by the general form.
__device__ __forceinline__ void basis_row_fast(double u, int level, const double* __restrict__ xf, double* tab,
                                               int stride) {
  auto out = [&](int id, double v) { tab[id * stride] = v; };
  if (!basis_in_range(u)) level = -level;
  switch (level) {
    case 1: return basis_row_t<1>(u, xf, out);
    case 2: return basis_row_t<2>(u, xf, out);
    case 3: return basis_row_t<3>(u, xf, out);
    case 4: return basis_row_t<4>(u, xf, out);
    case 5: return basis_row_t<5>(u, xf, out);
    default: return basis_row(u, abs(level), xf, tab, stride);
  }
}


struct df {
  float hi, lo;
};

__device__ __forceinline__ df df_from(double x) {
  const float hi = __double2float_rn(x);
  return {hi, __double2float_rn(x - static_cast<double>(hi))};
}

__device__ __forceinline__ df df_norm(float s, float e) {
  const float hi = __fadd_rn(s, e);
  return {hi, __fsub_rn(e, __fsub_rn(hi, s))};
}

__device__ __forceinline__ df df_add(df a, df b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return df_norm(s, e);
}

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, {-b.hi, -b.lo}); }

__device__ __forceinline__ df df_mul(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_norm(p, e);
}

__device__ __forceinline__ df df_scale(df a, float s) {   // s exact power-of-two multiple of +-1
  return {__fmul_rn(a.hi, s), __fmul_rn(a.lo, s)};
}

__device__ __forceinline__ df df_recip(df a) {
  // the hardware's approximate reciprocal (a few ulp); the Newton correction
  // below takes the pair to the same accuracy as from a rounded one
  float q;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(a.hi));
  // residual 1 - a q, with a = hi + lo
  float r = __fmaf_rn(-a.hi, q, 1.0f);
  r = __fmaf_rn(-a.lo, q, r);
  return df_norm(q, __fmul_rn(q, r));
}

// All 1-D basis values at u (FP64 in [0,1]) for levels 1..L+1, as pairs, in
// barycentric form on the finest set (see basis_row in interp.cu).
// The same for a level fixed at compile time: every loop unrolls, so the
// reciprocals stay in registers (the general form indexes them at run time,
// which puts them in local memory).
template <int L, typename Out>
__device__ __forceinline__ void basis_row_df_t(double u, const float2* __restrict__ xf, Out out) {
  constexpr int fine_n = 1 << L;
  out(0, df{1.0f, 0.0f});
  const df uu = df_from(u);
  df rinv[fine_n + 1];
  int hit = -1;
#pragma unroll
  for (int p = 0; p <= fine_n; ++p) {
    const df d = df_sub(uu, {xf[p].x, xf[p].y});
    if (d.hi == 0.0f && d.lo == 0.0f) {
      hit = p;
      rinv[p] = {0.0f, 0.0f};
    } else {
      rinv[p] = df_recip(d);
    }
  }
  int id = 1;
#pragma unroll
  for (int l = 2; l <= L + 1; ++l) {
    const int n = 1 << (l - 1);
    const int sf = fine_n / n;
    const bool exact = hit >= 0 && (hit % sf) == 0;
    df inv_denom = {0.0f, 0.0f};
    if (!exact) {
      df den = {0.0f, 0.0f};
#pragma unroll
      for (int m = 0; m <= n; ++m) {
        float wm = (m & 1) ? -1.0f : 1.0f;
        if (m == 0 || m == n) wm *= 0.5f;
        den = df_add(den, df_scale(rinv[m * sf], wm));
      }
      inv_denom = df_recip(den);
    }
    const int cnt = l == 2 ? 2 : (n >> 1);
#pragma unroll
    for (int j = 0; j < cnt; ++j) {
      const int m = l == 2 ? j * n : 2 * j + 1;
      df v;
      if (exact) {
        v = {(m * sf == hit) ? 1.0f : 0.0f, 0.0f};
      } else {
        float wm = (m & 1) ? -1.0f : 1.0f;
        if (m == 0 || m == n) wm *= 0.5f;
        v = df_mul(df_scale(rinv[m * sf], wm), inv_denom);
      }
      out(id + j, v);
    }
    id += cnt;
  }
}

template <typename Out>
__device__ inline void basis_row_df_out(double u, int level, const float2* __restrict__ xf, Out out) {
  switch (level) {
    case 1: return basis_row_df_t<1>(u, xf, out);
    case 2: return basis_row_df_t<2>(u, xf, out);
    case 3: return basis_row_df_t<3>(u, xf, out);
    case 4: return basis_row_df_t<4>(u, xf, out);
    case 5: return basis_row_df_t<5>(u, xf, out);
    default: break;
  }
  out(0, df{1.0f, 0.0f});
  if (level == 0) return;
  const int fine_n = 1 << level;
  const df uu = df_from(u);
  df rinv[kMaxFine + 1];
  int hit = -1;
  for (int p = 0; p <= fine_n; ++p) {
    const df d = df_sub(uu, {xf[p].x, xf[p].y});
    if (d.hi == 0.0f && d.lo == 0.0f) {
      hit = p;
      rinv[p] = {0.0f, 0.0f};
    } else {
      rinv[p] = df_recip(d);
    }
  }
  int id = 1;
  for (int l = 2; l <= level + 1; ++l) {
    const int n = 1 << (l - 1);
    const int sf = fine_n / n;
    const bool exact = hit >= 0 && (hit % sf) == 0;
    df inv_denom = {0.0f, 0.0f};
    if (!exact) {
      df den = {0.0f, 0.0f};
      for (int m = 0; m <= n; ++m) {
        float wm = (m & 1) ? -1.0f : 1.0f;
        if (m == 0 || m == n) wm *= 0.5f;
        den = df_add(den, df_scale(rinv[m * sf], wm));
      }
      inv_denom = df_recip(den);
    }
    const int cnt = l == 2 ? 2 : (n >> 1);
    for (int j = 0; j < cnt; ++j) {
      const int m = l == 2 ? j * n : 2 * j + 1;
      df v;
      if (exact) {
        v = {(m * sf == hit) ? 1.0f : 0.0f, 0.0f};
      } else {
        float wm = (m & 1) ? -1.0f : 1.0f;
        if (m == 0 || m == n) wm *= 0.5f;
        v = df_mul(df_scale(rinv[m * sf], wm), inv_denom);
      }
      out(id + j, v);
    }
    id += cnt;
  }
}

// Product of a pair with a pair, left unnormalised: the result (p, e) has
// p = fl(a.hi b.hi) and e = the exact rounding error of p plus the cross
// terms, so p + e carries the product to about 2^-46 relative.  Skipping the
// renormalisation is safe because |e| stays below about 2^-22 |p| and every
// consumer (the next product, the compensated dot) treats hi and lo only
// through products and exact sums.
__device__ __forceinline__ df df_mul_raw(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return {p, e};
}

// Writers of basis_row_df_out: the pairs, or their leading floats (the
// values rounded once to FP32).
struct DfPairOut {
  float2* tab;
  int stride;
  __device__ __forceinline__ void operator()(int id, df v) const { tab[id * stride] = make_float2(v.hi, v.lo); }
};
struct DfHiOut {
  float* tab;
  int stride;
  __device__ __forceinline__ void operator()(int id, df v) const { tab[id * stride] = v.hi; }
};

__device__ inline void basis_row_df(double u, int level, const float2* __restrict__ xf, float2* tab, int stride) {
  basis_row_df_out(u, level, xf, DfPairOut{tab, stride});
}

__device__ inline void basis_row_df_hi(double u, int level, const float2* __restrict__ xf, float* tab,
                                       int stride) {
  basis_row_df_out(u, level, xf, DfHiOut{tab, stride});
}

}  // namespace sg
