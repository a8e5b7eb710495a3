// Eigenvectors of the symmetric tridiagonal T (Eigh(T) of Algorithm 1): inverse
// iteration with partial-pivoting LU in double-float, modified Gram-Schmidt
// within clusters of close eigenvalues.
#pragma once

#include <cfloat>

#include "tridiag.cuh"

namespace sls {

// Eigenvectors of one cluster [first, last] of nearly equal Ritz values of
// a T of order n, written as columns of S: inverse iteration with
// partial-pivoting LU of T - shift I in double-float, two iterations, each
// followed by modified Gram-Schmidt against the cluster members already found.
// The recurrences carry their running values in registers (the factorisation the
// current pivot row, the solves the last one or two entries), so a step's
// dependent chain holds no memory access; pivoting selects operands instead of
// branching; the first forward solve rides along the factorisation; and the back
// substitution multiplies by the pivots' reciprocals.  The work arrays (n entries
// each) belong to the caller.  WARP: a warp's lanes share the loops over entries of
// arrays in shared memory; else one thread runs them (sums over n as four
// interleaved partial sums).
SLS_DEV dfloat sum4_df(dfloat (&acc)[4]) {
  return df_add(df_add(acc[0], acc[1]), df_add(acc[2], acc[3]));
}

// A power-of-two scale of T (the eigenvectors do not change):
// 1 / 2^ceil(log2 |T|), |T| from the extreme Ritz values.
SLS_DEV double eig_scale(const double* th, int n, double* tnorm_out) {
  const double tnorm = fmax(fabs(th[0]), fabs(th[n - 1])) + DBL_MIN;
  int ex = 0;
  frexp(tnorm, &ex);
  *tnorm_out = tnorm;
  return ldexp(1.0, -ex);
}

// The scaled diagonal sa[i] = a_i sc and off-diagonal sb[i] = b_i sc as
// double-float, entries i = t, t + nt, ... for the nt calling threads (t = their
// index): every eigenvector of the problem starts from them, and the float64
// products and splits, whose dependent latency is long on this part, run once
// per problem and in parallel.
SLS_DEV void eig_scaled_T(const double* a, const double* b, int n, double sc, int t, int nt,
                          float2* __restrict__ sa, float2* __restrict__ sb) {
  for (int i = t; i < n; i += nt) {
    sa[i] = f2(df_from_double(a[i] * sc));
    if (i < n - 1) sb[i] = f2(df_from_double(b[i] * sc));
  }
}

// LU of T - shift I with the forward solve of the running right-hand side y:
// d the pivots' reciprocals, du and du2 the rows of U, dl the multipliers, piv the
// interchanges.  Returns the last entry of the solved right-hand side.
template <typename Y0>
SLS_DEV dfloat eig_factor(int n, dfloat shift, dfloat pert, Y0 y0, const float2* __restrict__ sa,
                          const float2* __restrict__ sb, float2* __restrict__ d,
                          float2* __restrict__ du, float2* __restrict__ du2,
                          float2* __restrict__ dl, float2* __restrict__ y,
                          unsigned char* __restrict__ piv) {
  const dfloat one = df_make(1.f, 0.f), zero = df_make(0.f, 0.f);
  // cd, cu: the current pivot row's diagonal and superdiagonal entries as the
  // elimination has left them; cy: the running right-hand side
  dfloat cd = df_sub(dfv(sa[0]), shift), cu = dfv(sb[0]), cy = df_make(y0(0), 0.f);
  for (int i = 0; i < n - 1; ++i) {
    const dfloat li = dfv(sb[i]);
    const dfloat dn = df_sub(dfv(sa[i + 1]), shift);
    const dfloat un = (i < n - 2) ? dfv(sb[i + 1]) : zero;
    const dfloat yn = df_make(y0(i + 1), 0.f);
    const bool sw = !(fabsf(cd.hi) >= fabsf(li.hi));
    if (!sw && cd.hi == 0.f) cd = pert;
    const dfloat den = sw ? li : cd;
    const dfloat f = df_div(sw ? cd : li, den);
    const dfloat u1 = sw ? dn : cu, u2 = sw ? un : zero, ya = sw ? yn : cy;
    d[i] = f2(df_div(one, den));
    dl[i] = f2(f);
    du[i] = f2(u1);
    du2[i] = f2(u2);
    y[i] = f2(ya);
    piv[i] = sw ? 1 : 0;
    cd = df_sub(sw ? cu : dn, df_mul(f, u1));
    cy = df_sub(sw ? cy : yn, df_mul(f, ya));
    cu = sw ? df_neg(df_mul(f, un)) : un;
  }
  if (cd.hi == 0.f) cd = pert;
  d[n - 1] = f2(df_div(one, cd));
  return cy;
}

// Forward solve with the row interchanges; returns the last entry.
SLS_DEV dfloat eig_forward(int n, const float2* __restrict__ dl, float2* __restrict__ y,
                           const unsigned char* __restrict__ piv) {
  dfloat cy = dfv(y[0]);
  for (int i = 0; i < n - 1; ++i) {
    const dfloat yn = dfv(y[i + 1]);
    const bool sw = piv[i] != 0;
    const dfloat ya = sw ? yn : cy;
    y[i] = f2(ya);
    cy = df_sub(sw ? cy : yn, df_mul(dfv(dl[i]), ya));
  }
  return cy;
}

// Back substitution from the last entry cy; c1, c2: y[i + 1], y[i + 2].
SLS_DEV void eig_back(int n, dfloat cy, const float2* __restrict__ d,
                      const float2* __restrict__ du, const float2* __restrict__ du2,
                      float2* __restrict__ y) {
  dfloat c1 = df_mul(cy, dfv(d[n - 1])), c2 = df_make(0.f, 0.f);
  y[n - 1] = f2(c1);
  for (int i = n - 2; i >= 0; --i) {
    dfloat t = df_sub(dfv(y[i]), df_mul(dfv(du[i]), c1));
    if (i < n - 2) t = df_sub(t, df_mul(dfv(du2[i]), c2));
    c2 = c1;
    c1 = df_mul(t, dfv(d[i]));
    y[i] = f2(c1);
  }
}

// Deterministic start vector of column mm, entry i.
SLS_DEV float eig_start(int mm, int i) {
  unsigned h = (unsigned)(i + 1) * 2654435761u ^ (unsigned)(mm + 7) * 40503u;
  h ^= h >> 13;
  h *= 0x5bd1e995u;
  h ^= h >> 15;
  return 0.5f + (float)(h & 0xffffu) / 65536.f;
}

// The shift of column mm of the cluster that starts at column first: distinct
// inside a cluster.
SLS_DEV dfloat eig_shift(const double* th, int mm, int first, double pert, double sc) {
  return df_from_double((th[mm] - (double)(mm - first) * 4.0 * pert) * sc);
}

// Keep the iterate y in range (divide by its largest entry, a power of two).
template <bool WARP>
SLS_DEV void eig_rescale(int n, float2* __restrict__ y) {
  const int i0 = WARP ? (threadIdx.x & 31) : 0;
  constexpr int di = WARP ? 32 : 1;
  float ymax = 0.f;
  for (int i = i0; i < n; i += di) ymax = fmaxf(ymax, fabsf(y[i].x));
  if (WARP)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ymax = fmaxf(ymax, __shfl_xor_sync(0xffffffffu, ymax, o));
  if (ymax > 0.f && isfinite(ymax)) {
    int e2 = 0;
    frexpf(ymax, &e2);
    const float s2 = ldexpf(1.f, -e2);
    for (int i = i0; i < n; i += di) y[i] = f2(df_scale(dfv(y[i]), s2));
  }
}

// Orthogonalise y against columns first .. mm - 1 of S, the cluster members found
// so far, and normalise it.
template <bool WARP>
SLS_DEV void eig_orthonormalise(int n, int r, int first, int mm, const double* __restrict__ S,
                                float2* __restrict__ y) {
  const int i0 = WARP ? (threadIdx.x & 31) : 0;
  constexpr int di = WARP ? 32 : 1;
  auto dot_all = [&](auto term) {  // sum of term(i) over i < n
    if constexpr (WARP) {
      dfloat acc = df_make(0.f, 0.f);
      for (int i = i0; i < n; i += di) acc = df_add(acc, term(i));
      return warp_sum_df(acc);
    } else {
      dfloat acc[4] = {df_make(0.f, 0.f), df_make(0.f, 0.f), df_make(0.f, 0.f),
                       df_make(0.f, 0.f)};
      for (int i = 0; i < n; ++i) acc[i & 3] = df_add(acc[i & 3], term(i));
      return sum4_df(acc);
    }
  };
  for (int pm = first; pm < mm; ++pm) {
    const dfloat dot =
        dot_all([&](int i) { return df_mul(df_from_double(S[(size_t)i * r + pm]), dfv(y[i])); });
    for (int i = i0; i < n; i += di)
      y[i] = f2(df_sub(dfv(y[i]), df_mul(dot, df_from_double(S[(size_t)i * r + pm]))));
  }
  const double nr =
      sqrt(df_to_double(dot_all([&](int i) { return df_mul(dfv(y[i]), dfv(y[i])); })));
  if (!(nr > 0.0) || !isfinite(nr)) {
    for (int i = i0; i < n; i += di) y[i] = make_float2((i == mm) ? 1.f : 0.f, 0.f);
  } else {
    const dfloat inv = df_from_double(1.0 / nr);
    for (int i = i0; i < n; i += di) y[i] = f2(df_mul(dfv(y[i]), inv));
  }
}

// Column mm of S from y, its first entry made non-negative.
template <bool WARP>
SLS_DEV void eig_store(int n, int r, int mm, const float2* __restrict__ y,
                       double* __restrict__ S) {
  const double sg = (y[0].x < 0.f) ? -1.0 : 1.0;
#pragma unroll 4
  for (int i = WARP ? (threadIdx.x & 31) : 0; i < n; i += WARP ? 32 : 1)
    S[(size_t)i * r + mm] = sg * df_to_double(dfv(y[i]));
}

// The cluster [first, last] by one warp, on arrays in shared memory: lane 0 runs the
// recurrences (the solves are in place: a second lane running them alike would read
// entries that the first has already overwritten), all lanes share the loops over
// entries, and they meet between the two.
SLS_DEV void eigvec_cluster(int r, const double* th, double* S, int n, int first, int last,
                            double sc, double tnorm, const float2* __restrict__ sa,
                            const float2* __restrict__ sb, float2* __restrict__ d,
                            float2* __restrict__ du, float2* __restrict__ du2,
                            float2* __restrict__ dl, float2* __restrict__ y,
                            unsigned char* __restrict__ piv) {
  const int lane = threadIdx.x & 31;
  const double pert = 0x1p-44 * tnorm;
  const dfloat pert_df = df_from_double(pert * sc);
  for (int mm = first; mm <= last; ++mm) {
    if (n == 1) {
      if (lane == 0) y[0] = make_float2(1.f, 0.f);
      __syncwarp();
    } else {
      for (int it = 0; it < 2; ++it) {
        if (lane == 0) {
          const dfloat cy =
              it == 0 ? eig_factor(n, eig_shift(th, mm, first, pert, sc), pert_df,
                                   [mm](int i) { return eig_start(mm, i); }, sa, sb, d, du, du2,
                                   dl, y, piv)
                      : eig_forward(n, dl, y, piv);
          eig_back(n, cy, d, du, du2, y);
        }
        __syncwarp();
        eig_rescale<true>(n, y);
        eig_orthonormalise<true>(n, r, first, mm, S, y);
        __syncwarp();
      }
    }
    eig_store<true>(n, r, mm, y, S);
    __syncwarp();
  }
}

// Cluster bounds of eigenvalue m: [first, last] with neighbours closer than
// 1e-7 * |T| merged (the eigenvectors of a cluster are computed together).
SLS_DEV void eig_cluster(const double* th, int n, int m, int& first, int& last) {
  const double tnorm = fmax(fabs(th[0]), fabs(th[n - 1])) + DBL_MIN;
  const double ctol = 1e-7 * tnorm;
  first = m;
  while (first > 0 && th[first - 1] - th[first] <= ctol) --first;
  last = m;
  while (last + 1 < n && th[last] - th[last + 1] <= ctol) ++last;
}

}  // namespace sls
