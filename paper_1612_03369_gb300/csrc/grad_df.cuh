// grad_df.cuh -- the velocity gradient G = du_h/dx = (du_h/dx-hat) J^{-1} at a
// located point, in double-float arithmetic on the FP32 pipe (the FP64 pipe
// of GB300 issues ~1/75 of the FP32 rate).  Used by the property ODEs of
// Sec. 2.6 and by the adjoint sweep.
//
//   du/dx-hat   from the cell's monomial coefficients about its centre
//               (u_c = sum c_pqr s0^p s1^q s2^r, s = x-hat - 1/2, so
//               d/dx-hat = d/ds): Horner steps that carry each partial
//               sum's value and its derivatives along the axes already
//               passed
//   J           from the cell's monomial block (the map about vertex 0,
//               Phi = X_0 + sum_k a_k m_k(t)): J_ij = sum_k a_k,i dm_k/dt_j
//   J^{-1}      cofactors over the determinant, one double-float reciprocal
// Every product is a double-float product (two_prod), every sum a
// double-float sum, so G carries ~2^-44 relative error times the
// conditioning of J.
#pragma once

#include "df.cuh"
#include "fastpath.cuh"

namespace pic {

struct LdgLoader {
  __device__ __forceinline__ float4 ld(const float4* p) const { return __ldg(p); }
};

// 1 / a: FP32 reciprocal refined by one Newton step in double-float.
__device__ __forceinline__ df df_recip(df a) {
  const float r = __frcp_rn(a.hi);
  const df p = two_prod(a.hi, r);                  // a.hi r exactly
  const float e = __fsub_rn(__fsub_rn(1.0f, p.hi), __fmaf_rn(a.lo, r, p.lo));  // 1 - a r
  return fast_two_sum(r, __fmul_rn(r, e));
}

// Gu[c][j] = d u_c / d t_j in cell K at double-float reference coordinates
// t, from the cell's coefficient slices (u_c = sum_r slice_r(s0, s1) s2^r,
// s = t - 1/2).  In a slice each row q has its value h = c_0 + s0 (c_1 + s0 c_2)
// and its derivative along s0, h' = c_1 + 2 c_2 s0; the rows combine along s1
// to the slice's value g and derivatives g0 (along s0) and g1 = h_1 + 2 h_2 s1;
// along s2 the slices combine the same way.
template <int D>
__device__ __forceinline__ void q2_grad_mono_df(const float4* __restrict__ Qc, uint32_t K, const df t[D],
                                                df Gu[D][D]) {
  constexpr int NS = (D == 3 ? 3 : 1);
  const LdgLoader ld;
  df s[D];
#pragma unroll
  for (int a = 0; a < D; ++a) s[a] = centred(t[a]);
  const float4* cell = Qc + (size_t)K * D * (5 * NS);
#pragma unroll 1
  for (int comp = 0; comp < D; ++comp) {
    const float4* cq = cell + comp * (5 * NS);
    df g0, g1, g2;  // sums over the slices so far: the derivatives along s0, s1 and s2
#pragma unroll
    for (int r = NS - 1; r >= 0; --r) {
      float hi[10], lo[10];
      load_slice(ld, cq + 5 * r, hi, lo);
      auto c = [&](int k) { return df_make(hi[k], lo[k]); };
      df h[3], h0[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (D == 2 || r > 0 || q > 0) h[q] = df_horner(df_horner(c(3 * q + 2), s[0], c(3 * q + 1)), s[0], c(3 * q));
        h0[q] = df_horner(df_scale2(c(3 * q + 2), 2.0f), s[0], c(3 * q + 1));
      }
      const df r0 = df_horner(df_horner(h0[2], s[1], h0[1]), s[1], h0[0]);
      const df r1 = df_horner(df_scale2(h[2], 2.0f), s[1], h[1]);
      g0 = r == NS - 1 ? r0 : df_horner(g0, s[D - 1], r0);
      g1 = r == NS - 1 ? r1 : df_horner(g1, s[D - 1], r1);
      if constexpr (D == 3) {
        if (r == 0) continue;
        const df v = df_horner(df_horner(h[2], s[1], h[1]), s[1], h[0]);
        g2 = r == 2 ? df_scale2(v, 2.0f) : df_horner(g2, s[2], v);
      }
    }
    Gu[comp][0] = df_norm(g0);
    Gu[comp][1] = df_norm(g1);
    if constexpr (D == 3) Gu[comp][2] = df_norm(g2);
  }
}

// J_ij = dPhi_i/dt_j from the monomial block: in 3D the monomials are
// (t0, t1, t2, t0 t1, t0 t2, t1 t2, t0 t1 t2), in 2D (t0, t1, t0 t1).
template <int D, class Ld>
__device__ __forceinline__ void map_jacobian_df(const Ld& ld, const float4* B, const df t[D], df J[D][D]) {
  df t01, t02, t12;
  if constexpr (D == 3) {
    t01 = df_mul(t[0], t[1]);
    t02 = df_mul(t[0], t[2]);
    t12 = df_mul(t[1], t[2]);
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const MapRow<D> hi = load_row<D>(ld, B, 0, i), lo = load_row<D>(ld, B, 1, i);
    auto a = [&](int k) { return df_make(hi.a[k], lo.a[k]); };
    if constexpr (D == 3) {
      df_acc j0 = acc_init(a(0)), j1 = acc_init(a(1)), j2 = acc_init(a(2));
      acc_mad(j0, a(3), t[1]);
      acc_mad(j0, a(4), t[2]);
      acc_mad(j0, a(6), t12);
      acc_mad(j1, a(3), t[0]);
      acc_mad(j1, a(5), t[2]);
      acc_mad(j1, a(6), t02);
      acc_mad(j2, a(4), t[0]);
      acc_mad(j2, a(5), t[1]);
      acc_mad(j2, a(6), t01);
      J[i][0] = acc_result(j0);
      J[i][1] = acc_result(j1);
      J[i][2] = acc_result(j2);
    } else {
      df_acc j0 = acc_init(a(0)), j1 = acc_init(a(1));
      acc_mad(j0, a(2), t[1]);
      acc_mad(j1, a(2), t[0]);
      J[i][0] = acc_result(j0);
      J[i][1] = acc_result(j1);
    }
  }
}

// a b - c d
__device__ __forceinline__ df df_det2(df a, df b, df c, df d) {
  df_acc s = acc_zero();
  acc_mad(s, a, b);
  acc_mad(s, c, df_make(-d.hi, -d.lo));
  return acc_result(s);
}

template <int D>
__device__ __forceinline__ void invert_df(const df J[D][D], df Ji[D][D]) {
  if constexpr (D == 2) {
    const df inv = df_recip(df_det2(J[0][0], J[1][1], J[0][1], J[1][0]));
    Ji[0][0] = df_mul(J[1][1], inv);
    Ji[0][1] = df_mul(df_make(-J[0][1].hi, -J[0][1].lo), inv);
    Ji[1][0] = df_mul(df_make(-J[1][0].hi, -J[1][0].lo), inv);
    Ji[1][1] = df_mul(J[0][0], inv);
  } else {
    df c[3][3];
    c[0][0] = df_det2(J[1][1], J[2][2], J[1][2], J[2][1]);
    c[0][1] = df_det2(J[1][2], J[2][0], J[1][0], J[2][2]);
    c[0][2] = df_det2(J[1][0], J[2][1], J[1][1], J[2][0]);
    c[1][0] = df_det2(J[0][2], J[2][1], J[0][1], J[2][2]);
    c[1][1] = df_det2(J[0][0], J[2][2], J[0][2], J[2][0]);
    c[1][2] = df_det2(J[0][1], J[2][0], J[0][0], J[2][1]);
    c[2][0] = df_det2(J[0][1], J[1][2], J[0][2], J[1][1]);
    c[2][1] = df_det2(J[0][2], J[1][0], J[0][0], J[1][2]);
    c[2][2] = df_det2(J[0][0], J[1][1], J[0][1], J[1][0]);
    df_acc det = acc_zero();
    acc_mad(det, J[0][0], c[0][0]);
    acc_mad(det, J[0][1], c[0][1]);
    acc_mad(det, J[0][2], c[0][2]);
    const df inv = df_recip(acc_result(det));
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int q = 0; q < 3; ++q) Ji[r][q] = df_mul(c[q][r], inv);
  }
}

// z = J^{-T} v by double-float cofactors.  Out of line: the cells that
// solve_transposed_df cannot serve.
template <int D>
struct DfVec {
  df v[D];
};
template <int D>
__device__ __noinline__ DfVec<D> solve_transposed_cofactors_df(const MeshView& m, uint32_t K, DfVec<D> t, DfVec<D> v) {
  df J[D][D], Ji[D][D];
  map_jacobian_df<D>(LdgLoader(), m.blk + (size_t)K * block_float4s<D>(), t.v, J);
  invert_df<D>(J, Ji);
  DfVec<D> z;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    df_acc acc = acc_zero();
#pragma unroll
    for (int j = 0; j < D; ++j) acc_mad(acc, Ji[j][i], v.v[j]);
    z.v[i] = acc_result(acc);
  }
  return z;
}

// z = J^{-T} v in double-float, J = dPhi/dt at t in cell K: the FP32 inverse's
// solution and two corrections by the double-float residual v - J^T z, each of
// which takes the error down by the FP32 inverse's own, some 1e-7 times the
// condition of J (double-float cofactors and their product with the field's
// gradient took 660 operations, this 390).  The first correction shows that
// factor: above 2^-16 of z, where two of them would leave more than the
// cofactors do (a cell sheared to a condition of a few hundred), and where FP32
// has no inverse, the cofactors take over.  The inverse's entries, of order
// 1 / h, multiply the residual; cofactors would take it down by h^(D-1) first.
// The residuals go down to 2^-48 of v: the caller scales v where it may be small.
template <int D>
__device__ __forceinline__ void solve_transposed_df(const MeshView& m, uint32_t K, const df t[D], const df v[D],
                                                    df z[D]) {
  const LdgLoader ld;
  const float4* B = m.blk + (size_t)K * block_float4s<D>();
  df J[D][D];
  map_jacobian_df<D>(ld, B, t, J);
  float J32[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) J32[i][j] = J[i][j].hi;
  Adjugate32<D> A;
  bool ok = adjugate32<D>(J32, A);
  if (ok) {
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
      for (int j = 0; j < D; ++j) A.c[i][j] = __fmul_rn(A.c[i][j], A.inv);  // (J^{-T})_ij
#pragma unroll
    for (int i = 0; i < D; ++i) z[i] = df_make(0.f, 0.f);
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
      float r[D], first = 0.f, total = 0.f;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        df_acc acc = acc_init(v[j]);
#pragma unroll
        for (int i = 0; i < D; ++i) {
          if (pass == 1) acc_mad_f(acc, J[i][j], -z[i].hi);
          if (pass == 2) acc_mad(acc, J[i][j], df_make(-z[i].hi, -z[i].lo));
        }
        r[j] = __fadd_rn(acc.s, acc.e);
      }
#pragma unroll
      for (int i = 0; i < D; ++i) {
        float q = __fmul_rn(A.c[i][0], r[0]);
#pragma unroll
        for (int j = 1; j < D; ++j) q = __fmaf_rn(A.c[i][j], r[j], q);
        if (pass == 1) {
          first = __fadd_rn(first, fabsf(q));  // sums: not a number if any is not
          total = __fadd_rn(total, fabsf(z[i].hi));
        }
        z[i] = pass == 0 ? df_make(q, 0.f) : (pass == 1 ? two_sum(z[i].hi, q) : df_add(z[i], df_make(q, 0.f)));
      }
      if (pass == 1) ok = first <= 0x1p-16f * total;
    }
  }
  if (!ok) {
    DfVec<D> tv, vv;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      tv.v[i] = t[i];
      vv.v[i] = v[i];
    }
    const DfVec<D> zv = solve_transposed_cofactors_df<D>(m, K, tv, vv);
#pragma unroll
    for (int i = 0; i < D; ++i) z[i] = zv.v[i];
  }
}

// A power of two that takes values of magnitude up to `largest` near 1, and its
// inverse (both normal floats).
__device__ __forceinline__ void pow2_near_one(float largest, float& scale, float& back) {
  const int e = min(max(__float_as_int(largest) & 0x7f800000, 1 << 23), 253 << 23);
  scale = __int_as_float((254 << 23) - e);
  back = __int_as_float(e);
}

// G = du_h/dx at double-float reference coordinates t of cell K.
template <int D>
__device__ __forceinline__ void velocity_gradient_df(const MeshView& m, uint32_t K, const df t[D], df G[D][D]) {
  df Gu[D][D], J[D][D], Ji[D][D];
  q2_grad_mono_df<D>(m.Qc, K, t, Gu);
  map_jacobian_df<D>(LdgLoader(), m.blk + (size_t)K * block_float4s<D>(), t, J);
  invert_df<D>(J, Ji);
#pragma unroll
  for (int c = 0; c < D; ++c)
#pragma unroll
    for (int q = 0; q < D; ++q) {
      df_acc s = acc_zero();
#pragma unroll
      for (int j = 0; j < D; ++j) acc_mad(s, Gu[c][j], Ji[j][q]);
      G[c][q] = acc_result(s);
    }
}

// sqrt(a), a >= 0: FP32 root refined by one Newton step in double-float.
__device__ __forceinline__ df df_sqrt(df a) {
  if (!(a.hi > 0.f)) return df_make(0.f, 0.f);
  const float r = __fsqrt_rn(a.hi);
  const df r2 = two_prod(r, r);
  const float e = __fdiv_rn(__fadd_rn(__fsub_rn(a.hi, r2.hi), __fsub_rn(a.lo, r2.lo)), __fmul_rn(2.0f, r));
  return fast_two_sum(r, e);
}

}  // namespace pic
