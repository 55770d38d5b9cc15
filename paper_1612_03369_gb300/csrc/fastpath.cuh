// fastpath.cuh -- the advection hot path in double-float arithmetic on the
// FP32 pipe (Sec. 2.3 velocity evaluation, Sec. 2.4 location).
//
// Layouts (built once per mesh / velocity field):
//   cell block   per cell, the (bi/tri)linear map in monomial form about
//                vertex 0: Phi_K(t) = X_0 + sum_k a_k m_k(t) with
//                m = (t0, t1, t2, t0 t1, t0 t2, t1 t2, t0 t1 t2) in 3D and
//                (t0, t1, t0 t1) in 2D; X_0 and every a_k as double-floats
//                (192 B per hex, 64 B per quad, 16-byte aligned), the high
//                parts of every component's row (X_0, a_1, ...), then the low
//                parts of every row
//   U2           Q2 nodal values as double-floats, node-major [node][dim]
//                (the source of the coefficient slices below)
//
// Qc, the Q2 field's per-cell monomial coefficients about the cell centre
// (double-float, 720 B per hex), and Qf, their high parts alone for the
// FP32-basis form (336 B per hex), are built with the field (mesh.cu).
//
// Where a cell's blocks are read from is a template parameter: GlobalCells
// reads the mesh arrays; StagedCells a shared-memory copy of the cells a
// warp's particles start in (advect.cu), and the mesh arrays for any other
// cell.  The arithmetic is the same either way, so every kernel that inlines
// it computes the same bits.
//
// Inverse map (Newton, Sec. 2.2 / Remark 2.1): FP32 iterations on the local
// offset y - X_0 until the iterate is within ~2e-7 of the root, then one Newton
// step whose residual (y - X_0) - sum_k a_k m_k(t) is evaluated in double-float
// (absolute accuracy ~2^-47 h), with the FP32 Jacobian at the current iterate.
// That leaves |t - t*| ~ 1e-13.  A point the FP32 phase does not settle is left
// to the rare paths, where the FP64 Newton of pic_internal.cuh stands behind
// each cell.
#pragma once

#include "df.cuh"
#include "locate.cuh"
#include "pic_internal.cuh"

namespace pic {

// FP32 phase ends when max|update| <= kSettle32: the iterate is then within
// ~C*kSettle32^2 + 1e-7 of the root (C ~ 1 for cells jittered by 10%), and
// the double-float step takes that to ~C*(2e-7)^2 + 3e-7*2e-7 ~ 1e-13 (the
// FP32 Jacobian and the approximate reciprocal of solve32 scale the update).
constexpr float kSettle32 = 2e-4f;
constexpr int kMaxIt32 = 8;
// Ends the FP32 phase after a step with the second-order term q: the error
// left, ~2 |q|^2 / |d|, is then below 2e-9, well under the FP32 residual's own noise
// of ~1e-7.  (At a hundred times that, and kFinish32 at 1e-6, it showed: x of 6^3 cells
// 2.44e-16 rms off instead of 2.2e-16, dL/dU of 4^3 1.71e-15 instead of 1.5e-15, for
// no gain in time.)
constexpr float kSettleCheb32 = 1e-9f;
// A settled FP32 iterate this far outside [0,1] is still taken to the
// double-float step, which decides (the two differ by a few 1e-7).
constexpr float kInside32 = 5e-7f;
// Largest double-float step after which the root is taken as found: the FP32
// Jacobian leaves ~3e-7 of the step (at 2e-7 the FP32 phase's noise alone has it
// repeated: 2 % of the 64^3 step).
constexpr float kFinish32 = 4e-7f;
// Largest first double-float step of a root that is taken further: the FP32
// iterate is off by ~1e-7 times the condition of the Jacobian (~1e-7 in cells
// jittered by 10 %, 1e-4 in ones sheared 30 to 1).
constexpr float kStart32 = 1e-2f;

// One component's row of the map block (the high or the low parts).
template <int D>
struct MapRow {
  float x0;
  float a[(1 << D) - 1];
};

template <int D>
__host__ __device__ constexpr int block_float4s() {
  return (2 * D + 2 * D * ((1 << D) - 1)) / 4;  // 12 (3D) or 4 (2D)
}
// float4 per cell of Qc: per component NS slices of 5 float4 (ten high
// parts, then ten low parts; the tenth of each is zero).
template <int D>
__host__ __device__ constexpr int qc_float4s() {
  return D * 5 * (D == 3 ? 3 : 1);  // 45 (3D) or 10 (2D)
}
// Qf: per component the 3^D high parts in the order r*9 + q*3 + p (the
// coefficient of s2^r s1^q s0^p), padded to 28 (3D) or 12 (2D) floats.
template <int D>
__host__ __device__ constexpr int qf_floats_per_comp() {
  return D == 3 ? 28 : 12;
}
template <int D>
__host__ __device__ constexpr int qf_float4s() {
  return D * qf_floats_per_comp<D>() / 4;  // 21 (3D) or 6 (2D)
}

// ------------------------------------------------------ cell data source --

template <int D, bool F32B>
struct GlobalCells {
  static constexpr int NB = block_float4s<D>();
  static constexpr int NQ = F32B ? qf_float4s<D>() : qc_float4s<D>();
  const MeshView& m;
  __device__ __forceinline__ const float4* block(uint32_t K) const { return m.blk + (size_t)K * NB; }
  __device__ __forceinline__ const float4* coef(uint32_t K) const { return (F32B ? m.Qf : m.Qc) + (size_t)K * NQ; }
  __device__ __forceinline__ float4 ld(const float4* p) const { return __ldg(p); }
};

// Cells [K0, K0 + n) from shared memory (sbase: their map blocks in order,
// then from sbase + kStage * NB their coefficient blocks), every other cell
// from the mesh arrays.  Loads are generic, so one instruction serves both.
template <int D, bool F32B, int kStage>
struct StagedCells {
  static constexpr int NB = block_float4s<D>();
  static constexpr int NQ = F32B ? qf_float4s<D>() : qc_float4s<D>();
  const MeshView& m;
  const float4* sbase;
  uint32_t K0, n;
  __device__ __forceinline__ const float4* block(uint32_t K) const {
    const uint32_t o = K - K0;
    return o < n ? sbase + o * NB : m.blk + (size_t)K * NB;
  }
  __device__ __forceinline__ const float4* coef(uint32_t K) const {
    const uint32_t o = K - K0;
    return o < n ? sbase + kStage * NB + o * NQ : (F32B ? m.Qf : m.Qc) + (size_t)K * NQ;
  }
  __device__ __forceinline__ float4 ld(const float4* p) const { return *p; }
};

// Component c's row of the map block at B, high (half 0) or low parts (half 1).
// The code that uses the rows takes them one at a time, so that it never holds
// more than one component's coefficients in registers.
template <int D, class Cells>
__device__ __forceinline__ MapRow<D> load_row(const Cells& cs, const float4* B, int half, int c) {
  constexpr int NR = (1 << D) / 4;  // float4 per row
  const float4* p = B + (half * D + c) * NR;
  float f[1 << D];
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const float4 v = cs.ld(p + q);
    f[4 * q] = v.x;
    f[4 * q + 1] = v.y;
    f[4 * q + 2] = v.z;
    f[4 * q + 3] = v.w;
  }
  MapRow<D> r;
  r.x0 = f[0];
#pragma unroll
  for (int k = 0; k < (1 << D) - 1; ++k) r.a[k] = f[1 + k];
  return r;
}

// Monomials of degree >= 2 at t: t0 t1 (2D); t0 t1, t0 t2, t1 t2, t0 t1 t2 (3D).
template <int D>
__device__ __forceinline__ void mixed32(const float t[D], float m[4]) {
  m[0] = __fmul_rn(t[0], t[1]);
  if constexpr (D == 3) {
    m[1] = __fmul_rn(t[0], t[2]);
    m[2] = __fmul_rn(t[1], t[2]);
    m[3] = __fmul_rn(m[0], t[2]);
  }
}

// One component of the FP32 map offset phi(t) = sum_k a_k m_k(t).
template <int D>
__device__ __forceinline__ float map_row32(const MapRow<D>& w, const float t[D], const float m[4]) {
  if constexpr (D == 2) return __fmaf_rn(w.a[2], m[0], __fmaf_rn(w.a[1], t[1], __fmul_rn(w.a[0], t[0])));
  else
    return __fmaf_rn(
        w.a[6], m[3],
        __fmaf_rn(w.a[5], m[2],
                  __fmaf_rn(w.a[4], m[1],
                            __fmaf_rn(w.a[3], m[0],
                                      __fmaf_rn(w.a[2], t[2], __fmaf_rn(w.a[1], t[1], __fmul_rn(w.a[0], t[0])))))));
}

// One row of the FP32 Jacobian.
template <int D>
__device__ __forceinline__ void jacobian_row32(const MapRow<D>& w, const float t[D], const float m[4], float J[D]) {
  if constexpr (D == 2) {
    J[0] = __fmaf_rn(w.a[2], t[1], w.a[0]);
    J[1] = __fmaf_rn(w.a[2], t[0], w.a[1]);
  } else {
    J[0] = __fmaf_rn(w.a[6], m[2], __fmaf_rn(w.a[4], t[2], __fmaf_rn(w.a[3], t[1], w.a[0])));
    J[1] = __fmaf_rn(w.a[6], m[1], __fmaf_rn(w.a[5], t[2], __fmaf_rn(w.a[3], t[0], w.a[1])));
    J[2] = __fmaf_rn(w.a[6], m[0], __fmaf_rn(w.a[5], t[1], __fmaf_rn(w.a[4], t[0], w.a[2])));
  }
}

// J^{-1} as adjugate times reciprocal determinant, applied to any number of
// right-hand sides.  Every operation is an explicit rounded intrinsic, in a
// fixed order, so that every kernel inlining this (the advect kernel's template
// instances, the stage-recording kernel, the adjoint's stage kernel) computes
// the same iterates bit for bit, whatever the compiler would contract on its
// own.  The determinant's reciprocal is the hardware approximation (one
// instruction, within 2 ulp; the IEEE division took a dozen): it scales a
// Newton update whose last, double-float-residual step is ~1e-7, so it moves
// the root by ~3e-14, the size of the FP32 Jacobian's own error.  A zero or
// non-finite determinant fails; so does one of 2^126 and more, for which that
// reciprocal is 0 and the update with it; one so small that its reciprocal
// overflows gives an update the caller rejects (|d| > 1e3).
template <int D>
struct Adjugate32 {
  float c[D][D];  // cofactors: (J^{-1})_ij = c[j][i] inv
  float inv;
};

template <int D>
__device__ __forceinline__ bool adjugate32(const float J[D][D], Adjugate32<D>& A) {
  auto det2 = [](float a, float b, float c, float e) { return __fmaf_rn(a, b, -__fmul_rn(c, e)); };  // a b - c e
  if constexpr (D == 2) {
    const float det = det2(J[0][0], J[1][1], J[0][1], J[1][0]);
    if (!(fabsf(det) > 0.f && fabsf(det) < 0x1p126f)) return false;
    A.inv = __fdividef(1.0f, det);
    A.c[0][0] = J[1][1];
    A.c[0][1] = -J[1][0];
    A.c[1][0] = -J[0][1];
    A.c[1][1] = J[0][0];
  } else {
    A.c[0][0] = det2(J[1][1], J[2][2], J[1][2], J[2][1]);
    A.c[0][1] = det2(J[1][2], J[2][0], J[1][0], J[2][2]);
    A.c[0][2] = det2(J[1][0], J[2][1], J[1][1], J[2][0]);
    const float det = __fmaf_rn(J[0][2], A.c[0][2], __fmaf_rn(J[0][1], A.c[0][1], __fmul_rn(J[0][0], A.c[0][0])));
    if (!(fabsf(det) > 0.f && fabsf(det) < 0x1p126f)) return false;
    A.inv = __fdividef(1.0f, det);
    A.c[1][0] = det2(J[0][2], J[2][1], J[0][1], J[2][2]);
    A.c[1][1] = det2(J[0][0], J[2][2], J[0][2], J[2][0]);
    A.c[1][2] = det2(J[0][1], J[2][0], J[0][0], J[2][1]);
    A.c[2][0] = det2(J[0][1], J[1][2], J[0][2], J[1][1]);
    A.c[2][1] = det2(J[0][2], J[1][0], J[0][0], J[1][2]);
    A.c[2][2] = det2(J[0][0], J[1][1], J[0][1], J[1][0]);
  }
  return true;
}

template <int D>
__device__ __forceinline__ void apply32(const Adjugate32<D>& A, const float r[D], float d[D]) {
#pragma unroll
  for (int i = 0; i < D; ++i) {
    if constexpr (D == 2)  // c[0][i] r0 - (-c[1][i]) r1, each product rounded as in a 2 x 2 determinant
      d[i] = __fmul_rn(i == 0 ? __fmaf_rn(A.c[0][0], r[0], -__fmul_rn(-A.c[1][0], r[1]))
                              : __fmaf_rn(A.c[1][1], r[1], -__fmul_rn(-A.c[0][1], r[0])),
                       A.inv);
    else
      d[i] = __fmul_rn(__fmaf_rn(A.c[2][i], r[2], __fmaf_rn(A.c[1][i], r[1], __fmul_rn(A.c[0][i], r[0]))), A.inv);
  }
}

template <int D>
__device__ __forceinline__ bool solve32(const float J[D][D], const float r[D], float d[D]) {
  Adjugate32<D> A;
  if (!adjugate32<D>(J, A)) return false;
  apply32<D>(A, r, d);
  return true;
}

// The part of Phi_K(t + d) - Phi_K(t) beyond J d, exact for the (bi/tri)linear
// map: sum over the mixed monomials, FP32.
template <int D, class Cells>
__device__ __forceinline__ void second_order32(const Cells& cs, const float4* B, const float t[D], const float d[D],
                                               float w[D]) {
  if constexpr (D == 2) {
    const float d01 = __fmul_rn(d[0], d[1]);
#pragma unroll
    for (int c = 0; c < 2; ++c) w[c] = __fmul_rn(cs.ld(B + c).w, d01);
  } else {
    const float d01 = __fmul_rn(d[0], d[1]), d02 = __fmul_rn(d[0], d[2]), d12 = __fmul_rn(d[1], d[2]);
    const float d012 = __fmul_rn(d01, d[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float4 v = cs.ld(B + 2 * c + 1);  // a_t0t1, a_t0t2, a_t1t2, a_t0t1t2
      const float p = __fmul_rn(__fmaf_rn(v.w, t[2], v.x), d01);
      const float q = __fmaf_rn(__fmaf_rn(v.w, t[1], v.y), d02, p);
      w[c] = __fmaf_rn(v.w, d012, __fmaf_rn(__fmaf_rn(v.w, t[0], v.z), d12, q));
    }
  }
}

// One component of the double-float residual dloc - sum_k a_k m_k(t) at a
// single-float point t (mixed monomials m formed exactly with two_prod; hi, lo
// the component's row).
template <int D>
__device__ __forceinline__ float residual_row_df(const MapRow<D>& hi, const MapRow<D>& lo, df dloc, const float t[D],
                                                 const df m[4]) {
  auto A = [&](int k) { return df_make(-hi.a[k], -lo.a[k]); };
  df_acc acc = acc_init(dloc);
#pragma unroll
  for (int a = 0; a < D; ++a) acc_mad_f(acc, A(a), t[a]);
#pragma unroll
  for (int k = D; k < (1 << D) - 1; ++k) acc_mad(acc, A(k), m[k - D]);
  return __fadd_rn(acc.s, acc.e);
}

template <int D>
__device__ __forceinline__ void mixed_df(const float t[D], df m[4]) {
  m[0] = two_prod(t[0], t[1]);
  if constexpr (D == 3) {
    m[1] = two_prod(t[0], t[2]);
    m[2] = two_prod(t[1], t[2]);
    m[3] = df_mul_f(m[0], t[2]);
  }
}

// Outcome of the inverse map in one cell.
enum : int { kCellOut = 0, kCellIn = 1, kCellFail = -1 };

// Returned instead of a cell by the fast-path-only locate (kFast == true)
// where the full locate would enter a rare path (the FP64 Newton, the
// lowest-index test of the cells across a nearby facet, the FP64 walk): the
// caller hands the particle to a second kernel that runs the full step.  A
// kernel without those out-of-line calls needs no spill code around them.
constexpr uint32_t kDefer = 0xFFFFFFFEu;

// Points and results passed by value to and from the out-of-line rare paths,
// so that no variable of the hot loop has its address taken (an address-
// taken variable lives in local memory for its whole life).
template <int D>
struct DfPt {
  df v[D];
};
template <int D>
struct RarePath {
  DfPt<D> t;       // reference coordinates found
  uint32_t K;      // cell found (PIC_LOST: none)
  int r;           // kCellIn / kCellOut / kCellFail (single-cell tests)
  int iters;       // Newton iterations spent
  unsigned flags;  // flags raised
};
template <int D>
__device__ __forceinline__ DfPt<D> pack(const df a[D]) {
  DfPt<D> p;
#pragma unroll
  for (int i = 0; i < D; ++i) p.v[i] = a[i];
  return p;
}

// X_0 of the cell whose block is B.
template <int D, class Cells>
__device__ __forceinline__ void cell_origin_df(const Cells& cs, const float4* B, df x0[D]) {
  constexpr int NR = (1 << D) / 4;
#pragma unroll
  for (int a = 0; a < D; ++a) x0[a] = df_make(cs.ld(B + a * NR).x, cs.ld(B + (D + a) * NR).x);
}

// One Newton step at t32 with the double-float residual of the offset dloc =
// y - X_0 in the cell whose block is B (the end of the fast path's inverse
// map), repeated from the updated iterate while the step is above kFinish32
// (rare: the FP32 phase ends within ~2e-7 of the root, but in sheared cells; a
// first step of more than kStart32, or one that does not shrink 100 times, fails).
// t receives the double-float reference coordinates.
template <int D, class Cells>
__device__ __forceinline__ int finish_cell_df(const Cells& cs, const float4* B, const df dloc[D], float t32[D], df t[D],
                                              int& iters) {
  float most = kStart32;
#pragma unroll 1
  for (int rep = 0; rep < 3; ++rep) {
    float r[D], J[D][D], m32[4], dt[D];
    df m[4];
    ++iters;
    mixed32<D>(t32, m32);
    mixed_df<D>(t32, m);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const MapRow<D> hi = load_row<D>(cs, B, 0, c);
      r[c] = residual_row_df<D>(hi, load_row<D>(cs, B, 1, c), dloc[c], t32, m);
      jacobian_row32<D>(hi, t32, m32, J[c]);
    }
    if (!solve32<D>(J, r, dt)) return kCellFail;
    float mx = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) mx = fmaxf(mx, fabsf(dt[a]));
    if (!(mx <= most)) return kCellFail;
    if (mx <= kFinish32 || rep == 2) {
      bool in = true;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        t[a] = two_sum(t32[a], dt[a]);
        // t >= -eps  <=>  t32 >= -eps - dt ;  t <= 1 + eps  <=>  t32 - 1 <= eps - dt
        in = in && (t32[a] >= -(float)kInsideEps - dt[a]) && (t32[a] - 1.0f <= (float)kInsideEps - dt[a]);
      }
      return in ? kCellIn : kCellOut;
    }
#pragma unroll
    for (int a = 0; a < D; ++a) t32[a] += dt[a];
    most = rep == 0 ? fmaxf(1e-2f * mx, kFinish32) : 1e-5f;
  }
  return kCellFail;
}

// Inverse map of y in one cell (the candidates of the rare paths; the fast
// path's loop is locate_df).  t32 holds the FP32 start on entry; on return t
// holds the double-float reference coordinates.
constexpr float kSettle32Tight = 1e-5f;

template <int D, class Cells>
__device__ __forceinline__ int solve_cell_df(const Cells& cs, uint32_t K, const df y[D], float t32[D], df t[D],
                                             int& iters) {
  const float4* B = cs.block(K);
  df dloc[D];
  cell_origin_df<D>(cs, B, dloc);
#pragma unroll
  for (int a = 0; a < D; ++a) dloc[a] = df_sub(y[a], dloc[a]);
  float mx = 1.f;
#pragma unroll 1
  for (int it = 0; it < kMaxIt32 && mx > kSettle32; ++it) {
    ++iters;
    float J[D][D], r[D], dt[D], m[4];
    mixed32<D>(t32, m);
#pragma unroll
    for (int c = 0; c < D; ++c) {
      const MapRow<D> w = load_row<D>(cs, B, 0, c);
      r[c] = __fsub_rn(dloc[c].hi, map_row32<D>(w, t32, m));
      jacobian_row32<D>(w, t32, m, J[c]);
    }
    if (!solve32<D>(J, r, dt)) return kCellFail;
    mx = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      t32[a] += dt[a];
      mx = fmaxf(mx, fabsf(dt[a]));
    }
    if (!(mx <= 1e3f)) return kCellFail;  // diverging or NaN
    // clearly outside (see locate_df)
    if (mx < 0.05f) {
      float out = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) out = fmaxf(out, fmaxf(-t32[a], t32[a] - 1.0f));
      if (out > 4.f * mx + 1e-3f) return kCellOut;
    }
  }
  // not settled by kStart32: as good as FP32 gets in a sheared cell, perhaps
  return mx <= kStart32 ? finish_cell_df<D>(cs, B, dloc, t32, t, iters) : kCellFail;
}

// FP64 Newton for a cell the fast path could not settle (rare; out of line
// so that the hot loop stays small in the instruction cache); s32 holds the
// FP32 start in its high parts.
template <int D>
__device__ __noinline__ RarePath<D> test_cell_fp64(const MeshView& m, uint32_t K, DfPt<D> y, DfPt<D> s32) {
  RarePath<D> o;
  o.iters = 0;
  o.flags = 0;
  o.K = K;
  double yd[D], tt[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    yd[a] = df_to_double(y.v[a]);
    const float st = s32.v[a].hi;
    tt[a] = isfinite(st) && fabsf(st) < 4.f ? (double)st : 0.5;
  }
  bool conv = false;
  const bool in = try_cell<D>(m, K, yd, tt, o.iters, o.flags, &conv);
#pragma unroll
  for (int a = 0; a < D; ++a) o.t.v[a] = df_from_double(tt[a]);
  o.r = !conv ? kCellFail : (in ? kCellIn : kCellOut);
  return o;
}

// y inside cell K's padded bounding box (padding 1e-6 of the cell's extent,
// far wider than the kInsideEps band in reference coordinates): a point
// outside it is not in K.  The FP32 copy of the box is widened outward, so
// the test on y's high parts is conservative, with no FP64 instruction.
template <int D>
__device__ __forceinline__ bool in_cell_box(const MeshView& m, uint32_t K, const df y[D]) {
  const float4 lo = __ldg(m.bbox32 + 2 * (size_t)K), hi = __ldg(m.bbox32 + 2 * (size_t)K + 1);
  const float l[3] = {lo.x, lo.y, lo.z}, h[3] = {hi.x, hi.y, hi.z};
  bool in = true;
#pragma unroll
  for (int a = 0; a < D; ++a) in = in && y[a].hi >= l[a] && y[a].hi <= h[a];
  return in;
}

// Fast path, then the FP64 Newton when the fast path does not settle.
template <int D, class Cells>
__device__ __forceinline__ int test_cell(const Cells& cs, const MeshView& m, uint32_t K, const df y[D], float t32[D],
                                         df t[D], int& iters, unsigned& flags) {
  DfPt<D> s;
#pragma unroll
  for (int a = 0; a < D; ++a) s.v[a] = df_make(t32[a], 0.f);
  const int r = solve_cell_df<D>(cs, K, y, t32, t, iters);
  if (r != kCellFail) return r;
  const RarePath<D> o = test_cell_fp64<D>(m, K, pack<D>(y), s);
  iters += o.iters;
  flags |= o.flags | kFlagFallback64;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    t[a] = o.t.v[a];
    t32[a] = t[a].hi;
  }
  return o.r;
}

// Lowest-index rule (see lowest_owner in locate.cuh) on the fast path.  The
// band test is inline; the neighbour tests (rare) are out of line and read
// the cells from the mesh arrays.
template <int D>
__device__ __noinline__ RarePath<D> lowest_owner_df_slow(const MeshView& m, DfPt<D> y, uint32_t found, DfPt<D> t) {
  RarePath<D> o;
  o.iters = 0;
  o.flags = 0;
  o.r = kCellIn;
  int c[3];
  cell_ijk<D>(m, found, c);
  int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    lo[a] = (t.v[a].hi < (float)kTieBand && c[a] > 0) ? -1 : 0;
    hi[a] = (t.v[a].hi > 1.0f - (float)kTieBand && c[a] < m.n[a] - 1) ? 1 : 0;
  }
  uint32_t best = found;
  DfPt<D> tb = t;
  for (int o2 = (D == 3 ? lo[2] : 0); o2 <= (D == 3 ? hi[2] : 0); ++o2)
    for (int o1 = lo[1]; o1 <= hi[1]; ++o1)
      for (int o0 = lo[0]; o0 <= hi[0]; ++o0) {
        if (o0 == 0 && o1 == 0 && o2 == 0) continue;
        const uint32_t K = cell_index<D>(m, c[0] + o0, c[1] + o1, c[2] + o2);
        if (K >= best) continue;
        const int off[3] = {o0, o1, o2};
        float s[D];
        df tt[D];
#pragma unroll
        for (int a = 0; a < D; ++a) s[a] = t.v[a].hi - (float)off[a];
        if (test_cell<D>(GlobalCells<D, false>{m}, m, K, y.v, s, tt, o.iters, o.flags) == kCellIn) {
          best = K;
          tb = pack<D>(tt);
        }
      }
  o.K = best;
  o.t = tb;
  return o;
}

//
// The fast path leaves a particle to the full step only within the mesh's band
// of a facet: a redone particle holds its warp up by several times a step's
// latency, which a small store sees whole.  A cell across the facet holds the
// point within kInsideEps only if the point is that part of the cell's size away,
// in units of this one: no more than kInsideEps sqrt(D) times the largest |J| of
// the mesh times the largest |J^-1|, which the set-up takes at the cells' corners.
// Where that product is at most kTieRatio it makes 4.5e-8, and kTieBandFast, more
// than twice that, is enough (reference coordinates at hand are good to ~1e-12,
// accurate == true); meshes of more uneven cells keep kTieBand.
constexpr float kTieBandFast = 1e-7f;
constexpr double kTieRatio = 256.0;

template <int D, bool kFast = false>
__device__ __forceinline__ uint32_t lowest_owner_df(const MeshView& m, const df y[D], uint32_t found, df t[D],
                                                    int& iters, unsigned& flags, bool accurate) {
  // band test first (cheap); the cell's (i,j,k) only when some coordinate is
  // near a facet
  bool near = false;
  const float band = accurate ? m.tie_band : (float)kTieBand;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (accurate)
      near = near || t[a].hi < band || __fsub_rn(__fsub_rn(1.0f, t[a].hi), t[a].lo) < band;
    else
      near = near || t[a].hi < band || t[a].hi > 1.0f - band;
  }
  if (!near) return found;
  int c[3];
  cell_ijk<D>(m, found, c);
  bool any = false;
#pragma unroll
  for (int a = 0; a < D; ++a)
    any = any || (t[a].hi < (float)kTieBand && c[a] > 0) || (t[a].hi > 1.0f - (float)kTieBand && c[a] < m.n[a] - 1);
  if (!any) return found;
  if constexpr (kFast) return kDefer;
  const RarePath<D> o = lowest_owner_df_slow<D>(m, pack<D>(y), found, pack<D>(t));
  iters += o.iters;
  flags |= o.flags;
#pragma unroll
  for (int a = 0; a < D; ++a) t[a] = o.t.v[a];
  return o.K;
}

// Past the hint cell and its predicted neighbour: the walk over the hint's
// other vertex neighbours in the paper's order (Sec. 2.4: v the vertex of the
// hint closest to y, descending (y - v).(c_K' - v) over the neighbours' centres
// c_K'), each cell tested with the double-float inverse map (FP64 Newton only
// where that does not settle), then the all-cells search.  The order only
// affects the cost: the first cell found is settled by the lowest-index
// rule, so the ordering heuristic is computed in FP32.  Each candidate's
// Newton starts from the cell centre.
template <int D>
__device__ __noinline__ RarePath<D> locate_df_slow(const MeshView& m, DfPt<D> y, uint32_t hintK) {
  RarePath<D> o;
  o.iters = 0;
  o.flags = 0;
  o.r = kCellIn;
  double yd[D];
#pragma unroll
  for (int a = 0; a < D; ++a) yd[a] = df_to_double(y.v[a]);
  bool inside_box = true;
#pragma unroll
  for (int a = 0; a < D; ++a) inside_box = inside_box && yd[a] >= m.dlo[a] && yd[a] <= m.dhi[a];
  if (!inside_box) {
    // outside the padded domain box: in no cell (see locate in locate.cuh)
    o.K = PIC_LOST;
#pragma unroll
    for (int a = 0; a < D; ++a) o.t.v[a] = df_make(0.f, 0.f);
    return o;
  }
  if (hintK < m.C) {
    o.flags |= kFlagWalk;
    int c[3];
    cell_ijk<D>(m, hintK, c);
    // corner positions of cell (i,j,k) from the vertex array, in FP32
    auto vertex = [&](int i, int j, int k, float p[D]) {
      const int64_t v = (int64_t)i + (int64_t)m.nv[0] * ((int64_t)j + (D == 3 ? (int64_t)m.nv[1] * k : 0));
#pragma unroll
      for (int a = 0; a < D; ++a) p[a] = (float)__ldg(m.X + a * m.nverts + v);
    };
    float yf[D], v[D], best = 3.4e38f;
#pragma unroll
    for (int a = 0; a < D; ++a) yf[a] = y.v[a].hi;
    for (int q = 0; q < (1 << D); ++q) {
      float p[D], d2 = 0.f;
      vertex(c[0] + (q & 1), c[1] + ((q >> 1) & 1), D == 3 ? c[2] + ((q >> 2) & 1) : 0, p);
#pragma unroll
      for (int a = 0; a < D; ++a) d2 += (yf[a] - p[a]) * (yf[a] - p[a]);
      if (d2 < best) {
        best = d2;
#pragma unroll
        for (int a = 0; a < D; ++a) v[a] = p[a];
      }
    }
    constexpr int NN = (D == 3 ? 27 : 9);
    float score[NN];
    uint32_t cand = 0;  // bit mask of the neighbours still to test
    for (int q = 0; q < NN; ++q) {
      const int o0 = q % 3 - 1, o1 = (q / 3) % 3 - 1, o2 = (D == 3 ? q / 9 - 1 : 0);
      score[q] = 0.f;
      if (o0 == 0 && o1 == 0 && o2 == 0) continue;
      const int i = c[0] + o0, j = c[1] + o1, k = c[2] + o2;
      if (i < 0 || j < 0 || i >= m.n[0] || j >= m.n[1]) continue;
      if (D == 3 && (k < 0 || k >= m.n[2])) continue;
      float ctr[D] = {};
      for (int w = 0; w < (1 << D); ++w) {
        float p[D];
        vertex(i + (w & 1), j + ((w >> 1) & 1), D == 3 ? k + ((w >> 2) & 1) : 0, p);
#pragma unroll
        for (int a = 0; a < D; ++a) ctr[a] += p[a] * (1.f / (1 << D));
      }
      float sc = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) sc += (yf[a] - v[a]) * (ctr[a] - v[a]);
      score[q] = sc;
      cand |= 1u << q;
    }
    const GlobalCells<D, false> cs{m};
    bool at_hint = true;  // the hint cell itself first: the fast path may have failed to settle in it
    while (at_hint || cand) {
      int qb = NN / 2;
      if (!at_hint) {
        qb = __ffs(cand) - 1;  // a valid candidate even if every score is NaN
        float sb = score[qb];
        for (int q = qb + 1; q < NN; ++q)
          if (((cand >> q) & 1u) && score[q] > sb) {
            sb = score[q];
            qb = q;
          }
        cand &= ~(1u << qb);
      }
      at_hint = false;
      const int off[3] = {qb % 3 - 1, (qb / 3) % 3 - 1, D == 3 ? qb / 9 - 1 : 0};
      const uint32_t K = cell_index<D>(m, c[0] + off[0], c[1] + off[1], c[2] + off[2]);
      if (!in_cell_box<D>(m, K, y.v)) continue;  // cannot hold y: no Newton there
      float s32[D];
      df tt[D];
#pragma unroll
      for (int a = 0; a < D; ++a) s32[a] = 0.5f;  // from the cell centre (R2)
      if (test_cell<D>(cs, m, K, y.v, s32, tt, o.iters, o.flags) == kCellIn) {
        o.K = lowest_owner_df<D>(m, y.v, K, tt, o.iters, o.flags, true);
        o.t = pack<D>(tt);
        return o;
      }
    }
  }
  double to[D];
  o.K = global_search<D>(m, yd, to, o.iters, o.flags);
#pragma unroll
  for (int a = 0; a < D; ++a) o.t.v[a] = df_from_double(to[a]);
  return o;
}

template <int D>
__device__ __forceinline__ uint32_t locate_slow(const MeshView& m, const df y[D], uint32_t hintK, df t[D], int& iters,
                                                unsigned& flags) {
  const RarePath<D> o = locate_df_slow<D>(m, pack<D>(y), hintK);
  iters += o.iters;
  flags |= o.flags;
#pragma unroll
  for (int a = 0; a < D; ++a) t[a] = o.t.v[a];
  return o.K;
}

// Owner of y (lowest index) and its double-float reference coordinates.
// Search order: the hint cell, then up to two hops to the neighbour that the
// current cell's iterate points to (across every facet it violates), then
// (out of line) the walk over the hint's vertex neighbours in the paper's a.b
// order and the all-cells search.  The owner does not depend on the order: the
// first cell found to hold y is settled by the lowest-index rule.
//
// The FP32 iterations and the hops are one loop, an iteration per pass in
// whatever cell the lane is in, and the double-float step comes once, after
// it.  A warp's particles need two or three passes in one or two cells each;
// one Newton solve per visited cell, each ending in its own double-float step,
// made every warp run two or three whole solves with most lanes idle (26 of 32
// lanes active over the kernel).
//
// Convergence, accurate == true: above kSettle32 an update d also takes the
// map's second-order term (Chebyshev's method: the (bi/tri)linear map's
// Phi(t + d) - Phi(t) - J d is a short exact sum, and J^{-1} is at hand), q =
// J^{-1} of it; the next error is then ~2 |q|^2 / |d|, so steps up to a few
// 1e-3 settle in one iteration and a quarter cell in two (plain Newton: two
// and three).  accurate == false (stage points of the FP32-basis form) runs
// plain Newton to kSettle32Tight, which is what an FP32 basis can use.
constexpr int kPredictedHops = 2;

template <int D, bool kFast = false, class Cells>
__device__ __forceinline__ uint32_t locate_df(const Cells& cs, const MeshView& m, const df y[D], uint32_t hintK,
                                              const float hint_t[D], df t[D], int& iters, unsigned& flags,
                                              bool accurate = true) {
  if (hintK >= m.C) {
    if constexpr (kFast) return kDefer;
    flags |= kFlagBounds;
    return locate_slow<D>(m, y, hintK, t, iters, flags);
  }
  uint32_t K = hintK;
  float t32[D];
  df dloc[D];  // y - X_0 of the current cell
#pragma unroll
  for (int a = 0; a < D; ++a) t32[a] = hint_t[a];
  cell_origin_df<D>(cs, cs.block(K), dloc);
#pragma unroll
  for (int a = 0; a < D; ++a) dloc[a] = df_sub(y[a], dloc[a]);
  int left = kMaxIt32, hops = 0;
  bool ok = false;
  // to the neighbour across every facet that t32 violates; the offset from its
  // X_0 by the step between the two, so that y itself need not be kept.  Both
  // differences carry their low parts: added at the size of the coordinates, with
  // df_add's rounding, two hops left x-hat 1.04 times less exact on 32^2 cells.
  auto hop = [&]() {
    if (hops++ == kPredictedHops) return false;
    flags |= kFlagWalk;
    int c[3], pred[3] = {0, 0, 0};
    cell_ijk<D>(m, K, c);
    bool have_pred = false;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      pred[a] = t32[a] < 0.f ? -1 : (t32[a] >= 1.f ? 1 : 0);
      if (c[a] + pred[a] < 0 || c[a] + pred[a] >= m.n[a]) pred[a] = 0;
      have_pred = have_pred || pred[a] != 0;
      t32[a] -= (float)pred[a];
    }
    if (!have_pred) return false;
    df x0[D], x1[D];
    cell_origin_df<D>(cs, cs.block(K), x0);
    K = cell_index<D>(m, c[0] + pred[0], c[1] + pred[1], c[2] + pred[2]);
    cell_origin_df<D>(cs, cs.block(K), x1);
#pragma unroll
    for (int a = 0; a < D; ++a) dloc[a] = df_sub_accurate(dloc[a], df_sub_accurate(x1[a], x0[a]));
    left = kMaxIt32 - 1;
    return true;
  };
  bool leave = false;  // the double-float root of the current cell lies outside it
#pragma unroll 1
  for (;;) {
    ok = false;
#pragma unroll 1
    while (left-- > 0) {
      if (leave) {
        if (!hop()) break;
        leave = false;
      }
      ++iters;
      float d[D], mx = 0.f, slack;
      bool settled;
      {
        const float4* B = cs.block(K);
        float J[D][D], r[D], m32[4];
        Adjugate32<D> A;
        mixed32<D>(t32, m32);
#pragma unroll
        for (int c = 0; c < D; ++c) {
          const MapRow<D> w = load_row<D>(cs, B, 0, c);
          r[c] = __fsub_rn(dloc[c].hi, map_row32<D>(w, t32, m32));
          jacobian_row32<D>(w, t32, m32, J[c]);
        }
        if (!adjugate32<D>(J, A)) break;
        apply32<D>(A, r, d);
#pragma unroll
        for (int a = 0; a < D; ++a) mx = fmaxf(mx, fabsf(d[a]));
        if (!(mx <= 1e3f)) break;  // diverging or NaN
        if (accurate) {
          settled = mx <= kSettle32;
          slack = kInside32;
          if (!settled) {
            float w[D], q[D], mq = 0.f;
            second_order32<D>(cs, B, t32, d, w);
            apply32<D>(A, w, q);
#pragma unroll
            for (int a = 0; a < D; ++a) mq = fmaxf(mq, fabsf(q[a]));
            if (mq <= 0.25f * mx) {
#pragma unroll
              for (int a = 0; a < D; ++a) d[a] = __fsub_rn(d[a], q[a]);
              settled = mq * mq <= kSettleCheb32 * mx;
              if (!settled) slack = __fmaf_rn(4.f, __fdividef(mq * mq, mx), 1e-4f);
            } else {
              slack = 1e30f;
            }
          }
        } else {
          settled = mx <= kSettle32Tight;
          slack = settled ? (float)kInsideEps : 1e30f;
          if (mx < 0.05f && !settled) slack = __fadd_rn(__fmul_rn(4.f, mx), 1e-3f);
        }
      }
      // Clearly outside: the iterate lies outside [0,1] by more than its error,
      // so the root is outside too and the iterate tells where to go.  A wrong
      // call only costs time: another hop, or the rare path.
      float out = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        t32[a] = __fadd_rn(t32[a], d[a]);
        out = fmaxf(out, fmaxf(-t32[a], t32[a] - 1.0f));
      }
      leave = out > slack;
      ok = settled && !leave;
      if (ok) break;
      if (leave) left = 1;  // the next pass hops, which sets it again
    }
    if (!ok) break;
    if (!accurate) {
#pragma unroll
      for (int a = 0; a < D; ++a) t[a] = df_make(t32[a], 0.f);
      break;
    }
    const int r = finish_cell_df<D>(cs, cs.block(K), dloc, t32, t, iters);
    ok = r == kCellIn;
    if (r != kCellOut) break;
    // within a few 1e-7 of a facet and on its other side: that neighbour
#pragma unroll
    for (int a = 0; a < D; ++a) t32[a] = t[a].hi;
    leave = true;
    left = 1;
  }
  if (ok) return lowest_owner_df<D, kFast>(m, y, K, t, iters, flags, accurate);
  if constexpr (kFast) return kDefer;
  flags |= kFlagWalk | kFlagWalk64;
  return locate_slow<D>(m, y, hintK, t, iters, flags);
}

// The same reading every block from the mesh arrays.
template <int D>
__device__ __forceinline__ uint32_t locate_df(const MeshView& m, const df y[D], uint32_t hintK, const float hint_t[D],
                                              df t[D], int& iters, unsigned& flags, bool accurate = true) {
  return locate_df<D>(GlobalCells<D, false>{m}, m, y, hintK, hint_t, t, iters, flags, accurate);
}

// ---------------------------------------------------------- Q2 velocity --
// u_h = sum_{a,b,c} U[node(K; a,b,c)] l_a(t0) l_b(t1) l_c(t2) with the 1D
// quadratic Lagrange basis on {0, 1/2, 1}:
//   l0 = (1-t)(1-2t) = -w v,  l1 = 4 t w,  l2 = t v,  w = 1-t, v = 2t-1.
// lagrange2_df gives the basis in double-float (used by the gradient).

__device__ __forceinline__ void lagrange2_df(df t, df l[3]) {
  const df ws = two_sum(1.0f, -t.hi);
  const df w = fast_two_sum(ws.hi, __fsub_rn(ws.lo, t.lo));
  const df vs = two_sum(__fmul_rn(2.0f, t.hi), -1.0f);
  const df v = fast_two_sum(vs.hi, __fmaf_rn(2.0f, t.lo, vs.lo));
  const df wv = df_mul(w, v);
  l[0] = df_make(-wv.hi, -wv.lo);
  l[1] = df_scale2(df_mul(t, w), 4.0f);
  l[2] = df_mul(t, v);
}

// The evaluation itself uses the per-cell monomial form about the cell
// centre (built from the nodal values when the field is set):
//   u_c(s) = sum_{p,q,r} C_pqr s0^p s1^q s2^r,   s = t - 1/2,
// evaluated by nested Horner steps, 26 per component in 3D (8 in 2D),
// each a double-float multiply-add.  For smooth fields |C_pqr| falls
// with p + q + r (C_000 is the centre node's value), so the evaluation is
// well conditioned.  (Sums of order two and above with their high parts on one
// fixed grid take 7 operations a step for 12, and 8.02 ms for 8.85 in five 64^3 x
// 20 RK4 steps; but their low parts lose two or three bits of the largest sum,
// which made positions up to 1.4 times and gradients 2 to 10 times less exact on
// meshes below 16 cells a side.)

// c + a s in double-float, the result left unnormalised (its low part may
// exceed half an ulp of the high part slightly; the next step multiplies it
// exactly through two_prod and an FMA).
__device__ __forceinline__ df df_horner(df a, df s, df c) {
  const df p = two_prod(a.hi, s.hi);
  float e = __fmaf_rn(a.hi, s.lo, p.lo);
  e = __fmaf_rn(a.lo, s.hi, e);
  const df q = two_sum(p.hi, c.hi);
  return df_make(q.hi, __fadd_rn(q.lo, __fadd_rn(e, c.lo)));
}

// s = t - 1/2 in double-float.
__device__ __forceinline__ df centred(df t) {
  const df d = two_sum(t.hi, -0.5f);
  return fast_two_sum(d.hi, __fadd_rn(d.lo, t.lo));
}

// One slice of Qc (five float4: ten high parts, then ten low parts).
template <class Ld>
__device__ __forceinline__ void load_slice(const Ld& ld, const float4* p, float hi[10], float lo[10]) {
  float f[20];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float4 v = ld.ld(p + k);
    f[4 * k] = v.x;
    f[4 * k + 1] = v.y;
    f[4 * k + 2] = v.z;
    f[4 * k + 3] = v.w;
  }
#pragma unroll
  for (int e = 0; e < 10; ++e) {
    hi[e] = f[e];
    lo[e] = f[10 + e];
  }
}

// From the cell's Qc block `cell`, read through ld.ld().
template <int D, class Ld>
__device__ __forceinline__ void q2_eval_df(const Ld& ld, const float4* cell, const df t[D], df u[D]) {
  constexpr int NS = (D == 3 ? 3 : 1);
  df s[D];
#pragma unroll
  for (int a = 0; a < D; ++a) s[a] = centred(t[a]);
#pragma unroll 1
  for (int comp = 0; comp < D; ++comp) {
    const float4* cq = cell + comp * (5 * NS);
    df rr;
#pragma unroll
    for (int r = NS - 1; r >= 0; --r) {
      float hi[10], lo[10];
      load_slice(ld, cq + 5 * r, hi, lo);
      auto c = [&](int k) { return df_make(hi[k], lo[k]); };
      df h[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) h[q] = df_horner(df_horner(c(3 * q + 2), s[0], c(3 * q + 1)), s[0], c(3 * q));
      const df g = df_horner(df_horner(h[2], s[1], h[1]), s[1], h[0]);
      rr = r == NS - 1 ? g : df_horner(rr, s[D - 1], g);
    }
    rr = df_norm(rr);
    // constant indices keep u in registers under the rolled loop
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (a == comp) u[a] = rr;
  }
}

// FP32 basis and contraction (precision form) from the cell's Qf block: the
// same monomial form on the high parts, FP32 Horner steps.
template <int D, class Ld>
__device__ __forceinline__ void q2_eval_f32(const Ld& ld, const float4* cell, const df t[D], df u[D]) {
  constexpr int NS = (D == 3 ? 3 : 1);
  constexpr int NF4 = qf_floats_per_comp<D>() / 4;  // float4 per component
  float s[D];
#pragma unroll
  for (int a = 0; a < D; ++a) s[a] = t[a].hi - 0.5f;
#pragma unroll
  for (int comp = 0; comp < D; ++comp) {
    float c[4 * NF4];
#pragma unroll
    for (int k = 0; k < NF4; ++k) {
      const float4 v = ld.ld(cell + comp * NF4 + k);
      c[4 * k] = v.x;
      c[4 * k + 1] = v.y;
      c[4 * k + 2] = v.z;
      c[4 * k + 3] = v.w;
    }
    float g[NS];
#pragma unroll
    for (int r = 0; r < NS; ++r) {
      float h[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) h[q] = fmaf(fmaf(c[9 * r + 3 * q + 2], s[0], c[9 * r + 3 * q + 1]), s[0], c[9 * r + 3 * q]);
      g[r] = fmaf(fmaf(h[2], s[1], h[1]), s[1], h[0]);
    }
    const df rr = df_make((D == 3) ? fmaf(fmaf(g[2], s[2], g[1]), s[2], g[0]) : g[0], 0.f);
    // constant indices keep u in registers under a rolled loop
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (a == comp) u[a] = rr;
  }
}

}  // namespace pic
