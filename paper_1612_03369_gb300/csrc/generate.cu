// generate.cu -- particle generation with a density and from prescribed
// locations (Sec. 2.2 of Gassmoeller et al., arXiv 1612.03369).
//
//   pic_cell_weights       w_K = int_K rho_h dx, rho_h the (bi/tri)linear
//                          interpolant of vertex values; tensor 2-point Gauss
//                          (exact: the integrand has degree <= 3 per axis)
//   pic_draw_cell_counts   N draws over the accumulated weights (the listing's
//                          second and third loops, on one GPU)
//   pic_seed_particles_mh  in-cell Metropolis-Hastings with target
//                          rho-hat = rho_h(Phi_K(x-hat)) |det grad-hat Phi_K|
//                          and uniform proposals, thinned by J
//   pic_import_particles   owner search for every prescribed point, ids in
//                          input order among the points found
//
// The decisions that turn floating point into integers (which cell a draw
// falls in, whether a proposal is accepted) must not depend on the device:
// the accumulated weights are one left fold, and rho-hat is evaluated as a
// fixed sequence of correctly rounded IEEE operations (the _rn intrinsics
// keep the compiler from contracting or reordering them):
//   rho_h   = sum over local vertices v = 0..2^D-1 of rho_v * w_v(t),
//             w_v = product over axes a = 0..D-1 of (bit a of v ? t_a : 1 - t_a)
//   J_ij    = sum over v of X_{v,i} * dw_v/dt_j (the same product with the
//             factor of axis j replaced by +1 or -1)
//   det J   = J00 J11 - J01 J10 (2D);
//             J00 (J11 J22 - J12 J21) + J01 (J12 J20 - J10 J22)
//             + J02 (J10 J21 - J11 J20), summed left to right (3D)
//   rho-hat = rho_h * |det J|
#include <cmath>
#include <cstdlib>

#include "fastpath.cuh"
#include "grad_df.cuh"
#include "pic_internal.cuh"
#include "seed.cuh"

namespace pic {

template <int D>
__device__ __forceinline__ int64_t local_vertex(const MeshView& m, const int c[3], int v) {
  return (int64_t)(c[0] + (v & 1)) +
         (int64_t)m.nv[0] * ((int64_t)(c[1] + ((v >> 1) & 1)) + (D == 3 ? (int64_t)m.nv[1] * (c[2] + ((v >> 2) & 1)) : 0));
}

template <int D>
__device__ __forceinline__ double vweight_rn(int v, const double t[D], int skip = -1) {
  double w = 1.0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const bool hi = (v >> a) & 1;
    const double f = (a == skip) ? (hi ? 1.0 : -1.0) : (hi ? t[a] : __dsub_rn(1.0, t[a]));
    w = __dmul_rn(w, f);
  }
  return w;
}

template <int D>
__device__ __forceinline__ double det_rn(const double J[D][D]) {
  double det;
  if constexpr (D == 2) {
    det = __dsub_rn(__dmul_rn(J[0][0], J[1][1]), __dmul_rn(J[0][1], J[1][0]));
  } else {
    const double c0 = __dsub_rn(__dmul_rn(J[1][1], J[2][2]), __dmul_rn(J[1][2], J[2][1]));
    const double c1 = __dsub_rn(__dmul_rn(J[1][2], J[2][0]), __dmul_rn(J[1][0], J[2][2]));
    const double c2 = __dsub_rn(__dmul_rn(J[1][0], J[2][1]), __dmul_rn(J[1][1], J[2][0]));
    det = __dadd_rn(__dadd_rn(__dmul_rn(J[0][0], c0), __dmul_rn(J[0][1], c1)), __dmul_rn(J[0][2], c2));
  }
  return det;
}

template <int D>
__device__ double rho_hat_rn(const MeshView& m, uint32_t K, const double* __restrict__ rho, const double t[D]) {
  int c[3];
  cell_ijk<D>(m, K, c);
  double r = 0.0;
#pragma unroll
  for (int v = 0; v < (1 << D); ++v) r = __dadd_rn(r, __dmul_rn(__ldg(rho + local_vertex<D>(m, c, v)), vweight_rn<D>(v, t)));
  double J[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) {
      double s = 0.0;
#pragma unroll
      for (int v = 0; v < (1 << D); ++v)
        s = __dadd_rn(s, __dmul_rn(__ldg(m.X + i * m.nverts + local_vertex<D>(m, c, v)), vweight_rn<D>(v, t, j)));
      J[i][j] = s;
    }
  return __dmul_rn(r, fabs(det_rn<D>(J)));
}

// x = Phi_K(t) = sum_v X_v w_v(t), in the same rounded sequence.
template <int D>
__device__ __forceinline__ void phi_rn(const MeshView& m, uint32_t K, const double t[D], double x[D]) {
  int c[3];
  cell_ijk<D>(m, K, c);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    double s = 0.0;
#pragma unroll
    for (int v = 0; v < (1 << D); ++v)
      s = __dadd_rn(s, __dmul_rn(__ldg(m.X + i * m.nverts + local_vertex<D>(m, c, v)), vweight_rn<D>(v, t)));
    x[i] = s;
  }
}

__device__ __forceinline__ double unit53(uint64_t r) { return (double)(r >> 11) * 0x1.0p-53; }

// ------------------------------------------------------------ cell weights

// The Gauss points are the same in every cell, and so are the weights w_v and
// dw_v/dt_j there: each block forms them once, by the sequence's own operations,
// and a cell only takes the products with its vertices (the full sequence per
// cell, 1815 FP64 operations: 0.40 ms for 110,592 cells, FP64-pipe bound).
template <int D>
__global__ void __launch_bounds__(128) cell_weights_kernel(const __grid_constant__ MeshView m, const double* __restrict__ rho,
                                                           double* __restrict__ w) {
  constexpr int NV = 1 << D;
  __shared__ double s_w[NV][D + 1][NV];  // [point][j; D: the weight itself][vertex]
  for (int e = threadIdx.x; e < NV * (D + 1) * NV; e += blockDim.x) {
    const double g0 = __dsub_rn(0.5, __ddiv_rn(0.5, __dsqrt_rn(3.0)));
    const double g1 = __dadd_rn(0.5, __ddiv_rn(0.5, __dsqrt_rn(3.0)));
    const int v = e % NV, j = (e / NV) % (D + 1), q = e / (NV * (D + 1));
    double t[D];
#pragma unroll
    for (int a = 0; a < D; ++a) t[a] = ((q >> a) & 1) ? g1 : g0;
    s_w[q][j][v] = vweight_rn<D>(v, t, j == D ? -1 : j);
  }
  __syncthreads();
  for (uint32_t K = blockIdx.x * blockDim.x + threadIdx.x; K < m.C; K += gridDim.x * blockDim.x) {
    int c[3];
    cell_ijk<D>(m, K, c);
    double X[D][NV], r[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int64_t lv = local_vertex<D>(m, c, v);
      r[v] = __ldg(rho + lv);
#pragma unroll
      for (int i = 0; i < D; ++i) X[i][v] = __ldg(m.X + i * m.nverts + lv);
    }
    double s = 0.0;
#pragma unroll 1
    for (int q = 0; q < NV; ++q) {
      double rh = 0.0, J[D][D], wq = 1.0;
#pragma unroll
      for (int v = 0; v < NV; ++v) rh = __dadd_rn(rh, __dmul_rn(r[v], s_w[q][D][v]));
#pragma unroll
      for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) {
          double e = 0.0;
#pragma unroll
          for (int v = 0; v < NV; ++v) e = __dadd_rn(e, __dmul_rn(X[i][v], s_w[q][j][v]));
          J[i][j] = e;
        }
#pragma unroll
      for (int a = 0; a < D; ++a) wq = __dmul_rn(wq, 0.5);
      s = __dadd_rn(s, __dmul_rn(wq, __dmul_rn(rh, fabs(det_rn<D>(J)))));
    }
    w[K] = s;
  }
}

// ------------------------------------------------------------ cell counts

struct DrawInfo {
  double W;          // total weight
  long long last;    // last cell of positive weight, -1 if none
  unsigned bad;      // a weight was negative or not finite
};

// The accumulated weights as one left fold, rounded after every addition, by
// one block.
//
// Between two powers of two the running sum S is an integer multiple n of one
// spacing g = ulp(S), and adding w >= 0 moves it to n + RN(w / g): an integer
// that does not depend on S, except that a remainder of exactly g / 2 rounds
// to the even sum, so on n's parity.  So each weight is a pair of increments,
// one per parity of the sum it meets (FoldInc), pairs compose associatively,
// and a block scan of 4,096 pairs gives 4,096 sums of the sequential fold at
// once.  The first sum to reach the next power of two ends the run: it is
// formed by one rounded addition, and the scan goes on behind it with the new
// spacing (about log2(C) such breaks).  One warp folding value by value, each
// addition waiting for the last, took 6.0 ms for 110,592 cells; this 0.24.
struct FoldInc {
  unsigned long long d[2];  // increment of n when n is even / odd, at most kFoldCap
};
constexpr unsigned long long kFoldTop = 1ull << 53;  // n of the next power of two
constexpr unsigned long long kFoldCap = 1ull << 54;  // increments saturate here: past kFoldTop only the order counts

__host__ __device__ __forceinline__ unsigned long long fold_cap(unsigned long long v) {
  return v < kFoldCap ? v : kFoldCap;
}

// First a, then b.
__host__ __device__ __forceinline__ FoldInc fold_compose(FoldInc a, FoldInc b) {
  FoldInc r;
  r.d[0] = fold_cap(a.d[0] + b.d[a.d[0] & 1u]);
  r.d[1] = fold_cap(a.d[1] + b.d[(a.d[1] + 1u) & 1u]);
  return r;
}

// A non-negative finite double's significand as an integer multiple of
// 2^(exp - 1075), exp >= 1 (subnormals share the first binade's spacing).
__host__ __device__ __forceinline__ void fold_split(unsigned long long bits, unsigned long long& n, int& exp) {
  exp = (int)((bits >> 52) & 0x7ffu);
  n = bits & ((1ull << 52) - 1);
  if (exp)
    n += 1ull << 52;
  else
    exp = 1;
}

// The bits of the sum n 2^(exp - 1075), n < kFoldTop.
__host__ __device__ __forceinline__ unsigned long long fold_join(unsigned long long n, int exp) {
  return n < (1ull << 52) ? n : (((unsigned long long)exp << 52) + (n - (1ull << 52)));
}

// Increments of n by the weight with these bits where the spacing is
// 2^(exp - 1075).
__host__ __device__ __forceinline__ FoldInc fold_inc(unsigned long long wbits, int exp) {
  unsigned long long m;
  int ew;
  fold_split(wbits, m, ew);
  FoldInc r;
  const int up = ew - exp;
  if (up >= 0) {
    r.d[0] = r.d[1] = up >= 2 ? (m ? kFoldCap : 0ull) : fold_cap(m << up);
    return r;
  }
  const int down = -up;
  if (down > 54) {
    r.d[0] = r.d[1] = 0;
    return r;
  }
  const unsigned long long q = m >> down, rem = m & ((1ull << down) - 1), half = 1ull << (down - 1);
  r.d[0] = q + ((rem > half || (rem == half && (q & 1u))) ? 1u : 0u);
  r.d[1] = q + ((rem > half || (rem == half && !(q & 1u))) ? 1u : 0u);
  return r;
}

constexpr int kFoldThreads = 1024;
constexpr int kFoldItems = 4;

__device__ __forceinline__ FoldInc fold_shfl_up(FoldInc v, int o) {
  FoldInc r;
  r.d[0] = __shfl_up_sync(0xffffffffu, v.d[0], o);
  r.d[1] = __shfl_up_sync(0xffffffffu, v.d[1], o);
  return r;
}

__global__ void __launch_bounds__(kFoldThreads) accumulate_weights_kernel(const double* __restrict__ w, uint32_t C,
                                                                          double* __restrict__ acc,
                                                                          DrawInfo* __restrict__ info) {
  __shared__ FoldInc s_warp[kFoldThreads / 32];
  __shared__ unsigned long long s_sum;  // bits of the running sum
  __shared__ uint32_t s_stop;           // first position of the batch that the scan cannot form
  __shared__ unsigned s_bad;
  __shared__ uint32_t s_last;           // 1 + last position of a positive weight
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  if (tid == 0) {
    s_sum = 0;
    s_bad = 0;
    s_last = 0;
  }
  __syncthreads();
  // the first sums double within a few values, each a break of the scan: one
  // warp folds them value by value (256 values: 0.01 ms for eight breaks)
  constexpr uint32_t kPrologue = 256;
  const uint32_t pro = C < kPrologue ? C : kPrologue;
  if (warp == 0) {
    double sum = 0.0;
    for (uint32_t k0 = 0; k0 < pro; k0 += 32) {
      const uint32_t k = k0 + lane;
      double v = k < pro ? w[k] : 0.0, mine = 0.0;
      if (!(v >= 0.0) || !isfinite(v)) {
        s_bad = 1;
        v = 0.0;
      }
      if (v > 0.0) atomicMax(&s_last, k + 1u);
      for (int q = 0; q < 32; ++q) {
        sum = __dadd_rn(sum, __shfl_sync(0xffffffffu, v, q));
        if ((int)lane == q) mine = sum;
      }
      if (k < pro) acc[k] = mine;
    }
    if (lane == 0) s_sum = (unsigned long long)__double_as_longlong(sum);
  }
  __syncthreads();
  for (uint64_t base = pro; base < C;) {
    const unsigned long long sum = s_sum;
    unsigned long long n0;
    int exp;
    fold_split(sum, n0, exp);
    if (tid == 0) s_stop = 0xffffffffu;
    // the batch's weights, kFoldItems consecutive ones per thread; a weight
    // that is not a finite number >= 0 counts as 0 (the call then fails)
    unsigned long long wb[kFoldItems];
    FoldInc inc[kFoldItems], mine;
    uint32_t pos = 0xffffffffu;  // this thread's first positive weight
    mine.d[0] = mine.d[1] = 0;
    uint32_t last = 0;
#pragma unroll
    for (int q = 0; q < kFoldItems; ++q) {
      const uint64_t k = base + (uint64_t)tid * kFoldItems + q;
      // on the bits (an FP64 comparison holds the SM's FP64 pipe 16 clocks a
      // warp): -0 counts as 0
      const unsigned long long b = k < C ? (unsigned long long)__double_as_longlong(w[k]) : 0ull;
      const bool minus_zero = b == 1ull << 63;
      const bool good = (b >> 52) < 0x7ffu || minus_zero;
      if (!good) s_bad = 1;
      wb[q] = good && !minus_zero ? b : 0ull;
      if (wb[q]) {
        if (pos == 0xffffffffu) pos = tid * kFoldItems + q;
        last = (uint32_t)k + 1u;
      }
      inc[q] = fold_inc(wb[q], exp);
      mine = fold_compose(mine, inc[q]);
    }
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0 && last) atomicMax(&s_last, last);
    // exclusive composition over the threads before this one
    FoldInc inc_warp = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const FoldInc v = fold_shfl_up(inc_warp, o);
      if ((int)lane >= o) inc_warp = fold_compose(v, inc_warp);
    }
    if (lane == 31) s_warp[warp] = inc_warp;
    __syncthreads();
    if (warp == 0) {
      FoldInc v = s_warp[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const FoldInc u = fold_shfl_up(v, o);
        if ((int)lane >= o) v = fold_compose(u, v);
      }
      s_warp[lane] = v;
    }
    __syncthreads();
    unsigned long long n = n0;
    if (warp > 0) n += s_warp[warp - 1].d[n & 1u];
    const FoldInc before = fold_shfl_up(inc_warp, 1);
    if (lane > 0) n += before.d[n & 1u];
    // a sum of zero has no spacing: the first positive weight is the sum
    const bool zero = sum == 0;
    uint32_t stop = zero ? pos : 0xffffffffu;
    unsigned long long nq[kFoldItems];
#pragma unroll
    for (int q = 0; q < kFoldItems; ++q) {
      nq[q] = n;  // the sum that item q meets
      n += inc[q].d[n & 1u];
      if (!zero && n >= kFoldTop && stop == 0xffffffffu) stop = tid * kFoldItems + q;
    }
    if (stop != 0xffffffffu) atomicMin(&s_stop, stop);
    __syncthreads();
    const uint32_t end = s_stop;
#pragma unroll
    for (int q = 0; q < kFoldItems; ++q) {
      const uint32_t i = tid * kFoldItems + q;
      const uint64_t k = base + i;
      if (k >= C || i > end) continue;
      const unsigned long long after = q + 1 < kFoldItems ? nq[q + 1 < kFoldItems ? q + 1 : q] : n;
      unsigned long long bits = zero ? 0ull : fold_join(after, exp);
      if (i == end)
        bits = (unsigned long long)__double_as_longlong(
            __dadd_rn(__longlong_as_double((long long)(zero ? 0ull : fold_join(nq[q], exp))),
                      __longlong_as_double((long long)wb[q])));
      acc[k] = __longlong_as_double((long long)bits);
      if (i == end || (end == 0xffffffffu && (k + 1 == C || i + 1 == kFoldThreads * kFoldItems))) s_sum = bits;
    }
    __syncthreads();
    base += end == 0xffffffffu ? (uint64_t)(kFoldThreads * kFoldItems) : (uint64_t)end + 1u;
    if (((s_sum >> 52) & 0x7ffu) == 0x7ffu) break;  // overflowed: the call fails
  }
  if (tid == 0) {
    info->W = __longlong_as_double((long long)s_sum);
    info->last = (long long)s_last - 1;
    info->bad = s_bad;
  }
}

// Draw i: u = top 53 bits of SplitMix64 output i times 2^-53, r = W u, the
// first cell with acc > r (or the last cell of positive weight if W u
// rounded up to W).
__global__ void __launch_bounds__(256) draw_cells_kernel(const double* __restrict__ acc, uint32_t C,
                                                         const DrawInfo* __restrict__ info, uint64_t n,
                                                         uint64_t seed, uint32_t* __restrict__ counts) {
  const double W = info->W;
  const long long last = info->last;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const double r = __dmul_rn(W, unit53(splitmix64_at(seed, i)));
    uint32_t lo = 0, hi = C;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if (acc[mid] > r)
        hi = mid;
      else
        lo = mid + 1;
    }
    const long long K = lo < C ? (long long)lo : last;
    if (K >= 0) atomicAdd(counts + K, 1u);
  }
}

// ------------------------------------------------------ Metropolis-Hastings

// A point of the unit cell as the generator's raw outputs (coordinate a is
// unit53(r[a])).
template <int D>
struct RawPoint {
  uint64_t r[D];
};

template <int D>
__device__ __forceinline__ void raw_coordinates(RawPoint<D> p, double t[D]) {
#pragma unroll
  for (int a = 0; a < D; ++a) t[a] = unit53(p.r[a]);
}

// rho-hat in double-float.
template <int D>
__device__ df rho_hat_df(const MeshView& m, uint32_t K, const double* __restrict__ rho, const df t[D]) {
  int c[3];
  cell_ijk<D>(m, K, c);
  df_acc r = acc_zero();
  df w[1 << D];
  w[0] = df_make(1.0f, 0.f);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const df u = df_sub(df_make(1.0f, 0.f), t[a]);
#pragma unroll
    for (int v = 0; v < (1 << a); ++v) {
      w[v + (1 << a)] = df_mul(w[v], t[a]);
      w[v] = df_mul(w[v], u);
    }
  }
#pragma unroll
  for (int v = 0; v < (1 << D); ++v) acc_mad(r, w[v], df_from_double(__ldg(rho + local_vertex<D>(m, c, v))));
  df J[D][D], det;
  map_jacobian_df<D>(LdgLoader(), m.blk + (size_t)K * block_float4s<D>(), t, J);
  if constexpr (D == 2) {
    det = df_det2(J[0][0], J[1][1], J[0][1], J[1][0]);
  } else {
    df_acc s = acc_zero();
    acc_mad(s, J[0][0], df_det2(J[1][1], J[2][2], J[1][2], J[2][1]));
    acc_mad(s, J[0][1], df_det2(J[1][2], J[2][0], J[1][0], J[2][2]));
    acc_mad(s, J[0][2], df_det2(J[1][0], J[2][1], J[1][1], J[2][0]));
    det = acc_result(s);
  }
  const df p = df_mul(acc_result(r), det);
  return det.hi < 0.f ? df_make(-p.hi, -p.lo) : p;
}

// The acceptance test that FP32 values left open: by double-float ones where
// they differ by more than `sure`, and by the definition otherwise,
// u rho-hat(current) < rho-hat(proposal) in the written sequence of IEEE
// operations (two evaluations are 2000 FP64 operations, 33 k clocks of an SM's
// FP64 pipe, and came 1.6 times per warp with FP32 alone before them).
template <int D>
__device__ __noinline__ bool mh_accept_rn(const MeshView& m, uint32_t K, const double* __restrict__ rho, RawPoint<D> cur,
                                          RawPoint<D> prop, bool at_centre, double u, float sure) {
  double t[D], y[D];
  raw_coordinates<D>(cur, t);
  if (at_centre)
#pragma unroll
    for (int a = 0; a < D; ++a) t[a] = 0.5;
  raw_coordinates<D>(prop, y);
  if (sure < INFINITY) {
    df td[D], yd[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      td[a] = df_from_double(t[a]);
      yd[a] = df_from_double(y[a]);
    }
    const df lhs = df_mul(df_from_double(u), rho_hat_df<D>(m, K, rho, td));
    const df diff = df_sub(rho_hat_df<D>(m, K, rho, yd), lhs);
    if (diff.hi > sure) return true;
    if (diff.hi < -sure) return false;
  }
  const double rc = rho_hat_rn<D>(m, K, rho, t), ry = rho_hat_rn<D>(m, K, rho, y);
  return __dmul_rn(u, rc) < ry;
}

// Writes particle q of cell K at the chain's state.  Out of line: its two dozen
// FP64 vertex values would otherwise be held through the steps.
template <int D>
__device__ __noinline__ void mh_emit(const MeshView& m, const StoreView& s, uint32_t K, RawPoint<D> cur, bool at_centre,
                                     uint32_t q, uint64_t id) {
  double t[D], x[D];
  raw_coordinates<D>(cur, t);
  if (at_centre)
#pragma unroll
    for (int a = 0; a < D; ++a) t[a] = 0.5;
  phi_rn<D>(m, K, t, x);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    s.x[a * s.cap + q] = x[a];
    const float hi = __double2float_rn(t[a]);
    s.xhat[a * s.cap + q] = make_float2(hi, __double2float_rn(t[a] - (double)hi));
  }
  s.id[q] = id;
  s.cell[q] = K;
  for (int p = 0; p < s.n_props; ++p) s.props[(size_t)p * s.cap + q] = 0.0;
}

// rho-hat in FP32: the density's monomial coefficients in the cell and the rows
// of the map's Jacobian; and how far u rho-hat(current) - rho-hat(proposal) has
// to be from 0 for its FP32 and its double-float value to have the right sign
// (infinite where they cannot decide).
template <int D>
struct RhoHat32 {
  float c[1 << D];      // 1, t0, t1, (t2,) mixed ones
  MapRow<D> row[D];
  float sure32, sure_df;

  __device__ __forceinline__ void load(const MeshView& m, uint32_t K, const double* __restrict__ rho) {
    int ijk[3];
    cell_ijk<D>(m, K, ijk);
    double v[1 << D];
#pragma unroll
    for (int q = 0; q < (1 << D); ++q) v[q] = __ldg(rho + local_vertex<D>(m, ijk, q));
    // differences along each axis: v[q] becomes the coefficient of the monomial
    // with the axes of q's set bits
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
      for (int q = 0; q < (1 << D); ++q)
        if ((q >> a) & 1) v[q] -= v[q & ~(1 << a)];
    constexpr int order[8] = {0, 1, 2, D == 2 ? 3 : 4, 3, 5, 6, 7};  // as mixed32 orders the monomials
    float R = 0.f;
#pragma unroll
    for (int q = 0; q < (1 << D); ++q) {
      c[q] = (float)v[order[q]];
      R += fabsf(c[q]);
    }
    const GlobalCells<D, false> cs{m};
    const float4* B = cs.block(K);
    float s[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      row[a] = load_row<D>(cs, B, 0, a);
      // bounds every entry of the row: its largest linear coefficient and the
      // mixed ones
      float r = 0.f, mixed = 0.f;
#pragma unroll
      for (int k = 0; k < D; ++k) r = fmaxf(r, fabsf(row[a].a[k]));
#pragma unroll
      for (int k = D; k < (1 << D) - 1; ++k) mixed += fabsf(row[a].a[k]);
      s[a] = r + mixed;
    }
    // With s_i the bound of row i and e = 2^-24: every entry of J is off by at
    // most 7 e s_i (coefficient, coordinate and FMA roundings), the determinant,
    // a sum of D! products, by 26 e D! s_0..s_(D-1), rho_h by 11 e R; the product
    // by less than 256 e R S = tau.  The double-float form keeps ~2^-46 where FP32
    // keeps 2^-24, so its bound is 2^-20 tau.  Two evaluations and u's own rounding
    // make 2.5 tau, and four times the bound in double-float.
    //
    // The written sequence has an error of its own, since it sums whole
    // coordinates: with f = 2^-53 and A_i the largest |x_i| of the mesh, an entry of
    // row i is off by at most 22 f A_i (the derivative weights' magnitudes sum to
    // 2; 11 roundings), the determinant by D! S f (22 sum A_i / s_i + 20), rho_h by
    // 11 f R; the product by less than 2^-29 tau (2 + sum A_i / s_i).  A decision has
    // to be clear of that too, twice, to be the sequence's (at |x| / h = 1e10 one in
    // 2e5 was not).
    float far = 2.f;
#pragma unroll
    for (int a = 0; a < D; ++a) far += __double2float_ru(fmax(fabs(m.dlo[a]), fabs(m.dhi[a]))) / s[a];
    const float minor = D == 3 ? s[1] * s[D - 1] : s[1];
    const float S = s[0] * minor, tau = 0x1p-16f * R * S;
    // These are relative roundings, true while every product of the evaluation,
    // and in double-float its part of 2^-48 too, is a normal float: R, the rows
    // and the products of rows that the determinant forms lie far enough inside
    // that range, or the filter declines (2D, uniform cells, density 1e-42: an
    // FP32 product is a few of the smallest float there, and 3 in 1,000 of the
    // decisions taken from it were wrong).
    float least = fminf(fminf(R, S), fminf(minor, R * S)), most = fmaxf(fmaxf(R, S), fmaxf(minor, R * S));
#pragma unroll
    for (int a = 0; a < D; ++a) {
      least = fminf(least, s[a]);
      most = fmaxf(most, s[a]);
    }
    const bool normal32 = least > 0x1p-100f && most < 0x1p100f, normal_df = least > 0x1p-74f && normal32;
    const float sequence = 0x1.4p-28f * far * tau;
    sure32 = normal32 ? 2.5f * tau + sequence : INFINITY;
    sure_df = normal_df ? 0x1p-18f * tau + sequence : INFINITY;
  }

  __device__ __forceinline__ float at(const float t[D]) const {
    float m[4], J[D][D], r;
    mixed32<D>(t, m);
    if constexpr (D == 2) {
      r = c[0] + (c[1] * t[0] + (c[2] * t[1] + c[3] * m[0]));
    } else {
      r = c[0] + (c[1] * t[0] + (c[2] * t[1] + (c[3] * t[2] + (c[4] * m[0] + (c[5] * m[1] + (c[6] * m[2] + c[7] * m[3]))))));
    }
#pragma unroll
    for (int i = 0; i < D; ++i) jacobian_row32<D>(row[i], t, m, J[i]);
    float det;
    if constexpr (D == 2)
      det = J[0][0] * J[1][1] - J[0][1] * J[1][0];
    else
      det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) + J[0][1] * (J[1][2] * J[2][0] - J[1][0] * J[2][2]) +
            J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
    return r * fabsf(det);
  }
};

// Thread per cell: the cell's chain, started at the centre; step st of the
// chain is global step g = J * cell_off[K] + st and uses SplitMix64 outputs
// g (D+1) + a (proposal coordinate a) and g (D+1) + D (acceptance uniform).
// States J, 2J, ... become the cell's particles, in order.
//
// A step only needs the sign of u rho-hat(current) - rho-hat(proposal).  It is
// taken from FP32 values where they differ by more than their error bound, and
// in double-float or by the written IEEE sequence otherwise (mh_accept_rn), so
// the decisions are those of the sequence.  Evaluating the sequence at every
// proposal, 239 FP64 operations, held the FP64 pipe 83 % busy: 12.8 ms for
// 1.77 M particles at J = 8.
template <int D>
__global__ void __launch_bounds__(128, 5) mh_seed_kernel(const __grid_constant__ MeshView m, const __grid_constant__ StoreView s, const uint32_t* __restrict__ cell_off,
                                                      const double* __restrict__ rho, uint32_t J, uint64_t seed,
                                                      uint64_t first_id) {
  constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
  for (uint32_t K = blockIdx.x * blockDim.x + threadIdx.x; K < m.C; K += gridDim.x * blockDim.x) {
    const uint32_t beg = cell_off[K], end = cell_off[K + 1];
    if (end > s.cap || beg >= end) continue;
    RhoHat32<D> f;
    f.load(m, K, rho);
    RawPoint<D> cur;
    float t32[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      cur.r[a] = 0;
      t32[a] = 0.5f;
    }
    bool at_centre = true;
    float rc = f.at(t32);
    const uint64_t g0 = (uint64_t)J * beg, len = (uint64_t)J * (end - beg);
    uint64_t z = seed + g0 * (D + 1) * kGamma;  // the generator's state before the step's first output
    uint32_t q = beg;
    uint32_t phase = 0;
    for (uint64_t st = 0; st < len; ++st) {
      RawPoint<D> y;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        y.r[a] = splitmix64_mix(z += kGamma);
        t32[a] = (float)(uint32_t)(y.r[a] >> 40) * 0x1p-24f;
      }
      const uint64_t ur = splitmix64_mix(z += kGamma);
      const float ry = f.at(t32);
      const float diff = ry - (float)(uint32_t)(ur >> 40) * 0x1p-24f * rc;
      bool accept = diff > f.sure32;
      if (!(fabsf(diff) > f.sure32)) accept = mh_accept_rn<D>(m, K, rho, cur, y, at_centre, unit53(ur), f.sure_df);
      if (accept) {
        cur = y;
        rc = ry;
        at_centre = false;
      }
      if (++phase == J) {
        phase = 0;
        mh_emit<D>(m, s, K, cur, at_centre, q, first_id + q);
        ++q;
      }
    }
  }
}

// ------------------------------------------------------- prescribed points

__global__ void found_flags_kernel(const uint32_t* __restrict__ cell, size_t n, uint32_t C, uint32_t* __restrict__ f) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    f[i] = cell[i] < C ? 1u : 0u;
}

__global__ void import_ids_kernel(const uint32_t* __restrict__ rank, size_t n, uint64_t first_id,
                                  uint64_t* __restrict__ id) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    id[i] = first_id + rank[i];
}

template <int D>
__global__ void import_gather_kernel(const __grid_constant__ StoreView s, const uint32_t* __restrict__ perm, const uint32_t* __restrict__ kept_p,
                                     size_t n, const double* __restrict__ x, const double* __restrict__ xh,
                                     const uint32_t* __restrict__ cell, const uint64_t* __restrict__ id) {
  const uint32_t kept = *kept_p;
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < kept; j += gridDim.x * blockDim.x) {
    const uint32_t i = perm[j];
    if (i >= n || j >= s.cap) continue;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      s.x[a * s.cap + j] = x[a * n + i];
      const double t = xh[a * n + i];
      const float hi = __double2float_rn(t);
      s.xhat[a * s.cap + j] = make_float2(hi, __double2float_rn(t - (double)hi));
    }
    s.id[j] = id[i];
    s.cell[j] = cell[i];
    for (int p = 0; p < s.n_props; ++p) s.props[(size_t)p * s.cap + j] = 0.0;
  }
}

static int gen_grid(size_t n, int block) {
  size_t g = (n + block - 1) / block;
  const size_t cap = (size_t)num_sms() * 16;
  if (g > cap) g = cap;
  return (int)(g ? g : 1);
}

}  // namespace pic

using namespace pic;

extern "C" pic_status pic_cell_weights(pic_mesh mesh, const double* rho, double* w, void* stream) {
  if (!mesh || !rho || !w) return (set_error("pic_cell_weights: null argument"), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  const MeshView m = mesh_view(mesh);
  if (mesh->dim == 2)
    cell_weights_kernel<2><<<gen_grid(m.C, 128), 128, 0, st>>>(m, rho, w);
  else
    cell_weights_kernel<3><<<gen_grid(m.C, 128), 128, 0, st>>>(m, rho, w);
  count_launches(1);
  PIC_CUDA(cudaGetLastError());
  return PIC_OK;
}

extern "C" pic_status pic_draw_cell_counts(uint32_t n_cells, const double* w, uint64_t n_particles, uint64_t seed,
                                           uint32_t* counts, void* stream) {
  if (!w || !counts || n_cells == 0) return (set_error("pic_draw_cell_counts: null argument or no cells"), PIC_ERR_ARG);
  if (n_particles >= 0xFFFFFFF0ull)
    return (set_error("pic_draw_cell_counts: %llu particles exceed the 32-bit store",
                      (unsigned long long)n_particles),
            PIC_ERR_CAPACITY);
  cudaStream_t st = (cudaStream_t)stream;
  double* acc = nullptr;
  DrawInfo* info = nullptr;
  void* scratch = nullptr;
  Slab slab;
  slab.add(&acc, n_cells);
  slab.add(&info, 1);
  if (!slab.allocate(&scratch))
    return (set_error("pic_draw_cell_counts: device allocation failed"), PIC_ERR_OOM);
  accumulate_weights_kernel<<<1, kFoldThreads, 0, st>>>(w, n_cells, acc, info);
  DrawInfo h{};
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, info, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    cudaFree(scratch);
    return cuda_fail(e, "pic_draw_cell_counts: accumulate");
  }
  if (h.bad || !(h.W > 0.0) || !std::isfinite(h.W)) {
    cudaFree(scratch);
    return (set_error("pic_draw_cell_counts: weights must be finite and >= 0 with a positive sum"), PIC_ERR_ARG);
  }
  e = cudaMemsetAsync(counts, 0, sizeof(uint32_t) * n_cells, st);
  if (e == cudaSuccess && n_particles > 0) {
    draw_cells_kernel<<<gen_grid((size_t)n_particles, 256), 256, 0, st>>>(acc, n_cells, info, n_particles, seed,
                                                                          counts);
    e = cudaGetLastError();
  }
  count_launches(n_particles > 0 ? 2 : 1);
  cudaFreeAsync(scratch, st);
  if (e != cudaSuccess) return cuda_fail(e, "pic_draw_cell_counts: draws");
  return PIC_OK;
}

extern "C" pic_status pic_seed_particles_mh(pic_mesh mesh, const uint32_t* per_cell, const double* rho,
                                            uint32_t thinning, uint64_t seed, uint64_t first_id, int n_props,
                                            size_t capacity, void* stream, pic_particles* out) {
  if (!out) return (set_error("pic_seed_particles_mh: out is NULL"), PIC_ERR_ARG);
  *out = nullptr;
  if (!mesh || !per_cell || !rho) return (set_error("pic_seed_particles_mh: null argument"), PIC_ERR_ARG);
  if (thinning < 1) return (set_error("pic_seed_particles_mh: thinning must be >= 1"), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  pic_particles_s* p = nullptr;
  size_t N = 0;
  pic_status r = seed_prepare(mesh, per_cell, 0, n_props, capacity, st, "pic_seed_particles_mh", &p, &N);
  if (r != PIC_OK) return r;
  const MeshView m = mesh_view(mesh);
  if (mesh->dim == 2)
    mh_seed_kernel<2><<<gen_grid(m.C, 128), 128, 0, st>>>(m, store_view(p, 0), p->cell_off, rho, thinning, seed,
                                                          first_id);
  else
    mh_seed_kernel<3><<<gen_grid(m.C, 128), 128, 0, st>>>(m, store_view(p, 0), p->cell_off, rho, thinning, seed,
                                                          first_id);
  count_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    pic_destroy_particles(p);
    return cuda_fail(e, "pic_seed_particles_mh: kernel");
  }
  *out = p;
  return PIC_OK;
}

extern "C" pic_status pic_import_particles(pic_mesh mesh, size_t n, const double* x, uint64_t first_id, int n_props,
                                           size_t capacity, void* stream, pic_particles* out, size_t* n_outside) {
  if (!out) return (set_error("pic_import_particles: out is NULL"), PIC_ERR_ARG);
  *out = nullptr;
  if (!mesh || (n > 0 && !x)) return (set_error("pic_import_particles: null argument"), PIC_ERR_ARG);
  if (n >= 0xFFFFFFF0ull) return (set_error("pic_import_particles: n exceeds the 32-bit store"), PIC_ERR_CAPACITY);
  if (n_props < 0 || n_props > kMaxProps)
    return (set_error("pic_import_particles: n_props must be in [0, %d]", kMaxProps), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  const uint32_t C = mesh->C;
  const int d = mesh->dim;
  const size_t nn = n > 0 ? n : 1;
  uint32_t *cell = nullptr, *flag = nullptr, *rank = nullptr, *sums = nullptr, *total = nullptr, *perm = nullptr,
           *off = nullptr;
  double* xh = nullptr;
  uint64_t* id = nullptr;
  void* scratch = nullptr;
  Slab slab;
  slab.add(&cell, nn);
  slab.add(&flag, nn);
  slab.add(&rank, nn + 1);
  slab.add(&sums, scan_scratch_bytes((uint32_t)nn) / sizeof(uint32_t));
  slab.add(&total, 2);
  slab.add(&perm, nn);
  slab.add(&xh, (size_t)d * nn);
  slab.add(&id, nn);
  const bool ok = slab.allocate(&scratch) && cudaMalloc(&off, sizeof(uint32_t) * (C + 1)) == cudaSuccess;
  auto release = [&](bool keep_off) {
    cudaFree(scratch);
    if (!keep_off) cudaFree(off);
  };
  if (!ok) {
    cudaGetLastError();
    release(false);
    return (set_error("pic_import_particles: device allocation failed"), PIC_ERR_OOM);
  }
  pic_status r = PIC_OK;
  uint32_t kept = 0;
  if (n > 0) {
    r = pic_locate_points(mesh, n, x, nullptr, cell, xh, stream);
    if (r == PIC_OK) {
      found_flags_kernel<<<gen_grid(n, 256), 256, 0, st>>>(cell, n, C, flag);
      r = scan_u32(flag, rank, (uint32_t)n, sums, total, nullptr, st);
    }
    if (r == PIC_OK) {
      import_ids_kernel<<<gen_grid(n, 256), 256, 0, st>>>(rank, n, first_id, id);
      count_launches(2);
      r = pic_sort_by_cell(n, cell, id, C, perm, off, stream);
    }
    if (r == PIC_OK) {
      cudaError_t e = cudaMemcpyAsync(&kept, off + C, sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) r = cuda_fail(e, "pic_import_particles: count");
    }
  } else {
    cudaError_t e = cudaMemsetAsync(off, 0, sizeof(uint32_t) * (C + 1), st);
    if (e != cudaSuccess) r = cuda_fail(e, "pic_import_particles: offsets");
  }
  if (r == PIC_OK && capacity == 0) capacity = kept;
  if (r == PIC_OK && capacity < kept)
    r = (set_error("pic_import_particles: capacity %zu < %u particles", capacity, kept), PIC_ERR_CAPACITY);
  if (r != PIC_OK) {
    release(false);
    return r;
  }
  pic_particles_s* p = store_alloc(d, n_props, C, capacity, off);  // takes `off`
  if (!p) {
    release(true);
    return PIC_ERR_OOM;
  }
  p->mesh = mesh;
  p->stream = st;
  cudaError_t e = store_init(p, kept, st);
  if (e == cudaSuccess && kept > 0) {
    if (d == 2)
      import_gather_kernel<2><<<gen_grid(kept, 128), 128, 0, st>>>(store_view(p, 0), perm, off + C, n, x, xh, cell, id);
    else
      import_gather_kernel<3><<<gen_grid(kept, 128), 128, 0, st>>>(store_view(p, 0), perm, off + C, n, x, xh, cell, id);
    count_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  release(true);
  if (e != cudaSuccess) {
    pic_destroy_particles(p);
    return cuda_fail(e, "pic_import_particles: gather");
  }
  p->cur = 0;
  if (n_outside) *n_outside = n - kept;
  *out = p;
  return PIC_OK;
}
