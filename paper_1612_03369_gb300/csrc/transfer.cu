// transfer.cu -- particle -> field transfers of Sec. 2.7 beyond cell
// averages, both linear in the number of particles because the store is
// sorted by cell:
//   (iv) shape-function-weighted averages at the mesh vertices,
//        p_v = sum_i phi_v(x_i) p_i / sum_i phi_v(x_i) over the particles of
//        the cells around v, phi_v the (bi/tri)linear nodal basis function
//   (v)  per-cell linear least squares in reference coordinates,
//        f(x-hat) = c_0 + sum_j c_{j+1} (x-hat_j - 1/2)
// No atomics, so the results are reproducible run to run.  The linear fit folds a
// cell's particles in store order.  The vertex sums are formed per cell first (one
// left fold, or four strided ones added in a fixed pattern, by the cells' counts) and
// the cells' partial sums then added in increasing cell index, which rounds differently
// from one left fold over the support (the definition) by a few ulps of the sum.
#include "df.cuh"
#include "pic_internal.cuh"

namespace pic {

// The arithmetic per particle is double-float on the FP32 pipe (the stored
// x-hat already is a double-float pair; the property is split once): GB300's
// FP64 pipe runs about 1/80 of the FP32 rate, and the FP64 form of these
// kernels was bound by it.  Every product keeps ~2^-47 of its value and the
// sums are compensated (acc_mad, acc_add), so the per-cell sums carry a
// relative error of a few 2^-47 against the FP64 definition.
__device__ __forceinline__ df one_minus(df t) {  // 1 - t
  const df d = two_sum(1.0f, -t.hi);
  return fast_two_sum(d.hi, __fsub_rn(d.lo, t.lo));
}
__device__ __forceinline__ df minus_half(df t) {  // t - 1/2
  const df d = two_sum(t.hi, -0.5f);
  return fast_two_sum(d.hi, __fadd_rn(d.lo, t.lo));
}
__device__ __forceinline__ double df_to_f64(df a) { return (double)a.hi + (double)a.lo; }

// In the vertex sums a cell is taken by one lane or by kLanes neighbouring ones,
// lane q then folding its particles q, q + kLanes, ..., and the lanes' compensated
// sums are added in a fixed pattern of exchanges.  Shared, the lanes' loads are
// consecutive, a 32-byte sector per cell and array, and a long cell holds its warp
// up a quarter as long; alone, every load of a warp touches 32 sectors of as many
// lines, but there are no exchanges.  The choice falls for 32 cells at a time, by the
// largest of them, so that the order of the sums is a function of the store's
// particles and the mesh (chosen by the store's capacity, two stores of the same
// particles differed in the last bits).  64^3 cells, the call with the vertices' pass
// and the launches, all alone / all shared: 6 per cell 61 / 78 us, 10 77 / 91, 14 94 /
// 102, 16 134 / 102, 36 197 / 164; unevenly filled, 4.9 per cell on average and up to 48
// in one, 135 / 107, 13 297 / 199; 500^2 cells cross at 13 per cell.  This rule: 65, 79,
// 93, 103, 164; 111, 211.
constexpr int kLanes = 4;
constexpr uint32_t kAloneUpTo = 14;

// The group's sums, dealt to its lanes: own[j] of lane q becomes the sum over the
// group of acc[kLanes j + q].  Each round halves what a lane holds, so an entry
// costs a lane 3/4 of an exchange and addition, 2 if every lane took every sum.
__device__ __forceinline__ df_acc exchange_add(const df_acc& even, const df_acc& odd, uint32_t bit, int mask) {
  const float s = __shfl_xor_sync(0xffffffffu, bit ? even.s : odd.s, mask);
  const float e = __shfl_xor_sync(0xffffffffu, bit ? even.e : odd.e, mask);
  df_acc r = bit ? odd : even;
  const df t = two_sum(r.s, s);
  r.s = t.hi;
  r.e = __fadd_rn(__fadd_rn(r.e, e), t.lo);
  return r;
}
template <int N>
__device__ __forceinline__ void group_sums(const df_acc (&acc)[N], df_acc (&own)[N / kLanes], uint32_t q) {
  static_assert(kLanes == 4 && N % 4 == 0, "two rounds");
  df_acc half[N / 2];
#pragma unroll
  for (int k = 0; k < N / 2; ++k) half[k] = exchange_add(acc[2 * k], acc[2 * k + 1], q & 1u, 1);
#pragma unroll
  for (int j = 0; j < N / 4; ++j) own[j] = exchange_add(half[2 * j], half[2 * j + 1], q >> 1, 2);
}

// One particle's loads, issued an iteration ahead of their use.
template <int D>
struct ParticleLoads {
  float2 t[D];
  double p;
  __device__ __forceinline__ void load(const float2* __restrict__ xh, const double* __restrict__ prop, size_t cap,
                                       uint32_t i, uint32_t end) {
    if (i >= end) return;
#pragma unroll
    for (int a = 0; a < D; ++a) t[a] = xh[a * cap + i];
    p = prop[i];
  }
};

// A cell's particles (none past the last cell); a segment outside the store is
// flagged and taken as empty.
__device__ __forceinline__ void cell_segment(const uint32_t* __restrict__ cell_off, uint32_t K, uint32_t C, size_t cap,
                                             uint32_t& beg, uint32_t& end, DevCounters* __restrict__ ctr) {
  beg = K < C ? cell_off[K] : 0u;
  end = K < C ? cell_off[K + 1] : 0u;
  if (end > cap || beg > end) {
    latch_status(ctr, PIC_STATUS_BOUNDS);
    beg = end = 0;
  }
}

// Two phases, both deterministic.
// Phase 1, L lanes (kLanes or 1) per cell: each particle of the cell is read once and
// its 2^D corner weights (the tensor product of (1 - t_a, t_a), multiplied in
// axis order) are folded into the cell's partial sums
//   num[c][K] = sum w_c(x-hat_i) p_i,   den[c][K] = sum w_c(x-hat_i)
// stored as double-float pairs, corner-major ([c][C]) so that the phase-2
// reads of a warp coalesce.
template <int D, int L>
__device__ __forceinline__ void vertex_partial_sums(uint32_t K, uint32_t beg, uint32_t end, uint32_t q,
                                                    const float2* __restrict__ xh, const double* __restrict__ prop,
                                                    uint32_t C, size_t cap, float2* __restrict__ part) {
  constexpr int NC = 1 << D;
  df_acc num[NC], den[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) num[c] = den[c] = acc_zero();
  ParticleLoads<D> next;
  next.load(xh, prop, cap, beg + q, end);
  for (uint32_t i = beg + q; i < end; i += L) {
    const ParticleLoads<D> now = next;
    next.load(xh, prop, cap, i + L, end);
    df f[D][2];  // f[a][0] = 1 - t_a, f[a][1] = t_a
#pragma unroll
    for (int a = 0; a < D; ++a) {
      f[a][1] = df_make(now.t[a].x, now.t[a].y);
      f[a][0] = one_minus(f[a][1]);
    }
    const df p = split_f64(now.p);
    df w01[4];  // the first two axes' products, corner bits 0 and 1
#pragma unroll
    for (int c = 0; c < 4; ++c) w01[c] = df_mul(f[0][c & 1], f[1][(c >> 1) & 1]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const df w = D == 3 ? df_mul(w01[c & 3], f[D - 1][(c >> 2) & 1]) : w01[c];
      acc_mad(num[c], w, p);
      acc_add(den[c], w);
    }
  }
  df_acc num_q[NC / L], den_q[NC / L];
  if constexpr (L == 1) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      num_q[c] = num[c];
      den_q[c] = den[c];
    }
  } else {
    group_sums(num, num_q, q);
    group_sums(den, den_q, q);
  }
  if (K < C)
#pragma unroll
    for (int j = 0; j < NC / L; ++j) {
      const size_t c = (size_t)(L * j) + q;
      const df a = acc_result(num_q[j]), b = acc_result(den_q[j]);
      part[c * C + K] = make_float2(a.hi, a.lo);
      part[(NC + c) * C + K] = make_float2(b.hi, b.lo);
    }
}

// A block takes `per_block` (1 or 4) groups of 32 cells at a time: alone, one of its
// warps takes a group; shared, every warp eight of the group's cells.
template <int D>
__global__ void __launch_bounds__(128) vertex_partial_kernel(const uint32_t* __restrict__ cell_off,
                                                             const float2* __restrict__ xh, const double* __restrict__ prop,
                                                             uint32_t C, size_t cap, uint32_t per_block,
                                                             float2* __restrict__ part, DevCounters* __restrict__ ctr) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t groups = (C + 31u) / 32u;
  for (uint32_t g0 = blockIdx.x * per_block; g0 < groups; g0 += gridDim.x * per_block) {
    for (uint32_t g = 0; g < per_block && g0 + g < groups; ++g) {
      const uint32_t K0 = (g0 + g) * 32u;
      uint32_t beg, end;
      cell_segment(cell_off, K0 + lane, C, cap, beg, end, ctr);
      if (__reduce_max_sync(0xffffffffu, end - beg) <= kAloneUpTo) {
        if (warp == g) vertex_partial_sums<D, 1>(K0 + lane, beg, end, 0u, xh, prop, C, cap, part);
      } else {
        const uint32_t k = warp * (32 / kLanes) + lane / kLanes;
        beg = __shfl_sync(0xffffffffu, beg, k);
        end = __shfl_sync(0xffffffffu, end, k);
        vertex_partial_sums<D, kLanes>(K0 + k, beg, end, lane % kLanes, xh, prop, C, cap, part);
      }
    }
  }
}

// Phase 2, thread per vertex: the partial sums of the cells around the
// vertex, added in increasing cell index (double-float), then one FP64
// division.
template <int D>
__global__ void __launch_bounds__(256) vertex_gather_kernel(const __grid_constant__ MeshView m, const float2* __restrict__ part,
                                                            double empty_fill, double* __restrict__ avg,
                                                            double* __restrict__ weight) {
  constexpr int NC = 1 << D;
  const uint32_t nv = (uint32_t)m.nverts, C = m.C;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    int vc[3];
    vc[0] = (int)(v % (uint32_t)m.nv[0]);
    const uint32_t r = v / (uint32_t)m.nv[0];
    vc[1] = D == 3 ? (int)(r % (uint32_t)m.nv[1]) : (int)r;
    vc[2] = D == 3 ? (int)(r / (uint32_t)m.nv[1]) : 0;
    df_acc num = acc_zero(), den = acc_zero();
#pragma unroll
    for (int o = 0; o < NC; ++o) {
      // bit a of o is the offset along axis a (x fastest, the last axis
      // slowest), so the cells come in increasing index
      int c[3] = {0, 0, 0}, corner = 0;
      bool ok = true;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        c[a] = vc[a] - 1 + ((o >> a) & 1);
        ok = ok && c[a] >= 0 && c[a] < m.n[a];
        corner |= (vc[a] - c[a]) << a;
      }
      if (!ok) continue;
      const uint32_t K = cell_index<D>(m, c[0], c[1], c[2]);
      const float2 a = part[(size_t)corner * C + K], b = part[(size_t)(NC + corner) * C + K];
      acc_add(num, df_make(a.x, a.y));
      acc_add(den, df_make(b.x, b.y));
    }
    const double dn = df_to_f64(acc_result(den));
    avg[v] = dn > 0.0 ? df_to_f64(acc_result(num)) / dn : empty_fill;
    if (weight) weight[v] = dn;
  }
}

// Thread per cell: normal equations (A^T A) c = A^T p of the cell's design
// matrix, rows (1, x-hat_i - 1/2), folded in store order; Gaussian
// elimination with partial pivoting; the mean where the cell has at most D
// particles or a pivot is <= 1e-12 of the largest diagonal entry.
// The fold stays one left fold per sum: a pivot may be 1e-12 of the diagonal, and a
// sum folded in another order (four lanes a cell: 115 -> 104 us a call at 64^3 x 20) would
// move such a cell's coefficients by 1e12 times its rounding.
template <int D>
__global__ void __launch_bounds__(128) lsq_linear_kernel(const uint32_t* __restrict__ cell_off,
                                                         const float2* __restrict__ xh, const double* __restrict__ prop,
                                                         uint32_t C, size_t cap, double empty_fill,
                                                         double* __restrict__ coef, uint32_t* __restrict__ count,
                                                         DevCounters* __restrict__ ctr) {
  constexpr int NB = D + 1;
  for (uint32_t K = blockIdx.x * blockDim.x + threadIdx.x; K < C; K += gridDim.x * blockDim.x) {
    const uint32_t beg = cell_off[K], end = cell_off[K + 1];
    if (end > cap || beg > end) {
      latch_status(ctr, PIC_STATUS_BOUNDS);
      continue;
    }
    // the upper triangle of A^T A, A^T p and sum p, accumulated in
    // double-float (row a = (1, x-hat - 1/2)), then converted once
    df_acc Ma[NB][NB + 1];
#pragma unroll
    for (int r = 0; r < NB; ++r)
#pragma unroll
      for (int q = 0; q <= NB; ++q) Ma[r][q] = acc_zero();
    ParticleLoads<D> next;
    next.load(xh, prop, cap, beg, end);
    for (uint32_t i = beg; i < end; ++i) {
      const ParticleLoads<D> now = next;
      next.load(xh, prop, cap, i + 1, end);
      df a[NB];
      a[0] = df_make(1.0f, 0.f);
#pragma unroll
      for (int j = 0; j < D; ++j) a[j + 1] = minus_half(df_make(now.t[j].x, now.t[j].y));
      const df p = split_f64(now.p);
#pragma unroll
      for (int r = 0; r < NB; ++r) {
#pragma unroll
        for (int q = r; q < NB; ++q) {
          if (r == 0 && q == 0) continue;  // the count
          if (r == 0)
            acc_add(Ma[r][q], a[q]);  // a[0] = 1
          else
            acc_mad(Ma[r][q], a[r], a[q]);
        }
        if (r == 0)
          acc_add(Ma[r][NB], p);
        else
          acc_mad(Ma[r][NB], a[r], p);
      }
    }
    double M[NB][NB + 1];
#pragma unroll
    for (int r = 0; r < NB; ++r)
#pragma unroll
      for (int q = r; q <= NB; ++q) M[r][q] = df_to_f64(acc_result(Ma[r][q]));
    M[0][0] = (double)(end - beg);
    const double sum = M[0][NB];
#pragma unroll
    for (int r = 1; r < NB; ++r)
#pragma unroll
      for (int q = 0; q < r; ++q) M[r][q] = M[q][r];
    const uint32_t n = end - beg;
    double c[NB];
#pragma unroll
    for (int r = 0; r < NB; ++r) c[r] = 0.0;
    if (n == 0) {
      c[0] = empty_fill;
    } else {
      bool ok = n > (uint32_t)D;
      double dmax = 0.0, invd[NB];
#pragma unroll
      for (int r = 0; r < NB; ++r) dmax = M[r][r] > dmax ? M[r][r] : dmax;
#pragma unroll
      for (int col = 0; col < NB; ++col) {
        if (!ok) break;
        int piv = col;
        double best = fabs(M[col][col]);
#pragma unroll
        for (int r = col + 1; r < NB; ++r)
          if (fabs(M[r][col]) > best) {
            best = fabs(M[r][col]);
            piv = r;
          }
        if (!(best > 1e-12 * dmax)) {
          ok = false;
          break;
        }
        // the swap with compile-time row indices keeps M in registers
#pragma unroll
        for (int r = col + 1; r < NB; ++r)
          if (r == piv) {
#pragma unroll
            for (int q = 0; q <= NB; ++q) {
              const double t = M[col][q];
              M[col][q] = M[r][q];
              M[r][q] = t;
            }
          }
        // one reciprocal per pivot (FP64 divisions are sequences on the FP64
        // pipe; the solve's rounding is covered by the kappa-scaled bound)
        const double inv = 1.0 / M[col][col];
        invd[col] = inv;
#pragma unroll
        for (int r = col + 1; r < NB; ++r) {
          const double f = M[r][col] * inv;
#pragma unroll
          for (int q = col; q <= NB; ++q) M[r][q] -= f * M[col][q];
        }
      }
      if (ok) {
#pragma unroll
        for (int r = NB - 1; r >= 0; --r) {
          double s = M[r][NB];
#pragma unroll
          for (int q = r + 1; q < NB; ++q) s -= M[r][q] * c[q];
          c[r] = s * invd[r];
        }
      } else {
        c[0] = sum / (double)n;
      }
    }
#pragma unroll
    for (int r = 0; r < NB; ++r) coef[(size_t)r * C + K] = c[r];
    if (count) count[K] = n;
  }
}

static int transfer_grid(size_t n, int block) {
  size_t g = (n + block - 1) / block;
  const size_t cap = (size_t)num_sms() * 16;
  if (g > cap) g = cap;
  return (int)(g ? g : 1);
}

}  // namespace pic

using namespace pic;

extern "C" pic_status pic_interpolate_to_vertices(pic_particles p, pic_mesh mesh, int prop, double* avg,
                                                  double* weight, double empty_fill, void* stream) {
  if (!p || !mesh || !avg) return (set_error("pic_interpolate_to_vertices: null argument"), PIC_ERR_ARG);
  if (p->mesh != mesh) return (set_error("pic_interpolate_to_vertices: mesh mismatch"), PIC_ERR_ARG);
  if (prop < 0 || prop >= p->n_props)
    return (set_error("pic_interpolate_to_vertices: property %d out of range", prop), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  {
    const pic_status r0 = settle_order(p, st);
    if (r0 != PIC_OK) return r0;
  }
  const MeshView m = mesh_view(mesh);
  if (!p->xfer) {
    const size_t bytes = sizeof(double) * 2 * ((size_t)1 << mesh->dim) * (size_t)p->C;
    if (cudaMalloc(&p->xfer, bytes) != cudaSuccess) {
      cudaGetLastError();
      p->xfer = nullptr;
      return (set_error("pic_interpolate_to_vertices: cannot allocate %zu bytes", bytes), PIC_ERR_OOM);
    }
  }
  const double* pv = p->props[p->cur] + (size_t)prop * p->capacity;
  // four groups per block where that leaves every SM its blocks and groups may be taken
  // alone, so that each warp has one (64^3 x 12: 86 us, 101 with one group per block);
  // otherwise one, as shared groups are 2 to 5 % faster that way.  Only the time depends
  // on it.
  const size_t groups = ((size_t)p->C + 31) / 32;
  const uint32_t per_block = groups >= (size_t)num_sms() * 16 && p->capacity < (size_t)p->C * (kAloneUpTo + 1) ? 4u : 1u;
  const int g1 = transfer_grid((groups + per_block - 1) / per_block * 128, 128), g2 = transfer_grid((size_t)m.nverts, 256);
  float2* part = reinterpret_cast<float2*>(p->xfer);  // [2 * 2^dim][C] double-float pairs
  if (mesh->dim == 2) {
    vertex_partial_kernel<2><<<g1, 128, 0, st>>>(p->cell_off, p->xhat[p->cur], pv, p->C, p->capacity, per_block, part,
                                                  p->ctr);
    vertex_gather_kernel<2><<<g2, 256, 0, st>>>(m, part, empty_fill, avg, weight);
  } else {
    vertex_partial_kernel<3><<<g1, 128, 0, st>>>(p->cell_off, p->xhat[p->cur], pv, p->C, p->capacity, per_block, part,
                                                  p->ctr);
    vertex_gather_kernel<3><<<g2, 256, 0, st>>>(m, part, empty_fill, avg, weight);
  }
  count_launches(2);
  PIC_CUDA(cudaGetLastError());
  return PIC_OK;
}

extern "C" pic_status pic_project_linear(pic_particles p, pic_mesh mesh, int prop, double* coef, uint32_t* count,
                                         double empty_fill, void* stream) {
  if (!p || !mesh || !coef) return (set_error("pic_project_linear: null argument"), PIC_ERR_ARG);
  if (p->mesh != mesh) return (set_error("pic_project_linear: mesh mismatch"), PIC_ERR_ARG);
  if (prop < 0 || prop >= p->n_props)
    return (set_error("pic_project_linear: property %d out of range", prop), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  {
    const pic_status r0 = settle_order(p, st);
    if (r0 != PIC_OK) return r0;
  }
  const double* pv = p->props[p->cur] + (size_t)prop * p->capacity;
  const int g = transfer_grid((size_t)p->C, 128);
  if (mesh->dim == 2)
    lsq_linear_kernel<2><<<g, 128, 0, st>>>(p->cell_off, p->xhat[p->cur], pv, p->C, p->capacity, empty_fill, coef,
                                            count, p->ctr);
  else
    lsq_linear_kernel<3><<<g, 128, 0, st>>>(p->cell_off, p->xhat[p->cur], pv, p->C, p->capacity, empty_fill, coef,
                                            count, p->ctr);
  count_launches(1);
  PIC_CUDA(cudaGetLastError());
  return PIC_OK;
}
