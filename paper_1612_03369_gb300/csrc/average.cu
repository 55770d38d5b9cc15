// average.cu -- particle -> cell transfer, scheme (ii) of Sec. 2.7
// (arithmetic average of the particles of each cell; linear in the particle
// count because the store is sorted by cell).
#include "pic_internal.cuh"

namespace pic {

// Thread per cell: the particles of a cell are folded in store order (the
// order of the definition), then combined with their number.  The threads of
// a warp read neighbouring segments, so every sector fetched from HBM is used
// by the following iterations through L1.  Kinds (Sec. 2.7 (ii)):
//   0 arithmetic  sum v / n
//   1 geometric   (product v)^(1/n)     (NaN if the cell holds a v <= 0)
//   2 harmonic    n / sum (1 / v)      (NaN if the cell holds a v <= 0)
// The geometric mean multiplies significands and adds exponents, so it takes
// one logarithm per cell instead of one per particle: with v_i = m_i 2^e_i, P 2^E
// their product and E = q n + r, it is 2^q exp((r log 2 + log P) / n).  The
// product's relative rounding, sqrt(n) 2^-53, counts 1/n of itself in the mean.
// (An FP64 logarithm per particle: 332 us at 64^3 x 20, FP64-pipe bound.)
// PERM (an order left pending by pic_advect): slot i's value is
// prop[perm[i]], the same values in the same order as after the gather.
struct ProductAcc {
  double P = 1.0;     // in [1, 2)
  long long E = 0;
  bool infinite = false;

  // Takes v in (0, inf]; false for anything else.  The tests are on the bits:
  // an FP64 comparison would cost as much as the product.
  __device__ __forceinline__ bool mul(double v) {
    int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    if (hi < 0 || ((unsigned)hi | lo) == 0u) return false;
    if (hi >= 0x7ff00000) {
      infinite = true;
      return hi == 0x7ff00000 && lo == 0u;
    }
    int e = hi >> 20;
    if (e == 0) {  // subnormal
      v *= 0x1p54;
      hi = __double2hiint(v);
      e = (hi >> 20) - 54;
    }
    P *= __hiloint2double((hi & 0xfffff) | 0x3ff00000, __double2loint(v));
    const int top = __double2hiint(P);
    const int carry = (top >> 20) - 1023;  // 0 or 1
    P = __hiloint2double(top - (carry << 20), __double2loint(P));
    E += e - 1023 + carry;
    return true;
  }
  __device__ __forceinline__ double mean(uint32_t n) const {
    if (infinite) return __longlong_as_double(0x7ff0000000000000ll);
    long long q = E / (long long)n, r = E % (long long)n;
    if (r < 0) {
      r += n;
      --q;
    }
    return ldexp(exp(((double)r * 0.6931471805599453094 + log(P)) / (double)n), (int)q);
  }
};

template <int KIND, bool PERM>
__global__ void __launch_bounds__(256) cell_average_kernel(const uint32_t* __restrict__ cell_off,
                                                           const double* __restrict__ prop,
                                                           const uint32_t* __restrict__ perm, uint32_t C, size_t cap,
                                                           double empty_fill, double* __restrict__ avg,
                                                           uint32_t* __restrict__ count, DevCounters* __restrict__ ctr) {
  for (uint32_t K = blockIdx.x * blockDim.x + threadIdx.x; K < C; K += gridDim.x * blockDim.x) {
    const uint32_t beg = cell_off[K], end = cell_off[K + 1];
    if (end > cap || beg > end) {
      latch_status(ctr, PIC_STATUS_BOUNDS);
      continue;
    }
    double s = 0.0;
    bool bad = false;
    ProductAcc product;
    // kBatch particles at a time: their loads (two dependent ones with PERM) are
    // in flight together, then folded in store order: 14 -> 7 us for 16^3 cells
    // and 42 -> 31 us for 64^3 through a pending order (settled, 4 at a time is
    // enough for 20 particles a cell)
    constexpr int kBatch = PERM ? 8 : 4;
    for (uint32_t i0 = beg; i0 < end; i0 += kBatch) {
      uint32_t src[kBatch];
      double v[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        src[q] = i0 + q;
        if constexpr (PERM) src[q] = i0 + q < end ? perm[i0 + q] : 0u;
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) v[q] = i0 + q < end && src[q] < cap ? prop[src[q]] : 0.0;
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        if (i0 + q >= end) break;
        if (PERM && src[q] >= cap) {
          bad = true;
          latch_status(ctr, PIC_STATUS_BOUNDS);
          continue;
        }
        if constexpr (KIND == 0) {
          s += v[q];
        } else {
          if constexpr (KIND == 1) {
            if (!product.mul(v[q])) bad = true;
          } else {
            bad = bad || !(v[q] > 0.0);
            s += 1.0 / v[q];
          }
        }
      }
    }
    const uint32_t n = end - beg;
    double r = empty_fill;
    if (n) {
      if constexpr (KIND == 0)
        r = s / (double)n;
      else if (bad)
        r = __longlong_as_double(0x7ff8000000000000ll);
      else
        r = (KIND == 1) ? product.mean(n) : (double)n / s;
    }
    avg[K] = r;
    if (count) count[K] = n;
  }
}

}  // namespace pic

using namespace pic;

extern "C" pic_status pic_interpolate_to_cells(pic_particles p, pic_mesh mesh, int prop, pic_average kind, double* avg,
                                               uint32_t* count, double empty_fill, void* stream) {
  if (!p || !mesh || !avg) return (set_error("pic_interpolate_to_cells: null argument"), PIC_ERR_ARG);
  if (p->mesh != mesh) return (set_error("pic_interpolate_to_cells: mesh mismatch"), PIC_ERR_ARG);
  if (prop < 0 || prop >= p->n_props)
    return (set_error("pic_interpolate_to_cells: property %d out of range", prop), PIC_ERR_ARG);
  if (kind != PIC_AVG_ARITHMETIC && kind != PIC_AVG_GEOMETRIC && kind != PIC_AVG_HARMONIC)
    return (set_error("pic_interpolate_to_cells: unknown average %d", (int)kind), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  size_t grid = ((size_t)p->C + 255) / 256;
  const size_t cap = (size_t)num_sms() * 16;
  if (grid > cap) grid = cap;
  const int g = (int)(grid ? grid : 1);
  const double* pv = p->props[p->cur] + (size_t)prop * p->capacity;
  // read through a pending order, do not apply it
  const uint32_t* pm = p->perm;
  const uint32_t C = p->C;
  const size_t cp = p->capacity;
  if (p->pending_order) {
    if (kind == PIC_AVG_ARITHMETIC)
      cell_average_kernel<0, true><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
    else if (kind == PIC_AVG_GEOMETRIC)
      cell_average_kernel<1, true><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
    else
      cell_average_kernel<2, true><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
  } else {
    if (kind == PIC_AVG_ARITHMETIC)
      cell_average_kernel<0, false><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
    else if (kind == PIC_AVG_GEOMETRIC)
      cell_average_kernel<1, false><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
    else
      cell_average_kernel<2, false><<<g, 256, 0, st>>>(p->cell_off, pv, pm, C, cp, empty_fill, avg, count, p->ctr);
  }
  count_launches(1);
  PIC_CUDA(cudaGetLastError());
  return PIC_OK;
}
