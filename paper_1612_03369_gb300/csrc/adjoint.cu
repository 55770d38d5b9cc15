// adjoint.cu -- gradients of a function of the final particle positions with
// respect to the Q2 nodal velocities (the adjoint of the Sec. 2.3 integrators
// over located stages), for inverse flow reconstruction from tracer
// endpoints.
//
// pic_advect_record advances the store like pic_advect and keeps, for every
// step, each particle's stage records (the located cell and double-float
// x-hat of every stage point, exactly as the step used them) and the rebin's
// permutation (new slot -> old slot).  A checkpoint tape keeps instead the
// store at the start of each step and replays the step in the sweep with the
// same particle step, which rewrites the same records (half the memory, one
// more advect per step).  pic_tape_adjoint then sweeps the steps backwards.  For one step, with y_s = x + a_s k_{s-1}, k_s = dt u(y_s),
// x' = x + sum_s b_s k_s and G_s = du/dx at y_s (cell held fixed):
//   lambda_k_s = b_s lambda' + a_{s+1} lambda_y_{s+1}
//   lambda_y_s = dt G_s^T lambda_k_s,       lambda = lambda' + sum_s lambda_y_s
//   dL/dU_i   += dt phi-hat_i(x-hat_s) lambda_k_s
// G and lambda in double-float.  Each stage's contribution (stage cell,
// x-hat_s, dt lambda_k_s) is a record keyed by (stage, slot); the records are
// sorted by (cell, stage, slot), summed per cell in that order, and the cells' sums
// are added into the nodes in increasing cell order.  No floating-point
// atomics, so the gradient is bit-for-bit reproducible.
#include <cmath>
#include <cstdlib>

#include "advect.cuh"
#include "fastpath.cuh"
#include "grad_df.cuh"
#include "locate.cuh"
#include "pic_internal.cuh"
#include "rebin.cuh"

struct pic_tape_s {
  pic_particles_s* parts;
  const pic_mesh_s* mesh;
  int dim, n_steps, integrator;
  double dt;
  size_t cap;
  uint32_t C;
  int kind;          // pic_tape_kind
  int n_rec;         // stage-record sets: n_steps (stage tapes) or 1 (the replay's, checkpoint tapes)
  uint32_t** rcell;  // [n_rec] of [4][cap]: stage cells (StageRec layout, slots of the start of the step)
  float2** rt;       // [n_rec] of [dim][4][cap]: stage x-hat, double-float
  double** x;        // checkpoint tapes: [n_steps] of [dim][cap], the store at the start of the step
  float2** xhat;     //   [n_steps] of [dim][cap]
  uint32_t** cell;   //   [n_steps] of [cap]
  double* sink_x;    //   [dim][cap] the replayed step's new positions (discarded)
  float2* sink_xhat; //   [dim][cap]
  uint32_t** perm;   // [n_steps] of [cap] (new slot -> old slot)
  uint32_t* n_dev;   // [n_steps + 1] particles at the start of each step (and at the end)
  // reverse-sweep work
  float2* lam[2];      // [dim][cap] double-float
  float2* rec_w;       // [dim][4 cap] double-float dt lambda_k
  uint32_t* rec_perm;  // [4 cap] the step's records sorted by (cell, stage, slot)
  uint32_t* rec_off;   // [4 C + 1] their offsets per (cell, stage)
  uint32_t *rec_counts, *rec_cursor;  // [4 C] sort scratch
  uint32_t *rec_scan, *rec_src;       // scan scratch, [4 cap]
  double* partial;     // [C][3^dim][dim]
  void* slab;          // the allocation that holds every device array above
};

namespace pic {

constexpr int kRecPerParticle = 4;

// The tableaux with a_s (a power of two or zero) as float and b_s as a
// double-float (1/6 and 1/3 to ~2^-48).
template <int RK>
struct AdjTableau;
template <>
struct AdjTableau<1> {
  static constexpr int S = 1;
  __device__ static float a(int) { return 0.f; }
  __device__ static df b(int) { return df_make(1.f, 0.f); }
};
template <>
struct AdjTableau<2> {
  static constexpr int S = 2;
  __device__ static float a(int s) { return s == 1 ? 0.5f : 0.f; }
  __device__ static df b(int s) { return df_make(s == 1 ? 1.f : 0.f, 0.f); }
};
template <>
struct AdjTableau<4> {
  static constexpr int S = 4;
  __device__ static float a(int s) { return s == 3 ? 1.f : (s == 0 ? 0.f : 0.5f); }
  __device__ static df b(int s) {
    return (s == 0 || s == 3) ? df_make(0.1666666716337204f, -4.967053879312289e-09f)
                              : df_make(0.3333333432674408f, -9.934107758624577e-09f);
  }
};

struct TapeStep {
  const uint32_t* rcell;
  const float2* rt;
  const uint32_t* perm;
  const uint32_t* n_next;  // particles after the step
};

// Resident blocks per SM requested from the register allocator for the
// lambda sweep (swept at build time with -DPIC_REVERSE_MIN_BLOCKS=n).
#ifndef PIC_REVERSE_MIN_BLOCKS
#define PIC_REVERSE_MIN_BLOCKS 4
#endif

// One reverse step, thread per particle alive after the step (new slot j,
// old slot i = perm[j]): the stages backwards with G_s = du/dx at the
// recorded stage points, all in double-float on the FP32 pipe:
//   lambda_k_s = b_s lambda' + a_{s+1} lambda_y_{s+1}
//   lambda_y_s = dt G_s^T lambda_k_s,   lambda = lambda' + sum_s lambda_y_s
// and record r = s cap + i gets its weight dt lambda_k_s and is counted at
// (its cell, s).
template <int D, int RK>
__global__ void __launch_bounds__(128, PIC_REVERSE_MIN_BLOCKS) reverse_lambda_kernel(
    const __grid_constant__ MeshView m, const __grid_constant__ TapeStep tp, size_t cap, df dt, const float2* __restrict__ lam_in, float2* __restrict__ lam_out,
    uint32_t* __restrict__ rec_counts, float2* __restrict__ rec_w, DevCounters* __restrict__ ctr) {
  using TB = AdjTableau<RK>;
  constexpr int S = TB::S;
  const uint32_t n = *tp.n_next;
  const size_t rcap = kRecPerParticle * cap;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t base = blockIdx.x * blockDim.x + threadIdx.x - lane; base < n; base += gridDim.x * blockDim.x) {
    const uint32_t j = base + lane;
    uint32_t i = 0, Ks[S];
    bool ok = j < n;
#pragma unroll
    for (int s = 0; s < S; ++s) Ks[s] = PIC_LOST;
    if (ok) {
      i = tp.perm[j];
      ok = i < cap;
#pragma unroll
      for (int s = 0; s < S; ++s) {
        if (ok) Ks[s] = tp.rcell[(size_t)s * cap + i];
        ok = ok && Ks[s] < m.C;
      }
      if (!ok) latch_status(ctr, PIC_STATUS_BOUNDS);  // cannot happen for a particle that survived the step
    }
    // the counts of the records' sort, one atomic per distinct (cell, stage) of
    // the warp
#pragma unroll
    for (int s = 0; s < S; ++s) (void)aggregated_increment(rec_counts, Ks[s] * kRecPerParticle + s, ok);
    if (!ok) continue;
    df lam[D], lam_x[D], lam_ynext[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const float2 v = lam_in[a * cap + j];
      lam[a] = df_make(v.x, v.y);
      lam_x[a] = lam[a];
      lam_ynext[a] = df_make(0.f, 0.f);
    }
#pragma unroll 1
    for (int s = S - 1; s >= 0; --s) {
      const size_t r = (size_t)s * cap + i;
      df t[D];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float2 v = tp.rt[a * rcap + r];
        t[a] = df_make(v.x, v.y);
      }
      uint32_t K = Ks[0];
#pragma unroll
      for (int q = 1; q < S; ++q) K = (s == q) ? Ks[q] : K;
      const df bs = TB::b(s);
      const float an = s + 1 < S ? TB::a(s + 1) : 0.f;
      df lk[D];
#pragma unroll
      for (int a = 0; a < D; ++a) lk[a] = df_add(df_mul(bs, lam[a]), df_scale2(lam_ynext[a], an));
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const df w = df_mul(dt, lk[a]);
        rec_w[a * rcap + r] = make_float2(w.hi, w.lo);
      }
      // G_s^T lambda_k = J^{-T} ((du/dx-hat)^T lambda_k), linear in lambda_k, which
      // takes whatever scale the loss has: solved for a lambda_k near 1
      df Gu[D][D], v[D], z[D];
      float largest = 0.f, scale, back;
#pragma unroll
      for (int a = 0; a < D; ++a) largest = fmaxf(largest, fabsf(lk[a].hi));
      pow2_near_one(largest, scale, back);
#pragma unroll
      for (int a = 0; a < D; ++a) lk[a] = df_scale2(lk[a], scale);
      q2_grad_mono_df<D>(m.Qc, K, t, Gu);
#pragma unroll
      for (int q = 0; q < D; ++q) {
        df_acc acc = acc_zero();
#pragma unroll
        for (int c = 0; c < D; ++c) acc_mad(acc, Gu[c][q], lk[c]);
        v[q] = acc_result(acc);
      }
      solve_transposed_df<D>(m, K, t, v, z);
#pragma unroll
      for (int q = 0; q < D; ++q) {
        lam_ynext[q] = df_mul(dt, df_scale2(z[q], back));
        lam_x[q] = df_add(lam_x[q], lam_ynext[q]);
      }
    }
#pragma unroll
    for (int a = 0; a < D; ++a) lam_out[a * cap + i] = make_float2(lam_x[a].hi, lam_x[a].lo);
  }
}

// The records of the step's survivors into their (cell, stage) segments.  The
// sums want them by (cell, stage, slot): with a segment per stage the rank that
// follows only compares slots, over a quarter of the cell's records (128 of
// them at 32 particles per cell: 160 us a step for 4.2 M records ranked by a
// 64-bit key per cell; this and the rank over 4 C segments take 55).
__global__ void __launch_bounds__(256) scatter_records_kernel(const __grid_constant__ TapeStep tp, int S, uint32_t C,
                                                              size_t cap, uint32_t* __restrict__ cursor,
                                                              uint32_t* __restrict__ src, DevCounters* __restrict__ ctr) {
  const uint32_t n = *tp.n_next;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t base = blockIdx.x * blockDim.x + threadIdx.x - lane; base < n; base += gridDim.x * blockDim.x) {
    const uint32_t j = base + lane;
    const uint32_t i = j < n ? tp.perm[j] : PIC_LOST;
    // all stages or none, as the lambda sweep counted them
    uint32_t K[kRecPerParticle];
    bool ok = i < cap;
#pragma unroll
    for (int s = 0; s < kRecPerParticle; ++s) {
      K[s] = ok && s < S ? tp.rcell[(size_t)s * cap + i] : 0u;
      ok = ok && K[s] < C;
    }
#pragma unroll
    for (int s = 0; s < kRecPerParticle; ++s) {
      if (s >= S) break;
      const uint32_t slot = aggregated_increment(cursor, K[s] * kRecPerParticle + s, ok);
      if (!ok) continue;
      if (slot < kRecPerParticle * cap)
        src[slot] = (uint32_t)(s * cap + i);
      else
        latch_status(ctr, PIC_STATUS_BOUNDS);
    }
  }
}

__global__ void __launch_bounds__(256) rank_records_kernel(const uint32_t* __restrict__ off, const uint32_t* __restrict__ src,
                                                           uint32_t* __restrict__ perm, uint32_t segments, size_t rcap,
                                                           DevCounters* __restrict__ ctr) {
  rank_phase(off, src, src, perm, (uint32_t*)nullptr, segments, rcap, &ctr->status,
             (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

// Checkpoint tapes: the step replayed from the store as it was at the start
// of the step, for every particle then alive, by the forward's own
// advect_particle_step (so the stage records are the forward's bit for bit); the
// new positions go to a sink.
template <int D, int RK>
__global__ void __launch_bounds__(128, PIC_ADVECT_MIN_BLOCKS) replay_step_kernel(const __grid_constant__ MeshView m, const __grid_constant__ StoreView s, const __grid_constant__ StoreView sink,
                                                                                const uint32_t* __restrict__ n_start,
                                                                                df dt, const __grid_constant__ StageRec rec) {
  const uint32_t n = *n_start;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int iters = 0;
    unsigned flags = 0;
    uint32_t full = 0;
    (void)advect_particle_step<D, RK, false, kSteady>(GlobalCells<D, false>{m}, m, s, i, sink, i, s.cell[i], dt, iters,
                                                    flags, full, RecordHook{rec, i});
  }
}

// Warp per cell: the records of the cell, in (cell, stage, slot) order, summed
// into the cell's 3^D x D block of nodal gradient entries, in double-float on
// the FP32 pipe; every cell is written (FP64), empty ones with zeros.  The entry
// (node (a, b, c), comp) of a record is (w_comp l_a(t0)) (l_b(t1) l_c(t2)):
// records are taken 32 at a time, lane i forms record i's D x 3 left factors and
// 3^(D-1) right factors once and leaves them in shared memory, then every lane
// adds its entries' products over those records in record order.  Lane (left
// factor, c) owns the entries of that left factor with the three right factors
// of c (2D: of one right factor): 27 lanes (18) and four loads a record, where
// entries dealt out evenly took six.
template <int D>
__global__ void __launch_bounds__(256) cell_partial_kernel(uint32_t C, const uint32_t* __restrict__ rec_off,
                                                           const uint32_t* __restrict__ rec_perm,
                                                           const float2* __restrict__ rec_t,
                                                           const float2* __restrict__ rec_w, size_t rcap,
                                                           double* __restrict__ partial) {
  constexpr int NN = (D == 3 ? 27 : 9);
  constexpr int NE = NN * D;
  constexpr int NA = 3 * D;             // w_comp l_a(t0), index comp * 3 + a
  constexpr int NB = (D == 3 ? 9 : 3);  // l_b(t1) l_c(t2), index c * 3 + b (2D: l_b(t1))
  constexpr int PER = D == 3 ? 3 : 1;   // right factors per lane
  __shared__ float2 fac[256 / 32][32][NA + NB];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const bool mine = lane < 3 * NA;
  const int left = lane % NA, group = mine ? lane / NA : 0;
  for (uint32_t K = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; K < C; K += warps) {
    df_acc acc[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) acc[q] = acc_zero();
    const uint32_t beg = rec_off[K * kRecPerParticle], end = rec_off[(K + 1) * kRecPerParticle];
    for (uint32_t e0 = beg; e0 < end; e0 += 32) {
      const uint32_t e = e0 + lane;
      if (e < end) {
        const uint32_t r = rec_perm[e];
        df l[D][3], w[D];
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const float2 tv = rec_t[a * rcap + r], wv = rec_w[a * rcap + r];
          lagrange2_df(df_make(tv.x, tv.y), l[a]);
          w[a] = df_make(wv.x, wv.y);
        }
#pragma unroll
        for (int comp = 0; comp < D; ++comp)
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const df v = df_mul(w[comp], l[0][a]);
            fac[wib][lane][comp * 3 + a] = make_float2(v.hi, v.lo);
          }
#pragma unroll
        for (int c = 0; c < (D == 3 ? 3 : 1); ++c)
#pragma unroll
          for (int b = 0; b < 3; ++b) {
            const df v = (D == 3) ? df_mul(l[1][b], l[2 % D][c]) : l[1][b];
            fac[wib][lane][NA + c * 3 + b] = make_float2(v.hi, v.lo);
          }
      }
      __syncwarp();
      const int cnt = (end - e0) < 32u ? (int)(end - e0) : 32;
      if (mine) {
#pragma unroll 2
        for (int j = 0; j < cnt; ++j) {
          const float2 A = fac[wib][j][left];
#pragma unroll
          for (int q = 0; q < PER; ++q) {
            const float2 B = fac[wib][j][NA + group * PER + q];
            acc_mad(acc[q], df_make(A.x, A.y), df_make(B.x, B.y));
          }
        }
      }
      __syncwarp();
    }
    if (mine) {
      const int comp = left / 3, a = left % 3;
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        const int node = a + 3 * (group * PER + q);
        partial[(size_t)K * NE + node * D + comp] = df_to_double(acc_result(acc[q]));
      }
    }
  }
}

// Thread per (node, component): add the blocks of the cells that share the
// node, in increasing cell order.
template <int D>
__global__ void node_reduce_kernel(const __grid_constant__ MeshView m, const double* __restrict__ partial, double* __restrict__ grad) {
  constexpr int NN = (D == 3 ? 27 : 9);
  const size_t total = (size_t)m.nnodes * D;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const size_t comp = q / m.nnodes, node = q % m.nnodes;
    int I[3] = {(int)(node % m.nq[0]), (int)((node / m.nq[0]) % m.nq[1]), (int)(node / ((size_t)m.nq[0] * m.nq[1]))};
    // cells touching the node along each axis: node index I = 2i + a, a in {0,1,2}
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (a >= D) continue;
      if (I[a] % 2 == 1) {
        lo[a] = hi[a] = I[a] / 2;
      } else {
        lo[a] = I[a] / 2 - 1;
        hi[a] = I[a] / 2;
        if (lo[a] < 0) lo[a] = 0;
        if (hi[a] > m.n[a] - 1) hi[a] = m.n[a] - 1;
      }
    }
    double s = 0.0;
    for (int ck = lo[2]; ck <= hi[2]; ++ck)
      for (int cj = lo[1]; cj <= hi[1]; ++cj)
        for (int ci = lo[0]; ci <= hi[0]; ++ci) {
          const uint32_t K = cell_index<D>(m, ci, cj, ck);
          const int a = I[0] - 2 * ci, b = I[1] - 2 * cj, c = (D == 3 ? I[2] - 2 * ck : 0);
          const int local = a + 3 * b + 9 * c;
          s += partial[((size_t)K * NN + local) * D + comp];
        }
    grad[comp * m.nnodes + node] += s;
  }
}

// lam[a*cap + j] = src[a*n + j] for j < n (dense caller layout -> strided,
// FP64 -> double-float).
__global__ void copy_in_kernel(const double* __restrict__ src, float2* __restrict__ dst, const uint32_t* n_dev, int dim,
                               size_t cap) {
  const uint32_t n = *n_dev;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < (size_t)n * dim; q += (size_t)gridDim.x * blockDim.x) {
    const df v = df_from_double(src[q]);
    dst[(q / n) * cap + q % n] = make_float2(v.hi, v.lo);
  }
}

__global__ void copy_out_kernel(const float2* __restrict__ src, double* __restrict__ dst, const uint32_t* n_dev, int dim,
                                size_t cap) {
  const uint32_t n = *n_dev;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < (size_t)n * dim; q += (size_t)gridDim.x * blockDim.x) {
    const float2 v = src[(q / n) * cap + q % n];
    dst[q] = df_to_double(df_make(v.x, v.y));
  }
}

static int grid_of(size_t n, int block) {
  size_t g = (n + block - 1) / block;
  const size_t cap = (size_t)num_sms() * 16;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

template <int D, int RK>
static void launch_reverse(pic_tape_s* tp, const MeshView& m, int step, const TapeStep& ts, const float2* lin,
                           float2* lout, cudaStream_t st) {
  const float hi = (float)tp->dt;
  const df dtd = {hi, (float)(tp->dt - (double)hi)};
  if (tp->kind == PIC_TAPE_CHECKPOINTS) {
    StoreView s{}, sink{};
    s.x = tp->x[step];
    s.xhat = tp->xhat[step];
    s.cell = tp->cell[step];
    s.cap = tp->cap;
    sink.x = tp->sink_x;
    sink.xhat = tp->sink_xhat;
    sink.cap = tp->cap;
    replay_step_kernel<D, RK><<<grid_of(tp->cap, 128), 128, 0, st>>>(m, s, sink, tp->n_dev + step, dtd,
                                                                     StageRec{tp->rcell[0], tp->rt[0], tp->cap});
    count_launches(1);
  }
  reverse_lambda_kernel<D, RK><<<grid_of(tp->cap, 128), 128, 0, st>>>(m, ts, tp->cap, dtd, lin, lout,
                                                                       tp->rec_counts, tp->rec_w, tp->parts->ctr);
}

}  // namespace pic

using namespace pic;

extern "C" pic_status pic_destroy_tape(pic_tape tp) {
  if (!tp) return PIC_OK;
  free(tp->rcell);
  free(tp->rt);
  free(tp->perm);
  free(tp->x);
  free(tp->xhat);
  free(tp->cell);
  cudaFree(tp->slab);
  free(tp);
  return PIC_OK;
}

extern "C" pic_status pic_advect_record_tape(pic_particles parts, pic_mesh mesh, double dt, pic_integrator integrator,
                                             int n_steps, pic_tape_kind kind, void* stream, pic_tape* out) {
  if (!out) return (set_error("pic_advect_record: out is NULL"), PIC_ERR_ARG);
  *out = nullptr;
  if (kind != PIC_TAPE_STAGES && kind != PIC_TAPE_CHECKPOINTS)
    return (set_error("pic_advect_record: unknown tape kind %d", (int)kind), PIC_ERR_ARG);
  if (!parts || !mesh || parts->mesh != mesh || parts->dim != mesh->dim)
    return (set_error("pic_advect_record: bad handles"), PIC_ERR_ARG);
  if (!std::isfinite(dt)) return (set_error("pic_advect_record: dt not finite"), PIC_ERR_ARG);
  if (n_steps < 1) return (set_error("pic_advect_record: n_steps must be >= 1"), PIC_ERR_ARG);
  if (integrator != PIC_EULER && integrator != PIC_RK2 && integrator != PIC_RK4)
    return (set_error("pic_advect_record: unknown integrator"), PIC_ERR_ARG);
  if (!mesh->has_velocity) return (set_error("pic_advect_record: velocity not set"), PIC_ERR_ARG);
  if (mesh->has_next)
    return (set_error("pic_advect_record: the adjoint supports a steady field only (no U_next)"), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  pic_tape_s* tp = (pic_tape_s*)calloc(1, sizeof(pic_tape_s));
  if (!tp) return (set_error("pic_advect_record: host allocation failed"), PIC_ERR_OOM);
  tp->parts = parts;
  tp->mesh = mesh;
  tp->dim = mesh->dim;
  tp->n_steps = n_steps;
  tp->integrator = (int)integrator;
  tp->dt = dt;
  tp->cap = parts->capacity;
  tp->C = mesh->C;
  tp->kind = (int)kind;
  const bool ckpt = kind == PIC_TAPE_CHECKPOINTS;
  tp->n_rec = ckpt ? 1 : n_steps;
  const size_t cap = tp->cap, d = (size_t)tp->dim, rcap = kRecPerParticle * cap;
  const int NE = (tp->dim == 3 ? 27 : 9) * tp->dim;
  tp->rcell = (uint32_t**)calloc(tp->n_rec, sizeof(uint32_t*));
  tp->rt = (float2**)calloc(tp->n_rec, sizeof(float2*));
  tp->perm = (uint32_t**)calloc(n_steps, sizeof(uint32_t*));
  bool ok = tp->rcell && tp->rt && tp->perm;
  if (ckpt) {
    tp->x = (double**)calloc(n_steps, sizeof(double*));
    tp->xhat = (float2**)calloc(n_steps, sizeof(float2*));
    tp->cell = (uint32_t**)calloc(n_steps, sizeof(uint32_t*));
    ok = ok && tp->x && tp->xhat && tp->cell;
  }
  // per-step arrays one after another, a stride of whole 256-byte lines apart
  const size_t cap64 = (cap + 63) / 64 * 64;
  uint32_t *rcell0 = nullptr, *perm0 = nullptr, *cell0 = nullptr;
  float2 *rt0 = nullptr, *xhat0 = nullptr;
  double* x0 = nullptr;
  if (ok) {
    const size_t steps = (size_t)n_steps, recs = (size_t)tp->n_rec;
    Slab slab;
    slab.add(&rcell0, recs * kRecPerParticle * cap64);
    slab.add(&rt0, recs * d * kRecPerParticle * cap64);
    slab.add(&perm0, steps * cap64);
    if (ckpt) {
      slab.add(&x0, steps * d * cap64);
      slab.add(&xhat0, steps * d * cap64);
      slab.add(&cell0, steps * cap64);
      slab.add(&tp->sink_x, d * cap);
      slab.add(&tp->sink_xhat, d * cap);
    }
    slab.add(&tp->n_dev, steps + 1);
    slab.add(&tp->lam[0], d * cap);
    slab.add(&tp->lam[1], d * cap);
    slab.add(&tp->rec_w, d * rcap);
    slab.add(&tp->rec_perm, rcap);
    const uint32_t segments = kRecPerParticle * tp->C;
    slab.add(&tp->rec_off, (size_t)segments + 1);
    slab.add(&tp->rec_counts, segments);
    slab.add(&tp->rec_cursor, segments);
    slab.add(&tp->rec_scan, scan_scratch_bytes(segments) / sizeof(uint32_t));
    slab.add(&tp->rec_src, rcap);
    slab.add(&tp->partial, (size_t)NE * tp->C);
    ok = slab.allocate(&tp->slab);
  }
  for (int s = 0; s < tp->n_rec && ok; ++s) {
    tp->rcell[s] = rcell0 + (size_t)s * kRecPerParticle * cap64;
    tp->rt[s] = rt0 + (size_t)s * d * kRecPerParticle * cap64;
  }
  for (int s = 0; s < n_steps && ok; ++s) {
    tp->perm[s] = perm0 + (size_t)s * cap64;
    if (ckpt) {
      tp->x[s] = x0 + (size_t)s * d * cap64;
      tp->xhat[s] = xhat0 + (size_t)s * d * cap64;
      tp->cell[s] = cell0 + (size_t)s * cap64;
    }
  }
  if (!ok) {
    cudaGetLastError();
    pic_destroy_tape(tp);
    return (set_error("pic_advect_record: device allocation failed"), PIC_ERR_OOM);
  }
  const MeshView m = mesh_view(mesh);
  for (int s = 0; s < n_steps; ++s) {
    cudaError_t e = cudaMemcpyAsync(tp->n_dev + s, &parts->ctr->n_alive, sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
    if (ckpt) {
      // the checkpoint is the sorted store
      const pic_status r0 = settle_order(parts, st);
      if (r0 != PIC_OK) {
        pic_destroy_tape(tp);
        return r0;
      }
      const int c = parts->cur;
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(tp->x[s], parts->x[c], sizeof(double) * d * cap, cudaMemcpyDeviceToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(tp->xhat[s], parts->xhat[c], sizeof(float2) * d * cap, cudaMemcpyDeviceToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(tp->cell[s], parts->cell[c], sizeof(uint32_t) * cap, cudaMemcpyDeviceToDevice, st);
    }
    if (e != cudaSuccess) {
      pic_destroy_tape(tp);
      return cuda_fail(e, "pic_advect_record: checkpoint");
    }
    // a checkpoint tape keeps one record set, which the sweep's replay rewrites
    pic_status r = launch_advect_record(parts, m, dt, (int)integrator,
                                        StageRec{tp->rcell[ckpt ? 0 : s], tp->rt[ckpt ? 0 : s], cap}, st);
    if (r == PIC_OK) r = rebin_order_from_counts(parts, st);
    if (r != PIC_OK) {
      pic_destroy_tape(tp);
      return r;
    }
    parts->pending_order = 1;  // applied by the next step, or by whoever needs the sorted arrays
    e = cudaMemcpyAsync(tp->perm[s], parts->perm, sizeof(uint32_t) * cap, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) {
      pic_destroy_tape(tp);
      return cuda_fail(e, "pic_advect_record: permutation");
    }
  }
  cudaError_t e = cudaMemcpyAsync(tp->n_dev + n_steps, &parts->ctr->n_alive, sizeof(uint32_t), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) {
    pic_destroy_tape(tp);
    return cuda_fail(e, "pic_advect_record: count");
  }
  *out = tp;
  return PIC_OK;
}

extern "C" pic_status pic_advect_record(pic_particles parts, pic_mesh mesh, double dt, pic_integrator integrator,
                                        int n_steps, void* stream, pic_tape* out) {
  return pic_advect_record_tape(parts, mesh, dt, integrator, n_steps, PIC_TAPE_STAGES, stream, out);
}

extern "C" pic_status pic_tape_adjoint(pic_tape tp, const double* dL_dxfinal, double* dL_dU, double* dL_dx0,
                                       void* stream) {
  if (!tp || !dL_dxfinal || !dL_dU) return (set_error("pic_tape_adjoint: null argument"), PIC_ERR_ARG);
  const pic_mesh_s* mesh = tp->mesh;
  cudaStream_t st = (cudaStream_t)stream;
  const MeshView m = mesh_view(mesh);
  const size_t cap = tp->cap, d = (size_t)tp->dim, rcap = kRecPerParticle * cap;
  PIC_CUDA(cudaMemsetAsync(dL_dU, 0, sizeof(double) * d * (size_t)mesh->nnodes, st));
  PIC_CUDA(cudaMemsetAsync(tp->lam[0], 0, sizeof(float2) * d * cap, st));
  copy_in_kernel<<<grid_of(d * cap, 256), 256, 0, st>>>(dL_dxfinal, tp->lam[0], tp->n_dev + tp->n_steps, tp->dim, cap);
  count_launches(1);
  int cur = 0;
  const uint32_t segments = kRecPerParticle * tp->C;
  for (int s = tp->n_steps - 1; s >= 0; --s) {
    TapeStep ts;
    ts.rcell = tp->rcell[tp->kind == PIC_TAPE_CHECKPOINTS ? 0 : s];
    ts.rt = tp->rt[tp->kind == PIC_TAPE_CHECKPOINTS ? 0 : s];
    ts.perm = tp->perm[s];
    ts.n_next = tp->n_dev + s + 1;
    PIC_CUDA(cudaMemsetAsync(tp->lam[1 - cur], 0, sizeof(float2) * d * cap, st));
    PIC_CUDA(cudaMemsetAsync(tp->rec_counts, 0, sizeof(uint32_t) * segments, st));
    const float2* lin = tp->lam[cur];
    float2* lout = tp->lam[1 - cur];
    if (tp->dim == 2) {
      if (tp->integrator == 1) launch_reverse<2, 1>(tp, m, s, ts, lin, lout, st);
      else if (tp->integrator == 2) launch_reverse<2, 2>(tp, m, s, ts, lin, lout, st);
      else launch_reverse<2, 4>(tp, m, s, ts, lin, lout, st);
    } else {
      if (tp->integrator == 1) launch_reverse<3, 1>(tp, m, s, ts, lin, lout, st);
      else if (tp->integrator == 2) launch_reverse<3, 2>(tp, m, s, ts, lin, lout, st);
      else launch_reverse<3, 4>(tp, m, s, ts, lin, lout, st);
    }
    count_launches(1);
    PIC_CUDA(cudaGetLastError());
    pic_status r = scan_u32(tp->rec_counts, tp->rec_off, segments, tp->rec_scan, nullptr, tp->rec_cursor, st,
                            &tp->parts->ctr->status);
    if (r != PIC_OK) return r;
    scatter_records_kernel<<<grid_of(cap, 256), 256, 0, st>>>(ts, tp->integrator, tp->C, cap, tp->rec_cursor, tp->rec_src,
                                                              tp->parts->ctr);
    rank_records_kernel<<<grid_of((size_t)segments * 32, 256), 256, 0, st>>>(tp->rec_off, tp->rec_src, tp->rec_perm,
                                                                             segments, rcap, tp->parts->ctr);
    count_launches(2);
    const int gp = grid_of((size_t)tp->C * 32, 256);
    const int gn = grid_of(d * (size_t)mesh->nnodes, 256);
    if (tp->dim == 2) {
      cell_partial_kernel<2><<<gp, 256, 0, st>>>(tp->C, tp->rec_off, tp->rec_perm, ts.rt, tp->rec_w, rcap, tp->partial);
      node_reduce_kernel<2><<<gn, 256, 0, st>>>(m, tp->partial, dL_dU);
    } else {
      cell_partial_kernel<3><<<gp, 256, 0, st>>>(tp->C, tp->rec_off, tp->rec_perm, ts.rt, tp->rec_w, rcap, tp->partial);
      node_reduce_kernel<3><<<gn, 256, 0, st>>>(m, tp->partial, dL_dU);
    }
    count_launches(2);
    PIC_CUDA(cudaGetLastError());
    cur = 1 - cur;
  }
  if (dL_dx0) {
    copy_out_kernel<<<grid_of(d * cap, 256), 256, 0, st>>>(tp->lam[cur], dL_dx0, tp->n_dev, tp->dim, cap);
    count_launches(1);
    PIC_CUDA(cudaGetLastError());
  }
  return PIC_OK;
}
