// particles.cu -- the particle store (Sec. 2.1): generation from local
// coordinates (Sec. 2.2), properties (Sec. 2.6), state queries and export.
#include <cstdlib>
#include <cstring>

#include "pic_internal.cuh"
#include "seed.cuh"

namespace pic {

// double-float reference coordinates -> FP64 (export)
__global__ void xhat_to_double_kernel(const float2* __restrict__ src, double* __restrict__ dst, size_t cap, size_t n,
                                      int dim) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n * dim; i += (size_t)gridDim.x * blockDim.x) {
    const size_t a = i / n, j = i % n;
    const float2 v = src[a * cap + j];
    dst[a * n + j] = (double)v.x + (double)v.y;
  }
}

// Every field of the packed particles in one pass.  With perm the order that
// pic_advect left pending is read through, not applied (cells are already in
// the new order, in the other buffer).  At 64^3 x 20 with three properties, in
// place of a gather, one copy per array and the x-hat conversion (150 + 120 +
// 105 us; the conversion alone is FP64-pipe bound, and hides behind the copies'
// memory time here): see pic_export.
template <int D>
__global__ void __launch_bounds__(256) pack_kernel(const __grid_constant__ StoreView s, const uint32_t* __restrict__ cell,
                                                   const uint32_t* __restrict__ perm, size_t first, size_t n,
                                                   uint32_t cell_base, const __grid_constant__ PackedOut o,
                                                   unsigned int* __restrict__ status) {
  for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < n; j += (size_t)gridDim.x * blockDim.x) {
    size_t i = first + j;
    if (perm) {
      i = perm[j];
      if (i >= s.cap) {
        atomicOr(status, PIC_STATUS_BOUNDS);
        continue;
      }
    }
    double x[D];
    float2 t[D];
    uint64_t id = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (o.x) x[a] = s.x[a * s.cap + i];
      if (o.xhat) t[a] = s.xhat[a * s.cap + i];
    }
    if (o.id) id = s.id[i];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (o.x) o.x[a * n + j] = x[a];
      if (o.xhat) o.xhat[a * n + j] = (double)t[a].x + (double)t[a].y;
    }
    if (o.id) o.id[j] = id;
    if (o.cell) o.cell[j] = cell[first + j] - cell_base;
    if (o.props)
      for (int q = 0; q < s.n_props; ++q) o.props[q * n + j] = s.props[q * s.cap + i];
  }
}

void launch_pack(pic_particles_s* p, int buf, const uint32_t* perm, size_t first, size_t n, uint32_t cell_base,
                 const PackedOut& o, cudaStream_t s) {
  if (n == 0) return;
  const StoreView v = store_view(p, buf);
  const uint32_t* cell = perm ? p->cell[1 - buf] : p->cell[buf];
  const size_t want = (n + 255) / 256, most = (size_t)num_sms() * 32;
  const int g = (int)(want < most ? want : most);
  if (p->dim == 2)
    pack_kernel<2><<<g, 256, 0, s>>>(v, cell, perm, first, n, cell_base, o, &p->ctr->status);
  else
    pack_kernel<3><<<g, 256, 0, s>>>(v, cell, perm, first, n, cell_base, o, &p->ctr->status);
  count_launches(1);
}

// Device memory of the current device that a kernel may write as elements of
// `align` bytes (a copy takes any address).
bool on_device(const void* ptr, size_t align) {
  if ((uintptr_t)ptr % align) return false;
  cudaPointerAttributes at;
  int here = 0;
  const bool dev = cudaGetDevice(&here) == cudaSuccess && cudaPointerGetAttributes(&at, ptr) == cudaSuccess &&
                   at.type == cudaMemoryTypeDevice && at.device == here;
  cudaGetLastError();
  return dev;
}

__global__ void set_prop_kernel(double* __restrict__ dst, const double* __restrict__ src, const DevCounters* ctr) {
  const uint32_t n = ctr->n_alive;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

}  // namespace pic

using namespace pic;

extern "C" pic_status pic_destroy_particles(pic_particles p) {
  if (!p) return PIC_OK;
  cudaFree(p->cell_off);
  cudaFree(p->slab);
  cudaFree(p->xfer);
  cudaFree(p->stage_rec);
  for (int k = 0; k < 3 * p->ev_cap; ++k) cudaEventDestroy(p->ev[k]);
  free(p->ev);
  free(p);
  return PIC_OK;
}

namespace pic {

// A store of `capacity` particles over C cells (both rebin buffers and the
// rebin scratch).  Takes ownership of cell_off.  NULL (error message set,
// cell_off freed) if an allocation fails.
pic_particles_s* store_alloc(int dim, int n_props, uint32_t C, size_t capacity, uint32_t* cell_off) {
  pic_particles_s* p = (pic_particles_s*)calloc(1, sizeof(pic_particles_s));
  if (!p) {
    cudaFree(cell_off);
    set_error("store_alloc: host allocation failed");
    return nullptr;
  }
  p->dim = dim;
  p->n_props = n_props;
  p->C = C;
  p->capacity = capacity > 0 ? capacity : 1;
  p->cell_off = cell_off;
  const size_t cap = p->capacity, d = (size_t)dim;
  Slab slab;
  for (int b = 0; b < 2; ++b) {
    slab.add(&p->x[b], d * cap);
    slab.add(&p->xhat[b], d * cap);
    slab.add(&p->id[b], cap);
    slab.add(&p->cell[b], cap);
    slab.add(&p->props[b], (size_t)(n_props > 0 ? n_props : 1) * cap);
  }
  slab.add(&p->cell_new, cap);
  slab.add(&p->cursor, C);
  slab.add(&p->counts, C);
  slab.add(&p->block_sums, scan_scratch_bytes(C) / sizeof(uint32_t));
  slab.add(&p->tile_next, 1);
  slab.add(&p->key_id, cap);
  slab.add(&p->key_src, cap);
  slab.add(&p->perm, cap);
  slab.add(&p->ctr, 1);
  if (!slab.allocate(&p->slab)) {
    pic_destroy_particles(p);
    set_error("store_alloc: device allocation failed (capacity %zu)", cap);
    return nullptr;
  }
  return p;
}

cudaError_t store_init(pic_particles_s* p, uint32_t n, cudaStream_t s) {
  DevCounters h{};
  h.n_alive = n;
  h.n_next = n;
  const cudaError_t e = cudaMemcpyAsync(p->ctr, &h, sizeof(h), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  p->scratch_clear = 0;
  if (clear_step_scratch(p, s) != PIC_OK) return cudaErrorUnknown;
  p->scratch_clear = 1;
  return cudaSuccess;
}

}  // namespace pic

namespace pic {

// The part of seeding shared by every generator: per-cell numbers (device
// array, or `uniform_count` everywhere) -> cell offsets -> an allocated store
// of `capacity` (0 = exactly the number created) whose counters say N
// particles.  The generator's kernel then fills slots cell_off[K] ..
// cell_off[K+1]-1 of buffer 0.
pic_status seed_prepare(pic_mesh mesh, const uint32_t* per_cell, uint32_t uniform_count, int n_props, size_t capacity,
                        cudaStream_t st, const char* who, pic_particles_s** out, size_t* n_out) {
  *out = nullptr;
  if (n_props < 0 || n_props > kMaxProps) return (set_error("%s: n_props must be in [0, %d]", who, kMaxProps), PIC_ERR_ARG);
  const uint32_t C = mesh->C;
  uint32_t *counts = nullptr, *off = nullptr, *sums = nullptr, *total = nullptr;
  void* tmp = nullptr;
  Slab slab;
  slab.add(&counts, C);
  slab.add(&sums, scan_scratch_bytes(C) / sizeof(uint32_t));
  slab.add(&total, 2);
  if (!slab.allocate(&tmp) || cudaMalloc(&off, sizeof(uint32_t) * (C + 1)) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(tmp);
    return (set_error("%s: device allocation failed", who), PIC_ERR_OOM);
  }
  auto cleanup_tmp = [&]() { cudaFree(tmp); };
  fill_counts_kernel<<<(C + 255) / 256 < 4096 ? (C + 255) / 256 : 4096, 256, 0, st>>>(per_cell, uniform_count, counts, C);
  // 64-bit total check: the scan is 32-bit, so guard against overflow first
  uint64_t total64 = 0;
  if (per_cell) {
    uint32_t* h = (uint32_t*)malloc(sizeof(uint32_t) * C);
    cudaError_t e = h ? cudaMemcpyAsync(h, per_cell, sizeof(uint32_t) * C, cudaMemcpyDefault, st) : cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
      free(h);
      cleanup_tmp();
      cudaFree(off);
      return cuda_fail(e, who);
    }
    for (uint32_t K = 0; K < C; ++K) total64 += h[K];
    free(h);
  } else {
    total64 = (uint64_t)uniform_count * C;
  }
  if (total64 >= 0xFFFFFFF0ull) {
    cleanup_tmp();
    cudaFree(off);
    return (set_error("%s: %llu particles exceed the 32-bit store", who, (unsigned long long)total64), PIC_ERR_CAPACITY);
  }
  const size_t N = (size_t)total64;
  if (capacity == 0) capacity = N;
  if (capacity < N) {
    cleanup_tmp();
    cudaFree(off);
    return (set_error("%s: capacity %zu < %zu particles", who, capacity, N), PIC_ERR_CAPACITY);
  }
  if (capacity >= 0xFFFFFFF0ull) {
    cleanup_tmp();
    cudaFree(off);
    return (set_error("%s: capacity exceeds the 32-bit store", who), PIC_ERR_CAPACITY);
  }
  pic_status r = scan_u32(counts, off, C, sums, total, nullptr, st);
  cleanup_tmp();
  if (r != PIC_OK) {
    cudaFree(off);
    return r;
  }
  pic_particles_s* p = store_alloc(mesh->dim, n_props, C, capacity, off);
  if (!p) return PIC_ERR_OOM;
  p->mesh = mesh;
  p->stream = st;
  const cudaError_t e = store_init(p, (uint32_t)N, st);
  if (e != cudaSuccess) {
    pic_destroy_particles(p);
    return cuda_fail(e, who);
  }
  p->cur = 0;
  *out = p;
  *n_out = N;
  return PIC_OK;
}

}  // namespace pic

extern "C" pic_status pic_seed_particles(pic_mesh mesh, const uint32_t* per_cell, uint32_t uniform_count, uint64_t seed,
                                         uint64_t first_id, int n_props, size_t capacity, void* stream,
                                         pic_particles* out) {
  if (!out) return (set_error("pic_seed_particles: out is NULL"), PIC_ERR_ARG);
  *out = nullptr;
  if (!mesh) return (set_error("pic_seed_particles: null mesh"), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  pic_particles_s* p = nullptr;
  size_t N = 0;
  pic_status r = seed_prepare(mesh, per_cell, uniform_count, n_props, capacity, st, "pic_seed_particles", &p, &N);
  if (r != PIC_OK) return r;
  const uint32_t C = mesh->C;
  const MeshView m = mesh_view(mesh);
  const int grid = (int)((C + 127) / 128 < 8192 ? (C + 127) / 128 : 8192);
  if (mesh->dim == 2)
    seed_kernel<2><<<grid, 128, 0, st>>>(m, store_view(p, 0), p->cell_off, seed, first_id, 0u);
  else
    seed_kernel<3><<<grid, 128, 0, st>>>(m, store_view(p, 0), p->cell_off, seed, first_id, 0u);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    pic_destroy_particles(p);
    return cuda_fail(e, "pic_seed_particles: seed kernel");
  }
  *out = p;
  return PIC_OK;
}

extern "C" pic_status pic_set_properties(pic_particles p, int prop, const double* values, void* stream) {
  if (!p || !values) return (set_error("pic_set_properties: null argument"), PIC_ERR_ARG);
  if (prop < 0 || prop >= p->n_props) return (set_error("pic_set_properties: property %d out of range", prop), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  {
    const pic_status r0 = settle_order(p, st);
    if (r0 != PIC_OK) return r0;
  }
  set_prop_kernel<<<1024, 256, 0, st>>>(p->props[p->cur] + (size_t)prop * p->capacity, values, p->ctr);
  count_launches(1);
  PIC_CUDA(cudaGetLastError());
  return PIC_OK;
}

static pic_status read_counters(pic_particles p, DevCounters* h) {
  PIC_CUDA(cudaDeviceSynchronize());
  PIC_CUDA(cudaMemcpy(h, p->ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost));
  return PIC_OK;
}

extern "C" pic_status pic_get_state(pic_particles p, size_t* n_alive, size_t* n_lost, uint32_t* status_word) {
  if (!p) return (set_error("pic_get_state: null handle"), PIC_ERR_ARG);
  DevCounters h;
  pic_status r = read_counters(p, &h);
  if (r != PIC_OK) return r;
  if (n_alive) *n_alive = h.n_alive;
  if (n_lost) *n_lost = (size_t)h.lost_total;
  if (status_word) *status_word = h.status;
  return PIC_OK;
}

extern "C" pic_status pic_get_stats(pic_particles p, uint64_t* particle_steps, uint64_t* walks, uint64_t* global_searches,
                                    uint64_t* newton_iterations) {
  if (!p) return (set_error("pic_get_stats: null handle"), PIC_ERR_ARG);
  DevCounters h;
  pic_status r = read_counters(p, &h);
  if (r != PIC_OK) return r;
  if (particle_steps) *particle_steps = h.particle_steps;
  if (walks) *walks = h.walks;
  if (global_searches) *global_searches = h.global_searches;
  if (newton_iterations) *newton_iterations = h.newton_iterations;
  return PIC_OK;
}

extern "C" pic_status pic_get_counters(pic_particles p, uint64_t* values, int n_values) {
  if (!p || (!values && n_values > 0) || n_values < 0) return (set_error("pic_get_counters: bad argument"), PIC_ERR_ARG);
  DevCounters h;
  pic_status r = read_counters(p, &h);
  if (r != PIC_OK) return r;
  const uint64_t v[PIC_N_COUNTERS] = {h.particle_steps, h.walks, h.global_searches, h.newton_iterations,
                                      h.lost_total, h.fallback64, h.walk64, h.deferred};
  for (int k = 0; k < n_values && k < PIC_N_COUNTERS; ++k) values[k] = v[k];
  return PIC_OK;
}

extern "C" pic_status pic_export(pic_particles p, double* x, double* xhat, uint64_t* id, uint32_t* cell, double* props,
                                 void* stream) {
  if (!p) return (set_error("pic_export: null handle"), PIC_ERR_ARG);
  cudaStream_t st = (cudaStream_t)stream;
  // into device arrays: one kernel, through a pending order; with any host
  // array: the order applied, then a copy per array
  const bool packed = (!x || on_device(x, sizeof(double))) && (!xhat || on_device(xhat, sizeof(double))) &&
                      (!id || on_device(id, sizeof(uint64_t))) && (!cell || on_device(cell, sizeof(uint32_t))) &&
                      (!props || on_device(props, sizeof(double)));
  if (!packed) {
    const pic_status r0 = settle_order(p, st);
    if (r0 != PIC_OK) return r0;
  }
  DevCounters h;
  pic_status r = read_counters(p, &h);
  if (r != PIC_OK) return r;
  const size_t N = h.n_alive, cap = p->capacity;
  const int c = p->cur;
  if (N == 0) return PIC_OK;
  if (packed) {
    launch_pack(p, c, p->pending_order ? p->perm : nullptr, 0, N, 0, PackedOut{x, xhat, id, cell, props}, st);
    PIC_CUDA(cudaGetLastError());
    return PIC_OK;
  }
  for (int a = 0; a < p->dim; ++a) {
    if (x) PIC_CUDA(cudaMemcpyAsync(x + a * N, p->x[c] + a * cap, sizeof(double) * N, cudaMemcpyDefault, st));
  }
  if (xhat) {
    const bool dev = on_device(xhat, sizeof(double));
    double* tmp = xhat;
    if (!dev) PIC_CUDA(cudaMallocAsync((void**)&tmp, sizeof(double) * p->dim * N, st));
    xhat_to_double_kernel<<<1024, 256, 0, st>>>(p->xhat[c], tmp, cap, N, p->dim);
    PIC_CUDA(cudaGetLastError());
    if (!dev) {
      PIC_CUDA(cudaMemcpyAsync(xhat, tmp, sizeof(double) * p->dim * N, cudaMemcpyDefault, st));
      PIC_CUDA(cudaFreeAsync(tmp, st));
    }
  }
  if (id) PIC_CUDA(cudaMemcpyAsync(id, p->id[c], sizeof(uint64_t) * N, cudaMemcpyDefault, st));
  if (cell) PIC_CUDA(cudaMemcpyAsync(cell, p->cell[c], sizeof(uint32_t) * N, cudaMemcpyDefault, st));
  for (int q = 0; q < p->n_props && props; ++q)
    PIC_CUDA(cudaMemcpyAsync(props + q * N, p->props[c] + q * cap, sizeof(double) * N, cudaMemcpyDefault, st));
  return PIC_OK;
}

extern "C" pic_status pic_cell_offsets(pic_particles p, uint32_t* off, void* stream) {
  if (!p || !off) return (set_error("pic_cell_offsets: null argument"), PIC_ERR_ARG);
  PIC_CUDA(cudaMemcpyAsync(off, p->cell_off, sizeof(uint32_t) * ((size_t)p->C + 1), cudaMemcpyDefault,
                           (cudaStream_t)stream));
  return PIC_OK;
}
