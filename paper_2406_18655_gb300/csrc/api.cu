// Host side of the C ABI declared in include/lsd.h: decoder construction, device
// memory, launches.  No decoding arithmetic runs on the host.
#include <algorithm>
#include <climits>
#include <cstdlib>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "lsd_internal.cuh"

using namespace lsdgb;

namespace lsdgb {
// Chunks of the copy / decode pipeline of the host-buffer entry points (measured on GB300
// with 10^6 BB144 shots: 4 chunks 152 M shots/s end to end, 6 chunks 151 M, 8 chunks 149 M).
constexpr int kHostChunks = 4;
}  // namespace lsdgb

struct lsd_decoder {
  int m = 0, n = 0, E = 0;
  int bp_iters = 0, order = 0, osd_cs = -1;
  int io_packed = 0;  // set for the duration of a bit-packed decode call
  lsd_options opt{};
  float alpha = 0.625f;
  cudaStream_t st = nullptr;
  DevGraph g{};
  // owned device memory
  std::vector<void*> allocs;
  size_t bytes = 0;
  DevCounters* d_ctr = nullptr;
  DevCounters* h_ctr = nullptr;  // pinned
  int32_t* d_queue = nullptr;
  float* d_queue_llr = nullptr;
  size_t cap_shots = 0;
  uint8_t* d_stage = nullptr;  // host-buffer entry point: syndromes | corrections | status
  size_t stage_cap = 0;
  // host-buffer entry point: copy streams and per-chunk events of the pipelined path
  cudaStream_t cp_in = nullptr, cp_out = nullptr;
  cudaEvent_t cev[2 * lsdgb::kHostChunks] = {};
  // second compute stream and per-chunk counters: consecutive chunks decode on alternate
  // streams, so that one chunk's BP fills the SMs that the previous chunk's LSD tail leaves
  cudaStream_t st2 = nullptr;
  cudaEvent_t join = nullptr;
  DevCounters* d_ctr_chunks = nullptr;  // [kHostChunks]
  // launch shapes
  int bp_variant = -1, bp_grid = 0, bp_block = 0;
  size_t bp_smem = 0;
  bool lsd_ok = false;
  bool dense = false;        // the dense LSD kernel takes this matrix
  int lsd_warps = 0, lsd_grid = 0, lsd_W = 0;
  size_t lsd_smem = 0;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  long long launches = 0;
  int64_t last_shots = 0;
  int last_kind = 0;  // 0 none, 1 decode, 2 bp only, 3 lsd only
  float* d_probs = nullptr;  // channel probabilities (sampler)
  // sparse LSD (large matrices)
  bool sparse = false;
  int sparse_rc = 0;         // its tables found no room: every LSD call returns this
  int sp_grid_small = 0, sp_grid_big = 0;  // (large: 0 when no shot can outgrow the small one)
  unsigned char* d_sp_small = nullptr;
  unsigned char* d_sp_big = nullptr;
  int* d_spill = nullptr;
  size_t sp_tables = 0;      // bytes of g.chk_pad and g.var_pad together
  size_t sp_stride_small = 0, sp_stride_big = 0, spill_cap = 0;
};

struct lsd_prior {
  lsd_decoder* dec = nullptr;
  int rounds = 4;
  int np = 0;
  float *d_params = nullptr, *d_grads = nullptr, *d_m = nullptr, *d_v = nullptr;
  double* d_loss = nullptr;
  double* h_loss = nullptr;  // pinned
  float* d_scratch = nullptr;
  int* d_flag = nullptr;     // set by the tensor-memory kernel when a wait runs out
  int grid_train = 0, grid_fwd = 0;
  int grid_tc = 0;           // > 0: inference may run on the tensor-memory kernel
  int kernel = 0;            // 0 auto, 1 per-node mma.sync kernel, 2 tensor-memory kernel
  int step = 0;
};

namespace {

thread_local char g_last_error[160] = "";

int cuda_fail(cudaError_t e) {
  lsdgb::record_cuda_error(e);
  if (e == cudaErrorMemoryAllocation) return LSD_ERR_OOM;
  return LSD_ERR_CUDA;
}

// Inference of the prior on the tensor-memory kernel: chosen automatically when the graph
// fits it, or on request.
bool prior_uses_tc(const lsd_prior* p) {
  return p->grid_tc > 0 && p->kernel != 1;
}

// Device allocation charged to the decoder (and to its memory budget).
constexpr size_t alloc_size(size_t bytes) { return bytes ? bytes : 16; }
int try_alloc(lsd_decoder* d, void** p, size_t bytes) {
  bytes = alloc_size(bytes);
  if (d->opt.mem_budget && d->bytes + bytes > d->opt.mem_budget) return LSD_ERR_ADMISSION;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_fail(e);
  }
  d->allocs.push_back(*p);
  d->bytes += bytes;
  return LSD_OK;
}

void dev_free(lsd_decoder* d, void* p, size_t bytes) {
  if (!p) return;
  auto it = std::find(d->allocs.begin(), d->allocs.end(), p);
  if (it != d->allocs.end()) d->allocs.erase(it);
  cudaFree(p);
  d->bytes -= bytes;
}

bool no_room(int rc) { return rc == LSD_ERR_ADMISSION || rc == LSD_ERR_OOM; }

// A matrix that both LSD kernels take goes over to the dense one, which holds no scratch (the
// same results): whatever a budget has room for with that kernel, it has room for.  False when
// the sparse kernel is not in use or is the only one.
bool drop_sparse(lsd_decoder* d) {
  if (!d->sparse || !d->dense) return false;
  cudaStreamSynchronize(d->st);  // (an error of earlier work is reported by the next call)
  dev_free(d, d->d_sp_small, alloc_size((size_t)d->sp_grid_small * d->sp_stride_small));
  dev_free(d, d->d_sp_big, alloc_size((size_t)d->sp_grid_big * d->sp_stride_big));
  dev_free(d, d->d_spill, d->spill_cap * sizeof(int));
  dev_free(d, const_cast<uint16_t*>(d->g.chk_pad), d->sp_tables);
  d->g.chk_pad = d->g.var_pad = nullptr;
  d->d_sp_small = d->d_sp_big = nullptr;
  d->d_spill = nullptr;
  d->spill_cap = 0;
  d->sparse = false;
  return true;
}

int dev_alloc(lsd_decoder* d, void** p, size_t bytes) {
  const int rc = try_alloc(d, p, bytes);
  return no_room(rc) && drop_sparse(d) ? try_alloc(d, p, bytes) : rc;
}

template <typename T>
int upload(lsd_decoder* d, T** dst, const std::vector<T>& src) {
  int rc = dev_alloc(d, reinterpret_cast<void**>(dst), src.size() * sizeof(T));
  if (rc) return rc;
  cudaError_t e = cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T),
                                  cudaMemcpyHostToDevice, d->st);
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

// Queue and LLR buffer for `shots` unconverged shots.
int ensure_workspace(lsd_decoder* d, int64_t shots) {
  if ((size_t)shots <= d->cap_shots) return LSD_OK;
  cudaError_t e = cudaStreamSynchronize(d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  dev_free(d, d->d_queue, d->cap_shots * sizeof(int32_t));
  dev_free(d, d->d_queue_llr, d->cap_shots * (size_t)d->n * sizeof(float));
  d->d_queue = nullptr;
  d->d_queue_llr = nullptr;
  d->cap_shots = 0;
  int rc = dev_alloc(d, reinterpret_cast<void**>(&d->d_queue), (size_t)shots * sizeof(int32_t));
  if (rc) return rc;
  rc = dev_alloc(d, reinterpret_cast<void**>(&d->d_queue_llr),
                 (size_t)shots * (size_t)d->n * sizeof(float));
  if (rc) {
    dev_free(d, d->d_queue, (size_t)shots * sizeof(int32_t));
    d->d_queue = nullptr;
    return rc;
  }
  d->cap_shots = (size_t)shots;
  return LSD_OK;
}

int reset_counters(lsd_decoder* d) {
  cudaError_t e = cudaMemsetAsync(d->d_ctr, 0, sizeof(DevCounters), d->st);
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

BPArgs bp_args(lsd_decoder* d, int64_t shots, const uint8_t* syn) {
  BPArgs a{};
  a.g = d->g;
  a.shots = shots;
  a.syndromes = syn;
  a.iters = d->bp_iters;
  a.alpha = d->alpha;
  a.method = d->opt.bp_method;
  a.early_exit = d->opt.no_early_exit ? 0 : 1;
  a.ctr = d->d_ctr;
  a.packed = d->io_packed;
  return a;
}

int fill_stats(lsd_decoder* d, int64_t shots, lsd_stats* stats, bool timed_lsd) {
  cudaError_t e = cudaMemcpyAsync(d->h_ctr, d->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost,
                                  d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  e = cudaStreamSynchronize(d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  std::memset(stats, 0, sizeof(*stats));
  stats->shots = shots;
  stats->bp_converged = (int64_t)d->h_ctr->bp_converged;
  stats->lsd_shots = (int64_t)d->h_ctr->lsd_count;
  stats->unsolvable = (int64_t)d->h_ctr->unsolvable;
  stats->bp_iterations = (int64_t)d->h_ctr->bp_iterations;
  stats->lsd_steps = (int64_t)d->h_ctr->lsd_steps;
  stats->kappa_max = d->h_ctr->kappa_max;
  stats->nu_max = d->h_ctr->nu_max;
  stats->lsd_spilled = (int64_t)d->h_ctr->spill_count;
  float ms = 0.f;
  if (d->last_kind != 3 && cudaEventElapsedTime(&ms, d->ev[0], d->ev[1]) == cudaSuccess)
    stats->ms_bp = ms;
  if (timed_lsd && d->last_kind != 2 && cudaEventElapsedTime(&ms, d->ev[1], d->ev[2]) == cudaSuccess)
    stats->ms_lsd = ms;
  cudaGetLastError();
  return LSD_OK;
}

bool valid_lanes(int l) { return l == 0 || l == 8 || l == 16 || l == 32; }

// BP + dense LSD of one chunk of a pipelined batch, on stream st with its own counters and
// its own part of the queue (the rows of its shots).
int decode_chunk(lsd_decoder* d, int64_t shots, const uint8_t* syn, uint8_t* corr,
                 uint8_t* status, DevCounters* ctr, int32_t* queue, float* queue_llr,
                 cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(ctr, 0, sizeof(DevCounters), st);
  if (e != cudaSuccess) return cuda_fail(e);
  BPArgs a = bp_args(d, shots, syn);
  a.ctr = ctr;
  a.corrections = corr;
  a.status = status;
  a.queue = queue;
  a.queue_llr = queue_llr;
  e = launch_bp(a, d->bp_variant, d->bp_grid, d->bp_block, d->bp_smem, st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  LSDArgs l{};
  l.packed = d->io_packed;
  l.g = d->g;
  l.count_from_ctr = 1;
  l.queue = queue;
  l.llr = queue_llr;
  l.llr_by_item = 1;
  l.syndromes = syn;
  l.corrections = corr;
  l.status = status;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = ctr;
  e = launch_lsd(l, d->lsd_warps, d->lsd_grid, d->lsd_smem, st);
  d->launches++;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

// Scratch of the sparse LSD for a launch of up to max_items shots.
int ensure_sparse(lsd_decoder* d, int64_t max_items) {
  if (d->sparse_rc) return d->sparse_rc;
  int rc;
  // (each by its own pointer: a call after one that found no room for the second keeps the first)
  if (!d->d_sp_small && (rc = try_alloc(d, reinterpret_cast<void**>(&d->d_sp_small),
                                        (size_t)d->sp_grid_small * d->sp_stride_small)))
    return rc;
  if (!d->d_sp_big && (rc = try_alloc(d, reinterpret_cast<void**>(&d->d_sp_big),
                                      (size_t)d->sp_grid_big * d->sp_stride_big)))
    return rc;
  if (d->sp_grid_big > 0 && (size_t)max_items > d->spill_cap) {
    cudaError_t e = cudaStreamSynchronize(d->st);
    if (e != cudaSuccess) return cuda_fail(e);
    dev_free(d, d->d_spill, d->spill_cap * sizeof(int));
    d->d_spill = nullptr;
    d->spill_cap = 0;
    if ((rc = try_alloc(d, reinterpret_cast<void**>(&d->d_spill), (size_t)max_items * sizeof(int))))
      return rc;
    d->spill_cap = (size_t)max_items;
  }
  return LSD_OK;
}

// LSD launch on the decoder's queue or batch: the dense kernel, or the sparse kernel followed by
// its large instance for the shots that outgrew the small one.
int run_lsd(lsd_decoder* d, const LSDArgs& l, int64_t max_items) {
  if (d->sparse) {
    const int rc = ensure_sparse(d, max_items);
    if (rc && !(no_room(rc) && drop_sparse(d))) return rc;
  }
  cudaError_t e;
  if (!d->sparse) {
    e = launch_lsd(l, d->lsd_warps, d->lsd_grid, d->lsd_smem, d->st);
    d->launches++;
    return e == cudaSuccess ? LSD_OK : cuda_fail(e);
  }
  e = launch_sparse(l, false, d->sp_grid_small, d->d_sp_small, d->sp_stride_small, d->d_spill,
                    nullptr, d->st);
  d->launches++;
  if (d->sp_grid_big == 0) return e == cudaSuccess ? LSD_OK : cuda_fail(e);
  if (e == cudaSuccess)
    e = launch_sparse(l, true, d->sp_grid_big, d->d_sp_big, d->sp_stride_big, nullptr, d->d_spill,
                      d->st);
  d->launches++;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

}  // namespace

void lsdgb::record_cuda_error(cudaError_t e) {
  std::snprintf(g_last_error, sizeof(g_last_error), "%s: %s", cudaGetErrorName(e),
                cudaGetErrorString(e));
}

extern "C" {

const char* lsd_last_error(void) { return g_last_error; }

const char* lsd_status_string(int code) {
  switch (code) {
    case LSD_OK: return "ok";
    case LSD_ERR_INVALID_ARG: return "invalid argument";
    case LSD_ERR_CUDA: return "CUDA error";
    case LSD_ERR_OOM: return "out of device memory";
    case LSD_ERR_ADMISSION: return "work does not fit in the memory budget";
    case LSD_ERR_TIMEOUT: return "device wait timed out";
    case LSD_ERR_UNSUPPORTED: return "matrix shape beyond the kernel limits";
    case LSD_SHOT_OK_BP: return "shot decoded by BP";
    case LSD_SHOT_OK_LSD: return "shot decoded by LSD";
    case LSD_SHOT_UNSOLVABLE: return "syndrome not in the image of H";
    default: return "unknown code";
  }
}

int lsd_destroy(lsd_decoder* d) {
  if (!d) return LSD_OK;
  if (d->st || d->allocs.size()) cudaStreamSynchronize(d->st);
  for (void* p : d->allocs) cudaFree(p);
  if (d->h_ctr) cudaFreeHost(d->h_ctr);
  for (auto& e : d->ev)
    if (e) cudaEventDestroy(e);
  if (d->join) cudaEventDestroy(d->join);
  for (cudaStream_t c : {d->cp_in, d->cp_out, d->st2})
    if (c) {
      cudaStreamSynchronize(c);
      cudaStreamDestroy(c);
    }
  for (auto& e : d->cev)
    if (e) cudaEventDestroy(e);
  cudaGetLastError();
  delete d;
  return LSD_OK;
}

int lsd_create(lsd_decoder** out, int32_t m, int32_t n, int64_t nnz, const int32_t* rows,
               const int32_t* cols, const float* channel_probs, int32_t bp_iters,
               int32_t lsd_order, const lsd_options* opt) {
  if (!out) return LSD_ERR_INVALID_ARG;
  *out = nullptr;
  if (m < 1 || n < 1 || nnz < 0 || (nnz > 0 && (!rows || !cols)) || !channel_probs ||
      bp_iters < 0 || lsd_order < 0)
    return LSD_ERR_INVALID_ARG;
  lsd_options o{};
  if (opt) o = *opt;
  if (o.bp_method < 0 || o.bp_method > 1 || !valid_lanes(o.bp_lanes) || o.lsd_warps < 0 ||
      o.lsd_warps > 16 || o.bp_kernel < 0 || o.bp_kernel > 3 || o.lsd_kernel < 0 ||
      o.lsd_kernel > 2 || o.reserved || o.ms_scaling < 0.f || o.osd_method < 0 ||
      o.osd_method > 1 || o.osd_cs_order < 0 || o.osd_cs_order > kMaxCsOrder ||
      (o.osd_method == 0 && o.osd_cs_order != 0) ||
      lsd_order > (o.osd_method == 1 ? kMaxCsGrowth : kMaxOrder))
    return LSD_ERR_INVALID_ARG;
  for (int j = 0; j < n; ++j)
    if (!(channel_probs[j] > 0.f && channel_probs[j] < 1.f)) return LSD_ERR_INVALID_ARG;
  // Tanner graph: edges sorted by (row, column); duplicates are an error
  std::vector<std::pair<int, int>> e((size_t)nnz);
  for (int64_t k = 0; k < nnz; ++k) {
    if (rows[k] < 0 || rows[k] >= m || cols[k] < 0 || cols[k] >= n) return LSD_ERR_INVALID_ARG;
    e[(size_t)k] = {rows[k], cols[k]};
  }
  std::sort(e.begin(), e.end());
  for (size_t k = 1; k < e.size(); ++k)
    if (e[k] == e[k - 1]) return LSD_ERR_INVALID_ARG;
  const int E = (int)e.size();
  if (E >= 65536 || n >= 65536 || m >= 65536) return LSD_ERR_UNSUPPORTED;
  std::vector<int32_t> chk_ptr(m + 1, 0), var_ptr(n + 1, 0);
  std::vector<uint16_t> chk_var(E), var_edge(E), var_chk(E);
  for (auto& p : e) {
    chk_ptr[p.first + 1]++;
    var_ptr[p.second + 1]++;
  }
  int max_row = 0, max_col = 0, min_row = INT_MAX, min_col = INT_MAX;
  for (int i = 0; i < m; ++i) {
    max_row = std::max(max_row, chk_ptr[i + 1]);
    min_row = std::min(min_row, chk_ptr[i + 1]);
  }
  for (int j = 0; j < n; ++j) {
    max_col = std::max(max_col, var_ptr[j + 1]);
    min_col = std::min(min_col, var_ptr[j + 1]);
  }
  if (max_row > kMaxRowDeg) return LSD_ERR_UNSUPPORTED;
  for (int i = 0; i < m; ++i) chk_ptr[i + 1] += chk_ptr[i];
  for (int j = 0; j < n; ++j) var_ptr[j + 1] += var_ptr[j];
  std::vector<int32_t> vfill(var_ptr.begin(), var_ptr.end() - 1);
  for (int k = 0; k < E; ++k) {  // edge k is (row e[k].first, column e[k].second)
    chk_var[k] = (uint16_t)e[k].second;
    const int slot = vfill[e[k].second]++;  // rows arrive in ascending order per column
    var_edge[slot] = (uint16_t)k;
    var_chk[slot] = (uint16_t)e[k].first;
  }

  lsd_decoder* d = new (std::nothrow) lsd_decoder();
  if (!d) return LSD_ERR_OOM;
  d->m = m;
  d->n = n;
  d->E = E;
  d->bp_iters = bp_iters;
  d->order = lsd_order;
  d->osd_cs = o.osd_method == 1 ? o.osd_cs_order : -1;
  d->opt = o;
  d->alpha = o.ms_scaling > 0.f ? o.ms_scaling : 0.625f;
  d->st = static_cast<cudaStream_t>(o.stream);
  int rc = LSD_OK;
  int32_t *d_chk_ptr = nullptr, *d_var_ptr = nullptr;
  uint16_t *d_chk_var = nullptr, *d_var_edge = nullptr, *d_var_chk = nullptr;
  float *d_prior = nullptr, *d_probs = nullptr;
  long long* d_wfix = nullptr;
  std::vector<float> probs(channel_probs, channel_probs + n);
  if ((rc = upload(d, &d_chk_ptr, chk_ptr)) || (rc = upload(d, &d_var_ptr, var_ptr)) ||
      (rc = upload(d, &d_chk_var, chk_var)) || (rc = upload(d, &d_var_edge, var_edge)) ||
      (rc = upload(d, &d_var_chk, var_chk)) || (rc = upload(d, &d_probs, probs)) ||
      (rc = dev_alloc(d, reinterpret_cast<void**>(&d_prior), (size_t)n * sizeof(float))) ||
      (rc = dev_alloc(d, reinterpret_cast<void**>(&d_wfix), (size_t)n * sizeof(long long))) ||
      (rc = dev_alloc(d, reinterpret_cast<void**>(&d->d_ctr), sizeof(DevCounters)))) {
    lsd_destroy(d);
    return rc;
  }
  if (cudaMallocHost(reinterpret_cast<void**>(&d->h_ctr), sizeof(DevCounters)) != cudaSuccess) {
    cudaGetLastError();
    lsd_destroy(d);
    return LSD_ERR_OOM;
  }
  for (auto& ev : d->ev)
    if (cudaEventCreate(&ev) != cudaSuccess) {
      lsd_destroy(d);
      return LSD_ERR_CUDA;
    }
  DevGraph& g = d->g;
  g.m = m;
  g.n = n;
  g.E = E;
  g.max_row_deg = max_row;
  g.max_col_deg = max_col;
  g.min_row_deg = min_row;
  g.min_col_deg = min_col;
  g.chk_ptr = d_chk_ptr;
  g.chk_var = d_chk_var;
  g.var_ptr = d_var_ptr;
  g.var_edge = d_var_edge;
  g.var_chk = d_var_chk;
  g.prior = d_prior;
  g.wfix = d_wfix;
  d->d_probs = d_probs;
  cudaError_t ce = launch_priors(d_probs, d_prior, d_wfix, n, d->st);
  d->launches++;
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(d->st);
  if (ce != cudaSuccess) {
    lsd_destroy(d);
    return cuda_fail(ce);
  }
  d->bp_variant = -1;
  ce = bp_config(g, o.bp_lanes, o.bp_method, o.bp_kernel, &d->bp_variant, &d->bp_grid,
                 &d->bp_block, &d->bp_smem);
  if (ce != cudaSuccess) {
    cudaGetLastError();
    lsd_destroy(d);
    return LSD_ERR_UNSUPPORTED;
  }
  ce = o.lsd_kernel == 2 ? cudaErrorInvalidValue
                         : lsd_config(g, lsd_order, o.lsd_warps, &d->lsd_warps, &d->lsd_grid,
                                      &d->lsd_smem, &d->lsd_W);
  if (ce == cudaSuccess)
    d->dense = d->lsd_ok = true;
  else
    cudaGetLastError();
  // The sparse LSD takes the matrices that the dense kernel does not, and those whose dense
  // ranking is a sort in shared memory (more than 144 detectors or 288 faults), where it is the
  // faster one also when every shot of a batch reaches LSD: dense / sparse of 16 to 50 000 shots
  // 3.1-7.6 for LSD-0 of a 144 x 324 space-time matrix (7.41 / 0.97 ms for 50 000), 1.7-4.5 for
  // its LSD-6 and LSD-14 with OSD-CS-4; 1.4-5.5 and 1.8-4.2 for (3,6)-regular 150 x 300 and 240 x
  // 480 at p = 0.01 to 0.08 (percolating at the last: 21.4 / 15.0 ms); 11-45 beyond 256 detectors
  // or 768 faults.  Not for the single-cluster mode, whose one cluster holds every detector from
  // the start.
  const bool prefer_sparse = !d->dense || (o.lsd_kernel == 0 && (m > 144 || n > 288));
  if (prefer_sparse && o.lsd_kernel != 1 && !o.single_cluster) {
    if (sparse_config(g, lsd_order, &d->sp_grid_small, &d->sp_grid_big) == cudaSuccess) {
      // one allocation: the rows' columns padded to the largest row, the columns' first four rows
      const int D = std::max(max_row, 1);
      const size_t rows_at = ((size_t)m * D + 3) & ~(size_t)3;  // (read eight bytes at a time)
      std::vector<uint16_t> pad(rows_at + (size_t)n * 4, 0xffff);
      for (int i = 0; i < m; ++i)
        for (int q = chk_ptr[i]; q < chk_ptr[i + 1]; ++q) pad[(size_t)i * D + q - chk_ptr[i]] = chk_var[q];
      for (int j = 0; j < n; ++j)
        for (int q = var_ptr[j]; q < std::min(var_ptr[j + 1], var_ptr[j] + 4); ++q)
          pad[rows_at + (size_t)j * 4 + q - var_ptr[j]] = var_chk[q];
      uint16_t* d_pad = nullptr;
      rc = upload(d, &d_pad, pad);
      if (rc == LSD_OK && (ce = cudaStreamSynchronize(d->st)) != cudaSuccess) rc = cuda_fail(ce);
      if (rc != LSD_OK && !no_room(rc)) {
        lsd_destroy(d);
        return rc;
      }
      // no room for the tables: the dense kernel if it takes the matrix, else BP alone
      d->sparse = rc == LSD_OK || !d->dense;
      d->sparse_rc = d->sparse ? rc : LSD_OK;
      d->lsd_ok = true;
      if (rc == LSD_OK) {
        g.chk_pad = d_pad;
        g.var_pad = d_pad + rows_at;
        d->sp_tables = pad.size() * sizeof(uint16_t);
      }
      d->sp_stride_small = sparse_scratch_bytes(m, n, false, lsd_order > 0);
      d->sp_stride_big = sparse_scratch_bytes(m, n, true, lsd_order > 0);
    } else {
      cudaGetLastError();  // BP still works; LSD entry points report LSD_ERR_UNSUPPORTED
    }
  }
  *out = d;
  return LSD_OK;
}

int lsd_decode_batch(lsd_decoder* d, int64_t shots, const uint8_t* syndromes,
                     uint8_t* corrections, uint8_t* status, float* posteriors, lsd_stats* stats) {
  if (!d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) {
    if (stats) {
      std::memset(stats, 0, sizeof(*stats));
    }
    return LSD_OK;
  }
  if (!syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  if (!d->lsd_ok) return LSD_ERR_UNSUPPORTED;
  int rc = ensure_workspace(d, shots);
  if (rc) return rc;
  if ((rc = reset_counters(d))) return rc;
  BPArgs a = bp_args(d, shots, syndromes);
  a.corrections = corrections;
  a.status = status;
  a.posteriors = posteriors;
  a.queue = d->d_queue;
  a.queue_llr = d->d_queue_llr;
  cudaEventRecord(d->ev[0], d->st);
  cudaError_t e = launch_bp(a, d->bp_variant, d->bp_grid, d->bp_block, d->bp_smem, d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  cudaEventRecord(d->ev[1], d->st);
  LSDArgs l{};
  l.packed = d->io_packed;
  l.g = d->g;
  l.count_from_ctr = 1;
  l.queue = d->d_queue;
  l.llr = d->d_queue_llr;
  l.llr_by_item = 1;
  l.syndromes = syndromes;
  l.corrections = corrections;
  l.status = status;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = d->d_ctr;
  rc = run_lsd(d, l, shots);
  if (rc) return rc;
  cudaEventRecord(d->ev[2], d->st);
  d->last_shots = shots;
  d->last_kind = 1;
  if (stats) return fill_stats(d, shots, stats, true);
  return LSD_OK;
}

int lsd_decode_batch_host(lsd_decoder* d, int64_t shots, const uint8_t* syndromes,
                          uint8_t* corrections, uint8_t* status, lsd_stats* stats) {
  if (!d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return lsd_decode_batch(d, 0, nullptr, nullptr, nullptr, nullptr, stats);
  if (!syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  // row bytes of syndromes and corrections: bytes, or 32-bit words when bit-packed
  const size_t srow = d->io_packed ? 4 * (size_t)((d->m + 31) / 32) : (size_t)d->m;
  const size_t crow = d->io_packed ? 4 * (size_t)((d->n + 31) / 32) : (size_t)d->n;
  const size_t need = (size_t)shots * (srow + crow + 1);
  if (need > d->stage_cap) {
    cudaError_t e = cudaStreamSynchronize(d->st);
    if (e != cudaSuccess) return cuda_fail(e);
    dev_free(d, d->d_stage, d->stage_cap);
    d->d_stage = nullptr;
    d->stage_cap = 0;
    int rc = dev_alloc(d, reinterpret_cast<void**>(&d->d_stage), need);
    if (rc) return rc;
    d->stage_cap = need;
  }
  uint8_t* dsyn = d->d_stage;
  uint8_t* dcor = dsyn + (size_t)shots * srow;
  uint8_t* dst = dcor + (size_t)shots * crow;
  // Large batches without statistics run as a pipeline of chunks: chunk i+1's syndromes
  // copy in and chunk i-1's corrections copy out (two copy streams) while chunk i decodes.
  constexpr int64_t kMinChunk = 65536;
  constexpr int kMaxChunks = lsdgb::kHostChunks;
  const int chunks = (int)std::min<int64_t>(kMaxChunks, shots / kMinChunk);
  if (!stats && chunks >= 2) {
    cudaError_t e = cudaSuccess;
    if (!d->cp_in) e = cudaStreamCreateWithFlags(&d->cp_in, cudaStreamNonBlocking);
    if (e == cudaSuccess && !d->cp_out) e = cudaStreamCreateWithFlags(&d->cp_out, cudaStreamNonBlocking);
    for (int i = 0; i < 2 * kMaxChunks && e == cudaSuccess; ++i)
      if (!d->cev[i]) e = cudaEventCreateWithFlags(&d->cev[i], cudaEventDisableTiming);
    // dense LSD: two compute lanes (no per-decoder scratch beyond counters and queue rows)
    const bool lanes2 = !d->sparse && d->lsd_ok;
    if (lanes2) {
      if (e == cudaSuccess && !d->st2) e = cudaStreamCreateWithFlags(&d->st2, cudaStreamNonBlocking);
      if (e == cudaSuccess && !d->join) e = cudaEventCreateWithFlags(&d->join, cudaEventDisableTiming);
    }
    if (e != cudaSuccess) return cuda_fail(e);
    if (lanes2 && !d->d_ctr_chunks) {
      const int rc = dev_alloc(d, reinterpret_cast<void**>(&d->d_ctr_chunks),
                               kMaxChunks * sizeof(DevCounters));
      if (rc) return rc;
    }
    if (lanes2) {
      const int rc = ensure_workspace(d, shots);
      if (rc) return rc;
      // the second lane starts after everything already queued on the decoder's stream
      e = cudaEventRecord(d->join, d->st);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(d->st2, d->join, 0);
      if (e != cudaSuccess) return cuda_fail(e);
    }
    int64_t base = 0;
    for (int i = 0; i < chunks; ++i) {
      const int64_t cnt = shots * (i + 1) / chunks - base;
      const size_t sm = (size_t)base * srow, sn = (size_t)base * crow;
      const size_t ln = (size_t)base * d->n;  // LLR rows of the chunk's queue
      cudaStream_t cs = (lanes2 && (i & 1)) ? d->st2 : d->st;
      e = cudaMemcpyAsync(dsyn + sm, syndromes + sm, (size_t)cnt * srow, cudaMemcpyHostToDevice,
                          d->cp_in);
      if (e == cudaSuccess) e = cudaEventRecord(d->cev[2 * i], d->cp_in);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, d->cev[2 * i], 0);
      if (e != cudaSuccess) return cuda_fail(e);
      const int rc =
          lanes2 ? decode_chunk(d, cnt, dsyn + sm, dcor + sn, dst + base, d->d_ctr_chunks + i,
                                d->d_queue + base, d->d_queue_llr + ln, cs)
                 : lsd_decode_batch(d, cnt, dsyn + sm, dcor + sn, dst + base, nullptr, nullptr);
      if (rc) return rc;
      e = cudaEventRecord(d->cev[2 * i + 1], cs);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(d->cp_out, d->cev[2 * i + 1], 0);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(corrections + sn, dcor + sn, (size_t)cnt * crow,
                            cudaMemcpyDeviceToHost, d->cp_out);
      if (e == cudaSuccess && status)
        e = cudaMemcpyAsync(status + base, dst + base, (size_t)cnt, cudaMemcpyDeviceToHost,
                            d->cp_out);
      if (e != cudaSuccess) return cuda_fail(e);
      base += cnt;
    }
    e = cudaStreamSynchronize(d->cp_out);
    if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
    if (e == cudaSuccess && lanes2) e = cudaStreamSynchronize(d->st2);
    return e == cudaSuccess ? LSD_OK : cuda_fail(e);
  }
  cudaError_t e = cudaMemcpyAsync(dsyn, syndromes, (size_t)shots * srow, cudaMemcpyHostToDevice,
                                  d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  int rc = lsd_decode_batch(d, shots, dsyn, dcor, dst, nullptr, nullptr);
  if (rc) return rc;
  e = cudaMemcpyAsync(corrections, dcor, (size_t)shots * crow, cudaMemcpyDeviceToHost, d->st);
  if (e == cudaSuccess && status)
    e = cudaMemcpyAsync(status, dst, (size_t)shots, cudaMemcpyDeviceToHost, d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  if (stats) return fill_stats(d, shots, stats, true);
  e = cudaStreamSynchronize(d->st);
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

int lsd_decode_batch_packed(lsd_decoder* d, int64_t shots, const uint32_t* syndromes,
                            uint32_t* corrections, uint8_t* status, lsd_stats* stats) {
  if (!d) return LSD_ERR_INVALID_ARG;
  d->io_packed = 1;
  const int rc = lsd_decode_batch(d, shots, reinterpret_cast<const uint8_t*>(syndromes),
                                  reinterpret_cast<uint8_t*>(corrections), status, nullptr, stats);
  d->io_packed = 0;
  return rc;
}

int lsd_decode_batch_host_packed(lsd_decoder* d, int64_t shots, const uint32_t* syndromes,
                                 uint32_t* corrections, uint8_t* status, lsd_stats* stats) {
  if (!d) return LSD_ERR_INVALID_ARG;
  d->io_packed = 1;
  const int rc = lsd_decode_batch_host(d, shots, reinterpret_cast<const uint8_t*>(syndromes),
                                       reinterpret_cast<uint8_t*>(corrections), status, stats);
  d->io_packed = 0;
  return rc;
}

int lsd_bp_batch(lsd_decoder* d, int64_t shots, const uint8_t* syndromes, float* posteriors,
                 uint8_t* converged, int32_t* iterations) {
  if (!d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return LSD_OK;
  if (!syndromes || !posteriors) return LSD_ERR_INVALID_ARG;
  int rc = reset_counters(d);
  if (rc) return rc;
  BPArgs a = bp_args(d, shots, syndromes);
  a.posteriors = posteriors;
  a.converged_out = converged;
  a.iters_out = iterations;
  cudaEventRecord(d->ev[0], d->st);
  cudaError_t e = launch_bp(a, d->bp_variant, d->bp_grid, d->bp_block, d->bp_smem, d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  cudaEventRecord(d->ev[1], d->st);
  d->last_shots = shots;
  d->last_kind = 2;
  return LSD_OK;
}

int lsd_postprocess_batch(lsd_decoder* d, int64_t shots, const float* llrs,
                          const uint8_t* syndromes, uint8_t* corrections, uint8_t* status,
                          int32_t* shot_info) {
  if (!d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return LSD_OK;
  if (!llrs || !syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  if (!d->lsd_ok) return LSD_ERR_UNSUPPORTED;
  int rc = reset_counters(d);
  if (rc) return rc;
  LSDArgs l{};
  l.g = d->g;
  l.count = shots;
  l.count_from_ctr = 0;
  l.queue = nullptr;
  l.llr = llrs;
  l.llr_by_item = 0;
  l.syndromes = syndromes;
  l.corrections = corrections;
  l.status = status;
  l.shot_info = shot_info;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = d->d_ctr;
  cudaEventRecord(d->ev[1], d->st);
  rc = run_lsd(d, l, shots);
  if (rc) return rc;
  cudaEventRecord(d->ev[2], d->st);
  d->last_shots = shots;
  d->last_kind = 3;
  return LSD_OK;
}

int lsd_get_stats(lsd_decoder* d, lsd_stats* stats) {
  if (!d || !stats) return LSD_ERR_INVALID_ARG;
  if (d->last_kind == 0) {
    std::memset(stats, 0, sizeof(*stats));
    return LSD_OK;
  }
  return fill_stats(d, d->last_shots, stats, true);
}

int lsd_get_priors(lsd_decoder* d, float* priors) {
  if (!d || !priors) return LSD_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(priors, d->g.prior, (size_t)d->n * sizeof(float),
                                  cudaMemcpyDeviceToHost, d->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

int lsd_workspace_bytes(const lsd_decoder* d, size_t* bytes) {
  if (!d || !bytes) return LSD_ERR_INVALID_ARG;
  *bytes = d->bytes;
  return LSD_OK;
}

int lsd_kernel_launches(const lsd_decoder* d, int64_t* count) {
  if (!d || !count) return LSD_ERR_INVALID_ARG;
  *count = d->launches;
  return LSD_OK;
}

const char* lsd_bp_variant_name(int32_t variant) {
  const char* s = bp_variant_name(variant);
  return s ? s : "";
}

}  // extern "C"

// ---------------------------------------------------------------------------------------
// Allocation-free decode (lsd_decode_batch_static).  The scratch of the BP and LSD kernels
// (counters, queue, LLR rows) comes from one file-scope device array instead of the
// decoder's workspace.  Its device address is looked up once per device, on that device.
// ---------------------------------------------------------------------------------------
namespace {

static __device__ __align__(256) unsigned char g_static_scratch[LSD_STATIC_SCRATCH_BYTES];

constexpr int kMaxStaticDevices = 64;

std::mutex g_static_mu;
void* g_static_ptr[kMaxStaticDevices] = {};

// Device address of g_static_scratch on the current device.  Only a successful lookup is
// kept: a failed one (for example a first call made during stream capture) clears the
// runtime's error state and is retried by the next call.
int static_scratch(void** ptr) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (dev < 0 || dev >= kMaxStaticDevices) return LSD_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return cuda_fail(e != cudaSuccess ? e : cudaErrorInvalidSymbol);
    }
    g_static_ptr[dev] = p;
  }
  *ptr = g_static_ptr[dev];
  return LSD_OK;
}

size_t round256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

extern "C" int lsd_decode_batch_static(lsd_decoder* d, int64_t shots, const uint8_t* syndromes,
                                       uint8_t* corrections, uint8_t* status) {
  if (!d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return LSD_OK;
  if (!syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  if (!d->dense) return LSD_ERR_UNSUPPORTED;
  const size_t ctr_bytes = round256(sizeof(DevCounters));
  const size_t queue_bytes = round256((size_t)shots * sizeof(int32_t));
  const size_t llr_bytes = (size_t)shots * (size_t)d->n * sizeof(float);
  if (ctr_bytes + queue_bytes + llr_bytes > LSD_STATIC_SCRATCH_BYTES) return LSD_ERR_ADMISSION;
  void* base = nullptr;
  int rc = static_scratch(&base);
  if (rc) return rc;
  unsigned char* p = static_cast<unsigned char*>(base);
  DevCounters* ctr = reinterpret_cast<DevCounters*>(p);
  int32_t* queue = reinterpret_cast<int32_t*>(p + ctr_bytes);
  float* queue_llr = reinterpret_cast<float*>(p + ctr_bytes + queue_bytes);
  // the array keeps the previous call's contents: the counters must start at zero
  cudaError_t e = cudaMemsetAsync(ctr, 0, sizeof(DevCounters), d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  BPArgs a = bp_args(d, shots, syndromes);
  a.ctr = ctr;
  a.corrections = corrections;
  a.status = status;
  a.queue = queue;
  a.queue_llr = queue_llr;
  e = launch_bp(a, d->bp_variant, d->bp_grid, d->bp_block, d->bp_smem, d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  LSDArgs l{};
  l.g = d->g;
  l.count_from_ctr = 1;
  l.queue = queue;
  l.llr = queue_llr;
  l.llr_by_item = 1;
  l.syndromes = syndromes;
  l.corrections = corrections;
  l.status = status;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = ctr;
  e = launch_lsd(l, d->lsd_warps, d->lsd_grid, d->lsd_smem, d->st);
  d->launches++;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

// ---------------------------------------------------------------------------------------
// Learned prior
// ---------------------------------------------------------------------------------------
namespace {

void prior_free(lsd_prior* p) {
  if (!p) return;
  cudaStreamSynchronize(p->dec ? p->dec->st : nullptr);
  for (void* q : {(void*)p->d_params, (void*)p->d_grads, (void*)p->d_m, (void*)p->d_v,
                  (void*)p->d_loss, (void*)p->d_scratch, (void*)p->d_flag})
    if (q) cudaFree(q);
  if (p->h_loss) cudaFreeHost(p->h_loss);
  cudaGetLastError();
  delete p;
}

int prior_alloc(void** q, size_t bytes) {
  cudaError_t e = cudaMalloc(q, bytes ? bytes : 16);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_fail(e);
  }
  return LSD_OK;
}

int prior_grads(lsd_prior* p, int64_t shots, const uint8_t* syn, const uint8_t* err) {
  lsd_decoder* d = p->dec;
  if (p->grid_train <= 0) return LSD_ERR_UNSUPPORTED;
  cudaError_t e = cudaMemsetAsync(p->d_grads, 0, sizeof(float) * p->np, d->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->d_loss, 0, sizeof(double), d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  e = launch_prior(true, p->grid_train, d->g, p->rounds, p->d_params, shots, syn, err, nullptr,
                   p->d_scratch, p->d_grads, p->d_loss, d->st);
  d->launches++;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

}  // namespace

extern "C" {

int lsd_prior_num_params(void) { return prior_num_params(); }

int lsd_prior_destroy(lsd_prior* p) {
  prior_free(p);
  return LSD_OK;
}

int lsd_prior_create(lsd_prior** out, lsd_decoder* d, int32_t rounds, const float* params) {
  if (!out || !d || rounds < 1 || rounds > kPriorMaxRounds) return LSD_ERR_INVALID_ARG;
  *out = nullptr;
  lsd_prior* p = new (std::nothrow) lsd_prior();
  if (!p) return LSD_ERR_OOM;
  p->dec = d;
  p->rounds = rounds;
  p->np = prior_num_params();
  cudaError_t ce = prior_config(d->m, d->n, d->E, false, &p->grid_fwd);
  if (ce != cudaSuccess) {
    cudaGetLastError();
    prior_free(p);
    return LSD_ERR_UNSUPPORTED;
  }
  if (prior_tc_config(d->g, &p->grid_tc) != cudaSuccess) {
    cudaGetLastError();
    p->grid_tc = 0;
  }
  // training is optional: its kernel keeps more per-shot state
  if (d->m > 96 || d->n > 192 ||
      prior_config(d->m, d->n, d->E, true, &p->grid_train) != cudaSuccess) {
    cudaGetLastError();
    p->grid_train = 0;
  }
  int rc;
  const size_t nb = sizeof(float) * p->np;
  if ((rc = prior_alloc((void**)&p->d_params, nb)) || (rc = prior_alloc((void**)&p->d_grads, nb)) ||
      (rc = prior_alloc((void**)&p->d_m, nb)) || (rc = prior_alloc((void**)&p->d_v, nb)) ||
      (rc = prior_alloc((void**)&p->d_loss, sizeof(double))) ||
      (rc = prior_alloc((void**)&p->d_flag, sizeof(int))) ||
      (p->grid_train > 0 &&
       (rc = prior_alloc((void**)&p->d_scratch,
                         sizeof(float) * prior_scratch_floats(d->m, d->n, rounds, p->grid_train))))) {
    prior_free(p);
    return rc;
  }
  if (cudaMallocHost((void**)&p->h_loss, sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    prior_free(p);
    return LSD_ERR_OOM;
  }
  *out = p;
  cudaMemsetAsync(p->d_flag, 0, sizeof(int), d->st);
  if (params) return lsd_prior_set_params(p, params);
  cudaMemsetAsync(p->d_params, 0, nb, d->st);
  cudaMemsetAsync(p->d_m, 0, nb, d->st);
  cudaMemsetAsync(p->d_v, 0, nb, d->st);
  ce = cudaStreamSynchronize(d->st);
  return ce == cudaSuccess ? LSD_OK : cuda_fail(ce);
}

int lsd_prior_set_params(lsd_prior* p, const float* params) {
  if (!p || !params) return LSD_ERR_INVALID_ARG;
  lsd_decoder* d = p->dec;
  const size_t nb = sizeof(float) * p->np;
  cudaError_t e = cudaMemcpyAsync(p->d_params, params, nb, cudaMemcpyHostToDevice, d->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->d_m, 0, nb, d->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->d_v, 0, nb, d->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
  p->step = 0;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

int lsd_prior_get_params(lsd_prior* p, float* params) {
  if (!p || !params) return LSD_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(params, p->d_params, sizeof(float) * p->np,
                                  cudaMemcpyDeviceToHost, p->dec->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->dec->st);
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

int lsd_prior_forward(lsd_prior* p, int64_t shots, const uint8_t* syndromes, float* llrs) {
  if (!p || shots < 0) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return LSD_OK;
  if (!syndromes || !llrs) return LSD_ERR_INVALID_ARG;
  lsd_decoder* d = p->dec;
  cudaError_t e;
  if (prior_uses_tc(p)) {
    e = cudaMemsetAsync(p->d_flag, 0, sizeof(int), d->st);
    if (e == cudaSuccess)
      e = launch_prior_tc(p->grid_tc, d->g, p->rounds, p->d_params, shots, syndromes, llrs,
                          nullptr, nullptr, nullptr, nullptr, nullptr, p->d_flag, d->st);
  } else {
    e = launch_prior(false, p->grid_fwd, d->g, p->rounds, p->d_params, shots, syndromes,
                     nullptr, llrs, nullptr, nullptr, nullptr, d->st);
  }
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  if (!prior_uses_tc(p)) return LSD_OK;
  // the tensor-memory kernel reports a completion wait that ran out (a device fault, never
  // expected): synchronize and read its flag
  int flag = 0;
  e = cudaMemcpyAsync(&flag, p->d_flag, sizeof(int), cudaMemcpyDeviceToHost, d->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  return flag ? LSD_ERR_TIMEOUT : LSD_OK;
}

int lsd_prior_get_kernel(const lsd_prior* p, int32_t* kernel, int32_t* grid) {
  if (!p || !kernel || !grid) return LSD_ERR_INVALID_ARG;
  const bool tc = prior_uses_tc(p);
  *kernel = tc ? 2 : 1;
  *grid = tc ? p->grid_tc : p->grid_fwd;
  return LSD_OK;
}

int lsd_prior_set_kernel(lsd_prior* p, int32_t kernel) {
  if (!p || kernel < 0 || kernel > 2) return LSD_ERR_INVALID_ARG;
  if (kernel == 2 && p->grid_tc <= 0) return LSD_ERR_UNSUPPORTED;
  p->kernel = kernel;
  return LSD_OK;
}

int lsd_prior_gradient(lsd_prior* p, int64_t shots, const uint8_t* syndromes,
                       const uint8_t* errors, double* loss, float* grads) {
  if (!p || shots <= 0 || !syndromes || !errors || !loss) return LSD_ERR_INVALID_ARG;
  int rc = prior_grads(p, shots, syndromes, errors);
  if (rc) return rc;
  lsd_decoder* d = p->dec;
  cudaError_t e = cudaMemcpyAsync(p->h_loss, p->d_loss, sizeof(double), cudaMemcpyDeviceToHost,
                                  d->st);
  if (e == cudaSuccess && grads)
    e = cudaMemcpyAsync(grads, p->d_grads, sizeof(float) * p->np, cudaMemcpyDeviceToHost, d->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  *loss = *p->h_loss / ((double)shots * d->n);
  return LSD_OK;
}

int lsd_prior_train_step(lsd_prior* p, int64_t shots, const uint8_t* syndromes,
                         const uint8_t* errors, float lr, double* loss) {
  if (!p || shots <= 0 || !syndromes || !errors || !(lr > 0.f)) return LSD_ERR_INVALID_ARG;
  int rc = prior_grads(p, shots, syndromes, errors);
  if (rc) return rc;
  lsd_decoder* d = p->dec;
  p->step++;
  cudaError_t e = launch_adam(p->d_params, p->d_grads, p->d_m, p->d_v, p->np, lr, p->step, d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  if (loss) {
    e = cudaMemcpyAsync(p->h_loss, p->d_loss, sizeof(double), cudaMemcpyDeviceToHost, d->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
    if (e != cudaSuccess) return cuda_fail(e);
    *loss = *p->h_loss / ((double)shots * d->n);
  }
  return LSD_OK;
}

int lsd_sample(lsd_decoder* d, uint64_t seed, int64_t first_shot, int64_t shots,
               uint8_t* errors, uint8_t* syndromes) {
  if (!d || shots < 0 || first_shot < 0) return LSD_ERR_INVALID_ARG;
  if (shots == 0) return LSD_OK;
  if (!errors || !syndromes) return LSD_ERR_INVALID_ARG;
  cudaError_t e = launch_sample(d->g, d->d_probs, seed, first_shot, shots, errors, syndromes, d->st);
  d->launches++;
  return e == cudaSuccess ? LSD_OK : cuda_fail(e);
}

int lsd_decode_learned(lsd_decoder* d, lsd_prior* p, int64_t shots, const uint8_t* syndromes,
                       uint8_t* corrections, uint8_t* status, lsd_stats* stats) {
  if (!d || !p || p->dec != d || shots < 0 || shots > INT32_MAX) return LSD_ERR_INVALID_ARG;
  if (shots == 0) {
    if (stats) std::memset(stats, 0, sizeof(*stats));
    return LSD_OK;
  }
  if (!syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  if (!d->lsd_ok) return LSD_ERR_UNSUPPORTED;
  int rc = ensure_workspace(d, shots);
  if (rc) return rc;
  // the fallback needs the status of every shot
  uint8_t* st = status;
  if (!st) return LSD_ERR_INVALID_ARG;
  if ((rc = reset_counters(d))) return rc;
  cudaEventRecord(d->ev[0], d->st);
  cudaError_t e =
      prior_uses_tc(p)
          ? launch_prior_tc(p->grid_tc, d->g, p->rounds, p->d_params, shots, syndromes, nullptr,
                            corrections, st, d->d_queue, d->d_queue_llr, d->d_ctr,
                            &d->d_ctr->timeout_flag, d->st)
          : launch_prior_decode(p->grid_fwd, d->g, p->rounds, p->d_params, shots, syndromes,
                                nullptr, corrections, st, d->d_queue, d->d_queue_llr, d->d_ctr,
                                d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  cudaEventRecord(d->ev[1], d->st);
  LSDArgs l{};
  l.g = d->g;
  l.count_from_ctr = 1;
  l.queue = d->d_queue;
  l.llr = d->d_queue_llr;
  l.llr_by_item = 1;
  l.syndromes = syndromes;
  l.corrections = corrections;
  l.status = st;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = d->d_ctr;
  rc = run_lsd(d, l, shots);
  if (rc) return rc;
  cudaEventRecord(d->ev[2], d->st);
  d->last_shots = shots;
  d->last_kind = 1;
  // fallback: BP + LSD for the shots LSD could not solve
  e = cudaMemcpyAsync(d->h_ctr, d->d_ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, d->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(d->st);
  if (e != cudaSuccess) return cuda_fail(e);
  const DevCounters learned = *d->h_ctr;
  if (learned.timeout_flag) return LSD_ERR_TIMEOUT;
  if (learned.unsolvable > 0) {
    std::vector<uint8_t> hs((size_t)shots);
    e = cudaMemcpy(hs.data(), st, (size_t)shots, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e);
    for (int64_t k = 0; k < shots; ++k) {
      if (hs[(size_t)k] != LSD_SHOT_UNSOLVABLE) continue;
      rc = lsd_decode_batch(d, 1, syndromes + k * d->m, corrections + k * d->n, st + k, nullptr,
                            nullptr);
      if (rc) return rc;
    }
  }
  if (stats) {
    std::memset(stats, 0, sizeof(*stats));
    stats->shots = shots;
    stats->bp_converged = (int64_t)learned.bp_converged;
    stats->lsd_shots = (int64_t)learned.lsd_count;
    stats->unsolvable = (int64_t)learned.unsolvable;
    stats->lsd_steps = (int64_t)learned.lsd_steps;
    stats->kappa_max = learned.kappa_max;
    stats->nu_max = learned.nu_max;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, d->ev[0], d->ev[1]) == cudaSuccess) stats->ms_bp = ms;
    if (cudaEventElapsedTime(&ms, d->ev[1], d->ev[2]) == cudaSuccess) stats->ms_lsd = ms;
    cudaGetLastError();
  }
  return LSD_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------
// Autotuner
// ---------------------------------------------------------------------------------------
extern "C" int lsd_autotune(lsd_decoder* d, int64_t shots, const uint8_t* syndromes,
                            lsd_tune_report* report) {
  if (!d || shots <= 0 || shots > INT32_MAX || !syndromes) return LSD_ERR_INVALID_ARG;
  lsd_tune_report rep{};
  float* post = nullptr;
  uint8_t *corr = nullptr, *st = nullptr;
  cudaError_t e = cudaMalloc(&post, (size_t)shots * d->n * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&corr, (size_t)shots * d->n);
  if (e == cudaSuccess) e = cudaMalloc(&st, (size_t)shots);
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  int rc = e == cudaSuccess ? LSD_OK : cuda_fail(e);
  // A candidate that fails at launch leaves the stream and the context usable; anything
  // else (an error the stream reports) ends the search.
  auto skippable = [&](int r) -> bool {
    if (r != LSD_ERR_CUDA) return false;
    cudaGetLastError();
    return cudaStreamSynchronize(d->st) == cudaSuccess;
  };
  auto timed = [&](auto&& fn, float* ms) -> int {
    float best = 0.f;
    for (int rep_i = 0; rep_i < 3; ++rep_i) {  // first run warms up; keep the best of the rest
      cudaEventRecord(t0, d->st);
      int r = fn();
      if (r) return r;
      cudaEventRecord(t1, d->st);
      cudaError_t ee = cudaEventSynchronize(t1);
      if (ee != cudaSuccess) return cuda_fail(ee);
      float v = 0.f;
      cudaEventElapsedTime(&v, t0, t1);
      if (rep_i == 1 || (rep_i > 1 && v < best)) best = v;
    }
    *ms = best;
    return LSD_OK;
  };
  // ---- BP variants ----
  if (!rc) {
    const int v0 = d->bp_variant, g0 = d->bp_grid, b0 = d->bp_block;
    const size_t s0 = d->bp_smem;
    int best_v = v0, best_g = g0, best_b = b0;
    size_t best_s = s0;
    float best_ms = 0.f;
    for (int v = 0; v < bp_num_variants() && !rc; ++v) {
      int vv = v, grid = 0, block = 0;
      size_t smem = 0;
      if (bp_config(d->g, 0, d->opt.bp_method, 0, &vv, &grid, &block, &smem) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      d->bp_variant = vv;
      d->bp_grid = grid;
      d->bp_block = block;
      d->bp_smem = smem;
      float ms = 0.f;
      rc = timed([&]() { return lsd_bp_batch(d, shots, syndromes, post, nullptr, nullptr); }, &ms);
      if (rc && skippable(rc)) {  // the candidate did not launch: drop it
        rc = LSD_OK;
        continue;
      }
      if (rc) break;
      rep.bp_candidates++;
      if (v == v0) rep.ms_bp_first = ms;
      if (best_ms == 0.f || ms < best_ms) {
        best_ms = ms;
        best_v = vv;
        best_g = grid;
        best_b = block;
        best_s = smem;
      }
    }
    d->bp_variant = best_v;
    d->bp_grid = best_g;
    d->bp_block = best_b;
    d->bp_smem = best_s;
    rep.bp_variant = best_v;
    rep.ms_bp_best = best_ms;
  }
  // ---- LSD: warps per CTA of the dense kernel, and the sparse kernel (candidate 0) where it
  // was chosen for a matrix that the dense one takes too ----
  if (!rc && d->dense) {
    const bool sparse0 = d->sparse;
    const int w0 = sparse0 ? 0 : d->lsd_warps;
    int best_w = d->lsd_warps, best_g = d->lsd_grid;
    size_t best_s = d->lsd_smem;
    float best_ms = 0.f;
    bool best_sparse = sparse0;
    const int cand[] = {0, 2, 4, 8, 16};
    for (int w : cand) {
      if (w == 0 && !sparse0) continue;
      int ww = 0, grid = 0, words = 0;
      size_t smem = 0;
      d->sparse = w == 0;
      if (w && (lsd_config(d->g, d->order, w, &ww, &grid, &smem, &words) != cudaSuccess || ww != w)) {
        cudaGetLastError();
        continue;
      }
      if (w) {
        d->lsd_warps = ww;
        d->lsd_grid = grid;
        d->lsd_smem = smem;
      }
      float ms = 0.f;
      rc = timed([&]() { return lsd_decode_batch(d, shots, syndromes, corr, st, nullptr, nullptr); },
                 &ms);
      if (rc && skippable(rc)) {
        rc = LSD_OK;
        continue;
      }
      if (rc) break;
      rep.lsd_candidates++;
      if (w == w0) rep.ms_lsd_first = ms;
      if (best_ms == 0.f || ms < best_ms) {
        best_ms = ms;
        best_sparse = d->sparse;
        if (w) {
          best_w = ww;
          best_g = grid;
          best_s = smem;
        }
      }
    }
    d->lsd_warps = best_w;
    d->lsd_grid = best_g;
    d->lsd_smem = best_s;
    // (a decoder that found no room for the sparse kernel's scratch above has dropped its tables)
    d->sparse = sparse0 && d->g.chk_pad;
    if (!best_sparse) drop_sparse(d);
    rep.lsd_warps = d->sparse ? 0 : best_w;
    rep.ms_lsd_best = best_ms;
  }
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  if (post) cudaFree(post);
  if (corr) cudaFree(corr);
  if (st) cudaFree(st);
  cudaGetLastError();
  if (report) *report = rep;
  return rc;
}

// ---------------------------------------------------------------------------------------
// Decode with a device-side shot count (graph capture by the serving runtime).  The
// workspace must already hold max_shots (no allocation may happen during a capture).
// ---------------------------------------------------------------------------------------
int lsdgb::bp_batch_counted(lsd_decoder* d, int64_t max_shots, const long long* shots_dev,
                            const uint8_t* syndromes, uint8_t* corrections, uint8_t* status) {
  if (!d || max_shots <= 0 || !shots_dev || !syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  if (!d->lsd_ok) return LSD_ERR_UNSUPPORTED;
  if ((size_t)max_shots > d->cap_shots) return LSD_ERR_ADMISSION;
  if (d->sparse && (!d->d_sp_big || (d->sp_grid_big > 0 && (size_t)max_shots > d->spill_cap)))
    return LSD_ERR_ADMISSION;
  int rc = reset_counters(d);
  if (rc) return rc;
  BPArgs a = bp_args(d, max_shots, syndromes);
  a.shots_dev = shots_dev;
  a.corrections = corrections;
  a.status = status;
  a.queue = d->d_queue;
  a.queue_llr = d->d_queue_llr;
  cudaError_t e = launch_bp(a, d->bp_variant, d->bp_grid, d->bp_block, d->bp_smem, d->st);
  d->launches++;
  if (e != cudaSuccess) return cuda_fail(e);
  return LSD_OK;
}

int lsdgb::lsd_batch_counted(lsd_decoder* d, int64_t max_shots, const uint8_t* syndromes,
                             uint8_t* corrections, uint8_t* status) {
  if (!d || max_shots <= 0 || !syndromes || !corrections) return LSD_ERR_INVALID_ARG;
  LSDArgs l{};
  l.g = d->g;
  l.count_from_ctr = 1;
  l.queue = d->d_queue;
  l.llr = d->d_queue_llr;
  l.llr_by_item = 1;
  l.syndromes = syndromes;
  l.corrections = corrections;
  l.status = status;
  l.order = d->order;
  l.osd_cs = d->osd_cs;
  l.single_cluster = d->opt.single_cluster;
  l.ctr = d->d_ctr;
  return run_lsd(d, l, max_shots);
}

int lsdgb::decode_batch_counted(lsd_decoder* d, int64_t max_shots, const long long* shots_dev,
                                const uint8_t* syndromes, uint8_t* corrections, uint8_t* status) {
  const int rc = bp_batch_counted(d, max_shots, shots_dev, syndromes, corrections, status);
  return rc ? rc : lsd_batch_counted(d, max_shots, syndromes, corrections, status);
}
