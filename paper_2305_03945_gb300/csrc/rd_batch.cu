// Batched, continuously served implicit steps (many independent solves of uneven grid sizes).
//
// Every admitted request owns a slot: device buffers cut from one arena sized by the caller's
// HBM budget, two descriptors (FP32 inner sweeps, FP64 outer loop) and a control block whose
// phase drives FP64 defect correction and the time-step loop on the device:
//   BEGIN  -> build the step's rhs from U^k and the outer threshold (k_step_b)
//   RESID  -> r = F(u) in FP64, outer stopping rule, arm the FP32 inner solve (k_step_b)
//   INNER  -> FP32 G-prox PDHG iterations on the correction equation (the line kernels of
//             rd_batch_lines.cuh; k_res_b, k_col_b, k_upd_b with a side below 16 points; one launch
//             per inner solve for small grids), returning to AXPY when the inner solve stops
//   AXPY   -> u += d in FP64 (k_axpy_b)
//   DONE / FAILED after the last step or on divergence.
// One CUDA graph holds graph_k iterations of [axpy, step, sweeps] for each equation kind present, a
// branch per kind and sort of slot; every launch covers all slots of that kind through a work list of (slot, block)
// pairs, so instances of different sizes share one launch.  A host worker thread admits queued
// requests when a slot and arena space are free, relaunches the graph, and retires finished
// slots while the others keep running (continuous batching).
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <map>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "../../include/rd_pdhg.h"
#include "rd_3d.cuh"
#include "rd_batch3.h"
#include "rd_batch_lines.h"
#include "rd_launch3.h"
#include "rd_launch_small.h"
#include "rd_mu.h"

namespace rd {

// ---------------------------------------------------------------------------------------
// batched kernels
// ---------------------------------------------------------------------------------------
template <class T, int K>
__global__ void __launch_bounds__(MaxThreads<T>::value, MinBlocks<T>::value)
    k_res_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (*((volatile const int*)&slots[w.x].phase) != PH_INNER) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  res_body<T, K>(sd, &slots[w.x].inner, slots + w.x, w.y, smem_raw);
}

template <class T>
__global__ void __launch_bounds__(MaxThreads<T>::value, MinBlocks<T>::value)
    k_col_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (*((volatile const int*)&slots[w.x].phase) != PH_INNER) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  col_body<T, false>(sd, &slots[w.x].inner, slots + w.x, w.y, smem_raw);
}

template <class T, int K>
__global__ void __launch_bounds__(MaxThreads<T>::value, MinBlocks<T>::value)
    k_upd_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (*((volatile const int*)&slots[w.x].phase) != PH_INNER) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  upd_body<T, K>(sd, &slots[w.x].inner, slots + w.x, w.y, smem_raw);
}

// FP64 state of a slot read through the boundary map
struct UAcc {
  const double* u;
  int nx, ny, bc;
  __device__ __forceinline__ double operator()(int i, int j) const {
    return u[(size_t)bcmap(i, ny, bc) * nx + bcmap(j, nx, bc)];
  }
};

// PH_BEGIN: rhs of the step from U^k (kind constants, the explicit part of the convex split),
//           ||U^k||, outer threshold, -> PH_RESID.
// PH_RESID: r = F(u) in FP64; r and u rounded to FP32 for the inner solve; d = 0, P_0 = 0;
//           outer stopping rule -> next step / DONE / FAILED, or arm the inner solve -> PH_INNER.
template <int K>
__global__ void __launch_bounds__(256) k_step_b(const Desc* __restrict__ d64s, Slot* __restrict__ slots,
                                                const int2* __restrict__ items) {
  __shared__ Desc sd;
  __shared__ double red[32];
  const int2 w = items[blockIdx.x];
  Slot* sl = slots + w.x;
  const int ph = *((volatile const int*)&sl->phase);
  if (ph != PH_BEGIN && ph != PH_RESID) return;
  load_desc(sd, d64s + w.x);
  __syncthreads();
  const Desc& d = sd;
  const int nx = d.nx, ny = d.ny, bc = d.bc;
  const size_t plane = (size_t)nx * ny;
  const int band = w.y;
  const int y0 = band * d.band_rows;
  const int rows = min(d.band_rows, ny - y0);
  double* u = static_cast<double*>(d.X);
  double* rhs = static_cast<double*>(const_cast<void*>(d.rhs));
  constexpr int nc = KT<K>::two ? 2 : 1;
  State* outer = &sl->outer;
  if (ph == PH_BEGIN) {
    double acc = 0.0;
    for (int idx = threadIdx.x; idx < nc * rows * nx; idx += blockDim.x) {
      const int c = idx / (rows * nx);
      const int rem = idx - c * rows * nx;
      const int r = rem / nx, j = rem - r * nx;
      const int i = y0 + r;
      const size_t o = c * plane + (size_t)i * nx + j;
      const double uv = u[o];
      double v = uv;
      if constexpr (K == KK_CH_SPLIT) {
        const UAcc f{u, nx, ny, bc};
        v = uv - d.dt * d.b * lap5(f, i, j, uv, d.hx2, d.hy2);
      } else if constexpr (K == KK_GS) {
        if (c == 0) v = uv + d.dt * d.p[2];
      } else if constexpr (K == KK_SCHNAK) {
        v = uv + d.dt * d.p[2] * (c == 0 ? d.p[3] : d.p[4]);
      }
      rhs[o] = v;
      acc += uv * uv;
    }
    const double s = block_sum(acc, red);
    if (threadIdx.x == 0) d.partials[band] = s;
    if (last_block(outer, d.nbands)) {
      __threadfence();
      const double tot = sum_partials(d.partials, d.nbands, red);
      if (threadIdx.x == 0) {
        outer->ticket = 0u;
        outer->aux = sqrt(tot);
        outer->thresh = sl->tol_kind == 1 ? sl->tol * sqrt(tot) : sl->tol;
        outer->n = 0;
        outer->r = 0.0;
        outer->r0 = 0.0;
        outer->status = ST_ACTIVE;
        sl->phase = PH_RESID;
      }
    }
    return;
  }
  // PH_RESID
  const UAcc f0{u, nx, ny, bc}, f1{u + plane, nx, ny, bc};
  double acc0 = 0.0, acc1 = 0.0;
  for (int idx = threadIdx.x; idx < rows * nx; idx += blockDim.x) {
    const int r = idx / nx, j = idx - r * nx;
    const int i = y0 + r;
    const size_t o = (size_t)i * nx + j;
    double wv[2] = {0.0, 0.0};
    residual_pt<double, K, false>(d, f0, f1, f0, f1, i, j, rhs[o], nc > 1 ? rhs[plane + o] : 0.0, wv);
    for (int c = 0; c < nc; ++c) {
      const size_t oc = c * plane + o;
      d.f32_r[oc] = (float)wv[c];
      d.f32_u[oc] = (float)u[oc];
      d.f32_d[oc] = 0.f;
      d.f32_p0[oc] = 0.f;
    }
    acc0 += wv[0] * wv[0];
    acc1 += wv[1] * wv[1];
  }
  const double s0 = block_sum(acc0, red);
  const double s1 = nc > 1 ? block_sum(acc1, red) : 0.0;
  if (threadIdx.x == 0) {
    d.partials[band] = s0;
    if (nc > 1) d.partials[d.nbands + band] = s1;
  }
  if (last_block(outer, d.nbands)) {
    __threadfence();
    double tot = 0.0;
    for (int c = 0; c < nc; ++c) tot += sqrt(sum_partials(d.partials + c * d.nbands, d.nbands, red));
    if (threadIdx.x == 0) {
      const double meas = d.meas_div_dt ? tot / d.dt : tot;
      const double prev = outer->r;
      outer->ticket = 0u;
      outer->r = meas;
      const int n = outer->n;
      if (n == 0) outer->r0 = meas;
      const double r0 = n == 0 ? meas : outer->r0;
      outer->n = n + 1;
      sl->outer_total += 1;
      if (meas <= outer->thresh) {
        outer->status = ST_CONVERGED;
        sl->steps_done += 1;
        sl->phase = sl->steps_done >= sl->nsteps ? PH_DONE : PH_BEGIN;
      } else if (!isfinite(meas) || meas > kDivergeFactor * r0 || outer->n > sl->max_outer) {
        outer->status = isfinite(meas) && meas <= kDivergeFactor * r0 ? ST_NOT_CONVERGED : ST_DIVERGED;
        sl->phase = PH_FAILED;
      } else {
        State* in = &sl->inner;
        in->stall_mul = next_stall_mul(n, meas, prev, in->stall_mul);
        in->n = 0;
        in->r = 0.0;
        in->r0 = 0.0;
        in->thresh = fmax(sl->rtol * tot, 0.5 * outer->thresh * (d.meas_div_dt ? d.dt : 1.0));
        in->status = ST_ACTIVE;
        in->ticket = 0u;
        sl->phase = PH_INNER;
      }
    }
  }
}

// PH_AXPY: u += d (FP64 += FP32), pointwise over the band, -> PH_RESID.
__global__ void __launch_bounds__(256) k_axpy_b(const Desc* __restrict__ d64s, Slot* __restrict__ slots,
                                                const int2* __restrict__ items) {
  const int2 w = items[blockIdx.x];
  Slot* sl = slots + w.x;
  if (*((volatile const int*)&sl->phase) != PH_AXPY) return;
  const Desc& d = d64s[w.x];
  const int nx = d.nx, ny = d.ny, nc = d.ncomp;
  const size_t plane = (size_t)nx * ny;
  const int y0 = w.y * d.band_rows;
  const int rows = min(d.band_rows, ny - y0);
  double* u = static_cast<double*>(d.X);
  const float* dl = d.f32_d;
  for (int idx = threadIdx.x; idx < nc * rows * nx; idx += blockDim.x) {
    const int c = idx / (rows * nx);
    const size_t o = c * plane + (size_t)y0 * nx + (idx - c * rows * nx);
    u[o] += (double)dl[o];
  }
  if (last_block(&sl->outer, d.nbands) && threadIdx.x == 0) {
    sl->outer.ticket = 0u;
    sl->phase = PH_RESID;
  }
}

}  // namespace rd

using namespace rd;

// ---------------------------------------------------------------------------------------
// host runtime
// ---------------------------------------------------------------------------------------
namespace {

constexpr int kBatchThreads = 256;      // FP32 sweep blocks
constexpr int kBatchMaxSide = 1024;     // batch grids: sides 4 .. 1024, powers of two
constexpr int kBatchMaxSide3 = 512;     // 3-D batch grids: sides 4 .. 512
constexpr int kBatchMaxBlk3 = 1024;     // blocks per 3-D slot (plan3's cap)
constexpr int kBatchBandRows = 4;
constexpr int kBatchColWidth = 4;
constexpr int kBatchGroups = 7;         // equation kinds served
constexpr int kBatchParts = 5;          // branches of a group's graph: see launch_branch
// Entries one slot adds to the work lists at most.  2-D: ny / 4 bands, and ny / 2 blocks of the line kernels or
// 2 nx / 4 column blocks of two components; 3-D: its blocks.
constexpr int kBatchSlotItems =
    std::max(kBatchMaxSide / kBatchBandRows + std::max(kBatchMaxSide / 2, 2 * kBatchMaxSide / kBatchColWidth), kBatchMaxBlk3);
const int kGroupKey[kBatchGroups] = {KK_NONE_LAP, KK_AC, KK_CH_IMPL, KK_CH_SPLIT, KK_NONE_BIH, KK_GS, KK_SCHNAK};

double now_s() {
  using namespace std::chrono;
  return duration<double>(steady_clock::now().time_since_epoch()).count();
}

// first-fit allocator over one device arena (offsets aligned to 256 bytes)
struct Arena {
  char* base = nullptr;
  size_t size = 0;
  std::map<size_t, size_t> free_;  // offset -> length
  void init(char* b, size_t s) {
    base = b;
    size = s;
    free_.clear();
    free_[0] = s;
  }
  static size_t up(size_t v) { return (v + 255) & ~(size_t)255; }
  char* alloc(size_t n) {
    n = up(n);
    for (auto it = free_.begin(); it != free_.end(); ++it) {
      if (it->second >= n) {
        const size_t off = it->first, len = it->second;
        free_.erase(it);
        if (len > n) free_[off + n] = len - n;
        return base + off;
      }
    }
    return nullptr;
  }
  void release(char* p, size_t n) {
    n = up(n);
    size_t off = (size_t)(p - base);
    auto nx = free_.lower_bound(off);
    if (nx != free_.end() && off + n == nx->first) {
      n += nx->second;
      free_.erase(nx);
    }
    auto pv = free_.lower_bound(off);
    if (pv != free_.begin()) {
      --pv;
      if (pv->first + pv->second == off) {
        off = pv->first;
        n += pv->second;
        free_.erase(pv);
      }
    }
    free_[off] = n;
  }
};

// A work list of (slot, block) pairs: built on the host, and its part of the batch's device array (rd_batch::d_items).
struct ItemList {
  int2* d = nullptr;
  int n = 0;
  std::vector<int2> h;
};

struct Request {
  uint64_t id = 0;
  rd_request req{};
  std::vector<double> u0;
  double t_submit = 0;
};

struct SlotHost {
  bool used = false;
  uint64_t id = 0;
  rd_request req{};
  int key = 0, group = 0;
  char* mem = nullptr;
  size_t mem_bytes = 0;
  size_t npts = 0;
  double t_submit = 0, t_admit = 0;
  bool nd3 = false;  // a 3-D request
  bool fast = false; // every side 16 points or more: the line kernels of rd_batch_lines.cuh
  int small = 0;     // a 2-D request whose inner solves run in one launch (1 one block, 2 a cluster)
  Desc d32{}, d64{};
  // what else admission copies to the device.  A copy from pageable memory may read its source after the
  // call has returned (it does where the device reads host memory through the host's page tables), so the
  // sources live here until the stream has been synchronised: no wait per admission.
  std::vector<double> u0;
  std::vector<float> mu;
  Slot ctl{};
};

size_t slot_bytes(const rd_request& r, size_t* npts_out) {
  const bool nd3 = r.grid.ndim == 3;
  const int nz = nd3 ? r.grid.n[2] : 1;
  const size_t npts = (size_t)r.reaction.ncomp * r.grid.n[0] * r.grid.n[1] * nz;
  if (npts_out) *npts_out = npts;
  const int nx = r.grid.n[0], ny = r.grid.n[1];
  size_t b = 0;
  if (nd3) {
    b += Arena::up(npts * 8) * 2;                       // u, rhs (FP64)
    b += Arena::up(npts * 4) * 5;                       // d, P, WY, r32, u32
    b += Arena::up((size_t)(nx + ny + nz) * 2 * 8);     // twiddles + rotations (FP32 complex)
    b += Arena::up((size_t)(nx + ny + nz) * 4);         // mu tables
    b += Arena::up((size_t)2 * kBatchMaxBlk3 * 8);      // partials
    return b;
  }
  b += Arena::up(npts * 8) * 2;                       // u, rhs (FP64)
  b += Arena::up(npts * 4) * 6;                       // d, P0, P1, WY, r32, u32
  b += Arena::up((size_t)(nx + ny) * 2 * 8) * 1;      // twiddles + rotations (FP32 complex)
  b += Arena::up((size_t)(nx + ny) * 4);              // mu tables
  b += Arena::up((size_t)2 * (ny / 2 + 1) * 8);  // partials (two-row bands at the finest tile)
  return b;
}

}  // namespace

struct rd_batch {
  cudaStream_t stream = nullptr;
  cudaStream_t cap_stream = nullptr;
  rd_opts opts{};
  int max_slots = 0;
  size_t budget = 0;
  Arena arena;
  char* arena_mem = nullptr;
  Desc* d_d32 = nullptr;
  Desc* d_d64 = nullptr;
  Slot* d_slots = nullptr;
  Slot* h_slots = nullptr;  // pinned mirror
  // Work lists per group.  Slots with a one-launch inner solve: one entry per slot in small1 / small2
  // (one block / a cluster each) and the bands of their step phases (axpy, step) in small_phase.  2-D
  // slots: bands and column blocks of the Stockham sweeps (band, col), or, with line kernels, the bands
  // of the step phases and the blocks of the line kernels (line_phase, line2).  3-D slots: blocks of
  // either set of kernels (old3, line3).
  struct Lists {
    ItemList band, col, small_phase, small1, small2, line_phase, line2, old3, line3;
    int smem_small[2] = {};
    int smem_line2[2] = {}, smem_line3[2] = {};  // row and column kernels
    int thr3[3] = {}, smem3[3] = {};             // transform passes of the old3 slots
  } lists[kBatchGroups];
  int2* d_items = nullptr;   // the entries of all lists, kBatchSlotItems per slot (allocated once: serving
  int2* h_items = nullptr;   // allocates no device memory but the graph's), and their pinned source
  int smem_usable = 0;
  // one capture stream and join event per branch of the graph (see rebuild_graph)
  cudaStream_t branch_stream[kBatchParts * kBatchGroups] = {};
  cudaEvent_t ev_join[kBatchParts * kBatchGroups] = {};
  cudaEvent_t ev_fork = nullptr;
  int stale = 0;  // slots of the current work lists that have been retired
  // twiddle and DCT rotation tables of every line length 4 .. kBatchMaxSide, shared by all slots: those
  // of length n at n - 4 complex entries each (twiddles), and behind all of them (rotations); sines of
  // pi k / (2 kBatchMaxSide) for the eigenvalues
  cx<float>* d_tables = nullptr;
  std::vector<double> sines;
  std::vector<long double> sines_l;
  std::vector<SlotHost> slots;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  bool graph_dirty = true;
  bool lists_dirty = false;  // the slots have changed since the work lists were built
  int smem_sweep = 0;
  int smem_sweep2 = 0;  // the band kernels of the two-species kinds
  // queues.  mu guards the queues, outputs, stats, worker_error, stop and the arena's free list
  // (allocated and released by the worker, read by rd_batch_get_stats); never held across a
  // CUDA call that waits on the device.
  std::mutex mu;
  std::condition_variable cv;
  std::deque<Request> queue;
  std::deque<rd_result> done;
  std::map<uint64_t, double*> outputs;  // request id -> caller's host output buffer
  uint64_t next_id = 1;
  bool stop = false;
  std::thread worker;
  std::string worker_error;
  rd_batch_stats stats{};
};

namespace {

rd_status bfail(rd_status s, const std::string& m) {
  rd::set_last_error(m.c_str());
  return s;
}

int key_of(const rd_request& r) {
  if (r.reaction.kind == RD_RX_NONE) return r.op == RD_OP_NEG_BIHARMONIC ? KK_NONE_BIH : KK_NONE_LAP;
  return r.reaction.kind;
}

int group_of(int key) {
  for (int g = 0; g < kBatchGroups; ++g)
    if (kGroupKey[g] == key) return g;
  return -1;
}

// Tables of every line length, once per batch: one pass of long double trigonometry (software on this
// host) for all admissions.  w_n^k = w_N^{k N/n} with N = kBatchMaxSide, an exact scaling of the argument.
rd_status make_tables(rd_batch* b) {
  const long double pi = 3.141592653589793238462643383279502884L;
  constexpr int N = kBatchMaxSide;
  b->sines.resize(2 * N + 1);
  b->sines_l.resize(2 * N + 1);
  std::vector<cx<float>> tab(2 * (2 * N - 4));
  std::vector<cx<float>> tw(N), dc(N);
  for (int k = 0; k < N; ++k) {
    const long double t = 2.0L * pi * k / N;
    tw[k] = cx<float>{(float)cosl(t), (float)(-sinl(t))};
    const long double q = pi * k / (2.0L * N);
    dc[k] = cx<float>{(float)cosl(q), (float)sinl(q)};
  }
  for (int k = 0; k <= 2 * N; ++k) {
    b->sines_l[k] = sinl(pi * k / (2.0L * N));
    b->sines[k] = (double)b->sines_l[k];
  }
  for (int n = 4; n <= N; n *= 2)
    for (int k = 0; k < n; ++k) {
      tab[n - 4 + k] = tw[k * (N / n)];
      tab[2 * N - 4 + n - 4 + k] = dc[k * (N / n)];
    }
  cudaError_t e = cudaMalloc(&b->d_tables, tab.size() * sizeof(cx<float>));
  if (e == cudaSuccess) e = cudaMemcpy(b->d_tables, tab.data(), tab.size() * sizeof(cx<float>), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? RD_OK : bfail(RD_ERR_OOM, std::string("batch tables: ") + cudaGetErrorString(e));
}

const cx<float>* twiddles_of(const rd_batch* b, int n) { return b->d_tables + (n - 4); }
const cx<float>* rotations_of(const rd_batch* b, int n) { return b->d_tables + (2 * kBatchMaxSide - 4) + (n - 4); }

// eigenvalues of -Lap along one axis, mu(k) = 4/h^2 sin^2(pi k / (d n)), d = 1 periodic, 2 Neumann
void append_mu(const rd_batch* b, int n, bool neumann, double h, std::vector<float>& mu) {
  const int step = (neumann ? 1 : 2) * (kBatchMaxSide / n);
  for (int k = 0; k < n; ++k) {
    const int q = k * step;
    mu.push_back(eigenvalue32(b->sines[q], b->sines_l[q], h));
  }
}

template <class T, int K>
cudaError_t allow_batch_kernels(int optin) {
  cudaFuncAttributes fa;
  cudaError_t e;
  if ((e = cudaFuncGetAttributes(&fa, k_res_b<T, K>)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(k_res_b<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                optin - (int)fa.sharedSizeBytes)) != cudaSuccess)
    return e;
  if ((e = cudaFuncGetAttributes(&fa, k_upd_b<T, K>)) != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_upd_b<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              optin - (int)fa.sharedSizeBytes);
}

// The chain of one graph iteration for part `part` of group g: 0 the 2-D slots on the Stockham sweeps,
// 1 the slots with a one-launch inner solve, 2 the 3-D slots on the Stockham passes, 3 and 4 the 2-D and
// 3-D slots on the line kernels.
template <int K>
void launch_group(rd_batch* b, int g, int part, cudaStream_t s) {
  const rd_batch::Lists& l = b->lists[g];
  const ItemList& ph = part == 0 ? l.band : (part == 1 ? l.small_phase : l.line_phase);
  k_axpy_b<<<ph.n, 256, 0, s>>>(b->d_d64, b->d_slots, ph.d);
  k_step_b<K><<<ph.n, 256, 0, s>>>(b->d_d64, b->d_slots, ph.d);
  if (part == 0) {
    const int smem_res = KT<K>::two ? b->smem_sweep2 : b->smem_sweep, smem_col = b->smem_sweep;
    k_res_b<float, K><<<l.band.n, kBatchThreads, smem_res, s>>>(b->d_d32, b->d_slots, l.band.d);
    k_col_b<float><<<l.col.n, kBatchThreads, smem_col, s>>>(b->d_d32, b->d_slots, l.col.d);
    k_upd_b<float, K><<<l.band.n, kBatchThreads, smem_res, s>>>(b->d_d32, b->d_slots, l.band.d);
  } else if (part == 1) {
    launch_small_batch(K, 1, b->d_d32, b->d_slots, l.small1.d, l.small1.n, l.smem_small[0], s);
    launch_small_batch(K, 2, b->d_d32, b->d_slots, l.small2.d, l.small2.n, l.smem_small[1], s);
  } else {
    batch_lines2(K, BatchLines{b->d_d32, b->d_slots, l.line2.d, l.line2.n, l.smem_line2[0], l.smem_line2[1]}, s);
  }
}

// entries of the list that decides whether a part has work
int part_items(const rd_batch* b, int g, int part) {
  const rd_batch::Lists& l = b->lists[g];
  const ItemList* of[kBatchParts] = {&l.band, &l.small_phase, &l.old3, &l.line2, &l.line3};
  return of[part]->n;
}

void launch_branch(rd_batch* b, int g, int part, cudaStream_t s) {
  const rd_batch::Lists& l = b->lists[g];
  if (part == 2 || part == 4) {
    const ItemList& it = part == 2 ? l.old3 : l.line3;
    Batch3Launch L{b->d_d32, b->d_d64, b->d_slots, it.d, it.n, {}, {}};
    for (int a = 0; a < 3; ++a) {
      L.thr[a] = l.thr3[a];
      L.smem[a] = l.smem3[a];
    }
    if (part == 2) {
      batch3_launch_group(kGroupKey[g], L, s);
    } else {
      batch3_launch_phases(kGroupKey[g], L, s);
      batch_lines3(kGroupKey[g], BatchLines{b->d_d32, b->d_slots, it.d, it.n, l.smem_line3[0], l.smem_line3[1]}, s);
    }
    return;
  }
  switch (kGroupKey[g]) {
    case KK_NONE_LAP: launch_group<KK_NONE_LAP>(b, g, part, s); break;
    case KK_AC: launch_group<KK_AC>(b, g, part, s); break;
    case KK_CH_IMPL: launch_group<KK_CH_IMPL>(b, g, part, s); break;
    case KK_CH_SPLIT: launch_group<KK_CH_SPLIT>(b, g, part, s); break;
    case KK_GS: launch_group<KK_GS>(b, g, part, s); break;
    case KK_SCHNAK: launch_group<KK_SCHNAK>(b, g, part, s); break;
    default: launch_group<KK_NONE_BIH>(b, g, part, s); break;
  }
}

// (Re)capture the graph of graph_k iterations over the current work lists.  Slots of different
// groups, and the sweep, one-launch and 3-D slots of one group, share nothing: each such part is a
// branch of its own through all its iterations, so that the kernels of one fill the launch gaps and
// idle SMs of the others (one chain through all of them: 28 launches in a row per iteration of a mix
// of two kinds with cubes).  An iteration of the one-launch slots is a whole inner solve, as long as
// several sweeps: their branch has a quarter of the iterations, so that no branch waits long for it, or
// half where no other kind of branch is there to wait (16 runs of 5 steps, a quarter / half / all: 4 x 4 3.0 / 2.1 /
// 2.4 ms, 64 x 64 3.8 / 3.6 / 3.6 ms; of one step: 64 x 64 1.51 / 1.57 / 1.68 ms).
rd_status rebuild_graph(rd_batch* b) {
  if (b->gexec) {
    cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
  }
  if (b->graph) {
    cudaGraphDestroy(b->graph);
    b->graph = nullptr;
  }
  cudaError_t e = cudaSuccess;
  std::vector<int> live;
  bool only_small = true;
  for (int k = 0; k < kBatchParts * kBatchGroups; ++k) {
    if (part_items(b, k / kBatchParts, k % kBatchParts) == 0) continue;
    live.push_back(k);
    only_small = only_small && k % kBatchParts == 1;
    if (!b->branch_stream[k]) e = cudaStreamCreateWithFlags(&b->branch_stream[k], cudaStreamNonBlocking);
    if (e == cudaSuccess && !b->ev_join[k]) e = cudaEventCreateWithFlags(&b->ev_join[k], cudaEventDisableTiming);
    if (e != cudaSuccess) return bfail(RD_ERR_CUDA, std::string("batch branches: ") + cudaGetErrorString(e));
  }
  e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return bfail(RD_ERR_CUDA, std::string("batch capture: ") + cudaGetErrorString(e));
  cudaEventRecord(b->ev_fork, b->cap_stream);
  for (int k : live) {
    const int part = k % kBatchParts;
    cudaStream_t s = b->branch_stream[k];
    cudaStreamWaitEvent(s, b->ev_fork, 0);
    const int iters = part == 1 ? std::max(1, b->opts.graph_k / (only_small ? 2 : 4)) : b->opts.graph_k;
    for (int i = 0; i < iters; ++i) launch_branch(b, k / kBatchParts, part, s);
    cudaEventRecord(b->ev_join[k], s);
    cudaStreamWaitEvent(b->cap_stream, b->ev_join[k], 0);
  }
  cudaError_t el = cudaGetLastError();
  e = cudaStreamEndCapture(b->cap_stream, &b->graph);
  if (el != cudaSuccess || e != cudaSuccess)
    return bfail(RD_ERR_CUDA, std::string("batch capture: ") + cudaGetErrorString(el != cudaSuccess ? el : e));
  e = cudaGraphInstantiate(&b->gexec, b->graph, 0);
  if (e != cudaSuccess) return bfail(RD_ERR_CUDA, std::string("batch instantiate: ") + cudaGetErrorString(e));
  b->graph_dirty = false;
  return RD_OK;
}

// Upload the work lists of all groups from the slot table, one behind the other; at most once between two
// synchronisations of the stream (the copy may still read the entries of the last time until then).
rd_status rebuild_items(rd_batch* b) {
  for (int g = 0; g < kBatchGroups; ++g) {
    rd_batch::Lists& l = b->lists[g];
    for (ItemList* it : {&l.band, &l.col, &l.small_phase, &l.small1, &l.small2, &l.line_phase, &l.line2, &l.old3, &l.line3})
      it->h.clear();
    for (int m = 0; m < 2; ++m) l.smem_small[m] = l.smem_line2[m] = l.smem_line3[m] = 0;
    for (int a = 0; a < 3; ++a) l.thr3[a] = l.smem3[a] = 0;
  }
  for (int s = 0; s < b->max_slots; ++s) {
    const SlotHost& sh = b->slots[s];
    if (!sh.used) continue;
    const Desc& d = sh.d32;
    rd_batch::Lists& l = b->lists[sh.group];
    auto list = [s](ItemList& it, int n) {
      for (int k = 0; k < n; ++k) it.h.push_back(make_int2(s, k));
    };
    if (sh.fast) {
      list(sh.nd3 ? l.line3 : l.line2, d.blk3);
      if (!sh.nd3) list(l.line_phase, d.nbands);
      int* sm = sh.nd3 ? l.smem_line3 : l.smem_line2;
      int row = 0, col = 0;
      if (sh.nd3) batch_lines3_plan(d, 1, &row, &col);
      else batch_lines2_plan(d, 1, &row, &col);
      sm[0] = std::max(sm[0], row);
      sm[1] = std::max(sm[1], col);
    } else if (sh.nd3) {
      list(l.old3, d.blk3);
      const int n_ax[3] = {d.nx, d.ny, d.nz};
      for (int a = 0; a < 3; ++a) {
        l.thr3[a] = std::max(l.thr3[a], d.thr3[a]);
        l.smem3[a] = std::max(l.smem3[a], lines3_smem_bytes<float>(n_ax[a], d.lw3[a], d.bc == BC_NEUMANN));
      }
    } else if (sh.small) {
      list(l.small_phase, d.nbands);
      list(sh.small == 1 ? l.small1 : l.small2, 1);
      int& sm = l.smem_small[sh.small - 1];
      sm = std::max(sm, small_smem_of(sh.small, d.nx, d.ny, d.ncomp, sh.key, d.bc == BC_NEUMANN));
    } else {
      list(l.band, d.nbands);
      list(l.col, d.ncomp * d.ncolblk);
    }
  }
  size_t n = 0;
  const size_t cap = (size_t)b->max_slots * kBatchSlotItems;
  for (int g = 0; g < kBatchGroups; ++g) {
    rd_batch::Lists& l = b->lists[g];
    for (ItemList* it : {&l.band, &l.col, &l.small_phase, &l.small1, &l.small2, &l.line_phase, &l.line2, &l.old3, &l.line3}) {
      if (n + it->h.size() > cap) return bfail(RD_ERR_CUDA, "batch work lists beyond their bound");
      it->d = b->d_items + n;
      it->n = (int)it->h.size();
      std::copy(it->h.begin(), it->h.end(), b->h_items + n);
      n += it->h.size();
    }
  }
  const cudaError_t e = cudaMemcpyAsync(b->d_items, b->h_items, n * sizeof(int2), cudaMemcpyHostToDevice, b->stream);
  if (e != cudaSuccess) return bfail(RD_ERR_CUDA, cudaGetErrorString(e));
  b->graph_dirty = true;
  b->lists_dirty = false;
  b->stale = 0;
  return RD_OK;
}

// Set-up of an admitted 3-D request in slot s (arena block mem): arrays, the FP32 and FP64
// descriptors with the 3-D plan, tables, state and control block.
void admit3(rd_batch* b, Request& q, int s, char* mem, size_t npts, rd_status* err) {
  SlotHost& sh = b->slots[s];
  const rd_request& r = q.req;
  const int nx = r.grid.n[0], ny = r.grid.n[1], nz = r.grid.n[2];
  char* p = mem;
  auto take = [&](size_t n) {
    char* q2 = p;
    p += Arena::up(n);
    return q2;
  };
  double* u = (double*)take(npts * 8);
  double* rhs = (double*)take(npts * 8);
  float* dl = (float*)take(npts * 4);
  float* p0 = (float*)take(npts * 4);
  float* wy = (float*)take(npts * 4);
  float* r32 = (float*)take(npts * 4);
  float* u32 = (float*)take(npts * 4);
  take((size_t)(nx + ny + nz) * 2 * 8);  // (the tables are the batch's; the request's size stays as it was)
  float* mus = (float*)take((size_t)(nx + ny + nz) * 4);
  double* parts = (double*)take((size_t)2 * kBatchMaxBlk3 * 8);
  const double hx = r.grid.length[0] / nx, hy = r.grid.length[1] / ny, hz = r.grid.length[2] / nz;
  Desc d{};
  d.nx = nx;
  d.ny = ny;
  d.nz = nz;
  d.ncomp = 1;
  d.lognx = ilog2i(nx);
  d.logny = ilog2i(ny);
  d.lognz = ilog2i(nz);
  d.bc = r.bc;
  d.op = r.op;
  d.kind = r.reaction.kind;
  d.precond = 1;
  d.mode = MODE_PDHG;
  d.hx2 = 1.0 / (hx * hx);
  d.hy2 = 1.0 / (hy * hy);
  d.hz2 = 1.0 / (hz * hz);
  d.dt = r.dt;
  d.a = r.reaction.a;
  d.b = r.reaction.b;
  for (int k = 0; k < 6; ++k) d.p[k] = r.reaction.p[k];
  d.tau_u = r.tau;
  d.tau_p = r.sigma;
  d.omega = b->opts.omega;
  d.batched = 1;
  d.partials = parts;
  for (int c = 0; c < 2; ++c) {
    d.gc1[c] = r.op == RD_OP_LAPLACIAN ? r.reaction.a * r.dt : 0.0;
    d.gc2[c] = r.op == RD_OP_LAPLACIAN ? 0.0 : r.reaction.a * r.dt;
  }
  d.inv_nn = 1.0 / ((double)nx * ny * nz);
  const char* why = nullptr;
  if (!plan3(nx, ny, nz, 1, 4, r.bc == RD_BC_NEUMANN, 226 * 1024, d, &why)) {
    *err = bfail(RD_ERR_UNSUPPORTED, std::string("admission: ") + why);
    return;
  }
  Desc d64 = d, d32 = d;
  d64.dc = 0;
  d64.meas_div_dt = r.tol_kind == RD_TOL_RES_ABS;
  d64.X = u;
  d64.rhs = rhs;
  d64.f32_d = dl;
  d64.f32_p0 = p0;
  d64.f32_r = r32;
  d64.f32_u = u32;
  d32.dc = 1;
  d32.meas_div_dt = 0;
  d32.stall_window = b->opts.dc_stall_window > 0 ? b->opts.dc_stall_window : 8;
  d32.X = dl;
  d32.base = u32;
  d32.rhs = r32;
  d32.P[0] = p0;
  d32.P[1] = p0;
  d32.WY = wy;
  d32.twx = twiddles_of(b, nx);
  d32.dcx = rotations_of(b, nx);
  d32.twy = twiddles_of(b, ny);
  d32.dcy = rotations_of(b, ny);
  d32.twz = twiddles_of(b, nz);
  d32.dcz = rotations_of(b, nz);
  d32.mux = mus;
  d32.muy = mus + nx;
  d32.muz = mus + nx + ny;
  sh.fast = nx >= 16 && ny >= 16 && nz >= 16;
  if (sh.fast) {
    int row = 0, col = 0;
    d32.blk3 = d64.blk3 = batch_lines3_plan(d32, kBatchMaxBlk3, &row, &col);
    d32.P[1] = wy;
  }
  sh.d32 = d32;
  sh.d64 = d64;
  sh.nd3 = true;
  const int n_ax[3] = {nx, ny, nz};
  const double h_ax[3] = {hx, hy, hz};
  for (int a = 0; a < 3; ++a) append_mu(b, n_ax[a], r.bc == RD_BC_NEUMANN, h_ax[a], sh.mu);
  sh.u0 = std::move(q.u0);
  Slot& ctl = sh.ctl;
  ctl.outer.max_iter = 1 << 30;
  ctl.inner.max_iter = b->opts.max_iter;
  ctl.phase = PH_BEGIN;
  ctl.nsteps = r.nsteps;
  ctl.max_outer = b->opts.dc_max_outer;
  ctl.tol = r.tol;
  ctl.rtol = b->opts.dc_inner_rtol;
  ctl.tol_kind = r.tol_kind;
  cudaStream_t st = b->stream;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaMemcpyAsync(mus, sh.mu.data(), sh.mu.size() * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(u, sh.u0.data(), npts * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_d32 + s, &sh.d32, sizeof(Desc), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_d64 + s, &sh.d64, sizeof(Desc), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_slots + s, &ctl, sizeof(Slot), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) *err = bfail(RD_ERR_CUDA, std::string("admission: ") + cudaGetErrorString(e));
}

// Try to admit the request into a free slot.  Returns false when no slot or memory is free.
bool admit(rd_batch* b, Request& q, rd_status* err) {
  *err = RD_OK;
  int s = -1;
  for (int k = 0; k < b->max_slots; ++k)
    if (!b->slots[k].used) {
      s = k;
      break;
    }
  if (s < 0) return false;
  size_t npts = 0;
  const size_t bytes = slot_bytes(q.req, &npts);
  char* mem = nullptr;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    mem = b->arena.alloc(bytes);
  }
  if (!mem) return false;
  SlotHost& sh = b->slots[s];
  sh.used = true;
  sh.id = q.id;
  sh.req = q.req;
  sh.key = key_of(q.req);
  sh.group = group_of(sh.key);
  sh.mem = mem;
  sh.mem_bytes = bytes;
  sh.npts = npts;
  sh.t_submit = q.t_submit;
  sh.t_admit = now_s();
  sh.nd3 = sh.fast = false;
  if (q.req.grid.ndim == 3) {
    admit3(b, q, s, mem, npts, err);
    std::lock_guard<std::mutex> lk(b->mu);
    b->stats.admitted += 1;
    return true;
  }
  const rd_request& r = q.req;
  const int nx = r.grid.n[0], ny = r.grid.n[1], nc = r.reaction.ncomp;
  char* p = mem;
  auto take = [&](size_t n) {
    char* q2 = p;
    p += Arena::up(n);
    return q2;
  };
  double* u = (double*)take(npts * 8);
  double* rhs = (double*)take(npts * 8);
  float* dl = (float*)take(npts * 4);
  float* p0 = (float*)take(npts * 4);
  float* p1 = (float*)take(npts * 4);
  float* wy = (float*)take(npts * 4);
  float* r32 = (float*)take(npts * 4);
  float* u32 = (float*)take(npts * 4);
  take((size_t)(nx + ny) * 2 * 8);  // (the tables are the batch's; the request's size stays as it was)
  float* mus = (float*)take((size_t)(nx + ny) * 4);
  double* parts = (double*)take((size_t)2 * (ny / 2 + 1) * 8);
  const double hx = r.grid.length[0] / nx, hy = r.grid.length[1] / ny;
  // descriptors
  Desc d{};
  d.nx = nx;
  d.ny = ny;
  d.ncomp = nc;
  d.lognx = ilog2i(nx);
  d.logny = ilog2i(ny);
  d.bc = r.bc;
  d.op = r.op;
  d.kind = r.reaction.kind;
  d.precond = 1;
  d.mode = MODE_PDHG;
  d.band_rows = std::min(kBatchBandRows, ny);
  d.nbands = (ny + d.band_rows - 1) / d.band_rows;
  d.col_width = std::min(kBatchColWidth, nx);
  d.ncolblk = nx / d.col_width;
  d.hx2 = 1.0 / (hx * hx);
  d.hy2 = 1.0 / (hy * hy);
  d.dt = r.dt;
  d.a = r.reaction.a;
  d.b = r.reaction.b;
  for (int k = 0; k < 6; ++k) d.p[k] = r.reaction.p[k];
  d.tau_u = r.tau;
  d.tau_p = r.sigma;
  d.omega = b->opts.omega;
  d.batched = 1;
  d.partials = parts;
  const bool two = r.reaction.kind == RD_RX_GRAY_SCOTT || r.reaction.kind == RD_RX_SCHNAKENBERG;
  for (int c = 0; c < 2; ++c) {
    const double D = two ? r.reaction.p[c] : r.reaction.a;  // two species: each its own diffusivity
    d.gc1[c] = r.op == RD_OP_LAPLACIAN ? D * r.dt : 0.0;
    d.gc2[c] = r.op == RD_OP_LAPLACIAN ? 0.0 : r.reaction.a * r.dt;
  }
  d.inv_nn = 1.0 / ((double)nx * ny);
  Desc d64 = d, d32 = d;
  d64.dc = 0;
  d64.meas_div_dt = r.tol_kind == RD_TOL_RES_ABS;
  d64.X = u;
  d64.rhs = rhs;
  d64.f32_d = dl;
  d64.f32_p0 = p0;
  d64.f32_r = r32;
  d64.f32_u = u32;
  d32.dc = 1;
  d32.meas_div_dt = 0;
  d32.stall_window = b->opts.dc_stall_window > 0 ? b->opts.dc_stall_window : 8;
  d32.X = dl;
  d32.base = u32;
  d32.rhs = r32;
  d32.P[0] = p0;
  d32.P[1] = p1;
  d32.WY = wy;
  d32.twx = twiddles_of(b, nx);
  d32.dcx = rotations_of(b, nx);
  d32.twy = twiddles_of(b, ny);
  d32.dcy = rotations_of(b, ny);
  d32.mux = mus;
  d32.muy = mus + nx;
  // small grids: each inner solve in one launch (one block, or a cluster of eight)
  sh.small = b->opts.small_solve ? small_mode(nx, ny, nc, sh.key, r.bc == RD_BC_NEUMANN, b->smem_usable) : 0;
  sh.fast = !sh.small && nx >= 16 && ny >= 16;
  if (sh.fast) {
    int row = 0, col = 0;
    // (at most ny / 2 blocks: the partial sums of the norm)
    d32.blk3 = batch_lines2_plan(d32, ny / 2, &row, &col);
    d32.P[1] = wy;
  }
  sh.d32 = d32;
  sh.d64 = d64;
  // eigenvalues, state, control block
  append_mu(b, nx, r.bc == RD_BC_NEUMANN, hx, sh.mu);
  append_mu(b, ny, r.bc == RD_BC_NEUMANN, hy, sh.mu);
  sh.u0 = std::move(q.u0);
  Slot& ctl = sh.ctl;
  ctl.outer.max_iter = 1 << 30;
  ctl.inner.max_iter = b->opts.max_iter;
  ctl.phase = PH_BEGIN;
  ctl.nsteps = r.nsteps;
  ctl.max_outer = b->opts.dc_max_outer;
  ctl.tol = r.tol;
  ctl.rtol = b->opts.dc_inner_rtol;
  ctl.tol_kind = r.tol_kind;
  cudaStream_t st = b->stream;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaMemcpyAsync(mus, sh.mu.data(), sh.mu.size() * 4, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(u, sh.u0.data(), npts * 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_d32 + s, &sh.d32, sizeof(Desc), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_d64 + s, &sh.d64, sizeof(Desc), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_slots + s, &ctl, sizeof(Slot), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) *err = bfail(RD_ERR_CUDA, std::string("admission: ") + cudaGetErrorString(e));
  std::lock_guard<std::mutex> lk(b->mu);
  b->stats.admitted += 1;
  return true;
}

void retire(rd_batch* b, int s, const Slot& ctl) {
  SlotHost& sh = b->slots[s];
  rd_result res{};
  res.id = sh.id;
  res.tag = sh.req.tag;
  res.status = ctl.phase == PH_DONE ? RD_OK
               : (ctl.outer.status == ST_DIVERGED || ctl.inner.status == ST_DIVERGED ? RD_ERR_DIVERGED
                                                                                   : RD_ERR_NOT_CONVERGED);
  res.steps = ctl.steps_done;
  res.iterations = ctl.inner_total;
  res.outer_rounds = ctl.outer_total;
  res.residual = ctl.outer.r;
  double* out = nullptr;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    auto it = b->outputs.find(sh.id);
    if (it != b->outputs.end()) {
      out = it->second;
      b->outputs.erase(it);
    }
  }
  // the result copy and the wait for it: a failure of either reports the request as RD_ERR_CUDA
  // (its host output would hold stale data) and is kept as the worker's error
  cudaError_t ce = cudaSuccess;
  if (out) ce = cudaMemcpyAsync(out, sh.d64.X, sh.npts * 8, cudaMemcpyDeviceToHost, b->stream);
  const cudaError_t se = cudaStreamSynchronize(b->stream);
  if (ce == cudaSuccess) ce = se;
  std::string copy_error;
  if (ce != cudaSuccess) {
    res.status = RD_ERR_CUDA;
    copy_error = std::string("result copy of request ") + std::to_string(sh.id) + ": " + cudaGetErrorString(ce);
  }
  res.t_submit = sh.t_submit;
  res.t_admit = sh.t_admit;
  res.t_done = now_s();
  char* mem = sh.mem;
  const size_t mem_bytes = sh.mem_bytes;
  static_assert(PH_IDLE == 0, "a cleared control block is an idle slot's");
  cudaMemsetAsync(b->d_slots + s, 0, sizeof(Slot), b->stream);
  sh = SlotHost{};
  std::lock_guard<std::mutex> lk(b->mu);
  b->arena.release(mem, mem_bytes);
  b->stats.completed += 1;
  if (!copy_error.empty()) b->worker_error = copy_error;
  b->done.push_back(res);
  b->cv.notify_all();
}

void worker_loop(rd_batch* b) {
  cudaStream_t st = b->stream;
  while (true) {
    // admit what fits
    {
      std::unique_lock<std::mutex> lk(b->mu);
      int active = 0;
      for (const SlotHost& sh : b->slots) active += sh.used;
      if (active == 0)
        b->cv.wait(lk, [&] { return b->stop || !b->queue.empty(); });
      if (b->stop) return;  // destroy: running slots are abandoned
      while (!b->queue.empty()) {
        Request q = std::move(b->queue.front());
        b->queue.pop_front();
        lk.unlock();
        rd_status err;
        const bool ok = admit(b, q, &err);
        lk.lock();
        if (!ok) {
          b->queue.push_front(std::move(q));
          break;
        }
        if (err != RD_OK) b->worker_error = rd_last_error();
        b->lists_dirty = true;
      }
    }
    int active = 0;
    for (const SlotHost& sh : b->slots) active += sh.used;
    if (active == 0) {
      std::lock_guard<std::mutex> lk(b->mu);
      if (b->stop && b->queue.empty()) return;
      continue;
    }
    // without its work lists a graph must not run: they may name slots that changed since, or be freed
    if ((b->lists_dirty && rebuild_items(b) != RD_OK) || (b->graph_dirty && rebuild_graph(b) != RD_OK)) {
      b->worker_error = rd_last_error();
      std::lock_guard<std::mutex> lk(b->mu);
      b->stop = true;
      b->cv.notify_all();
      return;
    }
    cudaGraphLaunch(b->gexec, st);
    cudaMemcpyAsync(b->h_slots, b->d_slots, sizeof(Slot) * b->max_slots, cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) {
      b->worker_error = std::string("batch graph: ") + cudaGetErrorString(cudaGetLastError());
      std::lock_guard<std::mutex> lk(b->mu);
      b->stop = true;
      b->cv.notify_all();
      return;
    }
    {
      std::lock_guard<std::mutex> lk(b->mu);
      b->stats.graph_launches += 1;
    }
    int retired = 0, running = 0;
    for (int s = 0; s < b->max_slots; ++s) {
      if (!b->slots[s].used) continue;
      std::vector<double>().swap(b->slots[s].u0);  // the admission's copies have run
      std::vector<float>().swap(b->slots[s].mu);
      const Slot ctl = b->h_slots[s];
      if (ctl.phase == PH_DONE || ctl.phase == PH_FAILED) {
        retire(b, s, ctl);
        ++retired;
      } else {
        ++running;
      }
    }
    // the blocks of a retired slot return at once (its control block is idle), so the lists and the
    // graph, whose capture takes as long as several sweeps, stay until half their slots are gone (or
    // a request is admitted)
    b->stale += retired;
    if (retired && running > 0 && b->stale >= running) b->lists_dirty = true;
  }
}

}  // namespace

extern "C" {

rd_status rd_batch_create(rd_batch** out, size_t hbm_budget_bytes, int max_slots, const rd_opts* opts,
                          void* cuda_stream) {
  if (!out) return bfail(RD_ERR_INVALID_ARG, "out must not be NULL");
  *out = nullptr;
  if (max_slots < 1 || max_slots > 4096) return bfail(RD_ERR_INVALID_ARG, "max_slots must be in [1, 4096]");
  if (hbm_budget_bytes < (1u << 20)) return bfail(RD_ERR_INVALID_ARG, "HBM budget below 1 MiB");
  rd_batch* b = new (std::nothrow) rd_batch();
  if (!b) return bfail(RD_ERR_OOM, "host allocation failed");
  if (opts) b->opts = *opts; else rd_opts_default(&b->opts);
  if (b->opts.graph_k < 1) b->opts.graph_k = 8;
  b->max_slots = max_slots;
  b->budget = hbm_budget_bytes;
  b->stream = static_cast<cudaStream_t>(cuda_stream);
  b->slots.assign(max_slots, SlotHost{});
  auto cleanup = [&](rd_status s) {
    rd_batch_destroy(b);
    return s;
  };
  cudaError_t e;
  if ((e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking)) != cudaSuccess ||
      (e = cudaEventCreateWithFlags(&b->ev_fork, cudaEventDisableTiming)) != cudaSuccess)
    return cleanup(bfail(RD_ERR_CUDA, cudaGetErrorString(e)));
  if ((e = cudaMalloc(&b->arena_mem, hbm_budget_bytes)) != cudaSuccess) {
    cudaGetLastError();
    return cleanup(bfail(RD_ERR_OOM, std::string("arena: ") + cudaGetErrorString(e)));
  }
  b->arena.init(b->arena_mem, hbm_budget_bytes);
  if ((e = cudaMalloc(&b->d_d32, sizeof(Desc) * max_slots)) != cudaSuccess ||
      (e = cudaMalloc(&b->d_d64, sizeof(Desc) * max_slots)) != cudaSuccess ||
      (e = cudaMalloc(&b->d_slots, sizeof(Slot) * max_slots)) != cudaSuccess ||
      (e = cudaMalloc(&b->d_items, sizeof(int2) * max_slots * kBatchSlotItems)) != cudaSuccess ||
      (e = cudaMallocHost(&b->h_items, sizeof(int2) * max_slots * kBatchSlotItems)) != cudaSuccess ||
      (e = cudaMallocHost(&b->h_slots, sizeof(Slot) * max_slots)) != cudaSuccess)
    return cleanup(bfail(RD_ERR_OOM, cudaGetErrorString(e)));
  cudaMemset(b->d_slots, 0, sizeof(Slot) * max_slots);
  // shared memory of the batched sweeps: the largest grid the batch accepts
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int tabs = table_bytes<float>(kBatchMaxSide, true, true);
  b->smem_sweep = std::max(res_smem_bytes<float>(1, kBatchBandRows, 2, kBatchMaxSide, 1, 0, tabs),
                           std::max(lines_smem_bytes<float>((kBatchBandRows + 4) / 2, kBatchMaxSide, 0, tabs),
                                    lines_smem_bytes<float>(kBatchColWidth / 2, kBatchMaxSide, 0, tabs)));
  if ((e = batch_lines2_allow(optin)) != cudaSuccess || (e = batch_lines3_allow(optin)) != cudaSuccess)
    return cleanup(bfail(RD_ERR_CUDA, cudaGetErrorString(e)));
  {
    const rd_status ts = make_tables(b);
    if (ts != RD_OK) return cleanup(ts);
  }
  if ((e = batch3_allow(optin)) != cudaSuccess || (e = allow_small(optin)) != cudaSuccess)
    return cleanup(bfail(RD_ERR_CUDA, cudaGetErrorString(e)));
  b->smem_usable = optin - 1024;
  b->smem_sweep2 = std::max(res_smem_bytes<float>(2, kBatchBandRows, 1, kBatchMaxSide, 0, 0, tabs),
                            lines_smem_bytes<float>(2 * ((kBatchBandRows + 2) / 2), kBatchMaxSide, 0, tabs));
  if ((e = allow_batch_kernels<float, KK_GS>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_SCHNAK>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_NONE_LAP>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_AC>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_CH_IMPL>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_CH_SPLIT>(optin)) != cudaSuccess ||
      (e = allow_batch_kernels<float, KK_NONE_BIH>(optin)) != cudaSuccess)
    return cleanup(bfail(RD_ERR_CUDA, cudaGetErrorString(e)));
  {
    cudaFuncAttributes fa;
    cudaFuncGetAttributes(&fa, k_col_b<float>);
    cudaFuncSetAttribute(k_col_b<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  }
  if ((e = cudaDeviceSynchronize()) != cudaSuccess) return cleanup(bfail(RD_ERR_CUDA, cudaGetErrorString(e)));
  b->worker = std::thread(worker_loop, b);
  *out = b;
  return RD_OK;
}

rd_status rd_batch_submit(rd_batch* b, const rd_request* req, double* u_out_host, uint64_t* id) {
  if (!b || !req || !req->u0_host) return bfail(RD_ERR_INVALID_ARG, "NULL batch, request or u0");
  const rd_request& r = *req;
  if (r.grid.ndim != 2 && r.grid.ndim != 3) return bfail(RD_ERR_UNSUPPORTED, "batch: 2-D and 3-D grids only");
  for (int k = 0; k < r.grid.ndim; ++k) {
    const int n = r.grid.n[k];
    if (r.grid.ndim == 2 && (n < 4 || n > kBatchMaxSide || (n & (n - 1))))
      return bfail(RD_ERR_UNSUPPORTED, "batch: sides must be powers of two in [4, 1024]");
    if (r.grid.ndim == 3 && (n < 4 || n > kBatchMaxSide3 || (n & (n - 1))))
      return bfail(RD_ERR_UNSUPPORTED, "batch: 3-D sides must be powers of two in [4, 512]");
    if (!(r.grid.length[k] > 0)) return bfail(RD_ERR_INVALID_ARG, "lengths must be > 0");
  }
  if (r.bc != RD_BC_PERIODIC && r.bc != RD_BC_NEUMANN) return bfail(RD_ERR_INVALID_ARG, "bad boundary condition");
  if (r.reaction.kind == RD_RX_FCH || r.op == RD_OP_FUNCTIONALIZED)
    return bfail(RD_ERR_UNSUPPORTED, "batch: the sixth-order equation is not batched");
  const bool two = r.reaction.kind == RD_RX_GRAY_SCOTT || r.reaction.kind == RD_RX_SCHNAKENBERG;
  if (group_of(key_of(r)) < 0) return bfail(RD_ERR_UNSUPPORTED, "batch: kind not served");
  if (r.reaction.ncomp != (two ? 2 : 1)) return bfail(RD_ERR_INVALID_ARG, "ncomp does not match the reaction kind");
  if (two && r.grid.ndim == 3) return bfail(RD_ERR_UNSUPPORTED, "batch: 3-D grids are served for the scalar kinds");
  if (two && r.op != RD_OP_LAPLACIAN) return bfail(RD_ERR_INVALID_ARG, "two species need RD_OP_LAPLACIAN");
  if (r.op != RD_OP_LAPLACIAN && r.op != RD_OP_NEG_BIHARMONIC) return bfail(RD_ERR_INVALID_ARG, "bad operator");
  if (r.reaction.kind == RD_RX_ALLEN_CAHN && r.op != RD_OP_LAPLACIAN)
    return bfail(RD_ERR_INVALID_ARG, "Allen-Cahn needs RD_OP_LAPLACIAN");
  if ((r.reaction.kind == RD_RX_CH_IMPLICIT || r.reaction.kind == RD_RX_CH_SPLIT) && r.op != RD_OP_NEG_BIHARMONIC)
    return bfail(RD_ERR_INVALID_ARG, "Cahn-Hilliard needs RD_OP_NEG_BIHARMONIC");
  if (!(r.reaction.a >= 0) || !(r.reaction.b >= 0)) return bfail(RD_ERR_INVALID_ARG, "a and b must be >= 0");
  if (r.tol_kind != RD_TOL_RES_ABS && r.tol_kind != RD_TOL_F_REL) return bfail(RD_ERR_INVALID_ARG, "bad tol_kind");
  if (!(r.dt > 0) || !(r.tau > 0) || !(r.sigma > 0)) return bfail(RD_ERR_INVALID_ARG, "dt, tau, sigma must be > 0");
  if (r.nsteps < 1) return bfail(RD_ERR_INVALID_ARG, "nsteps must be >= 1");
  size_t npts = 0;
  if (slot_bytes(r, &npts) > b->budget) return bfail(RD_ERR_BUSY, "request larger than the whole HBM budget");
  Request q;
  q.req = r;
  q.u0.assign(r.u0_host, r.u0_host + npts);
  q.t_submit = now_s();
  std::lock_guard<std::mutex> lk(b->mu);
  if (b->stop) return bfail(RD_ERR_CUDA, "batch worker stopped: " + b->worker_error);
  q.id = b->next_id++;
  q.req.u0_host = nullptr;
  if (u_out_host) b->outputs[q.id] = u_out_host;
  if (id) *id = q.id;
  b->queue.push_back(std::move(q));
  b->stats.submitted += 1;
  b->cv.notify_all();
  return RD_OK;
}

rd_status rd_batch_poll(rd_batch* b, rd_result* done, int cap, int* n_done, double timeout_s) {
  if (!b || !n_done || (cap > 0 && !done)) return bfail(RD_ERR_INVALID_ARG, "NULL argument");
  *n_done = 0;
  std::unique_lock<std::mutex> lk(b->mu);
  if (timeout_s > 0 && b->done.empty() && !b->stop)
    b->cv.wait_for(lk, std::chrono::duration<double>(timeout_s), [&] { return !b->done.empty() || b->stop; });
  while (*n_done < cap && !b->done.empty()) {
    done[(*n_done)++] = b->done.front();
    b->done.pop_front();
  }
  if (b->stop && !b->worker_error.empty()) return bfail(RD_ERR_CUDA, "batch worker stopped: " + b->worker_error);
  return RD_OK;
}

rd_status rd_batch_get_stats(rd_batch* b, rd_batch_stats* out) {
  if (!b || !out) return bfail(RD_ERR_INVALID_ARG, "NULL argument");
  std::lock_guard<std::mutex> lk(b->mu);
  *out = b->stats;
  out->queued = (long long)b->queue.size();
  size_t fr = 0;
  for (auto& kv : b->arena.free_) fr += kv.second;
  out->arena_free_bytes = (long long)fr;
  return RD_OK;
}

void rd_batch_destroy(rd_batch* b) {
  if (!b) return;
  if (b->worker.joinable()) {
    {
      std::lock_guard<std::mutex> lk(b->mu);
      b->stop = true;
      b->queue.clear();
      b->cv.notify_all();
    }
    b->worker.join();
  }
  cudaStreamSynchronize(b->stream);  // (NULL: the legacy default stream, whose copies read the slots' memory too)
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->d_items) cudaFree(b->d_items);
  if (b->h_items) cudaFreeHost(b->h_items);
  if (b->d_tables) cudaFree(b->d_tables);
  if (b->d_d32) cudaFree(b->d_d32);
  if (b->d_d64) cudaFree(b->d_d64);
  if (b->d_slots) cudaFree(b->d_slots);
  if (b->h_slots) cudaFreeHost(b->h_slots);
  if (b->arena_mem) cudaFree(b->arena_mem);
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
  for (cudaStream_t s : b->branch_stream)
    if (s) cudaStreamDestroy(s);
  for (cudaEvent_t ev : b->ev_join)
    if (ev) cudaEventDestroy(ev);
  if (b->ev_fork) cudaEventDestroy(b->ev_fork);
  delete b;
}

}  // extern "C"
