// Sweep kernels of one G-prox PDHG iteration (arxiv 2305.03945, Section 2.1, Algorithm 1) on 2-D
// grids, on the register-resident line transforms of rd_fft.cuh:
//
//   k_fcol    (column blocks) forward column transform of the row spectrum along y, multiplication
//             by 1/g_hat, inverse column transform, in place in WY;
//   k_dual    (row pairs)     inverse row transform of Y = G^{-1} W, P_{n+1} = P_n + tau_p Y in
//             place, P~ = P_n + (1 + omega) tau_p Y to its own array (eqs. G-prox dynamic 1-2);
//   k_primal  (row bands)     U_{n+1} = U_n - tau_u dF(U_n)^T P~ (eq. G-prox dynamic 3), then on the
//             same band W = F(U_{n+1}), its norm partials and stopping decision, and the forward
//             row transform of W into WY.
//
// k_primal without an update (`first`) starts a solve.  The order (column, dual, primal with the
// next residual) puts the only halo on the primal update, whose recomputation on 2H rows is a
// stencil; k_upd and the former fused kernel recomputed the inverse row transform on them.
// k_rowfwd is the forward row transform alone (preconditioner-only solve).
#pragma once

#include <cuda.h>

#include <type_traits>

#include "rd_fft.cuh"
#include "rd_sweep.cuh"

namespace rd {

// the spectral symbol 1 / (g_hat nx ny), g_hat = (1 + c1 mu + c2 mu^2 + c3 mu^3)^2
template <class T>
struct Symbol {
  T c1, c2, c3, inn;
  __device__ __forceinline__ Symbol(const Desc& d, int c)
      : c1(T(d.gc1[c])), c2(T(d.gc2[c])), c3(T(d.gc3[c])), inn(T(d.inv_nn)) {}
  __device__ __forceinline__ T operator()(T mu) const {
    const T g = T(1) + mu * (c1 + mu * (c2 + c3 * mu));
    if constexpr (sizeof(T) == 4) return inn * __frcp_rn(g * g);
    else return inn / (g * g);
  }
};

// Spectral scaling of a pair of real columns (a, b) with the symbols of their own frequencies, on
// the paired middle order v (see rf_pair).  sym(k, sa, sb): the symbols of the two columns at
// frequency k of the line.  Periodic: with A = (Z + conj Z')/2 and iB = (Z - conj Z')/2 the scaled
// spectrum is sa A + sb iB = (sa + sb)/2 Z + (sa - sb)/2 conj Z', and the symbols are even in k.
// Neumann: the DCT-II coefficients, scaled, and back.
template <class T, int N, int V, class Sym>
__device__ __forceinline__ void scale_pairs(cx<T>* v, int t, bool per, const Sym& sym, const cx<T>* __restrict__ dc) {
  auto one = [&](int k, cx<T> z, cx<T> zp, cx<T>& o, cx<T>& op) {
    T sa, sb;
    sym(k, sa, sb);
    if (per) {
      const T sp = T(0.5) * (sa + sb), sm = T(0.5) * (sa - sb);
      o = cx<T>{sp * z.x + sm * zp.x, sp * z.y - sm * zp.y};
      op = cx<T>{sp * zp.x + sm * z.x, sp * zp.y - sm * z.y};
    } else {
      const cx<T> w = ldg(dc + k);
      cx<T> h, hp;
      pair_fwd(false, z, zp, w, h, hp);
      T ta, tb;
      sym(k == 0 ? 0 : N - k, ta, tb);
      h = cx<T>{h.x * sa, h.y * sb};
      hp = k == 0 ? cx<T>{T(0), T(0)} : cx<T>{hp.x * ta, hp.y * tb};
      pair_inv(false, h, hp, w, o, op);
    }
  };
  rf_pair<T, V>(v, t);
  cx<T> v0 = v[0], vm = v[V - 1];
#pragma unroll
  for (int i = 1; i < V / 2; ++i) {
    cx<T> o, op;
    one(rf_freq<V>(N, t, i), v[i], v[V - 1 - i], o, op);
    v[i] = o;
    v[V - 1 - i] = op;
  }
  cx<T> o, op;
  if (t == 0) {
    one(0, v0, v0, o, op);
    v[0] = o;
    one(N / 2, vm, vm, o, op);
    v[V - 1] = o;
  } else {
    one(rf_freq<V>(N, t, 0), v0, vm, o, op);
    v[0] = o;
    v[V - 1] = op;
  }
  rf_unpair<T, V>(v, t);
}

// The symbols of the columns with eigenvalues ma, mb from the line axis' eigenvalues mul.
template <class T>
struct SymMu {
  Symbol<T> s;
  const T* __restrict__ mul;
  T ma, mb;
  __device__ __forceinline__ void operator()(int k, T& sa, T& sb) const {
    const T m = __ldg(mul + k);
    sa = s(ma + m);
    sb = s(mb + m);
  }
};
// The same from a table (FP64, whose division and polynomial would take a sixth of the kernel's FP64
// operations): p points at the pair of columns in row 0, rs elements per row.
template <class T>
struct SymTab {
  const T* __restrict__ p;
  size_t rs;
  __device__ __forceinline__ void operator()(int k, T& sa, T& sb) const {
    const cx<T> v = ldg(reinterpret_cast<const cx<T>*>(p + (size_t)k * rs));
    sa = v.x;
    sb = v.y;
  }
};

// fills the table of one descriptor: [ncomp][ny][nx]
static __global__ void __launch_bounds__(256) k_symbol(const __grid_constant__ Desc d, double* __restrict__ out) {
  const size_t plane = (size_t)d.nx * d.ny;
  for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < plane * d.ncomp; q += (size_t)gridDim.x * blockDim.x) {
    const int c = q >= plane ? 1 : 0;
    const size_t r = q - c * plane;
    out[q] = Symbol<double>(d, c)(static_cast<const double*>(d.mux)[r & (size_t)(d.nx - 1)] +
                                  static_cast<const double*>(d.muy)[r >> d.lognx]);
  }
}

// ---------------------------------------------------------------------------------------
// k_fcol
// ---------------------------------------------------------------------------------------
template <class T, int LOGN, int V, bool PER>
__device__ __forceinline__ void fcol_body(const Desc& d, int blk, unsigned char* smem_raw) {
  using F = Rf<LOGN, V>;
  using P1 = Pass<T, LOGN, V, true, 1>;
  constexpr int N = F::N;
  const int nx = d.nx;
  const int c = blk / d.ncolblk, cb = blk - c * d.ncolblk;
  const int nl = d.col_width >> 1, lnl = ilog2i(nl);
  const int m = threadIdx.x & (nl - 1), t = threadIdx.x >> lnl;
  const int col = cb * d.col_width + 2 * m;
  constexpr bool per = PER;
  cx<T>* G = reinterpret_cast<cx<T>*>(static_cast<T*>(d.WY) + (size_t)c * nx * N + col);
  const size_t rs = (size_t)(nx >> 1);  // row stride in pairs
  cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw) + m;
  const cx<T>* tw = static_cast<const cx<T>*>(d.twy);
  cx<T> v[V];
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int n = P1::natural(t, e);
    v[e] = G[(size_t)(per ? n : mk_perm(n, N)) * rs];
  }
  auto sync = [] { __syncthreads(); };
  rf_forward<T, LOGN, V, true>(v, buf, nl, tw, t, sync);
  const cx<T>* dc = static_cast<const cx<T>*>(d.dcy);
  if constexpr (sizeof(T) == 8) {
    scale_pairs<T, N, V>(v, t, per, SymTab<T>{static_cast<const T*>(d.scale) + (size_t)c * nx * N + col, (size_t)nx}, dc);
  } else {
    const T* mux = static_cast<const T*>(d.mux);
    scale_pairs<T, N, V>(v, t, per, SymMu<T>{Symbol<T>(d, c), static_cast<const T*>(d.muy), __ldg(mux + col), __ldg(mux + col + 1)}, dc);
  }
  rf_inverse<T, LOGN, V, true>(v, buf, nl, tw, t, sync);
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int n = P1::natural(t, e);
    G[(size_t)(per ? n : mk_perm(n, N)) * rs] = v[e];
  }
}

// Threads of a block at most: 128 registers per thread; FP64 at V = 16 holds 64 in its values alone
// and takes up to 255 (the same rule as band_threads_max).
template <class T, int V>
struct BandThreads { static constexpr int value = sizeof(T) == 8 && V == 16 ? 256 : 512; };
// of k_fcol: FP32 lines of 4096 and 8192 points take 1024 threads to hold two lines or more; at 64
// registers these and the 2048-point ones spill 160 to 240 bytes (k_fcol_tma 50 to 130)
template <class T, int LOGN, int V>
struct ColThreads {
  static constexpr int value = LOGN >= 12 && sizeof(T) == 4 ? 1024 : BandThreads<T, V>::value;
  static constexpr int blocks = sizeof(T) == 4 && V == 16 && LOGN == 11 ? 2 : 1;
};

// st = nullptr: the preconditioner alone, whatever the solve's state
template <class T, int LOGN, int V, bool PER>
__global__ void __launch_bounds__(ColThreads<T, LOGN, V>::value, ColThreads<T, LOGN, V>::blocks) k_fcol(const __grid_constant__ Desc d, State* __restrict__ st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  if (st && !sweep_active(st, nullptr)) return;
  fcol_body<T, LOGN, V, PER>(d, blockIdx.x, smem_raw);
}

// ---------------------------------------------------------------------------------------
// k_fcol_tma: k_fcol<float> at V = 16 on lines of 2048 points and more, whose tile of narrow row segments
// TMA moves between global and shared memory: by threads, a warp's load or store of such a tile is 8 or 16
// separate requests, and their issue was the kernel's first stall (lg_throttle).  Measured, k_fcol ->
// k_fcol_tma: 2048^2 x 2 (32-byte segments) 50 -> 37 us, 1.8 TB/s; 8192^2 (16-byte segments) 578 -> 394 us,
// 1.4 TB/s.  On 1024^2, a block or two per SM, it was slower (step 0.749 -> 0.785 ms): the tile's way
// through shared memory has nothing to hide behind.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Waits for phase 0 of a transaction barrier, with a bound (false: it ran out).
__device__ __forceinline__ bool mbar_wait0(unsigned bar) {
  for (int i = 0; i < (1 << 20); ++i) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar)
        : "memory");
    if (done) return true;
  }
  return false;
}

constexpr int kTmaRows = 256;  // rows of one TMA box (the largest)

template <int LOGN>
struct TmaCol {
  static constexpr int threads = LOGN >= 12 ? 1024 : 512;
  static constexpr int blocks = LOGN >= 12 ? 1 : 2;
};

template <int LOGN, bool PER>
__global__ void __launch_bounds__(TmaCol<LOGN>::threads, TmaCol<LOGN>::blocks)
    k_fcol_tma(const __grid_constant__ Desc d, State* __restrict__ st, const __grid_constant__ CUtensorMap map) {
  constexpr int V = 16;
  using F = Rf<LOGN, V>;
  using P1 = Pass<float, LOGN, V, true, 1>;
  constexpr int N = F::N;
  extern __shared__ __align__(128) unsigned char smem_tma[];
  __shared__ __align__(8) unsigned long long bar;
  pdl_wait();
  if (!sweep_active(st, nullptr)) return;
  const int nl = d.col_width >> 1, lnl = ilog2i(nl);
  const int m = threadIdx.x & (nl - 1), t = threadIdx.x >> lnl;
  const int c = blockIdx.x / d.ncolblk, x0 = (blockIdx.x - c * d.ncolblk) * d.col_width;
  const int col = x0 + 2 * m;
  const unsigned mb = smem_u32(&bar), box = kTmaRows * d.col_width * 4;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"((unsigned)(N / kTmaRows) * box) : "memory");
    for (int k = 0; k < N / kTmaRows; ++k)
      asm volatile(
          "cp.async.bulk.tensor.2d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
              smem_u32(smem_tma) + k * box),
          "l"(&map), "r"(x0), "r"(c * N + k * kTmaRows), "r"(mb)
          : "memory");
  }
  __syncthreads();  // the barrier is initialised
  cx<float>* buf = reinterpret_cast<cx<float>*>(smem_tma) + m;
  const bool here = mbar_wait0(mb);
  cx<float> v[V];
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int n = P1::natural(t, e);
    v[e] = buf[(PER ? n : mk_perm(n, N)) * nl];
  }
  // The wait cannot run out while the memory system works.  One thread's is the block's: all stop, the tile
  // stays as it was and the solve ends with an error.
  if (!__syncthreads_and(here)) {
    if (threadIdx.x == 0) st->status = ST_FAULT;
    mbar_wait0(mb);  // (the copies in flight write this block's shared memory)
    return;
  }
  auto sync = [] { __syncthreads(); };
  const cx<float>* tw = static_cast<const cx<float>*>(d.twy);
  rf_forward<float, LOGN, V, true>(v, buf, nl, tw, t, sync);
  const float* mux = static_cast<const float*>(d.mux);
  scale_pairs<float, N, V>(
      v, t, PER, SymMu<float>{Symbol<float>(d, c), static_cast<const float*>(d.muy), __ldg(mux + col), __ldg(mux + col + 1)},
      static_cast<const cx<float>*>(d.dcy));
  rf_inverse<float, LOGN, V, true>(v, buf, nl, tw, t, sync);
  sync();
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int n = P1::natural(t, e);
    buf[(PER ? n : mk_perm(n, N)) * nl] = v[e];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < N / kTmaRows; ++k)
      asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(&map), "r"(x0),
                   "r"(c * N + k * kTmaRows), "r"(smem_u32(smem_tma) + k * box)
                   : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
}

// ---------------------------------------------------------------------------------------
// rows: shared pieces
// ---------------------------------------------------------------------------------------

// four adjacent values
template <class T>
__device__ __forceinline__ void ld4(const T* __restrict__ p, T* v) {
  vld<T, V16<T>::n>(p, v);
  if constexpr (sizeof(T) == 8) vld<T, 2>(p + 2, v + 2);
}
template <class T>
__device__ __forceinline__ void st4(T* __restrict__ p, const T* v) {
  vst<T, V16<T>::n>(p, v);
  if constexpr (sizeof(T) == 8) vst<T, 2>(p + 2, v + 2);
}

// A pair of rows (a, b) at columns j0 .. j0+3 to / from the line buffer's natural order (pass-1
// input of the forward transform): column j at entry j (periodic) or at its Makhoul slot.
template <class T>
__device__ __forceinline__ void put4(cx<T>* line, int N, bool per, int j0, const T* a, const T* b) {
  if (per) {
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
      T w[4] = {a[q], b[q], a[q + 1], b[q + 1]};
      st4(reinterpret_cast<T*>(line + j0 + q), w);
    }
  } else {
    T w[4] = {a[0], b[0], a[2], b[2]};
    st4(reinterpret_cast<T*>(line + (j0 >> 1)), w);
    T u[4] = {a[3], b[3], a[1], b[1]};
    st4(reinterpret_cast<T*>(line + (N - 2 - (j0 >> 1))), u);
  }
}
template <class T>
__device__ __forceinline__ void get4(const cx<T>* line, int N, bool per, int j0, T* a, T* b) {
  T w[4], u[4];
  if (per) {
    ld4(reinterpret_cast<const T*>(line + j0), w);
    ld4(reinterpret_cast<const T*>(line + j0 + 2), u);
    a[0] = w[0], b[0] = w[1], a[1] = w[2], b[1] = w[3];
    a[2] = u[0], b[2] = u[1], a[3] = u[2], b[3] = u[3];
  } else {
    ld4(reinterpret_cast<const T*>(line + (j0 >> 1)), w);
    ld4(reinterpret_cast<const T*>(line + (N - 2 - (j0 >> 1))), u);
    a[0] = w[0], b[0] = w[1], a[2] = w[2], b[2] = w[3];
    a[3] = u[0], b[3] = u[1], a[1] = u[2], b[1] = u[3];
  }
}

// Forward row transform of one pair line held in `line` in natural order, coefficients to the two
// rows Wa, Wa + nx.  Called by the TPL threads of the line; the line buffer is overwritten.
template <class T, int LOGN, int V, class Sync>
__device__ __forceinline__ void row_forward(const Desc& d, cx<T>* line, T* __restrict__ Wa, int t, bool live, Sync sync) {
  using F = Rf<LOGN, V>;
  using P1 = Pass<T, LOGN, V, false, 1>;
  constexpr int N = F::N;
  const bool per = d.bc == BC_PERIODIC;
  cx<T> v[V];
#pragma unroll
  for (int e = 0; e < V; ++e) v[e] = line[P1::natural(t, e)];
  sync();  // the exchange layout differs from the natural order
  rf_forward<T, LOGN, V, false>(v, line, 1, static_cast<const cx<T>*>(d.twx), t, sync);
  rf_pair<T, V>(v, t);
  const cx<T>* dc = static_cast<const cx<T>*>(d.dcx);
  T* __restrict__ Wb = Wa + N;
  if (!live) return;
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const int k = rf_freq<V>(N, t, i);
    const cx<T> w = per ? cx<T>{T(0), T(0)} : ldg(dc + k);
    cx<T> o, op;
    if (i == 0 && t == 0) {
      cx<T> skip;
      pair_fwd(per, v[0], v[0], w, o, skip);
      pair_fwd(per, v[V - 1], v[V - 1], per ? w : ldg(dc + N / 2), op, skip);
      Wa[0] = o.x;
      Wb[0] = o.y;
      Wa[N / 2] = op.x;
      Wb[N / 2] = op.y;
    } else {
      pair_fwd(per, v[i], v[V - 1 - i], w, o, op);
      Wa[k] = o.x;
      Wb[k] = o.y;
      Wa[N - k] = op.x;
      Wb[N - k] = op.y;
    }
  }
}

// Inverse row transform of the rows Wa, Wa + nx into `line` in natural order (see put4 / get4),
// complete when the caller has passed a barrier of the line's threads.
template <class T, int LOGN, int V, class Sync>
__device__ __forceinline__ void row_inverse(const Desc& d, const T* Wa, cx<T>* line, int t, Sync sync) {
  using F = Rf<LOGN, V>;
  using P1 = Pass<T, LOGN, V, false, 1>;
  constexpr int N = F::N;
  const bool per = d.bc == BC_PERIODIC;
  const cx<T>* dc = static_cast<const cx<T>*>(d.dcx);
  const T* Wb = Wa + N;
  cx<T> v[V];
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const int k = rf_freq<V>(N, t, i);
    const int kp = i == 0 && t == 0 ? N / 2 : N - k;
    v[i] = cx<T>{Wa[k], Wb[k]};
    v[V - 1 - i] = cx<T>{Wa[kp], Wb[kp]};
  }
#pragma unroll
  for (int i = 0; i < V / 2; ++i) {
    const int k = rf_freq<V>(N, t, i);
    const cx<T> w = per ? cx<T>{T(0), T(0)} : ldg(dc + k);
    cx<T> z, zp;
    if (i == 0 && t == 0) {
      cx<T> skip;
      pair_inv(per, v[0], per ? v[0] : cx<T>{T(0), T(0)}, w, z, skip);
      pair_inv(per, v[V - 1], v[V - 1], per ? w : ldg(dc + N / 2), zp, skip);
    } else {
      pair_inv(per, v[i], v[V - 1 - i], w, z, zp);
    }
    v[i] = z;
    v[V - 1 - i] = zp;
  }
  rf_unpair<T, V>(v, t);
  rf_inverse<T, LOGN, V, false>(v, line, 1, static_cast<const cx<T>*>(d.twx), t, sync);
  sync();  // the exchange layout differs from the natural order
#pragma unroll
  for (int e = 0; e < V; ++e) line[P1::natural(t, e)] = v[e];
}

// ---------------------------------------------------------------------------------------
// k_rowfwd: forward row transform of X into WY (preconditioner-only solve)
// ---------------------------------------------------------------------------------------
template <class T, int LOGN, int V>
__global__ void __launch_bounds__(BandThreads<T, V>::value) k_rowfwd(const __grid_constant__ Desc d) {
  using F = Rf<LOGN, V>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  constexpr int N = F::N;
  const int lline = threadIdx.x / F::TPL, t = threadIdx.x % F::TPL;
  const int lines = d.ncomp * (d.ny >> 1);
  const int gl = blockIdx.x * (blockDim.x / F::TPL) + lline;
  const bool live = gl < lines;
  cx<T>* line = reinterpret_cast<cx<T>*>(smem_raw) + lline * Lay<T, LOGN, V, false>::len;
  const bool per = d.bc == BC_PERIODIC;
  const size_t o = (size_t)(live ? gl : 0) * 2 * N;  // rows 2 gl, 2 gl + 1 of the stacked components
  const T* X = static_cast<const T*>(d.X) + o;
#pragma unroll
  for (int i = 0; i < V / 4; ++i) {
    const int j0 = 4 * (t + i * F::TPL);
    T a[4], b[4];
    ld4(X + j0, a);
    ld4(X + N + j0, b);
    put4(line, N, per, j0, a, b);
  }
  auto sync = [lline] { line_sync<F::TPL>(lline); };
  sync();
  row_forward<T, LOGN, V>(d, line, static_cast<T*>(d.WY) + o, t, live, sync);
}

// ---------------------------------------------------------------------------------------
// k_dual
// ---------------------------------------------------------------------------------------
// The lines of group `grp` (blockDim.x / TPL row pairs of the stacked components and planes).  P~ may
// overwrite Y (d.P[1] = d.WY): a line's coefficients are all read before its first store.
template <class T, int LOGN, int V, bool PC>
__device__ __forceinline__ void dual_body(const Desc& d, int grp, unsigned char* smem_raw) {
  using F = Rf<LOGN, V>;
  constexpr int N = F::N;
  const int lline = threadIdx.x / F::TPL, t = threadIdx.x % F::TPL;
  const int lines = d.ncomp * (d.ny >> 1) * (d.nz > 1 ? d.nz : 1);
  const int gl = grp * (blockDim.x / F::TPL) + lline;
  const bool live = gl < lines;
  cx<T>* line = reinterpret_cast<cx<T>*>(smem_raw) + lline * Lay<T, LOGN, V, false>::len;
  const bool per = d.bc == BC_PERIODIC;
  const size_t o = (size_t)(live ? gl : 0) * 2 * N;
  auto sync = [lline] { line_sync<F::TPL>(lline); };
  row_inverse<T, LOGN, V>(d, static_cast<const T*>(d.WY) + o, line, t, sync);
  sync();
  if (!live) return;
  if constexpr (PC) {
    T* X = static_cast<T*>(d.X) + o;
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
      const int j0 = 4 * (t + i * F::TPL);
      T a[4], b[4];
      get4(line, N, per, j0, a, b);
      st4(X + j0, a);
      st4(X + N + j0, b);
    }
  } else {
    T* P = static_cast<T*>(d.P[0]) + o;
    T* Pt = static_cast<T*>(d.P[1]) + o;
    const T tp = T(d.tau_p), tpe = T((1.0 + d.omega) * d.tau_p);
    T pa[V / 4][4], pb[V / 4][4];
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
      const int j0 = 4 * (t + i * F::TPL);
      ld4(P + j0, pa[i]);
      ld4(P + N + j0, pb[i]);
    }
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
      const int j0 = 4 * (t + i * F::TPL);
      T ya[4], yb[4], na[4], nb[4];
      get4(line, N, per, j0, ya, yb);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        na[q] = pa[i][q] + tp * ya[q];
        nb[q] = pb[i][q] + tp * yb[q];
        pa[i][q] += tpe * ya[q];
        pb[i][q] += tpe * yb[q];
      }
      st4(P + j0, na);
      st4(P + N + j0, nb);
      st4(Pt + j0, pa[i]);
      st4(Pt + N + j0, pb[i]);
    }
  }
}

template <class T, int LOGN, int V, bool PC>
__global__ void __launch_bounds__(BandThreads<T, V>::value) k_dual(const __grid_constant__ Desc d, State* __restrict__ st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  if (!PC && !sweep_active(st, nullptr)) return;
  dual_body<T, LOGN, V, PC>(d, blockIdx.x, smem_raw);
}

// ---------------------------------------------------------------------------------------
// k_primal
// ---------------------------------------------------------------------------------------

// Values of a field around four adjacent points (rows -H..H, columns -H..3+H), as the accessor
// the pointwise formulas of rd_sweep.cuh take; entries no stencil of radius H reads stay unset.
template <class T, int H>
struct Patch {
  T v[2 * H + 1][4 + 2 * H];
  __device__ __forceinline__ T operator()(int i, int j) const { return v[i + H][j + H]; }
  // rows[H + di]: row di of the field, boundary-mapped
  __device__ __forceinline__ void load(const T* const* rows, int j0, int nx, bool per) {
    int jl[2], jr[2];
    jl[0] = j0 > 0 ? j0 - 1 : (per ? nx - 1 : 0);
    jr[0] = j0 + 4 < nx ? j0 + 4 : (per ? 0 : nx - 1);
    if constexpr (H > 1) {
      jl[1] = j0 > 0 ? j0 - 2 : (per ? nx - 2 : 1);
      jr[1] = j0 + 4 < nx ? j0 + 5 : (per ? 1 : nx - 2);
    }
#pragma unroll
    for (int di = -H; di <= H; ++di) {
      const T* r = rows[H + di];
      ld4(r + j0, &v[H + di][H]);
      const int side = H - (di < 0 ? -di : di);  // columns the stencil reads beyond the four
#pragma unroll
      for (int s = 0; s < H; ++s)
        if (s < side) {
          v[H + di][H - 1 - s] = r[jl[s]];
          v[H + di][H + 4 + s] = r[jr[s]];
        }
    }
  }
};

// the base state at the four points, for kinds whose residual reads it there only
template <class T>
struct Pt4 {
  T v[4];
  __device__ __forceinline__ T operator()(int, int j) const { return v[j]; }
};

template <int K>
__host__ __device__ constexpr int ncomp_of() { return KT<K>::two ? 2 : 1; }

// Bytes of a k_primal block's table of row offsets, (rows + 2H)(2H + 1) of them: whole 16-byte vectors, since
// what lies behind it is read and written in such.
__host__ __device__ constexpr int primal_table_bytes(int rows, int H) {
  return ((rows + 2 * H) * (2 * H + 1) * (int)sizeof(int) + 15) / 16 * 16;
}

// Shared-memory bytes of a k_primal block: the table, and behind it the band's rows of U with H halo rows,
// whose place the line buffers of the forward transform take afterwards.
template <class T>
__host__ __device__ inline int primal_smem_bytes(int nc, int rows, int H, int nx, int line_len, int line_bufs) {
  const int u = nc * (rows + 2 * H) * nx * (int)sizeof(T);
  const int l = line_bufs * line_len * (int)sizeof(cx<T>);
  return primal_table_bytes(rows, H) + (u > l ? u : l);
}

// Threads of a k_primal block at most, and the blocks an SM shall hold (the register cap).  FP32 lines of
// 2048 points and more: 1024 threads, 64 registers (two species spill 20 to 40 bytes): two blocks of four rows
// or one of eight per SM; but 512 threads at 128 registers for Cahn-Hilliard, whose thirteen-point stencils of d and
// u spill 240 to 380 bytes at 64 (steps at 64 / 128 registers: split 2048^2 6.20 / 5.36 ms, 4096^2 22.3 / 21.2 ms, 256 x 4096
// 2.44 / 2.40 ms; implicit 2048^2 5.97 / 5.13 ms; the biharmonic alone, which does not spill, 3.85 / 4.01 ms).  FP32
// five-point kinds at V = 16 on shorter lines: two blocks of 512.  (primal_wide: the same rule for the planner.)
inline bool primal_wide(const Desc& d, int H, int elem, int vals) {
  return elem == 4 && vals == 16 && d.nx >= 2048 && !(H == 2 && d.kind != RX_NONE);
}
template <class T, int K, int LOGN, int V>
struct PrimalBlock {
  static constexpr bool wide = sizeof(T) == 4 && V == 16 && LOGN >= 11 && !(KT<K>::biharm && KT<K>::nonlinear);
  static constexpr int threads = wide ? 1024 : BandThreads<T, V>::value;
  static constexpr int blocks = sizeof(T) == 4 && V == 16 && !wide && !KT<K>::biharm ? 2 : 1;
};

template <class T, int K, int LOGN, int V>
__device__ __forceinline__ void primal_body(const Desc& d, State* __restrict__ st, int band, bool first,
                                            unsigned char* smem_raw) {
  using F = Rf<LOGN, V>;
  constexpr int N = F::N;
  constexpr int H = KT<K>::H;
  constexpr int NC = ncomp_of<K>();
  constexpr bool DC = sizeof(T) == 4;
  constexpr bool BASE = DC && KT<K>::nonlinear;
  constexpr int HB = base_stencil<K>() ? 1 : 0;  // the residual's reach on the base state
  __shared__ double red[32];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ny = d.ny, bc = d.bc;
  const bool per = bc == BC_PERIODIC;
  const size_t plane = (size_t)N * ny;
  const int B = d.upd_rows;
  const int y0 = band * B;
  const int rows = min(B, ny - y0);
  const int srows = rows + 2 * H;
  // offsets of the rows the stencils of every staged row read, boundary-mapped (a row beyond a wall is
  // updated exactly as the row it maps to, by that row's neighbours); mapped per group of four points they
  // cost 7% of the kernel's instructions (steps: 1024 x 128 805 -> 782 us, 512^2 716 -> 705 us)
  int* roff = reinterpret_cast<int*>(smem_raw);
  T* us = reinterpret_cast<T*>(smem_raw + primal_table_bytes(rows, H));
  for (int k = tid; k < srows * (2 * H + 1); k += nt) {
    const int r = k / (2 * H + 1), di = k - r * (2 * H + 1) - H;
    roff[k] = bcmap(bcmap(y0 + r - H, ny, bc) + di, ny, bc) << LOGN;
  }
  T* X = static_cast<T*>(d.X);
  T* Hb = static_cast<T*>(d.halo) + (size_t)band * NC * 2 * H * N;
  const T* Bs = static_cast<const T*>(d.base);
  const T* Pt = static_cast<const T*>(d.P[1]);
  constexpr int LV = LOGN - 2;  // log2 of the four-point groups of a row

  // 1. U_{n+1} on the band and its halo rows: band rows in place in X, halo rows in this block's
  //    own copy (rows that other blocks update), all rows staged in shared memory.  `first`: U_0.
  const T tu = T(d.tau_u);
  __syncthreads();
  for (int g = tid; g < (srows << LV); g += nt) {
    const int r = (g >> LV) - H, j0 = (g & ((1 << LV) - 1)) * 4;
    const bool own = r >= 0 && r < rows;
    const int* ro = roff + (r + H) * (2 * H + 1);
    const int at = ro[H] + j0;
    T* u[2];
    const int slot = r < 0 ? r + H : r - rows + H;
    const int hat = (slot << LOGN) + j0;
    u[0] = own || first ? X + at : Hb + hat;
    u[1] = own || first ? u[0] + plane : Hb + (2 * H << LOGN) + hat;
    T x[2][4];
#pragma unroll
    for (int c = 0; c < NC; ++c) ld4(u[c], x[c]);
    if (!first) {
      T s[2][4] = {};
      if constexpr (BASE)
#pragma unroll
        for (int c = 0; c < NC; ++c) ld4(Bs + c * plane + at, s[c]);
      Patch<T, H> p[NC];
      const T* rp[2 * H + 1];
#pragma unroll
      for (int di = 0; di <= 2 * H; ++di) rp[di] = Pt + ro[di];
      p[0].load(rp, j0, N, per);
      if constexpr (NC == 2) {
#pragma unroll
        for (int di = 0; di <= 2 * H; ++di) rp[di] += plane;
        p[NC - 1].load(rp, j0, N, per);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        T g2[2] = {T(0), T(0)};
        gradT_pt<T, K>(d, p[0], p[NC - 1], x[0][q] + s[0][q], NC == 2 ? x[1][q] + s[1][q] : T(0), 0, q, g2);
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c][q] -= tu * g2[c];
      }
    }
    if (!own) {
      u[0] = Hb + hat;
      u[1] = Hb + (2 * H << LOGN) + hat;
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (!first || !own) st4(u[c], x[c]);
      st4(us + ((c * srows + r + H) << LOGN) + j0, x[c]);
    }
  }
  __syncthreads();

  // 2. W = F(U_{n+1}) on the band, two rows by four columns at a time; the values stay in registers
  //    until every read of the staged rows is done (the line buffers share their memory)
  constexpr int MI = V / 4 / NC > 0 ? V / 4 / NC : 1;  // groups per thread at most (a thread per V values of a line)
  const int groups = (rows >> 1) << LV;
  T w[MI][NC][2][4];
#pragma unroll
  for (int m = 0; m < MI; ++m) {
    const int g = tid + m * nt;
    if (g < groups) {
      const int r = 2 * (g >> LV), j0 = (g & ((1 << LV) - 1)) * 4;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int* ro = roff + (r + h + H) * (2 * H + 1);
        const int at = ro[H] + j0;
        T rr[2][4];
#pragma unroll
        for (int c = 0; c < NC; ++c) ld4(static_cast<const T*>(d.rhs) + c * plane + at, rr[c]);
        Patch<T, H> x[NC];
        const T* rp[2 * H + 1];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
#pragma unroll
          for (int di = -H; di <= H; ++di) rp[H + di] = us + ((c * srows + r + h + H + di) << LOGN);
          x[c].load(rp, j0, N, per);
        }
        auto points = [&](const auto& b0, const auto& b1) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            T ww[2] = {T(0), T(0)};
            residual_pt<T, K, DC>(d, x[0], x[NC - 1], b0, b1, 0, q, rr[0][q], NC == 2 ? rr[1][q] : T(0), ww);
#pragma unroll
            for (int c = 0; c < NC; ++c) w[m][c][h][q] = ww[c];
          }
        };
        if constexpr (BASE && HB > 0) {
          Patch<T, 1> b;
          const T* bp[3];
#pragma unroll
          for (int di = -1; di <= 1; ++di) bp[1 + di] = Bs + ro[H + di];
          b.load(bp, j0, N, per);
          points(b, b);
        } else if constexpr (BASE) {
          Pt4<T> b[NC];
#pragma unroll
          for (int c = 0; c < NC; ++c) ld4(Bs + c * plane + at, b[c].v);
          points(b[0], b[NC - 1]);
        } else {
          points(x[0], x[NC - 1]);
        }
      }
    }
  }
  __syncthreads();
  cx<T>* lines = reinterpret_cast<cx<T>*>(us);
  constexpr int LEN = Lay<T, LOGN, V, false>::len;
  const int hr = rows >> 1;
  SumSq<T> acc[NC];  // (summed here, not beside the stencils that need the registers)
#pragma unroll
  for (int m = 0; m < MI; ++m) {
    const int g = tid + m * nt;
    if (g < groups) {
      const int pr = g >> LV, j0 = (g & ((1 << LV) - 1)) * 4;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        put4(lines + (c * hr + pr) * LEN, N, per, j0, w[m][c][0], w[m][c][1]);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[c].add(w[m][c][q >> 2][q & 3]);
      }
    }
  }
  __syncthreads();

  // 3. forward row transform, one line per TPL threads (whole warps: a short line's spare threads
  //    run on a spare line buffer)
  const int nlines = NC * hr;
  const int lline = tid / F::TPL, t = tid % F::TPL;
  if ((tid & ~31) < nlines * F::TPL) {
    const bool live = lline < nlines;
    const int c = NC == 2 && lline >= hr ? 1 : 0, pr = lline - c * hr;
    T* Wa = static_cast<T*>(d.WY) + c * plane + (size_t)(y0 + 2 * pr) * N;
    auto sync = [lline] { line_sync<F::TPL>(lline); };
    row_forward<T, LOGN, V>(d, lines + lline * LEN, live ? Wa : nullptr, t, live, sync);
  }

  // 4. partial norms, ticket, stopping decision in the last block
  const double s0 = block_sum(acc[0].value(), red);
  const double s1 = NC == 2 ? block_sum(acc[NC - 1].value(), red) : 0.0;
  if (tid == 0) {
    d.partials[band] = s0;
    if (NC == 2) d.partials[d.nupd + band] = s1;
  }
  if (last_block(st, d.nupd)) finalize_measure(d, st, red, nullptr, d.nupd);
}

template <class T, int K, int LOGN, int V>
__global__ void __launch_bounds__(PrimalBlock<T, K, LOGN, V>::threads, PrimalBlock<T, K, LOGN, V>::blocks) k_primal(const __grid_constant__ Desc d, State* __restrict__ st,
                                                                 int first) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  if (!sweep_active(st, nullptr)) return;
  primal_body<T, K, LOGN, V>(d, st, blockIdx.x, first != 0, smem_raw);
}

// Line lengths: V = 4 (few threads' worth of work on the grid) 16 .. 2048 points, V = 16 512 .. 8192
// in FP32, 512 .. 4096 in FP64; a block of BandThreads threads holds at least one line.
template <class T>
constexpr bool has_len(int logn, int v) {
  return v == 16 ? logn >= 9 && logn <= (sizeof(T) == 4 ? 13 : 12) : logn >= 4 && logn <= 11;
}

// f(LOGN, V) as integral constants, of a line length and V at run time
template <class T, class Fn>
inline cudaError_t by_len(int logn, int v, Fn f) {
  auto go = [&](auto l, auto vv) { return f(l, vv); };
#define RD_LEN(L, V) \
  case L: return go(std::integral_constant<int, L>(), std::integral_constant<int, V>());
  if (v == 16) {
    switch (logn) {
      RD_LEN(9, 16)
      RD_LEN(10, 16)
      RD_LEN(11, 16)
      RD_LEN(12, 16)
      case 13:
        if constexpr (sizeof(T) == 4) return go(std::integral_constant<int, 13>(), std::integral_constant<int, 16>());
        break;
      default: break;
    }
  } else {
    switch (logn) {
      RD_LEN(4, 4)
      RD_LEN(5, 4)
      RD_LEN(6, 4)
      RD_LEN(7, 4)
      RD_LEN(8, 4)
      RD_LEN(9, 4)
      RD_LEN(10, 4)
      RD_LEN(11, 4)
      default: break;
    }
  }
#undef RD_LEN
  return cudaErrorNotSupported;
}

// The launcher and the shared-memory limit of k_primal for key K in arithmetic T; one unit per group
// of keys, compiled in parallel.
#define RD_PRIMAL_KIND(T, K)                                                                           \
  template <>                                                                                          \
  cudaError_t launch_primal_kind<T, K>(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool first) { \
    return by_len<T>(d.lognx, c.vrow, [&](auto l, auto v) {                                            \
      return launch_pdl(k_primal<T, K, decltype(l)::value, decltype(v)::value>, d.nupd, c.thr_primal,  \
                        c.smem_primal, s, d, st, first ? 1 : 0);                                       \
    });                                                                                                \
  }                                                                                                    \
  template <>                                                                                          \
  cudaError_t allow_primal_kind<T, K>(const Desc& d, const LaunchCfg& c, int optin) {                  \
    return by_len<T>(d.lognx, c.vrow, [&](auto l, auto v) {                                            \
      return allow_smem_k(k_primal<T, K, decltype(l)::value, decltype(v)::value>, optin);              \
    });                                                                                                \
  }

}  // namespace rd
