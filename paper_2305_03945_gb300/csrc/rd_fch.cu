// The sixth-order functionalized Cahn-Hilliard step (arxiv 2305.03945, Section 3.3) in FP64:
//
//   mu(U) = a Lap U - b W'(U),   A(U) = a Lap - b diag(W''(U)) + a I,   B(U) = a Lap - b diag(W''(U))
//   F(U)  = U - U^k - dt Lap A(U) mu(U)
//   dF(U)^T P = P - dt B(U) A(U) Lap P + dt b mu(U) W'''(U) Lap P
//
// with W(u) = (u^2 - 1)^2 / 4 (W' = u^3 - u, W'' = 3u^2 - 1, W''' = 6u).  F nests three
// five-point Laplacians and the adjoint three more, each with pointwise nonlinear factors in
// between, so one PDHG iteration is a chain of simple stencil passes over whole grids (which
// at the paper's 128^2 stay in L2), with the preconditioner solve of the other equations in the
// middle (symbol g = (1 + dt a mu^2 (a mu + 2b - a))^2 of
// G = (I - dt Lap (a Lap - (2b - a) I) a Lap)^2):
//
//   k_fch_mu    M = mu(U)                           (skips once the solve has stopped)
//   k_fch_a     N = A(U) M
//   k_fch_wrow  W = U - U^k - dt Lap N, ||W||^2 partials, forward row transform of W; last block:
//               the stopping decision
//   k_fcol      column solve
//   k_dual      inverse rows, P += tau_p Y, P~ = P + (1 + omega) tau_p Y
//   k_fch_lap   Q = Lap P~
//   k_fch_a     N = A(U) Q
//   k_fch_upd   U -= tau_u (P~ - dt B(U) N + dt b M W'''(U) Q)   (pointwise in U: in place)
//
// At 128^2 each launch is a few microseconds of latency around a microsecond of FP64 work.  Fusing a
// stencil with the one it feeds (mu with A mu, Lap P~ with A Lap P~: two launches less) gained
// nothing: the inner stencil recomputed on five points costs the FP64 pipes what the launch costs
// (14.6 ms per step either way).
// Where the row kernels do not run (G = I, sides below 16 points): k_fch_w, the preconditioner-only
// sweeps and k_fch_dual.
//
// The pointwise kernels run one wave of blocks over a grid-stride loop.
#include <algorithm>

#include "rd_band.cuh"

namespace rd {

namespace {

// Threads per block of the pointwise kernels: four warps, one for each FP64 pipe of an SM, so that the
// 512 warps of a 128^2 grid spread over 128 SMs.
constexpr int kFchThreads = 128;

__device__ __forceinline__ bool fch_active(const State* st) {
  return st == nullptr || *((volatile const int*)&st->status) == ST_ACTIVE;
}

struct FchPt {
  int i, j;
  size_t o;
};

template <class Body>
__device__ __forceinline__ void fch_points(const Desc& d, Body body) {
  const size_t np = (size_t)d.nx * d.ny;
  for (size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x; g < np; g += (size_t)gridDim.x * blockDim.x)
    body(FchPt{(int)(g >> d.lognx), (int)(g & (size_t)(d.nx - 1)), g});
}

__global__ void __launch_bounds__(kFchThreads) k_fch_mu(const __grid_constant__ Desc d, const State* st,
                                                        const double* __restrict__ U, double* __restrict__ M) {
  pdl_wait();
  if (!fch_active(st)) return;
  const GField<double> u{U, d.nx, d.ny, d.bc};
  fch_points(d, [&](FchPt p) {
    const double c = U[p.o];
    M[p.o] = d.a * lap5(u, p.i, p.j, c, d.hx2, d.hy2) - d.b * (c * c * c - c);
  });
}

// N = A(U) X = a Lap X - b W''(U) X + a X
__global__ void __launch_bounds__(kFchThreads) k_fch_a(const __grid_constant__ Desc d, const State* st,
                                                       const double* __restrict__ U, const double* __restrict__ X,
                                                       double* __restrict__ N) {
  pdl_wait();
  if (!fch_active(st)) return;
  const GField<double> x{X, d.nx, d.ny, d.bc};
  fch_points(d, [&](FchPt p) {
    const double c = X[p.o], u = U[p.o];
    N[p.o] = d.a * lap5(x, p.i, p.j, c, d.hx2, d.hy2) - d.b * (3.0 * u * u - 1.0) * c + d.a * c;
  });
}

// W = U - U^k - dt Lap N; with st, the block partials of ||W||^2 and the stopping decision.
__global__ void __launch_bounds__(kFchThreads) k_fch_w(const __grid_constant__ Desc d, State* st, const double* __restrict__ U,
                                               const double* __restrict__ Uk, const double* __restrict__ N,
                                               double* __restrict__ W) {
  __shared__ double red[32];
  pdl_wait();
  if (!fch_active(st)) return;
  const GField<double> n{N, d.nx, d.ny, d.bc};
  double acc = 0.0;
  fch_points(d, [&](FchPt p) {
    const double w = U[p.o] - Uk[p.o] - d.dt * lap5(n, p.i, p.j, N[p.o], d.hx2, d.hy2);
    W[p.o] = w;
    acc += w * w;
  });
  if (st == nullptr) return;
  const double s = block_sum(acc, red);
  if (threadIdx.x == 0) d.partials[blockIdx.x] = s;
  if (last_block(st, gridDim.x)) finalize_measure(d, st, red, nullptr, gridDim.x);
}

// P~ = P + (1 + omega) tau_p Y, P <- P + tau_p Y
__global__ void __launch_bounds__(kFchThreads) k_fch_dual(const __grid_constant__ Desc d, const State* st,
                                                  const double* __restrict__ Y, double* __restrict__ P,
                                                  double* __restrict__ Pt) {
  pdl_wait();
  if (!fch_active(st)) return;
  const double tp = d.tau_p, tpe = (1.0 + d.omega) * d.tau_p;
  fch_points(d, [&](FchPt p) {
    const double y = Y[p.o], pn = P[p.o];
    Pt[p.o] = pn + tpe * y;
    P[p.o] = pn + tp * y;
  });
}

// W as k_fch_w, and the forward row transform of W into d.WY, one pair of rows per TPL threads.
template <int LOGN, int V>
__global__ void __launch_bounds__(BandThreads<double, V>::value)
    k_fch_wrow(const __grid_constant__ Desc d, State* st, const double* __restrict__ U, const double* __restrict__ Uk,
               const double* __restrict__ N) {
  using F = Rf<LOGN, V>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  pdl_wait();
  if (!fch_active(st)) return;
  constexpr int NX = F::N;
  const int lline = threadIdx.x / F::TPL, t = threadIdx.x % F::TPL;
  const int gl = blockIdx.x * (blockDim.x / F::TPL) + lline;
  const bool live = gl < d.ny >> 1;
  const int row = live ? 2 * gl : 0;
  cx<double>* line = reinterpret_cast<cx<double>*>(smem_raw) + lline * Lay<double, LOGN, V, false>::len;
  const bool per = d.bc == BC_PERIODIC;
  double acc = 0.0;
#pragma unroll 1
  for (int m = 0; m < V / 4; ++m) {
    const int j0 = 4 * (t + m * F::TPL);
    double w[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const size_t o = (size_t)(row + h) * NX + j0;
      const double* rp[3];
#pragma unroll
      for (int di = -1; di <= 1; ++di) rp[1 + di] = N + (size_t)bcmap(row + h + di, d.ny, d.bc) * NX;
      Patch<double, 1> n;
      n.load(rp, j0, NX, per);
      double u[4], uk[4];
      ld4(U + o, u);
      ld4(Uk + o, uk);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        w[h][q] = u[q] - uk[q] - d.dt * lap5(n, 0, q, n(0, q), d.hx2, d.hy2);
        acc += w[h][q] * w[h][q];
      }
    }
    put4(line, NX, per, j0, w[0], w[1]);
  }
  auto sync = [lline] { line_sync<F::TPL>(lline); };
  sync();
  row_forward<double, LOGN, V>(d, line, static_cast<double*>(d.WY) + (size_t)row * NX, t, live, sync);
  const double s = block_sum(live ? acc : 0.0, red);
  if (threadIdx.x == 0) d.partials[blockIdx.x] = s;
  if (last_block(st, gridDim.x)) finalize_measure(d, st, red, nullptr, gridDim.x);
}

__global__ void __launch_bounds__(kFchThreads) k_fch_lap(const __grid_constant__ Desc d, const State* st,
                                                         const double* __restrict__ X, double* __restrict__ Q) {
  pdl_wait();
  if (!fch_active(st)) return;
  const GField<double> x{X, d.nx, d.ny, d.bc};
  fch_points(d, [&](FchPt p) { Q[p.o] = lap5(x, p.i, p.j, X[p.o], d.hx2, d.hy2); });
}

// U -= tau_u (P~ - dt B(U) R + dt b mu W'''(U) Q), B(U) R = a Lap R - b W''(U) R
__global__ void __launch_bounds__(kFchThreads) k_fch_upd(const __grid_constant__ Desc d, const State* st,
                                                 double* __restrict__ U, const double* __restrict__ M,
                                                 const double* __restrict__ Q, const double* __restrict__ R,
                                                 const double* __restrict__ Pt) {
  pdl_wait();
  if (!fch_active(st)) return;
  const GField<double> r{R, d.nx, d.ny, d.bc};
  fch_points(d, [&](FchPt p) {
    const double u = U[p.o], rc = R[p.o];
    const double s = d.a * lap5(r, p.i, p.j, rc, d.hx2, d.hy2) - d.b * (3.0 * u * u - 1.0) * rc;
    const double g = Pt[p.o] - d.dt * s + d.dt * d.b * M[p.o] * (6.0 * u) * Q[p.o];
    U[p.o] = u - d.tau_u * g;
  });
}

template <class F>
int fch_grid(F kernel, size_t npts) {
  int dev = 0, sms = 0, occ = 0;
  const int want = (int)std::min<size_t>((npts + kFchThreads - 1) / kFchThreads, (size_t)1 << 20);
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kFchThreads, 0) != cudaSuccess)
    return std::max(1, want);
  return std::max(1, std::min(want, std::max(1, occ) * std::max(1, sms)));
}

}  // namespace

cudaError_t launch_fch_residual(const Desc& d, State* st, const FchBuffers& b, const double* U, const double* Uk,
                                double* W, int max_blocks, cudaStream_t s) {
  const size_t np = (size_t)d.nx * d.ny;
  cudaError_t e = launch_pdl(k_fch_mu, fch_grid(k_fch_mu, np), kFchThreads, 0, s, d, st, U, b.M);
  if (e == cudaSuccess) e = launch_pdl(k_fch_a, fch_grid(k_fch_a, np), kFchThreads, 0, s, d, st, U, b.M, b.N);
  if (e == cudaSuccess) e = launch_pdl(k_fch_w, std::min(max_blocks, fch_grid(k_fch_w, np)), kFchThreads, 0, s, d, st, U, Uk, b.N, W);
  return e;
}

bool fch_fused(const LaunchCfg& cpc) { return cpc.transform && cpc.fast_row && cpc.fast_col; }

cudaError_t allow_fch(const Desc& d, const LaunchCfg& cpc, int optin) {
  return by_len<double>(d.lognx, cpc.vrow, [&](auto l, auto v) {
    return allow_smem_k(k_fch_wrow<decltype(l)::value, decltype(v)::value>, optin);
  });
}

cudaError_t launch_fch_iteration(const Desc& d, const Desc& dpc, State* st, State* st_pc, const LaunchCfg& cpc,
                                 const FchBuffers& b, int max_blocks, cudaStream_t s, cudaEvent_t* ev) {
  unsigned flags;
  cudaError_t e = record_flags(s, ev, &flags);
  if (e != cudaSuccess) return e;
  auto mark = [&](int i) {
    if (ev && e == cudaSuccess) e = cudaEventRecordWithFlags(ev[i], s, flags);
  };
  const size_t np = (size_t)d.nx * d.ny;
  double* U = static_cast<double*>(d.X);
  const double* Uk = static_cast<const double*>(d.rhs);
  double* P = static_cast<double*>(d.P[0]);
  double* W = static_cast<double*>(dpc.X);  // F(U), then G^{-1} F(U) in place
  mark(0);
  if (fch_fused(cpc)) {
    Desc dd = d;
    dd.P[1] = b.Pt;
    if (e == cudaSuccess) e = launch_pdl(k_fch_mu, fch_grid(k_fch_mu, np), kFchThreads, 0, s, d, st, U, b.M);
    if (e == cudaSuccess) e = launch_pdl(k_fch_a, fch_grid(k_fch_a, np), kFchThreads, 0, s, d, st, U, b.M, b.N);
    if (e == cudaSuccess)
      e = by_len<double>(d.lognx, cpc.vrow, [&](auto l, auto v) {
        constexpr int L = decltype(l)::value, V = decltype(v)::value;
        const int lpb = cpc.thr_dual / Rf<L, V>::TPL;
        return launch_pdl(k_fch_wrow<L, V>, (d.ny / 2 + lpb - 1) / lpb, cpc.thr_dual, cpc.smem_dual, s, dd, st, U, Uk, b.N);
      });
    mark(1);
    if (e == cudaSuccess) e = launch_fcol<double>(dd, st, cpc, s, false);
    mark(2);
    if (e == cudaSuccess) e = launch_dual<double>(dd, st, cpc, s, false);
  } else {
    if (e == cudaSuccess) e = launch_fch_residual(d, st, b, U, Uk, W, max_blocks, s);
    mark(1);
    if (e == cudaSuccess && d.precond != 0) e = launch_iteration<double>(dpc, st_pc, cpc, s, nullptr);
    mark(2);
    if (e == cudaSuccess) e = launch_pdl(k_fch_dual, fch_grid(k_fch_dual, np), kFchThreads, 0, s, d, st, W, P, b.Pt);
  }
  if (e == cudaSuccess) e = launch_pdl(k_fch_lap, fch_grid(k_fch_lap, np), kFchThreads, 0, s, d, st, b.Pt, b.Q);
  if (e == cudaSuccess) e = launch_pdl(k_fch_a, fch_grid(k_fch_a, np), kFchThreads, 0, s, d, st, U, b.Q, b.N);
  if (e == cudaSuccess) e = launch_pdl(k_fch_upd, fch_grid(k_fch_upd, np), kFchThreads, 0, s, d, st, U, b.M, b.Q, b.N, b.Pt);
  mark(3);
  return e;
}

}  // namespace rd
