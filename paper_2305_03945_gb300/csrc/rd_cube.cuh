// Kernels of one G-prox PDHG iteration on 3-D grids (scalar equations; see rd_3d.cuh for the scheme
// and its pointwise formulas) on the register-resident line transforms of rd_fft.cuh:
//
//   k3_rowres          W = F(U_n) on pairs of x rows, norm partials and stopping decision, and the
//                      forward transform along x of the pair, into WY;
//   k3_axis<1, FWD>    forward along y, in place in WY;
//   k3_axis<2, FSI>    forward along z, times 1 / (g_hat nx ny nz), inverse along z;
//   k3_axis<1, INV>    inverse along y;
//   k_dual             inverse along x, the dual update and P~ (rd_band.cuh);
//   k3_primal          U_{n+1} = U_n - tau_u dF(U_n)^T P~.
//
// Against the kernels of rd_3d.cuh the forward x pass is part of the residual (one launch and 8 bytes
// per point less in FP32), every stencil reads vectors of four points, and a transform crosses shared
// memory once per exchange.
#pragma once

#include "rd_3d.cuh"
#include "rd_band.cuh"

namespace rd {

// Values of a field around four adjacent points of row (l, i), boundary-mapped: rows (l + dl, i + di)
// with |dl| + |di| <= H and H - |dl| - |di| columns on either side, as the accessor of the pointwise
// formulas (at offsets from the first point); the other entries stay unset.
template <class T, int H>
struct Patch3 {
  T v[2 * H + 1][2 * H + 1][4 + 2 * H];
  __device__ __forceinline__ T operator()(int l, int i, int j) const { return v[l + H][i + H][j + H]; }
  __device__ __forceinline__ void load(const T* __restrict__ p, const Desc& d, int l, int i, int j0) {
    const bool per = d.bc == BC_PERIODIC;
    const int nx = d.nx;
    int jl[2], jr[2];
    jl[0] = j0 > 0 ? j0 - 1 : (per ? nx - 1 : 0);
    jr[0] = j0 + 4 < nx ? j0 + 4 : (per ? 0 : nx - 1);
    if constexpr (H > 1) {
      jl[1] = j0 > 0 ? j0 - 2 : (per ? nx - 2 : 1);
      jr[1] = j0 + 4 < nx ? j0 + 5 : (per ? 1 : nx - 2);
    }
#pragma unroll
    for (int dl = -H; dl <= H; ++dl) {
      const size_t zo = (size_t)bcmap(l + dl, d.nz, d.bc) * d.ny;
#pragma unroll
      for (int di = -H; di <= H; ++di) {
        const int side = H - (dl < 0 ? -dl : dl) - (di < 0 ? -di : di);
        if (side < 0) continue;
        const T* r = p + (zo + bcmap(i + di, d.ny, d.bc)) * nx;
        ld4(r + j0, &v[H + dl][H + di][H]);
#pragma unroll
        for (int s = 0; s < H; ++s)
          if (s < side) {
            v[H + dl][H + di][H - 1 - s] = r[jl[s]];
            v[H + dl][H + di][H + 4 + s] = r[jr[s]];
          }
      }
    }
  }
};

// the base state at the four points
template <class T>
struct Pt4z {
  T v[4];
  __device__ __forceinline__ T operator()(int, int, int j) const { return v[j]; }
};

// ---------------------------------------------------------------------------------------
// k3_rowres
// ---------------------------------------------------------------------------------------
// The lines of group `blk`; the squares of the thread's residuals are added to acc_out (in twice FP32's
// precision, see SumSq).
template <class T, int K, int LOGN, int V>
__device__ __forceinline__ void rowres3_body(const Desc& d, int blk, unsigned char* smem_raw, double& acc_out) {
  using F = Rf<LOGN, V>;
  constexpr int N = F::N;
  constexpr int H = KT<K>::H;
  constexpr bool DC = sizeof(T) == 4;
  constexpr bool BASE = DC && KT<K>::nonlinear;
  const int lline = threadIdx.x / F::TPL, t = threadIdx.x % F::TPL;
  const int lines = d.nz * (d.ny >> 1);
  const int gl = blk * (blockDim.x / F::TPL) + lline;
  const bool live = gl < lines;
  cx<T>* line = reinterpret_cast<cx<T>*>(smem_raw) + lline * Lay<T, LOGN, V, false>::len;
  const bool per = d.bc == BC_PERIODIC;
  const size_t o = (size_t)(live ? gl : 0) * 2 * N;
  const int row0 = (live ? gl : 0) * 2, l = row0 >> d.logny, i0 = row0 & (d.ny - 1);
  const T* X = static_cast<const T*>(d.X);
  const T* Bs = static_cast<const T*>(d.base);
  const T* R = static_cast<const T*>(d.rhs);
  SumSq<T> acc;
#pragma unroll 1
  for (int m = 0; m < V / 4; ++m) {
    const int j0 = 4 * (t + m * F::TPL);
    T w[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T rr[4];
      ld4(R + o + (size_t)h * N + j0, rr);
      Patch3<T, H> x;
      x.load(X, d, l, i0 + h, j0);
      auto points = [&](const auto& b) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          w[h][q] = residual3_pt<T, K, DC>(d, x, b, 0, 0, q, rr[q]);
          acc.add(w[h][q]);
        }
      };
      if constexpr (BASE && base_stencil<K>()) {
        Patch3<T, 1> b;
        b.load(Bs, d, l, i0 + h, j0);
        points(b);
      } else if constexpr (BASE) {
        Pt4z<T> b;
        ld4(Bs + o + (size_t)h * N + j0, b.v);
        points(b);
      } else {
        points(x);
      }
    }
    put4(line, N, per, j0, w[0], w[1]);
  }
  auto sync = [lline] { line_sync<F::TPL>(lline); };
  sync();
  row_forward<T, LOGN, V>(d, line, static_cast<T*>(d.WY) + o, t, live, sync);
  if (live) acc_out += acc.value();
}

// Partial norm of block `blk` of `nblk`, stopping decision in the last one.
__device__ __forceinline__ void rowres_finish(const Desc& d, State* __restrict__ st, Slot* slot, int blk, int nblk, double a0,
                                              double a1) {
  __shared__ double red[32];
  const double s0 = block_sum(a0, red);
  const double s1 = d.ncomp == 2 ? block_sum(a1, red) : 0.0;
  if (threadIdx.x == 0) {
    d.partials[blk] = s0;
    if (d.ncomp == 2) d.partials[nblk + blk] = s1;
  }
  if (last_block(st, nblk)) finalize_measure(d, st, red, slot, nblk);
}

template <class T, int K, int LOGN, int V>
__global__ void __launch_bounds__(256) k3_rowres(const __grid_constant__ Desc d, State* __restrict__ st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  if (!sweep_active(st, nullptr)) return;
  double acc = 0.0;
  rowres3_body<T, K, LOGN, V>(d, blockIdx.x, smem_raw, acc);
  rowres_finish(d, st, nullptr, blockIdx.x, gridDim.x, acc, 0.0);
}

// ---------------------------------------------------------------------------------------
// k3_axis: transforms along y (AX = 1) and z (AX = 2), `nl` adjacent column pairs per block; `sync` is a
// barrier of the nl TPL threads.  Scalar 3-D grids; 2-D grids (nz <= 1, AX = 1) with either number of
// components.
// ---------------------------------------------------------------------------------------
template <class T, int AX, int MODE, int LOGN, int V, class Sync>
__device__ __forceinline__ void axis3_body(const Desc& d, int nl, int blk, unsigned char* smem_raw, Sync sync) {
  using F = Rf<LOGN, V>;
  using P1 = Pass<T, LOGN, V, true, 1>;
  constexpr int N = F::N;
  const int hx = d.nx >> 1;
  const int m = threadIdx.x % nl, t = threadIdx.x / nl;
  const int ntx = hx / nl;
  const int third = blk / ntx;                    // z of a y line, y of a z line (2-D: the component)
  const int col = (blk - third * ntx) * nl + m;   // pair of columns
  const size_t plane = (size_t)hx * d.ny;
  const size_t rs = AX == 1 ? hx : plane;         // pairs between the elements of a line
  cx<T>* G = reinterpret_cast<cx<T>*>(d.WY) + (AX == 1 ? (size_t)third * plane : (size_t)third * hx) + col;
  const bool per = d.bc == BC_PERIODIC;
  const cx<T>* tw = static_cast<const cx<T>*>(AX == 1 ? d.twy : d.twz);
  const cx<T>* dc = static_cast<const cx<T>*>(AX == 1 ? d.dcy : d.dcz);
  cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw) + m;
  cx<T> v[V];
  // frequency of paired value i and its partner (the self-paired 0 and N/2 in thread 0)
  auto freq = [&](int i) { return rf_freq<V>(N, t, i); };
  auto part = [&](int i, int k) { return i == 0 && t == 0 ? N / 2 : N - k; };
  if constexpr (MODE != L3_INV) {
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int n = P1::natural(t, e);
      v[e] = G[(size_t)(per ? n : mk_perm(n, N)) * rs];
    }
    rf_forward<T, LOGN, V, true>(v, buf, nl, tw, t, sync);
  }
  if constexpr (MODE == L3_FSI) {
    const T* mux = static_cast<const T*>(d.mux);
    const T* muo = static_cast<const T*>(AX == 1 ? d.muz : d.muy);
    const T mo = d.nz > 1 ? __ldg(muo + third) : T(0);
    scale_pairs<T, N, V>(v, t, per,
                         SymMu<T>{Symbol<T>(d, d.nz > 1 ? 0 : third), static_cast<const T*>(AX == 1 ? d.muy : d.muz),
                                  __ldg(mux + 2 * col) + mo, __ldg(mux + 2 * col + 1) + mo},
                         dc);
  }
  if constexpr (MODE == L3_FWD) {
    rf_pair<T, V>(v, t);
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      const int k = freq(i);
      const cx<T> w = per ? cx<T>{T(0), T(0)} : ldg(dc + k);
      cx<T> a, b;
      if (i == 0 && t == 0) {
        cx<T> skip;
        pair_fwd(per, v[0], v[0], w, a, skip);
        pair_fwd(per, v[V - 1], v[V - 1], per ? w : ldg(dc + N / 2), b, skip);
      } else {
        pair_fwd(per, v[i], v[V - 1 - i], w, a, b);
      }
      G[(size_t)k * rs] = a;
      G[(size_t)part(i, k) * rs] = b;
    }
  }
  if constexpr (MODE == L3_INV) {
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      const int k = freq(i);
      v[i] = G[(size_t)k * rs];
      v[V - 1 - i] = G[(size_t)part(i, k) * rs];
    }
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      const int k = freq(i);
      const cx<T> w = per ? cx<T>{T(0), T(0)} : ldg(dc + k);
      cx<T> a, b;
      if (i == 0 && t == 0) {
        cx<T> skip;
        pair_inv(per, v[0], per ? v[0] : cx<T>{T(0), T(0)}, w, a, skip);
        pair_inv(per, v[V - 1], v[V - 1], per ? w : ldg(dc + N / 2), b, skip);
      } else {
        pair_inv(per, v[i], v[V - 1 - i], w, a, b);
      }
      v[i] = a;
      v[V - 1 - i] = b;
    }
    rf_unpair<T, V>(v, t);
  }
  if constexpr (MODE != L3_FWD) {
    rf_inverse<T, LOGN, V, true>(v, buf, nl, tw, t, sync);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int n = P1::natural(t, e);
      G[(size_t)(per ? n : mk_perm(n, N)) * rs] = v[e];
    }
  }
}

template <class T, int AX, int MODE, int LOGN, int V>
__global__ void __launch_bounds__(BandThreads<T, V>::value) k3_axis(const __grid_constant__ Desc d, State* __restrict__ st,
                                                                    int nl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  if (!sweep_active(st, nullptr)) return;
  axis3_body<T, AX, MODE, LOGN, V>(d, nl, blockIdx.x, smem_raw, [] { __syncthreads(); });
}

// ---------------------------------------------------------------------------------------
// k3_primal: four points per thread
// ---------------------------------------------------------------------------------------
template <class T, int K>
__device__ __forceinline__ void primal3_body(const Desc& d, int blk) {
  constexpr int H = KT<K>::H;
  constexpr bool BASE = sizeof(T) == 4 && KT<K>::nonlinear;
  const size_t g = (size_t)blk * blockDim.x + threadIdx.x;
  const size_t q = 4 * g;
  if (q >= (size_t)d.nx * d.ny * d.nz) return;
  int l, i, j0;
  point3(d, q, l, i, j0);
  T* X = static_cast<T*>(d.X) + q;
  T x[4], s[4] = {T(0), T(0), T(0), T(0)};
  ld4(X, x);
  if constexpr (BASE) ld4(static_cast<const T*>(d.base) + q, s);
  Patch3<T, H> p;
  p.load(static_cast<const T*>(d.P[1]), d, l, i, j0);
  const T tu = T(d.tau_u);
#pragma unroll
  for (int k = 0; k < 4; ++k) x[k] -= tu * gradT3_pt<T, K>(d, p, x[k] + s[k], 0, 0, k);
  st4(X, x);
}

template <class T, int K>
__global__ void __launch_bounds__(256) k3_primal(const __grid_constant__ Desc d, State* __restrict__ st) {
  pdl_wait();
  if (!sweep_active(st, nullptr)) return;
  primal3_body<T, K>(d, blockIdx.x);
}

}  // namespace rd
