// Batched PDHG iteration of the slots whose sides are all 16 points or more, on the register-resident
// line transforms (rd_fft.cuh): residual with the forward x pass, column solve (2-D) or y, z, y passes
// (3-D), inverse x with the dual update, primal update.  P~ takes the place of Y in the transform
// buffer, so a slot needs no array beyond those of the Stockham sweeps.
//
// A launch covers all slots of its group through a work list of (slot, block) pairs; every slot runs
// blk3 blocks of 256 threads in each kernel, each looping over its share of the slot's line groups, so
// that a slot does the same work in the same order whatever else shares the launch.  Values per thread
// follow the line length alone, for the same reason: 4 up to 64 (3-D) / 512 (2-D) points, 16 beyond.  Few threads
// with long chains pay on a full chip, many with short ones on an empty one; the lines lie where a lone slot gains
// more than a full batch loses.  Runs of five steps at 4 / 16 values: 2-D 256 and 512 points, one slot of 256^2 4.39 / 6.13 ms,
// of 512^2 5.37 / 7.33 ms, eight of 256^2 7.79 / 8.84 ms, of 512^2 16.9 / 13.5 ms; 3-D 128 points, one cube of 128 19.0 / 15.7 ms,
// four 60.8 / 48.1 ms, one 128 x 64 x 64 7.17 / 7.71 ms.
#pragma once

#include "rd_cube.cuh"

namespace rd {

constexpr int kLineThreads = 256;

// f(LOGN, V) for a line of a 2-D (16 .. 1024) or 3-D (16 .. 512) slot
template <bool D3, class Fn>
__host__ __device__ __forceinline__ void batch_len(int logn, Fn f) {
#define RD_LEN(L, V) \
  case L: f(std::integral_constant<int, L>(), std::integral_constant<int, V>()); break;
  if constexpr (D3) {
    switch (logn) {
      RD_LEN(4, 4)
      RD_LEN(5, 4)
      RD_LEN(6, 4)
      RD_LEN(7, 16)
      RD_LEN(8, 16)
      RD_LEN(9, 16)
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
      RD_LEN(10, 16)
      default: break;
    }
  }
#undef RD_LEN
}

// Column pairs of a block along y or z: what 256 threads hold, at most 16 and the row; their threads are
// whole warps (8 pairs of 4 threads at least).
template <class F>
__host__ __device__ constexpr int axis_lines(int nx) {
  const int fit = kLineThreads / F::TPL, most = (nx >> 1) < 16 ? nx >> 1 : 16;
  return fit < most ? fit : most;
}

// line groups of one kernel: rows (dual: of every component), columns along y and z
template <bool D3>
inline int batch_groups(const Desc& d) {
  int most = 1;
  const int nz = D3 ? d.nz : 1;
  batch_len<D3>(d.lognx, [&](auto l, auto v) {
    using F = Rf<decltype(l)::value, decltype(v)::value>;
    const int lpb = kLineThreads / F::TPL;
    most = (nz * (d.ny / 2) + lpb - 1) / lpb;
  });
  batch_len<D3>(d.logny, [&](auto l, auto v) {
    using F = Rf<decltype(l)::value, decltype(v)::value>;
    const int g = (D3 ? d.nz : d.ncomp) * (d.nx / 2 / axis_lines<F>(d.nx));
    most = g > most ? g : most;
  });
  return most;
}

// dynamic shared memory of the row and the column kernels for slot d
template <bool D3>
inline void batch_smem(const Desc& d, int* row, int* col) {
  batch_len<D3>(d.lognx, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    *row = d.ncomp * (kLineThreads / Rf<L, V>::TPL) * Lay<float, L, V, false>::len * (int)sizeof(cx<float>);
  });
  *col = 0;
  for (int a = 1; a <= (D3 ? 2 : 1); ++a)
    batch_len<D3>(a == 1 ? d.logny : d.lognz, [&](auto l, auto v) {
      constexpr int L = decltype(l)::value, V = decltype(v)::value;
      const int b = axis_lines<Rf<L, V>>(d.nx) * Lay<float, L, V, true>::len * (int)sizeof(cx<float>);
      *col = b > *col ? b : *col;
    });
}

__device__ __forceinline__ bool slot_inner(const Slot* sl) { return *((volatile const int*)&sl->phase) == PH_INNER; }

// ---------------------------------------------------------------------------------------
// 2-D pieces
// ---------------------------------------------------------------------------------------

// W = F(U_n) on the row pairs of group `grp` and its forward row transform into WY
template <int K, int LOGN, int V>
__device__ __forceinline__ void rowres2_body(const Desc& d, int grp, unsigned char* smem_raw, double* acc_out) {
  using F = Rf<LOGN, V>;
  constexpr int N = F::N;
  constexpr int H = KT<K>::H;
  constexpr int NC = ncomp_of<K>();
  constexpr bool BASE = KT<K>::nonlinear;
  constexpr int LEN = Lay<float, LOGN, V, false>::len;
  const int lpb = blockDim.x / F::TPL;
  const int lline = threadIdx.x / F::TPL, t = threadIdx.x % F::TPL;
  const int gl = grp * lpb + lline;
  const bool live = gl < d.ny >> 1;
  const int row0 = live ? 2 * gl : 0;
  const size_t plane = (size_t)N * d.ny;
  const bool per = d.bc == BC_PERIODIC;
  cx<float>* lines = reinterpret_cast<cx<float>*>(smem_raw);
  const float* X = static_cast<const float*>(d.X);
  const float* Bs = static_cast<const float*>(d.base);
  const float* R = static_cast<const float*>(d.rhs);
  SumSq<float> acc[NC];
#pragma unroll 1
  for (int m = 0; m < V / 4; ++m) {
    const int j0 = 4 * (t + m * F::TPL);
    float w[NC][2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = row0 + h;
      const size_t o = (size_t)row * N + j0;
      float rr[NC][4];
      Patch<float, H> x[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        ld4(R + c * plane + o, rr[c]);
        const float* rp[2 * H + 1];
#pragma unroll
        for (int di = -H; di <= H; ++di) rp[H + di] = X + c * plane + (size_t)bcmap(row + di, d.ny, d.bc) * N;
        x[c].load(rp, j0, N, per);
      }
      auto points = [&](const auto& b0, const auto& b1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float ww[2] = {0.f, 0.f};
          residual_pt<float, K, true>(d, x[0], x[NC - 1], b0, b1, 0, q, rr[0][q], rr[NC - 1][q], ww);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            w[c][h][q] = ww[c];
            acc[c].add(ww[c]);
          }
        }
      };
      if constexpr (BASE && base_stencil<K>()) {
        Patch<float, 1> b;
        const float* bp[3];
#pragma unroll
        for (int di = -1; di <= 1; ++di) bp[1 + di] = Bs + (size_t)bcmap(row + di, d.ny, d.bc) * N;
        b.load(bp, j0, N, per);
        points(b, b);
      } else if constexpr (BASE) {
        Pt4<float> b[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) ld4(Bs + c * plane + o, b[c].v);
        points(b[0], b[NC - 1]);
      } else {
        points(x[0], x[NC - 1]);
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) put4(lines + (c * lpb + lline) * LEN, N, per, j0, w[c][0], w[c][1]);
  }
  auto sync = [lline] { line_sync<F::TPL>(lline); };
  sync();
#pragma unroll 1
  for (int c = 0; c < NC; ++c)
    row_forward<float, LOGN, V>(d, lines + (c * lpb + lline) * LEN, static_cast<float*>(d.WY) + c * plane + (size_t)row0 * N, t,
                                live, sync);
  if (live) {
    acc_out[0] += acc[0].value();
    if constexpr (NC == 2) acc_out[1] += acc[1].value();
  }
}

// U_{n+1} = U_n - tau_u dF(U_n)^T P~ at the four points of group q4
template <int K>
__device__ __forceinline__ void primal2_body(const Desc& d, int q4) {
  constexpr int H = KT<K>::H;
  constexpr int NC = ncomp_of<K>();
  const int nx = d.nx, ny = d.ny;
  const size_t plane = (size_t)nx * ny;
  const int i = (q4 * 4) >> d.lognx, j0 = (q4 * 4) & (nx - 1);
  const size_t o = (size_t)i * nx + j0;
  float* X = static_cast<float*>(d.X);
  const float* Bs = static_cast<const float*>(d.base);
  const float* Pt = static_cast<const float*>(d.P[1]);
  float x[NC][4], s[NC][4] = {};
  Patch<float, H> p[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    ld4(X + c * plane + o, x[c]);
    if constexpr (KT<K>::nonlinear) ld4(Bs + c * plane + o, s[c]);
    const float* rp[2 * H + 1];
#pragma unroll
    for (int di = -H; di <= H; ++di) rp[H + di] = Pt + c * plane + (size_t)bcmap(i + di, ny, d.bc) * nx;
    p[c].load(rp, j0, nx, d.bc == BC_PERIODIC);
  }
  const float tu = float(d.tau_u);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float g[2] = {0.f, 0.f};
    gradT_pt<float, K>(d, p[0], p[NC - 1], x[0][q] + s[0][q], x[NC - 1][q] + s[NC - 1][q], 0, q, g);
#pragma unroll
    for (int c = 0; c < NC; ++c) x[c][q] -= tu * g[c];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) st4(X + c * plane + o, x[c]);
}

// ---------------------------------------------------------------------------------------
// batched kernels
// ---------------------------------------------------------------------------------------
template <int K, bool D3>
__global__ void __launch_bounds__(kLineThreads)
    k_rowres_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (!slot_inner(slots + w.x)) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  const Desc& d = sd;
  double acc[2] = {0.0, 0.0};
  batch_len<D3>(d.lognx, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const int lpb = kLineThreads / Rf<L, V>::TPL;
    const int n = ((D3 ? d.nz : 1) * (d.ny >> 1) + lpb - 1) / lpb;
    for (int g = w.y; g < n; g += d.blk3) {
      if constexpr (D3) rowres3_body<float, K, L, V>(d, g, smem_raw, acc[0]);
      else rowres2_body<K, L, V>(d, g, smem_raw, acc);
      __syncthreads();
    }
  });
  rowres_finish(d, &slots[w.x].inner, slots + w.x, w.y, d.blk3, acc[0], acc[1]);
}

template <bool D3, int AX, int MODE>
__global__ void __launch_bounds__(kLineThreads)
    k_axis_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (!slot_inner(slots + w.x)) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  const Desc& d = sd;
  batch_len<D3>(AX == 1 ? d.logny : d.lognz, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const int nl = axis_lines<Rf<L, V>>(d.nx), cnt = nl * Rf<L, V>::TPL;  // a multiple of 32
    const int n = (AX == 2 ? d.ny : (D3 ? d.nz : d.ncomp)) * ((d.nx >> 1) / nl);
    auto sync = [cnt] { asm volatile("bar.sync 1, %0;" ::"r"(cnt) : "memory"); };
    for (int g = w.y; g < n; g += d.blk3) {
      if ((int)threadIdx.x < cnt) axis3_body<float, AX, MODE, L, V>(d, nl, g, smem_raw, sync);
      __syncthreads();
    }
  });
}

template <bool D3>
__global__ void __launch_bounds__(kLineThreads)
    k_dual_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (!slot_inner(slots + w.x)) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  const Desc& d = sd;
  batch_len<D3>(d.lognx, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const int lpb = kLineThreads / Rf<L, V>::TPL;
    const int n = (d.ncomp * (D3 ? d.nz : 1) * (d.ny >> 1) + lpb - 1) / lpb;
    for (int g = w.y; g < n; g += d.blk3) {
      dual_body<float, L, V, false>(d, g, smem_raw);
      __syncthreads();
    }
  });
}

template <int K, bool D3>
__global__ void __launch_bounds__(kLineThreads)
    k_primal_b(const Desc* __restrict__ descs, Slot* __restrict__ slots, const int2* __restrict__ items) {
  __shared__ Desc sd;
  const int2 w = items[blockIdx.x];
  if (!slot_inner(slots + w.x)) return;
  load_desc(sd, descs + w.x);
  __syncthreads();
  const Desc& d = sd;
  const size_t n4 = (size_t)d.nx * d.ny * (D3 ? d.nz : 1) / 4;
  for (size_t g = w.y; g * kLineThreads < n4; g += d.blk3) {
    if constexpr (D3) {
      primal3_body<float, K>(d, (int)g);
    } else {
      const size_t q4 = g * kLineThreads + threadIdx.x;
      if (q4 < n4) primal2_body<K>(d, (int)q4);
    }
  }
}

}  // namespace rd
