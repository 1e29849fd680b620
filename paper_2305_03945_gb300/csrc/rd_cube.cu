// Launchers and planning rule of the FP32 3-D kernels of rd_cube.cuh.
#include <algorithm>

#include "rd_cube.cuh"
#include "rd_launch3.h"

namespace rd {

namespace {

// line lengths: V = 16 for 128 .. 1024 points, V = 4 for 16 .. 1024
bool has_len3(int logn, int v) { return logn >= (v == 16 ? 7 : 4) && logn <= 10; }

// f(LOGN, V) as integral constants
template <class Fn>
cudaError_t by_len3(int logn, int v, Fn f) {
#define RD_LEN(L, V) \
  case L: return f(std::integral_constant<int, L>(), std::integral_constant<int, V>());
  if (v == 16) {
    switch (logn) {
      RD_LEN(7, 16)
      RD_LEN(8, 16)
      RD_LEN(9, 16)
      RD_LEN(10, 16)
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
      default: break;
    }
  }
#undef RD_LEN
  return cudaErrorNotSupported;
}

template <bool COLS>
int line_len3(int logn, int vals) {
  int n = 0;
  by_len3(logn, vals, [&](auto l, auto v) {
    n = Lay<float, decltype(l)::value, decltype(v)::value, COLS>::len;
    return cudaSuccess;
  });
  return n;
}

template <int AX, int MODE>
cudaError_t launch_axis(const Desc& d, const Cube3& c, State* st, cudaStream_t s) {
  return by_len3(AX == 1 ? d.logny : d.lognz, c.v[AX], [&](auto l, auto v) {
    return launch_pdl(k3_axis<float, AX, MODE, decltype(l)::value, decltype(v)::value>, c.grid[AX], c.thr[AX], c.smem[AX],
                      s, d, st, c.nl[AX]);
  });
}

template <int K>
cudaError_t iteration_k(const Desc& d, const Cube3& c, State* st, cudaStream_t s, cudaEvent_t* ev) {
  unsigned flags;
  cudaError_t e = record_flags(s, ev, &flags);
  auto mark = [&](int i) {
    if (ev && e == cudaSuccess) e = cudaEventRecordWithFlags(ev[i], s, flags);
  };
  mark(0);
  if (e == cudaSuccess)
    e = by_len3(d.lognx, c.v[0], [&](auto l, auto v) {
      return launch_pdl(k3_rowres<float, K, decltype(l)::value, decltype(v)::value>, c.grid[0], c.thr[0], c.smem[0], s, d, st);
    });
  mark(1);
  if (e == cudaSuccess) e = launch_axis<1, L3_FWD>(d, c, st, s);
  if (e == cudaSuccess) e = launch_axis<2, L3_FSI>(d, c, st, s);
  if (e == cudaSuccess) e = launch_axis<1, L3_INV>(d, c, st, s);
  if (e == cudaSuccess)
    e = by_len3(d.lognx, c.v[0], [&](auto l, auto v) {
      return launch_pdl(k_dual<float, decltype(l)::value, decltype(v)::value, false>, c.grid[0], c.thr[0], c.smem[0], s, d, st);
    });
  mark(2);
  if (e == cudaSuccess)
    e = launch_pdl(k3_primal<float, K>, (unsigned)(((size_t)d.nx * d.ny * d.nz / 4 + 255) / 256), 256, 0, s, d, st);
  mark(3);
  return e;
}

template <int K>
cudaError_t allow_k(const Desc& d, const Cube3& c, int optin) {
  return by_len3(d.lognx, c.v[0], [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const cudaError_t e = allow_smem_k(k3_rowres<float, K, L, V>, optin);
    return e != cudaSuccess ? e : allow_smem_k(k_dual<float, L, V, false>, optin);
  });
}

}  // namespace

cudaError_t launch_cube(const Desc& d, const Cube3& c, State* st, cudaStream_t s, cudaEvent_t* ev) {
  switch (kind_key(d)) {
    case KK_NONE_LAP: return iteration_k<KK_NONE_LAP>(d, c, st, s, ev);
    case KK_AC: return iteration_k<KK_AC>(d, c, st, s, ev);
    case KK_CH_IMPL: return iteration_k<KK_CH_IMPL>(d, c, st, s, ev);
    case KK_CH_SPLIT: return iteration_k<KK_CH_SPLIT>(d, c, st, s, ev);
    case KK_NONE_BIH: return iteration_k<KK_NONE_BIH>(d, c, st, s, ev);
    default: return cudaErrorNotSupported;
  }
}

cudaError_t allow_cube(const Desc& d, const Cube3& c, int optin) {
  cudaError_t e = cudaErrorNotSupported;
  switch (kind_key(d)) {
    case KK_NONE_LAP: e = allow_k<KK_NONE_LAP>(d, c, optin); break;
    case KK_AC: e = allow_k<KK_AC>(d, c, optin); break;
    case KK_CH_IMPL: e = allow_k<KK_CH_IMPL>(d, c, optin); break;
    case KK_CH_SPLIT: e = allow_k<KK_CH_SPLIT>(d, c, optin); break;
    case KK_NONE_BIH: e = allow_k<KK_NONE_BIH>(d, c, optin); break;
    default: break;
  }
  if (e == cudaSuccess)
    e = by_len3(d.logny, c.v[1], [&](auto l, auto v) {
      constexpr int L = decltype(l)::value, V = decltype(v)::value;
      const cudaError_t r = allow_smem_k(k3_axis<float, 1, L3_FWD, L, V>, optin);
      return r != cudaSuccess ? r : allow_smem_k(k3_axis<float, 1, L3_INV, L, V>, optin);
    });
  if (e == cudaSuccess)
    e = by_len3(d.lognz, c.v[2], [&](auto l, auto v) {
      return allow_smem_k(k3_axis<float, 2, L3_FSI, decltype(l)::value, decltype(v)::value>, optin);
    });
  return e;
}

void plan_cube(const Desc& d, int smem_limit, Cube3& c) {
  c.on = 0;
  const int logn[3] = {d.lognx, d.logny, d.lognz};
  const size_t pts = (size_t)d.nx * d.ny * d.nz;
  if (d.nz < 2) return;
  for (int a = 0; a < 3; ++a) {
    // values per thread: the line kernels' rule (see plan_vals)
    c.v[a] = pts >= ((size_t)1 << 20) && has_len3(logn[a], 16) ? 16 : 4;
    if (!has_len3(logn[a], c.v[a])) return;
  }
  // rows: blocks of 256 threads, fewer while the grid has less than two blocks per SM
  const int tpl = d.nx / c.v[0], lines = d.nz * (d.ny / 2);
  int thr = std::max(32, std::min(256, tpl));
  while (thr < 256 && lines / (2 * thr / tpl) >= 2 * 152) thr *= 2;
  c.thr[0] = thr;
  c.nl[0] = thr / tpl;
  c.grid[0] = (lines + c.nl[0] - 1) / c.nl[0];
  c.smem[0] = c.nl[0] * line_len3<false>(d.lognx, c.v[0]) * (int)sizeof(cx<float>);
  if (c.smem[0] > smem_limit) return;
  // y and z: 16 column pairs (128-byte row segments) per block, fewer where the block is too large
  // or the grid too small
  for (int a = 1; a < 3; ++a) {
    const int t = (a == 1 ? d.ny : d.nz) / c.v[a], len = line_len3<true>(logn[a], c.v[a]) * (int)sizeof(cx<float>);
    const int third = a == 1 ? d.nz : d.ny;
    int nl = std::min(16, d.nx / 2);
    while (nl > 1 && (nl * t > 512 || nl * len > smem_limit / 2 ||
                      (third * (d.nx / 2 / nl) < 152 && nl * t > 64 && nl > 4)))
      nl /= 2;
    if (nl * t > 512) return;
    c.nl[a] = nl;
    c.thr[a] = nl * t;
    c.smem[a] = nl * len;
    c.grid[a] = third * (d.nx / 2 / nl);
  }
  c.on = 1;
}

}  // namespace rd
