// k_fcol, k_rowfwd and k_dual in float and double, the fused iteration's dispatch and the planning
// rule of the register-resident sweep kernels (k_primal is in rd_band_{f32,f64}_{lap,two,bih}.cu).
#include <algorithm>

#include "rd_band.cuh"

namespace rd {

namespace {

// complex entries of an exchange buffer
template <class T, bool COLS>
int line_len(int logn, int vals) {
  int n = 0;
  by_len<T>(logn, vals, [&](auto l, auto v) {
    n = Lay<T, decltype(l)::value, decltype(v)::value, COLS>::len;
    return cudaSuccess;
  });
  return n;
}

}  // namespace

template <class T>
cudaError_t launch_fcol(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool pc) {
  if (sizeof(T) == 8 && !d.scale) return cudaErrorInvalidValue;  // the handle holds no symbol table
  return by_len<T>(d.logny, c.vcol, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    if constexpr (sizeof(T) == 4 && V == 16 && L >= 11) {
      if (c.tmap && !pc)
        return launch_pdl(d.bc == BC_PERIODIC ? k_fcol_tma<L, true> : k_fcol_tma<L, false>, c.grid_cols, c.thr_fcol, c.smem_fcol,
                          s, d, st, *static_cast<const CUtensorMap*>(c.tmap));
    }
    return launch_pdl(d.bc == BC_PERIODIC ? k_fcol<T, L, V, true> : k_fcol<T, L, V, false>, c.grid_cols, c.thr_fcol,
                      c.smem_fcol, s, d, pc ? nullptr : st);
  });
}

cudaError_t launch_symbol(const Desc& d, double* table, cudaStream_t s) {
  const size_t n = (size_t)d.ncomp * d.nx * d.ny;
  k_symbol<<<(unsigned)std::min<size_t>((n + 255) / 256, 8 * 152), 256, 0, s>>>(d, table);
  return cudaGetLastError();
}

bool make_col_map(const Desc& d, const LaunchCfg& c, void* map) {
  if (!c.fast_col || c.vcol != 16 || d.ny < 2048 || d.col_width < 4) return false;
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    return false;
  }
  const cuuint64_t dims[2] = {(cuuint64_t)d.nx, (cuuint64_t)d.ncomp * d.ny};
  const cuuint64_t strides[1] = {(cuuint64_t)d.nx * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)d.col_width, (cuuint32_t)kTmaRows};
  const cuuint32_t one[2] = {1, 1};
  return reinterpret_cast<Encode>(fn)(static_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, d.WY, dims, strides, box,
                                      one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                      CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <>
cudaError_t launch_rowfwd<double>(const Desc& d, const LaunchCfg& c, cudaStream_t s) {
  using T = double;
  return by_len<T>(d.lognx, c.vrow, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const int lpb = c.thr_dual / Rf<L, V>::TPL;
    return launch_pdl(k_rowfwd<T, L, V>, (d.ncomp * (d.ny / 2) + lpb - 1) / lpb, c.thr_dual, c.smem_dual, s, d);
  });
}

template <class T>
cudaError_t launch_dual(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool pc) {
  return by_len<T>(d.lognx, c.vrow, [&](auto l, auto v) {
    constexpr int L = decltype(l)::value, V = decltype(v)::value;
    const int lpb = c.thr_dual / Rf<L, V>::TPL;
    const int grid = (d.ncomp * (d.ny / 2) + lpb - 1) / lpb;
    if constexpr (sizeof(T) == 8)
      if (pc) return launch_pdl(k_dual<T, L, V, true>, grid, c.thr_dual, c.smem_dual, s, d, st);
    return pc ? cudaErrorNotSupported : launch_pdl(k_dual<T, L, V, false>, grid, c.thr_dual, c.smem_dual, s, d, st);
  });
}

namespace {
template <class T>
cudaError_t launch_primal(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool first) {
  switch (kind_key(d)) {
    case KK_NONE_LAP: return launch_primal_kind<T, KK_NONE_LAP>(d, st, c, s, first);
    case KK_AC: return launch_primal_kind<T, KK_AC>(d, st, c, s, first);
    case KK_CH_IMPL: return launch_primal_kind<T, KK_CH_IMPL>(d, st, c, s, first);
    case KK_CH_SPLIT: return launch_primal_kind<T, KK_CH_SPLIT>(d, st, c, s, first);
    case KK_GS: return launch_primal_kind<T, KK_GS>(d, st, c, s, first);
    case KK_SCHNAK: return launch_primal_kind<T, KK_SCHNAK>(d, st, c, s, first);
    case KK_NONE_BIH: return launch_primal_kind<T, KK_NONE_BIH>(d, st, c, s, first);
    default: return cudaErrorNotSupported;
  }
}

template <class T>
cudaError_t allow_primal(const Desc& d, const LaunchCfg& c, int optin) {
  switch (kind_key(d)) {
    case KK_NONE_LAP: return allow_primal_kind<T, KK_NONE_LAP>(d, c, optin);
    case KK_AC: return allow_primal_kind<T, KK_AC>(d, c, optin);
    case KK_CH_IMPL: return allow_primal_kind<T, KK_CH_IMPL>(d, c, optin);
    case KK_CH_SPLIT: return allow_primal_kind<T, KK_CH_SPLIT>(d, c, optin);
    case KK_GS: return allow_primal_kind<T, KK_GS>(d, c, optin);
    case KK_SCHNAK: return allow_primal_kind<T, KK_SCHNAK>(d, c, optin);
    case KK_NONE_BIH: return allow_primal_kind<T, KK_NONE_BIH>(d, c, optin);
    default: return cudaErrorNotSupported;
  }
}
}  // namespace

template <class T>
cudaError_t launch_fused(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, cudaEvent_t* ev, bool first) {
  unsigned flags;
  cudaError_t e = record_flags(s, ev, &flags);
  if (e != cudaSuccess) return e;
  auto mark = [&](int i) {
    if (ev && e == cudaSuccess) e = cudaEventRecordWithFlags(ev[i], s, flags);
  };
  mark(0);
  if (first && e == cudaSuccess) e = launch_primal<T>(d, st, c, s, true);
  mark(1);
  if (e == cudaSuccess) e = launch_col<T>(d, st, c, s, false);
  mark(2);
  if (e == cudaSuccess) e = launch_dual<T>(d, st, c, s, false);
  if (e == cudaSuccess) e = launch_primal<T>(d, st, c, s, false);
  mark(3);
  return e;
}

template <class T>
cudaError_t allow_band(const Desc& d, const LaunchCfg& c, int optin, bool primal, bool tune) {
  cudaError_t e = cudaSuccess;
  if (c.transform && has_len<T>(d.logny, c.vcol))
    e = by_len<T>(d.logny, c.vcol, [&](auto l, auto v) {
      constexpr int L = decltype(l)::value, V = decltype(v)::value;
      if constexpr (sizeof(T) == 4 && V == 16 && L >= 11) {
        if (c.tmap || tune) {
          const cudaError_t r =
              d.bc == BC_PERIODIC ? allow_smem_k(k_fcol_tma<L, true>, optin) : allow_smem_k(k_fcol_tma<L, false>, optin);
          if (r != cudaSuccess || !tune) return r;
        }
      }
      return d.bc == BC_PERIODIC ? allow_smem_k(k_fcol<T, L, V, true>, optin) : allow_smem_k(k_fcol<T, L, V, false>, optin);
    });
  if (c.fast_row && e == cudaSuccess)
    e = by_len<T>(d.lognx, c.vrow, [&](auto l, auto v) {
      constexpr int L = decltype(l)::value, V = decltype(v)::value;
      cudaError_t r = allow_smem_k(k_dual<T, L, V, false>, optin);
      if constexpr (sizeof(T) == 8) {  // the preconditioner alone
        if (r == cudaSuccess) r = allow_smem_k(k_dual<T, L, V, true>, optin);
        if (r == cudaSuccess) r = allow_smem_k(k_rowfwd<T, L, V>, optin);
      }
      return r;
    });
  if (c.fast_row && primal && e == cudaSuccess) e = allow_primal<T>(d, c, optin);
  return e;
}

// Values per thread: 16 has the fewest instructions and barriers, 4 four times the threads.  A grid of
// 2^20 points gives a GB300 seven warps per SM at V = 16, half of that is too little to cover the
// latency of a pass; FP64 runs on four narrow pipes per SM (a warp's instruction holds one of them
// for 64 cycles), which the same warps just keep busy.  Measured, step time at V = 16 / V = 4:
// FP32 1024^2 0.753 / 0.912 ms, 512^2 0.828 / 0.769 ms; FP64 1024^2 4.85 / 5.16 ms; 128^2 x 2
// preconditioner solve FP64 115 / 55 us.
template <class T>
static int plan_vals(const Desc& d, int logn) {
  const int v = (size_t)d.ncomp * d.nx * d.ny >= ((size_t)1 << 20) ? 16 : 4;
  return has_len<T>(logn, v) ? v : 20 - v;
}

template <class T>
void plan_band(const Desc& d, int H, int smem_limit, LaunchCfg& c) {
  c.fast_col = c.fast_row = 0;
  if (!c.transform) return;
  const int nc = d.ncomp;
  c.vcol = plan_vals<T>(d, d.logny);
  c.vrow = plan_vals<T>(d, d.lognx);
  if (has_len<T>(d.logny, c.vcol)) {
    const int nl = d.col_width >> 1, tpl = d.ny / c.vcol;
    c.thr_fcol = nl * tpl;
    c.smem_fcol = nl * line_len<T, true>(d.logny, c.vcol) * (int)sizeof(cx<T>);
    const int cap = d.ny > 2048 && sizeof(T) == 4 ? 1024 : band_threads_max(sizeof(T), c.vcol);
    c.fast_col = (nl & (nl - 1)) == 0 && c.thr_fcol <= cap && c.smem_fcol <= smem_limit;
  }
  if (has_len<T>(d.lognx, c.vrow)) {
    const int tpl = d.nx / c.vrow, len = line_len<T, false>(d.lognx, c.vrow);
    const int cap = primal_wide(d, H, sizeof(T), c.vrow) ? 1024 : band_threads_max(sizeof(T), c.vrow);  // k_primal
    // k_dual: blocks of one warp or one line at least, of up to 256 threads once the lines give
    // two blocks per SM
    const int lines = nc * (d.ny / 2);
    int thr = std::max(32, tpl);
    while (thr < 256 && lines / (2 * thr / tpl) >= 2 * 152) thr *= 2;
    c.thr_dual = thr;
    c.smem_dual = thr / tpl * len * (int)sizeof(cx<T>);
    // k_primal: a thread per V values of the band's lines, more (up to 256) for the stencils of
    // narrow bands
    const int need = (nc * (d.upd_rows / 2) * tpl + 31) / 32 * 32;
    const int groups = nc * (d.upd_rows / 2) * (d.nx / 4);
    c.thr_primal = std::max(need, std::min(std::min(256, cap), (groups + 31) / 32 * 32));
    c.smem_primal = primal_smem_bytes<T>(nc, d.upd_rows, H, d.nx, len, need / tpl);
    c.fast_row = need <= cap && c.smem_primal <= smem_limit && c.smem_dual <= smem_limit;
  }
}

#define RD_BAND_COMMON(T)                                                                              \
  template cudaError_t launch_fcol<T>(const Desc&, State*, const LaunchCfg&, cudaStream_t, bool);      \
  template cudaError_t launch_dual<T>(const Desc&, State*, const LaunchCfg&, cudaStream_t, bool);      \
  template cudaError_t launch_fused<T>(const Desc&, State*, const LaunchCfg&, cudaStream_t, cudaEvent_t*, bool); \
  template cudaError_t allow_band<T>(const Desc&, const LaunchCfg&, int, bool, bool);                  \
  template void plan_band<T>(const Desc&, int, int, LaunchCfg&);
RD_BAND_COMMON(float)
RD_BAND_COMMON(double)

}  // namespace rd
