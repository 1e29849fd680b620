// The batched line kernels of 2-D slots and their launchers.
#include "rd_batch_lines.cuh"
#include "rd_batch_lines.h"

namespace rd {

namespace {

template <int K>
void iteration(const BatchLines& L, cudaStream_t s) {
  k_rowres_b<K, false><<<L.nitems, kLineThreads, L.smem_row, s>>>(L.d32s, L.slots, L.items);
  k_axis_b<false, 1, L3_FSI><<<L.nitems, kLineThreads, L.smem_col, s>>>(L.d32s, L.slots, L.items);
  k_dual_b<false><<<L.nitems, kLineThreads, L.smem_row, s>>>(L.d32s, L.slots, L.items);
  k_primal_b<K, false><<<L.nitems, kLineThreads, 0, s>>>(L.d32s, L.slots, L.items);
}

}  // namespace

cudaError_t batch_lines2(int key, const BatchLines& L, cudaStream_t s) {
  if (L.nitems == 0) return cudaSuccess;
  switch (key) {
    case KK_NONE_LAP: iteration<KK_NONE_LAP>(L, s); break;
    case KK_AC: iteration<KK_AC>(L, s); break;
    case KK_CH_IMPL: iteration<KK_CH_IMPL>(L, s); break;
    case KK_CH_SPLIT: iteration<KK_CH_SPLIT>(L, s); break;
    case KK_NONE_BIH: iteration<KK_NONE_BIH>(L, s); break;
    case KK_GS: iteration<KK_GS>(L, s); break;
    case KK_SCHNAK: iteration<KK_SCHNAK>(L, s); break;
    default: return cudaErrorNotSupported;
  }
  return cudaGetLastError();
}

cudaError_t batch_lines2_allow(int optin) {
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto k) {
    if (e == cudaSuccess) e = allow_smem_k(k, optin);
  };
  allow(k_rowres_b<KK_NONE_LAP, false>);
  allow(k_rowres_b<KK_AC, false>);
  allow(k_rowres_b<KK_CH_IMPL, false>);
  allow(k_rowres_b<KK_CH_SPLIT, false>);
  allow(k_rowres_b<KK_NONE_BIH, false>);
  allow(k_rowres_b<KK_GS, false>);
  allow(k_rowres_b<KK_SCHNAK, false>);
  allow(k_axis_b<false, 1, L3_FSI>);
  allow(k_dual_b<false>);
  return e;
}

int batch_lines2_plan(const Desc& d, int most, int* smem_row, int* smem_col) {
  batch_smem<false>(d, smem_row, smem_col);
  const int g = batch_groups<false>(d);
  return g < most ? g : most;
}

}  // namespace rd
