// Launchers of the batched line kernels (rd_batch_lines.cuh), 2-D and 3-D slots.
#pragma once

#include <cuda_runtime.h>

#include "rd_internal.h"

namespace rd {

// One launch of each kernel of a PDHG iteration over the (slot, block) list `items`.
struct BatchLines {
  const Desc* d32s;
  Slot* slots;
  const int2* items;
  int nitems;
  int smem_row, smem_col;  // the largest any listed slot needs
};
cudaError_t batch_lines2(int key, const BatchLines& L, cudaStream_t s);
cudaError_t batch_lines3(int key, const BatchLines& L, cudaStream_t s);
cudaError_t batch_lines2_allow(int optin);
cudaError_t batch_lines3_allow(int optin);
// Blocks of slot d in each kernel (at most `most`) and the shared memory of its row and column kernels.
int batch_lines2_plan(const Desc& d, int most, int* smem_row, int* smem_col);
int batch_lines3_plan(const Desc& d, int most, int* smem_row, int* smem_col);

}  // namespace rd
