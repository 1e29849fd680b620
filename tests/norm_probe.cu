// Runs one residual kernel on U_0 = 0, where W = F(0) is the right-hand side itself, and returns the
// norm its last block computed (test_gpu_norms.py).
#include <vector>

#include "rd_batch_lines.cuh"

using namespace rd;

namespace {
std::vector<void*> g_mem;
template <class T>
T* dev(size_t n) {
  void* p = nullptr;
  if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) return nullptr;
  cudaMemset(p, 0, n * sizeof(T));
  g_mem.push_back(p);
  return static_cast<T*>(p);
}
}  // namespace

// which: 0 k3_rowres (128 x 16 x 16), 1 k_primal (a line of 4096 points, 16 rows), 2 and 3 k_rowres_b on a
// 3-D slot (128 x 16 x 16) in one block and a 2-D slot (1024 x 64) in two.  *side receives nx, ny, nz.
extern "C" __attribute__((visibility("default"))) int norm_probe(int which, int* side, const float* rhs, double* norm) {
  Desc d{};
  const int sides[4][3] = {{128, 16, 16}, {4096, 16, 1}, {128, 16, 16}, {1024, 64, 1}};
  for (int k = 0; k < 3; ++k) side[k] = sides[which][k];
  if (!rhs) return 0;
  d.nx = side[0], d.ny = side[1], d.nz = side[2];
  auto lg = [](int n) { int l = 0; while ((1 << l) < n) ++l; return l; };
  d.lognx = lg(d.nx), d.logny = lg(d.ny), d.lognz = lg(d.nz);
  d.ncomp = 1, d.bc = BC_PERIODIC, d.op = OP_LAP, d.kind = RX_NONE, d.precond = 1, d.dc = 1;
  d.hx2 = d.hy2 = d.hz2 = 1.0, d.dt = 0.1, d.a = 1.0, d.tau_u = d.tau_p = 1.0;
  const size_t n = (size_t)d.nx * d.ny * d.nz;
  d.upd_rows = 4, d.nupd = d.ny / 4;
  float* r = dev<float>(n);
  d.X = dev<float>(n), d.P[0] = dev<float>(n), d.P[1] = dev<float>(n), d.WY = dev<float>(n), d.rhs = r;
  d.twx = dev<cx<float>>(d.nx), d.dcx = dev<cx<float>>(d.nx);
  d.halo = dev<float>((size_t)d.nupd * 2 * d.nx);
  d.partials = dev<double>(4096);
  State st{};
  st.status = ST_ACTIVE, st.max_iter = 1000, st.thresh = -1.0;
  Slot sl{};
  sl.inner = st, sl.phase = PH_INNER;
  State* dst = dev<State>(1);
  Slot* dsl = dev<Slot>(1);
  Desc* dd = dev<Desc>(1);
  int2* items = dev<int2>(2);
  const int2 it[2] = {{0, 0}, {0, 1}};
  d.blk3 = which == 3 ? 2 : 1;
  cudaMemcpy(r, rhs, n * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemcpy(dst, &st, sizeof(st), cudaMemcpyHostToDevice);
  cudaMemcpy(dsl, &sl, sizeof(sl), cudaMemcpyHostToDevice);
  cudaMemcpy(dd, &d, sizeof(d), cudaMemcpyHostToDevice);
  cudaMemcpy(items, it, sizeof(it), cudaMemcpyHostToDevice);
  cudaError_t e = cudaGetLastError();
  int row = 0, col = 0;
  if (which == 0) {
    using F = Rf<7, 16>;
    const int lpb = 256 / F::TPL, lines = d.nz * d.ny / 2;
    k3_rowres<float, KK_NONE_LAP, 7, 16><<<(lines + lpb - 1) / lpb, 256, lpb * Lay<float, 7, 16, false>::len * 8>>>(d, dst);
  } else if (which == 1) {
    const int len = Lay<float, 12, 16, false>::len, smem = primal_smem_bytes<float>(1, 4, 1, d.nx, len, 2);
    if (e == cudaSuccess) e = allow_smem_k(k_primal<float, KK_NONE_LAP, 12, 16>, 232448);
    k_primal<float, KK_NONE_LAP, 12, 16><<<d.nupd, 512, smem>>>(d, dst, 1);
  } else if (which == 2) {
    batch_smem<true>(d, &row, &col);
    if (e == cudaSuccess) e = allow_smem_k(k_rowres_b<KK_NONE_LAP, true>, 232448);
    k_rowres_b<KK_NONE_LAP, true><<<1, kLineThreads, row>>>(dd, dsl, items);
  } else {
    batch_smem<false>(d, &row, &col);
    if (e == cudaSuccess) e = allow_smem_k(k_rowres_b<KK_NONE_LAP, false>, 232448);
    k_rowres_b<KK_NONE_LAP, false><<<2, kLineThreads, row>>>(dd, dsl, items);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  const cudaError_t se = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = se;
  cudaMemcpy(&st, dst, sizeof(st), cudaMemcpyDeviceToHost);
  cudaMemcpy(&sl, dsl, sizeof(sl), cudaMemcpyDeviceToHost);
  *norm = which < 2 ? st.r : sl.inner.r;
  for (void* p : g_mem) cudaFree(p);
  g_mem.clear();
  return (int)e;
}
