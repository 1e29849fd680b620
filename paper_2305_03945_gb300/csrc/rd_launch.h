// Host-side launchers of the PDHG kernels (defined in rd_kernels.cu).
#pragma once

#include <cuda_runtime.h>

#include "rd_internal.h"

namespace rd {

// Launch shape of one PDHG iteration over `ninst` instances (grid.y = instance).
struct LaunchCfg {
  int grid_bands;    // max row bands over the instances
  int grid_cols;     // max ncomp * column blocks
  int thr_res, thr_col, thr_upd;
  int smem_res, smem_col, smem_upd;
  int transform;     // 0 when G = I (no spectral solve)
  int grid_upd;      // k_upd bands (0: grid_bands)
  // kernels on the register-resident transforms (rd_band.cuh), where the sides allow them
  int fast_col;      // k_fcol in place of k_col
  int fast_row;      // k_rowfwd, k_dual, k_primal
  int vcol, vrow;    // values of a line per thread (rd_fft.cuh): 16 or 4
  int thr_fcol, smem_fcol;
  const void* tmap;  // tensor map of WY for k_fcol_tma (make_col_map); nullptr: k_fcol
  int thr_dual, smem_dual;      // k_rowfwd, k_dual
  int thr_primal, smem_primal;
};

// Equation keys of the sweep templates (kind_key maps a Desc to one).
enum KKey {
  KK_NONE_LAP = 0, KK_AC = 1, KK_CH_IMPL = 2, KK_CH_SPLIT = 3, KK_GS = 4, KK_SCHNAK = 5,
  KK_NONE_BIH = 6, KK_PCONLY = 7
};

// Per-key pieces of the sweep, specialised for every (T, K) in the rd_sweep_*.cu units (one unit
// per group of keys, so that the kernels compile in parallel): one iteration and
// the shared-memory limits of k_res and k_upd.
template <class T, int K>
cudaError_t launch_iter_kind(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, cudaEvent_t* ev);
template <class T, int K>
cudaError_t allow_kind(int optin);
// The column-transform kernel (pc: the preconditioner-only variant), rd_sweep_col.cu: k_fcol where
// the plan allows it, else k_col.
template <class T>
cudaError_t launch_col(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool pc);

// The kernels of rd_band.cuh: launchers (rd_band_*.cu), the shared-memory limits of the ones the
// plan (d, c) launches (tune: and of those the tuner tries), and the planning rule of their launch shapes.  The
// preconditioner alone (launch_rowfwd, pc = true) runs in double only.
template <class T>
cudaError_t launch_fcol(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool pc);
// Encodes the tensor map of d.WY for tiles of d.col_width columns into *map (a CUtensorMap) where
// k_fcol_tma can run them (FP32 lines of 2048 points and more); false elsewhere.
bool make_col_map(const Desc& d, const LaunchCfg& c, void* map);
// The FP64 symbol table k_fcol<double> reads through Desc::scale ([ncomp][ny][nx]).
cudaError_t launch_symbol(const Desc& d, double* table, cudaStream_t s);
template <class T>
cudaError_t launch_rowfwd(const Desc& d, const LaunchCfg& c, cudaStream_t s);
template <class T>
cudaError_t launch_dual(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool pc);
template <class T, int K>
cudaError_t launch_primal_kind(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, bool first);
template <class T, int K>
cudaError_t allow_primal_kind(const Desc& d, const LaunchCfg& c, int optin);
template <class T>
cudaError_t allow_band(const Desc& d, const LaunchCfg& c, int optin, bool primal, bool tune);
// threads of a block of these kernels at most, for the element size and values per thread
inline int band_threads_max(int elem, int vals) { return elem == 8 && vals == 16 ? 256 : 512; }
// Fills the fast_* part of c for the tiles of d (col_width, upd_rows) and the equation's halo H;
// col / row: whether k_fcol / the row kernels can run those tiles.
template <class T>
void plan_band(const Desc& d, int H, int smem_limit, LaunchCfg& c);

// Raise the dynamic shared-memory limit of the PDHG kernels; *usable receives the bytes a launch may ask.
template <class T> cudaError_t set_kernel_smem_limits(int* usable);
// One PDHG iteration (k_res, k_col, k_upd) of the solve described by d (passed by value to the
// kernels); with ev != NULL, events ev[0..3] are recorded around the three kernels.
template <class T>
cudaError_t launch_iteration(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, cudaEvent_t* ev);
// One PDHG iteration with the fused update (d.fused = 1): k_primal on U_0 (first only), the column
// kernel, k_dual and k_primal; events ev[0..3] around the three groups (k_dual and k_primal
// together).
template <class T>
cudaError_t launch_fused(const Desc& d, State* st, const LaunchCfg& c, cudaStream_t s, cudaEvent_t* ev, bool first);


// The step-level kernels (begin, FP64 residual, mass) run point_blocks(nx, ny) blocks of 256
// threads, two points per thread; d.partials must hold ncomp * point_blocks(nx, ny) doubles.
inline int point_blocks(int nx, int ny) { return (int)(((size_t)nx * ny / 2 + 255) / 256); }

cudaError_t launch_begin(const Desc* d64, State* st, const double* uk, double* rhs, double tol, int tol_kind,
                         int nblocks, cudaStream_t s);
cudaError_t launch_resid64(const Desc& hd, const Desc* d64, State* outer, State* inner, const double* u,
                           const double* rhs, double* w64, float* r32, float* u32, float* z0, float* z1, int decide,
                           double rtol, int max_outer, int nblocks, cudaStream_t s);

// Work arrays of the sixth-order functionalized Cahn-Hilliard iteration (rd_fch.cu): P~, mu(U),
// A(U) mu / A(U) Lap P~, Lap P~; each ny * nx doubles.
struct FchBuffers {
  double* Pt;
  double* M;
  double* N;
  double* Q;
};
// W = F(U) of that equation (st != NULL: also the stopping decision of the solve st, on at most
// max_blocks blocks of d.partials).
cudaError_t launch_fch_residual(const Desc& d, State* st, const FchBuffers& b, const double* U, const double* Uk,
                                double* W, int max_blocks, cudaStream_t s);
// One PDHG iteration of that equation on d (X = U, rhs = U^k, P[0] = P); dpc is the
// preconditioner-only descriptor whose X holds W (and then G^{-1} W), run on st_pc with cpc.
// Events ev[0..3] (may be NULL) around the residual, the preconditioner solve and the update.
cudaError_t launch_fch_iteration(const Desc& d, const Desc& dpc, State* st, State* st_pc, const LaunchCfg& cpc,
                                 const FchBuffers& b, int max_blocks, cudaStream_t s, cudaEvent_t* ev);

// Whether that iteration runs its fused form (eight launches; else ten with G, seven without), and the
// shared-memory limit of its kernels.
bool fch_fused(const LaunchCfg& cpc);
cudaError_t allow_fch(const Desc& d, const LaunchCfg& cpc, int optin);

// Set the thread-local detail string returned by rd_last_error().
void set_last_error(const char* msg);

// Device-side loop decision (one thread): adds `sweeps` to st->trips and clears the graph
// conditional `cond` when the solve has ended (or the launch bound is passed).
cudaError_t launch_loop_cond(State* st, unsigned long long cond, unsigned sweeps, cudaStream_t s);
cudaError_t launch_axpy_dc(double* u, const float* dlt, size_t n, State* outer, const State* inner, cudaStream_t s);
cudaError_t launch_mass(const Desc* d64, State* st, const double* u, const State* gate, int nblocks, cudaStream_t s);

}  // namespace rd
