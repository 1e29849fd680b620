// The whole FP32 inner PDHG solve of a small 2-D grid in ONE thread block (Section 2.1,
// Algorithm 1's inner loop, on the correction equation of FP64 defect correction): every array
// of the solve -- the unknown d, the base state u, the right-hand side r = F(u), the dual P, the
// transform array -- lives in shared memory, and the phases of an iteration are separated by
// block barriers instead of kernel boundaries.  Per iteration:
//   A  W = F~(d) by the five- or thirteen-point stencil, ||W_c||^2 by a block reduction, and the
//      stopping rule (the same rule as the multi-kernel sweeps);
//   B  forward row transform of W (pair-packed Hartley / Makhoul DCT-II), spectrum to the array;
//   C  column transform forward, times 1 / (g_hat nx ny), inverse;
//   D  inverse row transform of Y = G^{-1} W, P_{n+1} = P_n + tau_p Y, P~ = P_n + (1+omega) tau_p Y;
//   E  d_{n+1} = d_n - tau_u dF(u + d_n)^T P~.
// A launch runs the solve from the state the FP64 residual armed until it stops, then writes d
// and the solve state back to global memory.  The paper's method is unchanged: only where the
// arrays live and how the phases are synchronised differ from the band / column kernels.
#pragma once

#include <cooperative_groups.h>

#include "rd_band.cuh"

namespace rd {

constexpr int kSmallThreads = 256;

__host__ __device__ inline int up16(int b) { return (b + 15) & ~15; }

// Shared-memory bytes of the small solve of an nx x ny grid with nc components: the FP32 tables
// (twiddles, DCT rotations, eigenvalues of both axes), five real arrays (d, u, r, P, transform
// array) and the complex line buffer of the larger of the row and column passes.
__host__ __device__ inline int small_smem_bytes(int nx, int ny, int nc, bool neumann) {
  int b = 0;
  b += up16(tw_entries(nx) * 8) + (neumann ? up16(nx * 8) : 0);
  b += up16(tw_entries(ny) * 8) + (neumann ? up16(ny * 8) : 0);
  b += up16(nx * 4) + up16(ny * 4);
  b += 5 * up16(nc * nx * ny * 4);
  const int lines_r = nc * (ny / 2) * padded_len(nx), lines_c = nc * (nx / 2) * padded_len(ny);
  b += up16((lines_r > lines_c ? lines_r : lines_c) * 8);
  return b;
}

template <int K>
__device__ __forceinline__ void small_solve_body(const Desc& d, State* __restrict__ gst, Slot* slot,
                                                 unsigned char* smem) {
  if (!sweep_active(gst, slot)) return;
  constexpr bool TWO = KT<K>::two;
  constexpr int NCC = TWO ? 2 : 1;
  const int nx = d.nx, ny = d.ny, lognx = d.lognx, logny = d.logny;
  const int N = nx * ny, NC = NCC * N;
  const bool per = d.bc == BC_PERIODIC;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int hnx = nx >> 1, hny = ny >> 1, lhx = lognx - 1, lhy = logny - 1;
  const int lsx = padded_len(nx), lsy = padded_len(ny);
  // carve the shared memory (the layout of small_smem_bytes)
  unsigned char* p = smem;
  cx<float>* twx = reinterpret_cast<cx<float>*>(p);
  p += up16(tw_entries(nx) * 8);
  cx<float>* dcx = reinterpret_cast<cx<float>*>(p);
  p += per ? 0 : up16(nx * 8);
  cx<float>* twy = reinterpret_cast<cx<float>*>(p);
  p += up16(tw_entries(ny) * 8);
  cx<float>* dcy = reinterpret_cast<cx<float>*>(p);
  p += per ? 0 : up16(ny * 8);
  float* mux = reinterpret_cast<float*>(p);
  p += up16(nx * 4);
  float* muy = reinterpret_cast<float*>(p);
  p += up16(ny * 4);
  float* X = reinterpret_cast<float*>(p);
  p += up16(NC * 4);
  float* B = reinterpret_cast<float*>(p);
  p += up16(NC * 4);
  float* R = reinterpret_cast<float*>(p);
  p += up16(NC * 4);
  float* P = reinterpret_cast<float*>(p);
  p += up16(NC * 4);
  float* WY = reinterpret_cast<float*>(p);
  p += up16(NC * 4);
  cx<float>* buf = reinterpret_cast<cx<float>*>(p);

  __shared__ State s;
  __shared__ double red[32];
  __shared__ int go;
  load_table(twx, static_cast<const cx<float>*>(d.twx), tw_entries(nx));
  load_table(twy, static_cast<const cx<float>*>(d.twy), tw_entries(ny));
  if (!per) {
    load_table(dcx, static_cast<const cx<float>*>(d.dcx), nx);
    load_table(dcy, static_cast<const cx<float>*>(d.dcy), ny);
  }
  for (int k = tid; k < nx; k += nt) mux[k] = static_cast<const float*>(d.mux)[k];
  for (int k = tid; k < ny; k += nt) muy[k] = static_cast<const float*>(d.muy)[k];
  {
    const float* gX = static_cast<const float*>(d.X);
    const float* gB = static_cast<const float*>(d.base);
    const float* gR = static_cast<const float*>(d.rhs);
    const float* gP = static_cast<const float*>(d.P[0]);
    for (int q = tid; q < NC; q += nt) {
      X[q] = gX[q];
      B[q] = KT<K>::nonlinear ? gB[q] : 0.f;
      R[q] = gR[q];
      P[q] = gP[q];
    }
  }
  if (tid == 0) s = *gst;
  __syncthreads();

  const GField<float> x0{X, nx, ny, d.bc}, x1{X + N, nx, ny, d.bc};
  const GField<float> b0{B, nx, ny, d.bc}, b1{B + N, nx, ny, d.bc};
  const GField<float> t0{WY, nx, ny, d.bc}, t1{WY + N, nx, ny, d.bc};
  const float tu = float(d.tau_u), tp = float(d.tau_p), tpe = float((1.0 + d.omega) * d.tau_p);
  const float inn = float(d.inv_nn);
  for (;;) {
    // A. W = F~(d) into the row-pair lines, norms, the stopping rule
    float acc0 = 0.f, acc1 = 0.f;
    for (int q = tid; q < N; q += nt) {
      const int i = q >> lognx, j = q & (nx - 1);
      float w[2] = {0.f, 0.f};
      residual_pt<float, K, true>(d, x0, x1, b0, b1, i, j, R[q], TWO ? R[N + q] : 0.f, w);
      acc0 += w[0] * w[0];
      acc1 += w[1] * w[1];
      const int sj = per ? j : mk_slot(j, nx);
      reinterpret_cast<float*>(buf + (i >> 1) * lsx + pidx(sj))[i & 1] = w[0];
      if (TWO) reinterpret_cast<float*>(buf + (hny + (i >> 1)) * lsx + pidx(sj))[i & 1] = w[1];
    }
    const double q0 = block_sum((double)acc0, red);
    const double q1 = TWO ? block_sum((double)acc1, red) : 0.0;
    if (tid == 0) {
      measure_decide(d, &s, sqrt(q0) + (TWO ? sqrt(q1) : 0.0), slot);
      go = s.status == ST_ACTIVE;
    }
    __syncthreads();
    if (!go) break;
    // B. forward row transform; real coefficients of rows 2m, 2m+1 into WY
    {
      const cx<float>* res = block_fft_loop<float, -1>(buf, buf, NCC * hny, lognx, lsx, twx, tid, nt);
      for (int g = tid; g < ((NCC * hny) << lhx); g += nt) {
        const int line = g >> lhx, k = g & (hnx - 1);
        const int c = line / hny, m = line - c * hny;
        float* Wa = WY + c * N + (2 * m) * nx;
        float* Wb = Wa + nx;
        cx<float> ok, okp;
        fwd_post(res + line * lsx, nx, d.bc, dcx, k, ok, okp);
        Wa[k] = ok.x;
        Wb[k] = ok.y;
        if (k != 0) {
          Wa[nx - k] = okp.x;
          Wb[nx - k] = okp.y;
        } else {
          fwd_post(res + line * lsx, nx, d.bc, dcx, hnx, ok, okp);
          Wa[hnx] = ok.x;
          Wb[hnx] = ok.y;
        }
      }
      __syncthreads();
    }
    // C. column transform: forward, 1 / (g_hat nx ny), inverse (pairs of columns per line)
    {
      for (int g = tid; g < NCC * hnx * ny; g += nt) {
        const int line = g / ny, row = g - line * ny;
        const int c = line / hnx, pp = line - c * hnx;
        const float* Wr = WY + c * N + row * nx + 2 * pp;
        buf[line * lsy + pidx(per ? row : mk_slot(row, ny))] = cx<float>{Wr[0], Wr[1]};
      }
      __syncthreads();
      cx<float>* cur = block_fft_loop<float, -1>(buf, buf, NCC * hnx, logny, lsy, twy, tid, nt);
      for (int g = tid; g < ((NCC * hnx) << lhy); g += nt) {
        const int line = g >> lhy, k = g & (hny - 1);
        const int c = line / hnx, pp = line - c * hnx;
        const float c1 = float(d.gc1[c]), c2 = float(d.gc2[c]), c3 = float(d.gc3[c]);
        auto sym = [&](float mu) -> float {
          const float gg = 1.f + mu * (c1 + mu * (c2 + c3 * mu));
          return inn * __frcp_rn(gg * gg);
        };
        cx<float>* L = cur + line * lsy;
        cx<float> ok, okp;
        fwd_post(L, ny, d.bc, dcy, k, ok, okp);
        const int k2 = k == 0 ? hny : ny - k;
        if (k == 0) {
          cx<float> tt;
          fwd_post(L, ny, d.bc, dcy, hny, okp, tt);
        }
        const float ma = mux[2 * pp], mb = mux[2 * pp + 1], m1 = muy[k], m2 = muy[k2];
        L[pidx(k)] = cx<float>{ok.x * sym(ma + m1), ok.y * sym(mb + m1)};
        L[pidx(k2)] = cx<float>{okp.x * sym(ma + m2), okp.y * sym(mb + m2)};
      }
      __syncthreads();
      if (!per) {
        for (int g = tid; g < ((NCC * hnx) << lhy); g += nt) {
          const int line = g >> lhy, k = g & (hny - 1);
          cx<float>* L = cur + line * lsy;
          const cx<float> w = dcy[k];
          cx<float> zk, zkp;
          if (k == 0) {
            dct_inv_pre(L[pidx(0)], cx<float>{0.f, 0.f}, w.x, w.y, zk, zkp);
            const cx<float> Xm = L[pidx(hny)];
            const cx<float> wm = dcy[hny];
            cx<float> zm, zmp;
            dct_inv_pre(Xm, Xm, wm.x, wm.y, zm, zmp);
            L[pidx(0)] = cx<float>{zk.x, -zk.y};
            L[pidx(hny)] = cx<float>{zm.x, -zm.y};
          } else {
            dct_inv_pre(L[pidx(k)], L[pidx(ny - k)], w.x, w.y, zk, zkp);
            L[pidx(k)] = cx<float>{zk.x, -zk.y};
            L[pidx(ny - k)] = cx<float>{zkp.x, -zkp.y};
          }
        }
        __syncthreads();
      }
      cur = block_fft_loop<float, -1>(cur, cur, NCC * hnx, logny, lsy, twy, tid, nt);
      if (per) {
        post_inplace(cur, NCC * hnx, logny, lsy, d.bc, dcy);
        __syncthreads();
      }
      for (int g = tid; g < NCC * hnx * ny; g += nt) {
        const int line = g / ny, n = g - line * ny;
        const int c = line / hnx, pp = line - c * hnx;
        const cx<float> v = cur[line * lsy + pidx(n)];
        float* Wr = WY + c * N + (per ? n : mk_perm(n, ny)) * nx + 2 * pp;
        Wr[0] = v.x;
        Wr[1] = per ? v.y : -v.y;
      }
      __syncthreads();
    }
    // D. inverse row transform of Y; P_{n+1} and P~ (into WY)
    {
      if (per) {
        for (int g = tid; g < NCC * hny * nx; g += nt) {
          const int line = g >> lognx, k = g & (nx - 1);
          const int c = line / hny, m = line - c * hny;
          const float* Wa = WY + c * N + (2 * m) * nx;
          buf[line * lsx + pidx(k)] = cx<float>{Wa[k], Wa[nx + k]};
        }
      } else {
        for (int g = tid; g < ((NCC * hny) << lhx); g += nt) {
          const int line = g >> lhx, k = g & (hnx - 1);
          const int c = line / hny, m = line - c * hny;
          const float* Wa = WY + c * N + (2 * m) * nx;
          const float* Wb = Wa + nx;
          cx<float>* L = buf + line * lsx;
          const cx<float> w = dcx[k];
          cx<float> zk, zkp;
          if (k == 0) {
            dct_inv_pre(cx<float>{Wa[0], Wb[0]}, cx<float>{0.f, 0.f}, w.x, w.y, zk, zkp);
            const cx<float> Xm{Wa[hnx], Wb[hnx]};
            const cx<float> wm = dcx[hnx];
            cx<float> zm, zmp;
            dct_inv_pre(Xm, Xm, wm.x, wm.y, zm, zmp);
            L[pidx(0)] = cx<float>{zk.x, -zk.y};
            L[pidx(hnx)] = cx<float>{zm.x, -zm.y};
          } else {
            dct_inv_pre(cx<float>{Wa[k], Wb[k]}, cx<float>{Wa[nx - k], Wb[nx - k]}, w.x, w.y, zk, zkp);
            L[pidx(k)] = cx<float>{zk.x, -zk.y};
            L[pidx(nx - k)] = cx<float>{zkp.x, -zkp.y};
          }
        }
      }
      __syncthreads();
      cx<float>* cur = block_fft_loop<float, -1>(buf, buf, NCC * hny, lognx, lsx, twx, tid, nt);
      if (per) {
        post_inplace(cur, NCC * hny, lognx, lsx, d.bc, dcx);
        __syncthreads();
      }
      for (int q = tid; q < NC; q += nt) {
        const int c = q / N, r = q - c * N;
        const int i = r >> lognx, j = r & (nx - 1);
        const cx<float> v = cur[(c * hny + (i >> 1)) * lsx + pidx(per ? j : mk_slot(j, nx))];
        const float y = (i & 1) ? (per ? v.y : -v.y) : v.x;
        const float po = P[q];
        P[q] = po + tp * y;
        WY[q] = po + tpe * y;
      }
      __syncthreads();
    }
    // E. d_{n+1} = d_n - tau_u dF(u + d_n)^T P~
    for (int q = tid; q < N; q += nt) {
      const int i = q >> lognx, j = q & (nx - 1);
      float s0 = X[q], s1 = TWO ? X[N + q] : 0.f;
      if constexpr (KT<K>::nonlinear) {
        s0 += B[q];
        if constexpr (TWO) s1 += B[N + q];
      }
      float g[2] = {0.f, 0.f};
      gradT_pt<float, K>(d, t0, t1, s0, s1, i, j, g);
      X[q] -= tu * g[0];
      if constexpr (TWO) X[N + q] -= tu * g[1];
    }
    __syncthreads();
  }
  // the correction and the final solve state back to global memory
  float* gX = static_cast<float*>(d.X);
  for (int q = tid; q < NC; q += nt) gX[q] = X[q];
  if (tid == 0) {
    s.trips = (unsigned)s.n + 1u;
    s.ticket = 0u;
    *gst = s;
  }
}


// ---------------------------------------------------------------------------------------
// The same inner solve on a cluster of kClusterCtas blocks (distributed shared memory): block r
// owns rows [r R, (r+1) R) (R = ny / 8) of every array and columns [r C, (r+1) C) (C = nx / 8) of the
// spectrum.  The solve is a chain of short dependent phases, so what counts is how few barriers and
// how few instructions in a row an iteration has.  Transforms stay in registers (rd_fft.cuh, V = 4:
// all lines of a block at once); a line of up to 128 points is exchanged within a warp.  Spectra are
// stored straight into the shared memory of the block that transforms them next.  Three cluster
// barriers per iteration:
//   A  W = F~(d) on own rows, partial norms; forward row transform, coefficients to the owners of
//      their columns; partial norms to every block                           -> barrier 1
//      every block sums the partials in rank order and takes the same stopping decision
//   C  columns: forward, 1 / g_hat, inverse, results to the owners of their rows -> barrier 2
//   D  inverse row transform, P_{n+1}, P~ on own rows                        -> barrier 3
//   E  2H halo rows of P~ from their owners; d_{n+1} on own rows and, recomputed, on H halo rows.
// (The row transform runs before the decision: on the last iteration it is wasted.)
// ---------------------------------------------------------------------------------------
constexpr int kClusterCtas = 8;
constexpr int kClusterVals = 4;  // values of a line per thread: nx ny / 64 threads <= 256 per component pair

// complex entries of a line's exchange buffer (the layout of Lay for V = 4), even
__host__ __device__ inline int cluster_line_len(int n) { return (n + (n >> 4) + (n >> 6) + 2) & ~1; }
// lines of a block's buffer: those of the whole warps that transform them
__host__ __device__ inline int cluster_lines(int lines, int n) {
  const int tpl = n / kClusterVals;
  return (lines * tpl + 31) / 32 * 32 / tpl;
}

__host__ __device__ inline int cluster_smem_bytes(int nx, int ny, int nc, int H) {
  const int R = ny / kClusterCtas, C = nx / kClusterCtas;
  int b = 0;
  b += 2 * up16(nc * (R + 2 * H) * nx * 4);  // d, u with H halo rows
  b += up16(nc * (R + 4 * H) * nx * 4);      // P~ with 2H halo rows
  b += 3 * up16(nc * R * nx * 4);            // r, P, Y's row spectrum
  b += up16(cluster_lines(nc * (R / 2), nx) * cluster_line_len(nx) * 8);  // row pairs
  b += up16(cluster_lines(nc * (C / 2), ny) * cluster_line_len(ny) * 8);  // column pairs
  return b;
}

// f(LOGN) as an integral constant, for the line lengths of a cluster solve (16 .. 1024)
template <class Fn>
__device__ __forceinline__ void cluster_len(int logn, Fn f) {
  switch (logn) {
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    case 9: f(std::integral_constant<int, 9>()); break;
    case 10: f(std::integral_constant<int, 10>()); break;
    default: break;
  }
}

// Forward row transform of the block's row pairs in `buf` (natural order); coefficient k of local row
// r goes to block k / C, into its column-pair line k % C / 2 at the position of row y0 + r.
__device__ __noinline__ void cluster_rows_fwd(const Desc& d, cx<float>* buf, float* S, int nlines, int y0, int lR, int lC) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x;
  const bool per = d.bc == BC_PERIODIC;
  const int lsx = cluster_line_len(d.nx), lsy = cluster_line_len(d.ny);
  const int lhR = lR - 1, lhC = lC - 1;
  cluster_len(d.lognx, [&](auto ln) {
    constexpr int LOGN = decltype(ln)::value, V = kClusterVals;
    using F = Rf<LOGN, V>;
    using P1 = Pass<float, LOGN, V, false, 1>;
    constexpr int N = F::N;
    const int lline = tid / F::TPL, t = tid % F::TPL;
    if ((tid & ~31) >= nlines * F::TPL) return;
    auto sync = [lline] { line_sync<F::TPL>(lline); };
    cx<float>* line = buf + lline * lsx;
    cx<float> v[V];
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = line[P1::natural(t, e)];
    sync();
    rf_forward<float, LOGN, V, false>(v, line, 1, static_cast<const cx<float>*>(d.twx), t, sync);
    rf_pair<float, V>(v, t);
    if (lline >= nlines) return;
    const cx<float>* dc = static_cast<const cx<float>*>(d.dcx);
    const int c = lline >> lhR, r0 = y0 + 2 * (lline & ((1 << lhR) - 1));
    const int sa = per ? r0 : mk_slot(r0, d.ny), sb = per ? r0 + 1 : mk_slot(r0 + 1, d.ny);
    auto put = [&](int k, cx<float> w) {  // both rows' coefficient k
      float* dst = cl.map_shared_rank(S, k >> lC);
      const int kl = k & ((1 << lC) - 1);
      dst += 2 * (((c << lhC) + (kl >> 1)) * lsy) + (kl & 1);
      dst[2 * sa] = w.x;
      dst[2 * sb] = w.y;
    };
#pragma unroll
    for (int i = 0; i < V / 2; ++i) {
      const int k = rf_freq<V>(N, t, i);
      const cx<float> w = per ? cx<float>{0.f, 0.f} : ldg(dc + k);
      cx<float> o, op;
      if (i == 0 && t == 0) {
        cx<float> skip;
        pair_fwd(per, v[0], v[0], w, o, skip);
        pair_fwd(per, v[V - 1], v[V - 1], per ? w : ldg(dc + N / 2), op, skip);
        put(0, o);
        put(N / 2, op);
      } else {
        pair_fwd(per, v[i], v[V - 1 - i], w, o, op);
        put(k, o);
        put(N - k, op);
      }
    }
  });
}

// The column solve of the block's column pairs in S; the results go to the row owners' W arrays
// ([c][R][nx]).
__device__ __noinline__ void cluster_cols(const Desc& d, cx<float>* S, float* W, int nlines, int x0, int lR, int lC) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x;
  const bool per = d.bc == BC_PERIODIC;
  const int lsy = cluster_line_len(d.ny), lhC = lC - 1;
  cluster_len(d.logny, [&](auto ln) {
    constexpr int LOGN = decltype(ln)::value, V = kClusterVals;
    using F = Rf<LOGN, V>;
    using P1 = Pass<float, LOGN, V, false, 1>;
    constexpr int N = F::N;
    const int lline = tid / F::TPL, t = tid % F::TPL;
    if ((tid & ~31) >= nlines * F::TPL) return;
    auto sync = [lline] { line_sync<F::TPL>(lline); };
    cx<float>* line = S + lline * lsy;
    const bool live = lline < nlines;
    const int c = live ? lline >> lhC : 0, col = x0 + 2 * (lline & ((1 << lhC) - 1));
    const cx<float>* tw = static_cast<const cx<float>*>(d.twy);
    cx<float> v[V];
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = line[P1::natural(t, e)];
    sync();
    rf_forward<float, LOGN, V, false>(v, line, 1, tw, t, sync);
    const float* mux = static_cast<const float*>(d.mux);
    scale_pairs<float, N, V>(
        v, t, per, SymMu<float>{Symbol<float>(d, c), static_cast<const float*>(d.muy), __ldg(mux + col), __ldg(mux + col + 1)},
        static_cast<const cx<float>*>(d.dcy));
    rf_inverse<float, LOGN, V, false>(v, line, 1, tw, t, sync);
    if (!live) return;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int n = P1::natural(t, e), row = per ? n : mk_perm(n, N);
      float* dst = cl.map_shared_rank(W, row >> lR) + ((size_t)((c << lR) + (row & ((1 << lR) - 1))) << d.lognx) + col;
      *reinterpret_cast<cx<float>*>(dst) = v[e];
    }
  });
}

// Inverse row transform of the rows of W ([c][R][nx]) into the pair lines of `buf`, natural order.
__device__ __noinline__ void cluster_rows_inv(const Desc& d, const float* W, cx<float>* buf, int nlines) {
  const int tid = threadIdx.x;
  const int lsx = cluster_line_len(d.nx);
  cluster_len(d.lognx, [&](auto ln) {
    constexpr int LOGN = decltype(ln)::value, V = kClusterVals;
    using F = Rf<LOGN, V>;
    const int lline = tid / F::TPL, t = tid % F::TPL;
    if ((tid & ~31) >= nlines * F::TPL) return;
    auto sync = [lline] { line_sync<F::TPL>(lline); };
    // pair m of component c holds rows 2m, 2m + 1: line c hR + m starts at row 2 (c hR + m) of [c][R]
    row_inverse<float, LOGN, V>(d, W + (size_t)(lline < nlines ? lline : 0) * 2 * F::N, buf + lline * lsx, t, sync);
  });
}

template <int K>
__device__ __forceinline__ void small_cluster_body(const Desc& d, State* __restrict__ gst, Slot* slot,
                                                   unsigned char* smem) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  // the state is the same for every block of the cluster: all return, or none
  if (!sweep_active(gst, slot)) return;
  constexpr bool TWO = KT<K>::two;
  constexpr int NCC = TWO ? 2 : 1;
  constexpr int H = KT<K>::biharm ? 2 : 1;
  const int nx = d.nx, ny = d.ny, lognx = d.lognx;
  const size_t N = (size_t)nx * ny;
  const int lR = d.logny - 3, lC = lognx - 3;  // kClusterCtas = 8
  const int R = 1 << lR, RH = R + 2 * H, RT = R + 4 * H;
  const int y0 = rank << lR, x0 = rank << lC;
  const bool per = d.bc == BC_PERIODIC;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nrow = NCC * (R >> 1), ncol = NCC << (lC - 1);  // row and column pairs of the block
  const int lsx = cluster_line_len(nx);
  unsigned char* p = smem;
  auto take = [&p](int bytes) {
    unsigned char* q = p;
    p += up16(bytes);
    return q;
  };
  float* X = reinterpret_cast<float*>(take(NCC * RH * nx * 4));   // [c][RH][nx], own rows at H
  float* B = reinterpret_cast<float*>(take(NCC * RH * nx * 4));   // [c][RH][nx]
  float* T = reinterpret_cast<float*>(take(NCC * RT * nx * 4));   // P~ [c][RT][nx], own rows at 2H
  float* Rr = reinterpret_cast<float*>(take(NCC * R * nx * 4));   // [c][R][nx]
  float* P = reinterpret_cast<float*>(take(NCC * R * nx * 4));    // [c][R][nx]
  float* W = reinterpret_cast<float*>(take(NCC * R * nx * 4));    // Y's row spectrum [c][R][nx]
  cx<float>* buf = reinterpret_cast<cx<float>*>(take(cluster_lines(nrow, nx) * lsx * 8));
  cx<float>* S = reinterpret_cast<cx<float>*>(p);

  __shared__ State s;
  __shared__ double red[32];
  __shared__ double parts[kClusterCtas][2];
  __shared__ int go;
  const float* gB = static_cast<const float*>(d.base);
  // d and u with their halo rows (periodic wrap or half-cell mirror of the global row), r and P
  for (int q = tid; q < (NCC * RH << lognx); q += nt) {
    const int rr = q >> lognx, j = q & (nx - 1);
    const int c = TWO && rr >= RH ? 1 : 0;
    const size_t g = c * N + ((size_t)bcmap(y0 + rr - c * RH - H, ny, d.bc) << lognx) + j;
    X[q] = static_cast<const float*>(d.X)[g];
    B[q] = KT<K>::nonlinear ? gB[g] : 0.f;
  }
  for (int q = tid; q < (NCC * R << lognx); q += nt) {
    const int c = q >> (lR + lognx), rem = q & ((R << lognx) - 1);
    const size_t g = c * N + ((size_t)y0 << lognx) + rem;
    Rr[q] = static_cast<const float*>(d.rhs)[g];
    P[q] = static_cast<const float*>(d.P[0])[g];
  }
  if (tid == 0) s = *gst;
  cl.sync();  // every block runs before any stores into another's shared memory

  const Rows<float, true> x0r{X, nx, d.bc}, x1r{X + RH * nx, nx, d.bc};
  const Rows<float, true> b0r{B, nx, d.bc}, b1r{B + RH * nx, nx, d.bc};
  const Rows<float, true> t0r{T, nx, d.bc}, t1r{T + RT * nx, nx, d.bc};
  const float tu = float(d.tau_u), tp = float(d.tau_p), tpe = float((1.0 + d.omega) * d.tau_p);
  const int hR = R >> 1;
  for (;;) {
    // A. W = F~(d) on own rows into the row-pair lines, partial norms, forward row transform
    float acc0 = 0.f, acc1 = 0.f;
    for (int q = tid; q < (R << lognx); q += nt) {
      const int r = q >> lognx, j = q & (nx - 1);
      float w[2] = {0.f, 0.f};
      residual_pt<float, K, true>(d, x0r, x1r, b0r, b1r, H + r, j, Rr[q], TWO ? Rr[(R << lognx) + q] : 0.f, w);
      acc0 += w[0] * w[0];
      acc1 += w[1] * w[1];
      const int sj = per ? j : mk_slot(j, nx);
      reinterpret_cast<float*>(buf + (r >> 1) * lsx + sj)[r & 1] = w[0];
      if (TWO) reinterpret_cast<float*>(buf + (hR + (r >> 1)) * lsx + sj)[r & 1] = w[1];
    }
    const double q0 = block_sum((double)acc0, red);  // (its barriers also complete the lines)
    const double q1 = TWO ? block_sum((double)acc1, red) : 0.0;
    if (tid == 0) {
      parts[rank][0] = q0;
      parts[rank][1] = q1;
    }
    cluster_rows_fwd(d, buf, reinterpret_cast<float*>(S), nrow, y0, lR, lC);
    __syncthreads();
    if (tid < kClusterCtas && tid != rank) {
      double* pk = cl.map_shared_rank(&parts[rank][0], tid);
      pk[0] = parts[rank][0];
      pk[1] = parts[rank][1];
    }
    cl.sync();  // 1
    if (tid == 0) {
      double t0 = 0.0, t1 = 0.0;
      for (int k = 0; k < kClusterCtas; ++k) {
        t0 += parts[k][0];
        t1 += parts[k][1];
      }
      measure_decide(d, &s, sqrt(t0) + (TWO ? sqrt(t1) : 0.0), rank == 0 ? slot : nullptr);
      go = s.status == ST_ACTIVE;
    }
    // the column solve needs no decision: it overlaps with thread 0's
    cluster_cols(d, S, W, ncol, x0, lR, lC);
    cl.sync();  // 2
    if (!go) break;
    // D. inverse row transform; P_{n+1}, P~ on own rows
    cluster_rows_inv(d, W, buf, nrow);
    __syncthreads();
    for (int q = tid; q < (NCC * R << lognx); q += nt) {
      const int c = q >> (lR + lognx), r = (q >> lognx) & (R - 1), j = q & (nx - 1);
      const cx<float> v = buf[(c * hR + (r >> 1)) * lsx + (per ? j : mk_slot(j, nx))];
      const float y = (r & 1) ? v.y : v.x;
      const float po = P[q];
      P[q] = po + tp * y;
      T[((c * RT + 2 * H + r) << lognx) + j] = po + tpe * y;
    }
    cl.sync();  // 3
    // E. halo rows of P~; d_{n+1} on own and H halo rows
    for (int q = tid; q < (NCC * 4 * H << lognx); q += nt) {
      const int hh = q >> lognx, j = q & (nx - 1);
      const int c = TWO && hh >= 4 * H ? 1 : 0, hr = hh - c * 4 * H;
      const int lr = hr < 2 * H ? hr - 2 * H : R + (hr - 2 * H);  // local row -2H..-1, R..R+2H-1
      // the stencil of halo row y0 + l reads the neighbours of the row it maps to; beyond a wall the
      // mirror image of those rows is this same map
      const int g = bcmap(y0 + lr, ny, d.bc);
      const float* src = cl.map_shared_rank(T, g >> lR);
      T[((c * RT + 2 * H + lr) << lognx) + j] = src[((c * RT + 2 * H + (g & (R - 1))) << lognx) + j];
    }
    __syncthreads();
    for (int q = tid; q < (RH << lognx); q += nt) {
      const int r = q >> lognx, j = q & (nx - 1);
      const int o1 = (RH << lognx) + q;
      float s0 = X[q], s1 = TWO ? X[o1] : 0.f;
      if constexpr (KT<K>::nonlinear) {
        s0 += B[q];
        if constexpr (TWO) s1 += B[o1];
      }
      float g[2] = {0.f, 0.f};
      gradT_pt<float, K>(d, t0r, t1r, s0, s1, H + r, j, g);
      X[q] -= tu * g[0];
      if constexpr (TWO) X[o1] -= tu * g[1];
    }
    __syncthreads();
  }
  // own rows of the correction and (block 0) the final state back to global memory
  float* gX = static_cast<float*>(d.X);
  for (int q = tid; q < (NCC * R << lognx); q += nt) {
    const int c = q >> (lR + lognx), rem = q & ((R << lognx) - 1);
    gX[c * N + ((size_t)y0 << lognx) + rem] = X[((c * RH + H) << lognx) + rem];
  }
  if (rank == 0 && tid == 0) {
    s.trips = (unsigned)s.n + 1u;
    s.ticket = 0u;
    *gst = s;
  }
}

}  // namespace rd
