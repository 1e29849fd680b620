// Register-resident line transforms: complex DFTs of 2^LOGN points in which every thread holds V
// values of a line (a line of N points has N / V threads) and the threads exchange values through
// shared memory between passes.
//
//   forward  decimation in frequency, passes of radix R_1, R_2, ..., R_P (radix V while the length
//            lasts, R_P = V / 2).  Pass i splits the remaining index j (length L_{i-1}) as
//            a L_i + j', transforms over a into the digit k_i and multiplies by
//            w_{L_{i-1}}^{j' k_i}.  A value stays at its position (k_1, ..., k_i, j'), so every
//            thread writes exactly the positions it has read and one barrier per exchange is enough
//            (the Stockham passes of rd_device.cuh need two in place, or twice the shared memory).
//   middle   after pass P a thread holds the frequencies k = k_0 + (2N/V) r for two values of k_0:
//            t and 2N/V - t.  Frequency N - k of every k is then in the same thread, so what couples
//            k and N - k (splitting a pair of real lines, the DCT-II rotations, the spectral symbol
//            of two real columns) runs in registers.
//   inverse  the same passes backwards (decimation in time).
//
// V = 16 crosses shared memory twice for lines of up to 2048 points, against a store and a load per
// Stockham pass plus the pre- and post-processing passes; V = 4 has four times the threads and a
// chain a quarter as long, for grids that do not fill the chip.
#pragma once

#include "rd_device.cuh"

namespace rd {

template <int LOGN, int V>
struct Rf {
  static_assert(LOGN >= 4 && LOGN <= 13, "lines of 16 .. 8192 points");
  static_assert(V == 4 || V == 16, "values per thread");
  static constexpr int LV = V == 16 ? 4 : 2;
  static constexpr int N = 1 << LOGN;
  static constexpr int TPL = N / V;  // threads per line
  static constexpr int P = 1 + (LOGN - (LV - 1) + LV - 1) / LV;
  // log2 of the radix of pass i (1-based)
  static __host__ __device__ constexpr int lr(int i) {
    if (i == P) return LV - 1;
    const int rem = LOGN - (LV - 1) - (i - 1) * LV;
    return rem < LV ? rem : LV;
  }
  // log2 L_i, the length left after pass i
  static __host__ __device__ constexpr int ll(int i) { return i == 0 ? LOGN : ll(i - 1) - lr(i); }
};

// Shared-memory layout of a line: where the value at position p (natural digit order) is stored.
// V = 16: an offset per value of the first digit k_1 = p / L_1 (and of the second on four-pass
// lines), so that every access of a warp falls on distinct banks where that is possible: writes and
// reads of a pass run along j' (8 or more neighbours), the reads of pass P along k_1.
//   rows (lanes along the line), FP32, N >= 256: 8 k_1 + (k_1 >> 1) is distinct modulo 16 over the
//   16 values of k_1 and differs by 8 within a pair; FP64 and short lines: k_1;
//   columns (lanes along adjacent lines first, COLS): k_1, an odd stride.
// V = 4: p + p / 16 + p / 64 (at most 4 lanes on a bank).
template <class T, int LOGN, int V, bool COLS>
struct Lay {
  using F = Rf<LOGN, V>;
  static constexpr int R1 = 1 << F::lr(1);
  static constexpr int R2 = 1 << F::lr(2);
  static __host__ __device__ constexpr int skew2(int k2) { return F::P < 4 ? 0 : (COLS ? k2 : 8 * k2 + (k2 >> 1)); }
  static __host__ __device__ constexpr int skew1(int k1) {
    return (!COLS && sizeof(T) == 4 && LOGN >= 8 ? 8 * k1 + (k1 >> 1) : k1) + (F::P < 4 ? 0 : k1 * (COLS ? 16 : 128));
  }
  // stored position of natural position p
  static __host__ __device__ __forceinline__ constexpr int at(int p) {
    if constexpr (V == 4) return p + (p >> 4) + (p >> 6);
    else if constexpr (F::P < 4) return p + skew1(p >> F::ll(1));
    else return p + skew1(p >> F::ll(1)) + skew2((p >> F::ll(2)) & (R2 - 1));
  }
  // complex entries of a line's exchange buffer, even (16-byte vectors), and for the short lines of
  // which a warp holds several such that they start on the banks the others leave free
  static constexpr int raw = at(F::N - 1) + 1;
  static constexpr int want = F::TPL < 2 ? 2 : F::TPL;
  static constexpr int len =
      COLS || F::TPL >= 16 || sizeof(T) == 8 ? (raw + 1) / 2 * 2 : (raw - want + 15) / 16 * 16 + want;
};

// Synchronise the threads of one line (TPL of them, consecutive), or the block when `block`.
template <int TPL>
__device__ __forceinline__ void line_sync(int line) {
  if constexpr (TPL <= 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(line + 1), "n"(TPL) : "memory");
}

// w^1 .. w^{R-1} of one job from a few table entries (global table, cached), with no more rounding than in the
// radix-8 passes of rd_device.cuh, whose twiddles are products of three entries at most.  Radix 16: w^1, w^2, w^8 and
// w^13 are read, and every other power is the product of two of them, or of one and another's conjugate.  (Products
// of up to four of w^1, w^2, w^4, w^8 raised the rounding floor of the FP32 inner solves: 8192^2, error of a step
// against 64 bits 7.1e-12 -> 8.4e-12.)
template <class T, int R>
__device__ __forceinline__ void rf_twiddles(const cx<T>* __restrict__ tw, int step, cx<T>* w) {
  w[1] = ldg(tw + step);
  if constexpr (R > 2) {
    w[2] = ldg(tw + 2 * step);
    w[3] = cmul(w[1], w[2]);
  }
  if constexpr (R == 8) {
    w[4] = ldg(tw + 4 * step);
    w[5] = cmul(w[1], w[4]);
    w[6] = cmul(w[2], w[4]);
    w[7] = cmul(w[3], w[4]);
  }
  if constexpr (R == 16) {
    w[8] = ldg(tw + 8 * step);
    w[13] = ldg(tw + 13 * step);  // (step < N / 16)
    w[4] = cmul(w[2], w[2]);
    w[5] = cmul_tw<T, 1>(w[13], w[8]);  // w^13 conj(w^8), ...
    w[6] = cmul_tw<T, 1>(w[8], w[2]);
    w[7] = cmul_tw<T, 1>(w[8], w[1]);
    w[9] = cmul(w[1], w[8]);
    w[10] = cmul(w[2], w[8]);
    w[11] = cmul_tw<T, 1>(w[13], w[2]);
    w[12] = cmul_tw<T, 1>(w[13], w[1]);
    w[14] = cmul(w[1], w[13]);
    w[15] = cmul(w[2], w[13]);
  }
}

// One pass's view of a thread's V values: S = V / R jobs of R values, v[s R + r]; job
// q = t + s TPL of the pass's N / R jobs.
template <class T, int LOGN, int V, bool COLS, int I>
struct Pass {
  using F = Rf<LOGN, V>;
  using Y = Lay<T, LOGN, V, COLS>;
  static constexpr int LR = F::lr(I);
  static constexpr int R = 1 << LR;
  static constexpr int S = V / R;
  static constexpr int LL = F::ll(I);  // log2 L_i
  static constexpr int L = 1 << LL;
  static constexpr bool last = I == F::P;
  // frequency index k_0 of job s of thread t in the last pass
  static __device__ __forceinline__ int k0(int t, int s) {
    if (s == 0) return t;
    return t > 0 ? 2 * F::TPL - t : F::TPL;
  }
  // natural position of element 0 of job s; element r is r L further
  static __device__ __forceinline__ int first(int t, int s) {
    if constexpr (last) {
      // digits of k_0 = k_1 + R_1 k_2 + ... into the position order k_1, k_2, ...
      const int k = k0(t, s);
      int p = 0, sh = 0;
#pragma unroll
      for (int i = 1; i < F::P; ++i) {
        p = (p << F::lr(i)) | ((k >> sh) & ((1 << F::lr(i)) - 1));
        sh += F::lr(i);
      }
      return p << LR;
    } else {
      const int q = t + s * F::TPL;
      return I == 1 ? q : ((q >> LL) << F::ll(I - 1)) | (q & (L - 1));
    }
  }
  // stored offset of element r from element 0 (V = 16: fixed)
  static __device__ __forceinline__ constexpr int off(int r) {
    return r * L + (I == 1 ? Y::skew1(r) : 0) + (I == 2 && F::P == 4 ? Y::skew2(r) : 0);
  }
  // twiddle exponent step of job s: w_{L_{i-1}}^{j'} = w_N^{j' N / L_{i-1}}
  static __device__ __forceinline__ int step(int t, int s) {
    const int q = t + s * F::TPL;
    return (q & (L - 1)) << (LOGN - F::ll(I - 1));
  }
  // `buf` is the line's buffer; consecutive positions are st entries apart (columns: adjacent
  // lines interleave)
  static __device__ __forceinline__ void load(const cx<T>* buf, int st, int t, cx<T>* v) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int n = first(t, s);
      const cx<T>* p = buf + Y::at(n) * st;
#pragma unroll
      for (int r = 0; r < R; ++r) v[s * R + r] = V == 16 ? p[off(r) * st] : buf[Y::at(n + r * L) * st];
    }
  }
  static __device__ __forceinline__ void store(cx<T>* buf, int st, int t, const cx<T>* v) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int n = first(t, s);
      cx<T>* p = buf + Y::at(n) * st;
#pragma unroll
      for (int r = 0; r < R; ++r) (V == 16 ? p[off(r) * st] : buf[Y::at(n + r * L) * st]) = v[s * R + r];
    }
  }
  static __device__ __forceinline__ void forward(cx<T>* v, const cx<T>* __restrict__ tw, int t) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      dft_reg<T, R, -1>(v + s * R);
      if constexpr (!last) {
        cx<T> w[R];
        rf_twiddles<T, R>(tw, step(t, s), w);
#pragma unroll
        for (int r = 1; r < R; ++r) v[s * R + r] = cmul_tw<T, -1>(v[s * R + r], w[r]);
      }
    }
  }
  static __device__ __forceinline__ void inverse(cx<T>* v, const cx<T>* __restrict__ tw, int t) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if constexpr (!last) {
        cx<T> w[R];
        rf_twiddles<T, R>(tw, step(t, s), w);
#pragma unroll
        for (int r = 1; r < R; ++r) v[s * R + r] = cmul_tw<T, 1>(v[s * R + r], w[r]);
      }
      dft_reg<T, R, 1>(v + s * R);
    }
  }
  // line position (natural) of value e = s R + r of thread t before pass 1 / after its inverse
  static __device__ __forceinline__ int natural(int t, int e) { return t + (e / R) * F::TPL + (e % R) * L; }
};

// Forward transform of the values v (pass-1 order) to the middle order; `sync` is the barrier of
// the threads that share the buffer.  The buffer must be free on entry.
template <class T, int LOGN, int V, bool COLS, int I = 1, class Sync>
__device__ __forceinline__ void rf_forward(cx<T>* v, cx<T>* buf, int st, const cx<T>* __restrict__ tw, int t, Sync sync) {
  Pass<T, LOGN, V, COLS, I>::forward(v, tw, t);
  if constexpr (I < Rf<LOGN, V>::P) {
    Pass<T, LOGN, V, COLS, I>::store(buf, st, t, v);
    sync();
    Pass<T, LOGN, V, COLS, I + 1>::load(buf, st, t, v);
    rf_forward<T, LOGN, V, COLS, I + 1>(v, buf, st, tw, t, sync);
  }
}

// Inverse transform from the middle order to pass-1 order.  On entry the positions this thread
// writes first are the ones it read last in rf_forward (or the buffer is free).
template <class T, int LOGN, int V, bool COLS, int I = Rf<LOGN, V>::P, class Sync>
__device__ __forceinline__ void rf_inverse(cx<T>* v, cx<T>* buf, int st, const cx<T>* __restrict__ tw, int t, Sync sync) {
  Pass<T, LOGN, V, COLS, I>::inverse(v, tw, t);
  if constexpr (I > 1) {
    Pass<T, LOGN, V, COLS, I>::store(buf, st, t, v);
    sync();
    Pass<T, LOGN, V, COLS, I - 1>::load(buf, st, t, v);
    rf_inverse<T, LOGN, V, COLS, I - 1>(v, buf, st, tw, t, sync);
  }
}

// The middle order as pairs: after rf_pair, v[i] holds frequency k(i) and v[V - 1 - i] frequency
// N - k(i), i = 0 .. V/2 - 1; thread 0 holds the self-paired frequencies 0 (v[0]) and N/2
// (v[V - 1]) as its pair 0.  Its own inverse is rf_unpair.
template <int V>
__device__ __forceinline__ int rf_freq(int N, int t, int i) {
  constexpr int R = V / 2;
  return i * (N / R) + (t > 0 ? t : (i < R / 2 ? 0 : N / V - N / 2));
}
template <class T, int V>
__device__ __forceinline__ void rf_pair(cx<T>* v, int t) {
  constexpr int R = V / 2;
  if (t == 0) {
    cx<T> u[V];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      u[i] = i < R / 2 ? v[i] : v[R + i - R / 2];
      u[V - 1 - i] = i == 0 ? v[R / 2] : (i < R / 2 ? v[R - i] : v[R + R - 1 - (i - R / 2)]);
    }
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = u[i];
  }
}
template <class T, int V>
__device__ __forceinline__ void rf_unpair(cx<T>* v, int t) {
  constexpr int R = V / 2;
  if (t == 0) {
    cx<T> u[V];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      u[i < R / 2 ? i : R + i - R / 2] = v[i];
      u[i == 0 ? R / 2 : (i < R / 2 ? R - i : R + R - 1 - (i - R / 2))] = v[V - 1 - i];
    }
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = u[i];
  }
}

// ---------------------------------------------------------------------------------------
// what couples frequencies k and N - k of a pair of real lines (a in .x, b in .y)
// ---------------------------------------------------------------------------------------

// complex DFT values z = Z(k), zp = Z(N-k) -> real coefficients (a, b) at k and at N - k:
// Hartley (periodic), or the DCT-II with (c, s) = (cos, sin)(pi k / 2N) (Neumann).
template <class T>
__device__ __forceinline__ void pair_fwd(bool per, cx<T> z, cx<T> zp, cx<T> w, cx<T>& ok, cx<T>& okp) {
  const T sx = z.x + zp.x, dx = z.x - zp.x, sy = z.y + zp.y, dy = z.y - zp.y;
  if (per) {
    ok = cx<T>{T(0.5) * (sx - dy), T(0.5) * (sy + dx)};
    okp = cx<T>{T(0.5) * (sx + dy), T(0.5) * (sy - dx)};
  } else {
    const T c = T(0.5) * w.x, s = T(0.5) * w.y;
    ok = cx<T>{c * sx + s * dy, c * sy - s * dx};
    okp = cx<T>{s * sx - c * dy, s * sy + c * dx};
  }
}

// real coefficients (a, b) at k and N - k -> the values whose inverse complex DFT (unnormalised)
// is the pair of real lines (Neumann: in Makhoul order, times N).  On the self-paired frequencies
// of a DCT the partner of k = 0 is 0.
template <class T>
__device__ __forceinline__ void pair_inv(bool per, cx<T> h, cx<T> hp, cx<T> w, cx<T>& z, cx<T>& zp) {
  if (per) {
    const T sx = h.x + hp.x, dx = h.x - hp.x, sy = h.y + hp.y, dy = h.y - hp.y;
    z = cx<T>{T(0.5) * (sx + dy), T(0.5) * (sy - dx)};
    zp = cx<T>{T(0.5) * (sx - dy), T(0.5) * (sy + dx)};
  } else {
    dct_inv_pre(h, hp, w.x, w.y, z, zp);
  }
}

}  // namespace rd
