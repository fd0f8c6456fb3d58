// sweep.cuh -- the half sweeps of the two-ended pencil kernels (pencil.cu
// k_pencil, k_pencil_g): one lane runs one half of a pencil.
#pragma once

#include "internal.h"
#include "seg.cuh"

namespace ibm {

// Two lanes per pencil, Thomas in excess form from both ends ("twisted"
// elimination): the even lane eliminates rows 0 .. m-1 top-down, the odd
// lane rows n-1 .. m+1 bottom-up, and the two meet at row m = n/2, where
//   (g + a q^T_{m-1} + a q^B_{m+1}) x_m = f_m + a (y^T_{m-1} + y^B_{m+1})
// (a sum of non-negative terms, like every other pivot).  Each lane then
// substitutes back towards its end.  The serial depth per pencil is n
// instead of 2n.  Per row of a half sweep (r = 1/(a + e), w = a r = 1 - q):
//   forward   y_s = r f_s + w y_{s-1}      (y over f in the shared tile, w kept)
//   backward  x_s = y_s + w_s x_{s+1}      (straight to the spectrum)
// The excess of a pencil converges geometrically (all but the longest waves
// within some 20 to 40 rows), and once it has, the sweep goes on with constant
// r and w: 4 operations a complex row instead of 11, which is what the FP64
// sweeps are bound by.  In the working precision the recurrence then stays at one
// value or goes back and forth between two neighbours: a pencil has converged when
// e is what it was a row before, or two rows before, and from there on it takes
// the last row's r and w, or the last two rows' in turn, so that every row gets
// the pivot that the recurrence would give it.  (Without the pencils that go
// back and forth, 47 of 64 rows of 256 x 128 x 128 pass before a warp's pencils are
// all found, with them 30.  Stopping short of the fixed point makes the solve's
// error up to a tenth larger.)  The warp looks every kConvRows rows and goes on
// together.
// Measured FP64, with the reciprocal of seg.cuh in place of divisions: the
// streaming sweep of 256 x 128 x 128 74 -> 62 us (the FP64 pipe is busy for 40
// of them), the tile sweep of 96 x 65 x 64 27 -> 23 us, of the three fields of
// a stage there 30 -> 18 us.
constexpr int kConvRows = 4;  // even: a row's parity is its parity in its block

// Whether the recurrence repeats itself from the row of excess e on: e is the one
// of the last row, whose constants then stand for both parities, or of the row
// before it.
template <typename T>
__device__ __forceinline__ bool sweep_repeats(T e, T last, T back, T (&w)[2], T (&rs)[2], T (&qs)[2]) {
  if (e == last) {
    w[0] = w[1];
    rs[0] = rs[1];
    qs[0] = qs[1];
  }
  return e == last || e == back;
}

// One row of the half sweep: y, q and w from the row's e and f; returns the
// next row's e.
template <typename T>
__device__ __forceinline__ T sweep_row(T a, T g, T e, bool neg, cplx<T> f, cplx<T> &y, T &q, T &w, T &rs) {
  const T r = rcp<T>(a + e);
  q = e * r;
  w = a * r;
  rs = neg ? -r : r;
  y.x = fma(rs, f.x, w * y.x);
  y.y = fma(rs, f.y, w * y.y);
  return fma(a, q, g);
}

// len: the lane's rows (mlen >= len: the most of any lane of the warp); mask:
// the warp's lanes that take part.
template <typename T>
__device__ __forceinline__ void half_forward(cplx<T> *t, int stp, T *wc, int len, int mlen, T a, T g, T e0, bool neg,
                                             unsigned mask, cplx<T> &y, T &q) {
  constexpr int U = kConvRows;
  T e = e0, w[2], rs[2], qs[2];  // of the last even and odd row
  y = mk<T>(0, 0);
  bool conv = false;
  for (int s0 = 0; s0 < mlen; s0 += U) {
    const int nu = min(U, len - s0);
    auto constant_row = [&](T r, T wr) {
      const cplx<T> f = *t;
      y.x = fma(r, f.x, wr * y.x);
      y.y = fma(r, f.y, wr * y.y);
      *t = y;
      *wc = wr;
      t += stp;
      wc += stp;
    };
    if (conv) {
      for (int u = 0; u + 1 < nu; u += 2) {
        constant_row(rs[0], w[0]);
        constant_row(rs[1], w[1]);
      }
      if (nu > 0) q = qs[1];
      if (nu > 0 && (nu & 1)) {
        constant_row(rs[0], w[0]);
        q = qs[0];
      }
      continue;
    }
    bool same = false;
    if (nu == U) {
      cplx<T> f[U];
      T back = e, last = e;
#pragma unroll
      for (int u = 0; u < U; ++u) f[u] = t[u * stp];
#pragma unroll
      for (int u = 0; u < U; ++u, t += stp, wc += stp) {
        back = last;
        last = e;
        e = sweep_row<T>(a, g, e, neg, f[u], y, qs[u & 1], w[u & 1], rs[u & 1]);
        *t = y;
        *wc = w[u & 1];
      }
      same = sweep_repeats<T>(e, last, back, w, rs, qs);
      q = qs[1];
    } else {
      for (int u = 0; u < nu; ++u, t += stp, wc += stp) {
        e = sweep_row<T>(a, g, e, neg, *t, y, q, w[0], rs[0]);
        *t = y;
        *wc = w[0];
      }
    }
    conv = __all_sync(mask, same);
  }
}

template <typename T>
__device__ __forceinline__ void half_backward(const cplx<T> *t, int stp, const T *wc, int len, cplx<T> x,
                                              cplx<T> *gcol, long gstep) {
  t += (len - 1) * stp;
  wc += (len - 1) * stp;
  gcol += (len - 1) * gstep;
#pragma unroll 8
  for (int s = len; s > 0; --s, t -= stp, wc -= stp, gcol -= gstep) {
    const cplx<T> y = *t;
    const T w = *wc;
    x.x = fma(w, x.x, y.x);
    x.y = fma(w, x.y, y.y);
    *gcol = x;
  }
}

// Variant for grids with more pencils than the tile kernel keeps resident:
// no tile; the forward half sweep writes y_s over f_s in the spectrum itself
// (loads run U to 2U rows ahead of the recurrence), only w stays in shared
// memory, and the backward sweep reads y_s back (mostly from L2).
template <typename T> struct SweepDepth { static constexpr int U = 16; };
template <> struct SweepDepth<double> { static constexpr int U = 8; };

// (Constant rows leave no w in shared memory: kc is the first of them, wk
// those of the even and the odd ones.)
template <typename T, int U>
__device__ __forceinline__ void gl_forward(cplx<T> *col, long step, T *wc, int wstep, int len, int mlen, T a, T g,
                                           T e0, bool neg, unsigned mask, cplx<T> &y, T &q, int &kc, T (&wk)[2]) {
  constexpr int V = U / 2;  // rows between two looks
  static_assert(V % 2 == 0, "a row's parity is its parity in its block");
  cplx<T> fb[U];
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (u < len) fb[u] = col[u * step];
  T e = e0, rs[2], qs[2];
  wk[0] = wk[1] = (T)0;
  y = mk<T>(0, 0);
  kc = mlen;
  for (int s0 = 0; s0 < mlen; s0 += U) {
    cplx<T> fn[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (s0 + U + u < len) fn[u] = col[(s0 + U + u) * step];
#pragma unroll
    for (int v = 0; v < U; v += V) {
      if (s0 + v < kc) {
        bool same = false;
        T back = e, last = e;
#pragma unroll
        for (int u = v; u < v + V; ++u) {
          const int s = s0 + u;
          if (s < len) {
            back = last;
            last = e;
            e = sweep_row<T>(a, g, e, neg, fb[u], y, qs[u & 1], wk[u & 1], rs[u & 1]);
            if (u == v + V - 1) same = sweep_repeats<T>(e, last, back, wk, rs, qs);
            q = qs[u & 1];
            col[s * step] = y;
            wc[s * wstep] = wk[u & 1];
          }
        }
        if (__all_sync(mask, same)) kc = s0 + v + V;
      } else {
#pragma unroll
        for (int u = v; u < v + V; ++u) {
          const int s = s0 + u;
          if (s < len) {
            y.x = fma(rs[u & 1], fb[u].x, wk[u & 1] * y.x);
            y.y = fma(rs[u & 1], fb[u].y, wk[u & 1] * y.y);
            q = qs[u & 1];
            col[s * step] = y;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) fb[u] = fn[u];
  }
}

template <typename T, int U>
__device__ __forceinline__ void gl_backward(cplx<T> *col, long step, const T *wc, int wstep, int len, int kc,
                                            const T (&wk)[2], cplx<T> x) {
  cplx<T> yb[U];
  T wb[U];
  auto w_of = [&](int s) { return s < kc ? wc[s * wstep] : (s & 1) ? wk[1] : wk[0]; };
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int s = len - 1 - u;
    if (s >= 0) { yb[u] = col[s * step]; wb[u] = w_of(s); }
  }
  for (int s0 = len - 1; s0 >= 0; s0 -= U) {
    cplx<T> yn[U];
    T wn[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = s0 - U - u;
      if (s >= 0) { yn[u] = col[s * step]; wn[u] = w_of(s); }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = s0 - u;
      if (s >= 0) {
        x.x = fma(wb[u], x.x, yb[u].x);
        x.y = fma(wb[u], x.y, yb[u].y);
        col[s * step] = x;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) { yb[u] = yn[u]; wb[u] = wn[u]; }
  }
}

}  // namespace ibm
