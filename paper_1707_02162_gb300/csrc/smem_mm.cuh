// Shared-memory complex matrix products for N <= 64 (SIMT, FP64 or FP32).
#pragma once
#include "redo_internal.cuh"

namespace redo {

// ============================================================================
// Shared-memory complex matrix product  Y = A * X  (N x N, row-major)
// Thread lt of a chain owns rows ty + TY*a and columns tx + TX*c.
// ============================================================================
template <typename R, int N, int TM, int TN>
struct SmemMM {
  static constexpr int TY = N / TM, TX = N / TN, THREADS = TY * TX;
  static_assert(TY * TM == N && TX * TN == N, "tile must divide N");
  __device__ __forceinline__ static void run(const cplx<R>* __restrict__ A,
                                             const cplx<R>* __restrict__ X, int lt,
                                             cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) Y[a][c] = cmake<R>(R(0), R(0));
#pragma unroll 4
    for (int k = 0; k < N; ++k) {
      cplx<R> av[TM], xv[TN];
#pragma unroll
      for (int a = 0; a < TM; ++a) av[a] = A[(ty + TY * a) * N + k];
#pragma unroll
      for (int c = 0; c < TN; ++c) xv[c] = X[k * N + tx + TX * c];
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) cfma<R>(Y[a][c], av[a], xv[c]);
    }
  }
  // Y = A X with the terms of every 16 k summed on their own: a long FP32 sum then rounds at its own
  // size N / 16 times instead of 2 N times, and the chains of dependent additions are shorter.
  __device__ __forceinline__ static void run_blocked(const cplx<R>* __restrict__ A, const cplx<R>* __restrict__ X,
                                                     int lt, cplx<R> (&Y)[TM][TN]) {
    constexpr int KB = N < 16 ? N : 16;
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) Y[a][c] = cmake<R>(R(0), R(0));
#pragma unroll 1
    for (int k0 = 0; k0 < N; k0 += KB) {
      cplx<R> acc[TM][TN];
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) acc[a][c] = cmake<R>(R(0), R(0));
#pragma unroll
      for (int kk = 0; kk < KB; ++kk) {
        const int k = k0 + kk;
        cplx<R> av[TM], xv[TN];
#pragma unroll
        for (int a = 0; a < TM; ++a) av[a] = A[(ty + TY * a) * N + k];
#pragma unroll
        for (int c = 0; c < TN; ++c) xv[c] = X[k * N + tx + TX * c];
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
          for (int c = 0; c < TN; ++c) cfma<R>(acc[a][c], av[a], xv[c]);
      }
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) Y[a][c] = cmake<R>(Y[a][c].x + acc[a][c].x, Y[a][c].y + acc[a][c].y);
    }
  }
  // Y = A^dag X
  __device__ __forceinline__ static void run_adj(const cplx<R>* __restrict__ A,
                                                 const cplx<R>* __restrict__ X, int lt,
                                                 cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) Y[a][c] = cmake<R>(R(0), R(0));
#pragma unroll 4
    for (int k = 0; k < N; ++k) {
      cplx<R> av[TM], xv[TN];
#pragma unroll
      for (int a = 0; a < TM; ++a) {
        const cplx<R> v = A[k * N + ty + TY * a];
        av[a] = cmake<R>(v.x, -v.y);
      }
#pragma unroll
      for (int c = 0; c < TN; ++c) xv[c] = X[k * N + tx + TX * c];
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) cfma<R>(Y[a][c], av[a], xv[c]);
    }
  }
  // Q = (I - A^dag A) / 2 written to Q, computing only half of the Hermitian Gram matrix: the
  // T(T+1)/2 tiles (ty <= tx) of a square tiling go to the first threads (whole warps), each writes
  // its entries and, off the tile diagonal ty == tx, their conjugate mirrors (tile (ty, tx) and
  // tile (tx, ty) hold transposed entries).  In FP32 its diagonal is left to ns_diag.  Returns after
  // the caller's barrier is due.
  __device__ __forceinline__ static void ns_half_gram(const cplx<R>* __restrict__ A, cplx<R>* __restrict__ Q,
                                                      int lt) {
    static_assert(TY == TX && TM == TN, "square tiling");
    constexpr int T = TY, HALF = T * (T + 1) / 2;
    if (lt >= HALF) return;
    int ty = 0, rem = lt;
    while (rem >= T - ty) {
      rem -= T - ty;
      ++ty;
    }
    const int tx = ty + rem;
    cplx<R> Y[TM][TN];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) Y[a][c] = cmake<R>(R(0), R(0));
#pragma unroll 4
    for (int k = 0; k < N; ++k) {
      cplx<R> av[TM], xv[TN];
#pragma unroll
      for (int a = 0; a < TM; ++a) {
        const cplx<R> v = A[k * N + ty + TY * a];
        av[a] = cmake<R>(v.x, -v.y);
      }
#pragma unroll
      for (int c = 0; c < TN; ++c) xv[c] = A[k * N + tx + TX * c];
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) cfma<R>(Y[a][c], av[a], xv[c]);
    }
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        const int r = ty + TY * a, col = tx + TX * c;
        if (r != col || !kDiagApart)
          Q[r * N + col] = cmake<R>((r == col ? R(0.5) : R(0)) - R(0.5) * Y[a][c].x, -R(0.5) * Y[a][c].y);
        if (ty != tx) Q[col * N + r] = cmake<R>(-R(0.5) * Y[a][c].x, R(0.5) * Y[a][c].y);
      }
  }
  // Q[c][c] = (1 - sum_r |A[r][c]|^2) / 2.  A nearly unitary FP32 matrix has this near 1e-8, the
  // rounding of the plain sum: products are split by fma and added with compensation.  (FP64 takes
  // the plain sum: N threads with N dependent FP64 steps each made 512 matrices of N = 8 take 14.6 us
  // in place of 8.9.)
  static constexpr bool kDiagApart = sizeof(R) == 4;
  __device__ __forceinline__ static void ns_diag(const cplx<R>* __restrict__ A, cplx<R>* __restrict__ Q, int lt) {
    for (int c = lt; c < N; c += THREADS) {
      R s = R(-1), lo = R(0);
      for (int r = 0; r < N; ++r) {
        const cplx<R> v = A[r * N + c];
        const R h[2] = {v.x * v.x, v.y * v.y};
        lo += fma(v.x, v.x, -h[0]) + fma(v.y, v.y, -h[1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const R t = s + h[i], z = t - s;
          lo += (s - (t - z)) + (h[i] - z);
          s = t;
        }
      }
      Q[c * N + c] = cmake<R>(-R(0.5) * (s + lo), R(0));
    }
  }
  // Q = (I - A^dag A) / 2 by all threads (the caller's barrier is due afterwards)
  __device__ __forceinline__ static void ns_correction(const cplx<R>* __restrict__ A, cplx<R>* __restrict__ Q, int lt) {
    if constexpr (TY == TX && TM == TN && TM > 1) {
      ns_half_gram(A, Q, lt);                              // half the Gram tiles
    } else {
      cplx<R> Y[TM][TN];
      run_adj(A, A, lt, Y);                                // A^dag A (A read in column order)
      const int ty = lt / TX, tx = lt % TX;
#pragma unroll
      for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) {
          const int r = ty + TY * a, col = tx + TX * c;
          if (r != col || !kDiagApart)
            Q[r * N + col] = cmake<R>((r == col ? R(0.5) : R(0)) - R(0.5) * Y[a][c].x, -R(0.5) * Y[a][c].y);
        }
    }
    if constexpr (kDiagApart) ns_diag(A, Q, THREADS - 1 - lt);   // (the last threads have no half-Gram tile)
  }
  // Y = diag(p) X (a row scaling, p in FP64)
  __device__ __forceinline__ static void scale_rows(const double2* __restrict__ p,
                                                    const cplx<R>* __restrict__ X, int lt,
                                                    cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a) {
      const double2 pv = p[ty + TY * a];
      const cplx<R> pa = cmake<R>((R)pv.x, (R)pv.y);
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        Y[a][c] = cmake<R>(R(0), R(0));
        cfma<R>(Y[a][c], pa, X[(ty + TY * a) * N + tx + TX * c]);
      }
    }
  }
  __device__ __forceinline__ static void load(const cplx<R>* __restrict__ X, int lt, cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) Y[a][c] = X[(ty + TY * a) * N + tx + TX * c];
  }
  // X <- X + Y
  __device__ __forceinline__ static void add(cplx<R>* __restrict__ X, int lt, const cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) {
        cplx<R>& x = X[(ty + TY * a) * N + tx + TX * c];
        x = cmake<R>(x.x + Y[a][c].x, x.y + Y[a][c].y);
      }
  }
  __device__ __forceinline__ static void store(cplx<R>* __restrict__ X, int lt,
                                               const cplx<R> (&Y)[TM][TN]) {
    const int ty = lt / TX, tx = lt % TX;
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int c = 0; c < TN; ++c) X[(ty + TY * a) * N + tx + TX * c] = Y[a][c];
  }
};


// Square register tiles used by the one-matrix-per-CTA kernels.
template <int N> struct SqTile { static constexpr int TM = N >= 64 ? 4 : (N >= 32 ? 2 : 1); };

}  // namespace redo
