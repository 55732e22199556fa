// lu_inverse.cuh -- LU factors and inverse of a small matrix by one CTA, the
// matrix in registers.
//
// Gauss-Jordan elimination with partial pivoting, in place: at step j the row
// p with the largest |entry| of column j among the rows not yet used is
// scaled by its pivot and eliminated from every other row, column j being
// replaced by the multipliers.  The rows not yet used go through exactly the
// steps of an LU factorization, so their multipliers and the pivot rows are L
// and U; after r steps the registers hold the inverse (of P X, rows and columns
// in pivot order).  TG x TG threads (16 or 32), each with RB x RB entries (row
// ti + TG x, column tj + TG y).  A step is two barriers: the TG threads (a half
// or a whole warp) that hold column j pick the pivot and publish the column,
// the threads of row p publish the row, all update.
//
// Bound: the chain of r steps.  Separate stages (LU in shared memory, 39-56 us
// at r = 46-66, and a triangular solve per column for the inverse, 41-58 us)
// were most of an upper level's elimination launch (elimination of the 64^2 grid
// 2.24 -> 1.48 ms with this form, of the 100^2 grid in FP64 12.9 -> 10.1).
#pragma once
#include "common.cuh"

namespace rss {

template <typename T, int NMAX = 128> struct LuInvShared {
  T col[2][NMAX], row[2][NMAX], rd[2];
  int p[2];
  int piv[NMAX], pos[NMAX];
};

// X: r x r row-major in shared memory, leading dimension ldl; overwritten by
// L\U with physical row piv[j] holding row j of P X's factors.  store(i, c, v):
// entry (i, c) of X^{-1}.  r <= TG RB <= NMAX.  A zero or NaN pivot records
// DERR_NUMERIC.  s.piv, s.pos (its inverse) are complete on return.
template <typename T, int RB, int TG = 16, int NMAX = 128, typename Store>
__device__ __forceinline__ void lu_inverse(int r, T *X, int ldl, LuInvShared<T, NMAX> &s, int *err, Store store) {
  const int tid = threadIdx.x, ti = tid % TG, tj = tid / TG;
  T a[RB][RB];
#pragma unroll
  for (int x = 0; x < RB; x++)
#pragma unroll
    for (int y = 0; y < RB; y++) {
      const int i = ti + TG * x, c = tj + TG * y;
      a[x][y] = i < r && c < r ? X[i * ldl + c] : (T)0;
    }
  // FP64: rows and columns in use, in steps of TG; the products of the rest would
  // take the FP64 unit (r = 60 in 96 x 96: more than twice the operations;
  // elimination of the 100^2 grid 8.5 -> 7.7 ms).  In FP32 the branches cost more
  // than the products (64^2 grid 1.38 -> 1.52 ms).
  const int nx = sizeof(T) == 8 ? (r + TG - 1) / TG : RB;
  unsigned used = 0;  // bit x: row ti + TG x has been a pivot (or does not exist)
#pragma unroll
  for (int x = 0; x < RB; x++)
    if (ti + TG * x >= r) used |= 1u << x;
#pragma unroll
  for (int yj = 0; yj < RB; yj++) {
    for (int jj = 0; jj < TG; jj++) {
      const int j = TG * yj + jj, buf = j & 1;
      if (j >= r) break;
      if (tj == jj) {
        const unsigned half = TG == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
        // magnitudes compared in FP32 (NaN above infinity), ties to the lowest row
        unsigned key = 0;
        int row = 0x7fffffff;
#pragma unroll
        for (int x = 0; x < RB; x++)
          if (!(used >> x & 1)) {
            const unsigned kx = __float_as_uint((float)a[x][yj]) & 0x7fffffffu;
            if (row == 0x7fffffff || kx > key) key = kx, row = ti + TG * x;
          }
        const unsigned best = __reduce_max_sync(half, key);
        const int p = __reduce_min_sync(half, key == best ? row : 0x7fffffff);
        if (ti == 0) {
          s.p[buf] = p;
          s.piv[j] = p;
          s.pos[p] = j;
        }
#pragma unroll
        for (int x = 0; x < RB; x++) s.col[buf][ti + TG * x] = a[x][yj];
        if (ti == (p % TG)) {  // the pivot's reciprocal
          const int xp = p / TG;
          T d = a[0][yj];
#pragma unroll
          for (int x = 1; x < RB; x++) d = xp == x ? a[x][yj] : d;
          if (!(d < (T)0 || d > (T)0)) set_err(err, DERR_NUMERIC);
          s.rd[buf] = (T)1 / d;
        }
      }
      __syncthreads();
      const int p = s.p[buf];
      if (ti == (p % TG)) {
        const int xp = p / TG;
        used |= 1u << xp;
#pragma unroll
        for (int y = 0; y < RB; y++) {
          if (y >= nx) break;
          const int c = tj + TG * y;
          T v = a[0][y];
#pragma unroll
          for (int x = 1; x < RB; x++) v = xp == x ? a[x][y] : v;
          s.row[buf][c] = v;
          if (c >= j && c < r) X[p * ldl + c] = v;
        }
      }
      __syncthreads();
      const T rd = s.rd[buf];
      T rs[RB];  // the scaled pivot row, 1 / pivot in column j
#pragma unroll
      for (int y = 0; y < RB; y++)
        if (y < nx) rs[y] = (y == yj && tj == jj) ? rd : s.row[buf][tj + TG * y] * rd;
#pragma unroll
      for (int x = 0; x < RB; x++) {
        if (x >= nx) break;
        const int i = ti + TG * x;
        const T f = s.col[buf][i];
        if (tj == jj) {
          if (!(used >> x & 1)) X[i * ldl + j] = f * rd;
          a[x][yj] = (T)0;
        }
        if (i == p) {
#pragma unroll
          for (int y = 0; y < RB; y++)
            if (y < nx) a[x][y] = rs[y];
        } else {
#pragma unroll
          for (int y = 0; y < RB; y++)
            if (y < nx) a[x][y] -= f * rs[y];
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < RB; x++)
#pragma unroll
    for (int y = 0; y < RB; y++) {
      const int i = ti + TG * x, c = tj + TG * y;
      if (i < r && c < r) store(s.pos[i], s.piv[c], a[x][y]);
    }
  __syncthreads();
}

// One Newton step on an FP32 inverse, X += X (I - A X), in FP32: in-place
// elimination alone doubled the factor's apply error against triangular
// solves, with the step it is theirs or less.  A: r x r row-major (ld lda),
// overwritten by the residual; X: column-major (ld ldx).  Same thread layout as
// lu_inverse, r <= 16 RB.
template <int RB> __device__ __forceinline__ void newton_inverse(int r, float *A, int lda, float *X, int ldx) {
  const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
  float out[RB][RB];
  for (int pass = 0; pass < 2; pass++) {
#pragma unroll
    for (int x = 0; x < RB; x++)
#pragma unroll
      for (int y = 0; y < RB; y++) out[x][y] = pass == 0 && ti + 16 * x == tj + 16 * y ? 1.f : 0.f;
    // pass 0: I - A X, pass 1: X R; rows past the matrix repeat its last one
    const float *ap[RB], *bp[RB];
    const int sa = pass == 0 ? 1 : ldx, sb = pass == 0 ? 1 : lda;
#pragma unroll
    for (int x = 0; x < RB; x++) {
      const int i = min(ti + 16 * x, r - 1), c = min(tj + 16 * x, r - 1);
      ap[x] = pass == 0 ? A + i * lda : X + i;
      bp[x] = pass == 0 ? X + c * ldx : A + c;
    }
    const float sign = pass == 0 ? -1.f : 1.f;
#pragma unroll 1
    for (int l = 0; l < r; l++) {
      float av[RB], bv[RB];
#pragma unroll
      for (int x = 0; x < RB; x++) av[x] = sign * ap[x][l * sa], bv[x] = bp[x][l * sb];
#pragma unroll
      for (int x = 0; x < RB; x++)
#pragma unroll
        for (int y = 0; y < RB; y++) out[x][y] = fmaf(av[x], bv[y], out[x][y]);
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < RB; x++)
#pragma unroll
      for (int y = 0; y < RB; y++) {
        const int i = ti + 16 * x, c = tj + 16 * y;
        if (i < r && c < r) {
          if (pass == 0) A[i * lda + c] = out[x][y];
          else X[i + c * ldx] += out[x][y];
        }
      }
    __syncthreads();
  }
}

}  // namespace rss
