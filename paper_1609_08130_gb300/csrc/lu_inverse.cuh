// lu_inverse.cuh -- LU factors and inverse of a small matrix by one CTA.
//
// Two stages: LU with partial pivoting (FP32: lu_registers, FP64: lu_shared),
// then the inverse's columns by substitution (solve_columns).
//
// The substitution is there for what it keeps: X X^{-1} = I up to rounding in
// every column, however ill-conditioned X is, and entries near 1 rounded once.
// In-place Gauss-Jordan elimination saves its chain of steps, but its error has
// the condition number of U in it as well: with it (and a Newton step in FP32)
// the apply error of FP32 factors of first-kind matrices was 5 times larger in
// the mean and up to 1000 times in single cases, and in FP64 the inverse's error
// 1.9 times larger on second-kind blocks, up to 6 times on first-kind ones.
// What the substitution costs beside that form: factor and refined solve of the
// 64^2 grid 5.06 -> 5.26 ms, FP64 100^2 56.7 -> 57.9 ms; 32^3 21.8 -> 21.3 ms, where it
// replaces the Newton step's products.
#pragma once
#include "common.cuh"

namespace rss {

template <int NMAX = 128> struct LuShared {
  float col[2][NMAX], row[2][NMAX];
  int p[2], piv[NMAX];
};
// what lu_shared keeps (an order of up to 128)
struct LuPivots {
  int piv[128];
};

// FP32.  X: r x r row-major in shared memory, leading dimension ldl;
// overwritten by L\U with physical row piv[j] holding row j of P X's factors.
// r <= TG RB <= NMAX.  A zero or NaN pivot records DERR_NUMERIC.  s.piv is
// complete on return.
//
// The matrix is in registers: TG x TG threads (16 or 32), each with RB x RB
// entries (row ti + TG x, column tj + TG y).  A step is two barriers: the TG
// threads (a half or a whole warp) that hold column j pick the pivot (the
// largest |entry| among the rows not yet used, ties to the lowest row) and
// publish the multipliers, the threads of the pivot's row publish it, all
// update the columns of their blocks not yet done.  Bound: the chain of r
// steps (in shared memory, a warp picking the pivot and swapping rows, 39-56 us
// at r = 46-66).  The pivot's entry comes with the search: picked from the tile
// by its row it would put the tile into local memory.
template <int RB, int TG = 16, int NMAX = 128>
__device__ __forceinline__ void lu_registers(int r, float *X, int ldl, LuShared<NMAX> &s, int *err) {
  const int tid = threadIdx.x, ti = tid % TG, tj = tid / TG;
  float a[RB][RB];
#pragma unroll
  for (int x = 0; x < RB; x++)
#pragma unroll
    for (int y = 0; y < RB; y++) {
      const int i = ti + TG * x, c = tj + TG * y;
      a[x][y] = i < r && c < r ? X[i * ldl + c] : 0.f;
    }
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
        // magnitudes compared as bits (NaN above infinity)
        unsigned key = 0;
        int row = 0x7fffffff;
        float d = 0.f;
#pragma unroll
        for (int x = 0; x < RB; x++)
          if (!(used >> x & 1)) {
            const unsigned kx = __float_as_uint(a[x][yj]) & 0x7fffffffu;
            if (row == 0x7fffffff || kx > key) key = kx, row = ti + TG * x, d = a[x][yj];
          }
        const unsigned best = __reduce_max_sync(half, key);
        const int p = __reduce_min_sync(half, key == best ? row : 0x7fffffff);
        d = __shfl_sync(half, d, TG == 32 ? p % TG : (int)(threadIdx.x & 16) + p % TG);
        if (ti == 0) {
          s.p[buf] = p;
          s.piv[j] = p;
          if (!(d < 0.f || d > 0.f)) set_err(err, DERR_NUMERIC);
        }
        const float rd = 1.f / d;
#pragma unroll
        for (int x = 0; x < RB; x++) {
          const int i = ti + TG * x;
          const bool below = !(used >> x & 1) && i != p;
          const float l = below ? a[x][yj] * rd : 0.f;
          s.col[buf][i] = l;
          if (below) X[i * ldl + j] = l;
        }
      }
      __syncthreads();
      const int p = s.p[buf];
      if (ti == (p % TG)) {
        const int xp = p / TG;
        used |= 1u << xp;
#pragma unroll
        for (int y = 0; y < RB; y++) {
          if (y < yj) continue;
          const int c = tj + TG * y;
          float v = a[0][y];
#pragma unroll
          for (int x = 1; x < RB; x++) v = xp == x ? a[x][y] : v;
          s.row[buf][c] = v;
          if (c >= j && c < r) X[p * ldl + c] = v;
        }
      }
      __syncthreads();
      float u[RB];
#pragma unroll
      for (int y = 0; y < RB; y++) u[y] = y < yj ? 0.f : s.row[buf][tj + TG * y];
#pragma unroll
      for (int x = 0; x < RB; x++) {
        const float l = s.col[buf][ti + TG * x];
#pragma unroll
        for (int y = 0; y < RB; y++)
          if (y >= yj) a[x][y] -= l * u[y];
      }
    }
  }
  __syncthreads();
}

// The same in shared memory, rows swapped in place (row j of X is row j of the
// factors), piv[j] = the row at j, by the whole CTA of 32 W threads; r <= 128.
// For FP64: rank-1 updates of the rows and columns left only, a lane per
// column, take half the FP64 operations of the register form, whose warps hold
// used and unused rows side by side.
template <typename T, int W>
__device__ __forceinline__ void lu_shared(int r, T *X, int ldl, int *piv, int *err) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // per column, warp 0 picks the pivot (largest |entry|, ties to the lowest
  // row), swaps the rows and scales the column; then every warp takes rows of
  // the rank-1 update, its lanes 32 consecutive columns
  for (int i = tid; i < r; i += 32 * W) piv[i] = i;
  __syncthreads();
  for (int j = 0; j < r; j++) {
    if (warp == 0) {
      T best = (T)-1;
      int bi = r;
      for (int i = j + lane; i < r; i += 32) {
        const T v = fabs(X[i * ldl + j]);
        if (v > best) {
          best = v;
          bi = i;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const T ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) {
          best = ov;
          bi = oi;
        }
      }
      if (bi >= r) {  // NaN column: keep the diagonal, report
        bi = j;
        if (lane == 0) set_err(err, DERR_NUMERIC);
      }
      if (best == (T)0 && lane == 0) set_err(err, DERR_NUMERIC);
      if (bi != j) {
        for (int c = lane; c < r; c += 32) {
          const T t = X[j * ldl + c];
          X[j * ldl + c] = X[bi * ldl + c];
          X[bi * ldl + c] = t;
        }
        if (lane == 0) {
          const int t = piv[j];
          piv[j] = piv[bi];
          piv[bi] = t;
        }
      }
      __syncwarp();
      const T d = X[j * ldl + j];
      for (int i = j + 1 + lane; i < r; i += 32) X[i * ldl + j] /= d;
    }
    __syncthreads();
    for (int i = j + 1 + warp; i < r; i += W) {
      const T l = X[i * ldl + j];
      for (int c = j + 1 + lane; c < r; c += 32) X[i * ldl + c] -= l * X[j * ldl + c];
    }
    __syncthreads();
  }
}

// One column of the inverse, x = U^{-1} L^{-1} e_i0, by PARTS neighbouring
// lanes; every lane of the warp takes part, for its own column (live: it has
// one), iw: the smallest i0 of the warp.  row(i): row i of L\U; entry i of the
// column at x[i xs].  A row's product is split over the lanes and two sums a
// lane, the solution kept where all of them read it.
template <typename T, int PARTS, typename Row>
__device__ __forceinline__ void solve_columns(int r, int i0, int iw, bool live, Row row, T *x, int xs) {
  const int part = threadIdx.x % PARTS;
  auto dot = [&](const T *R, int l, int end) {
    T s0 = (T)0, s1 = (T)0;
    if (live) {
      l += part;
#pragma unroll 2
      for (; l + PARTS < end; l += 2 * PARTS) {
        s0 += R[l] * x[l * xs];
        s1 += R[l + PARTS] * x[(l + PARTS) * xs];
      }
      if (l < end) s0 += R[l] * x[l * xs];
    }
    s0 += s1;
#pragma unroll
    for (int o = PARTS / 2; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
    return s0;
  };
  if (live)
    for (int i = part; i < i0; i += PARTS) x[i * xs] = (T)0;
  __syncwarp();
  for (int i = iw; i < r; i++) {
    const T s = dot(row(i), i0, i);
    if (live && part == 0 && i >= i0) x[i * xs] = (i == i0 ? (T)1 : (T)0) - s;
    __syncwarp();
  }
  for (int i = r - 1; i >= 0; i--) {
    const T *R = row(i);
    const T s = dot(R, i + 1, r);
    if (live && part == 0) x[i * xs] = (x[i * xs] - s) / R[i];
    __syncwarp();
  }
}

// All r columns of X^{-1} = U^{-1} L^{-1} P into Xi (row-major, ldx) by a CTA of
// 32 W threads: column piv[i0] from e_i0, in pivot order, so that a warp's
// columns start at neighbouring rows.
template <typename T, int W, int PARTS, typename Row>
__device__ __forceinline__ void inverse_columns(int r, const int *piv, Row row, T *Xi, int ldx) {
  constexpr int PER = 32 / PARTS;  // columns a warp
  for (int iw = (threadIdx.x >> 5) * PER; iw < r; iw += W * PER) {  // uniform over the warp
    const int i0 = iw + (threadIdx.x & 31) / PARTS;
    const bool live = i0 < r;
    solve_columns<T, PARTS>(r, i0, iw, live, row, Xi + (live ? piv[i0] : 0), ldx);
  }
  __syncthreads();
}

}  // namespace rss
