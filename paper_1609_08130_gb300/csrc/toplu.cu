// toplu.cu -- the dense top blocks (Sec. 3.3.3) of one or several problems: LU
// with partial pivoting and the inverse the solves multiply by.
//
// Right-looking blocked LU, every problem's block in each launch (grid
// dimension), a panel per step:
//   k_top_panel  one CTA per problem: a thread holds its rows of the panel in
//                registers; a column step is one barrier (every warp publishes
//                its best row, every warp picks the winner by a reduction over
//                the warps' keys); rows are moved once at the end;
//   k_top_trsm   the panel's row moves on the other columns, U12;
//   k_top_trail  A22 -= L21 U12.
// Each launch is a programmatic dependent of the one before.  Bound: the chain
// of n column steps.  Measured, LU and inverse: FP32 n = 305 1.29 -> 0.46 ms (a
// panel in shared memory with three barriers a column before), n = 1600
// 9.5 -> 5.7 ms (the LU alone before), FP64 n = 313 2.78 -> 1.49 ms, 32 problems of
// n = 310 10.4 -> 1.4 ms (one CTA each, unblocked, before).  A column's
// pivot row in 16-byte pieces and the winner by a warp reduction instead of 16
// reads and compares a thread are 0.08, 0.5 and 0.06 ms of it.
//
// k_top_inverse forms W = U^{-1} L^{-1}: the diagonal blocks' inverses first,
// then a CTA per group of columns goes through the row blocks of L and of U
// with its columns in shared memory.  Then a solve's D^{-1} on the top block is
// a matrix-vector product, or four of them with the correction of k_top_gemv,
// instead of 2 n dependent row steps (2.45 ms a solve at n = 1600; the product
// alone 10 us).
#include <algorithm>

#include "internal.h"

namespace rss {

namespace {

constexpr int PT = 512;   // panel threads
constexpr int LBMAX = 32; // widest panel
constexpr int DB = 32;    // diagonal blocks of the inverse

__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// 16 bytes of a pivot row
template <typename T> struct alignas(16) Pack {
  static constexpr int N = 16 / sizeof(T);
  T x[N];
};

// A magnitude's order as 32 bits, NaN above infinity: FP32 entries as they are,
// FP64 ones by their upper word (20 bits of the mantissa, the whole range of the
// exponent; a conversion to FP32 would make zeros of what is below 1e-45 and
// infinities of what is above 3e38), a zero below every other number.
__device__ __forceinline__ unsigned pivot_key(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned pivot_key(double v) {
  return ((unsigned)__double2hiint(v) & 0x7fffffffu) | (__double2loint(v) != 0);
}

// a panel's row moves: position dst[e] (from the panel's first row) takes the
// row that was at src[e]
struct Moves {
  int cnt, dst[2 * LBMAX], src[2 * LBMAX];
};

}  // namespace

// Panel of NB columns at kb, rows kb.. n-1, thread t holding rows t + PT q.
// Pivot: largest |entry| (by pivot_key), rows moved at the end as the
// sequence of interchanges would.
template <typename T, int NB, int RPT>
__global__ void __launch_bounds__(PT) k_top_panel(T *LUall, const int64_t *loff, const int *tn, int *pivall,
                                                  const int64_t *toff, int kb, Moves *moves, int *err) {
  constexpr int NW = PT / 32, VW = Pack<T>::N;
  __shared__ unsigned s_key[2][NW];
  __shared__ int s_idx[2][NW], s_prow[NB], s_at[PT * RPT], s_where[PT * RPT];
  __shared__ __align__(16) T s_row[2][NW][NB];
  __shared__ T s_rd;
  pdl_enter();
  const int p = blockIdx.x, n = tn[p];
  if (kb >= n) return;
  T *A = LUall + loff[p];
  int *piv = pivall + toff[p];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int h = n - kb, nb = min(NB, h);
  T a[RPT][NB];
#pragma unroll
  for (int q = 0; q < RPT; q++) {
    const int i = tid + PT * q;
#pragma unroll
    for (int c = 0; c < NB; c++) a[q][c] = i < h && c < nb ? A[(int64_t)(kb + i) * n + kb + c] : (T)0;
    s_at[i] = i;
    s_where[i] = i;
  }
  unsigned used = 0;
#pragma unroll
  for (int q = 0; q < RPT; q++)
    if (tid + PT * q >= h) used |= 1u << q;
#pragma unroll
  for (int j = 0; j < NB; j++) {
    if (j < nb) {
      const int buf = j & 1;
      unsigned key = 0;
      int qb = -1;
#pragma unroll
      for (int q = 0; q < RPT; q++)
        if (!(used >> q & 1)) {
          const unsigned k = pivot_key(a[q][j]);
          if (qb < 0 || k > key) key = k, qb = q;
        }
      // a thread with no row left offers nothing (zero keys of real rows win)
      const unsigned have = __ballot_sync(0xffffffffu, qb >= 0);
      const unsigned kw = __reduce_max_sync(0xffffffffu, key);
      const unsigned at = __ballot_sync(0xffffffffu, qb >= 0 && key == kw);
      if (have == 0) {
        if (lane == 0) s_idx[buf][warp] = -1;
      } else if (lane == __ffs(at) - 1) {
        s_key[buf][warp] = kw;
        s_idx[buf][warp] = tid + PT * qb;
#pragma unroll
        for (int c0 = j / VW * VW; c0 < NB; c0 += VW) {
          Pack<T> v;
#pragma unroll
          for (int c = 0; c < VW; c++) {
            v.x[c] = a[0][c0 + c];
#pragma unroll
            for (int q = 1; q < RPT; q++) v.x[c] = qb == q ? a[q][c0 + c] : v.x[c];
          }
          *reinterpret_cast<Pack<T> *>(&s_row[buf][warp][c0]) = v;
        }
      }
      __syncthreads();
      // the first of the warps' largest keys (0: a warp with no row left)
      const int wi = s_idx[buf][lane % NW];
      const unsigned wk = wi >= 0 ? s_key[buf][lane % NW] + 1u : 0u;
      const int bw = (__ffs(__ballot_sync(0xffffffffu, wk == __reduce_max_sync(0xffffffffu, wk))) - 1) % NW;
      const int pr = __shfl_sync(0xffffffffu, wi, bw);
      const T *row = s_row[buf][bw];
      T rd;
      if (sizeof(T) == 8) {  // one reciprocal on the FP64 pipe instead of one a warp
        if (tid == 0) s_rd = (T)1 / row[j];
        __syncthreads();
        rd = s_rd;
      } else {
        rd = (T)1 / row[j];
      }
      if (tid == 0) {
        s_prow[j] = pr;
        if (!(row[j] > (T)0 || row[j] < (T)0)) set_err(err, DERR_NUMERIC);
      }
      T l[RPT];
#pragma unroll
      for (int q = 0; q < RPT; q++) {
        if (tid + PT * q == pr) used |= 1u << q;
        l[q] = (T)0;
        if (!(used >> q & 1)) a[q][j] = l[q] = a[q][j] * rd;
      }
      auto update = [&](int q, int c0) {
        const Pack<T> v = *reinterpret_cast<const Pack<T> *>(row + c0);
#pragma unroll
        for (int c = 0; c < VW; c++)
          if (c0 + c > j) a[q][c0 + c] -= l[q] * v.x[c];
      };
      // FP64 row by row, so that a warp without rows left issues nothing
      if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int q = 0; q < RPT; q++)
          if (!(used >> q & 1)) {
#pragma unroll
            for (int c0 = (j + 1) / VW * VW; c0 < NB; c0 += VW) update(q, c0);
          }
      } else {
#pragma unroll
        for (int c0 = (j + 1) / VW * VW; c0 < NB; c0 += VW)
#pragma unroll
          for (int q = 0; q < RPT; q++)
            if (!(used >> q & 1)) update(q, c0);
      }
    }
  }
  __syncthreads();
  if (tid == 0)
    for (int j = 0; j < nb; j++) {  // interchange positions j and the pivot row's
      const int r = s_prow[j], x = s_where[r], o = s_at[j];
      s_at[x] = o;
      s_where[o] = x;
      s_at[j] = r;
      s_where[r] = j;
    }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < RPT; q++) {
    const int i = tid + PT * q;
    if (i < h) {
      T *o = A + (int64_t)(kb + s_where[i]) * n + kb;
#pragma unroll
      for (int c = 0; c < NB; c++)
        if (c < nb) o[c] = a[q][c];
    }
  }
  // the moves, for k_top_trsm, and on the permutation
  Moves &M = moves[p];
  int dst = -1, src = 0, pv = 0;
  if (tid < 2 * nb) {
    dst = tid < nb ? tid : s_prow[tid - nb];
    if (tid >= nb && dst < nb) dst = -1;  // listed by its position
    if (dst >= 0) {
      src = s_at[dst];
      M.dst[tid] = dst;
      M.src[tid] = src;
      pv = kb == 0 ? src : piv[kb + src];
    } else {
      M.dst[tid] = -1;
    }
  }
  if (tid == 0) M.cnt = 2 * nb;
  if (kb == 0)
    for (int i = tid; i < n; i += PT) piv[i] = i;
  __syncthreads();
  if (dst >= 0) piv[kb + dst] = pv;
}

// The panel's row moves on every column outside it (all loads of a column
// before its stores), then U12 = L11^{-1} A12 right of it; a thread per column.
template <typename T, int NB>
__global__ void __launch_bounds__(64) k_top_trsm(T *LUall, const int64_t *loff, const int *tn, int kb,
                                                const Moves *moves) {
  __shared__ T s_l[NB][NB + 1];
  __shared__ T s_v[2 * NB][64];
  __shared__ int s_dst[2 * NB], s_src[2 * NB];
  pdl_enter();
  const int p = blockIdx.y, n = tn[p], tid = threadIdx.x;
  if (kb >= n) return;
  T *A = LUall + loff[p];
  const int nb = min(NB, n - kb), cnt = 2 * nb;
  const Moves &M = moves[p];
  if (tid < cnt) {
    s_dst[tid] = M.dst[tid];
    s_src[tid] = M.dst[tid] >= 0 ? M.src[tid] : 0;
  }
  for (int e = tid; e < nb * nb; e += 64) s_l[e / nb][e % nb] = A[(int64_t)(kb + e / nb) * n + kb + e % nb];
  __syncthreads();
  const int cc = blockIdx.x * 64 + tid;
  if (cc >= n || (cc >= kb && cc < kb + nb)) return;
  T *col = A + (int64_t)kb * n + cc;
#pragma unroll 16
  for (int e = 0; e < cnt; e++) s_v[e][tid] = col[(int64_t)s_src[e] * n];
#pragma unroll 4
  for (int e = 0; e < cnt; e++)
    if (s_dst[e] >= nb || (s_dst[e] >= 0 && cc < kb)) col[(int64_t)s_dst[e] * n] = s_v[e][tid];
  if (cc < kb) return;
  // rows 0 .. nb-1 after the moves are the first nb entries
  T x[NB];
#pragma unroll
  for (int i = 0; i < NB; i++) {
    if (i < nb) {
      T s0 = s_v[i][tid], s1 = (T)0;
#pragma unroll
      for (int l = 0; l < i; l++) (l & 1 ? s1 : s0) -= s_l[i][l] * x[l];
      x[i] = s0 + s1;
      col[(int64_t)i * n] = x[i];
    }
  }
}

// A22 -= L21 U12 (64 x 64 tiles, inner dimension NB)
template <typename T, int NB>
__global__ void __launch_bounds__(256) k_top_trail(T *LUall, const int64_t *loff, const int *tn, int kb) {
  __shared__ T Ls[NB][64 + 1], Us[NB][64 + 1];
  pdl_enter();
  const int p = blockIdx.z, n = tn[p];
  const int s0 = kb + NB, i0 = s0 + blockIdx.y * 64, c0 = s0 + blockIdx.x * 64;
  if (i0 >= n || c0 >= n) return;
  T *A = LUall + loff[p];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  T cur[4][4];
#pragma unroll
  for (int x = 0; x < 4; x++)
#pragma unroll
    for (int y = 0; y < 4; y++) {
      const int i = i0 + ty + 16 * x, c = c0 + tx + 16 * y;
      cur[x][y] = i < n && c < n ? A[(int64_t)i * n + c] : (T)0;
    }
#pragma unroll
  for (int e = tid; e < 64 * NB; e += 256) {
    const int i = e / NB, l = e % NB;
    Ls[l][i] = i0 + i < n ? A[(int64_t)(i0 + i) * n + kb + l] : (T)0;
    const int l2 = e / 64, c2 = e % 64;
    Us[l2][c2] = c0 + c2 < n ? A[(int64_t)(kb + l2) * n + c0 + c2] : (T)0;
  }
  __syncthreads();
  T acc[4][4] = {};
#pragma unroll 8
  for (int l = 0; l < NB; l++) {
    T lv[4], uv[4];
#pragma unroll
    for (int x = 0; x < 4; x++) lv[x] = Ls[l][ty + 16 * x];
#pragma unroll
    for (int y = 0; y < 4; y++) uv[y] = Us[l][tx + 16 * y];
#pragma unroll
    for (int x = 0; x < 4; x++)
#pragma unroll
      for (int y = 0; y < 4; y++) acc[x][y] += lv[x] * uv[y];
  }
#pragma unroll
  for (int x = 0; x < 4; x++)
#pragma unroll
    for (int y = 0; y < 4; y++) {
      const int i = i0 + ty + 16 * x, c = c0 + tx + 16 * y;
      if (i < n && c < n) A[(int64_t)i * n + c] = cur[x][y] - acc[x][y];
    }
}

template <typename K, typename... A>
static void launch_pdl(K kernel, dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, args...);
  count_launch();
}

template <typename T, int NB, int RPT>
static void lu_step(T *LU, const int64_t *loff, int *piv, const int64_t *toff, const int *tn, int nprob, int maxn,
                    int kb, Moves *moves, int *err, cudaStream_t st) {
  launch_pdl(k_top_panel<T, NB, RPT>, dim3(nprob), PT, 0, st, LU, loff, tn, piv, toff, kb, moves, err);
  if (maxn <= NB) return;
  launch_pdl(k_top_trsm<T, NB>, dim3((maxn + 63) / 64, nprob), 64, 0, st, LU, loff, tn, kb, (const Moves *)moves);
  const int rem = maxn - kb - NB;
  if (rem > 0) {
    const int t = (rem + 63) / 64;
    launch_pdl(k_top_trail<T, NB>, dim3(t, t, nprob), 256, 0, st, LU, loff, tn, kb);
  }
}

int64_t top_lu_scratch_bytes(int nprob) { return (int64_t)nprob * sizeof(Moves); }
int top_lu_limit(int elem) { return elem == 4 ? 4096 : 2048; }

// The panel's width is what its rows leave of the register file: 32 columns up
// to 1024 rows (FP64: 512), 16 up to 2048 (1024), 8 up to 4096 (2048).
template <typename T>
void launch_top_lu(T *LU, const int64_t *loff, int *piv, const int64_t *toff, const int *tn, int nprob, int maxn,
                   void *scratch, cudaStream_t st, int *err) {
  Moves *m = static_cast<Moves *>(scratch);
  constexpr int F = sizeof(T) == 4 ? 2 : 1;
  for (int kb = 0; kb < maxn;) {
    const int h = maxn - kb;
    if (h <= PT * F) {
      if (h <= PT) lu_step<T, 32, 1>(LU, loff, piv, toff, tn, nprob, maxn, kb, m, err, st);
      else lu_step<T, 32, F>(LU, loff, piv, toff, tn, nprob, maxn, kb, m, err, st);
      kb += 32;
    } else if (h <= 2 * PT * F) {
      lu_step<T, 16, 2 * F>(LU, loff, piv, toff, tn, nprob, maxn, kb, m, err, st);
      kb += 16;
    } else {
      lu_step<T, 8, 4 * F>(LU, loff, piv, toff, tn, nprob, maxn, kb, m, err, st);
      kb += 8;
    }
  }
}

// Inverses of the DB x DB diagonal blocks of L (unit lower) and U, side by
// side per block: a warp each, lane c solving for column c.
template <typename T>
__global__ void __launch_bounds__(64) k_diag_inverse(const T *LUall, const int64_t *loff, const int *tn, int maxblk,
                                                     T *D) {
  __shared__ T s_a[DB][DB + 1];
  pdl_enter();
  const int p = blockIdx.y, q = blockIdx.x, n = tn[p], k0 = q * DB, nb = min(DB, n - k0);
  if (nb <= 0) return;
  const T *A = LUall + loff[p];
  T *o = D + ((int64_t)p * maxblk + q) * (2 * DB * DB);
  for (int e = threadIdx.x; e < DB * DB; e += 64) {
    const int i = e / DB, c = e % DB;
    s_a[i][c] = i < nb && c < nb ? A[(int64_t)(k0 + i) * n + k0 + c] : (T)(i == c);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  T x[DB];
  if (threadIdx.x < 32) {
#pragma unroll
    for (int i = 0; i < DB; i++) {
      T s = (T)(i == lane);
      if (i < nb)  // rows past the block are the identity's
#pragma unroll
        for (int l = 0; l < i; l++) s -= s_a[i][l] * x[l];
      x[i] = s;
      o[i * DB + lane] = s;
    }
  } else {
#pragma unroll
    for (int i = DB - 1; i >= 0; i--) {
      T s = (T)(i == lane);
      if (i < nb) {
#pragma unroll
        for (int l = DB - 1; l > i; l--) s -= s_a[i][l] * x[l];
        s /= s_a[i][i];
      }
      x[i] = s;
      o[DB * DB + i * DB + lane] = s;
    }
  }
}

// Columns c0 .. c0 + NC - 1 of W = U^{-1} L^{-1}: z in shared memory
// (column-major, ld n).  Row block by row block: the block's rows times the
// part of z already known (a warp per four rows, lanes along the row), then
// the diagonal block's inverse.
template <typename T, int NC>
__global__ void __launch_bounds__(256) k_top_inverse(const T *LUall, const int64_t *loff, const int *tn, int maxblk,
                                                     const T *D, T *Wall) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ T s_r[DB][NC];
  pdl_enter();
  const int p = blockIdx.y, n = tn[p], c0 = blockIdx.x * NC;
  if (c0 >= n) return;
  T *z = reinterpret_cast<T *>(sm);
  const T *A = LUall + loff[p];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nblk = (n + DB - 1) / DB, b0 = c0 / DB;
  for (int e = tid; e < n * NC; e += 256) z[e] = (T)(e % n == c0 + e / n);
  __syncthreads();
  for (int pass = 0; pass < 2; pass++)
    for (int s = 0; s < (pass == 0 ? nblk - b0 : nblk); s++) {
      const int q = pass == 0 ? b0 + s : nblk - 1 - s, k0 = q * DB, nb = min(DB, n - k0);
      // columns of the row block that multiply known entries: z is zero above
      // block b0 in the forward pass
      const int l0 = pass == 0 ? b0 * DB : k0 + nb, l1 = pass == 0 ? k0 : n;
      T acc[4][NC];
#pragma unroll
      for (int u = 0; u < 4; u++)
#pragma unroll
        for (int c = 0; c < NC; c++) acc[u][c] = (T)0;
      const T *row[4];
#pragma unroll
      for (int u = 0; u < 4; u++) row[u] = A + (int64_t)min(k0 + 4 * warp + u, n - 1) * n;
#pragma unroll 2
      for (int l = l0 + lane; l < l1; l += 32) {
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; u++) v[u] = __ldg(row[u] + l);
#pragma unroll
        for (int c = 0; c < NC; c++) {
          const T x = z[c * n + l];
#pragma unroll
          for (int u = 0; u < 4; u++) acc[u][c] += v[u] * x;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; u++)
#pragma unroll
        for (int c = 0; c < NC; c++) {
          const T t = warp_sum(acc[u][c]);
          if (lane == 0) {
            const int i = 4 * warp + u;
            s_r[i][c] = i < nb ? z[c * n + k0 + i] - t : (T)0;
          }
        }
      __syncthreads();
      const T *Dq = D + ((int64_t)p * maxblk + q) * (2 * DB * DB) + pass * DB * DB;
      for (int e = tid; e < DB * NC; e += 256) {
        const int i = e % DB, c = e / DB;
        if (i < nb) {
          T s0 = (T)0, s1 = (T)0;
#pragma unroll 8
          for (int l = 0; l < DB; l += 2) {
            s0 += __ldg(Dq + i * DB + l) * s_r[l][c];
            s1 += __ldg(Dq + i * DB + l + 1) * s_r[l + 1][c];
          }
          z[c * n + k0 + i] = s0 + s1;
        }
      }
      __syncthreads();
    }
  T *W = Wall + loff[p];
  for (int e = tid; e < n * NC; e += 256) {
    const int i = e / NC, c = e % NC;
    if (c0 + c < n) W[(int64_t)i * n + c0 + c] = z[c * n + i];
  }
}

// Largest row sums of |W|, |L| and |U| of every problem (as FP32 bits), a warp per
// row: their product bounds what a solve by W loses against triangular solves.
template <typename T>
__global__ void __launch_bounds__(256) k_top_norms(const T *LUall, const T *Wall, const int64_t *loff, const int *tn,
                                                   unsigned *norms) {
  const int p = blockIdx.y, n = tn[p], lane = threadIdx.x & 31, i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const T *a = LUall + loff[p] + (int64_t)i * n, *w = Wall + loff[p] + (int64_t)i * n;
  T sw = (T)0, sl = (T)0, su = (T)0;
  for (int l = lane; l < n; l += 32) {
    sw += fabs(w[l]);
    (l < i ? sl : su) += fabs(a[l]);
  }
  const float v[3] = {(float)warp_sum(sw), (float)warp_sum(sl) + 1.f, (float)warp_sum(su)};
  if (lane == 0)
    for (int q = 0; q < 3; q++) atomicMax(norms + 3 * p + q, __float_as_uint(v[q]) & 0x7fffffffu);
}

int64_t top_inverse_scratch_elems(int nprob, int maxn) {
  return (int64_t)nprob * ((maxn + DB - 1) / DB) * (2 * DB * DB);
}

template <typename T>
void launch_top_inverse(const T *LU, const int64_t *loff, const int *tn, int nprob, int maxn, T *W, T *D,
                        unsigned *norms, cudaStream_t st) {
  if (maxn == 0 || nprob == 0) return;
  const int maxblk = (maxn + DB - 1) / DB;
  launch_pdl(k_diag_inverse<T>, dim3(maxblk, nprob), 64, 0, st, LU, loff, tn, maxblk, D);
  auto run = [&](auto kern, int nc) {
    const size_t smem = (size_t)maxn * nc * sizeof(T);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(kern, dim3((maxn + nc - 1) / nc, nprob), 256, smem, st, LU, loff, tn, maxblk, (const T *)D, W);
  };
  // columns per CTA: as many as leave about a CTA per SM
  const int64_t cols = (int64_t)nprob * maxn;
  if (cols >= 8 * 152 && sizeof(T) == 4) run(k_top_inverse<T, 8>, 8);
  else if (cols >= 4 * 152) run(k_top_inverse<T, 4>, 4);
  else run(k_top_inverse<T, 2>, 2);
  cudaMemsetAsync(norms, 0, sizeof(unsigned) * 3 * (size_t)nprob, st);
  k_top_norms<T><<<dim3((maxn + 7) / 8, nprob), 256, 0, st>>>(LU, W, loff, tn, norms);
  count_launch();
}

#define RSS_INST(T)                                                                                                 \
  template void launch_top_lu<T>(T *, const int64_t *, int *, const int64_t *, const int *, int, int, void *,       \
                                 cudaStream_t, int *);                                                              \
  template void launch_top_inverse<T>(const T *, const int64_t *, const int *, int, int, T *, T *, unsigned *,         \
                                      cudaStream_t);
RSS_INST(float)
RSS_INST(double)

}  // namespace rss
