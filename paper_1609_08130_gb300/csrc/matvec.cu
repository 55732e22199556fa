// matvec.cu -- the exact operator y = A x by direct summation (scattered
// points), FP64 in and out, evaluated in sums of three FP32 numbers.
//
// FP64 arithmetic runs at 2.15 operations per clock and SM here, FP32 at 128:
// a plain FP64 sum does about 17 FP64 operations a pair of points and column.
// FP32 numbers in threes (tf.cuh) carry the distance, the kernel and the sums to
// about 2^-56, so the result's error is that of its last FP64 roundings:
//   - coordinates are three FP32 parts on fixed grids (24 + 24 bits and the
//     rest), so differences of the first two parts are exact and the distance
//     keeps its bits however near the points are (exceptions below);
//   - r^2 = sum of squares; log r^2 table-driven (log_tf.cuh), 1 / r by an FP32
//     seed and a Newton step of second order;
//   - products and sums, flushed into FP64 every 256 terms.
// The weight, the kernel's constant and the diagonal term are FP64.  The
// columns are scaled by powers of two per tile of 256 sources; a tile with
// a value that is not finite takes plain FP64 arithmetic, and so do points
// that (nearly) coincide.
//
// About 130 FP32 instructions a pair of points and 45 a column.  Two columns of
// 20000 3D points: plain FP64 34 ms, here 3.6 ms.  Relative error of the
// kernel's part (diag 0, 64 to 20000 points, right-hand sides of both signs):
// 1.4e-16 to 2.3e-16, of the FP64 sum 2.8e-16 to 6.3e-15.  Pairs of FP32
// numbers took 2.1 ms, but left 2.1e-15 to 2.4e-14.
#include <algorithm>
#include <vector>

#include "internal.h"
#include "log_table.h"
#include "log_tf.cuh"

namespace rss {

namespace {

constexpr int MVT = 256;    // sources per tile, threads per CTA
constexpr int MV_SHIFT = 40;  // scaled coordinates stay below 2^40
// Pairs of points with a scaled r^2 below this take FP64 arithmetic: R2_MIN,
// where the third part would underflow; R2_AXIS for a target with a coordinate
// below NEAR_AXIS, where a coordinate's last bits may be finer than the 2^-32
// that its third part holds (2^-72 of the largest coordinate) and matter
// against a distance below 2^22.
constexpr float R2_MIN = 0x1p-60f, R2_AXIS = 0x1p44f, NEAR_AXIS = 0x1p23f;
constexpr int KBAD = 1 << 30;  // column scale of a tile with values that are not finite

__device__ __forceinline__ double pow2(int k) { return __longlong_as_double((long long)(1023 + k) << 52); }

// largest |coordinate| (as FP64 bits)
__global__ void k_mv_extent(const double *xt, int64_t cnt, unsigned long long *mx) {
  unsigned long long m = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(xt[i]) & 0x7fffffffffffffffull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(mx, m);
}

// smallest E with every |coordinate| <= 2^E
__device__ __forceinline__ int extent_exp(unsigned long long mx) {
  const int e = (int)(mx >> 52) - 1023;
  return max(-900, min(900, (mx & 0xfffffffffffffull) ? e + 1 : e));
}

// part p (of 3) of coordinate d at out[(3 d + p) n + i], scaled by 2^(40 - E):
// multiples of 2^17, then of 2^-7 (differences of either are below 2^24 of
// them), then the rest; the first CTA also fills the logarithm's exponent table
__global__ void __launch_bounds__(256) k_mv_split(const double *xt, int64_t n, int dim, const unsigned long long *mx,
                                                  LogTables *T, float *out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int sh = MV_SHIFT - extent_exp(*mx);
  if (blockIdx.x == 0) T->et[threadIdx.x] = log_tables_exponent((int)threadIdx.x - 127 - 2 * sh);
  if (i >= n) return;
  for (int d = 0; d < dim; d++) {
    const double x = xt[i * dim + d] * pow2(sh / 2) * pow2(sh - sh / 2);
    const double h = rint(x * 0x1p-17) * 0x1p17, l = rint((x - h) * 0x1p7) * 0x1p-7;
    out[(3 * d) * n + i] = (float)h;
    out[(3 * d + 1) * n + i] = (float)l;
    out[(3 * d + 2) * n + i] = (float)((x - h) - l);
  }
}

// The columns in tree order in three parts (planes of n), scaled by 2^-k: k a
// multiple of 64 near the tile's largest exponent (0 for ordinary data).
__global__ void __launch_bounds__(MVT) k_mv_x(const int64_t *perm, const double *xin, int64_t n, int ncol,
                                              const int64_t *tstart, const int64_t *tend, float *xs, int *xk) {
  __shared__ unsigned s_e;
  const int q = blockIdx.x, c = blockIdx.y;
  const int64_t i = tstart[q] + threadIdx.x;
  const bool live = i < tend[q];
  if (threadIdx.x == 0) s_e = 0;
  __syncthreads();
  const double x = live ? xin[perm[i] + c * n] : 0.0;
  const unsigned e = (unsigned)(__double_as_longlong(x) >> 52) & 0x7ffu;
  const unsigned ew = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_e, ew);
  __syncthreads();
  const int em = (int)s_e;
  // 0x7ff: not finite; 0: zeros (and subnormals, which count as such beside FP64 rounding)
  const int k = em == 0x7ff ? KBAD : em == 0 ? 0 : ((em - 1023 + 32 + 1024) >> 6) * 64 - 1024;
  if (threadIdx.x == 0) xk[(int64_t)c * gridDim.x + q] = k;
  if (live) {
    Tf v{0.f, 0.f, 0.f};
    if (k != KBAD) {
      const double s = x * pow2(-(k / 2)) * pow2(-(k - k / 2));
      v.h = (float)s;
      const double r = s - (double)v.h;
      v.m = (float)r;
      v.l = (float)(r - (double)v.m);
    }
    float *o = xs + (int64_t)3 * c * n + i;
    o[0] = v.h;
    o[n] = v.m;
    o[2 * n] = v.l;
  }
}

// One CTA: 256 / parts targets of one tile, `parts` threads per target, each
// taking every parts-th source; grid.y: groups of NC columns.  parts = 4 or
// 16: enough CTAs for every SM down to a few hundred targets (79 CTAs of 256
// targets left half the chip idle at 20011 points).  Bound: FP32 issue.
template <int DIM, int KIND, int NC>
__global__ void __launch_bounds__(MVT, NC == 8 ? 2 : 3)
    k_mv(const float *cs, const double *xt, const unsigned long long *mx, KernelParams K, const double *wdof,
         const int64_t *perm, const double *xin, const float *xs, const int *xk, double *yout, int64_t n, int col0,
         int ncol, int ntile, int parts, const int64_t *tstart, const int64_t *tend, const int64_t *sbeg,
         const int64_t *send) {
  __shared__ float sc[3 * DIM][MVT];
  __shared__ float sx[NC][3][MVT];
  __shared__ float4 s_lt[KIND == 0 ? LOG_CELLS : 1], s_et[KIND == 0 ? 256 : 1];
  __shared__ double s_red[MVT];
  const int tid = threadIdx.x;
  const int q = blockIdx.x / parts, sub = blockIdx.x % parts;
  const int ntg = MVT / parts, tg = tid % ntg, part = tid / ntg;
  const int64_t t0 = tstart[q], i = t0 + sub * ntg + tg;
  if (t0 + sub * ntg >= tend[q]) return;  // uniform
  const bool live = i < tend[q];
  const int64_t ic = live ? i : t0;
  const int64_t j0b = sbeg[q], j1b = send[q];
  const int q0 = q - (int)((t0 - j0b) / MVT);  // the problem's first tile
  const int cb = col0 + blockIdx.y * NC;
  const int sh = MV_SHIFT - extent_exp(*mx);
  if (KIND == 0) {
    const LogTables *T = reinterpret_cast<const LogTables *>(mx + 2);
    for (int e = tid; e < LOG_CELLS; e += MVT) s_lt[e] = T->lt[e];
    s_et[tid] = T->et[tid];
  }
  float xi[3 * DIM];
#pragma unroll
  for (int d = 0; d < 3 * DIM; d++) xi[d] = cs[(int64_t)d * n + ic];
  float r2min = R2_MIN;
#pragma unroll
  for (int d = 0; d < DIM; d++)
    if (fabsf(xi[3 * d] + xi[3 * d + 1]) < NEAR_AXIS) r2min = R2_AXIS;
  Tf acc[NC];
  double sum[NC];
  int kc[NC];
#pragma unroll
  for (int c = 0; c < NC; c++) acc[c] = Tf{0.f, 0.f, 0.f}, sum[c] = 0.0, kc[c] = 0;
  // the scaled sums so far into the FP64 ones
  auto flush = [&]() {
#pragma unroll
    for (int c = 0; c < NC; c++) {
      sum[c] += ((double)acc[c].h + ((double)acc[c].m + (double)acc[c].l)) * pow2(kc[c] / 2) * pow2(kc[c] - kc[c] / 2);
      acc[c] = Tf{0.f, 0.f, 0.f};
    }
  };
  int terms = 0;
  for (int64_t j0 = j0b; j0 < j1b; j0 += MVT) {
    const int sq = q0 + (int)((j0 - j0b) / MVT);
    const int lim = (int)min((int64_t)MVT, j1b - j0);
    bool bad = false, change = false;
    int kn[NC];
#pragma unroll
    for (int c = 0; c < NC; c++) {
      kn[c] = cb + c < ncol ? xk[(int64_t)(cb + c) * ntile + sq] : 0;
      bad |= kn[c] == KBAD;
      change |= kn[c] != kc[c];
    }
    __syncthreads();  // the tile before is used up
    if (tid < lim) {
#pragma unroll
      for (int d = 0; d < 3 * DIM; d++) sc[d][tid] = cs[(int64_t)d * n + j0 + tid];
#pragma unroll
      for (int c = 0; c < NC; c++)
#pragma unroll
        for (int p = 0; p < 3; p++)
          sx[c][p][tid] = cb + c < ncol ? xs[(int64_t)(3 * (cb + c) + p) * n + j0 + tid] : 0.f;
    }
    __syncthreads();
    const int64_t self64 = i - j0;
    const int self = self64 >= 0 && self64 < lim ? (int)self64 : -1;
    // source s in plain FP64, in units of the scaled distances as the sums
    auto plain = [&](int s) {
      double r2 = 0.0;
      for (int d = 0; d < DIM; d++) {
        const double z = xt[ic * DIM + d] - xt[(j0 + s) * DIM + d];
        r2 += z * z;
      }
      const double a = KIND == 0 ? log(r2) : 1.0 / (sqrt(r2) * pow2(sh / 2) * pow2(sh - sh / 2));
      for (int c = 0; c < NC; c++)
        if (cb + c < ncol) sum[c] += a * xin[perm[j0 + s] + (int64_t)(cb + c) * n];
    };
    if (bad) {  // uniform
      for (int s = part; s < lim; s += parts)
        if (s != self) plain(s);
      continue;
    }
    if (change || terms >= MVT) {
      flush();
      terms = 0;
#pragma unroll
      for (int c = 0; c < NC; c++) kc[c] = kn[c];
    }
    terms += (lim + parts - 1) / parts;
#pragma unroll 2
    for (int s = part; s < lim; s += parts) {
      float dx[3 * DIM];
#pragma unroll
      for (int d = 0; d < 3 * DIM; d++) dx[d] = __fadd_rn(xi[d], -sc[d][s]);
      const Tf r2 = dist2_tf<DIM>(dx);
      Tf a = KIND == 0 ? log_tf(r2, s_lt, s_et) : rsqrt_tf(r2);
      if (!(r2.h >= r2min)) {  // the target itself, or a point (nearly) on it
        a = Tf{0.f, 0.f, 0.f};
        if (s != self) plain(s);
      }
#pragma unroll
      for (int c = 0; c < NC; c++) add_mul_tf(acc[c], a, Tf{sx[c][0][s], sx[c][1][s], sx[c][2][s]});
    }
  }
  flush();
  const double w = wdof ? wdof[ic] : K.w;
  const double f = KIND == 0 ? -w * (1.0 / (4.0 * kPi)) : w * (1.0 / (4.0 * kPi)) * pow2(sh / 2) * pow2(sh - sh / 2);
#pragma unroll
  for (int c = 0; c < NC; c++) {
    __syncthreads();
    s_red[tid] = sum[c];
    __syncthreads();
    if (part == 0 && live && cb + c < ncol) {
      double s = s_red[tg];
      for (int p = 1; p < parts; p++) s += s_red[p * ntg + tg];
      const int64_t g = perm[i] + (int64_t)(cb + c) * n;
      yout[g] = f * s + K.diag * xin[g];
    }
  }
}

// The same product with the kernel evaluated in FP32 (the inner GMRES of the
// refinement): the parts' differences (the leading two exact) added in FP32,
// at most 256 terms summed in FP32, those sums in FP64.
template <int DIM, int NC>
__global__ void __launch_bounds__(MVT, 4)
    k_mv_f32(const float *cs, const unsigned long long *mx, int kind, float wk, const double *wdof, float diag,
             const int64_t *perm, const double *xin, double *yout, int64_t n, int col0, int ncol, int parts,
             const int64_t *tstart, const int64_t *tend, const int64_t *sbeg, const int64_t *send) {
  __shared__ float sc[3 * DIM][MVT];
  __shared__ float sx[NC][MVT];
  __shared__ double s_red[MVT];
  const int tid = threadIdx.x;
  const int q = blockIdx.x / parts, sub = blockIdx.x % parts;
  const int ntg = MVT / parts, tg = tid % ntg, part = tid / ntg;
  const int64_t t0 = tstart[q], i = t0 + sub * ntg + tg;
  if (t0 + sub * ntg >= tend[q]) return;  // uniform
  const bool live = i < tend[q];
  const int64_t ic = live ? i : t0;
  const int64_t j0b = sbeg[q], j1b = send[q];
  const int cb = col0 + blockIdx.y * NC;
  const float us = exp2f((float)(extent_exp(*mx) - MV_SHIFT));  // back to the points' units
  float xi[3 * DIM];
#pragma unroll
  for (int d = 0; d < 3 * DIM; d++) xi[d] = us * cs[(int64_t)d * n + ic];
  float t[NC];
  double sum[NC];
#pragma unroll
  for (int c = 0; c < NC; c++) t[c] = 0.f, sum[c] = 0.0;
  int terms = 0;
  for (int64_t j0 = j0b; j0 < j1b; j0 += MVT) {
    const int lim = (int)min((int64_t)MVT, j1b - j0);
    __syncthreads();  // the tile before is used up
    if (tid < lim) {
#pragma unroll
      for (int d = 0; d < 3 * DIM; d++) sc[d][tid] = us * cs[(int64_t)d * n + j0 + tid];
      const int64_t g = perm[j0 + tid];
#pragma unroll
      for (int c = 0; c < NC; c++) sx[c][tid] = cb + c < ncol ? (float)xin[g + (int64_t)(cb + c) * n] : 0.f;
    }
    __syncthreads();
    const int64_t self64 = i - j0;
    const int self = self64 >= 0 && self64 < lim ? (int)self64 : -1;
    if (terms + (lim + parts - 1) / parts > MVT) {
#pragma unroll
      for (int c = 0; c < NC; c++) sum[c] += (double)t[c], t[c] = 0.f;
      terms = 0;
    }
    terms += (lim + parts - 1) / parts;
#pragma unroll 4
    for (int s = part; s < lim; s += parts) {
      float r2 = 0.f;
#pragma unroll
      for (int d = 0; d < DIM; d++) {
        const float z = ((xi[3 * d] - sc[3 * d][s]) + (xi[3 * d + 1] - sc[3 * d + 1][s])) + (xi[3 * d + 2] - sc[3 * d + 2][s]);
        r2 = fmaf(z, z, r2);
      }
      const float a = s == self ? 0.f : kof(kind, r2);
#pragma unroll
      for (int c = 0; c < NC; c++) t[c] = fmaf(a, sx[c][s], t[c]);
    }
  }
  const float w = wdof ? (float)wdof[ic] : wk;
#pragma unroll
  for (int c = 0; c < NC; c++) {
    __syncthreads();
    s_red[tid] = sum[c] + (double)t[c];
    __syncthreads();
    if (part == 0 && live && cb + c < ncol) {
      double s = s_red[tg];
      for (int p = 1; p < parts; p++) s += s_red[p * ntg + tg];
      const int64_t g = perm[i] + (int64_t)(cb + c) * n;
      yout[g] = (double)w * s + (double)(diag * (float)xin[g]);
    }
  }
}

// Threads per target: 4 threads give 1200 CTAs (two or more rounds of the
// chip) from about 300 tiles on; fewer tiles take 16.
int mv_parts(int ntile, int groups) { return (int64_t)ntile * groups * 4 >= 1200 ? 4 : 16; }

}  // namespace

// extent (16 bytes), the logarithm's tables, the parts
constexpr int64_t SPLIT_HEAD = 16 + (int64_t)sizeof(LogTables);
int64_t matvec_split_bytes(int64_t n, int dim) { return SPLIT_HEAD + (int64_t)sizeof(float) * 3 * dim * n; }
int64_t matvec_x_bytes(int64_t n, int nrhs, int ntile) {
  return (int64_t)nrhs * (n * 3 * (int64_t)sizeof(float) + ntile * (int64_t)sizeof(int));
}

void matvec_split(const double *x_tree, int64_t n, int dim, void *split, cudaStream_t st) {
  if (n == 0) return;
  static const std::vector<float> lt = [] {  // made once, never written again
    std::vector<float> t(4 * LOG_CELLS);
    for (int i = 0; i < LOG_CELLS; i++) log_table_entry(i, LOG_CELLS, LOG_M, &t[4 * i]);
    return t;
  }();
  unsigned long long *mx = static_cast<unsigned long long *>(split);
  cudaMemcpyAsync(reinterpret_cast<LogTables *>(mx + 2)->lt, lt.data(), sizeof(float4) * LOG_CELLS,
                  cudaMemcpyHostToDevice, st);
  float *cs = reinterpret_cast<float *>(static_cast<char *>(split) + SPLIT_HEAD);
  cudaMemsetAsync(mx, 0, 16, st);
  const int64_t cnt = n * dim;
  k_mv_extent<<<(unsigned)std::min<int64_t>((cnt + 1023) / 1024, 608), 256, 0, st>>>(x_tree, cnt, mx);
  k_mv_split<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x_tree, n, dim, mx, reinterpret_cast<LogTables *>(mx + 2), cs);
  count_launch(2);
}

template <int DIM, int KIND, int NC>
static void launch_mv(const float *cs, const double *xt, const unsigned long long *mx, const KernelParams &K,
                      const double *wdof, const int64_t *perm, const double *xin, const float *xs, const int *xk,
                      double *yout, int64_t n, int col0, int ncol, int ntile, const int64_t *tstart,
                      const int64_t *tend, const int64_t *sbeg, const int64_t *send, cudaStream_t st) {
  const int groups = std::max(1, (ncol - col0) / NC), parts = mv_parts(ntile, groups);
  k_mv<DIM, KIND, NC><<<dim3((unsigned)(ntile * parts), groups), MVT, 0, st>>>(
      cs, xt, mx, K, wdof, perm, xin, xs, xk, yout, n, col0, ncol, ntile, parts, tstart, tend, sbeg, send);
  count_launch();
}

void launch_matvec(const double *x_tree, int dim, const KernelParams &K, const double *wdof, const int64_t *perm,
                   const double *xin, double *yout, int64_t n, int nrhs, int ntile, const int64_t *tstart,
                   const int64_t *tend, const int64_t *sbeg, const int64_t *send, const void *split, void *xbuf,
                   cudaStream_t st) {
  if (n == 0 || ntile == 0 || nrhs == 0) return;
  const unsigned long long *mx = static_cast<const unsigned long long *>(split);
  const float *cs = reinterpret_cast<const float *>(static_cast<const char *>(split) + SPLIT_HEAD);
  float *xs = static_cast<float *>(xbuf);
  int *xk = reinterpret_cast<int *>(xs + (int64_t)3 * nrhs * n);
  k_mv_x<<<dim3((unsigned)ntile, nrhs), MVT, 0, st>>>(perm, xin, n, nrhs, tstart, tend, xs, xk);
  count_launch();
  // columns in groups of eight, then four to one: the distance and the kernel
  // cost as much as three columns' products
#define MV(D, KD, N) \
  launch_mv<D, KD, N>(cs, x_tree, mx, K, wdof, perm, xin, xs, xk, yout, n, c, nrhs, ntile, tstart, tend, sbeg, send, st)
#define MVN(N)                           \
  do {                                   \
    if (dim == 2 && K.kind == 0) MV(2, 0, N); \
    else if (dim == 2) MV(2, 1, N);      \
    else if (K.kind == 0) MV(3, 0, N);   \
    else MV(3, 1, N);                    \
  } while (0)
  for (int c = 0; c < nrhs;) {
    const int left = nrhs - c;
    if (left >= 8) {
      MVN(8);
      c += left / 8 * 8;
    } else if (left >= 4) {
      MVN(4);
      c += 4;
    } else if (left == 3) {
      MVN(3);
      c += 3;
    } else if (left == 2) {
      MVN(2);
      c += 2;
    } else {
      MVN(1);
      c += 1;
    }
  }
#undef MVN
#undef MV
}

template <int DIM, int NC>
static void launch_mv_f32(const float *cs, const unsigned long long *mx, const KernelParams &K, const double *wdof,
                          const int64_t *perm, const double *xin, double *yout, int64_t n, int col0, int ncol,
                          int ntile, const int64_t *tstart, const int64_t *tend, const int64_t *sbeg,
                          const int64_t *send, cudaStream_t st) {
  const int groups = std::max(1, (ncol - col0) / NC), parts = mv_parts(ntile, groups);
  k_mv_f32<DIM, NC><<<dim3((unsigned)(ntile * parts), groups), MVT, 0, st>>>(
      cs, mx, K.kind, (float)K.w, wdof, (float)K.diag, perm, xin, yout, n, col0, ncol, parts, tstart, tend, sbeg, send);
  count_launch();
}

void launch_matvec_f32(int dim, const KernelParams &K, const double *wdof, const int64_t *perm, const double *xin,
                       double *yout, int64_t n, int nrhs, int ntile, const int64_t *tstart, const int64_t *tend,
                       const int64_t *sbeg, const int64_t *send, const void *split, cudaStream_t st) {
  if (n == 0 || ntile == 0 || nrhs == 0) return;
  const unsigned long long *mx = static_cast<const unsigned long long *>(split);
  const float *cs = reinterpret_cast<const float *>(static_cast<const char *>(split) + SPLIT_HEAD);
  for (int c = 0; c < nrhs;) {
    const int left = nrhs - c;
#define MV(D, N) launch_mv_f32<D, N>(cs, mx, K, wdof, perm, xin, yout, n, c, nrhs, ntile, tstart, tend, sbeg, send, st)
    if (left >= 3) {
      if (dim == 2) MV(2, 4);
      else MV(3, 4);
      c += std::max(4, left / 4 * 4);
    } else {
      if (dim == 2) MV(2, 1);
      else MV(3, 1);
      c += left;
    }
#undef MV
  }
}

}  // namespace rss
