// refine.cu -- FP64 residual operator on grids and vector kernels of the
// iterative refinement (GMRES-IR) around the factorization.
//
// When the points are the cell centres of an s^d grid, K_ij = kappa(I_i - I_j)
// depends only on the integer offset of the two cells, so K x is a discrete
// convolution.  It is applied exactly (to rounding) by embedding the kernel in
// a circulant of side L = 2s and using a Stockham FFT written here (radix-4
// passes, the lines of a CTA held in shared memory).  Two real right-hand sides
// share one complex transform (x1 + i x2): the embedded kernel is real and
// even, so its spectrum is real and the real and imaginary parts of the product
// transform back to K x1 and K x2.
//
// FP64 arithmetic bounds it (2.15 operations per clock and SM), so the passes
// leave out what is known: the input is zero outside [0, s)^d and only that
// corner of the output is read, so a pass reads or writes half lines there and
// its first or last radix-4 step takes the zero or unread half as such; the
// forward pass along the last axis, the product with the spectrum and the
// inverse pass are one kernel, and all pairs of columns share the launches.
// (Pairs of FP32 numbers would take a third of the time, but their 48 bits
// showed in the product's last digits, so the arithmetic stays FP64.)  Two
// products of four columns on the 512^2 grid 1.46 -> 1.28 ms and the spectrum
// 0.25 -> 0.15 ms, of 16 columns on the 256^2 grid 1.52 -> 0.91 ms.
//
// The same transforms in FP32 are the operator products inside the refinement's
// inner GMRES for a FP32 factor: there an operator accurate to FP32 rounding is
// enough (the inner solve only has to shrink the correction's error by a
// bounded factor), and FP64 stays for the residuals and the update.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

namespace rss {

namespace {

constexpr int FT = 256;  // threads of an FFT CTA

// complex type of a real type, its constructor and fused multiply-add
template <typename R> struct Cx;
template <> struct Cx<double> {
  using t = double2;
  static __device__ __forceinline__ double2 mk(double x, double y) { return make_double2(x, y); }
  static __device__ __forceinline__ double fm(double a, double b, double c) { return fma(a, b, c); }
};
template <> struct Cx<float> {
  using t = float2;
  static __device__ __forceinline__ float2 mk(float x, float y) { return make_float2(x, y); }
  static __device__ __forceinline__ float fm(float a, float b, float c) { return fmaf(a, b, c); }
};

// Stockham FFT (sign -1 forward, +1 inverse, unscaled) of `nl` lines of length
// L in shared memory at a (line ln at a + ln L), b the other buffer; returns
// the buffer that holds the result.  A pass combines sub-transforms of length
// m = 2^lm into ones of length 2m (radix 2, once when log2 L is odd) or 4m
// (radix 4): output index (r k) m + j + q m from inputs k m + j + p L / r,
// twiddled by w_{r m}^{p j} (tw[x] = exp(-2 pi i x / L), conjugated for
// sign > 0) and combined by the r-point DFT.  half_in: the upper half of the
// input is zero; half_out: the upper half of the output is not needed (both
// only in radix-4 passes).
template <typename R>
__device__ __forceinline__ typename Cx<R>::t *fft_shared(typename Cx<R>::t *a, typename Cx<R>::t *b, int nl, int L,
                                                         int logL, const typename Cx<R>::t *tw, int sign,
                                                         bool half_in, bool half_out) {
  using C2 = typename Cx<R>::t;
  int lm = 0;
  if (logL & 1) {
    const int half = L >> 1;
    for (int e = threadIdx.x; e < nl * half; e += FT) {  // m = 1: no twiddle
      const int t = e & (half - 1), o = (e >> (logL - 1)) * L;
      const C2 u = a[o + t];
      if (half_in) {
        b[o + 2 * t] = u;
        b[o + 2 * t + 1] = u;
      } else {
        const C2 v = a[o + t + half];
        b[o + 2 * t] = Cx<R>::mk(u.x + v.x, u.y + v.y);
        b[o + 2 * t + 1] = Cx<R>::mk(u.x - v.x, u.y - v.y);
      }
    }
    __syncthreads();
    C2 *t0 = a;
    a = b;
    b = t0;
    lm = 1;
  }
  const R sg = sign > 0 ? (R)1 : (R)-1;
  for (; lm < logL; lm += 2) {
    const int m = 1 << lm, quarter = L >> 2, tsh = logL - lm - 2;
    const bool zero_in = half_in && lm == 0, skip = half_out && lm + 2 >= logL;
    for (int e = threadIdx.x; e < nl * quarter; e += FT) {
      const int t = e & (quarter - 1), o = (e >> (logL - 2)) * L;
      const int j = t & (m - 1), k = t >> lm;
      const C2 a0 = a[o + t], a1 = a[o + t + quarter];
      C2 *q = b + o + (k << (lm + 2)) + j;
      if (zero_in) {  // a2 = a3 = 0, no twiddles
        const C2 r = Cx<R>::mk(-sg * a1.y, sg * a1.x);
        q[0] = Cx<R>::mk(a0.x + a1.x, a0.y + a1.y);
        q[m] = Cx<R>::mk(a0.x + r.x, a0.y + r.y);
        if (!skip) {
          q[2 * m] = Cx<R>::mk(a0.x - a1.x, a0.y - a1.y);
          q[3 * m] = Cx<R>::mk(a0.x - r.x, a0.y - r.y);
        }
        continue;
      }
      C2 c1 = a1, c2 = a[o + t + 2 * quarter], c3 = a[o + t + 3 * quarter];
      if (lm > 0) {
        auto twiddle = [&](C2 &v, int at) {
          C2 w = __ldg(tw + at);
          if (sign > 0) w.y = -w.y;
          v = Cx<R>::mk(Cx<R>::fm(v.x, w.x, -v.y * w.y), Cx<R>::fm(v.x, w.y, v.y * w.x));
        };
        twiddle(c1, j << tsh);
        twiddle(c2, (2 * j) << tsh);
        twiddle(c3, (3 * j) << tsh);
      }
      const C2 t0 = Cx<R>::mk(a0.x + c2.x, a0.y + c2.y), t1 = Cx<R>::mk(a0.x - c2.x, a0.y - c2.y);
      const C2 t2 = Cx<R>::mk(c1.x + c3.x, c1.y + c3.y);
      // (c1 - c3) times w_4 = sign i
      const C2 t3 = Cx<R>::mk(-sg * (c1.y - c3.y), sg * (c1.x - c3.x));
      q[0] = Cx<R>::mk(t0.x + t2.x, t0.y + t2.y);
      q[m] = Cx<R>::mk(t1.x + t3.x, t1.y + t3.y);
      if (!skip) {
        q[2 * m] = Cx<R>::mk(t0.x - t2.x, t0.y - t2.y);
        q[3 * m] = Cx<R>::mk(t1.x - t3.x, t1.y - t3.y);
      }
    }
    __syncthreads();
    C2 *t0 = a;
    a = b;
    b = t0;
  }
  return a;
}

// nl neighbouring lines per CTA: line q (lo fastest) starts at
// (q / lo_lim) hi_mul + (q % lo_lim) lo_mul and has stride `stride`.  Elements
// from nin on are zero and not read, those from nout on not written.  With a
// spectrum (real, at the same positions): forward, product, inverse.
// grid.y: transforms `tot` apart.
template <typename R>
__global__ void __launch_bounds__(FT) k_fft_lines(typename Cx<R>::t *data, int64_t tot, int L, int logL, int nl,
                                                  int64_t lines, int64_t stride, int64_t lo_mul, int64_t lo_lim,
                                                  int64_t hi_mul, int nin, int nout,
                                                  const typename Cx<R>::t *tw, int sign, const R *spectrum) {
  using C = typename Cx<R>::t;
  extern __shared__ __align__(16) unsigned char fft_sh[];
  C *a = reinterpret_cast<C *>(fft_sh), *b = a + nl * L;
  C *X = data + blockIdx.y * tot;
  const int64_t q0 = (int64_t)blockIdx.x * nl;
  const int nq = (int)min((int64_t)nl, lines - q0);
  // element (line, i): along contiguous lines i is fastest, else the line
  const bool along = stride == 1;
  auto at = [&](int ln) { return ((q0 + ln) / lo_lim) * hi_mul + ((q0 + ln) % lo_lim) * lo_mul; };
  const C zero = Cx<R>::mk((R)0, (R)0);
  const bool half_in = 2 * nin <= L, half_out = 2 * nout <= L;
  for (int e = threadIdx.x; e < nl * L; e += FT) {
    const int ln = along ? e >> logL : e % nl, i = along ? e & (L - 1) : e / nl;
    a[ln * L + i] = ln < nq && i < nin ? X[at(ln) + (int64_t)i * stride] : zero;
  }
  __syncthreads();
  C *r = fft_shared<R>(a, b, nl, L, logL, tw, sign, half_in, half_out && !spectrum);
  if (spectrum) {
    for (int e = threadIdx.x; e < nl * L; e += FT) {
      const int ln = along ? e >> logL : e % nl, i = along ? e & (L - 1) : e / nl;
      if (ln < nq) {
        const R c = spectrum[at(ln) + (int64_t)i * stride];
        const C v = r[ln * L + i];
        r[ln * L + i] = Cx<R>::mk(v.x * c, v.y * c);
      }
    }
    __syncthreads();
    r = fft_shared<R>(r, r == a ? b : a, nl, L, logL, tw, -sign, false, half_out);
  }
  for (int e = threadIdx.x; e < nl * nout; e += FT) {
    const int ln = along ? e / nout : e % nl, i = along ? e % nout : e / nl;
    if (ln < nq) X[at(ln) + (int64_t)i * stride] = r[ln * L + i];
  }
}

// tw[k] = exp(-2 pi i k / L), k < L (a radix-4 pass reads up to 3L/4), in both precisions
__global__ void k_twiddle(double2 *tw, float2 *twf, int L) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= L) return;
  double s, c;
  sincospi(-2.0 * (double)k / (double)L, &s, &c);
  tw[k] = make_double2(c, s);
  twf[k] = make_float2((float)c, (float)s);
}

// Embedded kernel c[delta] on the L^d circulant: offsets e in (-s, s) per
// axis, 0 at e = 0 and at the unused index s.  A thread per offset in [0, s]^d
// writes its 2^d mirror images, so the FP64 logarithm is taken once for them.
__global__ void __launch_bounds__(256) k_embed_kernel(double2 *C, int64_t cnt, int dim, int s, int L, double h,
                                                      int kind, double w) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= cnt) return;
  int o[3] = {0, 0, 0};
  int64_t rem = e;
  double r2 = 0.0;
  bool zero = false;
  for (int d = 0; d < dim; d++) {
    o[d] = (int)(rem % (s + 1));
    rem /= s + 1;
    zero |= o[d] == s;
    r2 += (double)o[d] * o[d];
  }
  double v = 0.0;
  if (!zero && r2 > 0.0) v = w * kof(kind, r2 * h * h);
  for (int m = 0; m < (1 << dim); m++) {
    int64_t pos = 0, mul = 1;
    for (int d = 0; d < dim; d++) {
      pos += (int64_t)(m >> d & 1 ? (L - o[d]) % L : o[d]) * mul;
      mul *= L;
    }
    C[pos] = make_double2(v, 0.0);
  }
}
// the spectrum's real part over the transform's size, in both precisions
__global__ void k_spectrum(const double2 *X, int64_t tot, double scale, double *C, float *Cf) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= tot) return;
  const double v = X[e].x * scale;
  C[e] = v;
  Cf[e] = (float)v;
}

// position in the L^d array of point i (caller order) at linear index g of the s^d grid
__device__ __forceinline__ int64_t grid_pos(int64_t g, int dim, int s, int L) {
  int64_t pos = 0, mul = 1;
  for (int d = 0; d < dim; d++) {
    pos += (g % s) * mul;
    g /= s;
    mul *= L;
  }
  return pos;
}

// X[grid(i)] = x1[i] + i x2[i]; grid.y: the pair of columns.  Every position
// of the s^d corner is written.
template <typename R>
__global__ void k_pack(typename Cx<R>::t *X, int64_t tot, const int64_t *gidx, const double *x, int64_t n, int nrhs,
                       int c0, int dim, int s, int L) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = c0 + 2 * blockIdx.y;
  const double re = x[i + (int64_t)c * n], im = c + 1 < nrhs ? x[i + (int64_t)(c + 1) * n] : 0.0;
  X[blockIdx.y * tot + grid_pos(gidx[i], dim, s, L)] = Cx<R>::mk((R)re, (R)im);
}

// y = diag * x + (K x)
template <typename R>
__global__ void k_unpack(const typename Cx<R>::t *X, int64_t tot, const int64_t *gidx, const double *x, double *y,
                         int64_t n, int nrhs, int c0, int dim, int s, int L, double diag) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = c0 + 2 * blockIdx.y;
  const typename Cx<R>::t v = X[blockIdx.y * tot + grid_pos(gidx[i], dim, s, L)];
  y[i + (int64_t)c * n] = fma(diag, x[i + (int64_t)c * n], (double)v.x);
  if (c + 1 < nrhs) y[i + (int64_t)(c + 1) * n] = fma(diag, x[i + (int64_t)(c + 1) * n], (double)v.y);
}

int64_t grid_total(const GridOp &G) {
  int64_t tot = 1;
  for (int d = 0; d < G.dim; d++) tot *= G.L;
  return tot;
}

// One pass along axis `ax` over the lines whose other coordinates d lie below
// lim[d] (lines entirely outside hold zeros, or results nobody reads).
template <typename R>
void fft_pass(const GridOp &G, typename Cx<R>::t *X, const typename Cx<R>::t *tw, int sign, int ax,
              const int64_t *lim, int nin, int nout, const R *spectrum, int npair, cudaStream_t st) {
  int64_t stride[4] = {1, 1, 1, 1};
  for (int d = 0; d < G.dim; d++) stride[d + 1] = stride[d] * G.L;
  int o[2] = {-1, -1}, no = 0;
  for (int d = 0; d < G.dim; d++)
    if (d != ax) o[no++] = d;
  const int64_t lo_lim = no > 0 ? lim[o[0]] : 1, hi_lim = no > 1 ? lim[o[1]] : 1;
  const int64_t lines = lo_lim * hi_lim;
  if (lines == 0) return;
  // lines per CTA: up to 1024 elements and two neighbouring lines (which share
  // 32-byte sectors across the axis) while that leaves two CTAs per SM, so that
  // small grids spread over the FP64 units; 64 KB of buffers at most
  const size_t line = (size_t)2 * G.L * sizeof(typename Cx<R>::t);
  int nl = 1;
  while (nl < 16 && (nl == 1 || nl * G.L < 1024) && lines * npair >= (int64_t)2 * nl * 304) nl *= 2;
  while (nl > 1 && nl * line > (size_t)(64 << 10)) nl /= 2;
  k_fft_lines<R><<<dim3((unsigned)((lines + nl - 1) / nl), npair), FT, nl * line, st>>>(
      X, grid_total(G), G.L, G.logL, nl, lines, stride[ax], no > 0 ? stride[o[0]] : 0, lo_lim,
      no > 1 ? stride[o[1]] : 0, nin, nout, tw, sign, spectrum);
  count_launch();
}

template <typename R>
void grid_op_apply_t(const GridOp &G, typename Cx<R>::t *X, const R *C, const typename Cx<R>::t *tw, const double *x,
                     double *y, int nrhs, cudaStream_t st) {
  const int64_t tot = grid_total(G);
  const unsigned nb = (unsigned)((G.n + 255) / 256);
  for (int c0 = 0; c0 < nrhs; c0 += 2 * G.pairs) {
    const int np = std::min(G.pairs, (nrhs - c0 + 1) / 2);
    k_pack<R><<<dim3(nb, np), 256, 0, st>>>(X, tot, G.gidx, x, G.n, nrhs, c0, G.dim, G.s, G.L);
    // forward: the data sit in [0, s)^d, so an axis not yet transformed
    // limits the lines to its first s coordinates
    int64_t lim[3] = {G.s, G.s, G.s};
    for (int ax = 0; ax + 1 < G.dim; ax++) {
      fft_pass<R>(G, X, tw, -1, ax, lim, G.s, G.L, nullptr, np, st);
      lim[ax] = G.L;
    }
    fft_pass<R>(G, X, tw, -1, G.dim - 1, lim, G.s, G.s, C, np, st);
    // inverse, last axis first: only [0, s)^d is read
    for (int ax = G.dim - 2; ax >= 0; ax--) {
      for (int d = 0; d < G.dim; d++) lim[d] = d > ax ? G.s : G.L;
      fft_pass<R>(G, X, tw, +1, ax, lim, G.L, G.s, nullptr, np, st);
    }
    k_unpack<R><<<dim3(nb, np), 256, 0, st>>>(X, tot, G.gidx, x, y, G.n, nrhs, c0, G.dim, G.s, G.L, G.diag);
    count_launch(2);
  }
}

}  // namespace

// Transforms in flight (pairs of columns): at most 128 MB of work space
void grid_op_bytes(GridOp &G, size_t &spectrum, size_t &work, size_t &tables) {
  const int64_t tot = grid_total(G);
  G.pairs = (int)std::max<int64_t>(1, std::min<int64_t>(8, ((int64_t)128 << 20) / (tot * (int64_t)sizeof(double2))));
  spectrum = (size_t)tot * (sizeof(double) + sizeof(float));
  work = (size_t)tot * G.pairs * sizeof(double2);
  tables = (size_t)G.L * (sizeof(double2) + sizeof(float2));
}

void grid_op_setup(GridOp &G, cudaStream_t st) {
  const int64_t tot = grid_total(G);
  double2 *X = static_cast<double2 *>(G.work), *tw = static_cast<double2 *>(G.tables);
  double *C = static_cast<double *>(G.spectrum);
  cudaFuncSetAttribute(k_fft_lines<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 << 10);
  cudaFuncSetAttribute(k_fft_lines<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 << 10);
  k_twiddle<<<(G.L + 255) / 256, 256, 0, st>>>(tw, reinterpret_cast<float2 *>(tw + G.L), G.L);
  int64_t cnt = 1;
  for (int d = 0; d < G.dim; d++) cnt *= G.s + 1;
  k_embed_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(X, cnt, G.dim, G.s, G.L, G.h, G.kind, G.w);
  int64_t lim[3] = {G.L, G.L, G.L};
  for (int ax = 0; ax < G.dim; ax++)
    fft_pass<double>(G, X, tw, -1, ax, lim, G.L, G.L, nullptr, 1, st);
  k_spectrum<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(X, tot, 1.0 / (double)tot, C,
                                                           reinterpret_cast<float *>(C + tot));
  count_launch(3);
}

void grid_op_apply(const GridOp &G, const double *x, double *y, int nrhs, cudaStream_t st, bool f32) {
  const double2 *tw = static_cast<const double2 *>(G.tables);
  const double *C = static_cast<const double *>(G.spectrum);
  if (f32)
    grid_op_apply_t<float>(G, static_cast<float2 *>(G.work), reinterpret_cast<const float *>(C + grid_total(G)),
                           reinterpret_cast<const float2 *>(tw + G.L), x, y, nrhs, st);
  else
    grid_op_apply_t<double>(G, static_cast<double2 *>(G.work), C, tw, x, y, nrhs, st);
}

// ---------------------------------------------------------------------------
// FP64 vector kernels for the Krylov loop (column-major n x nrhs blocks).
// Reductions are two-pass and deterministic.
// ---------------------------------------------------------------------------

constexpr int RB = 256;      // threads per reduction block
constexpr int RBLK = 240;    // blocks per column in the first pass

// part[(c * nv + i) * RBLK + blk] = partial sum of V_i[:,c] . w[:,c]
__global__ void __launch_bounds__(RB) k_multidot_part(const double *V, int64_t vstride, int nv, const double *w,
                                                      int64_t n, int nrhs, double *part) {
  __shared__ double red[RB / 32];
  const int c = blockIdx.y, i = blockIdx.z, blk = blockIdx.x;
  const double *vi = V + (int64_t)i * vstride + (int64_t)c * n;
  const double *wc = w + (int64_t)c * n;
  double s = 0.0;
  for (int64_t e = blk * (int64_t)RB + threadIdx.x; e < n; e += (int64_t)RB * RBLK) s += vi[e] * wc[e];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < RB / 32 ? red[threadIdx.x] : 0.0;
    s = warp_sum(s);
    if (threadIdx.x == 0) part[((int64_t)c * nv + i) * RBLK + blk] = s;
  }
}

// a warp per result (a thread summing the 240 parts one after another took
// 15 us); the order is fixed by RBLK
__global__ void k_multidot_final(const double *part, int cnt, double *out) {
  const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (q >= cnt) return;
  double s = 0.0;
  for (int b = lane; b < RBLK; b += 32) s += part[(int64_t)q * RBLK + b];
  s = warp_sum(s);
  if (lane == 0) out[q] = s;
}

// out[c * nv + i] = V_i[:,c] . w[:,c]
void multidot(const double *V, int64_t vstride, int nv, const double *w, int64_t n, int nrhs, double *part,
              double *out, cudaStream_t st) {
  dim3 g(RBLK, nrhs, nv);
  k_multidot_part<<<g, RB, 0, st>>>(V, vstride, nv, w, n, nrhs, part); count_launch();
  int cnt = nrhs * nv;
  k_multidot_final<<<(cnt + 3) / 4, 128, 0, st>>>(part, cnt, out); count_launch();
}

// y[:,c] = alpha * y[:,c] + sum_i coef[c * nv + i] * V_i[:,c]
__global__ void k_combine(double *y, double alpha, const double *V, int64_t vstride, int nv, const double *coef,
                          int64_t n, int nrhs) {
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n * nrhs) return;
  int c = (int)(e / n);
  double s = alpha * y[e];
  for (int i = 0; i < nv; i++) s += coef[c * nv + i] * V[(int64_t)i * vstride + e];
  y[e] = s;
}

void combine(double *y, double alpha, const double *V, int64_t vstride, int nv, const double *coef, int64_t n,
             int nrhs, cudaStream_t st) {
  int64_t tot = n * nrhs;
  if (tot == 0) return;
  k_combine<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(y, alpha, V, vstride, nv, coef, n, nrhs); count_launch();
}

}  // namespace rss
