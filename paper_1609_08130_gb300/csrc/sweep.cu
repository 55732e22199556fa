// sweep.cu -- the sweeps of the factor's apply (Eq. 3.10) and solve (Eq. 3.11)
// over one colour phase, for groups of up to four right-hand sides.
//
// The columns are held in groups of NR <= 4: group g's tree-order vector is
// v + g * n * NR, entry (dof, c) at [dof * NR + c].  grid.y is the group, so a
// wide block of right-hand sides costs one launch per phase and its groups
// share each other's latency (16 columns of the 256^2 grid took 5.7 ms a solve
// with all columns in one CTA per box, 0.9 ms in four groups; the FP64 solve of
// one column on the 128^2 grid, 56 launches, 1.26 -> 0.74 ms).
//
// A box's rows of J are split into chunks of SWEEP_CHUNK over CTAs.  The CTAs
// of one box meet at a per-box counter: the last to finish (no waiting) writes
// the box's own S and R entries, which every CTA of the box reads first, so
// the result does not depend on which CTA is last.
//
// Bound: large phases by reading the factor once; the many phases of under a
// few hundred CTAs by the chain of dependent loads (box record, indices,
// vector, factor blocks, counter).  Everything before the vector is the same
// in every sweep, so each launch is a programmatic dependent of the one
// before: it reads its records and indices, stages T and prefetches its blocks
// of the factor while the phase before it is still running, then waits for
// that phase's vector entries.
#include <algorithm>

#include "internal.h"

namespace rss {

namespace {

constexpr int NT = 256;
constexpr int MLP = 8;            // independent loads a thread keeps in flight
constexpr int T_STAGE = 2048;     // entries of T staged in shared memory (every 2D box; wider boxes read it from L2)
constexpr int WIDE_ENTRIES = 64 * NT;  // X_RR^{-1} and E_S of a box shared by its CTAs above this
constexpr int SWEEP_SMEM = (200 << 10) + 64;

__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// a contiguous range, one 128-byte line per thread
__device__ __forceinline__ void prefetch_range(const void *p, int64_t bytes) {
  const char *c = static_cast<const char *>(p);
  for (int64_t o = (int64_t)threadIdx.x * 128; o < bytes; o += NT * 128) prefetch_l2(c + o);
}

// out[i] = sum_l A(i, l) x[l] (NR columns each): rows over the threads, the
// columns of A over the remaining groups of threads, the groups' sums added in
// group order.  part: NT x NR entries.  Barriers inside; out is complete on
// return.
template <typename T, int NR, typename A>
__device__ __forceinline__ void mat_vec(int nrow, int ncol, A &&at, const T *x, T *part, T *out) {
  const int tid = threadIdx.x, nr = min(nrow, NT);
  if (nrow == 0) return;
  const int ng = NT / nr;
  for (int i0 = 0; i0 < nrow; i0 += nr) {
    const int i = i0 + tid % nr, g = tid / nr;
    if (i < nrow && g < ng) {
      T acc[NR];
#pragma unroll
      for (int c = 0; c < NR; c++) acc[c] = (T)0;
      for (int l = g; l < ncol; l += MLP * ng) {
        T w[MLP];
#pragma unroll
        for (int u = 0; u < MLP; u++) w[u] = l + u * ng < ncol ? at(i, l + u * ng) : (T)0;
#pragma unroll
        for (int u = 0; u < MLP; u++)
          if (l + u * ng < ncol)
#pragma unroll
            for (int c = 0; c < NR; c++) acc[c] += w[u] * x[(l + u * ng) * NR + c];
      }
#pragma unroll
      for (int c = 0; c < NR; c++) part[(g * nr + (i - i0)) * NR + c] = acc[c];
    }
    __syncthreads();
    for (int e = tid; e < min(nr, nrow - i0) * NR; e += NT) {
      T s = (T)0;
      for (int g2 = 0; g2 < ng; g2++) s += part[g2 * nr * NR + e];
      out[i0 * NR + e] = s;
    }
    __syncthreads();
  }
}

// What a CTA reads before the vector: its box, the ids of its S and R DOFs,
// T when it is small.
template <typename T, int NR> struct Box {
  const FBox<T> &fb;
  int k, r, nj, ch, nchunk;
  int64_t *ids;          // S then R
  T *vB, *w, *part, *Ts;  // v_S then v_R; b x NR; NT x NR; staged T
  bool staged;
};
// Dynamic shared memory: ids, v_S/v_R, three b-vectors, partial sums, a chunk
// of v_J, staged T.
template <typename T> __host__ __device__ size_t sweep_smem(int b, int nr) {
  return (size_t)b * sizeof(int64_t) + ((size_t)4 * b + NT + SWEEP_CHUNK) * nr * sizeof(T) + T_STAGE * sizeof(T) + 64;
}

template <typename T, int NR>
__device__ __forceinline__ Box<T, NR> open_box(const FBox<T> *boxes, int bi, int ch, unsigned char *sm) {
  const FBox<T> &fb = boxes[bi];
  Box<T, NR> x{fb, fb.k, fb.r, fb.nj, ch, 0, nullptr, nullptr, nullptr, nullptr, nullptr, false};
  const int b = x.k + x.r;
  x.nchunk = max(1, (x.nj + SWEEP_CHUNK - 1) / SWEEP_CHUNK);
  x.ids = reinterpret_cast<int64_t *>(sm);
  x.vB = reinterpret_cast<T *>(x.ids + b);
  x.w = x.vB + (size_t)b * NR;
  x.part = x.w + (size_t)2 * b * NR;  // two b-vectors at w
  x.Ts = x.part + (size_t)NT * NR;
  x.staged = x.k * x.r <= T_STAGE;
  for (int e = threadIdx.x; e < b; e += NT) x.ids[e] = fb.ids[e];
  if (x.staged)
    for (int e = threadIdx.x; e < x.k * x.r; e += NT) x.Ts[e] = __ldg(fb.Tm + e);
  else
    prefetch_range(fb.Tm, (int64_t)x.k * x.r * sizeof(T));
  return x;
}
// T(q, ri)
template <typename T, int NR> __device__ __forceinline__ T tval(const Box<T, NR> &x, int q, int ri) {
  return x.staged ? x.Ts[q + ri * x.k] : __ldg(x.fb.Tm + q + (int64_t)ri * x.k);
}
template <typename T, int NR> __device__ __forceinline__ void gather_box(const Box<T, NR> &x, const T *v) {
  for (int e = threadIdx.x; e < (x.k + x.r) * NR; e += NT) x.vB[e] = v[x.ids[e / NR] * NR + e % NR];
}
// Whether this CTA is the last of its box to get here (uniform).
__device__ __forceinline__ bool last_of_box(int *cnt, int nchunk, int *s_last) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool last = nchunk == 1 || atomicAdd(cnt, 1) == nchunk - 1;
    if (last && nchunk > 1) *cnt = 0;
    *s_last = last;
  }
  __syncthreads();
  return *s_last != 0;
}

// v_N += sgn * E_N x_R over this CTA's rows of J past the box's own S: two
// threads per row, each over alternate columns.  x: r x NR.  Near DOFs are
// added to without reading them back (other boxes of a 2^d phase may add to
// them too).
template <typename T, int NR>
__device__ __forceinline__ void add_near(const Box<T, NR> &x, int64_t jid, const T *xr, T sgn, T *v) {
  const int a = x.ch * SWEEP_CHUNK + (threadIdx.x >> 1), h = threadIdx.x & 1;
  const bool mine = a < x.nj && a >= x.k;
  const T *ea = x.fb.E + a;
  T acc[NR];
#pragma unroll
  for (int c = 0; c < NR; c++) acc[c] = (T)0;
  for (int ri = mine ? h : x.r; ri < x.r; ri += 2 * MLP) {
    T ev[MLP];
#pragma unroll
    for (int u = 0; u < MLP; u++) ev[u] = ri + 2 * u < x.r ? __ldg(ea + (int64_t)(ri + 2 * u) * x.nj) : (T)0;
#pragma unroll
    for (int u = 0; u < MLP; u++)
      if (ri + 2 * u < x.r)
#pragma unroll
        for (int c = 0; c < NR; c++) acc[c] += ev[u] * xr[(ri + 2 * u) * NR + c];
  }
#pragma unroll
  for (int c = 0; c < NR; c++) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 1);
  if (mine && h == 0) {
    T *vg = v + jid * NR;
#pragma unroll
    for (int c = 0; c < NR; c++) atomicAdd(vg + c, sgn * acc[c]);
  }
}
// this thread's row of the chunk (add_near), and the chunk's part of E
template <typename T, int NR> __device__ __forceinline__ int64_t near_id(const Box<T, NR> &x) {
  const int a0 = x.ch * SWEEP_CHUNK, a = a0 + (threadIdx.x >> 1);
  const int rows = min(SWEEP_CHUNK, x.nj - a0);
  // one line per (column, 128 bytes of rows)
  if (rows > 0) {
    const int per = (rows * (int)sizeof(T) + 127) / 128 + 1;
    for (int e = threadIdx.x; e < x.r * per; e += NT) {
      const int ri = e / per, o = min((e % per) * (int)(128 / sizeof(T)), rows - 1);
      prefetch_l2(x.fb.E + a0 + o + (int64_t)ri * x.nj);
    }
  }
  return a < x.nj ? x.fb.J[a] : 0;
}

}  // namespace

// Solve, forward: y = v_R - T^T v_S; v_N -= E_N y; the last CTA: v_S -= E_S y,
// v_R = X_RR^{-1} y.  Where that last product is more than 64 entries a thread
// (the 32^3 grid's upper boxes: 137, a chain of 22 rounds of loads) every CTA
// forms its share of the rows and the last one only adds them in (32^3 case
// 22.9 -> 21.6 ms); below, the round trip through memory costs more than it
// saves.  For one or two columns: with more the registers it takes slowed the
// large phases (16 columns on the 256^2 grid by 1 %).
template <typename T, int NR>
__global__ void __launch_bounds__(NT) k_sweep_fwd(const FBox<T> *boxes, const int *wbox, const int *wchunk, T *vall,
                                                  int64_t vstride, int *cntall, int nbox, T *pball, int64_t pstride,
                                                  const int64_t *poff) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int s_last;
  pdl_launch_next();
  const int bi = wbox[blockIdx.x], ch = wchunk[blockIdx.x], tid = threadIdx.x;
  T *v = vall + blockIdx.y * vstride;
  Box<T, NR> x = open_box<T, NR>(boxes, bi, ch, sm);
  const int k = x.k, r = x.r, nj = x.nj;
  const int64_t jid = near_id(x);
  if (ch == 0) prefetch_range(x.fb.Xi, (int64_t)r * r * sizeof(T));
  __syncthreads();
  pdl_wait();
  gather_box(x, v);
  __syncthreads();
  T *y = x.w, *z = x.w + (size_t)(k + r) * NR;
  mat_vec<T, NR>(r, k, [&](int i, int q) { return tval(x, q, i); }, x.vB, x.part, y);
  for (int e = tid; e < r * NR; e += NT) y[e] = x.vB[k * NR + e] - y[e];
  __syncthreads();
  add_near(x, jid, y, (T)-1, v);
  // the k rows of E at the head of J and the r rows of X_RR^{-1} as one
  // product of b rows, i0 .. i0 + ni - 1 of them
  const T *E = x.fb.E, *Xi = x.fb.Xi;
  auto product = [&](int i0, int ni, T *out) {
    mat_vec<T, NR>(ni, r,
                   [&](int i, int l) {
                     return i0 + i < k ? __ldg(E + i0 + i + (int64_t)l * nj) : __ldg(Xi + (i0 + i - k) + (int64_t)l * r);
                   },
                   y, x.part, out);
  };
  // the partial sums' space of the backward sweep holds r rows a chunk
  const bool shared_rows = NR <= 2 && (k + r) * r > WIDE_ENTRIES && x.nchunk > 1 && k + r <= x.nchunk * r;
  T *p0 = pball + blockIdx.y * pstride + poff[bi];
  if (shared_rows) {
    const int per = (k + r + x.nchunk - 1) / x.nchunk, i0 = min(k + r, ch * per);
    product(i0, min(per, k + r - i0), p0 + (int64_t)i0 * NR);
    __threadfence();
  }
  if (!last_of_box(cntall + (int64_t)blockIdx.y * nbox + bi, x.nchunk, &s_last)) return;
  if (shared_rows) {
    __threadfence();
    for (int e = tid; e < (k + r) * NR; e += NT) z[e] = __ldcg(p0 + e);
    __syncthreads();
  } else {
    product(0, k + r, z);
  }
  for (int e = tid; e < (k + r) * NR; e += NT) v[x.ids[e / NR] * NR + e % NR] = e < k * NR ? x.vB[e] - z[e] : z[e];
}

// Partial sums of G v_J over this CTA's chunk of J into pb (r x NR); vJ: the
// chunk's entries in shared memory.
template <typename T, int NR>
__device__ __forceinline__ void near_product(const Box<T, NR> &x, const T *vJ, T *pb) {
  const int a0 = x.ch * SWEEP_CHUNK, na = min(x.nj, a0 + SWEEP_CHUNK) - a0;
  // G(i, a): the stored G, or E^T under symmetric storage
  const T *g = x.fb.G ? x.fb.G + (int64_t)a0 * x.r : x.fb.E + a0;
  const int64_t gsi = x.fb.G ? 1 : x.nj, gsa = x.fb.G ? x.r : 1;
  mat_vec<T, NR>(x.r, max(na, 0), [&](int i, int a) { return __ldg(g + i * gsi + a * gsa); }, vJ, x.part, pb);
}
// the sum over the chunks, once every CTA of the box has written its part
template <typename T, int NR>
__device__ __forceinline__ void sum_chunks(const Box<T, NR> &x, const T *p0, T *out, T sgn) {
  for (int e = threadIdx.x; e < x.r * NR; e += NT) {
    T s = (T)0;
    for (int c = 0; c < x.nchunk; c++) s += __ldcg(p0 + (int64_t)c * x.r * NR + e);
    out[e] += sgn * s;
  }
  __syncthreads();
}
// ids of the chunk of J (into shared memory) and prefetch of its part of G
template <typename T, int NR>
__device__ __forceinline__ int near_ids(const Box<T, NR> &x, int64_t *jids) {
  const int a0 = x.ch * SWEEP_CHUNK, na = max(0, min(x.nj, a0 + SWEEP_CHUNK) - a0);
  for (int e = threadIdx.x; e < na; e += NT) jids[e] = x.fb.J[a0 + e];
  if (x.fb.G) prefetch_range(x.fb.G + (int64_t)a0 * x.r, (int64_t)na * x.r * sizeof(T));
  return na;
}

// Solve, backward: v_R -= G v_J (partial sums per chunk); the last CTA adds
// them in chunk order, v_S -= T v_R, and writes v_R and v_S.
template <typename T, int NR>
__global__ void __launch_bounds__(NT) k_sweep_bwd(const FBox<T> *boxes, const int *wbox, const int *wchunk, T *vall,
                                                  int64_t vstride, int *cntall, int nbox, T *pball, int64_t pstride,
                                                  const int64_t *poff) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int64_t s_j[SWEEP_CHUNK];
  __shared__ int s_last;
  pdl_launch_next();
  const int bi = wbox[blockIdx.x], ch = wchunk[blockIdx.x], tid = threadIdx.x;
  T *v = vall + blockIdx.y * vstride, *p0 = pball + blockIdx.y * pstride + poff[bi];
  Box<T, NR> x = open_box<T, NR>(boxes, bi, ch, sm);
  const int k = x.k, r = x.r;
  const int na = near_ids(x, s_j);
  __syncthreads();
  pdl_wait();
  T *vJ = x.Ts + T_STAGE;
  for (int e = tid; e < na * NR; e += NT) vJ[e] = v[s_j[e / NR] * NR + e % NR];
  gather_box(x, v);
  __syncthreads();
  near_product(x, vJ, p0 + (int64_t)ch * r * NR);
  __threadfence();
  if (!last_of_box(cntall + (int64_t)blockIdx.y * nbox + bi, x.nchunk, &s_last)) return;
  __threadfence();
  T *vR = x.vB + (size_t)k * NR;
  sum_chunks(x, p0, vR, (T)-1);
  mat_vec<T, NR>(k, r, [&](int q, int ri) { return tval(x, q, ri); }, vR, x.part, x.w);
  for (int e = tid; e < (k + r) * NR; e += NT)
    v[x.ids[e / NR] * NR + e % NR] = e < k * NR ? x.vB[e] - x.w[e] : x.vB[e];
}

// Apply, forward: v_S += T v_R, v_R += G v_J (v_J with the new v_S; partial
// sums per chunk); the last CTA: v_R = P^T L U v_R.
template <typename T, int NR>
__global__ void __launch_bounds__(NT) k_apply_fwd(const FBox<T> *boxes, const int *wbox, const int *wchunk, T *vall,
                                                  int64_t vstride, int *cntall, int nbox, T *pball, int64_t pstride,
                                                  const int64_t *poff) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int64_t s_j[SWEEP_CHUNK];
  __shared__ int s_last;
  pdl_launch_next();
  const int bi = wbox[blockIdx.x], ch = wchunk[blockIdx.x], tid = threadIdx.x;
  T *v = vall + blockIdx.y * vstride, *p0 = pball + blockIdx.y * pstride + poff[bi];
  Box<T, NR> x = open_box<T, NR>(boxes, bi, ch, sm);
  const int k = x.k, r = x.r, a0 = ch * SWEEP_CHUNK;
  const int na = near_ids(x, s_j);
  if (ch == 0) prefetch_range(x.fb.LU, (int64_t)r * r * sizeof(T));
  __syncthreads();
  pdl_wait();
  T *vJ = x.Ts + T_STAGE, *vR = x.vB + (size_t)k * NR;
  for (int e = tid; e < na * NR; e += NT) vJ[e] = v[s_j[e / NR] * NR + e % NR];
  gather_box(x, v);
  __syncthreads();
  // every CTA forms the new v_S: the chunks with S rows need it, the last one writes it
  mat_vec<T, NR>(k, r, [&](int q, int ri) { return tval(x, q, ri); }, vR, x.part, x.w);
  for (int e = tid; e < k * NR; e += NT) {
    x.vB[e] += x.w[e];
    if (e >= a0 * NR && e < (a0 + na) * NR) vJ[e - a0 * NR] = x.vB[e];
  }
  __syncthreads();
  near_product(x, vJ, p0 + (int64_t)ch * r * NR);
  __threadfence();
  if (!last_of_box(cntall + (int64_t)blockIdx.y * nbox + bi, x.nchunk, &s_last)) return;
  __threadfence();
  sum_chunks(x, p0, vR, (T)1);
  // U v_R, then L of it (row-major LU), as full products with zeros: a warp per
  // row spent 20 FP64 additions of its lanes' sums on 4 results, 14 us of the
  // FP64 unit per triangle at r = 60
  const T *LU = x.fb.LU;
  T *y = x.w, *z = x.w + (size_t)(k + r) * NR;
  mat_vec<T, NR>(r, r, [&](int i, int l) { return l >= i ? __ldg(LU + (int64_t)i * r + l) : (T)0; }, vR, x.part, y);
  mat_vec<T, NR>(r, r, [&](int i, int l) { return l < i ? __ldg(LU + (int64_t)i * r + l) : (T)0; }, y, x.part, z);
  for (int e = tid; e < r * NR; e += NT) v[x.ids[k + x.fb.piv[e / NR]] * NR + e % NR] = y[e] + z[e];
  for (int e = tid; e < k * NR; e += NT) v[x.ids[e / NR] * NR + e % NR] = x.vB[e];
}

// Apply, backward: v_N += E_N v_R; the last CTA: v_S += E_S v_R, then
// v_R += T^T v_S.
template <typename T, int NR>
__global__ void __launch_bounds__(NT) k_apply_bwd(const FBox<T> *boxes, const int *wbox, const int *wchunk, T *vall,
                                                  int64_t vstride, int *cntall, int nbox) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int s_last;
  pdl_launch_next();
  const int bi = wbox[blockIdx.x], ch = wchunk[blockIdx.x], tid = threadIdx.x;
  T *v = vall + blockIdx.y * vstride;
  Box<T, NR> x = open_box<T, NR>(boxes, bi, ch, sm);
  const int k = x.k, r = x.r, nj = x.nj;
  const int64_t jid = near_id(x);
  __syncthreads();
  pdl_wait();
  gather_box(x, v);
  __syncthreads();
  T *vR = x.vB + (size_t)k * NR;
  add_near(x, jid, vR, (T)1, v);
  if (!last_of_box(cntall + (int64_t)blockIdx.y * nbox + bi, x.nchunk, &s_last)) return;
  const T *E = x.fb.E;
  mat_vec<T, NR>(k, r, [&](int i, int l) { return __ldg(E + i + (int64_t)l * nj); }, vR, x.part, x.w);
  for (int e = tid; e < k * NR; e += NT) x.vB[e] += x.w[e];
  __syncthreads();
  mat_vec<T, NR>(r, k, [&](int i, int q) { return tval(x, q, i); }, x.vB, x.part, x.w);
  for (int e = tid; e < (k + r) * NR; e += NT)
    v[x.ids[e / NR] * NR + e % NR] = e < k * NR ? x.vB[e] : x.vB[e] + x.w[e - k * NR];
}

size_t sweep_chunk_smem(int bmax, int nrhs, int elem) {
  return elem == 4 ? sweep_smem<float>(bmax, nrhs) : sweep_smem<double>(bmax, nrhs);
}

// One phase as a programmatic dependent of the launch before it.
template <typename... P, typename... A>
static void launch_dependent(void (*kernel)(P...), dim3 grid, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
  count_launch();
}

template <typename T, int NR> static void chunk_attributes() {
  cudaFuncSetAttribute(k_sweep_fwd<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_SMEM);
  cudaFuncSetAttribute(k_sweep_bwd<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_SMEM);
  cudaFuncSetAttribute(k_apply_fwd<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_SMEM);
  cudaFuncSetAttribute(k_apply_bwd<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_SMEM);
}

template <typename T, int NR>
static void launch_chunks(int mode, const SweepWork<T> &w, int bmax, T *v, int64_t n, int groups, cudaStream_t st) {
  const dim3 grid((unsigned)w.nwork, (unsigned)groups);
  const size_t smem = sweep_smem<T>(bmax, NR);
  // a limit raised by an earlier uncaptured launch also serves captured ones
  if (smem > (size_t)(48 << 10)) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone) chunk_attributes<T, NR>();
  }
  const int64_t vs = n * NR;
  if (mode == SWEEP_SOLVE_FWD)
    launch_dependent(k_sweep_fwd<T, NR>, grid, smem, st, w.boxes, w.wbox, w.wchunk, v, vs, w.cnt, w.nbox, w.pbuf,
                     w.pstride, w.poff);
  else if (mode == SWEEP_SOLVE_BWD)
    launch_dependent(k_sweep_bwd<T, NR>, grid, smem, st, w.boxes, w.wbox, w.wchunk, v, vs, w.cnt, w.nbox, w.pbuf,
                     w.pstride, w.poff);
  else if (mode == SWEEP_APPLY_FWD)
    launch_dependent(k_apply_fwd<T, NR>, grid, smem, st, w.boxes, w.wbox, w.wchunk, v, vs, w.cnt, w.nbox, w.pbuf,
                     w.pstride, w.poff);
  else
    launch_dependent(k_apply_bwd<T, NR>, grid, smem, st, w.boxes, w.wbox, w.wchunk, v, vs, w.cnt, w.nbox);
}

template <typename T>
void launch_sweep_chunks(int mode, const SweepWork<T> &w, int bmax, T *v, int64_t n, int nr, int groups,
                         cudaStream_t st) {
  if (w.nwork == 0) return;
  switch (nr) {
    case 1: launch_chunks<T, 1>(mode, w, bmax, v, n, groups, st); break;
    case 2: launch_chunks<T, 2>(mode, w, bmax, v, n, groups, st); break;
    case 3: launch_chunks<T, 3>(mode, w, bmax, v, n, groups, st); break;
    default: launch_chunks<T, 4>(mode, w, bmax, v, n, groups, st); break;
  }
}

void sweep_chunk_attributes() {
  chunk_attributes<float, 1>(), chunk_attributes<float, 2>(), chunk_attributes<float, 3>(), chunk_attributes<float, 4>();
  chunk_attributes<double, 1>(), chunk_attributes<double, 2>(), chunk_attributes<double, 3>(),
      chunk_attributes<double, 4>();
}

template void launch_sweep_chunks<float>(int, const SweepWork<float> &, int, float *, int64_t, int, int, cudaStream_t);
template void launch_sweep_chunks<double>(int, const SweepWork<double> &, int, double *, int64_t, int, int,
                                          cudaStream_t);

}  // namespace rss
