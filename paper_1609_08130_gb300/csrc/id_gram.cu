// id_gram.cu -- the FP32 factor's ID (Definition 2.1, Sec. 2.2) from the Gram
// matrix of its rows, formed exactly on the tensor cores (tcgen05).
//
// The ID of a box asks for a column-pivoted QR of its m x b matrix M (ring
// rows inside the proxy surface and proxy rows, m about 1100..7000, b <= 512).
// Pivots, ranks and T depend on M only through M^T M: the pivoted Cholesky
// factor of M^T M is the R of the pivoted QR.  Forming M^T M in floating point
// would square the rounding error; here it is formed in integers instead.
// Every 64- (or 96-) column block of a chunk of rows is scaled by its largest
// entry to 22.7-bit integers (an error below FP32 rounding of that largest
// entry; smaller ones keep fewer bits of their own), each integer is three
// base-240 digits in [-120, 120], and the digit products are bf16 MMAs with FP32
// accumulators in tensor memory (operands cut into exactly multiplied slices:
// K. Ozaki, T. Ogita, S. Oishi and S. M. Rump, Numer. Algorithms 59, 2012).  A product is at most
// 14400, so within the row limits below every partial sum stays below 2^24
// and is exact; the digits' sums are put together in 64-bit integers.  The
// result is M^T M of the quantised columns to 48 bits whatever the order.
// The pivoted Cholesky (k_pchol) runs in pairs of FP32 numbers (48 bits): at
// |R_jj| = 1e-6 |R_11| its pivots still carry two digits, as the FP32
// Householder reduction of the same rows does.  eps below ID_GRAM_EPS takes
// that reduction (the other ID kernels).  Errors against FP64: the ID's residual
// is the reduction's at eps 1e-2 to 1e-4 and 0.77 of it at 1e-6 (leaf rows of
// 2D boxes, k the same); the factor's apply error 0.95 of the one with that
// reduction (geometric mean of 40 problems and schedules, single ones 0.7 to
// 1.13: pivots differ).
#include <algorithm>

#include "df.cuh"
#include "internal.h"
#include "tc.cuh"

namespace rss {

namespace {

constexpr int NTG = 256;          // threads of k_gram: warp w stages rows 8 w .. 8 w + 7 of a chunk
constexpr int KC = 64;            // rows per staged chunk
constexpr int RCH_TILE = 1152;    // rows per CTA: 1152 * 120^2 < 2^24
constexpr int RCH_WIDE = 384;     // three products in one accumulator: 384 * 3 * 120^2 < 2^24
constexpr float Q1 = 240.f, Q2 = 57600.f;
constexpr float QMAX = 6911000.f; // below 120 * 240^2
constexpr long long Q = 240;
constexpr long long WAIT_POLLS = 1ll << 20;
constexpr int PC_L = 32;          // columns of L kept in shared memory by k_pchol

// Columns per block: 64 (tiles of two blocks), or one 96-wide block for boxes
// of 65..96 columns (the 2D upper levels), staged once instead of in three
// tiles.
__host__ __device__ constexpr int block_cols(int bmax) { return bmax > 64 && bmax <= 96 ? 96 : 64; }
__host__ __device__ constexpr uint32_t slab_bytes(int tb) { return 3u * tb * 32; }  // K = 16 of a block's digits
__host__ __device__ constexpr uint32_t stage_bytes(int tb) { return slab_bytes(tb) * (KC / 16); }

__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(tc::smem_desc(a, 128, 256)), "l"(tc::smem_desc(b, 128, 256)), "r"(idesc), "r"(acc)
      : "memory");
}
// small integers as bf16: the upper halves of their FP32 words
__device__ __forceinline__ uint32_t pack_bf16(float2 v) {
  return __byte_perm(__float_as_uint(v.x), __float_as_uint(v.y), 0x7632);
}
// nearest integers of x * c, |x c| < 2^22 (the product rounds once, in the sum)
__device__ __forceinline__ float2 rint2(float2 x, float c) {
  const float2 m = __ffma2_rn(x, make_float2(c, c), make_float2(12582912.f, 12582912.f));
  return __fadd2_rn(m, make_float2(-12582912.f, -12582912.f));
}

}  // namespace

static int gram_tiles(int bmax) {
  const int nb = (bmax + block_cols(bmax) - 1) / block_cols(bmax);
  return nb * (nb + 1) / 2;
}
// Rows per CTA: all that stays exact when the phase fills the GPU that way,
// else fewer, so that about two CTAs per SM share the phase; not below 256,
// since every chunk is another partial sum that k_pchol reads.
static int gram_rows(int nbox, int bmax, int m) {
  const int most = block_cols(bmax) == 96 ? RCH_WIDE : RCH_TILE;
  const int64_t per = (int64_t)nbox * gram_tiles(bmax);
  const int want = (int)std::max<int64_t>(1, std::min<int64_t>(64, (304 + per - 1) / per));
  const int rows = std::max(((m + want - 1) / want + KC - 1) / KC * KC, 256);
  const int need = (m + most - 1) / most;  // chunks of equal length within the exact range
  return std::min(rows, ((m + need - 1) / need + KC - 1) / KC * KC);
}
// Scratch of one phase: the chunks' partial Gram tiles, and for boxes wider
// than 128 their sum; L's columns past PC_L.
int64_t id_gram_scratch_bytes(int nbox, int bmax, int m) {
  const int rows = gram_rows(nbox, bmax, m), tb = block_cols(bmax);
  const int C = (m + rows - 1) / rows;
  const int64_t part = (int64_t)C * gram_tiles(bmax) * tb * tb;
  const int64_t full = bmax > 128 ? (int64_t)bmax * bmax : 0;
  const int64_t spill = bmax > PC_L ? (int64_t)(bmax - PC_L) * bmax : 0;
  return (int64_t)nbox * (part + full + spill) * (int64_t)sizeof(Df);
}

// One CTA per (box, chunk of `rch` rows, tile of two blocks I >= J).  Warp w
// loads rows 8 w .. 8 w + 7 of a 64-row step, lane l columns l, l + 32, ...,
// cuts them into digits and stores eight rows of a digit as one 16-byte
// K-major unit; one thread issues the step's MMAs while the next step is
// loaded (two buffers).  The rows are read twice (largest entry first, then
// digits): at the 2D leaf 262 KB a box from L2 / HBM against 2.2 us of MMAs.
// Measured (512^2 grid): leaf phase of 1024 boxes 205 us, a phase of 256
// boxes of 72 columns 180 us in one 96-column block (550 us in three 64-column
// tiles), phases of 4-64 boxes 40-70 us (load latency).
template <int TBW>
__global__ void __launch_bounds__(NTG) k_gram(LevelDev<float> lv, FBox<float> *boxes, const int *box_list, Points P,
                                              KernelParams K, ProxyParams px, const float *proxy_unit, int rch, int C,
                                              int ntile, int ring_max, Df *part, int *err) {
  constexpr bool WIDE = TBW == 96;
  constexpr int NS = TBW / 32;  // columns per lane and side
  constexpr int NSIDE = WIDE ? 1 : 2;
  constexpr uint32_t SLAB = slab_bytes(TBW), STAGE = stage_bytes(TBW);
  constexpr int LDV = TBW + 1;
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ int s_ocode[125], s_obase[126], s_no;
  __shared__ const float *s_row[WIDE ? RCH_WIDE : RCH_TILE];
  __shared__ unsigned s_max[2];
  __shared__ Df s_inv;
  __shared__ __align__(8) uint64_t s_mbar[2];
  __shared__ uint32_t s_tmem;
  const int bi = blockIdx.x / (C * ntile), rem = blockIdx.x % (C * ntile);
  const int chunk = rem / ntile, tile = rem % ntile;
  int I = 0;
  while ((I + 1) * (I + 2) / 2 <= tile) I++;
  const int J = tile - I * (I + 1) / 2;
  FBox<float> &fb = boxes[box_list[bi]];
  const int c = fb.cell, b = fb.b, dim = lv.dim;
  if (I * TBW >= b) return;
  const int nside = I == J ? 1 : 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tmem_cols = WIDE || nside == 2 ? 512 : 256;

  if (tid < 2) s_max[tid] = 0u;
  if (warp == 0) {  // the ring's cells and the first row of each (as in k_idw)
    const int ncode = dim == 3 ? 125 : 25;
    int no = 0, acc = 0;
    for (int base = 0; base < ncode; base += 32) {
      int code = base + lane, cnt = 0;
      if (code < ncode) {
        int dx = code % 5 - 2, dy = (code / 5) % 5 - 2, dz = dim == 3 ? code / 25 - 2 : 0;
        const int dist = max(abs(dx), max(abs(dy), abs(dz)));
        if (dist == 2 || (lv.weak && dist == 1)) {
          int nb = lv.cell_nbr[(int64_t)c * lv.NB + code];
          if (nb >= 0) cnt = lv.act_cnt[nb];
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, cnt > 0);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      const int pos = __popc(mask & ((1u << lane) - 1));
      if (cnt > 0) {
        s_ocode[no + pos] = code;
        s_obase[no + pos] = acc + incl - cnt;
      }
      no += __popc(mask);
      acc += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) {
      s_obase[no] = acc;
      s_no = no;
    }
  }
  // this lane's columns: their points relative to the box centre
  const double Dt = ldexp(1.0, -lv.t);
  const float w = (float)weight_of(P, K, lv.cell_dofs[lv.cell_dof_off[c]]);
  const float rad = (float)(px.radius * Dt);
  int col[NSIDE][NS];
  float xq[NSIDE][NS][3];
#pragma unroll
  for (int s = 0; s < NSIDE; s++)
#pragma unroll
    for (int u = 0; u < NS; u++) {
      const int q = (s == 0 ? I : J) * TBW + u * 32 + lane;
      col[s][u] = q < b ? q : -1;
      const int64_t g = lv.cell_dofs[lv.cell_dof_off[c] + min(q, b - 1)];
#pragma unroll
      for (int d = 0; d < 3; d++)
        xq[s][u][d] = d < dim ? (float)(P.x[g * dim + d] - (lv.cell_coord[3 * c + d] + 0.5) * Dt) : 0.f;
    }
  __syncthreads();
  const int nO = s_obase[s_no], m = nO + px.np;
  const int r0 = chunk * rch, rows = min(rch, m - r0);
  if (nO > ring_max) {  // uniform: every thread sees the same nO
    if (tid == 0) set_err(err, DERR_INTERNAL);
    return;
  }
  if (chunk == 0 && tile == 0 && tid == 0) fb.no = nO;
  if (rows <= 0) return;
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&s_tmem), tmem_cols);
  if (tid < 2) tc::mbar_init(tc::smem_u32(&s_mbar[tid]), 1);
  // this chunk's ring rows: the box's part of a ring DOF's column
  const int nring = max(0, min(rows, nO - r0));
  for (int i = tid; i < nring; i += NTG) {
    const int row = r0 + i;
    int lo = 0, hi = s_no - 1;  // the last cell starting at or before this row
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_obase[mid] <= row) lo = mid;
      else hi = mid - 1;
    }
    const int code = s_ocode[lo];
    const int nb = lv.cell_nbr[(int64_t)c * lv.NB + code];
    s_row[i] = lv.pool + lv.pair_off[(int64_t)c * lv.NB + code] +
               (int64_t)lv.act_idx[lv.cell_dof_off[nb] + (row - s_obase[lo])] * b;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = s_tmem;

  // rows 64 ck + 8 warp + (0..7) of the chunk, this lane's columns of side s
  auto load = [&](int ck, int s, float (&v)[NS][8]) {
    const int i0 = ck * KC + warp * 8;
    if (i0 + 8 <= nring) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float *r = s_row[i0 + i];
#pragma unroll
        for (int u = 0; u < NS; u++) v[u][i] = col[s][u] >= 0 ? r[col[s][u]] : 0.f;
      }
      return;
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const int ri = i0 + i;
      if (ri < nring) {
        const float *r = s_row[ri];
#pragma unroll
        for (int u = 0; u < NS; u++) v[u][i] = col[s][u] >= 0 ? r[col[s][u]] : 0.f;
      } else {
        const float *pu = proxy_unit + 3 * min(r0 + ri - nO, px.np - 1);
        const float y0 = rad * pu[0], y1 = rad * pu[1], y2 = rad * pu[2];
#pragma unroll
        for (int u = 0; u < NS; u++) {
          const float e0 = y0 - xq[s][u][0], e1 = y1 - xq[s][u][1], e2 = y2 - xq[s][u][2];
          const float r2 = e0 * e0 + e1 * e1 + e2 * e2;
          v[u][i] = ri < rows && col[s][u] >= 0 ? w * kof(K.kind, r2) : 0.f;
        }
      }
    }
  };

  const int nck = (rows + KC - 1) / KC;
  // pass 1: the largest magnitude of each block (as bits: NaN above infinity)
#pragma unroll
  for (int s = 0; s < NSIDE; s++) {
    if (s >= nside) break;
    unsigned mx = 0;
#pragma unroll 2
    for (int ck = 0; ck < nck; ck++) {
      float v[NS][8];
      load(ck, s, v);
#pragma unroll
      for (int u = 0; u < NS; u++)
#pragma unroll
        for (int i = 0; i < 8; i++) mx = max(mx, __float_as_uint(v[u][i]) & 0x7fffffffu);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) atomicMax(&s_max[s], mx);
  }
  __syncthreads();
  const float mxI = __uint_as_float(s_max[0]), mxJ = nside == 1 ? mxI : __uint_as_float(s_max[1]);
  const bool finite = mxI < 3.0e38f && mxJ < 3.0e38f;
  const float sc[2] = {finite && mxI > 1e-30f ? QMAX / mxI : 0.f, finite && mxJ > 1e-30f ? QMAX / mxJ : 0.f};
  if (tid == 0) {
    // back to units of the weight, so that the pairs' low parts stay normal
    const double ss = (double)sc[0] * (double)(nside == 1 ? sc[0] : sc[1]) * (double)w * (double)w;
    const double inv = !finite ? (double)NAN : ss > 0.0 ? 1.0 / ss : 0.0;
    s_inv.h = (float)inv;
    s_inv.l = (float)(inv - (double)s_inv.h);
  }

  // pass 2: digits of step ck into buffer ck & 1, then its MMAs
  float v[NSIDE][NS][8];
  const uint32_t base = tc::smem_u32(sm);
  bool ok = true;
#pragma unroll
  for (int s = 0; s < NSIDE; s++)
    if (s < nside) load(0, s, v[s]);
  for (int ck = 0; ck < nck; ck++) {
    const int buf = ck & 1;
    unsigned char *st = sm + (size_t)buf * nside * STAGE;
    bool free_ok = true;
    if (ck >= 2) free_ok = tc::mbar_wait(tc::smem_u32(&s_mbar[buf]), ((ck >> 1) - 1) & 1, WAIT_POLLS);
    if (free_ok) {
#pragma unroll
      for (int s = 0; s < NSIDE; s++) {
        if (s >= nside) break;
#pragma unroll
        for (int u = 0; u < NS; u++) {
          const int q = u * 32 + lane;
          uint32_t d[3][4];
#pragma unroll
          for (int h = 0; h < 4; h++) {
            const float2 t = __fmul2_rn(make_float2(v[s][u][2 * h], v[s][u][2 * h + 1]), make_float2(sc[s], sc[s]));
            const float2 a0 = rint2(t, 1.f / Q2);
            const float2 t1 = __ffma2_rn(a0, make_float2(-Q2, -Q2), t);
            const float2 a1 = rint2(t1, 1.f / Q1);
            const float2 a2 = rint2(__ffma2_rn(a1, make_float2(-Q1, -Q1), t1), 1.f);
            d[0][h] = pack_bf16(a0);
            d[1][h] = pack_bf16(a1);
            d[2][h] = pack_bf16(a2);
          }
          unsigned char *o =
              st + (size_t)s * STAGE + (warp >> 1) * SLAB + (q >> 3) * 256 + (warp & 1) * 128 + (q & 7) * 16;
#pragma unroll
          for (int k = 0; k < 3; k++)
            *reinterpret_cast<uint4 *>(o + k * (TBW * 32)) = make_uint4(d[k][0], d[k][1], d[k][2], d[k][3]);
        }
      }
    }
    if (ck + 1 < nck) {
#pragma unroll
      for (int s = 0; s < NSIDE; s++)
        if (s < nside) load(ck + 1, s, v[s]);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    if (__syncthreads_or(!free_ok)) {
      ok = false;
      break;
    }
    if (tid == 0) {
      tc::fence_after_sync();
      const uint32_t a = base + buf * nside * STAGE, bb = a + (nside - 1) * STAGE;
#pragma unroll 1
      for (int k = 0; k < KC / 16; k++) {
        const uint32_t acc = (ck > 0 || k > 0) ? 1u : 0u;
        const uint32_t ak = a + k * SLAB, bk = bb + k * SLAB;
        if (WIDE) {  // one accumulator per weight of the digit pair
          constexpr uint32_t PL = TBW * 32;
          const uint32_t id = idesc_bf16(128, TBW);
          mma_bf16(tmem, ak, ak, id, acc);
          mma_bf16(tmem + TBW, ak, ak + PL, id, acc);
          mma_bf16(tmem + 2 * TBW, ak, ak + 2 * PL, id, acc);
          mma_bf16(tmem + 2 * TBW, ak + 2 * PL, ak, id, 1u);
          mma_bf16(tmem + 2 * TBW, ak + PL, ak + PL, id, 1u);
          mma_bf16(tmem + 3 * TBW, ak + PL, ak + 2 * PL, id, acc);
          mma_bf16(tmem + 4 * TBW, ak + 2 * PL, ak + 2 * PL, id, acc);
        } else {
          // digits 0, 1 of I against all three of J, then digits 1, 2 of I
          // against digit 2 (diagonal tile) or all three
          mma_bf16(tmem, ak, bk, idesc_bf16(128, 192), acc);
          if (nside == 1) mma_bf16(tmem + 192, ak + TBW * 32, bk + 2 * TBW * 32, idesc_bf16(128, 64), acc);
          else mma_bf16(tmem + 192, ak + TBW * 32, bk, idesc_bf16(128, 192), acc);
        }
      }
      tc::mma_commit(tc::smem_u32(&s_mbar[buf]));
    }
  }
  // the last commit covers every MMA issued before it
  const int last = nck - 1;
  if (ok) {
    const bool done = tc::mbar_wait(tc::smem_u32(&s_mbar[last & 1]), (last >> 1) & 1, WAIT_POLLS);
    ok = !__syncthreads_or(!done);
  }
  if (!ok) {
    if (tid == 0) set_err(err, DERR_INTERNAL);
    tc::mbar_wait(tc::smem_u32(&s_mbar[0]), 0, WAIT_POLLS);  // one more bounded wait before the memory is freed
  } else {
    tc::fence_after_sync();
    // epilogue: sums of digit products by weight; on a diagonal tile V + V^T
    // is twice the Gram matrix
    long long *V = reinterpret_cast<long long *>(sm);
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    if (WIDE) {
      if ((warp & 3) < 3) {
        for (int j0 = half * (TBW / 2); j0 < (half + 1) * (TBW / 2); j0 += 16) {
          long long *o = V + row * LDV + j0;
          float a[16], e[16];
          tc::tmem_ld16(tl + j0, a);
          tc::tmem_ld16(tl + TBW + j0, e);
          int hi[16];
#pragma unroll
          for (int j = 0; j < 16; j++) o[j] = Q * Q * Q * (Q * __float2int_rn(a[j]) + 2ll * __float2int_rn(e[j]));
          tc::tmem_ld16(tl + 2 * TBW + j0, a);
          tc::tmem_ld16(tl + 3 * TBW + j0, e);
#pragma unroll
          for (int j = 0; j < 16; j++) hi[j] = __float2int_rn(e[j]);
          tc::tmem_ld16(tl + 4 * TBW + j0, e);
#pragma unroll
          for (int j = 0; j < 16; j++) o[j] += Q * (Q * __float2int_rn(a[j]) + 2ll * hi[j]) + __float2int_rn(e[j]);
        }
      }
      __syncthreads();
    } else {
      // lane i: row i of I, digit 0; lane 64 + i: digits 1 and 2
      const bool upper = row < TBW;
      for (int pass = 0; pass < 2; pass++) {
        if (upper == (pass == 1)) {  // warp-uniform: lanes 64.. first, then lanes 0..63 add theirs
          for (int j0 = half * (TBW / 2); j0 < (half + 1) * (TBW / 2); j0 += 16) {
            float a0[16], a1[16], a2[16];
            tc::tmem_ld16(tl + j0, a0);
            tc::tmem_ld16(tl + TBW + j0, a1);
            tc::tmem_ld16(tl + 2 * TBW + j0, a2);
            long long *o = V + (row & (TBW - 1)) * LDV + j0;
            if (upper) {
              const long long f = nside == 1 ? 2 : 1;
#pragma unroll
              for (int j = 0; j < 16; j++)
                o[j] += Q * Q * (Q * (Q * __float2int_rn(a0[j]) + f * __float2int_rn(a1[j])) + f * __float2int_rn(a2[j]));
            } else if (nside == 1) {
              tc::tmem_ld16(tl + 192 + j0, a0);
#pragma unroll
              for (int j = 0; j < 16; j++)
                o[j] = Q * (Q * __float2int_rn(a1[j]) + 2ll * __float2int_rn(a2[j])) + __float2int_rn(a0[j]);
            } else {
              float c0[16], c1[16], c2[16];
              tc::tmem_ld16(tl + 192 + j0, c0);
              tc::tmem_ld16(tl + 192 + TBW + j0, c1);
              tc::tmem_ld16(tl + 192 + 2 * TBW + j0, c2);
#pragma unroll
              for (int j = 0; j < 16; j++)
                o[j] = Q * (Q * (Q * __float2int_rn(a0[j]) + (long long)__float2int_rn(a1[j]) + __float2int_rn(c0[j])) +
                            (long long)__float2int_rn(a2[j]) + __float2int_rn(c1[j])) +
                       __float2int_rn(c2[j]);
            }
          }
        }
        __syncthreads();
      }
    }
    const Df inv = s_inv;
    Df *o = part + (((int64_t)bi * C + chunk) * ntile + tile) * (TBW * TBW);
    for (int e = tid; e < TBW * TBW; e += NTG) {
      const int i = e / TBW, j = e % TBW;
      const long long x = nside == 1 ? V[i * LDV + j] + V[j * LDV + i] : 2 * V[i * LDV + j];
      const float h = __ll2float_rn(x);
      o[e] = mul(Df{0.5f * h, 0.5f * __ll2float_rn(x - __float2ll_rn(h))}, inv);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_free(tmem, tmem_cols);
  }
}

// Pivoted Cholesky of a box's Gram matrix (one CTA per box, thread i carries
// row i): step j takes the largest remaining diagonal entry (ties to the
// lowest column), forms column j of L by the left-looking product and updates
// the diagonal; it stops at d <= eps^2 d_0, which is the ID's rule
// |R_jj| <= eps |R_11|.  T = R11^{-1} R12 by back substitution in FP32, a
// column per thread.  Only k of the b columns are ever formed, with one
// barrier each.  The arithmetic is pairs of FP32 numbers: an FP64 operation
// occupies this part's FP64 pipe for 64 cycles a warp, a pair operation 12
// issue slots (a 9-box phase 58 -> 35 us, the 1024-box leaf phase 117 -> 62).
// Bound: the chain of k dependent steps.
template <int NTH>
__global__ void __launch_bounds__(NTH < 256 ? 256 : NTH)
    k_pchol(LevelDev<float> lv, FBox<float> *boxes, const int *box_list, int np, double eps, int rch, int C, int ntile,
            int bmax, const Df *part, Df *full, Df *spill) {
  extern __shared__ __align__(16) unsigned char smp[];
  constexpr int NW = NTH / 32;
  __shared__ unsigned s_key[2][NW];
  __shared__ int s_idx[2][NW];
  __shared__ float s_dl[2][NW];
  __shared__ int s_perm[NTH], s_cnt[NW], s_k;
  const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  FBox<float> &fb = boxes[box_list[blockIdx.x]];
  const int b = fb.b, nch = (fb.no + np + rch - 1) / rch;
  const bool gsm = full == nullptr;
  const int ldg = gsm ? b + 1 : b;
  Df *L = reinterpret_cast<Df *>(smp);  // L[j][i], j < PC_L
  Df *G = gsm ? L + (size_t)PC_L * bmax : full + (int64_t)blockIdx.x * bmax * bmax;
  Df *Ls = spill ? spill + (int64_t)blockIdx.x * (bmax - PC_L) * bmax - (int64_t)PC_L * b : nullptr;
  const int tb = block_cols(bmax);
  const Df *pb = part + (int64_t)blockIdx.x * C * ntile * (tb * tb);
  // the chunks' partial sums, in chunk order: a lower tile at a time, both
  // triangles written
  const int nblk = (b + tb - 1) / tb;
  for (int I = 0; I < nblk; I++)
    for (int J = 0; J <= I; J++) {
      const Df *t0 = pb + (int64_t)(I * (I + 1) / 2 + J) * (tb * tb);
      const int ni = min(tb, b - I * tb), nj = min(tb, b - J * tb);
#pragma unroll 4
      for (int e = tid; e < ni * (tb / 2); e += nthr) {
        const int i = e / (tb / 2), j = 2 * (e % (tb / 2));
        if (j >= nj) continue;
        float4 x = __ldcg(reinterpret_cast<const float4 *>(t0 + i * tb + j));
        Df s0{x.x, x.y}, s1{x.z, x.w};
        for (int ch = 1; ch < nch; ch++) {
          x = __ldcg(reinterpret_cast<const float4 *>(t0 + (int64_t)ch * ntile * (tb * tb) + i * tb + j));
          s0 = add(s0, Df{x.x, x.y});
          s1 = add(s1, Df{x.z, x.w});
        }
        const int gi = I * tb + i, gj = J * tb + j;
        G[(int64_t)gi * ldg + gj] = s0;
        if (I != J) G[(int64_t)gj * ldg + gi] = s0;
        if (j + 1 < nj) {
          G[(int64_t)gi * ldg + gj + 1] = s1;
          if (I != J) G[(int64_t)(gj + 1) * ldg + gi] = s1;
        }
      }
    }
  __syncthreads();
  const bool own = tid < b && tid < NTH;
  int my = -1;  // pivot position of this thread's column
  if (tid < NTH) {
    Df d = own ? G[(int64_t)tid * ldg + tid] : Df{0.f, 0.f};
    float thr = 0.f;
    int j = 0;
    for (; j < b; j++) {
      const int pb2 = j & 1;
      const unsigned key = own && my < 0 && d.h > 0.f ? __float_as_uint(d.h) : 0u;
      const unsigned kw = __reduce_max_sync(0xffffffffu, key);
      const int wl = __ffs(__ballot_sync(0xffffffffu, key == kw)) - 1;
      if (lane == wl) {
        s_key[pb2][warp] = kw;
        s_idx[pb2][warp] = tid;
        s_dl[pb2][warp] = d.l;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(NTH) : "memory");
      int bw = 0;
      unsigned bk = s_key[pb2][0];
#pragma unroll
      for (int x = 1; x < NW; x++)
        if (s_key[pb2][x] > bk) bk = s_key[pb2][x], bw = x;
      const int p = s_idx[pb2][bw];
      const Df dp{__uint_as_float(bk), s_dl[pb2][bw]};
      if (j == 0) thr = (float)(eps * eps * (double)dp.h);
      if (bk == 0u || !(dp.h > thr)) break;
      if (tid == p) my = j;
      const Df y = rsqrt_df(dp);
      if (own) {
        Df s[4] = {G[(int64_t)p * ldg + tid], {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        const int js = min(j, PC_L);
        int l = 0;
        for (; l + 3 < js; l += 4)
#pragma unroll
          for (int u = 0; u < 4; u++) s[u] = sub_mul(s[u], L[(l + u) * b + tid], L[(l + u) * b + p]);
        for (; l < js; l++) s[0] = sub_mul(s[0], L[l * b + tid], L[l * b + p]);
        for (l = PC_L; l < j; l++) s[1] = sub_mul(s[1], Ls[(int64_t)l * b + tid], Ls[(int64_t)l * b + p]);
        const Df x = mul(add(add(s[0], s[1]), add(s[2], s[3])), y);
        (j < PC_L ? L : Ls)[(int64_t)j * b + tid] = x;
        d = sub_mul(d, x, x);
        d = quick_two_sum(d.h, d.l);
      }
    }
    if (tid == 0) s_k = j;
    // positions: pivots in pivot order, then the others in column order
    const unsigned rest = __ballot_sync(0xffffffffu, own && my < 0);
    if (lane == 0) s_cnt[warp] = __popc(rest);
    asm volatile("bar.sync 1, %0;" ::"n"(NTH) : "memory");
    if (own) {
      int pos = my;
      if (pos < 0) {
        pos = j + __popc(rest & ((1u << lane) - 1));
        for (int x = 0; x < warp; x++) pos += s_cnt[x];
      }
      s_perm[pos] = tid;
    }
  }
  __syncthreads();
  const int k = s_k, r = b - k;
  // R = L^T in FP32, rows in pivot order and columns in the final order
  // (over G, which is no longer needed; k x b)
  float *R = reinterpret_cast<float *>(G);
  for (int e = tid; e < k * b; e += nthr) {
    const int i = e / b, cpos = e - i * b;
    R[e] = (i < PC_L ? L : Ls)[(int64_t)i * b + s_perm[cpos]].h;
  }
  __syncthreads();
  for (int cc = k + tid; cc < b; cc += nthr)
    for (int i = k - 1; i >= 0; i--) {
      const float *Ri = R + (int64_t)i * b;
      float a0 = Ri[cc], a1 = 0.f, a2 = 0.f, a3 = 0.f;
      int l = i + 1;
      for (; l + 3 < k; l += 4) {
        a0 -= Ri[l] * R[(int64_t)l * b + cc];
        a1 -= Ri[l + 1] * R[(int64_t)(l + 1) * b + cc];
        a2 -= Ri[l + 2] * R[(int64_t)(l + 2) * b + cc];
        a3 -= Ri[l + 3] * R[(int64_t)(l + 3) * b + cc];
      }
      for (; l < k; l++) a0 -= Ri[l] * R[(int64_t)l * b + cc];
      R[(int64_t)i * b + cc] = ((a0 + a1) + (a2 + a3)) / Ri[i];
    }
  __syncthreads();
  for (int e = tid; e < k * r; e += nthr) {
    const int cc = e / k, i = e - cc * k;
    fb.Tm[e] = R[(int64_t)i * b + k + cc];
  }
  const int64_t coff = lv.cell_dof_off[fb.cell];
  for (int x = tid; x < b; x += nthr) {
    fb.loc[x] = s_perm[x];
    fb.ids[x] = lv.cell_dofs[coff + s_perm[x]];
  }
  if (tid == 0) {
    fb.k = k;
    fb.r = r;
  }
}

static size_t pchol_smem(int bmax) {
  size_t s = (size_t)PC_L * bmax * sizeof(Df);
  if (bmax <= 128) s += (size_t)bmax * (bmax + 1) * sizeof(Df);
  return s;
}

template <int NTH>
static void launch_pchol(const LevelDev<float> &lv, FBox<float> *boxes, const int *box_list, int nbox, int bmax, int np,
                         double eps, int rch, int C, int ntile, const Df *part, Df *full, Df *spill, cudaStream_t st) {
  const size_t smem = pchol_smem(bmax);
  cudaFuncSetAttribute(k_pchol<NTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_pchol<NTH><<<nbox, NTH < 256 ? 256 : NTH, smem, st>>>(lv, boxes, box_list, np, eps, rch, C, ntile, bmax, part, full,
                                                         spill);
  count_launch();
}

template <int TBW>
static void launch_gram(const LevelDev<float> &lv, FBox<float> *boxes, const int *box_list, int nbox, int bmax,
                        int ring_max, const Points &P, const KernelParams &K, const ProxyParams &px,
                        const float *proxy_unit, int rch, int C, int ntile, Df *part, cudaStream_t st, int *err) {
  // operands (one or two sides, two buffers; the 96-wide block's last digit
  // is read 32 rows past its end, into lanes that are not used); the
  // epilogue's exchange tile takes their place
  const int sides = TBW == 64 && bmax > TBW ? 2 : 1;
  const size_t smem = std::max<size_t>((size_t)2 * sides * stage_bytes(TBW) + (TBW == 96 ? 1024 : 0),
                                       (size_t)TBW * (TBW + 1) * sizeof(long long));
  cudaFuncSetAttribute(k_gram<TBW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_gram<TBW><<<(unsigned)((int64_t)nbox * C * ntile), NTG, smem, st>>>(lv, boxes, box_list, P, K, px, proxy_unit, rch,
                                                                       C, ntile, ring_max, part, err);
  count_launch();
}

void launch_id_gram(const LevelDev<float> &lv, FBox<float> *boxes, const int *box_list, int nbox, int bmax,
                    int ring_max, const Points &P, const KernelParams &K, const ProxyParams &px,
                    const float *proxy_unit, double eps, void *scratch, cudaStream_t st, int *err) {
  if (nbox == 0) return;
  const int m = ring_max + px.np, rch = gram_rows(nbox, bmax, m), C = (m + rch - 1) / rch;
  const int ntile = gram_tiles(bmax), tb = block_cols(bmax);
  Df *part = static_cast<Df *>(scratch);
  Df *next = part + (int64_t)nbox * C * ntile * (tb * tb);
  Df *full = nullptr, *spill = nullptr;
  if (bmax > 128) {
    full = next;
    next += (int64_t)nbox * bmax * bmax;
  }
  if (bmax > PC_L) spill = next;
  if (tb == 96)
    launch_gram<96>(lv, boxes, box_list, nbox, bmax, ring_max, P, K, px, proxy_unit, rch, C, ntile, part, st, err);
  else
    launch_gram<64>(lv, boxes, box_list, nbox, bmax, ring_max, P, K, px, proxy_unit, rch, C, ntile, part, st, err);
  if (bmax <= 64)
    launch_pchol<64>(lv, boxes, box_list, nbox, bmax, px.np, eps, rch, C, ntile, part, full, spill, st);
  else if (bmax <= 96)
    launch_pchol<96>(lv, boxes, box_list, nbox, bmax, px.np, eps, rch, C, ntile, part, full, spill, st);
  else if (bmax <= 128)
    launch_pchol<128>(lv, boxes, box_list, nbox, bmax, px.np, eps, rch, C, ntile, part, full, spill, st);
  else if (bmax <= 256)
    launch_pchol<256>(lv, boxes, box_list, nbox, bmax, px.np, eps, rch, C, ntile, part, full, spill, st);
  else
    launch_pchol<512>(lv, boxes, box_list, nbox, bmax, px.np, eps, rch, C, ntile, part, full, spill, st);
}

}  // namespace rss
