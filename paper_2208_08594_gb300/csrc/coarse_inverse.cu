// Dense FP64 inverse of the coarsest AMG matrix (Section 5: a direct solver).  The matrix is
// scaled by powers of two per row and column (exact; undone at the end), inverted by blocked
// in-place Gauss-Jordan with partial pivoting, and the inverse corrected once.  One step of the
// elimination takes the kP = 96 columns K:
//   1. LU with partial pivoting of the rows k0..n-1 of a copy of those columns, in
//      sub-panels of W columns by one thread-block cluster (lu_panel_kernel) with rank-W
//      updates of the rest of the copy in between (lu_update_kernel);
//   2. D = A_KK^-1 from the factors, one warp per column (diag_inverse_panel_kernel), and
//      the panel's row exchanges applied to all columns of A (swap_slice_kernel);
//   3. A_iK <- P_iK = -A_iK D for the rows outside K, A_KK <- D, and with T = A_K,: before
//      the step, A_ij += P_iK T_j outside K and A_Kj = D T_j (slice_gemm_kernel).
// Step 3 is 2 n^3 flops in all.  The FP64 pipes do 1.25 TFLOP/s on this part, so it runs on
// the fifth-generation tensor cores instead, by the error-free splitting of Ozaki, Ogita, Oishi
// and Rump (Numer. Algorithms 59, 2012): every FP64 operand is scaled by a power of two per row
// of P (per column of T) and written as eight signed radix-256 digits, integers that bf16 holds
// exactly.  The product of two digits is at most 2^14, and the sum over 96 terms and the up to
// eight digit pairs (i, j) with the same i + j at most 8 * 96 * 2^14 < 2^24, so every FP32
// accumulator holds an exact integer.  The 36 pairs with i + j <= 9 are kept (seven digits lost
// accuracy where a row's entries differ widely); an epilogue adds the eight sums in integer
// arithmetic and rounds when it adds them to C.  Every instruction multiplies digit i of P by
// the digits 1..9-i of T side by side (N = 32 (9 - i)), each into the accumulator columns of its
// i + j.
//
// Such a product errs by about 2^-56 of its row's times its column's largest operand: as an
// FP64 product in norm, but operands below 2^-10 of their row's or column's maximum keep fewer
// than 53 bits, so small entries of the inverse lose digits (5e-9 to 2e-7 of themselves), and
// where rows of A are in other units than the rest so do the large ones (four rows times 1e10:
// 2e-9 of the largest entry; FP64 elimination 7e-16).  Hence the scaling, and after the
// elimination one step X += X (I - B X): the residual in FP64 from the sparse matrix B, the
// product in six digits of the already small term.  Errors against an extended-precision
// inverse, digits alone / now / FP64 elimination, as a fraction of the largest entry and of the
// entry itself (emulated): coarsest level of 742 rows 2e-16 / 3e-16 / 8e-16 and 8e-9 / 4e-13 /
// 9e-13; permeabilities e^(4N) 9e-15 / 6e-15 / 1e-14 and 2e-7 / 4e-13 / 2e-11; rows times
// 10^U[-9,9] 4e-3 / 9e-17 / 1e-11 and 7e3 / 9e-16 / 7e-6; an exchange in every column, 1,000 rows,
// 3e-15 / 1e-14 / 2e-13 and 4e-9 / 2e-9 / 2e-8.
//
// One SETUP's inverse, with rank-32 updates on the FP64 pipes (two launches per column) and now:
// n = 2,048: 45 -> 14.5 ms, 4,231: 203 -> 36.5 ms, 5,867: 446 -> 60 ms, 9,836: 1,824 -> 164 ms; of
// it the correction 1, 6.5, 14 and 55 ms.  What bounds it: the panels' columns (3.5 us each, a
// chain of one cluster exchange, a reciprocal and the rank-1 update) up to about 6,000 rows,
// above that the products, a tile's chain of MMAs and an epilogue that keeps the FP64 pipe half
// busy (tensor pipe 19 to 28 %).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "setup_kernels.h"

namespace msp {

namespace {

namespace cg = cooperative_groups;

constexpr int kP = 96;         // columns of a Gauss-Jordan step
constexpr int kRowTile = 128;  // rows of a product tile (one MMA's M)
constexpr int kColTile = 32;   // columns of a product tile
constexpr int kKTiles = kP / kColTile;
constexpr int kChunk = 16;     // columns of K per copy (one MMA's K)
constexpr int kStages = 4;     // chunk buffers of a column tile's digits
// A product's operands in ND radix-256 digits over kK columns: eight digits and 96 columns in
// the elimination, six and 128 in the correction (the same bytes, and the same bound
// ND kK 2^14 < 2^24 on the sums).  Bytes of one K chunk of a row tile's / column tile's
// digits (bf16, core matrices of 8 rows x 16 bytes).
constexpr int kSliceA = kRowTile * kChunk * 2;            // one digit of a row tile
template <int ND>
struct Geo {
  static constexpr int kK = 8 * kP / ND;                  // columns of K per product
  static constexpr int kChunks = kK / kChunk;
  static constexpr int kChunkA = ND * kSliceA;            // 32,768 or 24,576
  static constexpr int kRowsB = ND * kColTile;            // digits side by side
  static constexpr int kChunkB = kRowsB * kChunk * 2;     // 8,192 or 6,144
  static constexpr int kDigitB = (kColTile / 8) * 128;    // one digit of a column tile's chunk
};
constexpr int kTileA = Geo<8>::kChunks * Geo<8>::kChunkA;  // 196,608
constexpr int kTileB = Geo<8>::kChunks * Geo<8>::kChunkB;  // 49,152
constexpr int kCorrDigits = 6;
using CorrGeo = Geo<kCorrDigits>;
static_assert(CorrGeo::kChunks * CorrGeo::kChunkA == kTileA && CorrGeo::kChunks * CorrGeo::kChunkB == kTileB);
constexpr int kZeroExp = -4000;                           // exponent of an all-zero row

inline int launch_status() { return launch_check(__FILE__, __LINE__); }

// The dense matrices are stored by tiles of 128 rows x 32 columns (row tiles of `nct` column
// tiles), a tile by pairs of columns, then rows: the 32 rows that a warp of the products'
// epilogue holds are 512 consecutive bytes.  (With rows of the whole matrix each lane
// touched its own line and the L1 was the busiest unit: n = 9,836 157 -> 126 ms, 5,867 57 -> 47 ms.)
__device__ __forceinline__ size_t tile_at(int nct, int i, int j) {
  return ((size_t)(i / kRowTile) * nct + j / kColTile) * (kRowTile * kColTile) +
         (size_t)((j % kColTile) / 2) * (2 * kRowTile) + (i % kRowTile) * 2 + (j & 1);
}

__device__ void raise_flag(DevFlags* f, int code, int index) {
  if (atomicCAS(&f->code, MSP_OK, code) == MSP_OK) f->index = index;
}

// ------------------------------------------------------------------ digits
// e with |x| < 2^e for every |x| <= amax; amax 0 -> kZeroExp; not finite -> a large
// exponent, so that every product with the row is not finite either
__device__ __forceinline__ int scale_exp(double amax) {
  if (amax == 0.0) return kZeroExp;
  const int e = (int)((__double_as_longlong(amax) >> 52) & 0x7ff);
  if (e == 0x7ff) return 1 << 20;
  return max(e - 1022, -900);  // entries below 2^-955 lose digits
}

// x / 2^e (below 1) as a signed 64-bit integer in units of 2^-63
__device__ __forceinline__ long long scaled_int(double x, int e) {
  if (e == kZeroExp) return 0;
  if (e > 2000) return 1LL << 40;  // any nonzero value: the exponent makes it infinite
  // 2^(63 - e) in two factors, both representable
  const int h = (63 - e) / 2, k = 63 - e - h;
  const double s0 = __longlong_as_double((long long)(h + 1023) << 52);
  const double s1 = __longlong_as_double((long long)(k + 1023) << 52);
  return __double2ll_rn(x * s0 * s1);
}

__device__ __forceinline__ unsigned bf16_of_int(int d) {  // exact for |d| <= 256
  return __float_as_uint((float)d) >> 16;
}

// the ND leading digits of eight consecutive operands along K, packed eight bf16 per digit:
// digit s (0 = most significant) to dst + s * stride
template <int ND>
__device__ __forceinline__ void store_digits8(const double (&x)[8], int e, char* dst,
                                              size_t stride) {
  long long v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v[q] = scaled_int(x[q], e);
    if (ND < 8) v[q] = ((v[q] >> (63 - 8 * ND)) + 1) >> 1;  // rounded to the digits kept
  }
#pragma unroll
  for (int s = ND - 1; s >= 0; --s) {
    unsigned w[4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int d;
      if (s > 0) {
        d = (int)(((unsigned)v[q] + 128u) & 255u) - 128;
        v[q] = (v[q] - d) >> 8;
      } else {
        d = (int)v[q];  // |v| <= 128
      }
      const unsigned h = bf16_of_int(d);
      if (q & 1)
        w[q / 2] |= h << 16;
      else
        w[q / 2] = h;
    }
    *reinterpret_cast<uint4*>(dst + (size_t)s * stride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// digit 0 of row i, 16-byte group kcg of K, in the row tiles' images
template <int ND>
__device__ __forceinline__ char* digit_a(char* S, int i, int kcg) {
  const int tr = i % kRowTile;
  return S + (size_t)(i / kRowTile) * kTileA + (size_t)(kcg / 2) * Geo<ND>::kChunkA +
         (kcg % 2) * (kRowTile / 8) * 128 + (tr / 8) * 128 + (tr % 8) * 16;
}
// digit 0 of column c (of a tile of 32), 16-byte group kcg of K, in a column tile's image
template <int ND>
__device__ __forceinline__ char* digit_b(char* tile, int c, int kcg) {
  return tile + (size_t)(kcg / 2) * Geo<ND>::kChunkB + (kcg % 2) * (Geo<ND>::kRowsB / 8) * 128 +
         (c / 8) * 128 + (c % 8) * 16;
}

// Digits of the rows of a tile of 32 rows of A[:, k0..k0+96) (A padded: whole tiles exist),
// and the row exponents.  With Y the rows [z0, z1) are taken as zeros, and Y (96 columns)
// receives A[:, k0..k0+96) with -I in the rows [z0, z1).
__global__ void __launch_bounds__(256) slice_rows_kernel(int nct, int k0, int z0, int z1,
                                                         const double* __restrict__ A,
                                                         char* __restrict__ S,
                                                         int* __restrict__ exps,
                                                         double* __restrict__ Y) {
  __shared__ double sh[32][kP + 1];
  __shared__ int se[32];
  const int r0 = blockIdx.x * 32;
#pragma unroll
  for (int t = threadIdx.x; t < 32 * (kP / 2); t += 256) {
    const int r = t % 32, q = t / 32 * 2, i = r0 + r;
    const bool z = Y && i >= z0 && i < z1;
    double2 x = make_double2(0.0, 0.0);
    if (!z) x = *reinterpret_cast<const double2*>(A + tile_at(nct, i, k0 + q));
    sh[r][q] = x.x;
    sh[r][q + 1] = x.y;
    if (Y) {
      if (z) x = make_double2(i - z0 == q ? -1.0 : 0.0, i - z0 == q + 1 ? -1.0 : 0.0);
      *reinterpret_cast<double2*>(Y + tile_at(kKTiles, i, q)) = x;
    }
  }
  __syncthreads();
  {
    const int r = threadIdx.x / 8, l = threadIdx.x % 8;  // eight lanes per row
    double m = 0.0;
    bool bad = false;
    for (int q = l; q < kP; q += 8) {
      const double a = fabs(sh[r][q]);
      bad |= !isfinite(a);
      m = fmax(m, a);
    }
    if (bad) m = __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o, 8));
    if (l == 0) {
      const int e = scale_exp(m);
      se[r] = e;
      exps[r0 + r] = e;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 32 * (kP / 8); t += 256) {
    const int r = t % 32, kcg = t / 32;
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = sh[r][kcg * 8 + q];
    store_digits8<8>(x, se[r], digit_a<8>(S, r0 + r, kcg), kSliceA);
  }
}

// The panel's row exchanges on a tile of 32 columns of A, and the digits of the exchanged
// rows K (T, for the tiles of K the block A_KK).  perm[0] = number of rows that change, then pairs
// (destination, source); the K rows of T are read after the exchange.
__global__ void __launch_bounds__(256) swap_slice_kernel(int nct, int k0, int kb,
                                                         double* __restrict__ A,
                                                         const int* __restrict__ perm,
                                                         char* __restrict__ S,
                                                         int* __restrict__ exps) {
  extern __shared__ double swap_smem[];  // [2 kP][33]
  double(*sh)[kColTile + 1] = reinterpret_cast<double(*)[kColTile + 1]>(swap_smem);
  __shared__ int sd[2 * kP];
  __shared__ double smax[8][kColTile];
  __shared__ int se[kColTile];
  const int ct = blockIdx.x, c0 = ct * kColTile;
  const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int cnt = perm[0];
  for (int t = w; t < cnt; t += 8) {
    if (lane == 0) sd[t] = perm[1 + 2 * t];
    sh[t][lane] = A[tile_at(nct, perm[2 + 2 * t], c0 + lane)];
  }
  __syncthreads();
  for (int t = w; t < cnt; t += 8) A[tile_at(nct, sd[t], c0 + lane)] = sh[t][lane];
  __syncthreads();  // the rows K below are read back by the block that wrote them
  for (int t = threadIdx.x; t < kP * (kColTile / 2); t += 256) {
    const int q = t % kP, c = t / kP * 2;
    double2 x = make_double2(0.0, 0.0);
    if (q < kb) x = *reinterpret_cast<const double2*>(A + tile_at(nct, k0 + q, c0 + c));
    sh[q][c] = x.x;
    sh[q][c + 1] = x.y;
  }
  __syncthreads();
  double m = 0.0;
  bool bad = false;
  for (int q = w; q < kP; q += 8) {
    const double a = fabs(sh[q][lane]);
    bad |= !isfinite(a);
    m = fmax(m, a);
  }
  smax[w][lane] = bad ? __longlong_as_double(0x7ff0000000000000LL) : m;
  __syncthreads();
  if (w == 0) {
    for (int u = 1; u < 8; ++u) m = fmax(m, smax[u][lane]);
    m = fmax(m, smax[0][lane]);
    const int e = scale_exp(m);
    se[lane] = e;
    exps[c0 + lane] = e;
  }
  __syncthreads();
  char* tile = S + (size_t)ct * kTileB;
  for (int t = threadIdx.x; t < kColTile * (kP / 8); t += 256) {
    const int c = t % kColTile, kcg = t / kColTile;
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = sh[kcg * 8 + q][c];
    store_digits8<8>(x, se[c], digit_b<8>(tile, c, kcg), Geo<8>::kDigitB);
  }
}

// ------------------------------------------------------------------ LU of the panel copy
// X[i][c] = A[k0 + i][k0 + c] for the rows below k0, columns past kb zero
__global__ void panel_copy_kernel(int m, int k0, int kb, int nct, const double* __restrict__ A,
                                  double* __restrict__ X) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < (size_t)m * (kP / 2);
       t += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % m), c = (int)(t / m) * 2;
    double2 x = *reinterpret_cast<const double2*>(A + tile_at(nct, k0 + i, k0 + c));
    if (c >= kb) x.x = 0.0;
    if (c + 1 >= kb) x.y = 0.0;
    *reinterpret_cast<double2*>(X + (size_t)i * kP + c) = x;
  }
}

// LU with partial pivoting (the first of equal largest entries wins) of the columns
// [c0, c0 + w) of the panel copy X (m rows of kP), rows c0..m-1, by one cluster: thread t of
// CTA c holds the rows c * rpc + t + r * blockDim, r < R, in registers, the columns still to
// be factored first: after every step they move one place left and the step's multiplier
// takes the last place, so that the loop over the columns stays a loop (unrolled, its
// once-run code missed the instruction cache: 5.4 us a column at 4,231 rows) and nothing is
// stored before it ends (the barrier's release would wait for the stores: 3.5 us).  A column costs one cluster barrier: the warp that holds a CTA's
// best pivot candidate sends that row to every CTA (and the owner of row k the row to be
// exchanged), so after the barrier every CTA has the pivot row; the slots alternate by the
// parity of the column.  Bound by that chain of latencies and by the FP64 rate of the
// cluster's SMs.  CTA 0 then
// exchanges the rows of the panel's other columns and solves for the U rows of the columns
// to the right.  piv[c0 + q] = row exchanged with row c0 + q.
constexpr int kLuThreads = 512;
constexpr int kMaxCluster = 16;

__device__ __forceinline__ unsigned long long magnitude(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
  return b > 0x7ff0000000000000ULL ? 0 : b;  // NaN is no candidate
}
// over the warp: the largest value, the smallest index among equal ones
__device__ __forceinline__ void warp_best(unsigned long long& v, int& i) {
  const unsigned hi = (unsigned)(v >> 32), lo = (unsigned)v;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  i = (int)__reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? (unsigned)i : 0x7fffffffu);
  v = ((unsigned long long)mh << 32) | ml;
}

template <int W, int R>
__global__ void __launch_bounds__(kLuThreads) lu_panel_kernel(int m, int c0, int w, int kb, int rpc,
                                                              double* __restrict__ X,
                                                              int* __restrict__ piv, int k0,
                                                              DevFlags* flags) {
  __shared__ __align__(16) double cand[2][kMaxCluster][W + 2];  // every CTA's best row, 1 / pivot
  __shared__ __align__(16) double rowk[2][W + 2];               // row k before the exchange
  __shared__ __align__(16) double out[kLuThreads / kWarp][2][W + 2];  // a warp's rows to send
  __shared__ unsigned long long cmag[2][kMaxCluster], wmag[2][kLuThreads / kWarp];
  __shared__ int cidx[2][kMaxCluster], widx[2][kLuThreads / kWarp], spiv[W], slot[W];
  __shared__ double xs[2 * W * kP];  // CTA 0: the rows that the exchanges move
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nct = (int)cluster.num_blocks();
  const int tid = threadIdx.x, lane = tid % kWarp, wid = tid / kWarp;
  const int nw = (int)blockDim.x / kWarp;
  const int base = c0 + rank * rpc;
  int row[R];  // m: none
  double a[R][W];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int q = tid + r * (int)blockDim.x;
    row[r] = q < rpc && base + q < m ? base + q : m;
#pragma unroll
    for (int c = 0; c < W; ++c)
      a[r][c] = row[r] < m && c < w ? X[(size_t)row[r] * kP + c0 + c] : 0.0;
  }
  cluster.sync();  // every CTA's shared memory is live before it is written remotely
  // the row held by the thread with `own` (at most one of the block, any of its R rows) to
  // the same place in every CTA: staged by the thread, sent by its warp, 16 bytes a lane
  auto send = [&](bool own, int r, int which, double* dst) {
    const unsigned has = __ballot_sync(0xffffffffu, own);
    if (!has) return;
    if (own) {
#pragma unroll
      for (int rr = 0; rr < R; ++rr)
        if (rr == r) {
          // the reciprocal is taken here, by one warp: by every warp after the barrier its
          // dozen FP64 instructions would fill the pipe
          if (which == 0) out[wid][0][W] = 1.0 / a[rr][0];
#pragma unroll
          for (int c = 0; c < W; ++c) out[wid][which][c] = a[rr][c];
        }
    }
    __syncwarp();
    constexpr int kPairs = W / 2 + 1;
    for (int t = lane; t < nct * kPairs; t += kWarp) {
      const int d = t / kPairs, c = t % kPairs;
      reinterpret_cast<double2*>(cluster.map_shared_rank(dst, d))[c] =
          reinterpret_cast<const double2*>(out[wid][which])[c];
    }
  };
#pragma unroll 1
  for (int k = 0; k < w; ++k) {
    const int par = k & 1, kr = c0 + k;  // row of the diagonal
    // best candidate among the rows >= kr (magnitudes compared as integers, 0: none)
    unsigned long long best = 0;
    int bi = m;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const unsigned long long v = row[r] >= kr && row[r] < m ? magnitude(a[r][0]) : 0;
      if (v > best) {
        best = v;
        bi = row[r];
      }
    }
    warp_best(best, bi);
    if (lane == 0) {
      wmag[par][wid] = best;
      widx[par][wid] = bi;
    }
    __syncthreads();
    best = lane < nw ? wmag[par][lane] : 0;
    bi = lane < nw ? widx[par][lane] : m;
    warp_best(best, bi);
    bool mine = false, diag = false;
    int rm = 0, rd = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (best && row[r] == bi) {
        mine = true;
        rm = r;
      }
      if (row[r] == kr) {
        diag = true;
        rd = r;
      }
    }
    send(mine, rm, 0, cand[par][rank]);
    send(diag, rd, 1, rowk[par]);
    if (wid == 0 && lane < nct) {
      cluster.map_shared_rank(&cmag[par][rank], lane)[0] = best;
      cluster.map_shared_rank(&cidx[par][rank], lane)[0] = bi;
    }
    cluster.sync();
    unsigned long long pb = lane < nct ? cmag[par][lane] : 0;
    int pi = lane < nct ? cidx[par][lane] : m;
    const unsigned long long pmine = pb;
    const int imine = pi;
    warp_best(pb, pi);
    const int pr = __ffs(__ballot_sync(0xffffffffu, pmine == pb && imine == pi)) - 1;
    const bool ok = pb != 0;  // no usable pivot: the column is left out, the flag raised
    if (!ok) pi = kr;
    const double* up = ok ? cand[par][pr] : rowk[par];
    double u[W];
#pragma unroll
    for (int c = 0; c < W; c += 2) {
      const double2 v = *reinterpret_cast<const double2*>(up + c);
      u[c] = v.x;
      u[c + 1] = v.y;
    }
    if (tid == 0) {
      spiv[k] = pi;
      if (rank == 0) {
        piv[c0 + k] = pi;
        if (!ok) raise_flag(flags, MSP_ERR_SINGULAR_BLOCK, k0 + kr);
      }
    }
    const double inv = ok ? up[W] : 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (row[r] == pi && pi != kr) {  // the row exchanged away from the diagonal
#pragma unroll
        for (int c = 0; c < W; ++c) a[r][c] = rowk[par][c];
      }
      if (row[r] == kr) {
#pragma unroll
        for (int c = 0; c < W; ++c) a[r][c] = u[c];
      } else if (row[r] > kr && row[r] < m) {
        const double l = a[r][0] * inv;
#pragma unroll
        for (int g = 0; g < W; g += 4) {
          if (g + k < W) {  // some of these places still hold columns to be factored
#pragma unroll
            for (int c = g; c < g + 4 && c < W; ++c)
              if (c > 0) a[r][c - 1] = c + k < W ? fma(-l, u[c], a[r][c]) : a[r][c];
          } else {
#pragma unroll
            for (int c = g; c < g + 4 && c < W; ++c)
              if (c > 0) a[r][c - 1] = a[r][c];
          }
        }
        a[r][W - 1] = l;
      }
    }
  }
  // place c of a row holds column (c + steps) % W; a row of U stopped at its own step
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (row[r] < m) {
      const int steps = min(row[r] - c0, w);
      double* x = X + (size_t)row[r] * kP + c0;
#pragma unroll
      for (int c = 0; c < W; ++c) {
        const int col = (c + steps) % W;
        if (col < w) x[col] = a[r][c];
      }
    }
  cluster.sync();  // remote writes and reads are done; the factored columns are stored
  if (rank != 0) return;
  // the other columns: rows c0 + q <-> spiv[q], slots 0..w-1 the rows c0.., slot w + q the
  // pivot row of step q unless it is one of those or an earlier step's
  if (tid < w) {
    const int p = spiv[tid];
    int s = W + tid;
    if (p < c0 + w) {
      s = p - c0;
    } else {
      for (int q = tid - 1; q >= 0; --q)
        if (spiv[q] == p) s = W + q;
    }
    slot[tid] = s;
  }
  __syncthreads();
  for (int t = tid; t < 2 * W * kP; t += blockDim.x) {
    const int s = t / kP, c = t % kP;
    const int q = s % W;
    if (q >= w || (s >= W && slot[q] != s)) continue;
    xs[t] = X[(size_t)(s < W ? c0 + q : spiv[q]) * kP + c];
  }
  __syncthreads();
  if (tid < kP && (tid < c0 || tid >= c0 + w)) {
    for (int q = 0; q < w; ++q) {
      const int s = slot[q];
      if (s != q) {
        const double t = xs[q * kP + tid];
        xs[q * kP + tid] = xs[s * kP + tid];
        xs[s * kP + tid] = t;
      }
    }
  }
  __syncthreads();
  {
    if (tid >= c0 + w && tid < kb) {
      double y[W];
#pragma unroll
      for (int q = 0; q < W; ++q) y[q] = q < w ? xs[q * kP + tid] : 0.0;
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k < w) {
#pragma unroll
          for (int q = k + 1; q < W; ++q)
            if (q < w) y[q] = fma(-xs[q * kP + c0 + k], y[k], y[q]);
        }
#pragma unroll
      for (int q = 0; q < W; ++q)
        if (q < w) xs[q * kP + tid] = y[q];
    }
  }
  __syncthreads();
  for (int t = tid; t < 2 * W * kP; t += blockDim.x) {
    const int s = t / kP, c = t % kP;
    const int q = s % W;
    if (q >= w || (s >= W && slot[q] != s)) continue;
    X[(size_t)(s < W ? c0 + q : spiv[q]) * kP + c] = xs[t];
  }
}

// X[i][j] -= sum_q X[i][c0 + q] X[c0 + q][j] for the rows below c0 + w and the columns right
// of it: 16 rows per block (64 left most SMs without a block on the usual 2,000 to 10,000
// rows: 27 us a launch at 4,231), the multipliers and the U rows staged in shared memory
constexpr int kUpdRows = 16;
template <int W>
__global__ void __launch_bounds__(256) lu_update_kernel(int m, int c0, int w, int kb,
                                                        double* __restrict__ X) {
  __shared__ double sl[kUpdRows][W + 1];
  __shared__ double su[W][kP];
  const int j0 = c0 + w, nj = kb - j0, r0 = c0 + w + blockIdx.x * kUpdRows;
  for (int t = threadIdx.x; t < kUpdRows * W; t += 256) {
    const int r = t / W, q = t % W;
    sl[r][q] = (r0 + r < m && q < w) ? X[(size_t)(r0 + r) * kP + c0 + q] : 0.0;
  }
  for (int t = threadIdx.x; t < W * kP; t += 256) {
    const int q = t / kP, j = t % kP;
    su[q][j] = (q < w && j < nj) ? X[(size_t)(c0 + q) * kP + j0 + j] : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x % 16, i = r0 + threadIdx.x / 16;
  if (i >= m) return;
  const double* l = sl[threadIdx.x / 16];
  for (int j = tx; j < nj; j += 16) {
    double a = X[(size_t)i * kP + j0 + j];
#pragma unroll
    for (int q = 0; q < W; ++q) a = fma(-l[q], su[q][j], a);
    X[(size_t)i * kP + j0 + j] = a;
  }
}

// D = A_KK^-1 (rows K exchanged) from the factors in X: one warp per column solves
// L y = e_j, U x = y by columns (lane l owns the rows l, l + 32, l + 64; a step is a
// broadcast and up to three FMAs).  D is stored (kP x kP, zero past kb) and so are its
// digits (as a T operand) with their exponents.  The last block composes the exchanges
// into the list of rows that change (perm) for all columns of A.
constexpr int kDiagWarps = 4;
__global__ void __launch_bounds__(kDiagWarps * kWarp) diag_inverse_panel_kernel(
    int k0, int kb, const double* __restrict__ X, const int* __restrict__ piv,
    double* __restrict__ D, char* __restrict__ S, int* __restrict__ exps,
    int* __restrict__ perm, int* __restrict__ piv_out) {
  extern __shared__ double sf[];  // kP x (kP + 1) factors, then kP reciprocal pivots
  if (blockIdx.x == gridDim.x - 1) {
    // exchanges in order on a small list: slot q < kb is row k0 + q, slot kb + q the pivot
    // row of step q when it lies below the block (the first step that names it)
    __shared__ int row[2 * kP], cur[2 * kP], sl[kP], sp[kP];
    for (int q = threadIdx.x; q < kb; q += blockDim.x) sp[q] = piv[q];
    __syncthreads();
    for (int q = threadIdx.x; q < kb; q += blockDim.x) {
      const int p = sp[q];
      int s = kb + q;
      if (p < kb) {
        s = p;
      } else {
        for (int r = q - 1; r >= 0; --r)
          if (sp[r] == p) s = kb + r;
      }
      sl[q] = s;
      row[q] = k0 + q;
      row[kb + q] = s == kb + q ? k0 + p : -1;
      piv_out[k0 + q] = k0 + p;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * kb; t += blockDim.x) cur[t] = t;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int q = 0; q < kb; ++q) {
        const int s = sl[q], a = cur[q];
        cur[q] = cur[s];
        cur[s] = a;
      }
    __syncthreads();
    if (threadIdx.x < kWarp) {  // compacted by one warp
      int cnt = 0;
      for (int t0 = 0; t0 < 2 * kb; t0 += kWarp) {
        const int t = t0 + threadIdx.x;
        const bool ch = t < 2 * kb && row[t] >= 0 && cur[t] != t;
        const unsigned b = __ballot_sync(0xffffffffu, ch);
        const int at = cnt + __popc(b & ((1u << threadIdx.x) - 1u));
        if (ch) {
          perm[1 + 2 * at] = row[t];
          perm[2 + 2 * at] = row[cur[t]];
        }
        cnt += __popc(b);
      }
      if (threadIdx.x == 0) perm[0] = cnt;
    }
    return;
  }
  constexpr int ld = kP + 1;
  double* rd = sf + kP * ld;
#pragma unroll 8
  for (int t = threadIdx.x; t < kP * kP; t += kDiagWarps * kWarp) {
    const int r = t / kP, c = t % kP;
    sf[r * ld + c] = (r < kb && c < kb) ? X[(size_t)r * kP + c] : 0.0;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kP; q += blockDim.x) {
    const double d = sf[q * ld + q];
    rd[q] = d != 0.0 ? 1.0 / d : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x % kWarp;
  const int j = blockIdx.x * kDiagWarps + threadIdx.x / kWarp;
  double y[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) y[a] = (lane + 32 * a == j && j < kb) ? 1.0 : 0.0;
#pragma unroll 4
  for (int k = j & ~3; k < kb; ++k) {  // rows above j stay zero
    const double mine = k < 32 ? y[0] : (k < 64 ? y[1] : y[2]);
    const double yk = __shfl_sync(0xffffffffu, mine, k & 31);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (lane + 32 * a > k) y[a] = fma(-sf[(lane + 32 * a) * ld + k], yk, y[a]);
  }
#pragma unroll 4
  for (int k = kb - 1; k >= 0; --k) {
    const double mine = (k < 32 ? y[0] : (k < 64 ? y[1] : y[2])) * rd[k];
    const double xk = __shfl_sync(0xffffffffu, mine, k & 31);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (lane + 32 * a < k)
        y[a] = fma(-sf[(lane + 32 * a) * ld + k], xk, y[a]);
      else if (lane + 32 * a == k)
        y[a] = xk;
    }
  }
  double m = 0.0;
  bool bad = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (lane + 32 * a >= kb || j >= kb) y[a] = 0.0;
    bad |= !isfinite(y[a]);
    m = fmax(m, fabs(y[a]));
    D[(size_t)(lane + 32 * a) * kP + j] = y[a];
  }
  if (bad) m = __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = scale_exp(m);
  if (lane == 0) exps[j] = e;
  char* tile = S + (size_t)(j / kColTile) * kTileB;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int q = lane + 32 * a;
    long long v = scaled_int(y[a], e);
    char* dst = digit_b<8>(tile, j % kColTile, q / 8) + (q % 8) * 2;
    for (int s = 7; s >= 0; --s) {
      int d = (int)v;
      if (s > 0) {
        d = (int)(((unsigned)v + 128u) & 255u) - 128;
        v = (v - d) >> 8;
      }
      *reinterpret_cast<unsigned short*>(dst + (size_t)s * Geo<8>::kDigitB) =
          (unsigned short)bf16_of_int(d);
    }
  }
}

// ------------------------------------------------------------------ the products
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Wait for the phase of the given parity for at most limit_ns (and 2^20 attempts); false (and
// the block's stop word set) when the limit runs out or another warp has stopped.  The first
// look does not suspend the thread, so that a limit of 0 gives up wherever there is a wait.
constexpr unsigned long long kWaitNs = InverseOptions::kWaitNs;
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* stop,
                                          unsigned long long limit_ns) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  if (done) return true;
  const unsigned long long t0 = now_ns();
  for (int it = 0; it < (1 << 20) && limit_ns > 0; ++it) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*stop) return false;
    if (now_ns() - t0 > limit_ns) break;
  }
  *stop = 1;
  return false;
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes,
                                          unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(bar)
      : "memory");
}
// shared-memory matrix descriptor: K-major, no swizzle, core matrices of 8 rows x 16 bytes;
// lbo: bytes between core matrices along K, sbo: along the rows
__device__ __forceinline__ unsigned long long mat_desc(unsigned addr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((addr & 0x3ffffu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(sbo >> 4) << 32) | (1ULL << 46);
}
// D (f32, TMEM) (+)= A (bf16) B (bf16)^T, M = 128, N = n, K = 16
__device__ __forceinline__ void mma_bf16(unsigned d, unsigned long long a, unsigned long long b,
                                         unsigned n, bool accumulate) {
  const unsigned idesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((unsigned)(kRowTile >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void tmem_ld8(unsigned addr, unsigned (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(addr));
}

// c + 2^(e + 16) sum_m S_m 2^(8 (5 - m)), m = 0..5, |S_m| <= (m + 1) 2^21: an integer below 2^62,
// taken without its last 12 bits (2^-49 of the largest product, as the digits left out) so that it
// becomes a double by one subtraction: two FP64 operations an element
__device__ __forceinline__ double add_digits(const float (&S)[6], int e, double, double c) {
  static_assert(CorrGeo::kK << 14 <= 1 << 21, "bound of the sums");
  const int s0 = __float2int_rn(S[0]), s1 = __float2int_rn(S[1]), s2 = __float2int_rn(S[2]);
  const int s3 = __float2int_rn(S[3]), s4 = __float2int_rn(S[4]), s5 = __float2int_rn(S[5]);
  const long long v = (long long)(s0 * 256 + s1) * 1048576 + (long long)(s2 * 256 + s3) * 16 +
                      ((s4 + (s5 >> 8) + 8) >> 4);
  const double d = __longlong_as_double(0x4338000000000000LL + v) - 6755399441055744.0;
  const int be = min(max(e + 1051, 0), 0x7ff);
  return fma(d, __longlong_as_double((long long)be << 52), c);
}
// c + sign 2^e sum_m S_m 2^(8 (7 - m)), m = 0..7, S_m exact integers below 2^24
__device__ __forceinline__ double add_digits(const float (&S)[8], int e, double sign, double c) {
  // two exact 64-bit integers, |lo| < 2^49 and |hi| < 2^49; the sum is hi 2^32 + lo
  const int s2 = __float2int_rn(S[0]), s3 = __float2int_rn(S[1]), s4 = __float2int_rn(S[2]);
  const int s5 = __float2int_rn(S[3]), s6 = __float2int_rn(S[4]), s7 = __float2int_rn(S[5]);
  const int s8 = __float2int_rn(S[6]), s9 = __float2int_rn(S[7]);
  const long long hi =
      (long long)s2 * 16777216 + ((long long)s3 * 65536 + ((long long)s4 * 256 + s5));
  const long long lo =
      (long long)s6 * 16777216 + ((long long)s7 * 65536 + ((long long)s8 * 256 + s9));
  // An integer below 2^51 added to the bits of M = 1.5 * 2^52 is the double M + integer.
  // The low word is used as it is, M too large, and M = 1.5 * 2^20 * 2^32 is taken from the
  // high word instead: three FP64 operations an element (the FP64 pipe bounds the epilogue).
  const double dh =
      __longlong_as_double(0x4338000000000000LL + (hi - 1572864)) - 6755399441055744.0;
  const double dl = __longlong_as_double(0x4338000000000000LL + lo);
  const int be = min(max(e + 1023, 0), 0x7ff), bh = min(max(e + 1055, 0), 0x7ff);
  const long long sg = __double_as_longlong(sign) & (1LL << 63);
  const double fl = __longlong_as_double(((long long)be << 52) | sg);
  const double fh = __longlong_as_double(((long long)bh << 52) | sg);
  return fma(dl, fl, fma(dh, fh, c));
}

// One product of a step on the tiles (128 x 32) of C (row tiles of ctiles column tiles; the
// product's first column tile is coff), V = SA SB:
//   kUpdate: C = A, the nct column tiles from cbegin, without the kskip tiles from kt0 on (the
//            columns K and those done by another launch): C += V, or C = V for the rows K;
//   kFirst:  C = the columns K: C = -V, or D for the rows K;
//   kResid:  C += V;  kCorrect: C -= V (both on 96 columns; with ND = 6, kResid on all of them).
enum Product { kUpdate, kFirst, kResid, kCorrect };
// Persistent blocks, each a contiguous run of tiles in row-major tile order; the digits of a
// row tile (192 KB) stay in shared memory while the column tiles' digits (48 KB) stream
// through four buffers of 16 columns of K, so L2 is read once per tile.  One warp copies, one thread of
// another issues the MMAs (48 per tile, into one of two TMEM buffers of 256 columns), sixteen
// warps turn the previous tile's accumulators into FP64 and update A.
constexpr int kEpiWarps = 16;
constexpr int kGemmThreads = (kEpiWarps + 2) * kWarp;
constexpr int kEpiCols = kColTile / (kEpiWarps / 4);  // columns of a tile per epilogue warp
constexpr size_t kGemmSmem = kTileA + kStages * Geo<8>::kChunkB + 512;
template <Product kMode, int ND = 8>
__global__ void __launch_bounds__(kGemmThreads, 1) slice_gemm_kernel(
    int ctiles, int coff, int k0, int kb, int nrt, int nct, int cbegin, int kt0, int kskip,
    double* __restrict__ C,
    const char* __restrict__ SA, const int* __restrict__ ea, const char* __restrict__ SB,
    const int* __restrict__ eb, const double* __restrict__ D, DevFlags* flags,
    unsigned long long wait_ns) {
  constexpr int kChunks = Geo<ND>::kChunks, kChunkA = Geo<ND>::kChunkA, kChunkB = Geo<ND>::kChunkB;
  extern __shared__ __align__(128) char sm[];
  __shared__ __align__(8) unsigned long long bars[1 + 2 * kStages + 5];
  __shared__ unsigned s_tmem;
  __shared__ volatile int s_stop;
  const int wid = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  const unsigned sbase = (smem_u32(sm) + 127u) & ~127u;
  const unsigned sA = sbase, sB = sbase + kTileA;
  const unsigned b_a = smem_u32(&bars[0]);
  const unsigned b_full = smem_u32(&bars[1]), b_empty = smem_u32(&bars[1 + kStages]);
  const unsigned b_tfull = smem_u32(&bars[1 + 2 * kStages]), b_tempty = b_tfull + 16;
  const unsigned b_end = b_tempty + 16;  // every MMA issued
  const long long total = (long long)nrt * nct;
  const long long t0 = total * blockIdx.x / gridDim.x, t1 = total * (blockIdx.x + 1) / gridDim.x;
  if (threadIdx.x == 0) {
    s_stop = 0;
    mbar_init(b_a, 1);
    mbar_init(b_end, 1);
    for (int c = 0; c < kStages; ++c) {
      mbar_init(b_full + 8 * c, 1);
      mbar_init(b_empty + 8 * c, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(b_tfull + 8 * b, 1);
      mbar_init(b_tempty + 8 * b, kEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wid == kEpiWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(&s_tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = s_tmem;

  if (wid == kEpiWarps) {
    if (lane == 0) {
      int prev = -1;
      unsigned g = 0;  // chunks so far: buffer g % kStages, its use g / kStages
      unsigned na = 0;  // row tiles so far
      bool run = true;
      for (long long t = t0; t < t1 && run; ++t) {
        const int rt = (int)(t / nct), q = (int)(t % nct);
        const int ct = kMode != kUpdate ? q : cbegin + q + (q >= kt0 ? kskip : 0);
        if (rt != prev) {
          // the previous row tile's digits are free once its last chunk has been used
          if (g > 0)
            run = mbar_wait(b_empty + 8 * ((g - 1) % kStages), ((g - 1) / kStages) & 1, &s_stop, wait_ns);
          if (!run) break;
          ++na;
          mbar_expect(b_a, kTileA);
          for (int c = 0; c < kChunks; ++c)
            bulk_load(sA + c * kChunkA, SA + (size_t)rt * kTileA + (size_t)c * kChunkA, kChunkA, b_a);
          prev = rt;
        }
        for (int c = 0; c < kChunks && run; ++c, ++g) {
          const unsigned st = g % kStages;
          if (g >= kStages) run = mbar_wait(b_empty + 8 * st, ((g / kStages) - 1) & 1, &s_stop, wait_ns);
          if (!run) break;
          mbar_expect(b_full + 8 * st, kChunkB);
          bulk_load(sB + st * kChunkB, SB + (size_t)ct * kTileB + (size_t)c * kChunkB, kChunkB,
                    b_full + 8 * st);
        }
      }
      // the copies in flight land before the block (and its shared memory) goes away, whoever
      // stopped: the last phase of each barrier that has a copy
      volatile int never = 0;
      if (na > 0) mbar_wait(b_a, (na - 1) & 1, &never, kWaitNs);
      for (unsigned q = g > kStages ? g - kStages : 0; q < g; ++q)
        mbar_wait(b_full + 8 * (q % kStages), (q / kStages) & 1, &never, kWaitNs);
    }
  } else if (wid == kEpiWarps + 1) {
    if (lane == 0) {
      int prev = -1;
      unsigned it = 0, na = 0, g = 0;
      bool run = true;
      for (long long t = t0; t < t1 && run; ++t, ++it) {
        const int rt = (int)(t / nct);
        if (rt != prev) {
          run = mbar_wait(b_a, na & 1, &s_stop, wait_ns);
          ++na;
          prev = rt;
        }
        const unsigned buf = it & 1;
        if (run && it >= 2) run = mbar_wait(b_tempty + 8 * buf, ((it >> 1) - 1) & 1, &s_stop, wait_ns);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        for (int c = 0; c < kChunks && run; ++c, ++g) {
          const unsigned st = g % kStages;
          run = mbar_wait(b_full + 8 * st, (g / kStages) & 1, &s_stop, wait_ns);
          if (!run) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const unsigned long long db = mat_desc(sB + st * kChunkB, (Geo<ND>::kRowsB / 8) * 128, 128);
          // digit i of P with the digits 0..ND-1-i of T; digit 0 of the first chunk starts the
          // ND sums
#pragma unroll
          for (int i = 0; i < ND; ++i)
            mma_bf16(tmem + buf * 256 + i * kColTile,
                     mat_desc(sA + c * kChunkA + i * kSliceA, (kRowTile / 8) * 128, 128), db,
                     kColTile * (ND - i), c > 0 || i > 0);
          mma_commit(b_empty + 8 * st);
        }
        if (run) mma_commit(b_tfull + 8 * buf);
      }
      // every MMA issued here ends before the accumulators and the buffers go away, also where
      // an epilogue warp has stopped
      volatile int never = 0;
      mma_commit(b_end);
      mbar_wait(b_end, 0, &never, kWaitNs);
    }
  } else {
    const int quad = wid & 3, part = wid >> 2;  // a warp reads the TMEM lanes of its quadrant
    constexpr double sign = kMode == kFirst || kMode == kCorrect ? -1.0 : 1.0;
    // this thread's first pair of columns in a tile of C
    auto c_pairs = [&](int rt, int ct) {
      return C + ((size_t)rt * ctiles + coff + ct) * (kRowTile * kColTile) +
             (size_t)(part * kEpiCols / 2) * (2 * kRowTile) + (quad * 32 + lane) * 2;
    };
    // what a tile's C starts from: the rows' and columns' values, loaded one tile ahead
    auto load_c = [&](long long t, double (&cv)[kEpiCols]) {
      const int rt = (int)(t / nct), q = (int)(t % nct);
      const int ct = kMode != kUpdate ? q : cbegin + q + (q >= kt0 ? kskip : 0);
      const int i = rt * kRowTile + quad * 32 + lane;
      const bool in_k = i >= k0 && i < k0 + kb;
      const int cb = ct * kColTile + part * kEpiCols;
      const double* src = kMode == kFirst ? D + (size_t)(i - k0) * kP + cb : c_pairs(rt, ct);
      constexpr int pitch = kMode == kFirst ? 2 : 2 * kRowTile;  // between pairs of columns
      const bool use = kMode == kFirst ? in_k : kMode != kUpdate || !in_k;
#pragma unroll
      for (int p = 0; p < kEpiCols / 2; ++p) {
        const double2 v = use ? *reinterpret_cast<const double2*>(src + p * pitch)
                              : make_double2(0.0, 0.0);
        cv[2 * p] = v.x;
        cv[2 * p + 1] = v.y;
      }
    };
    unsigned it = 0;
    double cn[kEpiCols];
    if (t0 < t1) load_c(t0, cn);
    for (long long t = t0; t < t1; ++t, ++it) {
      const int rt = (int)(t / nct), q = (int)(t % nct);
      const int ct = kMode != kUpdate ? q : cbegin + q + (q >= kt0 ? kskip : 0);
      const int i = rt * kRowTile + quad * 32 + lane;
      const bool in_k = i >= k0 && i < k0 + kb;
      const int cb = ct * kColTile + part * kEpiCols;
      double* cpair = c_pairs(rt, ct);
      double cv[kEpiCols];
#pragma unroll
      for (int p = 0; p < kEpiCols; ++p) cv[p] = cn[p];
      int ev[kEpiCols];  // exponents of row + column
      const int eai = __ldg(ea + i) - 70;
#pragma unroll
      for (int c = 0; c < kEpiCols; c += 4) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(eb + cb + c));
        ev[c] = v.x + eai;
        ev[c + 1] = v.y + eai;
        ev[c + 2] = v.z + eai;
        ev[c + 3] = v.w + eai;
      }
      if (t + 1 < t1) load_c(t + 1, cn);
      const unsigned buf = it & 1;
      const bool run = mbar_wait(b_tfull + 8 * buf, (it >> 1) & 1, &s_stop, wait_ns);
      if (!__all_sync(0xffffffffu, run)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      static_assert(kEpiCols == 8, "one load of eight columns per group");
      unsigned r[ND][8];
#pragma unroll
      for (int m = 0; m < ND; ++m)
        tmem_ld8(tmem + ((unsigned)(quad * 32) << 16) + buf * 256 + m * kColTile + part * kEpiCols,
                 r[m]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (lane == 0) mbar_arrive(b_tempty + 8 * buf);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        float S[ND];
#pragma unroll
        for (int m = 0; m < ND; ++m) S[m] = __uint_as_float(r[m][c]);
        const double v = add_digits(S, ev[c], sign, cv[c]);
        if (kMode != kFirst || !in_k) cv[c] = v;
      }
#pragma unroll
      for (int p = 0; p < kEpiCols / 2; ++p)
        *reinterpret_cast<double2*>(cpair + p * 2 * kRowTile) = make_double2(cv[2 * p], cv[2 * p + 1]);
    }
  }
  __syncthreads();
  if (s_stop && threadIdx.x == 0) raise_flag(flags, MSP_ERR_TIMEOUT, blockIdx.x);  // a wait ran out
  __syncwarp();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (wid == kEpiWarps + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// ------------------------------------------------------------------ scaling of the matrix
// Powers of two r_i, c_j, so that the entries 2^(r_i + c_j) a_ij are of one order of magnitude
// whatever units the rows and columns of A come in: the digits of an operand share an exponent
// per row or column, so the products are FP64 products only of rows and columns whose large
// entries meet.  Six rounds of geometric means (of the entries' binary exponents, as integers:
// the same on every run), then the largest entry of a row to [0.5, 1).
constexpr int kScaleRounds = 6;
__device__ __forceinline__ bool entry_exp(double x, int& e) {
  if (x == 0.0 || !isfinite(x)) return false;
  frexp(x, &e);
  return true;
}
// largest: r_i from the largest entry, else from the mean; csum[j], ccnt[j] += exponents, count
__global__ void row_scale_kernel(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                 const double* __restrict__ v, const int* __restrict__ c, bool largest,
                                 int* __restrict__ r, int* __restrict__ csum, int* __restrict__ ccnt) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int sum = 0, cnt = 0, top = -(1 << 30), e;
    for (int p = rp[i]; p < rp[i + 1]; ++p)
      if (entry_exp(v[p], e)) {
        e += c[ci[p]];
        sum += e;
        ++cnt;
        top = max(top, e);
      }
    const int ri = cnt == 0 ? 0 : (largest ? -top : -(int)rint((double)sum / cnt));
    r[i] = ri;
    if (largest) continue;
    for (int p = rp[i]; p < rp[i + 1]; ++p)
      if (entry_exp(v[p], e)) {
        atomicAdd(csum + ci[p], e + ri);
        atomicAdd(ccnt + ci[p], 1);
      }
  }
}
__global__ void col_scale_kernel(int n, int* __restrict__ csum, int* __restrict__ ccnt, int* __restrict__ c) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    c[j] = ccnt[j] == 0 ? 0 : -(int)rint((double)csum[j] / ccnt[j]);
    csum[j] = ccnt[j] = 0;
  }
}

// v <- the scaled entries, and A (zeroed) their dense copy
__global__ void csr_to_dense_kernel(int n, int nct, const int* __restrict__ rp,
                                    const int* __restrict__ ci, const double* __restrict__ v,
                                    const int* __restrict__ r, const int* __restrict__ c,
                                    double* __restrict__ vs, double* __restrict__ A) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
      const double x = scalbn(v[p], r[i] + c[ci[p]]);
      vs[p] = x;
      A[tile_at(nct, i, ci[p])] = x;
    }
  }
}

// ------------------------------------------------------------------ the correction
// R = I - B X for the scaled matrix B (CSR) and its inverse X, whose column j stands at place
// cols[j] of A's tiles (place[cols[j]] = j): R row-major, its columns in the order of the
// places, and rmax[q] = the largest |R| of a column (as bits).  A block takes 32 rows and 32
// columns at a time: a lane per row, so that neighbouring rows' entries of X share lines, the
// piece written along its rows.  n^2 entries of X are read once per stored entry of a row of B
// (from L2 mostly).
__global__ void __launch_bounds__(256) inverse_residual_kernel(
    int n, int nct, const int* __restrict__ rp, const int* __restrict__ ci,
    const double* __restrict__ vs, const double* __restrict__ X, const int* __restrict__ place,
    double* __restrict__ R, unsigned long long* __restrict__ rmax) {
  __shared__ double sh[32][33];
  const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int i0 = blockIdx.x * 32, i = i0 + lane;
  const int p0 = i < n ? rp[i] : 0, p1 = i < n ? rp[i + 1] : 0;
  for (int ct = blockIdx.y; ct * kColTile < n; ct += gridDim.y) {
    const int q0 = ct * kColTile;
#pragma unroll
    for (int t = 0; t < 2; ++t) {  // pairs of columns
      const int c = (w + 8 * t) * 2;
      double2 a = make_double2(0.0, 0.0);
      for (int p = p0; p < p1; ++p) {
        const double b = -__ldg(vs + p);
        const double2 x = *reinterpret_cast<const double2*>(X + tile_at(nct, __ldg(ci + p), q0 + c));
        a.x = fma(b, x.x, a.x);
        a.y = fma(b, x.y, a.y);
      }
      const bool h0 = i < n && q0 + c < n, h1 = i < n && q0 + c + 1 < n;
      if (h0 && place[q0 + c] == i) a.x += 1.0;
      if (h1 && place[q0 + c + 1] == i) a.y += 1.0;
      sh[lane][c] = h0 ? a.x : 0.0;
      sh[lane][c + 1] = h1 ? a.y : 0.0;
    }
    __syncthreads();
    if (w == 0 && q0 + lane < n) {
      unsigned long long m = 0;
      for (int r = 0; r < 32; ++r) {
        const unsigned long long b =
            (unsigned long long)__double_as_longlong(sh[r][lane]) & 0x7fffffffffffffffULL;
        m = b > m ? b : m;  // a NaN is larger than any number
      }
      atomicMax(rmax + q0 + lane, m);
    }
    for (int r = w; r < 32; r += 8)
      if (i0 + r < n && q0 + lane < n) R[(size_t)(i0 + r) * n + q0 + lane] = sh[r][lane];
    __syncthreads();
  }
}

// Six digits of the columns k0..k0+127 of X (at the places cols[k0..]) for 16 rows a block
constexpr int kCorrK = CorrGeo::kK;
constexpr int kCorrRows = 16;
__global__ void __launch_bounds__(256) slice_inverse_kernel(int n, int nct, int k0,
                                                            const double* __restrict__ X,
                                                            const int* __restrict__ cols,
                                                            char* __restrict__ S, int* __restrict__ exps) {
  __shared__ double sh[kCorrRows][kCorrK + 1];
  __shared__ int se[kCorrRows];
  const int r0 = blockIdx.x * kCorrRows;
  for (int t = threadIdx.x; t < kCorrRows * kCorrK; t += 256) {
    const int r = t % kCorrRows, q = t / kCorrRows;
    sh[r][q] = k0 + q < n ? X[tile_at(nct, r0 + r, __ldg(cols + k0 + q))] : 0.0;
  }
  __syncthreads();
  {
    const int r = threadIdx.x / 16, l = threadIdx.x % 16;  // sixteen lanes per row
    double m = 0.0;
    bool bad = false;
    for (int q = l; q < kCorrK; q += 16) {
      const double a = fabs(sh[r][q]);
      bad |= !isfinite(a);
      m = fmax(m, a);
    }
    if (bad) m = __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o, 16));
    if (l == 0) {
      const int e = scale_exp(m);
      se[r] = e;
      exps[r0 + r] = e;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kCorrRows * (kCorrK / 8); t += 256) {
    const int r = t % kCorrRows, kcg = t / kCorrRows;
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = sh[r][kcg * 8 + q];
    store_digits8<kCorrDigits>(x, se[r], digit_a<kCorrDigits>(S, r0 + r, kcg), kSliceA);
  }
}

// Six digits of the rows k0..k0+127 of R, a tile of 32 columns a block.  A column whose
// residual is not small (an inverse without correct digits, or not finite) is left as it is.
constexpr double kCorrLimit = 0.0078125;
__global__ void __launch_bounds__(256) slice_residual_kernel(int n, int k0, const double* __restrict__ R,
                                                             const unsigned long long* __restrict__ rmax,
                                                             char* __restrict__ S, int* __restrict__ exps) {
  extern __shared__ double swap_smem[];  // [kCorrK][33]
  double(*sh)[kColTile + 1] = reinterpret_cast<double(*)[kColTile + 1]>(swap_smem);
  __shared__ double smax[8][kColTile];
  __shared__ int se[kColTile];
  const int ct = blockIdx.x, lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int c = ct * kColTile + lane;
  const bool use = c < n && __longlong_as_double((long long)rmax[c < n ? c : 0]) <= kCorrLimit;
  double m = 0.0;
  for (int q = w; q < kCorrK; q += 8) {
    const double x = use && k0 + q < n ? R[(size_t)(k0 + q) * n + c] : 0.0;
    sh[q][lane] = x;
    m = fmax(m, fabs(x));
  }
  smax[w][lane] = m;
  __syncthreads();
  if (w == 0) {
    for (int u = 1; u < 8; ++u) m = fmax(m, smax[u][lane]);
    const int e = scale_exp(m);
    se[lane] = e;
    exps[c] = e;
  }
  __syncthreads();
  char* tile = S + (size_t)ct * kTileB;
  for (int t = threadIdx.x; t < kColTile * (kCorrK / 8); t += 256) {
    const int cc = t % kColTile, kcg = t / kColTile;
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = sh[kcg * 8 + q][cc];
    store_digits8<kCorrDigits>(x, se[cc], digit_b<kCorrDigits>(tile, cc, kcg), CorrGeo::kDigitB);
  }
}

// out (n x n, row-major) = A with its columns in the order colperm, the scaling undone: 32 x 32
// pieces through shared memory, read along the rows of A's tiles and written along those of out
__global__ void __launch_bounds__(256) unscramble_kernel(int n, int nct,
                                                         const int* __restrict__ colperm,
                                                         const double* __restrict__ A,
                                                         const int* __restrict__ rs,
                                                         const int* __restrict__ cs,
                                                         double* __restrict__ out) {
  __shared__ double sh[32][33];
  const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int i0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
#pragma unroll
  for (int c = w; c < 32; c += 8)
    sh[lane][c] = (i0 + lane < n && c0 + c < n)
                      ? scalbn(A[tile_at(nct, i0 + lane, colperm[c0 + c])], cs[i0 + lane] + rs[c0 + c])
                      : 0.0;
  __syncthreads();
#pragma unroll
  for (int r = w; r < 32; r += 8)
    if (i0 + r < n && c0 + lane < n) out[(size_t)(i0 + r) * n + c0 + lane] = sh[r][lane];
}

// The sub-panels of one step: LU of the m x kb panel copy X.
template <int W, int R>
int lu_panel(int m, int kb, int k0, int cluster, double* X, int* piv, DevFlags* flags,
             cudaStream_t s) {
  MSP_CUDA_TRY(cudaFuncSetAttribute(lu_panel_kernel<W, R>,
                                    cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (int c0 = 0; c0 < kb; c0 += W) {
    const int w = std::min(W, kb - c0), rows = m - c0;
    // about 128 rows per CTA: more CTAs make the barrier dearer, fewer the rank-1 updates
    int nct = 1;
    while (nct < cluster && nct * 128 < rows) nct *= 2;
    const int rpc = std::max(W, (rows + nct - 1) / nct);  // CTA 0 holds the rows c0..c0+w-1
    const int threads = std::max(kP, (int)div_up(div_up(rpc, R), kWarp) * kWarp);
    if (threads > kLuThreads) return MSP_ERR_ARG;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nct);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = nct;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MSP_CUDA_TRY(
        cudaLaunchKernelEx(&cfg, lu_panel_kernel<W, R>, m, c0, w, kb, rpc, X, piv, k0, flags));
    MSP_TRY(launch_status());
    if (c0 + w < kb && m > c0 + w) {
      lu_update_kernel<W><<<div_up(m - c0 - w, kUpdRows), 256, 0, s>>>(m, c0, w, kb, X);
      MSP_TRY(launch_status());
    }
  }
  return MSP_OK;
}

// CTAs of the panels' cluster: 16 is past the portable size, so the device is asked whether it
// can place one (of 512 threads and all their registers: a whole SM each); 8 always fit
int panel_cluster(int* out) {
  MSP_CUDA_TRY(cudaFuncSetAttribute(lu_panel_kernel<16, 1>,
                                    cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kMaxCluster);
  cfg.blockDim = dim3(kLuThreads);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kMaxCluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int fit = 0;
  if (cudaOccupancyMaxActiveClusters(&fit, lu_panel_kernel<16, 1>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    fit = 0;
  }
  *out = fit > 0 ? kMaxCluster : 8;
  return MSP_OK;
}

// A stream of its own for the panels, joined before it goes
struct SideStream {
  cudaStream_t stream = nullptr;
  cudaEvent_t ready = nullptr, copied = nullptr, factored = nullptr;
  SideStream() = default;
  SideStream(const SideStream&) = delete;
  SideStream& operator=(const SideStream&) = delete;
  int create() {
    MSP_CUDA_TRY(cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking));
    MSP_CUDA_TRY(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
    MSP_CUDA_TRY(cudaEventCreateWithFlags(&copied, cudaEventDisableTiming));
    MSP_CUDA_TRY(cudaEventCreateWithFlags(&factored, cudaEventDisableTiming));
    return MSP_OK;
  }
  ~SideStream() {
    if (stream) {
      cudaStreamSynchronize(stream);
      cudaStreamDestroy(stream);
    }
    if (ready) cudaEventDestroy(ready);
    if (copied) cudaEventDestroy(copied);
    if (factored) cudaEventDestroy(factored);
  }
};

}  // namespace

long long inverse_scratch_bytes(long long n) {
  const long long lda = (n + kP - 1) / kP * kP, rows = (n + kRowTile - 1) / kRowTile * kRowTile;
  return 8 * (rows * lda + (n + rows) * kP) + rows / kRowTile * kTileA + lda / kColTile * kTileB +
         4 * (rows + 2 * lda + 6 * n) + 8 * n + kP * kP * 8 + (long long)kKTiles * kTileB + 24 * kP;
}

int coarse_inverse_blocked(int n, int nnz, const int* rp, const int* ci, const double* v, double* out,
                           DevFlags* flags, cudaStream_t s, const InverseOptions& opt) {
  if (n <= 0) return MSP_ERR_ARG;
  int cluster = opt.cluster;
  if (cluster == 0) MSP_TRY(panel_cluster(&cluster));
  if (cluster < 1 || cluster > kMaxCluster) return MSP_ERR_ARG;
  const int lda = (int)(div_up(n, kP) * kP), nrt = (int)div_up(n, kRowTile);
  const int nct = (int)div_up(n, kColTile), act = lda / kColTile;  // column tiles used, stored
  const size_t rows = (size_t)nrt * kRowTile;
  DevBuf<double> A, X, Y, D;
  DevBuf<char> SA, ST, SD;
  DevBuf<double> vs;
  DevBuf<int> ea, et, ed, piv, pivots, perm, cols_d, rs, cs, csum;
  DevBuf<unsigned long long> rmax;
  MSP_TRY(A.alloc(rows * lda));
  MSP_TRY(X.alloc((size_t)n * kP));
  MSP_TRY(Y.alloc(rows * kP));
  MSP_TRY(D.alloc(kP * kP));
  MSP_TRY(SA.alloc((size_t)nrt * kTileA));
  MSP_TRY(ST.alloc((size_t)(lda / kColTile) * kTileB));
  MSP_TRY(SD.alloc((size_t)kKTiles * kTileB));
  MSP_TRY(ea.alloc(rows));
  MSP_TRY(et.alloc(lda));
  MSP_TRY(ed.alloc(kP));
  MSP_TRY(piv.alloc(kP));
  MSP_TRY(pivots.alloc((size_t)lda));
  MSP_TRY(perm.alloc(1 + 4 * kP));
  MSP_TRY(cols_d.alloc(2 * (size_t)n));
  MSP_TRY(vs.alloc((size_t)nnz));
  MSP_TRY(rs.alloc(n));
  MSP_TRY(cs.alloc(n));
  MSP_TRY(csum.alloc(2 * (size_t)n));
  MSP_TRY(rmax.alloc(n));
  MSP_CUDA_TRY(cudaMemsetAsync(cs.p, 0, n * sizeof(int), s));
  MSP_CUDA_TRY(cudaMemsetAsync(csum.p, 0, 2 * (size_t)n * sizeof(int), s));
  MSP_CUDA_TRY(cudaMemsetAsync(rmax.p, 0, n * sizeof(unsigned long long), s));
  MSP_CUDA_TRY(cudaMemsetAsync(A.p, 0, rows * lda * sizeof(double), s));
  for (int round = 0; round <= kScaleRounds; ++round) {
    row_scale_kernel<<<grid_for(n, 128), 128, 0, s>>>(n, rp, ci, v, cs.p, round == kScaleRounds, rs.p,
                                                      csum.p, csum.p + n);
    MSP_TRY(launch_status());
    if (round == kScaleRounds) break;
    col_scale_kernel<<<grid_for(n, 128), 128, 0, s>>>(n, csum.p, csum.p + n, cs.p);
    MSP_TRY(launch_status());
  }
  csr_to_dense_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, act, rp, ci, v, rs.p, cs.p, vs.p, A.p);
  MSP_TRY(launch_status());
  const size_t diag_smem = sizeof(double) * (kP * (kP + 1) + kP);
  MSP_CUDA_TRY(cudaFuncSetAttribute(diag_inverse_panel_kernel,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, (int)diag_smem));
  for (auto* k : {slice_gemm_kernel<kUpdate>, slice_gemm_kernel<kFirst>, slice_gemm_kernel<kResid>,
                  slice_gemm_kernel<kCorrect>, slice_gemm_kernel<kResid, kCorrDigits>})
    MSP_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kGemmSmem));
  const size_t swap_smem = sizeof(double) * 2 * kP * (kColTile + 1);
  MSP_CUDA_TRY(cudaFuncSetAttribute(swap_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)swap_smem));
  const unsigned srow = div_up(rows, 32);
  // The next step's panel is updated first and factored on a second stream, by one cluster's
  // SMs, while the others update the rest: the panel's latency-bound columns would otherwise
  // leave most of the GPU idle for a third of the time.  The rest waits until the panel has
  // been copied, so that the cluster (16 SMs of one processing cluster of the chip) is
  // placed before the update's blocks take their SMs (n = 16,700: 671 -> 503 ms, 4,231: 35 ->
  // 31 ms; without that wait the cluster found no place and nothing was gained).
  SideStream side;
  MSP_TRY(side.create());
  // The factors of a step's panel (X, D and its digits, the exchanges) on stream f
  auto factor = [&](int k0, cudaStream_t f) -> int {
    const int kb = std::min(kP, n - k0), m = n - k0;
    panel_copy_kernel<<<grid_for((size_t)m * kP / 2, 256), 256, 0, f>>>(m, k0, kb, act, A.p, X.p);
    MSP_TRY(launch_status());
    MSP_CUDA_TRY(cudaEventRecord(side.copied, f));
    // the widest sub-panel whose rows fit the registers of one cluster
    const int fits = (int)div_up(m, (size_t)cluster * kLuThreads);  // rows a thread
    const int r = std::max(fits, opt.panel_rows);
    if (r <= 1)
      MSP_TRY((lu_panel<16, 1>(m, kb, k0, cluster, X.p, piv.p, flags, f)));
    else if (r <= 2)
      MSP_TRY((lu_panel<8, 2>(m, kb, k0, cluster, X.p, piv.p, flags, f)));
    else if (r <= 4)
      MSP_TRY((lu_panel<4, 4>(m, kb, k0, cluster, X.p, piv.p, flags, f)));
    else if (r <= 16)
      MSP_TRY((lu_panel<2, 16>(m, kb, k0, cluster, X.p, piv.p, flags, f)));
    else if (r <= 32)
      MSP_TRY((lu_panel<2, 32>(m, kb, k0, cluster, X.p, piv.p, flags, f)));
    else
      return MSP_ERR_NOMEM;  // two dense copies of such a matrix exceed the device
    diag_inverse_panel_kernel<<<kP / kDiagWarps + 1, kDiagWarps * kWarp, diag_smem, f>>>(
        k0, kb, X.p, piv.p, D.p, SD.p, ed.p, perm.p, pivots.p);
    return launch_status();
  };
  MSP_TRY(factor(0, s));
  for (int k0 = 0; k0 < n; k0 += kP) {
    const int kb = std::min(kP, n - k0), kt0 = k0 / kColTile;
    if (k0 > 0) MSP_CUDA_TRY(cudaStreamWaitEvent(s, side.factored, 0));
    swap_slice_kernel<<<act, 256, swap_smem, s>>>(act, k0, kb, A.p, perm.p, ST.p, et.p);
    MSP_TRY(launch_status());
    // P = -A_iK D (D for the rows K), then one correction: with the digit products the
    // residual P A_KK + A_iK is nearly exact, so P ends as accurate as its last rounding,
    // however the explicit inverse D of an ill-conditioned block was
    const unsigned pt = (unsigned)std::min(sm_count(), nrt * kKTiles);
    const char* SK = ST.p + (size_t)kt0 * kTileB;
    slice_rows_kernel<<<srow, 256, 0, s>>>(act, k0, k0, k0 + kb, A.p, SA.p, ea.p, Y.p);
    MSP_TRY(launch_status());
    slice_gemm_kernel<kFirst><<<pt, kGemmThreads, kGemmSmem, s>>>(
        act, kt0, k0, kb, nrt, kKTiles, 0, 0, 0, A.p, SA.p, ea.p, SD.p, ed.p, D.p, flags, opt.wait_ns);
    MSP_TRY(launch_status());
    slice_rows_kernel<<<srow, 256, 0, s>>>(act, k0, 0, 0, A.p, SA.p, ea.p, nullptr);
    MSP_TRY(launch_status());
    slice_gemm_kernel<kResid><<<pt, kGemmThreads, kGemmSmem, s>>>(
        kKTiles, 0, k0, kb, nrt, kKTiles, 0, 0, 0, Y.p, SA.p, ea.p, SK, et.p + k0, D.p, flags, opt.wait_ns);
    MSP_TRY(launch_status());
    slice_rows_kernel<<<srow, 256, 0, s>>>(kKTiles, 0, 0, 0, Y.p, SA.p, ea.p, nullptr);
    MSP_TRY(launch_status());
    slice_gemm_kernel<kCorrect><<<pt, kGemmThreads, kGemmSmem, s>>>(
        act, kt0, k0, kb, nrt, kKTiles, 0, 0, 0, A.p, SA.p, ea.p, SD.p, ed.p, D.p, flags, opt.wait_ns);
    MSP_TRY(launch_status());
    const int nown = std::min(nct - kt0, kKTiles), nnext = std::min(nct - kt0 - nown, kKTiles);
    if (nct - nown <= 0) continue;
    slice_rows_kernel<<<srow, 256, 0, s>>>(act, k0, 0, 0, A.p, SA.p, ea.p, nullptr);
    MSP_TRY(launch_status());
    auto update = [&](int count, int cbegin, int skip_at, int skip, int blocks) -> int {
      const long long tiles = (long long)nrt * count;
      if (tiles <= 0) return MSP_OK;
      slice_gemm_kernel<kUpdate><<<(unsigned)std::min<long long>(blocks, tiles), kGemmThreads,
                                   kGemmSmem, s>>>(act, 0, k0, kb, nrt, count, cbegin, skip_at, skip,
                                                   A.p, SA.p, ea.p, ST.p, et.p, D.p, flags, opt.wait_ns);
      return launch_status();
    };
    MSP_TRY(update(nnext, kt0 + nown, nnext, 0, sm_count()));
    if (nnext > 0) {
      MSP_CUDA_TRY(cudaEventRecord(side.ready, s));
      MSP_CUDA_TRY(cudaStreamWaitEvent(side.stream, side.ready, 0));
      MSP_TRY(factor(k0 + kP, side.stream));
      MSP_CUDA_TRY(cudaEventRecord(side.factored, side.stream));
      MSP_CUDA_TRY(cudaStreamWaitEvent(s, side.copied, 0));
    }
    MSP_TRY(update(nct - nown - nnext, 0, kt0, nown + nnext,
                   nnext > 0 ? std::max(1, sm_count() - cluster) : sm_count()));
  }
  std::vector<int> hp(n), cols(n), place(n);
  DevFlags hf{};
  MSP_CUDA_TRY(cudaMemcpyAsync(hp.data(), pivots.p, n * sizeof(int), cudaMemcpyDeviceToHost, s));
  MSP_CUDA_TRY(cudaMemcpyAsync(&hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, s));
  MSP_CUDA_TRY(cudaStreamSynchronize(s));
  if (hf.code != MSP_OK) return hf.code;
  for (int c = 0; c < n; ++c) cols[c] = c;
  for (int k = n - 1; k >= 0; --k)
    if (hp[k] != k) std::swap(cols[k], cols[hp[k]]);
  for (int c = 0; c < n; ++c) place[cols[c]] = c;
  const int* cols_p = cols_d.p;
  const int* place_p = cols_d.p + n;
  MSP_CUDA_TRY(cudaMemcpyAsync(cols_d.p, cols.data(), n * sizeof(int), cudaMemcpyHostToDevice, s));
  MSP_CUDA_TRY(cudaMemcpyAsync(cols_d.p + n, place.data(), n * sizeof(int), cudaMemcpyHostToDevice, s));
  // X += X (I - B X), the residual in `out` until the end; 128 columns of X a step, which see
  // the steps before theirs (a second-order change)
  inverse_residual_kernel<<<dim3(div_up(n, 32), std::min(nct, 16)), 256, 0, s>>>(
      n, act, rp, ci, vs.p, A.p, place_p, out, rmax.p);
  MSP_TRY(launch_status());
  const size_t corr_smem = sizeof(double) * kCorrK * (kColTile + 1);
  MSP_CUDA_TRY(cudaFuncSetAttribute(slice_residual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)corr_smem));
  for (int k0 = 0; k0 < n; k0 += kCorrK) {
    slice_inverse_kernel<<<(unsigned)(rows / kCorrRows), 256, 0, s>>>(n, act, k0, A.p, cols_p, SA.p, ea.p);
    MSP_TRY(launch_status());
    slice_residual_kernel<<<nct, 256, corr_smem, s>>>(n, k0, out, rmax.p, ST.p, et.p);
    MSP_TRY(launch_status());
    slice_gemm_kernel<kResid, kCorrDigits><<<(unsigned)std::min<long long>(sm_count(), (long long)nrt * nct),
                                   kGemmThreads, kGemmSmem, s>>>(
        act, 0, 0, 0, nrt, nct, 0, 0, 0, A.p, SA.p, ea.p, ST.p, et.p, D.p, flags, opt.wait_ns);
    MSP_TRY(launch_status());
  }
  unscramble_kernel<<<dim3(div_up(n, 32), div_up(n, 32)), 256, 0, s>>>(n, act, cols_p, A.p, rs.p, cs.p,
                                                                       out);
  MSP_TRY(launch_status());
  MSP_CUDA_TRY(cudaMemcpyAsync(&hf, flags, sizeof(hf), cudaMemcpyDeviceToHost, s));
  MSP_CUDA_TRY(cudaStreamSynchronize(s));  // cols and the temporaries are in use until here
  return hf.code;
}

}  // namespace msp

// For tests of the variants that a whole GPU or a small matrix never takes: the inverse of a
// CSR matrix (device arrays) with panels of `cluster` CTAs and at least panel_rows rows a thread,
// and the limit of the products' waits (< 0: the usual one).  Not part of the interface.
extern "C" int msp_test_inverse(int32_t n, int32_t nnz, const int32_t* d_rp, const int32_t* d_ci,
                                const double* d_v, double* d_out, int32_t cluster, int32_t panel_rows,
                                int64_t wait_ns, void* stream) {
  using namespace msp;
  DevBuf<DevFlags> flags;
  MSP_TRY(flags.alloc(1));
  MSP_CUDA_TRY(cudaMemsetAsync(flags.p, 0, sizeof(DevFlags), (cudaStream_t)stream));
  InverseOptions opt;
  opt.cluster = cluster;
  opt.panel_rows = panel_rows;
  if (wait_ns >= 0) opt.wait_ns = (unsigned long long)wait_ns;
  return coarse_inverse_blocked(n, nnz, d_rp, d_ci, d_v, d_out, flags.p, (cudaStream_t)stream, opt);
}
