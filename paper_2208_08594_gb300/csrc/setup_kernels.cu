// Setup kernels without bit-exactness requirements: pattern validation, value
// gathers, stage-N sub-blocks, BILU(0) factorisation by colour, casts.
#include <cuda_runtime.h>

#include "common.cuh"
#include "setup_kernels.h"

namespace msp {

namespace {

constexpr int kThreads = 256;

inline int launch_status() { return launch_check(__FILE__, __LINE__); }

__device__ void raise_flag(DevFlags* f, int code, int index) {
  if (atomicCAS(&f->code, MSP_OK, code) == MSP_OK) f->index = index;
}

// Every read of ci stays inside [0, nnz): a row whose pointers leave that range or
// decrease is rejected before its columns are read (nnz = rp[nb], checked by the host).
__global__ void check_pattern_kernel(int nb, int nnz, const int* __restrict__ rp,
                                     const int* __restrict__ ci, int* __restrict__ dpos,
                                     DevFlags* flags) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int p0 = rp[i], p1 = rp[i + 1];
    if (p0 < 0 || p1 < p0 || p1 > nnz) {
      dpos[i] = -2;
      raise_flag(flags, MSP_ERR_PATTERN, i);
      continue;
    }
    int d = -1;
    for (int p = p0; p < p1; ++p) {
      const int j = ci[p];
      if (j < 0 || j >= nb || (p > p0 && j <= ci[p - 1])) {
        raise_flag(flags, MSP_ERR_PATTERN, i);
        d = -2;
        break;
      }
      if (j == i) d = p;
    }
    if (d == -1) raise_flag(flags, MSP_ERR_PATTERN, i);
    dpos[i] = d;
  }
}

// instance of an original row: the last i with off[i] <= r
__device__ __forceinline__ int instance_of(int r, int B, const int* __restrict__ off) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// MSP_ERR_PATTERN where a block couples two instances (rows and columns are positions of
// the permuted pattern; perm maps them to original rows)
__global__ void check_block_diagonal_kernel(int nb, const int* __restrict__ rp,
                                            const int* __restrict__ ci, const int* __restrict__ perm,
                                            int B, const int* __restrict__ off, DevFlags* flags) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    const int inst = instance_of(perm[i], B, off);
    for (int p = rp[i]; p < rp[i + 1]; ++p)
      if (instance_of(perm[ci[p]], B, off) != inst) {
        raise_flag(flags, MSP_ERR_PATTERN, i);
        break;
      }
  }
}

__global__ void check_finite_vals_kernel(size_t n, const double* __restrict__ v, DevFlags* flags) {
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
       k += (size_t)gridDim.x * blockDim.x)
    if (!isfinite(v[k])) {
      raise_flag(flags, MSP_ERR_NONFINITE, (int)(k < 0x7fffffff ? k : 0x7fffffff));
      return;
    }
}

__global__ void gather_values_kernel(size_t nnz, int bb, const int* __restrict__ src,
                                     const double* __restrict__ in, double* __restrict__ out) {
  const size_t total = nnz * bb;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const size_t q = t / bb, k = t % bb;
    out[t] = in[(size_t)src[q] * bb + k];
  }
}

__global__ void extract_N_kernel(int b, size_t nnzb, const double* __restrict__ v,
                                 double* __restrict__ aN) {
  const int bn = b - 1;
  const size_t total = nnzb * bn * bn;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const size_t p = t / (bn * bn);
    const int rc = (int)(t % (bn * bn)), r = rc / bn, c = rc % bn;
    aN[t] = v[p * b * b + (size_t)(r + 1) * b + c + 1];
  }
}

// Stage N works with the concentration sub-blocks scaled by the inverse of their row's
// diagonal sub-block: aN[p] <- D_N,i^-1 aN[p] for the off-diagonal blocks p of row i (the
// diagonal block is left as it is and never read by the sweeps).  One thread per row.
template <int BN>
__global__ void scale_N_rows_kernel(int nb, const int* __restrict__ rp, const int* __restrict__ dpos,
                                    const double* __restrict__ dNinv, double* __restrict__ aN) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nb; i += gridDim.x * blockDim.x) {
    double D[BN * BN];
#pragma unroll
    for (int e = 0; e < BN * BN; ++e) D[e] = dNinv[(size_t)i * BN * BN + e];
    const int pd = dpos[i];
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
      if (p == pd) continue;
      double* a = aN + (size_t)p * BN * BN;
      double in[BN * BN];
#pragma unroll
      for (int e = 0; e < BN * BN; ++e) in[e] = a[e];
#pragma unroll
      for (int r = 0; r < BN; ++r)
#pragma unroll
        for (int c = 0; c < BN; ++c) {
          double t = 0.0;
#pragma unroll
          for (int k = 0; k < BN; ++k) t = fma(D[r * BN + k], in[k * BN + c], t);
          a[r * BN + c] = t;
        }
    }
  }
}

__global__ void diag_pos_kernel(int n, const int* __restrict__ rp, const int* __restrict__ ci,
                                int* __restrict__ dpos) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int d = -1;
    for (int p = rp[i]; p < rp[i + 1]; ++p)
      if (ci[p] == i) {
        d = p;
        break;
      }
    dpos[i] = d;
  }
}

// Greedy first-fit colouring in Jones-Plassmann priority order (an alternative to
// Algorithms 4.1/4.2): priority keys, then rounds in which every vertex whose higher-
// priority neighbours are all coloured takes the smallest colour none of them has.  A
// vertex's colour depends only on those neighbours' final colours, so the result is the
// sequential greedy's in priority order whatever the rounds' timing (a neighbour coloured
// in the same round and not yet seen only delays a vertex to the next round).
__device__ __forceinline__ unsigned long long jp_splitmix64(unsigned long long x) {
  // SplitMix64 output function (Vigna)
  unsigned long long z = x + 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

// key: larger degree first, then the smaller high word of SplitMix64(v ^ seed); a stable
// sort of the keys in index order breaks the remaining ties by index
__global__ void jp_keys_kernel(int n, const int* __restrict__ srp, unsigned long long seed,
                               unsigned long long* __restrict__ key, int* __restrict__ idx) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const unsigned long long deg = (unsigned long long)(srp[v + 1] - srp[v]);
    key[v] = ((0x7FFFFFFFull - deg) << 32) | (jp_splitmix64((unsigned long long)v ^ seed) >> 32);
    idx[v] = v;
  }
}

__global__ void jp_round_kernel(int n, const int* __restrict__ srp, const int* __restrict__ sci,
                                const int* __restrict__ rank, int* colour,
                                int* __restrict__ counters) {
  int done_here = 0, gmax = 0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    if (colour[v] != 0) continue;
    const int rv = rank[v];
    const int q0 = srp[v], q1 = srp[v + 1];
    unsigned long long used = 0;  // colours 1..64 of the higher-priority neighbours
    bool ready = true, high = false;
    for (int q = q0; q < q1; ++q) {
      const int u = sci[q];
      if (rank[u] > rv) continue;
      const int cu = *(volatile int*)(colour + u);
      if (cu == 0) {
        ready = false;
        break;
      }
      if (cu <= 64)
        used |= 1ull << (cu - 1);
      else
        high = true;
    }
    if (!ready) continue;
    int c = __ffsll(~used);  // smallest colour in 1..64 not taken (0 if all 64 are)
    if (c == 0 || high) {  // rare: a colour above 64 among the neighbours
      c = 1;
      for (bool taken = true; taken; ++c) {
        taken = false;
        for (int q = q0; q < q1 && !taken; ++q) {
          const int u = sci[q];
          taken = rank[u] < rv && *(volatile int*)(colour + u) == c;
        }
        if (!taken) break;
      }
    }
    colour[v] = c;
    ++done_here;
    gmax = max(gmax, c);
  }
  if (done_here) {
    atomicAdd(counters, done_here);
    atomicMax(counters + 1, gmax);
  }
}

// Sizes of the two-hop lists of a graph for VerticesGrouping: for every vertex v the rows of
// its neighbours, with repeats (an upper bound of its second circle).
__global__ void twohop_count_kernel(int n, const int* __restrict__ srp,
                                    const int* __restrict__ sci, int* __restrict__ cnt,
                                    unsigned long long* __restrict__ total) {
  __shared__ unsigned long long part[kThreads / 32];
  unsigned long long mine = 0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    int c = 0;
    for (int q = srp[v]; q < srp[v + 1]; ++q) {
      const int k = sci[q];
      c += srp[k + 1] - srp[k];
    }
    cnt[v] = c;
    mine += (unsigned long long)c;
  }
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (threadIdx.x % 32 == 0) part[threadIdx.x / 32] = mine;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += part[w];
    atomicAdd(total, t);
  }
}

// Lists of VerticesGrouping, one warp per vertex: v's neighbours, then its second circle (the
// vertices of its neighbours' rows) without repeats and without v and its neighbours; a hash
// table in shared memory finds the repeats.  A second circle too large for the table is
// stored as it comes (the colouring passes over what is not in V or already in the
// frontier; it only tests more).  Place: start[v] = tp[v] + srp[v].
constexpr int kHashSlots = 512;
__global__ void __launch_bounds__(kThreads) twohop_lists_kernel(int n, const int* __restrict__ srp,
                                                                const int* __restrict__ sci,
                                                                const int* __restrict__ tp,
                                                                const int* __restrict__ cnt,
                                                                int4* __restrict__ meta,
                                                                int* __restrict__ list) {
  __shared__ int table[kThreads / 32][kHashSlots];
  const int lane = threadIdx.x % 32;
  int* tab = table[threadIdx.x / 32];
  const int warps = gridDim.x * (blockDim.x / 32);
  // true when x was not in the table yet
  auto insert = [&](int x) {
    unsigned h = ((unsigned)x * 2654435761u) >> 23;
    while (true) {
      const int old = atomicCAS(tab + h, -1, x);
      if (old == -1) return true;
      if (old == x) return false;
      h = (h + 1) & (kHashSlots - 1);
    }
  };
  for (int v = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; v < n; v += warps) {
    const int q0 = srp[v], deg = srp[v + 1] - q0;
    const int start = tp[v] + q0;
    const bool hashed = deg + cnt[v] < kHashSlots * 3 / 4;  // the table always keeps free slots
    if (hashed) {
      for (int k = lane; k < kHashSlots; k += 32) tab[k] = -1;
      __syncwarp();
      if (lane == 0) insert(v);
    }
    for (int q = lane; q < deg; q += 32) {
      const int j = sci[q0 + q];
      list[start + q] = j;
      if (hashed) insert(j);
    }
    __syncwarp();
    int pos = start + deg;
    for (int q = 0; q < deg; ++q) {
      const int k = sci[q0 + q], e0 = srp[k], e1 = srp[k + 1];
      for (int e = e0; e < e1; e += 32) {
        int x = 0;
        bool keep = false;
        if (e + lane < e1) {
          x = sci[e + lane];
          keep = !hashed || insert(x);
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) list[pos + __popc(m & ((1u << lane) - 1u))] = x;
        pos += __popc(m);
      }
    }
    if (lane == 0) meta[v] = make_int4(start, deg, pos - start, 0);
    __syncwarp();
  }
}

// ELL copy of the off-diagonal entries of a CSR level matrix for the colour sweeps and the
// restriction: slot k of row i at i*K + k, in the row's CSR order; unused slots hold (i, 0);
// diag[i] = a_ii.  meta[i] = number of off-diagonal entries | (entries left of the
// diagonal) << 16, or -1 for a row with more than K of them (that row keeps only its CSR
// form and every slot is unused).
__global__ void build_ell_kernel(int n, int K, const int* __restrict__ rp,
                                 const int* __restrict__ ci, const double* __restrict__ v,
                                 const int* __restrict__ dpos, int* __restrict__ ell_ci,
                                 double* __restrict__ ell_v, int* __restrict__ meta,
                                 double* __restrict__ diag) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int p0 = rp[i], p1 = rp[i + 1], pd = dpos[i];
    diag[i] = v[pd];
    const int len = p1 - p0 - 1;
    int k = 0;
    if (len <= K) {
      for (int p = p0; p < p1; ++p) {
        if (p == pd) continue;
        ell_ci[(size_t)i * K + k] = ci[p];
        ell_v[(size_t)i * K + k] = v[p];
        ++k;
      }
      meta[i] = len | ((pd - p0) << 16);
    } else {
      meta[i] = -1;
    }
    for (; k < K; ++k) {
      ell_ci[(size_t)i * K + k] = i;
      ell_v[(size_t)i * K + k] = 0.0;
    }
  }
}

__global__ void rdiag_kernel(int n, const int* __restrict__ dpos, const double* __restrict__ v,
                             double* __restrict__ rdiag, DevFlags* flags) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int d = dpos[i];
    const double a = d >= 0 ? v[d] : 0.0;
    if (!(a != 0.0)) {
      raise_flag(flags, MSP_ERR_SINGULAR_BLOCK, i);
      rdiag[i] = 0.0;
    } else {
      rdiag[i] = 1.0 / a;
    }
  }
}

template <int N>
__device__ bool small_inverse(const double* __restrict__ D, double* X) {
  double a[N][N], x[N][N];
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int c = 0; c < N; ++c) {
      a[r][c] = D[r * N + c];
      x[r][c] = (r == c) ? 1.0 : 0.0;
    }
  for (int c = 0; c < N; ++c) {
    int p = c;
    for (int r = c + 1; r < N; ++r)
      if (fabs(a[r][c]) > fabs(a[p][c])) p = r;
    if (!(a[p][c] != 0.0) || !isfinite(a[p][c])) return false;
    if (p != c) {
#pragma unroll
      for (int k = 0; k < N; ++k) {
        double t = a[p][k];
        a[p][k] = a[c][k];
        a[c][k] = t;
        t = x[p][k];
        x[p][k] = x[c][k];
        x[c][k] = t;
      }
    }
    const double inv = 1.0 / a[c][c];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      a[c][k] *= inv;
      x[c][k] *= inv;
    }
    for (int r = 0; r < N; ++r) {
      if (r == c) continue;
      const double f = a[r][c];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        a[r][k] -= f * a[c][k];
        x[r][k] -= f * x[c][k];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int c = 0; c < N; ++c) X[r * N + c] = x[r][c];
  return true;
}

// Block ILU(0) (IKJ form) of the rows of one colour: for every k < i in the pattern,
// L_ik = A_ik U_kk^-1 and A_ij -= L_ik A_kj for the later j of row i present in row k.
template <int B>
__global__ void bilu_factor_kernel(int r0, int r1, const int* __restrict__ rp,
                                   const int* __restrict__ ci, const int* __restrict__ dpos,
                                   double* __restrict__ lu, double* __restrict__ uinv,
                                   DevFlags* flags) {
  constexpr int BB = B * B;
  for (int i = r0 + blockIdx.x * blockDim.x + threadIdx.x; i < r1; i += gridDim.x * blockDim.x) {
    const int p0 = rp[i], pd = dpos[i], p1 = rp[i + 1];
    for (int p = p0; p < pd; ++p) {
      const int k = ci[p];
      double L[BB];
      const double* Ap = lu + (size_t)p * BB;
      const double* Uk = uinv + (size_t)k * BB;
#pragma unroll
      for (int r = 0; r < B; ++r)
#pragma unroll
        for (int c = 0; c < B; ++c) {
          double s = 0.0;
#pragma unroll
          for (int m = 0; m < B; ++m) s = fma(Ap[r * B + m], Uk[m * B + c], s);
          L[r * B + c] = s;
        }
#pragma unroll
      for (int t = 0; t < BB; ++t) lu[(size_t)p * BB + t] = L[t];
      const int k0 = rp[k], k1 = rp[k + 1];
      int kr = k0;
      for (int q = p + 1; q < p1; ++q) {
        const int j = ci[q];
        while (kr < k1 && ci[kr] < j) ++kr;  // both rows ascending
        if (kr >= k1) break;
        if (ci[kr] != j) continue;
        const double* Ukj = lu + (size_t)kr * BB;
        double* Aq = lu + (size_t)q * BB;
#pragma unroll
        for (int r = 0; r < B; ++r)
#pragma unroll
          for (int c = 0; c < B; ++c) {
            double s = 0.0;
#pragma unroll
            for (int m = 0; m < B; ++m) s = fma(L[r * B + m], Ukj[m * B + c], s);
            Aq[r * B + c] -= s;
          }
      }
    }
    double X[BB];
    if (!small_inverse<B>(lu + (size_t)pd * BB, X)) {
      raise_flag(flags, MSP_ERR_SINGULAR_BLOCK, i);
      continue;
    }
#pragma unroll
    for (int t = 0; t < BB; ++t) uinv[(size_t)i * BB + t] = X[t];
  }
}

__global__ void cast_vals_kernel(size_t n, const double* __restrict__ in, float* __restrict__ out) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n;
       t += (size_t)gridDim.x * blockDim.x)
    out[t] = (float)in[t];
}

__global__ void iota_kernel(int n, int* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = i;
}

__global__ void fill_int_kernel(size_t n, int value, int* out) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = value;
}

__global__ void scatter_inverse_kernel(int n, const int* __restrict__ perm, int* __restrict__ iperm) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
    iperm[perm[k]] = k;
}

}  // namespace

int launch_check_pattern(int nb, int nnz, const int* rp, const int* ci, int* dpos, DevFlags* flags,
                         cudaStream_t s) {
  check_pattern_kernel<<<grid_for(nb, kThreads), kThreads, 0, s>>>(nb, nnz, rp, ci, dpos, flags);
  return launch_status();
}

int launch_check_block_diagonal(int nb, const int* rp, const int* ci, const int* perm, int B,
                                const int* off, DevFlags* flags, cudaStream_t s) {
  if (nb <= 0) return MSP_OK;
  check_block_diagonal_kernel<<<grid_for(nb, kThreads), kThreads, 0, s>>>(nb, rp, ci, perm, B,
                                                                          off, flags);
  return launch_status();
}

int launch_check_finite_vals(size_t n, const double* v, DevFlags* flags, cudaStream_t s) {
  if (!n) return MSP_OK;
  check_finite_vals_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, v, flags);
  return launch_status();
}

int launch_gather_values(size_t nnz, int bb, const int* src, const double* in, double* out,
                         cudaStream_t s) {
  if (!nnz) return MSP_OK;
  gather_values_kernel<<<grid_for(nnz * bb, kThreads), kThreads, 0, s>>>(nnz, bb, src, in, out);
  return launch_status();
}

int launch_extract_N(int b, size_t nnzb, const double* v, double* aN, cudaStream_t s) {
  if (b < 2 || !nnzb) return MSP_OK;
  extract_N_kernel<<<grid_for(nnzb * (b - 1) * (b - 1), kThreads), kThreads, 0, s>>>(b, nnzb, v,
                                                                                     aN);
  return launch_status();
}

int launch_scale_N_rows(int b, int nb, const int* rp, const int* dpos, const double* dNinv,
                        double* aN, cudaStream_t s) {
  if (nb <= 0 || b < 2) return MSP_OK;
  const unsigned grid = grid_for(nb, kThreads);
  switch (b - 1) {
    case 1: scale_N_rows_kernel<1><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 2: scale_N_rows_kernel<2><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 3: scale_N_rows_kernel<3><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 4: scale_N_rows_kernel<4><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 5: scale_N_rows_kernel<5><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 6: scale_N_rows_kernel<6><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    case 7: scale_N_rows_kernel<7><<<grid, kThreads, 0, s>>>(nb, rp, dpos, dNinv, aN); break;
    default: return MSP_ERR_ARG;
  }
  return launch_status();
}

int launch_diag_pos(int n, const int* rp, const int* ci, int* dpos, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  diag_pos_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, rp, ci, dpos);
  return launch_status();
}

int launch_jp_keys(int n, const int* srp, unsigned long long seed, unsigned long long* key,
                   int* idx, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  jp_keys_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, srp, seed, key, idx);
  return launch_status();
}

int launch_jp_round(int n, const int* srp, const int* sci, const int* rank, int* colour,
                    int* counters, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  jp_round_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, srp, sci, rank, colour,
                                                             counters);
  return launch_status();
}

int launch_twohop_count(int n, const int* srp, const int* sci, int* cnt, unsigned long long* total,
                        cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  MSP_CUDA_TRY(cudaMemsetAsync(total, 0, sizeof(unsigned long long), s));
  twohop_count_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, srp, sci, cnt, total);
  return launch_status();
}

int launch_twohop_lists(int n, const int* srp, const int* sci, const int* tp, const int* cnt,
                        int4* meta, int* list, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  twohop_lists_kernel<<<grid_for((size_t)n * 32, kThreads), kThreads, 0, s>>>(n, srp, sci, tp, cnt,
                                                                             meta, list);
  return launch_status();
}

int launch_build_ell(int n, int K, const int* rp, const int* ci, const double* v, const int* dpos,
                     int* ell_ci, double* ell_v, int* meta, double* diag, cudaStream_t s) {
  if (n <= 0 || K <= 0) return MSP_OK;
  build_ell_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, K, rp, ci, v, dpos, ell_ci,
                                                              ell_v, meta, diag);
  return launch_status();
}

int launch_rdiag(int n, const int* dpos, const double* v, double* rdiag, DevFlags* flags,
                 cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  rdiag_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, dpos, v, rdiag, flags);
  return launch_status();
}

int launch_bilu_factor(int b, int r0, int r1, const int* rp, const int* ci, const int* dpos,
                       double* lu, double* uinv, DevFlags* flags, cudaStream_t s) {
  if (r1 <= r0) return MSP_OK;
  const unsigned grid = grid_for(r1 - r0, 128);
  switch (b) {
#define MSP_BF_CASE(BB)                                                                   \
  case BB:                                                                                \
    bilu_factor_kernel<BB><<<grid, 128, 0, s>>>(r0, r1, rp, ci, dpos, lu, uinv, flags);   \
    break;
    MSP_BF_CASE(1)
    MSP_BF_CASE(2)
    MSP_BF_CASE(3)
    MSP_BF_CASE(4)
    MSP_BF_CASE(5)
    MSP_BF_CASE(6)
    MSP_BF_CASE(7)
    MSP_BF_CASE(8)
#undef MSP_BF_CASE
    default:
      return MSP_ERR_ARG;
  }
  return launch_status();
}

int launch_cast_vals(size_t n, const double* in, float* out, cudaStream_t s) {
  if (!n) return MSP_OK;
  cast_vals_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, in, out);
  return launch_status();
}

int launch_iota(int n, int* out, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  iota_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, out);
  return launch_status();
}

int launch_fill_int(size_t n, int value, int* out, cudaStream_t s) {
  if (!n) return MSP_OK;
  fill_int_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, value, out);
  return launch_status();
}

int launch_scatter_inverse(int n, const int* perm, int* iperm, cudaStream_t s) {
  if (n <= 0) return MSP_OK;
  scatter_inverse_kernel<<<grid_for(n, kThreads), kThreads, 0, s>>>(n, perm, iperm);
  return launch_status();
}

}  // namespace msp
