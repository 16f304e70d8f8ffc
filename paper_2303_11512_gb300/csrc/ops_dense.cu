// Dense FP64 kernels: Gauss-Jordan inverses (SAP blocks, the coarsest level of
// Algorithm 2 whose trace is tau_L), the coarsest-level inverse apply, and the
// Hutch++ pieces of Algorithm 2: the Gram matrix and Cholesky factor of
// CholeskyQR2 and the projection coefficients Q^H x.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "ops.cuh"

namespace mg {

namespace {
template <typename T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffff, v, o);
  return v;
}
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ double cabs2(float2 a) { return (double)a.x * a.x + (double)a.y * a.y; }
__device__ __forceinline__ double2 crecip(double2 a) {
  const double s = 1.0 / cabs2(a);
  return make_double2(a.x * s, -a.y * s);
}
__device__ __forceinline__ float2 crecip(float2 a) {
  const float s = 1.0f / (a.x * a.x + a.y * a.y);
  return make_float2(a.x * s, -a.y * s);
}
}  // namespace

// ---- batched small inverse (one CTA per matrix) ------------------------------------------------
// Gauss-Jordan with partial pivoting in shared memory, three barriers per column: pivot search (warp 0, also
// the reciprocal of the pivot), then the row swap, pivot-row scaling and multipliers (read all, barrier,
// write all), then the rank-1 elimination.  BD = block dimension at compile time (0: runtime bd).
template <typename C, int BD>
__global__ void __launch_bounds__(256) k_invert_small(C* __restrict__ Ag, int bd_, int* fail) {
  const int bd = BD ? BD : bd_;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* A = reinterpret_cast<C*>(smem_raw);
  C* sf = A + bd * bd;
  int* perm = reinterpret_cast<int*>(sf + bd);
  __shared__ int s_p;
  __shared__ int s_bad;
  __shared__ C s_a;
  C* G = Ag + (size_t)blockIdx.x * bd * bd;
  for (int e = threadIdx.x; e < bd * bd; e += 256) A[e] = G[e];
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int k = 0; k < bd; ++k) {
    if (threadIdx.x < 32) {
      double best = -1.0;
      int bi = k;
      for (int i = k + threadIdx.x; i < bd; i += 32) {
        double v = cabs2(A[i * bd + k]);
        if (v > best) { best = v; bi = i; }
      }
      for (int o = 16; o; o >>= 1) {
        double ob = __shfl_xor_sync(0xffffffff, best, o);
        int oi = __shfl_xor_sync(0xffffffff, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (threadIdx.x == 0) {
        s_p = bi;
        perm[k] = bi;
        if (!(best > 0.0)) s_bad = 1;
        s_a = best > 0.0 ? crecip(A[bi * bd + k]) : czero<C>();
      }
    }
    __syncthreads();
    if (s_bad) break;
    const int p = s_p;
    const C a = s_a;
    // swap rows k and p, scale the pivot row, multipliers of the swapped column k
    C tk, tp, ck, akk;
    const int t = threadIdx.x;
    if (t < bd) {
      tk = A[k * bd + t];
      tp = A[p * bd + t];
      ck = A[t * bd + k];
      akk = A[k * bd + k];
    }
    __syncthreads();
    if (t < bd) {
      if (p != k) A[p * bd + t] = tk;
      A[k * bd + t] = (t == k) ? a : cmul(tp, a);
      sf[t] = (t == k) ? czero<C>() : cneg(t == p ? akk : ck);  // minus the multiplier
    }
    __syncthreads();
    for (int e = threadIdx.x; e < bd * bd; e += 256) {
      const int i = e / bd, j = e - i * bd;
      if (i != k) A[e] = cfma(sf[i], A[k * bd + j], j == k ? czero<C>() : A[e]);
    }
    __syncthreads();
  }
  if (s_bad) {
    if (threadIdx.x == 0) atomicExch(fail, 1);
    return;
  }
  for (int k = bd - 1; k >= 0; --k) {
    const int p = perm[k];
    if (p != k)
      for (int i = threadIdx.x; i < bd; i += 256) {
        C t = A[i * bd + k];
        A[i * bd + k] = A[i * bd + p];
        A[i * bd + p] = t;
      }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < bd * bd; e += 256) G[e] = A[e];
}

template <typename C>
void invert_small_batched(cudaStream_t st, C* A, int nmat, int bd, int* fail) {
  MG_CHECK_ARG(bd <= 64, "small inverse limited to 64 x 64");
  size_t sm = sizeof(C) * ((size_t)bd * bd + bd) + sizeof(int) * bd + 16;
  auto attr = [&](auto kern, int) { ensure_max_smem((const void*)kern, 100 * 1024); };
  if (bd == 64) {
    attr(k_invert_small<C, 64>, 0);
    MG_LAUNCH((k_invert_small<C, 64>), nmat, 256, sm, st, A, bd, fail);
  } else if (bd == 32) {
    attr(k_invert_small<C, 32>, 1);
    MG_LAUNCH((k_invert_small<C, 32>), nmat, 256, sm, st, A, bd, fail);
  } else {
    attr(k_invert_small<C, 0>, 2);
    MG_LAUNCH((k_invert_small<C, 0>), nmat, 256, sm, st, A, bd, fail);
  }
}
template void invert_small_batched<double2>(cudaStream_t, double2*, int, int, int*);
template void invert_small_batched<float2>(cudaStream_t, float2*, int, int, int*);

// ---- large in-place inverse: Gauss-Jordan with partial pivoting in one cooperative kernel ------------
// The CTAs of the grid (all resident, cooperative launch) sweep the columns in step: per column k the pivot
// p = argmax_{i >= k} |A_ik| (ties: smallest i) comes from per-CTA partial maxima, rows k and p are swapped,
// the pivot row is scaled by a = 1 / A_pk (its column-k entry becomes a) and every other row i loses
// f_i x (pivot row), its column-k entry becoming -f_i a.  Column k reads one matrix buffer and writes the
// other (ping-pong), so every CTA can read the pivot row and column while others already write: one grid
// barrier per column.  The barrier spins on a generation counter with an iteration limit (timeout flag, all
// CTAs then leave).  Columns are unscrambled afterwards by the recorded swaps in reverse order.
constexpr int GJ_T = 512;

// `expect` arrivals release the barrier (the grid size; one more in the bounded-wait self-test, where nothing
// releases it and every wait runs out after `polls` polls)
__device__ __forceinline__ bool gj_barrier(unsigned* bar, unsigned expect, long polls, int* timeout, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    int ok = 1;
    if (atomicAdd(bar, 1u) == expect - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long it = 0;
      while (*gen == g) {
        if (++it > polls) {
          atomicExch(timeout, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    *s_ok = ok && !*(volatile int*)timeout;
  }
  __syncthreads();
  return *s_ok;
}

// block-wide argmax (value, smallest index on ties), result in thread 0
__device__ __forceinline__ void gj_block_argmax(double& best, int& idx, double* sb, int* si) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffff, best, o);
    const int oi = __shfl_xor_sync(0xffffffff, idx, o);
    if (ob > best || (ob == best && oi < idx)) { best = ob; idx = oi; }
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) { sb[w] = best; si[w] = idx; }
  __syncthreads();
  if (w == 0) {
    best = l < GJ_T / 32 ? sb[l] : -1.0;
    idx = l < GJ_T / 32 ? si[l] : 0x7fffffff;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffff, best, o);
      const int oi = __shfl_xor_sync(0xffffffff, idx, o);
      if (ob > best || (ob == best && oi < idx)) { best = ob; idx = oi; }
    }
  }
}

// A0: the matrix (result written back here); A1: scratch of the same size; slots: per-CTA (max, index)
// of the next pivot column, double-buffered by column parity
template <typename C>
__global__ void __launch_bounds__(GJ_T, 1) k_gj_coop(C* __restrict__ A0, C* __restrict__ A1, int n,
                                                    int* __restrict__ piv, double* __restrict__ slot_v,
                                                    int* __restrict__ slot_i, unsigned* bar, int* fail,
                                                    int* timeout, long polls, unsigned expect) {
  __shared__ double sb[GJ_T / 32];
  __shared__ int si[GJ_T / 32];
  __shared__ int s_ok, s_p;
  __shared__ C s_a;
  extern __shared__ __align__(16) unsigned char gj_smem[];
  C* s_row = reinterpret_cast<C*>(gj_smem);  // the scaled pivot row of the current column
  const unsigned nb = gridDim.x;
  // column 0 partial maxima into slot set 0
  {
    double best = -1.0;
    int idx = 0x7fffffff;
    for (int i = blockIdx.x * GJ_T + threadIdx.x; i < n; i += nb * GJ_T) {
      const double v = cabs2(A0[(size_t)i * n]);
      if (v > best || (v == best && i < idx)) { best = v; idx = i; }
    }
    gj_block_argmax(best, idx, sb, si);
    if (threadIdx.x == 0) { slot_v[blockIdx.x] = best; slot_i[blockIdx.x] = idx; }
  }
  if (!gj_barrier(bar, expect, polls, timeout, &s_ok)) return;
  for (int k = 0; k < n; ++k) {
    const C* __restrict__ cur = (k & 1) ? A1 : A0;
    C* __restrict__ nxt = (k & 1) ? A0 : A1;
    const double* sv = slot_v + (k & 1) * 1024;
    const int* sx = slot_i + (k & 1) * 1024;
    // pivot from the partial maxima (every CTA reaches the same decision)
    if (threadIdx.x < 32) {
      double best = -1.0;
      int idx = 0x7fffffff;
      for (unsigned c = threadIdx.x; c < nb; c += 32) {
        const double v = sv[c];
        const int i = sx[c];
        if (v > best || (v == best && i < idx)) { best = v; idx = i; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffff, best, o);
        const int oi = __shfl_xor_sync(0xffffffff, idx, o);
        if (ob > best || (ob == best && oi < idx)) { best = ob; idx = oi; }
      }
      if (threadIdx.x == 0) {
        const bool good = best > 0.0 && idx >= k && idx < n;
        s_p = good ? idx : k;
        if (!good && blockIdx.x == 0) atomicExch(fail, 1);
        s_a = good ? crecip(cur[(size_t)s_p * n + k]) : czero<C>();
        if (blockIdx.x == 0) piv[k] = s_p;
      }
    }
    __syncthreads();
    const int p = s_p;
    const C a = s_a;
    const C fk = cur[(size_t)k * n + k];  // multiplier of row p after the swap
    for (int j = threadIdx.x; j < n; j += GJ_T) s_row[j] = (j == k) ? a : cmul(cur[(size_t)p * n + j], a);
    __syncthreads();
    // eliminate into nxt; track the next pivot column's partial maximum
    double best = -1.0;
    int idx = 0x7fffffff;
    const int kn = k + 1;
#pragma unroll 2
    for (int i = blockIdx.x; i < n; i += (int)nb) {
      const C f = (i == k) ? czero<C>() : (i == p ? fk : cur[(size_t)i * n + k]);
      const C* src = cur + (size_t)(i == p ? k : i) * n;  // row p takes the old row k
#pragma unroll 4
      for (int j = threadIdx.x; j < n; j += GJ_T) {
        const C r = s_row[j];  // new pivot row
        C v;
        if (i == k)
          v = r;
        else if (j == k)
          v = cneg(cmul(f, r));
        else
          v = csub(src[j], cmul(f, r));
        nxt[(size_t)i * n + j] = v;
        if (j == kn && i >= kn) {
          const double m = cabs2(v);
          if (m > best || (m == best && i < idx)) { best = m; idx = i; }
        }
      }
    }
    gj_block_argmax(best, idx, sb, si);
    if (threadIdx.x == 0) {
      slot_v[((k + 1) & 1) * 1024 + blockIdx.x] = best;
      slot_i[((k + 1) & 1) * 1024 + blockIdx.x] = idx;
    }
    if (!gj_barrier(bar, expect, polls, timeout, &s_ok)) return;
  }
}

// ---- the same inverse by block columns ------------------------------------------------------------------
// In-place Gauss-Jordan on GJ_NB columns at a time.  A panel kernel (one cluster of 8 CTAs, the n x GJ_NB panel in
// their shared memory) eliminates its columns with the pivot search over the rows below; what it leaves in the panel,
// G, is the whole transformation: with A' the rows swapped as the panel chose,
//   A_new(i, j) = [i not in the block] A'(i, j) + sum_q G(i, q) A'(k0 + q, j)
// for the other columns, a rank-GJ_NB update over the whole grid (ping-pong buffers, so that swapped rows are read
// where they were).  Pivots and their ties are those of k_gj_coop.  A grid barrier per column (22 us at n = 1024) is
// replaced by two cluster barriers (the panel takes about 5 us a column: barriers, remote rows, the reciprocal); the
// update runs at the FMA rate (FP64: two a clock and SM, 6.9 ms in all).  n = 256, 1024, 2304: FP64 2.7, 25.9, 213 ->
// 1.7, 16.0, 117 ms, FP32 2.3, 14.9, 87 -> 1.1, 6.6, 30 ms.
constexpr int GJ_NB = 8, GJ_CS = 8, GJ_PT = 256;

__device__ __forceinline__ long long gj_key(double v) {  // ordering of non-negative doubles as integers, NaN last
  return v >= 0.0 ? __double_as_longlong(v) : -1ll;
}

template <typename C>
__global__ void __cluster_dims__(GJ_CS, 1, 1) __launch_bounds__(GJ_PT)
    k_gj_panel(const C* __restrict__ A, int n, int k0, int nb, C* __restrict__ G, int* __restrict__ piv, int* fail) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = cl.block_rank(), tid = threadIdx.x, w = tid >> 5, l = tid & 31;
  const int rpc = (n + GJ_CS - 1) / GJ_CS, i0 = rank * rpc, nrow = max(0, min(rpc, n - i0));
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);  // [row][GJ_NB]
  __shared__ long long slot_v[2][GJ_CS];  // candidate of every CTA, double-buffered by column parity
  __shared__ int slot_i[2][GJ_CS];
  __shared__ long long wv[GJ_PT / 32];
  __shared__ int wi[GJ_PT / 32];
  __shared__ int s_p, s_good;
  __shared__ C s_a, prow[GJ_NB], krow[GJ_NB];
  for (int e = tid; e < nrow * GJ_NB; e += GJ_PT) {
    const int r = e / GJ_NB, q = e % GJ_NB;
    P[e] = q < nb ? A[(size_t)(i0 + r) * n + k0 + q] : czero<C>();
  }
  cl.sync();  // every CTA of the cluster runs before its shared memory is written to
  auto better = [](long long v, int i, long long v2, int i2) { return v > v2 || (v == v2 && i < i2); };
  for (int q = 0; q < nb; ++q) {
    const int k = k0 + q, par = q & 1;
    long long bv = -1;
    int bi = 0x7fffffff;
    for (int r = tid; r < nrow; r += GJ_PT) {
      const int i = i0 + r;
      if (i >= k) {
        const long long v = gj_key(cabs2(P[r * GJ_NB + q]));
        if (better(v, i, bv, bi)) { bv = v; bi = i; }
      }
    }
    auto warp_best = [&](int width) {
      for (int o = width / 2; o; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffff, bv, o);
        const int oi = __shfl_xor_sync(0xffffffff, bi, o);
        if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
      }
    };
    warp_best(32);
    if (l == 0) { wv[w] = bv; wi[w] = bi; }
    __syncthreads();
    if (w == 0) {
      bv = wv[l & 7];
      bi = wi[l & 7];
      warp_best(8);
      if (l < GJ_CS) {  // to the slot of this CTA in every CTA of the cluster
        *cl.map_shared_rank(&slot_v[par][rank], l) = bv;
        *cl.map_shared_rank(&slot_i[par][rank], l) = bi;
      }
    }
    cl.sync();
    if (w == 0) {
      bv = slot_v[par][l & 7];
      bi = slot_i[par][l & 7];
      warp_best(8);
      const bool good = bv > 0 && bi >= k && bi < n;
      const int p = good ? bi : k;
      // pivot row (lanes 0-7) and row k (lanes 8-15) from their owners
      const int row = l < GJ_NB ? p : k, c = l & (GJ_NB - 1);
      if (l < 2 * GJ_NB) {
        const C v = cl.map_shared_rank(P, row / rpc)[(row % rpc) * GJ_NB + c];
        (l < GJ_NB ? prow : krow)[c] = v;
        if (l == q) s_a = good ? crecip(v) : czero<C>();
      }
      if (l == 0) {
        s_p = p;
        s_good = good;
      }
    }
    cl.sync();  // everybody has read the two rows
    const int p = s_p, c = tid & (GJ_NB - 1);
    const C a = s_a, r = c == q ? a : cmul(prow[c], a);  // entry c of the scaled pivot row
    if (rank == 0 && tid == 0) {
      piv[k] = p;
      if (!s_good) atomicExch(fail, 1);
    }
    constexpr int STEP = GJ_PT / GJ_NB;
    for (int m = 0; m < (rpc + STEP - 1) / STEP; ++m) {  // the same trips for every lane: the 8 threads of a row sit
      const int rr = m * STEP + tid / GJ_NB, i = i0 + rr;  // in one warp and wait for each other
      C* row = P + rr * GJ_NB;
      C f = czero<C>(), src = f;
      if (rr < nrow) {
        f = i == p ? krow[q] : row[q];
        src = i == p ? krow[c] : row[c];
      }
      __syncwarp();
      if (rr < nrow) row[c] = i == k ? r : cfma(cneg(f), r, c == q ? czero<C>() : src);
      __syncwarp();
    }
    __syncthreads();
  }
  for (int e = tid; e < nrow * GJ_NB; e += GJ_PT) G[(size_t)i0 * GJ_NB + e] = P[e];
  cl.sync();  // no CTA leaves while another may still read its panel
}

// X -> Y by the panel's transformation: 32 x 32 entries per CTA, 8 rows of one column per thread
template <typename C>
__global__ void __launch_bounds__(128) k_gj_update(const C* __restrict__ X, C* __restrict__ Y, int n, int k0, int nb,
                                                   const C* __restrict__ G, const int* __restrict__ piv) {
  __shared__ __align__(16) C sG[32][GJ_NB];
  __shared__ int src[32 + GJ_NB];  // rows of X that the tile's rows, and the block's rows, come from
  const int tid = threadIdx.x, i0 = blockIdx.y * 32, j = blockIdx.x * 32 + (tid & 31);
  for (int e = tid; e < 32 * GJ_NB; e += 128) sG[e / GJ_NB][e % GJ_NB] = i0 * GJ_NB + e < n * GJ_NB ? G[(size_t)i0 * GJ_NB + e] : czero<C>();
  if (tid < 32 + GJ_NB) {
    int s = tid < 32 ? i0 + tid : k0 + tid - 32;
    for (int q = nb - 1; q >= 0; --q) {  // the swaps in reverse
      const int p = piv[k0 + q];
      s = s == k0 + q ? p : s == p ? k0 + q : s;
    }
    src[tid] = s;
  }
  __syncthreads();
  if (j >= n) return;
  const bool panel = j >= k0 && j < k0 + nb;
  C b[GJ_NB], v[8];
#pragma unroll
  for (int q = 0; q < GJ_NB; ++q) b[q] = q < nb ? X[(size_t)src[32 + q] * n + j] : czero<C>();
  const int r0 = (tid >> 5) * 8;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + r0 + u;
    v[u] = i < n && !(i >= k0 && i < k0 + nb) ? X[(size_t)src[r0 + u] * n + j] : czero<C>();
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int i = i0 + r0 + u;
    if (i >= n) break;
#pragma unroll
    for (int q = 0; q < GJ_NB; ++q) v[u] = cfma(sG[r0 + u][q], b[q], v[u]);
    Y[(size_t)i * n + j] = panel ? sG[r0 + u][j - k0] : v[u];
  }
}

// Undo the column swaps of the recorded pivots.  Skipped when the elimination stopped early (a barrier ran out or
// a zero pivot), since the pivot record is then incomplete; entries outside [k, n) are ignored.
template <typename C>
__global__ void k_gj_unscramble(C* __restrict__ A, int n, const int* __restrict__ piv, const int* __restrict__ fail,
                                const int* __restrict__ timeout) {
  if (*(volatile const int*)timeout || *(volatile const int*)fail) return;
  for (int k = n - 1; k >= 0; --k) {
    const int p = piv[k];
    if (p != k && p > k && p < n)
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        C t = A[(size_t)i * n + k];
        A[(size_t)i * n + k] = A[(size_t)i * n + p];
        A[(size_t)i * n + p] = t;
      }
    __syncthreads();
  }
}

size_t invert_large_work_bytes(int n) {
  return sizeof(double2) * ((size_t)n * n + (size_t)n * GJ_NB) + (sizeof(double) + sizeof(int)) * 2048 + 64;
}

// By block columns; the one-kernel form (below) where a poll limit of its grid barrier is asked for.
template <typename C>
static void invert_blocked(cudaStream_t st, C* A, int n, int* piv, void* work, int* fail, int* timeout) {
  C* buf[2] = {A, (C*)work};
  C* G = (C*)work + (size_t)n * n;
  const int sm = (int)sizeof(C) * ((n + GJ_CS - 1) / GJ_CS) * GJ_NB;
  ensure_max_smem((const void*)k_gj_panel<C>, 160 * 1024);
  MG_CHECK_ARG(sm <= 160 * 1024, "coarsest level too large for the panel in shared memory");
  int cur = 0;
  for (int k0 = 0; k0 < n; k0 += GJ_NB, cur ^= 1) {
    const int nb = std::min(GJ_NB, n - k0);
    MG_LAUNCH_W(sizeof(C) * 2.0 * n * nb, 8.0 * n * nb * nb, k_gj_panel<C>, GJ_CS, GJ_PT, sm, st, buf[cur], n, k0, nb, G,
                piv, fail);
    MG_LAUNCH_W(sizeof(C) * 2.0 * n * (double)n, 8.0 * n * (double)n * nb, k_gj_update<C>,
                dim3(cdiv(n, 32), cdiv(n, 32)), 128, 0, st, buf[cur], buf[cur ^ 1], n, k0, nb, G, piv);
  }
  if (cur) MG_CUDA(cudaMemcpyAsync(A, buf[1], sizeof(C) * (size_t)n * n, cudaMemcpyDeviceToDevice, st));
  MG_LAUNCH(k_gj_unscramble<C>, 1, 1024, 0, st, A, n, piv, fail, timeout);
}

template <typename C>
void invert_large(cudaStream_t st, C* A, int n, int* piv, void* work, int* fail, int* timeout, long polls) {
  // up to 32 rows one CTA in shared memory, with the same pivots (the launches of the block columns would take longer:
  // 0.2 ms at n = 8); the cooperative kernel only where a poll limit of its barrier is asked for
  if (polls == 0 && n > 32) return invert_blocked<C>(st, A, n, piv, work, fail, timeout);
  if (polls == 0) return invert_small_batched<C>(st, A, 1, n, fail);
  int dev = 0, nsm = 0, per = 0;
  MG_CUDA(cudaGetDevice(&dev));
  MG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const size_t sm = sizeof(C) * (size_t)n;
  ensure_max_smem((const void*)k_gj_coop<C>, 160 * 1024);
  MG_CHECK_ARG(sm <= 160 * 1024, "coarsest level too large for the pivot row in shared memory");
  MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gj_coop<C>, GJ_T, sm));
  // one resident CTA per SM (at most one row per CTA), all co-resident as the cooperative launch requires
  const int grid = std::max(1, std::min(std::min(nsm * std::min(std::max(per, 1), 1), 1024), n));
  char* w = (char*)work;
  C* A1 = (C*)w;
  double* slot_v = (double*)(w + sizeof(double2) * ((size_t)n * n + (size_t)n * GJ_NB));
  int* slot_i = (int*)(slot_v + 2048);
  unsigned* bar = (unsigned*)(slot_i + 2048);
  MG_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st));
  long lim = polls > 0 ? polls : -polls;  // < 0: bounded-wait self-test (one arrival more than the grid has)
  unsigned expect = (unsigned)grid + (polls < 0 ? 1u : 0u);
  void* args[] = {&A, &A1, &n, &piv, &slot_v, &slot_i, &bar, &fail, &timeout, &lim, &expect};
  KTimer* t = g_timer;
  cudaEvent_t ea = nullptr, eb = nullptr;
  const char* name = sizeof(C) == 8 ? "k_gj_coop<float2>" : "k_gj_coop<double2>";
  if (t && t->want(name)) { ea = t->get(); eb = t->get(); MG_CUDA(cudaEventRecord(ea, st)); }
  MG_CUDA(cudaLaunchCooperativeKernel((void*)k_gj_coop<C>, dim3(grid), dim3(GJ_T), args, sm, st));
  if (ea) {
    MG_CUDA(cudaEventRecord(eb, st));
    t->recs.push_back({name, __PRETTY_FUNCTION__, 2.0 * sizeof(C) * n * (double)n * n, 8.0 * n * (double)n * n, ea, eb});
  }
  if (g_launch_counter) ++*g_launch_counter;
  if (n & 1)  // odd column count: the last column wrote the scratch buffer
    MG_CUDA(cudaMemcpyAsync(A, A1, sizeof(C) * (size_t)n * n, cudaMemcpyDeviceToDevice, st));
  MG_LAUNCH(k_gj_unscramble<C>, 1, 1024, 0, st, A, n, piv, fail, timeout);
}
template void invert_large<double2>(cudaStream_t, double2*, int, int*, void*, int*, int*, long);
template void invert_large<float2>(cudaStream_t, float2*, int, int*, void*, int*, int*, long);

// ---- y = A x for the coarsest level (n x n dense, nrhs columns) --------------------------------
// Each result is one sum over j in order (a chain of 2 n dependent FMAs: 4 us at n = 1024), so the parallelism is in
// the results only: blocks of 64 threads with RI rows x NR right-hand sides each, tiles of A and x staged ST chunks of
// 32 columns deep by cp.async (L2 answers in about 1 us).  In FP32 the bytes that shared memory returns come next,
// hence 2 x 2 (32 bytes for 16 FMAs).  FP64: each quarter of an SM has its own share of the two FMAs a clock, so the
// results are spread over as many warps as there are, one a thread, and warps without a right-hand side multiply nothing.
// n = 1024 with 8, 17, 32, 64 rhs: FP32 31, 31, 31, 41 -> 20, 26, 26, 40 us, FP64 273, 273, 275, 521 -> 146, 183, 270, 488
// us (tiles of 16 x 16 results and a barrier every 16 columns before).
template <typename C, int RI, int NR, int ST>
struct DenseTile {
  static constexpr int KC = 32, TI = 8 * RI, TR = 8 * NR;
  static constexpr int AP = TI + 16 / (int)sizeof(C), XP = TR + 16 / (int)sizeof(C);  // padded, rows 16-byte aligned
  C As[ST][KC][AP];  // [column][row]
  C Xs[ST][KC][XP];  // [column][rhs]
};

template <typename C, int RI, int NR, int ST>
__global__ void __launch_bounds__(64) k_dense_apply(const C* __restrict__ A, int n, const C* x,
                                                    C* __restrict__ y, int nrhs, const int* active) {
  pdl_begin();
  typedef DenseTile<C, RI, NR, ST> DT;
  constexpr int KC = DT::KC, TI = DT::TI, TR = DT::TR;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  DT& t = *reinterpret_cast<DT*>(smem_raw);
  const int tid = threadIdx.x, i0 = blockIdx.x * TI, r0 = blockIdx.y * TR;
  const int ti = tid & 7, tr = tid >> 3;
  auto fetch = [&](int c) {  // chunk c into stage c % ST: a warp reads 32 consecutive columns of a row
    const int s = c % ST, j = c * KC + (tid & 31);
    if (j < n) {
#pragma unroll
      for (int q = tid >> 5; q < TI; q += 2)
        if (i0 + q < n) cp_async_elem(&t.As[s][tid & 31][q], A + (size_t)(i0 + q) * n + j);
#pragma unroll
      for (int q = tid >> 5; q < TR; q += 2)
        if (r0 + q < nrhs) cp_async_elem(&t.Xs[s][tid & 31][q], x + (size_t)(r0 + q) * n + j);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  C acc[RI][NR];
#pragma unroll
  for (int a = 0; a < RI; ++a)
#pragma unroll
    for (int b = 0; b < NR; ++b) acc[a][b] = czero<C>();
  const int nch = (n + KC - 1) / KC;
  for (int c = 0; c < ST - 1; ++c) fetch(c);  // chunks past the end fetch nothing
  for (int c = 0; c < nch; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
    __syncthreads();  // chunk c has landed and chunk c - 1 is consumed
    fetch(c + ST - 1);
    const int s = c % ST, cols = min(KC, n - c * KC);
    auto column = [&](int j) {
      C m[RI], v[NR];
#pragma unroll
      for (int a = 0; a < RI; ++a) m[a] = t.As[s][j][ti * RI + a];
#pragma unroll
      for (int b = 0; b < NR; ++b) v[b] = t.Xs[s][j][tr * NR + b];
#pragma unroll
      for (int a = 0; a < RI; ++a)
#pragma unroll
        for (int b = 0; b < NR; ++b) acc[a][b] = cfma(m[a], v[b], acc[a][b]);
    };
    if (sizeof(C) == 16 && r0 + tr * NR >= nrhs) continue;  // no right-hand side: FP64 units are the bound
    if (cols == KC) {
#pragma unroll 8
      for (int j = 0; j < KC; ++j) column(j);
    } else {
      for (int j = 0; j < cols; ++j) column(j);
    }
  }
#pragma unroll
  for (int b = 0; b < NR; ++b) {
    const int r = r0 + tr * NR + b;
    if (r >= nrhs || (active && !active[r])) continue;
#pragma unroll
    for (int a = 0; a < RI; ++a)
      if (i0 + ti * RI + a < n) y[(size_t)r * n + i0 + ti * RI + a] = acc[a][b];
  }
}

template <typename R>
void dense_apply(cudaStream_t st, const typename CT<R>::T* A, int n, const typename CT<R>::T* x,
                 typename CT<R>::T* y, int nrhs, const int* active) {
  typedef typename CT<R>::T C;
  if (nrhs <= 0) return;
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      dense_apply<R>(st, A, n, x + (size_t)r * n, y + (size_t)r * n, k, act);
    }
    return;
  }
  const double bytes = ((double)n * n + 2.0 * act_rhs(nrhs) * n) * sizeof(C), flops = 8.0 * n * (double)n * act_rhs(nrhs);
  auto go = [&](auto ri, auto nr, auto stages) {
    constexpr int RI = decltype(ri)::value, NR = decltype(nr)::value, ST = decltype(stages)::value;
    constexpr int sm = (int)sizeof(DenseTile<C, RI, NR, ST>);
    ensure_max_smem((const void*)k_dense_apply<C, RI, NR, ST>, sm);
    const dim3 grid(cdiv(n, 8 * RI), cdiv(nrhs, 8 * NR));
    // FP64: more CTAs than SMs are launched plainly, because beside the last blocks of the kernel before they come to lie
    // unevenly (V-cycle on level 1 at L = 128, n = 1024, with 16 right-hand sides 1164 us, 778 so)
    const bool early = bytes < PDL_BYTES && (sizeof(R) == 4 || grid.x * grid.y <= (unsigned)sm_count());
    MG_LAUNCH_PE(early, bytes, flops, (k_dense_apply<C, RI, NR, ST>), grid, 64, sm, st, A, n, x, y, nrhs, active);
  };
  typedef std::integral_constant<int, 1> I1;
  typedef std::integral_constant<int, 2> I2;
  if constexpr (sizeof(R) == 8) {
    // six CTAs in an SM with four stages, eight with three: those where they spare a second wave (n = 1024 with 64
    // right-hand sides 533, 488 us)
    const long ctas = (long)cdiv(n, 8) * cdiv(nrhs, 8), nsm = sm_count();
    if (ctas > 6 * nsm && ctas <= 7 * nsm)
      go(I1(), I1(), std::integral_constant<int, 3>());
    else
      go(I1(), I1(), std::integral_constant<int, 4>());
  } else {
    typedef std::integral_constant<int, 8> I8;
    nrhs <= 8 ? go(I2(), I1(), I8()) : go(I2(), I2(), I8());
  }
}
template void dense_apply<float>(cudaStream_t, const float2*, int, const float2*, float2*, int, const int*);
template void dense_apply<double>(cudaStream_t, const double2*, int, const double2*, double2*, int, const int*);

// sum_i w_i A_ii with w_i = 1, or (g5_dof > 0) the gamma5 sign of dof i % g5_dof (-1 in its upper half)
__global__ void k_trace(const double2* __restrict__ A, int n, int g5_dof, double2* out) {
  __shared__ double sr[32], si[32];
  double re = 0, im = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double w = (g5_dof > 0 && i % g5_dof >= g5_dof / 2) ? -1.0 : 1.0;
    re += w * A[(size_t)i * n + i].x;
    im += w * A[(size_t)i * n + i].y;
  }
  re = warp_sum(re);
  im = warp_sum(im);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sr[w] = re; si[w] = im; }
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    re = l < nw ? sr[l] : 0;
    im = l < nw ? si[l] : 0;
    re = warp_sum(re);
    im = warp_sum(im);
    if (l == 0) *out = make_double2(re, im);
  }
}
void trace_dense(cudaStream_t st, const double2* A, int n, double2* out, int g5_dof) {
  MG_LAUNCH(k_trace, 1, 1024, 0, st, A, n, g5_dof, out);
}

// ---- CholeskyQR2 pieces ---------------------------------------------------------------------------
namespace {
constexpr int GCH = 32;     // rows per shared-memory chunk
constexpr int GBLK = 128;   // blocks (partials)
}

size_t gram_work_bytes(int d, long n) {
  (void)n;
  return sizeof(double2) * (size_t)GBLK * d * d;
}

// G is Hermitian: the upper-triangle entries (i, j), i <= j, are packed in order (t = 0 .. d(d+1)/2 - 1) and
// thread tid accumulates entries tid, tid + blockDim.x, ... (at most GACC of them), writing each and its
// conjugate mirror.
constexpr int GACC = (SK_MAXD * (SK_MAXD + 1) / 2 + 1023) / 1024;
__global__ void __launch_bounds__(1024) k_gram_part(const double2* __restrict__ Y, int d, long n,
                                                    double2* __restrict__ part) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* Ys = reinterpret_cast<double2*>(smem_raw);  // [GCH][d]
  const int tid = threadIdx.x, ntri = d * (d + 1) / 2;
  int ii[GACC], jj[GACC];
#pragma unroll
  for (int u = 0; u < GACC; ++u) {
    int t = tid + u * (int)blockDim.x, i = 0;
    if (t >= ntri) { ii[u] = -1; jj[u] = 0; continue; }
    while (t >= d - i) { t -= d - i; ++i; }
    ii[u] = i;
    jj[u] = i + t;
  }
  double2 acc[GACC];
#pragma unroll
  for (int u = 0; u < GACC; ++u) acc[u] = make_double2(0, 0);
  for (long e0 = (long)blockIdx.x * GCH; e0 < n; e0 += (long)gridDim.x * GCH) {
    __syncthreads();
    for (int q = tid; q < GCH * d; q += blockDim.x) {
      const int c = q / GCH, e = q % GCH;
      Ys[e * d + c] = (e0 + e < n) ? Y[(size_t)c * n + e0 + e] : make_double2(0, 0);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < GACC; ++u)
      if (ii[u] >= 0)
#pragma unroll 8
        for (int e = 0; e < GCH; ++e) acc[u] = cfmac(Ys[e * d + ii[u]], Ys[e * d + jj[u]], acc[u]);
  }
#pragma unroll
  for (int u = 0; u < GACC; ++u) {
    if (ii[u] < 0) continue;
    const int i = ii[u], j = jj[u];
    part[((size_t)blockIdx.x * d + i) * d + j] = acc[u];
    if (i != j) part[((size_t)blockIdx.x * d + j) * d + i] = cconj(acc[u]);
  }
}

__global__ void k_gram_final(const double2* __restrict__ part, int d, int nb, double2* __restrict__ G) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= d * d) return;
  double2 s = make_double2(0, 0);
  for (int b = 0; b < nb; ++b) s = cadd(s, part[(size_t)b * d * d + e]);
  G[e] = s;
}

void gram(cudaStream_t st, const double2* Y, int d, long n, double2* G, void* work) {
  MG_CHECK_ARG(d >= 1 && d <= SK_MAXD, "sketch size d limited to 64");
  const int nb = (int)std::min<long>(GBLK, cdiv(n, GCH));
  double2* part = reinterpret_cast<double2*>(work);
  MG_LAUNCH(k_gram_part, nb, 1024, sizeof(double2) * GCH * d, st, Y, d, n, part);
  MG_LAUNCH(k_gram_final, cdiv(d * d, 256), 256, 0, st, part, d, nb, G);
}

// G = R^H R (R upper, real positive diagonal), Rinv = R^{-1}; both in dynamic shared memory.  One CTA; what it costs is
// the latency of dependent FP64 operations, so the factorisation updates the whole trailing matrix after each row
// (one dependent product per step instead of a sum over the rows before it), one thread forms a row's root and
// reciprocal, and the inverse is formed row by row from the bottom, four threads to a sum.  d = 32: 258 -> 106 us.
// Every entry of R takes its subtractions and roundings in the order of a sum over the rows before it: a rank-deficient
// Gram matrix is found by a pivot that rounds to zero or below.
__global__ void __launch_bounds__(256) k_chol_inv(const double2* __restrict__ Gg, int d, double2* __restrict__ Rinv,
                                                  int* fail) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* R = reinterpret_cast<double2*>(smem_raw);
  double2* X = R + d * d;
  __shared__ double rd[SK_MAXD];  // reciprocals of the diagonal of R
  __shared__ int bad;
  const int tid = threadIdx.x;
  for (int e = tid; e < d * d; e += 256) { R[e] = Gg[e]; X[e] = make_double2(0, 0); }
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int k = 0; k < d; ++k) {
    if (tid == 0) {
      const double s = R[k * d + k].x;
      if (!(s > 0.0)) bad = 1;
      const double root = sqrt(fmax(s, 1e-300));
      R[k * d + k] = make_double2(root, 0);
      rd[k] = 1.0 / root;
    }
    __syncthreads();
    const double inv = rd[k];
    for (int j = k + 1 + tid; j < d; j += 256) R[k * d + j] = cscale(R[k * d + j], inv);
    __syncthreads();
    const int m = d - k - 1;  // trailing rows i <= columns j
    for (int e = tid; e < m * m; e += 256) {
      const int i = k + 1 + e / m, j = k + 1 + e % m;
      if (j == i)
        R[i * d + i].x -= cabs2(R[k * d + i]);
      else if (j > i)
        R[i * d + j] = csub(R[i * d + j], cmulc(R[k * d + i], R[k * d + j]));
    }
    __syncthreads();
  }
  const int j = tid >> 2, part = tid & 3;
  for (int i = d - 1; i >= 0; --i) {  // X_ij = (delta_ij - sum_{i < m <= j} R_im X_mj) / R_ii
    double2 s = make_double2(0, 0);
    if (j < d)
      for (int m = i + 1 + part; m <= j; m += 4) s = cfma(R[i * d + m], X[m * d + j], s);
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      s.x += __shfl_xor_sync(0xffffffff, s.x, o);
      s.y += __shfl_xor_sync(0xffffffff, s.y, o);
    }
    if (part == 0 && j < d && j >= i) X[i * d + j] = j == i ? make_double2(rd[i], 0) : cscale(s, -rd[i]);
    __syncwarp();  // row i of column j is read by the same four threads only
  }
  __syncthreads();
  for (int e = tid; e < d * d; e += 256) Rinv[e] = X[e];
  if (tid == 0 && bad) atomicExch(fail, 1);
}

void chol_inv_upper(cudaStream_t st, const double2* G, int d, double2* Rinv, int* fail) {
  MG_CHECK_ARG(d >= 1 && d <= SK_MAXD, "sketch size d limited to 64");
  const int sm = (int)sizeof(double2) * 2 * d * d;
  ensure_max_smem((const void*)k_chol_inv, sizeof(double2) * 2 * SK_MAXD * SK_MAXD);
  MG_LAUNCH(k_chol_inv, 1, 256, sm, st, G, d, Rinv, fail);
}

// Y <- Y Rinv for Y = [d][n]: a block takes RMT consecutive elements e of all d vectors into shared memory and
// each thread forms new_j(e) = sum_{i <= j} Y_i(e) Rinv_ij for several (e, j)
constexpr int RMT = 32;
__global__ void __launch_bounds__(256) k_right_mul_upper(double2* __restrict__ Y, int d, long n,
                                                         const double2* __restrict__ Rinv) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* Rs = reinterpret_cast<double2*>(smem_raw);  // [d][d]
  double2* Ys = Rs + d * d;                             // [RMT][d + 1]
  for (int e = threadIdx.x; e < d * d; e += blockDim.x) Rs[e] = Rinv[e];
  for (long e0 = (long)blockIdx.x * RMT; e0 < n; e0 += (long)gridDim.x * RMT) {
    __syncthreads();
    for (int q = threadIdx.x; q < RMT * d; q += blockDim.x) {
      const int i = q / RMT, e = q % RMT;
      Ys[e * (d + 1) + i] = (e0 + e < n) ? Y[(size_t)i * n + e0 + e] : make_double2(0, 0);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < RMT * d; q += blockDim.x) {
      const int j = q / RMT, e = q % RMT;
      if (e0 + e >= n) continue;
      double2 acc = make_double2(0, 0);
      for (int i = 0; i <= j; ++i) acc = cfma(Ys[e * (d + 1) + i], Rs[i * d + j], acc);
      Y[(size_t)j * n + e0 + e] = acc;
    }
  }
}

void right_mul_upper(cudaStream_t st, double2* Y, int d, long n, const double2* Rinv) {
  MG_CHECK_ARG(d >= 1 && d <= SK_MAXD, "sketch size d limited to 64");
  const size_t sm = sizeof(double2) * ((size_t)d * d + (size_t)RMT * (d + 1));
  ensure_max_smem((const void*)k_right_mul_upper,
                  (int)(sizeof(double2) * ((size_t)SK_MAXD * SK_MAXD + (size_t)RMT * (SK_MAXD + 1))));
  MG_LAUNCH(k_right_mul_upper, std::min<long>(cdiv(n, RMT), 2048), 256, sm, st, Y, d, n, Rinv);
}

// ---- projection coefficients c[i][r] = Q_i^H x_r -----------------------------------------------------
namespace {
constexpr int PCH = 32;    // rows per chunk
constexpr int PBLK = 96;   // chunks (partials) at most
}

size_t proj_work_bytes(int d, long n, int nrhs) {
  (void)n;
  return sizeof(double2) * (size_t)PBLK * d * nrhs * 2;
}

// Bound by the FP64 units: TI basis vectors x 256 / TI columns per CTA, one result per thread (every lane at work
// whatever d is), chunks of the rows over blockIdx.y.  Columns 0 .. nrhs-1 are x, nrhs .. those of x2 (if any), so
// that one pass over Q serves both vectors of a projected sample.  Lanes bound to basis vectors i and i + 32 idled where
// d is small: d = 16, 24 right-hand sides, n = 131072: 2 x 786 -> 356 us (1.1 TF of FP64, its roof).
template <int TI>
__global__ void __launch_bounds__(256) k_proj_part(const double2* __restrict__ Q, int d, const double2* __restrict__ x,
                                                   const double2* __restrict__ x2, long n, int nrhs, int ncol,
                                                   double2* __restrict__ part) {
  constexpr int TR = 256 / TI;
  __shared__ double2 Qs[PCH][TI + 1];
  __shared__ double2 Xs[PCH][TR + 1];
  const int tid = threadIdx.x, ti = (d + TI - 1) / TI;
  const int i0 = (blockIdx.x % ti) * TI, r0 = (blockIdx.x / ti) * TR;
  const int i = tid % TI, g = tid / TI;
  double2 acc = make_double2(0, 0);
  for (long e0 = (long)blockIdx.y * PCH; e0 < n; e0 += (long)gridDim.y * PCH) {
    __syncthreads();
    const int e = tid & 31;
#pragma unroll
    for (int c = tid >> 5; c < TI; c += 8)
      Qs[e][c] = i0 + c < d && e0 + e < n ? Q[(size_t)(i0 + c) * n + e0 + e] : make_double2(0, 0);
#pragma unroll
    for (int c = tid >> 5; c < TR; c += 8) {
      const int r = r0 + c;
      const double2* v = r < nrhs ? x + (size_t)r * n : x2 + (size_t)(r - nrhs) * n;
      Xs[e][c] = r < ncol && e0 + e < n ? v[e0 + e] : make_double2(0, 0);
    }
    __syncthreads();
#pragma unroll 8
    for (int q = 0; q < PCH; ++q) acc = cfmac(Qs[q][i], Xs[q][g], acc);
  }
  if (i0 + i < d && r0 + g < ncol) part[((size_t)blockIdx.y * ncol + r0 + g) * d + i0 + i] = acc;
}

// c[(s d + i) nrhs + r], s = 0 for x and 1 for x2: sums over the chunks in order
__global__ void k_proj_final(const double2* __restrict__ part, int d, int nrhs, int ncol, int nb,
                             double2* __restrict__ c) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= d * ncol) return;
  double2 s = make_double2(0, 0);
  for (int b = 0; b < nb; ++b) s = cadd(s, part[(size_t)b * d * ncol + e]);
  const int col = e / d, i = e - col * d;
  c[(size_t)((col < nrhs ? 0 : d) + i) * nrhs + col % nrhs] = s;
}

void proj_coeffs(cudaStream_t st, const double2* Q, int d, const double2* x, const double2* x2, long n, int nrhs,
                 double2* c, void* work) {
  MG_CHECK_ARG(d >= 1 && d <= SK_MAXD, "sketch size d limited to 64");
  const int ncol = x2 ? 2 * nrhs : nrhs;
  double2* part = reinterpret_cast<double2*>(work);
  auto tiles = [&](int ti) { return cdiv(d, ti) * cdiv(ncol, 256 / ti); };
  // the tile shape that pads least; as many chunks as there are partials, whatever the tiles (chunks for six CTAs per SM
  // made the chains of sums longer, down to one of all rows, and 3 to 9 % slower: n = 32768, d = 64, 1024 right-hand
  // sides 31.5 -> 30.1 ms)
  const int ti = tiles(8) < tiles(16) ? 8 : tiles(16) <= tiles(32) ? 16 : 32;
  const int nb = (int)std::min<long>(PBLK, cdiv(n, PCH));
  const dim3 grid(tiles(ti), nb);
  const double flops = 8.0 * d * ncol * (double)n, bytes = 16.0 * (double)n * (d + ncol);
  if (ti == 8)
    MG_LAUNCH_W(bytes, flops, k_proj_part<8>, grid, 256, 0, st, Q, d, x, x2, n, nrhs, ncol, part);
  else if (ti == 16)
    MG_LAUNCH_W(bytes, flops, k_proj_part<16>, grid, 256, 0, st, Q, d, x, x2, n, nrhs, ncol, part);
  else
    MG_LAUNCH_W(bytes, flops, k_proj_part<32>, grid, 256, 0, st, Q, d, x, x2, n, nrhs, ncol, part);
  MG_LAUNCH(k_proj_final, cdiv((long)d * ncol, 128), 128, 0, st, part, d, nrhs, ncol, nb, c);
}

}  // namespace mg
