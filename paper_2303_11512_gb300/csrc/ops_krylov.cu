// The orthogonalisation step of the batched FGMRES: classical Gram-Schmidt with one re-orthogonalisation of
// w = D z_j against the basis V_0 .. V_j, the norm, the Givens update of the Hessenberg column and the next basis
// vector, per right-hand side:
//   h1 = V^H w,  w' = w - V h1,  h2 = V^H w',  hn^2 = |w'|^2 - |h2|^2,  v_{j+1} = (w' - V h2) / hn.
// hn is |w' - V h2| by Pythagoras: h2 is of the order of the rounding of h1, so nothing cancels while w' is much larger
// than that.  When w lies in the span of the basis up to rounding, w' is rounding itself and may lie in the span too: from
// |h2|^2 > |w'|^2 / 4 on the Krylov space counts as spent, the right-hand side's cycle ends with this column and the true
// residual decides (the difference could be 0 or of either sign, and v_{j+1} would be rounding of any length).
//
// Two forms.  Long vectors: three passes over V, each one launch; the block that finishes last for a right-hand
// side adds the partial sums in a fixed order (bitwise repeatable) and, after the second pass, does the Givens
// update, so no launches for finalising, scaling or the Hessenberg column remain (10 launches a step before).
// Short vectors (KRY_SMALL entries at most): one launch for the whole step, a thread-block cluster per right-hand
// side with w in registers; partial sums meet in distributed shared memory.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "ops.cuh"

namespace mg {
namespace {

template <typename C> struct RealOf;
template <> struct RealOf<float2> { typedef float R; };
template <> struct RealOf<double2> { typedef double R; };

constexpr int KT = 256;           // threads per block
constexpr int KRY_BLK = 64;       // blocks per right-hand side at most
constexpr long KRY_SMALL = 16384;  // entries of a vector that the one-launch form takes

// Transposed warp reduction: NV values per lane (NV a power of two <= 32); lane l returns the warp total of value
// l >> log2(32 / NV).
template <int NV>
__device__ __forceinline__ double warp_totals(double (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int half = NV / 2; half >= 1; half >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < half; ++q) {
      const double send = up ? v[q] : v[q + half];
      const double keep = up ? v[q + half] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffff, send, o);
    }
  }
  double r = v[0];
  for (; o; o >>= 1) r += __shfl_xor_sync(0xffffffff, r, o);
  return r;
}
constexpr int log2_of(int v) { return v <= 1 ? 0 : 1 + log2_of(v / 2); }
__device__ __forceinline__ double warp_sum1(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffff, v, o);
  return v;
}

// Column of the Hessenberg matrix under its Givens update, and the earlier rotations, in shared memory: the rotations
// are a serial chain of one thread, which from global memory would wait for two loads in each.
struct Givens {
  double2 col[65], s[64];
  double c[64];
};
// rotations before column j of rhs r, by the lanes of a warp (or all threads of a block, stride nt)
__device__ __forceinline__ void givens_load(const KryGm& g, int j, int r, Givens& v, int t, int nt) {
  for (int i = t; i < j; i += nt) {
    v.c[i] = g.cs[(size_t)i * g.nrhs + r];
    v.s[i] = g.sn[(size_t)i * g.nrhs + r];
  }
}
__device__ __forceinline__ bool kry_spent(double w2, double h22) { return 4 * h22 > w2; }
// Givens update of column j for right-hand side r by one thread; v.col: h1 + h2 (j + 1 entries, overwritten); hn2 =
// |w' - V h2|^2 (negative by rounding counts as 0); spent: see above, the right-hand side's cycle ends here.  FP64 latency is what it costs: reciprocal square roots in place
// of square roots and divisions, and the stop test on squares.
__device__ void givens_column(const KryGm& g, int j, int r, Givens& v, double hn2, bool spent) {
  const int nrhs = g.nrhs, m = g.m;
  double2* col = v.col;
  double2 a = col[0];
  for (int i = 0; i < j; ++i) {  // a: entry i after the rotations before it
    const double c = v.c[i];
    const double2 s = v.s[i], b = col[i + 1];
    col[i] = cadd(cscale(a, c), cmul(s, b));
    a = csub(cscale(b, c), cmulc(s, a));
  }
  if (!(hn2 > 0.0) && hn2 == hn2) hn2 = 0.0;
  // new rotation zeroing the real entry hh = sqrt(hn2) below the diagonal
  const double hh = hn2 > 0.0 ? hn2 * rsqrt(hn2) : hn2, na2 = a.x * a.x + a.y * a.y;
  double c;
  double2 s, rr;
  if (na2 == 0.0) {
    c = 0.0; s = make_double2(1, 0); rr = make_double2(hh, 0);
  } else {
    const double t2 = na2 + hn2, rt = rsqrt(t2), rn = rsqrt(na2);
    const double2 ph = cscale(a, rn);
    c = na2 * rn * rt;
    s = cscale(ph, hh * rt);
    rr = cscale(ph, t2 * rt);
  }
  g.cs[(size_t)j * nrhs + r] = c;
  g.sn[(size_t)j * nrhs + r] = s;
  for (int i = 0; i < j; ++i) g.H[((size_t)i * m + j) * nrhs + r] = col[i];
  g.H[((size_t)j * m + j) * nrhs + r] = rr;
  const double2 gj = g.g[(size_t)j * nrhs + r];
  const double2 gn = cneg(cmulc(s, gj));
  g.g[(size_t)(j + 1) * nrhs + r] = gn;
  g.g[(size_t)j * nrhs + r] = cscale(gj, c);
  const double res2 = gn.x * gn.x + gn.y * gn.y, goal = g.tol * g.bnorm[r];
  const int it = g.its[r] + 1;
  g.its[r] = it;
  g.kvec[r] = j + 1;
  g.hn[r] = hh;
  if (res2 <= goal * goal || it >= g.maxit || hh == 0.0 || spent || j + 1 == m || !(res2 == res2))
    g.iact[r] = 0;
  else
    atomicAdd(g.count + j, 1);
}

// ---- long vectors -----------------------------------------------------------------------------------------------
// Elements as vectors of VE complex numbers (16 bytes): two in FP32, one in FP64.
template <typename C> struct Vec;
template <> struct Vec<float2> { typedef float4 T; static constexpr int VE = 2; };
template <> struct Vec<double2> { typedef double2 T; static constexpr int VE = 1; };
__device__ __forceinline__ void split(const float4& v, float2* c) {
  c[0] = make_float2(v.x, v.y);
  c[1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ void split(const double2& v, double2* c) { c[0] = v; }
__device__ __forceinline__ float4 join(const float2* c) { return make_float4(c[0].x, c[0].y, c[1].x, c[1].y); }
__device__ __forceinline__ double2 join(const double2* c) { return c[0]; }

// Block totals of 2 KM + 1 values (KM complex dots, one norm) into part[(i * nrhs + rhs) * nblk + block]; the norm
// goes to slot KM_total.  Returns true in the block that finished last for this rhs (every thread).
template <int KM>
__device__ bool store_partials(double (&v)[2 * KM], double nrm, bool with_norm, int k, double2* part, int nrhs, int rhs,
                               unsigned* done) {
  __shared__ double sh[KT / 32][2 * KM + 1];
  __shared__ bool s_last;
  constexpr int NV = 2 * KM <= 2 ? 2 : 2 * KM <= 4 ? 4 : 2 * KM <= 8 ? 8 : 2 * KM <= 16 ? 16 : 32;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  constexpr int S = 5 - log2_of(NV);
  double u[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) u[q] = q < 2 * KM ? v[q < 2 * KM ? q : 0] : 0.0;
  const double t = warp_totals<NV>(u);
  if ((l & ((1 << S) - 1)) == 0 && (l >> S) < 2 * KM) sh[w][l >> S] = t;
  if (with_norm) {
    const double tn = warp_sum1(nrm);
    if (l == 0) sh[w][2 * KM] = tn;
  }
  __syncthreads();
  const int nblk = gridDim.x, tid = threadIdx.x;
  if (tid < 2 * k || (tid == 2 * KM && with_norm)) {
    double t2 = 0;
#pragma unroll
    for (int q = 0; q < KT / 32; ++q) t2 += sh[q][tid];
    const int i = tid == 2 * KM ? k : tid >> 1, c = tid == 2 * KM ? 0 : tid & 1;
    reinterpret_cast<double*>(part + ((size_t)i * nrhs + rhs) * nblk + blockIdx.x)[c] = t2;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicInc(done + rhs, nblk - 1) == (unsigned)nblk - 1;  // wraps to 0 for the next pass
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// sums of the partials of slots 0 .. cnt-1 for rhs into out[], a warp per slot
__device__ __forceinline__ void sum_partials(const double2* part, int cnt, int nrhs, int rhs, int nblk, double2* out) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int i = w; i < cnt; i += KT / 32) {
    const double2* p = part + ((size_t)i * nrhs + rhs) * nblk;
    double re = 0, im = 0;
    for (int b = l; b < nblk; b += 32) {
      const double2 v = __ldcg(p + b);
      re += v.x;
      im += v.y;
    }
    re = warp_sum1(re);
    im = warp_sum1(im);
    if (l == 0) out[i] = make_double2(re, im);
  }
}

// h[i * nrhs + rhs] = V_i^H w, i < k
template <typename C, int KM>
__global__ void __launch_bounds__(KT) k_kry_dot(const C* __restrict__ V, long vstride, int k, const C* __restrict__ w,
                                                long n, double2* __restrict__ h, double2* part, unsigned* done,
                                                const int* __restrict__ active) {
  typedef typename RealOf<C>::R R;
  typedef typename Vec<C>::T VT;
  constexpr int VE = Vec<C>::VE;
  const int rhs = blockIdx.y, nrhs = gridDim.y;
  if (active && !active[rhs]) return;  // the whole rhs: no block of it counts itself
  R dr[KM], di[KM];
#pragma unroll
  for (int q = 0; q < KM; ++q) dr[q] = di[q] = 0;
  const VT* W = reinterpret_cast<const VT*>(w + (size_t)rhs * n);
  const C* Vr = V + (size_t)rhs * n;
  const long nv = n / VE;
  for (long e = blockIdx.x * (long)KT + threadIdx.x; e < nv; e += (long)gridDim.x * KT) {
    C b[VE];
    split(W[e], b);
    VT av[KM];
#pragma unroll
    for (int q = 0; q < KM; ++q)
      if (q < k) av[q] = reinterpret_cast<const VT*>(Vr + (size_t)q * vstride)[e];
#pragma unroll
    for (int q = 0; q < KM; ++q)
      if (q < k) {
        C a[VE];
        split(av[q], a);
#pragma unroll
        for (int u = 0; u < VE; ++u) {
          dr[q] = fma(a[u].x, b[u].x, fma(a[u].y, b[u].y, dr[q]));
          di[q] = fma(a[u].x, b[u].y, fma(-a[u].y, b[u].x, di[q]));
        }
      }
  }
  double v[2 * KM];
#pragma unroll
  for (int q = 0; q < KM; ++q) { v[2 * q] = dr[q]; v[2 * q + 1] = di[q]; }
  if (!store_partials<KM>(v, 0.0, false, k, part, nrhs, rhs, done)) return;
  __shared__ double2 tot[KM];
  sum_partials(part, k, nrhs, rhs, gridDim.x, tot);
  __syncthreads();
  if ((int)threadIdx.x < k) h[(size_t)threadIdx.x * nrhs + rhs] = tot[threadIdx.x];
}

// w -= V h1, h2 = V^H w, hn and the Givens update (last block)
template <typename C, int KM>
__global__ void __launch_bounds__(KT, sizeof(C) == 16 && KM > 8 ? 2 : 1)
    k_kry_update_dot(const C* __restrict__ V, long vstride, int k, C* __restrict__ w, long n, KryGm gm, double2* part,
                     unsigned* done) {
  typedef typename RealOf<C>::R R;
  typedef typename Vec<C>::T VT;
  constexpr int VE = Vec<C>::VE;
  __shared__ C hs[KM];
  const int rhs = blockIdx.y, nrhs = gridDim.y;
  if (!gm.iact[rhs]) return;
  if ((int)threadIdx.x < k) {
    const double2 v = gm.h1[(size_t)threadIdx.x * nrhs + rhs];
    hs[threadIdx.x] = cmake((R)v.x, (R)v.y);
  }
  __syncthreads();
  R dr[KM], di[KM], nr = 0;
#pragma unroll
  for (int q = 0; q < KM; ++q) dr[q] = di[q] = 0;
  VT* W = reinterpret_cast<VT*>(w + (size_t)rhs * n);
  const C* Vr = V + (size_t)rhs * n;
  const long nv = n / VE;
  for (long e = blockIdx.x * (long)KT + threadIdx.x; e < nv; e += (long)gridDim.x * KT) {
    VT av[KM];
    const VT wv = W[e];
#pragma unroll
    for (int q = 0; q < KM; ++q)
      if (q < k) av[q] = reinterpret_cast<const VT*>(Vr + (size_t)q * vstride)[e];
    C acc[VE], x[VE];
#pragma unroll
    for (int u = 0; u < VE; ++u) acc[u] = czero<C>();
#pragma unroll
    for (int q = 0; q < KM; ++q)
      if (q < k) {
        C a[VE];
        split(av[q], a);
#pragma unroll
        for (int u = 0; u < VE; ++u) acc[u] = cfma(hs[q], a[u], acc[u]);
      }
    split(wv, x);
#pragma unroll
    for (int u = 0; u < VE; ++u) {
      x[u] = csub(x[u], acc[u]);
      nr = fma(x[u].x, x[u].x, fma(x[u].y, x[u].y, nr));
    }
    W[e] = join(x);
#pragma unroll
    for (int q = 0; q < KM; ++q)
      if (q < k) {
        C a[VE];
        split(av[q], a);
#pragma unroll
        for (int u = 0; u < VE; ++u) {
          dr[q] = fma(a[u].x, x[u].x, fma(a[u].y, x[u].y, dr[q]));
          di[q] = fma(a[u].x, x[u].y, fma(-a[u].y, x[u].x, di[q]));
        }
      }
  }
  double v[2 * KM];
#pragma unroll
  for (int q = 0; q < KM; ++q) { v[2 * q] = dr[q]; v[2 * q + 1] = di[q]; }
  if (!store_partials<KM>(v, (double)nr, true, k, part, nrhs, rhs, done)) return;
  __shared__ double2 tot[KM + 1];
  __shared__ Givens gv;
  sum_partials(part, k + 1, nrhs, rhs, gridDim.x, tot);
  givens_load(gm, k - 1, rhs, gv, threadIdx.x, KT);
  __syncthreads();
  if ((int)threadIdx.x < k) {
    gm.h2[(size_t)threadIdx.x * nrhs + rhs] = tot[threadIdx.x];
    gv.col[threadIdx.x] = cadd(gm.h1[(size_t)threadIdx.x * nrhs + rhs], tot[threadIdx.x]);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double hn2 = tot[k].x, h22 = 0;
    for (int i = 0; i < k; ++i) {
      const double q = tot[i].x * tot[i].x + tot[i].y * tot[i].y;
      hn2 -= q;
      h22 += q;
    }
    givens_column(gm, k - 1, rhs, gv, hn2, kry_spent(tot[k].x, h22));
  }
}

// v = (w - V h2) / hn, in place of w; any k (the basis in steps of KM)
template <typename C, int KM>
__global__ void __launch_bounds__(KT) k_kry_update_scale(const C* __restrict__ V, long vstride, int k,
                                                         C* __restrict__ w, long n, KryGm gm) {
  typedef typename RealOf<C>::R R;
  typedef typename Vec<C>::T VT;
  constexpr int VE = Vec<C>::VE;
  __shared__ C hs[64];
  const int rhs = blockIdx.y, nrhs = gridDim.y;
  if (!gm.iact[rhs]) return;
  for (int i = threadIdx.x; i < k; i += KT) {
    const double2 v = gm.h2[(size_t)i * nrhs + rhs];
    hs[i] = cmake((R)v.x, (R)v.y);
  }
  const R f = (R)(1.0 / gm.hn[rhs]);
  __syncthreads();
  VT* W = reinterpret_cast<VT*>(w + (size_t)rhs * n);
  const C* Vr = V + (size_t)rhs * n;
  const long nv = n / VE;
  for (long e = blockIdx.x * (long)KT + threadIdx.x; e < nv; e += (long)gridDim.x * KT) {
    C acc[VE], x[VE];
    const VT wv = W[e];
#pragma unroll
    for (int u = 0; u < VE; ++u) acc[u] = czero<C>();
    for (int i0 = 0; i0 < k; i0 += KM) {
      VT av[KM];
#pragma unroll
      for (int q = 0; q < KM; ++q)
        if (i0 + q < k) av[q] = reinterpret_cast<const VT*>(Vr + (size_t)(i0 + q) * vstride)[e];
#pragma unroll
      for (int q = 0; q < KM; ++q)
        if (i0 + q < k) {
          C a[VE];
          split(av[q], a);
#pragma unroll
          for (int u = 0; u < VE; ++u) acc[u] = cfma(hs[i0 + q], a[u], acc[u]);
        }
    }
    split(wv, x);
#pragma unroll
    for (int u = 0; u < VE; ++u) x[u] = cscale(csub(x[u], acc[u]), f);
    W[e] = join(x);
  }
}

// after more than 16 basis vectors the second pass is an update and separate dot products: their Givens update
__global__ void __launch_bounds__(32) k_kry_givens(KryGm gm, int k) {
  __shared__ Givens gv;
  const int r = blockIdx.x, l = threadIdx.x;
  if (!gm.iact[r]) return;
  givens_load(gm, k - 1, r, gv, l, 32);
  double h2n = 0;
  for (int i = l; i < k; i += 32) {
    const double2 b = gm.h2[(size_t)i * gm.nrhs + r];
    gv.col[i] = cadd(gm.h1[(size_t)i * gm.nrhs + r], b);
    h2n += b.x * b.x + b.y * b.y;
  }
  h2n = warp_sum1(h2n);
  __syncwarp();
  if (l == 0) {
    givens_column(gm, k - 1, r, gv, gm.wn2[r] - h2n, kry_spent(gm.wn2[r], h2n));
  }
}

// back substitution of the k x k triangle of every right-hand side (k = kvec, 0 where cact is 0), one warp each:
// y_i = g_i / H_ii, then g -= H_.i y_i on the rows above; y_i = 0 for i >= k
__global__ void __launch_bounds__(32) k_kry_trisolve(KryGm gm, const int* __restrict__ cact, double2* __restrict__ y) {
  const int r = blockIdx.x, l = threadIdx.x, m = gm.m, nrhs = gm.nrhs;
  const int k = cact[r] ? gm.kvec[r] : 0;
  double2 a[2];  // rows l and l + 32 of the right-hand side
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    a[q] = l + 32 * q < k ? gm.g[(size_t)(l + 32 * q) * nrhs + r] : make_double2(0, 0);
    if (l + 32 * q >= k && l + 32 * q < m) y[(size_t)(l + 32 * q) * nrhs + r] = make_double2(0, 0);
  }
  double2 di[2];  // reciprocal of the diagonal entries of this lane's rows (0 for a zero entry)
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = l + 32 * q;
    di[q] = make_double2(0, 0);
    if (i < k) {
      const double2 d = gm.H[((size_t)i * m + i) * nrhs + r];
      const double dn = d.x * d.x + d.y * d.y;
      if (dn > 0) di[q] = cscale(cconj(d), 1.0 / dn);
    }
  }
  double2 h[2], hn[2];  // column i, the next column fetched ahead
  auto column = [&](int i, double2* c) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
      c[q] = i >= 0 && l + 32 * q <= i ? gm.H[((size_t)(l + 32 * q) * m + i) * nrhs + r] : make_double2(0, 0);
  };
  column(k - 1, h);
  for (int i = k - 1; i >= 0; --i) {
    column(i - 1, hn);
    double2 yi = make_double2(0, 0);
    if (l == (i & 31)) {
      yi = cmul(i < 32 ? di[0] : di[1], i < 32 ? a[0] : a[1]);
      y[(size_t)i * nrhs + r] = yi;
    }
    yi.x = __shfl_sync(0xffffffff, yi.x, i & 31);
    yi.y = __shfl_sync(0xffffffff, yi.y, i & 31);
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (l + 32 * q < i) a[q] = csub(a[q], cmul(h[q], yi));
    h[0] = hn[0];
    h[1] = hn[1];
  }
}

// ---- short vectors ----------------------------------------------------------------------------------------------
// One cluster of CS blocks per right-hand side; element e = q CS T + rank T + tid (q < E) of w stays in a register
// through the step, V is re-read (its second and third reading hit L1).  In FP64 the two FMAs a clock of each SM
// bound it (16 FMAs per element and basis vector), hence clusters: 32 right-hand sides of 512 entries occupy 128 SMs.
template <typename C, int E, int T>
__global__ void __launch_bounds__(T) k_kry_small(const C* __restrict__ V, long vstride, int k, C* __restrict__ w, int n,
                                                 KryGm gm) {
  typedef typename RealOf<C>::R R;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = cl.num_blocks(), rank = cl.block_rank();
  constexpr int NW = T / 32, CH = E <= 2 ? 8 : 4;  // basis vectors at a time (their loads in flight together)
  __shared__ double wp[NW][2 * 64 + 1];
  __shared__ double hp1[2 * 64], hp2[2 * 64 + 1];
  __shared__ double2 h1[64], h2[65];
  __shared__ Givens gv;
  const int rhs = blockIdx.x / cs, nrhs = gm.nrhs;
  if (!gm.iact[rhs]) return;  // the whole cluster
  const int tid = threadIdx.x, wi = tid >> 5, l = tid & 31;
  C* W = w + (size_t)rhs * n;
  const C* Vr = V + (size_t)rhs * n;
  const int e0 = rank * T + tid, step = cs * T;
  C x[E];
#pragma unroll
  for (int q = 0; q < E; ++q) x[q] = e0 + q * step < n ? W[e0 + q * step] : czero<C>();
  auto fetch = [&](int i0, C (&a)[CH][E]) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const C* Vi = Vr + (size_t)(i0 + c) * vstride;
#pragma unroll
      for (int q = 0; q < E; ++q)
        a[c][q] = i0 + c < k && e0 + q * step < n ? Vi[e0 + q * step] : czero<C>();
    }
  };
  auto dots = [&]() {  // warp totals of V_i^H x into wp
    for (int i0 = 0; i0 < k; i0 += CH) {
      C a[CH][E];
      fetch(i0, a);
      double v[2 * CH];
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        R dr = 0, di = 0;
#pragma unroll
        for (int q = 0; q < E; ++q) {
          dr = fma(a[c][q].x, x[q].x, fma(a[c][q].y, x[q].y, dr));
          di = fma(a[c][q].x, x[q].y, fma(-a[c][q].y, x[q].x, di));
        }
        v[2 * c] = dr;
        v[2 * c + 1] = di;
      }
      const double t = warp_totals<2 * CH>(v);
      constexpr int S = 5 - log2_of(2 * CH);  // lane l holds value l >> S
      if ((l & ((1 << S) - 1)) == 0 && 2 * i0 + (l >> S) < 2 * k) wp[wi][2 * i0 + (l >> S)] = t;
    }
  };
  auto update = [&](const double2* h) {
    for (int i0 = 0; i0 < k; i0 += CH) {
      C a[CH][E], y[E];  // even and odd basis vectors apart: half the chain of dependent FMAs
      fetch(i0, a);
#pragma unroll
      for (int q = 0; q < E; ++q) y[q] = czero<C>();
#pragma unroll
      for (int c = 0; c < CH; ++c)
        if (i0 + c < k) {
          const double2 hd = h[i0 + c];
          const C hc = cmake((R)(-hd.x), (R)(-hd.y));
#pragma unroll
          for (int q = 0; q < E; ++q) {
            if (c & 1)
              y[q] = cfma(hc, a[c][q], y[q]);
            else
              x[q] = cfma(hc, a[c][q], x[q]);
          }
        }
#pragma unroll
      for (int q = 0; q < E; ++q) x[q] = cadd(x[q], y[q]);
    }
  };
  auto block_totals = [&](int cnt, double* out) {
    __syncthreads();
    for (int v = tid; v < cnt; v += T) {
      double t = 0;
#pragma unroll
      for (int q = 0; q < NW; ++q) t += wp[q][v];
      out[v] = t;
    }
  };
  auto cluster_totals = [&](int cnt, double* mine, double* out) {  // out in shared memory; ends with a block barrier
    cl.sync();
    for (int v = tid; v < cnt; v += T) {
      double t = 0;
      for (int c = 0; c < cs; ++c) t += cl.map_shared_rank(mine, c)[v];
      out[v] = t;
    }
    __syncthreads();
  };
  if (rank == 0) givens_load(gm, k - 1, rhs, gv, tid, T);
  dots();
  block_totals(2 * k, hp1);
  cluster_totals(2 * k, hp1, reinterpret_cast<double*>(h1));
  update(h1);
  dots();
  R nr = 0;
#pragma unroll
  for (int q = 0; q < E; ++q) nr = fma(x[q].x, x[q].x, fma(x[q].y, x[q].y, nr));
  {
    const double t = warp_sum1((double)nr);
    if (l == 0) wp[wi][2 * k] = t;
  }
  block_totals(2 * k + 1, hp2);
  cluster_totals(2 * k + 1, hp2, reinterpret_cast<double*>(h2));
  double h2n = 0;
  for (int i = l; i < k; i += 32) h2n += h2[i].x * h2[i].x + h2[i].y * h2[i].y;
  h2n = warp_sum1(h2n);
  const double hn2 = h2[k].x - h2n;
  if (rank == 0 && wi == 0) {
    for (int i = l; i < k; i += 32) gv.col[i] = cadd(h1[i], h2[i]);
    __syncwarp();
    if (l == 0) givens_column(gm, k - 1, rhs, gv, hn2, kry_spent(h2[k].x, h2n));
  }
  if (hn2 > 0) {
    update(h2);
    const R f = (R)rsqrt(hn2);
#pragma unroll
    for (int q = 0; q < E; ++q)
      if (e0 + q * step < n) W[e0 + q * step] = cscale(x[q], f);
  }
  cl.sync();  // no block leaves while another may still read its shared memory
}

template <typename C, int E, int T>
void launch_small(cudaStream_t st, const C* V, long vstride, int k, C* w, long n, const KryGm& gm, int cs, double bytes,
                  double flops) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs * gm.nrhs);
  cfg.blockDim = dim3(T);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const char* name = "k_kry_small";
  KTimer* t = g_timer;
  cudaEvent_t ea = nullptr, eb = nullptr;
  if (t && t->want(name)) { ea = t->get(); eb = t->get(); MG_CUDA(cudaEventRecord(ea, st)); }
  MG_CUDA(cudaLaunchKernelEx(&cfg, &k_kry_small<C, E, T>, V, vstride, k, w, (int)n, gm));
  if (ea) {
    MG_CUDA(cudaEventRecord(eb, st));
    t->recs.push_back({name, __PRETTY_FUNCTION__, bytes, flops, ea, eb});
  }
  if (g_launch_counter) ++*g_launch_counter;
}

template <typename F>
void with_km(int k, F&& f) {
  if (k <= 1) f(std::integral_constant<int, 1>());
  else if (k <= 2) f(std::integral_constant<int, 2>());
  else if (k <= 4) f(std::integral_constant<int, 4>());
  else if (k <= 6) f(std::integral_constant<int, 6>());
  else if (k <= 8) f(std::integral_constant<int, 8>());
  else if (k <= 12) f(std::integral_constant<int, 12>());
  else f(std::integral_constant<int, 16>());
}

// blocks per right-hand side: at least 4 elements a thread, at most KRY_BLK blocks (the FP32 sums of a thread stay
// at 32 elements for the largest vectors of the benchmark)
int kry_blocks(long n, int ve) { return (int)std::max<long>(1, std::min<long>(KRY_BLK, n / (4 * KT * ve))); }

}  // namespace

void kry_trisolve(cudaStream_t st, const KryGm& gm, const int* cact, double2* y) {
  MG_LAUNCH(k_kry_trisolve, gm.nrhs, 32, 0, st, gm, cact, y);
}

size_t kry_work_bytes(int nrhs, int m) {
  return sizeof(double2) * (size_t)nrhs * (m + 2) * KRY_BLK + sizeof(unsigned) * nrhs;
}
void kry_work_init(cudaStream_t st, void* work, int nrhs, int m) {
  MG_CUDA(cudaMemsetAsync((double2*)work + (size_t)nrhs * (m + 2) * KRY_BLK, 0, sizeof(unsigned) * nrhs, st));
}

template <typename C>
void kry_step(cudaStream_t st, const C* V, long vstride, int k, C* w, long n, const KryGm& gm, void* work) {
  MG_CHECK_ARG(k >= 1 && k <= 64 && n % 2 == 0, "1..64 basis vectors of an even number of entries");
  const double ar = act_rhs(gm.nrhs), vb = ar * n * sizeof(C);
  if (n <= KRY_SMALL) {
    // one element a thread up to 1024 entries (128 threads, at most 8 blocks), up to 8 with 256 threads beyond
    const bool wide = n > 1024;
    const int T = wide ? 256 : 128;
    int cs = 1;
    while (cs < 8 && cs * T < n) cs *= 2;
    const int e = (int)((n + (long)cs * T - 1) / (cs * T));
    const double bytes = vb * (k + 2.0), flops = ar * n * 32.0 * k;
    auto go = [&](auto ec, auto tc) {
      launch_small<C, decltype(ec)::value, decltype(tc)::value>(st, V, vstride, k, w, n, gm, cs, bytes, flops);
    };
    typedef std::integral_constant<int, 128> T1;
    typedef std::integral_constant<int, 256> T2;
    if (!wide)
      go(std::integral_constant<int, 1>(), T1());
    else if (e <= 2)
      go(std::integral_constant<int, 2>(), T2());
    else if (e <= 4)
      go(std::integral_constant<int, 4>(), T2());
    else
      go(std::integral_constant<int, 8>(), T2());
    return;
  }
  double2* part = reinterpret_cast<double2*>(work);
  unsigned* done = reinterpret_cast<unsigned*>(part + (size_t)gm.nrhs * (gm.m + 2) * KRY_BLK);
  const dim3 grid(kry_blocks(n, Vec<C>::VE), gm.nrhs);
  if (k > 16) {
    vmultidot<C>(st, V, vstride, k, w, n, gm.nrhs, gm.h1, part, gm.iact);
    vgs_update<C>(st, V, vstride, k, gm.h1, w, n, gm.nrhs, gm.iact);
    vmultidot<C>(st, V, vstride, k, w, n, gm.nrhs, gm.h2, part, gm.iact);
    vnorm2<C>(st, w, n, gm.nrhs, gm.wn2, part, gm.iact);
    MG_LAUNCH(k_kry_givens, gm.nrhs, 32, 0, st, gm, k);
  } else {
    with_km(k, [&](auto km) {
      constexpr int KM = decltype(km)::value;
      MG_LAUNCH_W(vb * (k + 1.0), ar * n * 8.0 * k, (k_kry_dot<C, KM>), grid, KT, 0, st, V, vstride, k, w, n, gm.h1,
                  part, done, gm.iact);
      MG_LAUNCH_W(vb * (k + 2.0), ar * n * 16.0 * k, (k_kry_update_dot<C, KM>), grid, KT, 0, st, V, vstride, k, w, n,
                  gm, part, done);
    });
  }
  with_km(k, [&](auto km) {
    constexpr int KM = decltype(km)::value;
    MG_LAUNCH_W(vb * (k + 2.0), ar * n * 8.0 * k, (k_kry_update_scale<C, KM>), grid, KT, 0, st, V, vstride, k, w, n, gm);
  });
}
template void kry_step<float2>(cudaStream_t, const float2*, long, int, float2*, long, const KryGm&, void*);
template void kry_step<double2>(cudaStream_t, const double2*, long, int, double2*, long, const KryGm&, void*);

}  // namespace mg
