// Fine-level kernels: the Schwinger Wilson-Dirac stencil (multi-rhs), its
// SAP block matrices and the fine SAP smoother.
//
// Operator (Section 4, Schwinger discretisation, Wilson form):
//   (D x)(s) = (m0+2) x(s) + sum_mu [ (1-sigma_mu) W_mu(s) x(s+mu)
//                                    + (1+sigma_mu) conj(W_mu(s-mu)) x(s-mu) ]
// with W_mu(s) = -1/2 eta U_mu(s) the prepared link (eta = -1 on the t links
// of the last time slice: antiperiodic fermions).  (1 -+ sigma_mu) has rank 1,
// so each hop is one complex projection, one complex multiply by the link and
// a reconstruction of the lower spin:
//   (1 - sigma_1) x = h (1, -1),  h = x0 - x1
//   (1 + sigma_1) x = h (1,  1),  h = x0 + x1
//   (1 - sigma_2) x = h (1, -i),  h = x0 + i x1
//   (1 + sigma_2) x = h (1,  i),  h = x0 - i x1
#include <algorithm>
#include <type_traits>

#include "ops.cuh"

namespace mg {

__global__ void k_prepare_links(const double2* __restrict__ U, int L, double2* __restrict__ l64,
                                float2* __restrict__ l32) {
  const int V = L * L;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * V) return;
  int s = i >> 1, mu = i & 1;
  int t = s / L;
  double f = -0.5;
  if (mu == 1 && t == L - 1) f = 0.5;
  double2 u = U[i];
  double2 w = make_double2(f * u.x, f * u.y);
  l64[i] = w;
  if (l32) l32[i] = make_float2((float)w.x, (float)w.y);
}

// bad = 1 if some link is not a finite complex number
__global__ void k_check_links(const double2* __restrict__ U, long count, int* bad) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x) {
    const double2 u = U[i];
    if (!isfinite(u.x) || !isfinite(u.y)) atomicExch(bad, 1);
  }
}
void check_links(cudaStream_t st, const double2* U, int L, int* bad) {
  MG_LAUNCH(k_check_links, cdiv(2L * L * L, 256), 256, 0, st, U, 2L * L * L, bad);
}

void prepare_links(cudaStream_t st, const double2* U, int L, double2* l64, float2* l32) {
  MG_LAUNCH(k_prepare_links, cdiv(2L * L * L, 256), 256, 0, st, U, L, l64, l32);
}

// ---- spinor loads ----------------------------------------------------------
__device__ __forceinline__ void ld_sp(const float2* __restrict__ p, long s, float2& a, float2& b) {
  float4 v = __ldg(reinterpret_cast<const float4*>(p) + s);
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld_sp(const double2* __restrict__ p, long s, double2& a, double2& b) {
  a = __ldg(p + 2 * s);
  b = __ldg(p + 2 * s + 1);
}
__device__ __forceinline__ void st_sp(float2* p, long s, float2 a, float2 b) {
  reinterpret_cast<float4*>(p)[s] = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_sp(double2* p, long s, double2 a, double2 b) {
  p[2 * s] = a;
  p[2 * s + 1] = b;
}

// Links of a site's hops: prepared ones (k_prepare_links), or straight from U (same values: a factor of +-1/2 before the
// rounding to R), which saves a launch and a workspace where a call is a few microseconds.
template <typename R>
struct PreparedLinks {
  const typename CT<R>::T* __restrict__ lk;
  __device__ __forceinline__ typename CT<R>::T x(int s) const { return __ldg(lk + 2 * s); }
  __device__ __forceinline__ typename CT<R>::T t(int s, bool) const { return __ldg(lk + 2 * s + 1); }
};
template <typename R>
struct RawLinks {
  const double2* __restrict__ U;
  __device__ __forceinline__ typename CT<R>::T x(int s) const {
    const double2 u = __ldg(U + 2 * s);
    return cmake((R)(-0.5 * u.x), (R)(-0.5 * u.y));
  }
  __device__ __forceinline__ typename CT<R>::T t(int s, bool last_slice) const {
    const double2 u = __ldg(U + 2 * s + 1);
    const double f = last_slice ? 0.5 : -0.5;
    return cmake((R)(f * u.x), (R)(f * u.y));
  }
};

// (D x)(s) for one site of one rhs (X points at that rhs).
template <typename R, typename LK>
__device__ __forceinline__ void wilson_site(const LK& lk, R diag, int L,
                                            const typename CT<R>::T* __restrict__ X, int s,
                                            typename CT<R>::T& o0, typename CT<R>::T& o1) {
  typedef typename CT<R>::T C;
  const int V = L * L;
  const int t = s / L, xx = s - t * L;
  const int sxp = s + (xx == L - 1 ? 1 - L : 1);
  const int sxm = s + (xx == 0 ? L - 1 : -1);
  const int stp = (t == L - 1) ? xx : s + L;
  const int stm = (t == 0) ? s + V - L : s - L;
  C a0, a1;
  ld_sp(X, s, a0, a1);
  o0 = cscale(a0, diag);
  o1 = cscale(a1, diag);
  {  // +x : (1 - sigma_1) W_0(s) x(s+x)
    ld_sp(X, sxp, a0, a1);
    C u = cmul(lk.x(s), csub(a0, a1));
    o0 = cadd(o0, u);
    o1 = csub(o1, u);
  }
  {  // -x : (1 + sigma_1) conj(W_0(s-x)) x(s-x)
    ld_sp(X, sxm, a0, a1);
    C u = cmulc(lk.x(sxm), cadd(a0, a1));
    o0 = cadd(o0, u);
    o1 = cadd(o1, u);
  }
  {  // +t : (1 - sigma_2) W_1(s) x(s+t)
    ld_sp(X, stp, a0, a1);
    C u = cmul(lk.t(s, t == L - 1), cadd(a0, cmuli(a1)));
    o0 = cadd(o0, u);
    o1 = cadd(o1, cmulmi(u));
  }
  {  // -t : (1 + sigma_2) conj(W_1(s-t)) x(s-t)
    ld_sp(X, stm, a0, a1);
    C u = cmulc(lk.t(stm, t == 0), cadd(a0, cmulmi(a1)));
    o0 = cadd(o0, u);
    o1 = cadd(o1, cmuli(u));
  }
}

// One thread per site and rhs.
template <typename R, bool RES, typename LK>
__global__ void __launch_bounds__(256) k_wilson(LK lk, R diag, int L, const typename CT<R>::T* __restrict__ x,
                                                typename CT<R>::T* __restrict__ y,
                                                const typename CT<R>::T* __restrict__ b,
                                                const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  const int V = L * L, s = blockIdx.x * blockDim.x + threadIdx.x, rhs = blockIdx.y;
  if (s >= V || (active && !active[rhs])) return;
  const size_t off = (size_t)rhs * 2 * V;
  C o0, o1;
  wilson_site<R>(lk, diag, L, x + off, s, o0, o1);
  if (RES) {
    C b0, b1;
    ld_sp(b + off, s, b0, b1);
    o0 = csub(b0, o0);
    o1 = csub(b1, o1);
  }
  st_sp(y + off, s, o0, o1);
}

// FP32, long batches: a thread walks WT time slices of its column, for RPT right-hand sides (blockIdx.y * RPT + j),
// with the spinors of the last, this and the next slice in registers, so that a spinor comes from L2 (1 + 2 / WT)
// times instead of three times and a link 1 / RPT times; its x neighbours are L1 hits of the same row.  One thread
// per site and rhs moved 80 bytes of L2 traffic per site and rhs for 32 of DRAM (5.0 TB/s at L = 512, 256 rhs).  The
// columns of all slice groups are numbered through, so that lattices whose side is no multiple of a block leave no lanes
// idle.
constexpr int WT = 8;
template <bool RES, int RPT>
__global__ void __launch_bounds__(128) k_wilson_walk(const float2* __restrict__ lk, float diag, int L,
                                                     const float2* __restrict__ x, float2* __restrict__ y,
                                                     const float2* __restrict__ b, const int* __restrict__ active,
                                                     int nrhs) {
  const int V = L * L, i = blockIdx.x * 128 + threadIdx.x, tb = i / L, xx = i - tb * L;
  const int t0 = tb * WT, t1 = min(t0 + WT, L);
  if (t0 >= L) return;
  const float4* X[RPT];
  bool on[RPT];
  float4 prev[RPT], cur[RPT];
  const int xr = xx == L - 1 ? 0 : xx + 1, xl = xx == 0 ? L - 1 : xx - 1, tp0 = t0 == 0 ? L - 1 : t0 - 1;
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int rhs = blockIdx.y * RPT + j;
    on[j] = rhs < nrhs && !(active && !active[rhs]);
    X[j] = reinterpret_cast<const float4*>(x + (size_t)(on[j] ? rhs : 0) * 2 * V);
    if (on[j]) {
      prev[j] = __ldg(X[j] + (size_t)tp0 * L + xx);
      cur[j] = __ldg(X[j] + (size_t)t0 * L + xx);
    }
  }
  float2 wt_prev = __ldg(lk + 2 * (tp0 * L + xx) + 1);
#pragma unroll 2
  for (int t = t0; t < t1; ++t) {
    const int row = t * L, s = row + xx, next = (t == L - 1 ? 0 : row + L) + xx;
    const float4 w = __ldg(reinterpret_cast<const float4*>(lk) + s);  // both links of the site
    const float2 wx = make_float2(w.x, w.y), wt = make_float2(w.z, w.w), wl = __ldg(lk + 2 * (row + xl));
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if (!on[j]) continue;
      const float4 nx = __ldg(X[j] + next), rt = __ldg(X[j] + row + xr), lf = __ldg(X[j] + row + xl);
      float2 o0 = cscale(make_float2(cur[j].x, cur[j].y), diag), o1 = cscale(make_float2(cur[j].z, cur[j].w), diag);
      float2 a0, a1;
      a0 = make_float2(rt.x, rt.y); a1 = make_float2(rt.z, rt.w);
      {
        const float2 u = cmul(wx, csub(a0, a1));
        o0 = cadd(o0, u);
        o1 = csub(o1, u);
      }
      a0 = make_float2(lf.x, lf.y); a1 = make_float2(lf.z, lf.w);
      {
        const float2 u = cmulc(wl, cadd(a0, a1));
        o0 = cadd(o0, u);
        o1 = cadd(o1, u);
      }
      a0 = make_float2(nx.x, nx.y); a1 = make_float2(nx.z, nx.w);
      {
        const float2 u = cmul(wt, cadd(a0, cmuli(a1)));
        o0 = cadd(o0, u);
        o1 = cadd(o1, cmulmi(u));
      }
      a0 = make_float2(prev[j].x, prev[j].y); a1 = make_float2(prev[j].z, prev[j].w);
      {
        const float2 u = cmulc(wt_prev, cadd(a0, cmulmi(a1)));
        o0 = cadd(o0, u);
        o1 = cadd(o1, cmuli(u));
      }
      const size_t off = (size_t)(blockIdx.y * RPT + j) * 2 * V;
      if (RES) {
        float2 b0, b1;
        ld_sp(b + off, s, b0, b1);
        o0 = csub(b0, o0);
        o1 = csub(b1, o1);
      }
      st_sp(y + off, s, o0, o1);
      prev[j] = cur[j];
      cur[j] = nx;
    }
    wt_prev = wt;
  }
}

template <typename R, typename LK>
static void wilson_sites(cudaStream_t st, LK lk, R diag, int L, const typename CT<R>::T* x, typename CT<R>::T* y,
                         const typename CT<R>::T* b, int nrhs, const int* active, double bytes, double flops) {
  // blocks of 64 threads where 256 would leave most SMs without one (FP64: two FMAs a clock and SM bound it)
  const int bt = (long)L * L * nrhs >= 512L * sm_count() ? 256 : 64;
  const dim3 grid(cdiv((long)L * L, bt), nrhs);
  if (b)
    MG_LAUNCH_W(bytes, flops, (k_wilson<R, true, LK>), grid, bt, 0, st, lk, diag, L, x, y, b, active);
  else
    MG_LAUNCH_W(bytes, flops, (k_wilson<R, false, LK>), grid, bt, 0, st, lk, diag, L, x, y, b, active);
}

// FP32: 0 one thread per site, else right-hand sides per thread of the walking form, the tuned number or 1 where that
// would leave the chip short of threads.  The line, with one rhs per thread, per site against walking: L = 512 with 4,
// 12, 49, 244 rhs 17.5, 30.8, 86.2, 378 against 15.6, 31.4, 84.2, 357 us; L = 136 with 52, 173, 3460 rhs 12.5, 26.7, 371
// against 12.3, 24.7, 366; below 64 columns a warp lies across slice groups and the per-site form wins (L = 16, 24, 48
// with 12.8 M sites x rhs: 73.9, 81.4, 78.0 against 88.0, 94.6, 82.6).  At L = 512 with 244 rhs the walk takes 357 us with
// one rhs per thread, 389 with two, 505 with four; with 256 rhs 367 us alone (0.88 of the copy bandwidth), 413 against 375
// in an earlier form with 16 slices instead of 8.
int wilson_variant(int L, int nrhs, int rpt) {
  const double threads = (double)L * L * nrhs / WT, least = 1024.0 * sm_count();
  if (L < 64 || threads < least) return 0;
  return threads / rpt >= least ? rpt : 1;
}

template <typename R>
void wilson_apply(cudaStream_t st, const typename CT<R>::T* links, R diag, int L, const typename CT<R>::T* x,
                  typename CT<R>::T* y, const typename CT<R>::T* b, int nrhs, const int* active) {
  if (nrhs <= 0) return;
  if (nrhs > 65535) {  // one row of the grid per rhs
    for (int r = 0; r < nrhs; r += 65535) {
      const size_t n = 2 * (size_t)L * L;
      wilson_apply<R>(st, links, diag, L, x + r * n, y + r * n, b ? b + r * n : nullptr, std::min(65535, nrhs - r),
                      active ? active + r : nullptr);
    }
    return;
  }
  // algorithmic traffic: x read + y written once per site and rhs (+ b), links once per launch
  const double V = (double)L * L, sp = 2.0 * sizeof(typename CT<R>::T), ar = act_rhs(nrhs);
  const double bytes = ar * V * sp * (b ? 3 : 2) + V * sp;
  const double flops = ar * V * (b ? 56.0 : 52.0);
  if constexpr (sizeof(R) == 4) {
    if (const int rpt = wilson_variant(L, nrhs, tune_lookup(TUNE_WILSON32, L, nrhs, 0, 1))) {
      const dim3 grid(cdiv((long)L * cdiv(L, WT), 128), cdiv(nrhs, rpt));
#define MG_WILSON_LAUNCH(RPT_)                                                                                        \
  do {                                                                                                                \
    if (b)                                                                                                            \
      MG_LAUNCH_W(bytes, flops, (k_wilson_walk<true, RPT_>), grid, 128, 0, st, links, diag, L, x, y, b, active,       \
                  nrhs);                                                                                              \
    else                                                                                                              \
      MG_LAUNCH_W(bytes, flops, (k_wilson_walk<false, RPT_>), grid, 128, 0, st, links, diag, L, x, y, b, active,      \
                  nrhs);                                                                                              \
  } while (0)
      if (rpt == 4)
        MG_WILSON_LAUNCH(4);
      else if (rpt == 2)
        MG_WILSON_LAUNCH(2);
      else
        MG_WILSON_LAUNCH(1);
#undef MG_WILSON_LAUNCH
      return;
    }
  }
  wilson_sites<R>(st, PreparedLinks<R>{links}, diag, L, x, y, b, nrhs, active, bytes, flops);
}

template <typename R>
void wilson_apply_raw(cudaStream_t st, const double2* U, R diag, int L, const typename CT<R>::T* x,
                      typename CT<R>::T* y, int nrhs) {
  const double V = (double)L * L, sp = 2.0 * sizeof(typename CT<R>::T);
  wilson_sites<R>(st, RawLinks<R>{U}, diag, L, x, y, (const typename CT<R>::T*)nullptr, nrhs, nullptr,
                  nrhs * V * sp * 2 + V * 32.0, nrhs * V * 52.0);
}
template void wilson_apply_raw<float>(cudaStream_t, const double2*, float, int, const float2*, float2*, int);
template void wilson_apply_raw<double>(cudaStream_t, const double2*, double, int, const double2*, double2*, int);
template void wilson_apply<float>(cudaStream_t, const float2*, float, int, const float2*, float2*, const float2*,
                                  int, const int*);
template void wilson_apply<double>(cudaStream_t, const double2*, double, int, const double2*, double2*,
                                   const double2*, int, const int*);

// ---- SAP block matrices ------------------------------------------------------
// Block (BT, BX) of bs x bs sites; local dof index (jt * bs + jx) * 2 + spin.
// out[block][bd][bd], bd = 2 bs^2, blocks ordered BT slow, BX fast.
__global__ void k_fine_blocks(const double2* __restrict__ lk, double diag, int L, int bs, double2* __restrict__ out) {
  const int nbx = L / bs;
  const int blk = blockIdx.x;
  const int BT = blk / nbx, BX = blk % nbx;
  const int bd = 2 * bs * bs;
  double2* A = out + (size_t)blk * bd * bd;
  for (int e = threadIdx.x; e < bd * bd; e += blockDim.x) A[e] = make_double2(0, 0);
  __syncthreads();
  for (int j = threadIdx.x; j < bs * bs; j += blockDim.x) {
    const int jt = j / bs, jx = j % bs;
    const int t = BT * bs + jt, x = BX * bs + jx;
    const int s = t * L + x;
    A[(2 * j) * bd + 2 * j] = make_double2(diag, 0);
    A[(2 * j + 1) * bd + 2 * j + 1] = make_double2(diag, 0);
    // (row spin a, col spin b) coefficients of the four projectors
    if (jx + 1 < bs) {  // +x, link W_0(s)
      const int k = j + 1;
      double2 w = lk[2 * s];
      A[(2 * j) * bd + 2 * k] = w;
      A[(2 * j) * bd + 2 * k + 1] = cneg(w);
      A[(2 * j + 1) * bd + 2 * k] = cneg(w);
      A[(2 * j + 1) * bd + 2 * k + 1] = w;
    }
    if (jx > 0) {  // -x, conj(W_0(s-x))
      const int k = j - 1;
      double2 w = cconj(lk[2 * (s - 1)]);
      A[(2 * j) * bd + 2 * k] = w;
      A[(2 * j) * bd + 2 * k + 1] = w;
      A[(2 * j + 1) * bd + 2 * k] = w;
      A[(2 * j + 1) * bd + 2 * k + 1] = w;
    }
    if (jt + 1 < bs) {  // +t, W_1(s); (1 - sigma_2) = [[1, i], [-i, 1]]
      const int k = j + bs;
      double2 w = lk[2 * s + 1];
      A[(2 * j) * bd + 2 * k] = w;
      A[(2 * j) * bd + 2 * k + 1] = cmuli(w);
      A[(2 * j + 1) * bd + 2 * k] = cmulmi(w);
      A[(2 * j + 1) * bd + 2 * k + 1] = w;
    }
    if (jt > 0) {  // -t, conj(W_1(s-t)); (1 + sigma_2) = [[1, -i], [i, 1]]
      const int k = j - bs;
      double2 w = cconj(lk[2 * (s - L) + 1]);
      A[(2 * j) * bd + 2 * k] = w;
      A[(2 * j) * bd + 2 * k + 1] = cmulmi(w);
      A[(2 * j + 1) * bd + 2 * k] = cmuli(w);
      A[(2 * j + 1) * bd + 2 * k + 1] = w;
    }
  }
}

void fine_block_matrices(cudaStream_t st, const double2* l64, double diag, int L, int bs, double2* out) {
  const int nb = (L / bs) * (L / bs);
  MG_LAUNCH(k_fine_blocks, nb, 128, 0, st, l64, diag, L, bs, out);
}

// ---- SAP half sweep on the fine level ----------------------------------------
// x_B += D_BB^{-1} (f - D x)_B on the blocks of one colour.  `known` says what of x is read: all of it (SAP_X),
// nothing (SAP_ZERO: x counts as zero, the first half sweep of a cycle), or the other colour only (SAP_OTHER: x
// counts as zero on this colour, the second half sweep).

// FP32, 4 x 4 blocks.  An item is one block; blockIdx.y picks the tile of RG right-hand sides, which a CTA keeps.
// Two warps per CTA and one shared-memory stage (21 KB at RG = 16, ten CTAs per SM, each in another phase):
//   fetch     f on the block, x on the block and on the 16 sites around it, the inverse, all by cp.async
//   residual  lane = rhs, consecutive sites per thread: f - D x replaces f in place
//   product   inv_B r: a thread owns two sites (4 complex rows) times NR = RG / 8 rhs
// What bounds it: the bytes that shared memory returns to registers (128 a clock and SM; 48 bytes for 32 FMAs in the
// product), then DRAM (390 MB at L = 512, 32 rhs: f and x come as whole 128-byte lines although a colour uses every
// other 64 bytes).  Half sweep at L = 512: 100 us with 32 rhs, 56 with 16, 37 with 8.  Measured at 32 rhs and left:
// loads to registers at the start of an item 147 us (global latency); one row and 8 rhs per thread (72 bytes for 32
// FMAs) 130 us whatever the occupancy, prefetch depth or packing of the FMAs.  The sums run over the columns in order.
// With RESTRICT the items are all aggregates (4 x 4 sites as well), `inv` holds the prolongator blocks and `out` the
// coarse vectors: xc_a = P_a^H (f - D x)_a, the residual never leaves the SM (residual and restriction in one: 185 ->
// 123 us at L = 512, 32 rhs).
template <int RG, bool RESTRICT>
struct SapF {
  static constexpr int RP = RG + 1;  // padded row: 8 sites of one rhs hit distinct banks in the final update
  float4 f[16 * RG];
  float4 x[32 * RP];    // block sites, then the sites around it: -x, +x (by row), -t, +t (by column)
  float2 inv[RESTRICT ? 256 : 1024];  // transposed: row j holds column j of the inverse; P: [chirality][site][vector]
  float2 lx[20];        // x links of sites (row, -1 .. 3)
  float2 lt[20];        // t links of sites (-1 .. 3, column)
};

template <int RG, bool RESTRICT>
__global__ void __launch_bounds__(64) k_sap_fine4_fp32(const float2* __restrict__ lk, float diag, int L,
                                                       const float2* __restrict__ inv, const float2* f,
                                                       const float2* x, float2* out, int color, int nrhs, int nitems,
                                                       int known, const int* active) {
  pdl_begin();
  typedef SapF<RG, RESTRICT> S;
  constexpr int RP = S::RP, T = 64, NR = RG / 8, RSTEP = T / (4 * RG) ? T / (4 * RG) : 1;
  constexpr int RTH = T / 4 < RG ? T / 4 : RG;  // rhs that the CTA's threads fetch at once
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S& s = *reinterpret_cast<S*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31;
  const int nbx = L / 4, half = nbx / 2, r0 = blockIdx.y * RG;
  const size_t n = 2 * (size_t)L * L;
  const unsigned live_mask =
      __ballot_sync(0xffffffffu, lane < RG && r0 + lane < nrhs && !(active && !active[r0 + lane]));
  // fetch: site fj of row fi + RSTEP m of rhs frr + RTH k (64 consecutive bytes per rhs and row)
  const int fj = tid & 3, frr = (tid >> 2) % RTH, fi = (tid >> 2) / RTH;
  const int g = tid & 7, rg = tid >> 3;  // row group and rhs group of the product
  for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int BT = RESTRICT ? item / nbx : item / half, t0 = 4 * BT;
    const int x0 = RESTRICT ? 4 * (item - BT * nbx) : 4 * (2 * (item - BT * half) + ((BT + color) & 1));
    const int tm = t0 == 0 ? L - 1 : t0 - 1, tp = t0 + 4 == L ? 0 : t0 + 4;
    const int xm = x0 == 0 ? L - 1 : x0 - 1, xp = x0 + 4 == L ? 0 : x0 + 4;
    {
      constexpr int NI = RESTRICT ? 256 : 1024;
      const char* I = reinterpret_cast<const char*>(inv + (size_t)(BT * nbx + x0 / 4) * NI);
#pragma unroll
      for (int q = 0; q < NI / 2 / T; ++q)
        cp_async16(reinterpret_cast<char*>(s.inv) + (tid + q * T) * 16, I + (tid + q * T) * 16);
      if (tid < 20) {
        const int i = tid / 5, j = tid - 5 * i;
        cp_async_elem(&s.lx[tid], lk + 2 * ((t0 + i) * L + (j ? x0 + j - 1 : xm)));
      } else if (tid >= 32 && tid < 52) {
        const int i = (tid - 32) >> 2, j = tid & 3;
        cp_async_elem(&s.lt[tid - 32], lk + 2 * ((i ? t0 + i - 1 : tm) * L + x0 + j) + 1);
      }
#pragma unroll
      for (int k = 0; k < RG / RTH; ++k) {
        const int rr = frr + RTH * k;
        if (!((live_mask >> rr) & 1)) continue;
        const float2* frow = f + (size_t)(r0 + rr) * n;
        const float2* xrow = x + (size_t)(r0 + rr) * n;
#pragma unroll
        for (int m = 0; m < 4 / RSTEP; ++m) {
          const int i = fi + RSTEP * m, q = 4 * i + fj;
          const int site = (t0 + i) * L + x0 + fj;
          cp_async16(&s.f[q * RG + rr], frow + 2 * site);
          if (known == SAP_X) cp_async16(&s.x[q * RP + rr], xrow + 2 * site);
          if (known != SAP_ZERO) {
            const int edge = i == 0 ? (t0 + fj) * L + xm : i == 1 ? (t0 + fj) * L + xp : (i == 2 ? tm : tp) * L + x0 + fj;
            cp_async16(&s.x[(16 + q) * RP + rr], xrow + 2 * edge);
          }
        }
      }
      asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    if (known != SAP_ZERO) {
      constexpr int SPT = 16 * RG / T;  // sites per thread: consecutive ones
      const int rr = tid % RG, j0 = (tid / RG) * SPT;
      float2 a0, a1;
      auto at = [&](int k) {
        const float4 v = k >= 16 || known == SAP_X ? s.x[k * RP + rr] : make_float4(0.f, 0.f, 0.f, 0.f);
        a0 = make_float2(v.x, v.y);
        a1 = make_float2(v.z, v.w);
      };
#pragma unroll
      for (int q = 0; q < SPT; ++q) {
        const int j = j0 + q, jx = j & 3, jt = j >> 2;
        at(j);
        float2 o0 = cscale(a0, diag), o1 = cscale(a1, diag);
        {
          at(jx < 3 ? j + 1 : 20 + jt);
          const float2 u = cmul(s.lx[5 * jt + jx + 1], csub(a0, a1));
          o0 = cadd(o0, u);
          o1 = csub(o1, u);
        }
        {
          at(jx > 0 ? j - 1 : 16 + jt);
          const float2 u = cmulc(s.lx[5 * jt + jx], cadd(a0, a1));
          o0 = cadd(o0, u);
          o1 = cadd(o1, u);
        }
        {
          at(jt < 3 ? j + 4 : 28 + jx);
          const float2 u = cmul(s.lt[4 * jt + 4 + jx], cadd(a0, cmuli(a1)));
          o0 = cadd(o0, u);
          o1 = cadd(o1, cmulmi(u));
        }
        {
          at(jt > 0 ? j - 4 : 24 + jx);
          const float2 u = cmulc(s.lt[4 * jt + jx], cadd(a0, cmulmi(a1)));
          o0 = cadd(o0, u);
          o1 = cadd(o1, cmuli(u));
        }
        const float4 fv = s.f[j * RG + rr];
        s.f[j * RG + rr] = make_float4(fv.x - o0.x, fv.y - o0.y, fv.z - o1.x, fv.w - o1.y);
      }
      __syncthreads();
    }
    if constexpr (RESTRICT) {  // 16 coarse dofs (chirality, vector) x RG rhs: 4 threads per dof, RG / 4 rhs each
      constexpr int RQ = RG / 4;
      const int o = tid & 15, c = o >> 3, m = o & 7, q0 = (tid >> 4) * RQ;
      float2 acc[RQ];
#pragma unroll
      for (int b = 0; b < RQ; ++b) acc[b] = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 p = s.inv[(c * 16 + j) * 8 + m];
#pragma unroll
        for (int b = 0; b < RQ; ++b)
          acc[b] = cfmac(p, reinterpret_cast<const float2*>(&s.f[j * RG + q0 + b])[c], acc[b]);
      }
#pragma unroll
      for (int b = 0; b < RQ; ++b)
        if ((live_mask >> (q0 + b)) & 1) out[(size_t)(r0 + q0 + b) * (n / 2) + 16 * (size_t)item + o] = acc[b];
    } else {
      float2 acc[4][NR];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < NR; ++b) acc[a][b] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int j = 0; j < 16; ++j) {
        float4 v[NR];
#pragma unroll
        for (int b = 0; b < NR; ++b) v[b] = s.f[j * RG + rg * NR + b];
#pragma unroll
        for (int sp = 0; sp < 2; ++sp) {
          const float4* mi = reinterpret_cast<const float4*>(s.inv + (2 * j + sp) * 32);
          const float4 m0 = mi[g], m1 = mi[8 + g];  // rows 2g, 2g + 1 and 16 + 2g, 17 + 2g
#pragma unroll
          for (int b = 0; b < NR; ++b) {
            const float2 w = sp ? make_float2(v[b].z, v[b].w) : make_float2(v[b].x, v[b].y);
            acc[0][b] = cfma(make_float2(m0.x, m0.y), w, acc[0][b]);
            acc[1][b] = cfma(make_float2(m0.z, m0.w), w, acc[1][b]);
            acc[2][b] = cfma(make_float2(m1.x, m1.y), w, acc[2][b]);
            acc[3][b] = cfma(make_float2(m1.z, m1.w), w, acc[3][b]);
          }
        }
      }
      const int site = (t0 + (g >> 2)) * L + x0 + (g & 3);
      float2* xo = out + (size_t)(r0 + rg * NR) * n;
#pragma unroll
      for (int b = 0; b < NR; ++b) {
        const int rr = rg * NR + b;
        if ((live_mask >> rr) & 1) {
          if (known == SAP_X) {
            const float4 p = s.x[g * RP + rr], q = s.x[(8 + g) * RP + rr];
            acc[0][b] = cadd(make_float2(p.x, p.y), acc[0][b]);
            acc[1][b] = cadd(make_float2(p.z, p.w), acc[1][b]);
            acc[2][b] = cadd(make_float2(q.x, q.y), acc[2][b]);
            acc[3][b] = cadd(make_float2(q.z, q.w), acc[3][b]);
          }
          st_sp(xo + (size_t)b * n, site, acc[0][b], acc[1][b]);
          st_sp(xo + (size_t)b * n, site + 2 * L, acc[2][b], acc[3][b]);
        }
      }
    }
    __syncthreads();  // the stage is refilled next
  }
}

// FP64, 4 x 4 blocks: bound by the FP64 units (two FMAs a clock and SM).  The blocks of one colour do not couple, so
// with E the hops that leave the block x_B + D_BB^{-1} (f - D x)_B = D_BB^{-1} (f - E x)_B: the hops inside the block
// and the old x_B drop out.  One CTA of two warps per block and tile of at most 16 right-hand sides.  A lane owns a row
// of the block and a warp takes every second live right-hand side of the tile, up to four at a time, so that neither the
// remainder of a tile nor a right-hand side that has stopped costs FMAs, and the hops have loops of their own, in which
// every lane has one.  With whole tiles of 8 and 16 in threads of 4 rows x 1 or 2 right-hand sides a sweep of one took
// as long as of eight: at L = 512 with 1, 8, 9, 17, 64 right-hand sides 940, 943, 1860, 3645, 7390 us, now 193, 948,
// 1118, 2035, 7410 (the products alone 107, 853, 960, 1810, 6825).  Which warp gets the odd one changes from block to
// block, because a CTA's first warp lands in the same quarters of an SM.
constexpr int SF64_TILE = 16;
__global__ void __launch_bounds__(64) k_sap_fine4_fp64(const double2* __restrict__ lk, int L,
                                                       const double2* __restrict__ inv, const double2* __restrict__ f,
                                                       double2* __restrict__ x, int color, int nrhs, int tile, int known,
                                                       const int* __restrict__ active) {
  constexpr int BD = 32, IS = BD + 1;
  __shared__ double2 sinv[BD * IS];  // transposed
  __shared__ double2 sres[SF64_TILE][BD];
  __shared__ int srhs[SF64_TILE];  // live right-hand sides of the tile
  __shared__ int scount;
  const int tid = threadIdx.x, lane = tid & 31;
  const int nbx = L / 4, half = nbx / 2;
  const int BT = blockIdx.x / half;
  const int BX = 2 * (blockIdx.x - BT * half) + ((BT + color) & 1);
  const double2* I = inv + (size_t)(BT * nbx + BX) * BD * BD;
#pragma unroll 4
  for (int e = tid; e < BD * BD; e += 64) sinv[(e % BD) * IS + e / BD] = I[e];
  const size_t n = 2 * (size_t)L * L;
  const int first = (tid >> 5) ^ ((blockIdx.x * 0x9E3779B1u) >> 31);  // this warp's first slot
  for (int r0 = blockIdx.y * tile; r0 < nrhs; r0 += gridDim.y * tile) {
    if (tid < 32) {
      const bool on = lane < tile && r0 + lane < nrhs && !(active && !active[r0 + lane]);
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) srhs[__popc(m & ((1u << lane) - 1))] = r0 + lane;
      if (lane == 0) scount = __popc(m);
    }
    __syncthreads();
    const int cnt = scount;
    for (int q = tid; q < 32 * cnt; q += 64)
      sres[q >> 5][q & 31] = __ldg(f + srhs[q >> 5] * n + 2 * ((size_t)(4 * BT + ((q >> 3) & 3)) * L + 4 * BX) + (q & 7));
    if (known != SAP_ZERO) {
      __syncthreads();
      for (int q = tid; q < 8 * cnt; q += 64) {  // (1 -+ sigma_1) hops out of the block
        const bool up = q & 1;
        const int jt = (q >> 1) & 3, j = 4 * jt + (up ? 3 : 0), xx = 4 * BX + (up ? 3 : 0), s = (4 * BT + jt) * L + xx;
        const int s2 = up ? (xx == L - 1 ? s + 1 - L : s + 1) : (xx == 0 ? s + L - 1 : s - 1);
        double2 a0, a1;
        ld_sp(x + srhs[q >> 3] * n, s2, a0, a1);
        const double2 w = up ? __ldg(lk + 2 * s) : cconj(__ldg(lk + 2 * s2));
        const double2 u = cmul(w, cadd(a0, up ? cneg(a1) : a1));
        double2* o = sres[q >> 3] + 2 * j;
        o[0] = csub(o[0], u);
        o[1] = csub(o[1], up ? cneg(u) : u);
      }
      __syncthreads();
      for (int q = tid; q < 8 * cnt; q += 64) {  // (1 -+ sigma_2) hops
        const bool up = q & 4;
        const int jx = q & 3, j = (up ? 12 : 0) + jx, t = 4 * BT + (up ? 3 : 0), xx = 4 * BX + jx, s = t * L + xx;
        const int s2 = up ? (t == L - 1 ? xx : s + L) : (t == 0 ? s + L * (L - 1) : s - L);
        double2 a0, a1;
        ld_sp(x + srhs[q >> 3] * n, s2, a0, a1);
        const double2 w = up ? __ldg(lk + 2 * s + 1) : cconj(__ldg(lk + 2 * s2 + 1));
        const double2 u = cmul(w, cadd(a0, up ? cmuli(a1) : cmulmi(a1)));
        double2* o = sres[q >> 3] + 2 * j;
        o[0] = csub(o[0], u);
        o[1] = cadd(o[1], up ? cmuli(u) : cmulmi(u));
      }
    }
    __syncthreads();
    auto product = [&](int k0, auto nrc) {  // slots k0, k0 + 2, ..
      constexpr int NR = decltype(nrc)::value;
      double2 acc[NR];
#pragma unroll
      for (int b = 0; b < NR; ++b) acc[b] = make_double2(0, 0);
#pragma unroll 4
      for (int j = 0; j < BD; ++j) {
        const double2 m = sinv[j * IS + lane];
#pragma unroll
        for (int b = 0; b < NR; ++b) acc[b] = cfma(m, sres[k0 + 2 * b][j], acc[b]);
      }
      const size_t o = 2 * ((size_t)(4 * BT + (lane >> 3)) * L + 4 * BX) + (lane & 7);
#pragma unroll
      for (int b = 0; b < NR; ++b) x[srhs[k0 + 2 * b] * n + o] = acc[b];
    };
    int k = first;
    for (; k + 6 < cnt; k += 8) product(k, std::integral_constant<int, 4>());
    for (; k + 2 < cnt; k += 4) product(k, std::integral_constant<int, 2>());
    if (k < cnt) product(k, std::integral_constant<int, 1>());
    __syncthreads();
  }
}

// 2 x 2 blocks (8 unknowns; mg_params.sap_block_fine = 2): one CTA per block, one thread per (row, rhs)
template <typename R>
__global__ void __launch_bounds__(256) k_sap_fine2(const typename CT<R>::T* __restrict__ lk, R diag, int L,
                                                   const typename CT<R>::T* __restrict__ inv, bool inv_t,
                                                   const typename CT<R>::T* __restrict__ f,
                                                   typename CT<R>::T* __restrict__ x, int color, int nrhs,
                                                   const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  constexpr int NS = 4, BD = 8, G = 64;
  __shared__ C sinv[BD * BD];  // sinv[j * BD + i] = inv[i][j]
  __shared__ C sres[G * BD];
  const int nbx = L / 2, half = nbx / 2;
  const int BT = blockIdx.x / half;
  const int BX = 2 * (blockIdx.x - BT * half) + ((BT + color) & 1);
  const C* I = inv + (size_t)(BT * nbx + BX) * BD * BD;
  for (int e = threadIdx.x; e < BD * BD; e += blockDim.x) sinv[inv_t ? e : (e % BD) * BD + e / BD] = I[e];
  const size_t n = 2 * (size_t)L * L;
  for (int r0 = 0; r0 < nrhs; r0 += G) {
    __syncthreads();
    {
      const int q = threadIdx.x, g = q / NS, j = q % NS, rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) {
        const int s = (BT * 2 + j / 2) * L + BX * 2 + (j % 2);
        C o0, o1, f0, f1;
        wilson_site<R>(PreparedLinks<R>{lk}, diag, L, x + rhs * n, s, o0, o1);
        ld_sp(f + rhs * n, s, f0, f1);
        sres[g * BD + 2 * j] = csub(f0, o0);
        sres[g * BD + 2 * j + 1] = csub(f1, o1);
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < G * BD; q += blockDim.x) {
      const int g = q / BD, i = q % BD, rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) {
        C acc = czero<C>();
#pragma unroll
        for (int j = 0; j < BD; ++j) acc = cfma(sinv[j * BD + i], sres[g * BD + j], acc);
        const int js = i >> 1, s = (BT * 2 + js / 2) * L + BX * 2 + (js % 2);
        C* px = x + rhs * n + 2 * s + (i & 1);
        *px = cadd(*px, acc);
      }
    }
  }
}

template <typename R>
void sap_half_fine(cudaStream_t st, const typename CT<R>::T* links, R diag, int L, int bs,
                   const typename CT<R>::T* inv, const typename CT<R>::T* f, typename CT<R>::T* x, int color,
                   int nrhs, const int* active, bool inv_transposed, int known) {
  MG_CHECK_ARG(bs == 4 || bs == 2, "fine SAP block side must be 2 or 4");
  if (nrhs <= 0) return;
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const size_t n = 2 * (size_t)L * L;
      sap_half_fine<R>(st, links, diag, L, bs, inv, f + r * n, x + r * n, color, std::min(RHS_SLICE, nrhs - r),
                       active ? active + r : nullptr, inv_transposed, known);
    }
    return;
  }
  const int nb = (L / bs) * (L / bs) / 2;
  // per block and rhs: f and the surrounding x read, x written on the block (bd complex each); inverse once per block
  const double bd = 2.0 * bs * bs, cs = sizeof(typename CT<R>::T), ar = act_rhs(nrhs);
  const double bytes = nb * (ar * (known == SAP_ZERO ? 2 : 3) * bd * cs + bd * bd * cs);
  const double flops = nb * ar * ((known == SAP_ZERO ? 0.0 : bs * bs * 56.0) + 8.0 * bd * bd);
  if (bs == 2) {
    MG_CHECK_ARG(known == SAP_X, "2 x 2 blocks read all of x");
    MG_LAUNCH_W(bytes, flops, k_sap_fine2<R>, nb, 256, 0, st, links, diag, L, inv, inv_transposed, f, x, color, nrhs,
                active);
    return;
  }
  if constexpr (sizeof(R) == 4) {
    MG_CHECK_ARG(inv_transposed, "the FP32 fine smoother reads transposed block inverses");
    const int nsm = sm_count();
    // tile of right-hand sides: 8 where that takes the batch, else 16.  A tile of 32 needs fewer reads of the
    // inverse per FMA but leaves 6 CTAs per SM instead of 10: 115 us against 100 at L = 512, 32 rhs.
    auto go = [&](auto rg) {
      constexpr int RG = decltype(rg)::value, sm = (int)sizeof(SapF<RG, false>);
      constexpr int per_sm = std::min(16, 227 * 1024 / (sm + 1024));
      const int ntile = (nrhs + RG - 1) / RG;
      const dim3 grid(std::max(1, std::min(nb, (nsm * per_sm + ntile - 1) / ntile)), ntile);
      ensure_max_smem((const void*)k_sap_fine4_fp32<RG, false>, sm);
      MG_LAUNCH_P(bytes, flops, (k_sap_fine4_fp32<RG, false>), grid, 64, sm, st, links, diag, L, inv, f, x, x, color,
                  nrhs, nb, known, active);
    };
    if (nrhs <= 8)
      go(std::integral_constant<int, 8>());
    else
      go(std::integral_constant<int, 16>());
  } else {
    // lattices with few blocks spread a batch over blockIdx.y, in tiles as small as give every SM eight CTAs (at least
    // two right-hand sides, one per warp); those with many keep the inverse in shared memory across the tiles
    const int nsm = sm_count();
    int tile = SF64_TILE;
    while (tile > 2 && (long)nb * cdiv(nrhs, tile) < 8L * nsm) tile /= 2;
    const dim3 grid(nb, nb >= 4096 ? 1 : cdiv(nrhs, tile));
    MG_LAUNCH_W(bytes, flops, k_sap_fine4_fp64, grid, 64, 0, st, links, L, inv, f, x, color, nrhs, tile, known, active);
  }
}
template void sap_half_fine<float>(cudaStream_t, const float2*, float, int, int, const float2*, const float2*,
                                   float2*, int, int, const int*, bool, int);
template void sap_half_fine<double>(cudaStream_t, const double2*, double, int, int, const double2*,
                                    const double2*, double2*, int, int, const int*, bool, int);

void residual_restrict_fine(cudaStream_t st, const float2* links, float diag, int L, const float2* P, const float2* x,
                            const float2* f, float2* xc, int nrhs, const int* active) {
  MG_CHECK_ARG(L % 4 == 0, "4 x 4 aggregates");
  if (nrhs <= 0) return;
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      const size_t n = 2 * (size_t)L * L;
      residual_restrict_fine(st, links, diag, L, P, x + r * n, f + r * n, xc + r * (n / 2), k, act);
    }
    return;
  }
  const int na = (L / 4) * (L / 4);
  const double ar = act_rhs(nrhs);
  const double bytes = na * (ar * (16 * 16 * 2 + 128.0) + 2048.0), flops = na * ar * (16 * 56.0 + 8.0 * 256);
  const int nsm = sm_count();
  auto go = [&](auto rg) {
    constexpr int RG = decltype(rg)::value, sm = (int)sizeof(SapF<RG, true>);
    constexpr int per_sm = std::min(16, 227 * 1024 / (sm + 1024));
    const int ntile = (nrhs + RG - 1) / RG;
    const dim3 grid(std::max(1, std::min(na, (nsm * per_sm + ntile - 1) / ntile)), ntile);
    ensure_max_smem((const void*)k_sap_fine4_fp32<RG, true>, sm);
    MG_LAUNCH_P(bytes, flops, (k_sap_fine4_fp32<RG, true>), grid, 64, sm, st, links, diag, L, P, f, x, xc, 0, nrhs, na,
                SAP_X, active);
  };
  if (nrhs <= 8)
    go(std::integral_constant<int, 8>());
  else
    go(std::integral_constant<int, 16>());
}

// out[b][j][i] = (float) in[b][i][j] for nb blocks of bd x bd
__global__ void k_blocks_to_fp32_transposed(const double2* __restrict__ in, int nb, int bd, float2* __restrict__ out) {
  const size_t total = (size_t)nb * bd * bd;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const size_t b = e / ((size_t)bd * bd);
    const int r = (int)(e - b * bd * bd), i = r / bd, j = r - i * bd;
    const double2 v = in[e];
    out[b * bd * bd + (size_t)j * bd + i] = make_float2((float)v.x, (float)v.y);
  }
}

void blocks_to_fp32_transposed(cudaStream_t st, const double2* in, int nb, int bd, float2* out) {
  MG_LAUNCH(k_blocks_to_fp32_transposed, 1024, 256, 0, st, in, nb, bd, out);
}

}  // namespace mg
