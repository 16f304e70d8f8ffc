// Coarse-level kernels: 5-point block stencil apply, SAP block matrices and
// smoother on coarse levels, aggregation restriction/prolongation (R = P^H,
// Section 3.1), the per-aggregate orthonormalisation of the test vectors and
// the Galerkin construction D_{l+1} = P_l^H D_l P_l, block by block.
//
// Stencil layout: st[site][dir][i][j], dir = 0 self, 1 +x, 2 -x, 3 +t, 4 -t;
// (D x)(s)_i = sum_dir sum_j st[s][dir][i][j] x(s + dir)_j, periodic (the
// fermion boundary sign is already inside the Galerkin blocks).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "ops.cuh"

namespace mg {

// two consecutive complex numbers (16-byte aligned in FP32)
__device__ __forceinline__ void load2(const float2* p, float2* v) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = make_float2(q.x, q.y);
  v[1] = make_float2(q.z, q.w);
}
__device__ __forceinline__ void load2(const double2* p, double2* v) { v[0] = p[0]; v[1] = p[1]; }
__device__ __forceinline__ void store2(float2* p, const float2* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
__device__ __forceinline__ void store2(double2* p, const double2* v) { p[0] = v[0]; p[1] = v[1]; }

__device__ __forceinline__ int nbr_site(int s, int dir, int Ls) {
  const int t = s / Ls, x = s - t * Ls;
  switch (dir) {
    case 1: return t * Ls + (x + 1 == Ls ? 0 : x + 1);
    case 2: return t * Ls + (x == 0 ? Ls - 1 : x - 1);
    case 3: return (t + 1 == Ls ? 0 : t + 1) * Ls + x;
    case 4: return (t == 0 ? Ls - 1 : t - 1) * Ls + x;
    default: return s;
  }
}

// ---- coarse stencil apply -----------------------------------------------------
// FP64, other block sizes than 16, FP32 vectors off a 16-byte boundary and small batches on few sites.
// CTA per site: the 5 stencil blocks (transposed in shared memory) are applied to the
// rhs in groups of 256 / d; DT = d at compile time (0: runtime d).
template <typename R, bool RES, int DT>
__global__ void __launch_bounds__(256) k_coarse_apply(const typename CT<R>::T* __restrict__ st, int Ls, int d_,
                                                      const typename CT<R>::T* __restrict__ x,
                                                      typename CT<R>::T* __restrict__ y,
                                                      const typename CT<R>::T* __restrict__ b, int nrhs,
                                                      const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  const int d = DT ? DT : d_;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sst = reinterpret_cast<C*>(smem_raw);  // [dir][j][i] (transposed)
  const int G = 256 / d;
  C* sx = sst + 5 * d * d;                  // [g][dir][j]
  const int s = blockIdx.x;
  const int dd = d * d;
  const C* S = st + (size_t)s * 5 * dd;
  for (int e = threadIdx.x; e < 5 * dd; e += 256) {
    const int dir = e / dd, r = e - dir * dd, i = r / d, j = r - i * d;
    sst[dir * dd + j * d + i] = S[e];
  }
  const size_t n = (size_t)Ls * Ls * d;
  const int g = threadIdx.x / d, i = threadIdx.x - g * d;
  for (int r0 = 0; r0 < nrhs; r0 += G) {
    __syncthreads();
    for (int q = threadIdx.x; q < G * 5 * d; q += 256) {
      const int gg = q / (5 * d), rem = q - gg * 5 * d, dir = rem / d, j = rem - dir * d;
      const int rhs = r0 + gg;
      if (rhs < nrhs && !(active && !active[rhs]))
        sx[q] = __ldg(x + rhs * n + (size_t)nbr_site(s, dir, Ls) * d + j);
    }
    __syncthreads();
    const int rhs = r0 + g;
    if (rhs < nrhs && !(active && !active[rhs])) {
      C acc = czero<C>();
#pragma unroll
      for (int dir = 0; dir < 5; ++dir) {
        const C* a = sst + dir * dd + i;
        const C* v = sx + (g * 5 + dir) * d;
#pragma unroll 16
        for (int j = 0; j < d; ++j) acc = cfma(a[j * d], v[j], acc);
      }
      const size_t o = rhs * n + (size_t)s * d + i;
      y[o] = RES ? csub(b[o], acc) : acc;
    }
  }
}

// FP32, 16 dof per site: one CTA per site and tile of RG right-hand sides, RI rows x 2 rhs per thread (64 threads), the
// blocks and the five neighbour slabs by cp.async.  Bound by what shared memory returns: one result per thread took 16
// bytes for 4 FMAs, 4 x 2 results take 96 for 64.  64 x 64 sites, 24 right-hand sides: 49 -> 41 us (17 TF; the tile of
// 32 holds 24); a copy of the blocks transposed on the way in, 49 (8-way bank conflicts).  Tiles of 16 up to 16
// right-hand sides, so that half a tile is not padding.
template <bool RES, int RG, int RI>
__global__ void __launch_bounds__(64) k_coarse_apply16(const float2* __restrict__ st, int Ls, const float2* __restrict__ x,
                                                       float2* __restrict__ y, const float2* __restrict__ b, int nrhs,
                                                       const int* __restrict__ active) {
  constexpr int XP = 18, NG = 16 / RI;  // padded slab row (16-byte aligned), row groups
  static_assert(NG * (RG / 2) == 64, "64 threads");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* sw = reinterpret_cast<float2*>(smem_raw);  // [dir][i][j]
  float2* sx = sw + 80 * XP;                         // [dir][rhs][j]
  const int s = blockIdx.x, r0 = blockIdx.y * RG, tid = threadIdx.x;
  const size_t n = (size_t)Ls * Ls * 16;
#pragma unroll 5
  for (int q = tid; q < 5 * RG * 8; q += 64) {
    const int c = q & 7, g = (q >> 3) % RG, dir = (q >> 3) / RG, rhs = r0 + g;
    if (rhs < nrhs && !(active && !active[rhs]))
      cp_async16(sx + (dir * RG + g) * XP + 2 * c, x + rhs * n + (size_t)nbr_site(s, dir, Ls) * 16 + 2 * c);
  }
#pragma unroll 5
  for (int q = tid; q < 640; q += 64)
    cp_async16(sw + (q >> 3) * XP + 2 * (q & 7), st + (size_t)s * 1280 + 2 * q);
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const int ig = tid % NG, g0 = tid / NG * 2;  // rows ig, ig + NG, ...: different banks
  float2 acc[RI][2];
#pragma unroll
  for (int u = 0; u < RI; ++u) acc[u][0] = acc[u][1] = make_float2(0.f, 0.f);
#pragma unroll
  for (int dir = 0; dir < 5; ++dir) {
#pragma unroll 4
    for (int j = 0; j < 16; j += 2) {
      float2 v[2][2];
      load2(sx + (dir * RG + g0) * XP + j, v[0]);
      load2(sx + (dir * RG + g0 + 1) * XP + j, v[1]);
#pragma unroll
      for (int u = 0; u < RI; ++u) {
        float2 m[2];
        load2(sw + (dir * 16 + ig + NG * u) * XP + j, m);
#pragma unroll
        for (int p = 0; p < 2; ++p) acc[u][p] = cfma(m[1], v[p][1], cfma(m[0], v[p][0], acc[u][p]));
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int rhs = r0 + g0 + p;
    if (rhs >= nrhs || (active && !active[rhs])) continue;
    const size_t o = rhs * n + (size_t)s * 16 + ig;
#pragma unroll
    for (int u = 0; u < RI; ++u) y[o + NG * u] = RES ? csub(b[o + NG * u], acc[u][p]) : acc[u][p];
  }
}

template <typename K>
static void set_smem_attr(K kernel) {
  ensure_max_smem((const void*)kernel, 200 * 1024);
}

template <typename R, bool RES>
static void coarse_apply_launch(cudaStream_t stm, const typename CT<R>::T* st, int Ls, int d,
                                const typename CT<R>::T* x, typename CT<R>::T* y, const typename CT<R>::T* b,
                                int nrhs, const int* active, size_t sm, double bytes, double flops) {
  if (d == 16) {
    set_smem_attr(k_coarse_apply<R, RES, 16>);
    MG_LAUNCH_W(bytes, flops, (k_coarse_apply<R, RES, 16>), Ls * Ls, 256, sm, stm, st, Ls, d, x, y, b, nrhs, active);
  } else {
    set_smem_attr(k_coarse_apply<R, RES, 0>);
    MG_LAUNCH_W(bytes, flops, (k_coarse_apply<R, RES, 0>), Ls * Ls, 256, sm, stm, st, Ls, d, x, y, b, nrhs, active);
  }
}

template <typename R>
void coarse_apply(cudaStream_t stm, const typename CT<R>::T* st, int Ls, int d, const typename CT<R>::T* x,
                  typename CT<R>::T* y, const typename CT<R>::T* b, int nrhs, const int* active) {
  typedef typename CT<R>::T C;
  MG_CHECK_ARG(d <= 64 && 256 % d == 0, "coarse dof must divide 256");
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      const size_t n = (size_t)Ls * Ls * d;
      coarse_apply<R>(stm, st, Ls, d, x + r * n, y + r * n, b ? b + r * n : nullptr, k, act);
    }
    return;
  }
  const int G = 256 / d;
  size_t sm = sizeof(C) * (5 * d * d + G * 5 * d);
  const double ns = (double)Ls * Ls, cs = sizeof(C), ar = act_rhs(nrhs);
  const double bytes = ar * ns * d * cs * (b ? 3 : 2) + ns * 5.0 * d * d * cs;
  const double flops = ar * ns * 8.0 * 5.0 * d * d;
  if constexpr (sizeof(R) == 4) {
    // 16-byte copies: other vectors take the general kernel, as do lattices of less than a site per SM up to 16
    // right-hand sides, where its 256 threads per site are the shorter chain (8 x 8 sites with 1, 16: 4.9, 6.2 us
    // against 6.2, 8.2; 16 x 16 sites 5.9, 8.2 against 6.2, 8.2)
    const bool few = Ls * Ls < sm_count() && nrhs <= 16;
    if (d == 16 && ((uintptr_t)x & 15) == 0 && !few) {
      auto go = [&](auto rg, auto ri) {
        constexpr int RG = decltype(rg)::value, RI = decltype(ri)::value, smb = (80 + 5 * RG) * 18 * 8;
        ensure_max_smem((const void*)k_coarse_apply16<false, RG, RI>, smb);
        ensure_max_smem((const void*)k_coarse_apply16<true, RG, RI>, smb);
        const dim3 grid(Ls * Ls, cdiv(nrhs, RG));
        if (b)
          MG_LAUNCH_W(bytes, flops, (k_coarse_apply16<true, RG, RI>), grid, 64, smb, stm, st, Ls, x, y, b, nrhs, active);
        else
          MG_LAUNCH_W(bytes, flops, (k_coarse_apply16<false, RG, RI>), grid, 64, smb, stm, st, Ls, x, y, b, nrhs, active);
      };
      if (nrhs <= 16)
        go(std::integral_constant<int, 16>(), std::integral_constant<int, 2>());
      else
        go(std::integral_constant<int, 32>(), std::integral_constant<int, 4>());
      return;
    }
  }
  if (b)
    coarse_apply_launch<R, true>(stm, st, Ls, d, x, y, b, nrhs, active, sm, bytes, flops);
  else
    coarse_apply_launch<R, false>(stm, st, Ls, d, x, y, b, nrhs, active, sm, bytes, flops);
}
template void coarse_apply<float>(cudaStream_t, const float2*, int, int, const float2*, float2*, const float2*,
                                  int, const int*);
template void coarse_apply<double>(cudaStream_t, const double2*, int, int, const double2*, double2*,
                                   const double2*, int, const int*);

// ---- SAP on coarse levels --------------------------------------------------------
// Block (BT, BX) of bs x bs sites, local index (jt * bs + jx) * d + k.
__global__ void k_coarse_blocks(const double2* __restrict__ st, int Ls, int d, int bs, double2* __restrict__ out) {
  const int nbx = Ls / bs;
  const int blk = blockIdx.x;
  const int BT = blk / nbx, BX = blk % nbx;
  const int ns = bs * bs, bd = ns * d, dd = d * d;
  double2* A = out + (size_t)blk * bd * bd;
  for (int e = threadIdx.x; e < bd * bd; e += blockDim.x) A[e] = make_double2(0, 0);
  __syncthreads();
  for (int j = 0; j < ns; ++j) {
    const int s = (BT * bs + j / bs) * Ls + BX * bs + j % bs;
    for (int dir = 0; dir < 5; ++dir) {
      const int nbs = nbr_site(s, dir, Ls);
      const int nt = nbs / Ls, nx = nbs % Ls;
      if (nt / bs != BT || nx / bs != BX) continue;
      const int jj = (nt % bs) * bs + nx % bs;
      const double2* S = st + ((size_t)s * 5 + dir) * dd;
      for (int e = threadIdx.x; e < dd; e += blockDim.x) {
        const int i = e / d, k = e % d;
        double2* a = A + (size_t)(j * d + i) * bd + jj * d + k;
        *a = cadd(*a, S[e]);
      }
      __syncthreads();
    }
  }
}

void coarse_block_matrices(cudaStream_t stm, const double2* st, int Ls, int d, int bs, double2* out) {
  const int nb = (Ls / bs) * (Ls / bs);
  MG_LAUNCH(k_coarse_blocks, nb, 256, 0, stm, st, Ls, d, bs, out);
}

// SAP half sweep.  The blocks of one colour do not couple, so with E the hops that leave the block
// x_B + D_BB^{-1} (f - D x)_B = D_BB^{-1} (f - E x)_B: the hops inside the block and the old x_B drop out (of the 5
// stencil blocks of a site in a 2 x 2 block 2 remain).  One CTA per block and tile of at most G right-hand sides; a
// thread owns one row of the block (lanes: consecutive rows) and every ng-th live right-hand side of the tile, up to 4:
// the remainder of a tile and right-hand sides that have stopped are not computed.
// FP64 is bound by its units (two FMAs a clock and SM, a share in each quarter): the rows of the inverse and the
// stencil come straight from global memory (32 lines per load, which costs an eighth of the FMAs they feed) and the
// CTA stays small, so that lattices with few blocks fill the chip (one 150 KB CTA of 4 rhs per SM before: 0.70 TF).
// FP32 stages both transposed in shared memory, by cp.async into rows padded by one.  Level 1 at L = 512 with 1, 8, 9,
// 64 right-hand sides, a sweep in FP64 1585, 1590, 3038, 12050 us with whole tiles of 8, now 222, 1590, 1733, 12050; in
// FP32 230, 254, 433, 1760 us with a transposing store that met in one bank, now 72, 117, 166, 789 (tiles of 16: 89,
// 144, 168, 888).
constexpr int SC_T = 128, SC_R = 4;
struct SapCoarseShape {
  int bs, d, bd, ng, G, GP, nslot;
  __host__ __device__ SapCoarseShape(int bs_, int d_) : bs(bs_), d(d_) {
    bd = bs * bs * d;
    ng = SC_T / bd;
    G = ng * SC_R;
    GP = G + 1;
    nslot = 4 * bs;
  }
  __host__ __device__ int complexes(bool stage) const {
    return bd * GP + nslot * d * GP + (stage ? bd * (bd + 1) + nslot * d * (d + 1) : 0);
  }
};

template <typename R, int BS, int DT>  // BS, DT: block side and dof at compile time (0: runtime)
__global__ void __launch_bounds__(SC_T) k_sap_coarse(const typename CT<R>::T* __restrict__ st, int Ls, int d_, int bs_,
                                                     const typename CT<R>::T* __restrict__ inv,
                                                     const typename CT<R>::T* __restrict__ f,
                                                     typename CT<R>::T* __restrict__ x, int color, int nrhs, bool zero,
                                                     const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  constexpr bool STAGE = sizeof(R) == 4;
  const SapCoarseShape sh(BS ? BS : bs_, DT ? DT : d_);
  const int bs = sh.bs, d = sh.d, bd = sh.bd, ng = sh.ng, GP = sh.GP, dd = d * d;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sres = reinterpret_cast<C*>(smem_raw);      // [row][group][its rhs]
  C* sx = sres + bd * GP;                        // [slot][k][group][its rhs]: x on the sites around the block
  C* sinv = sx + sh.nslot * d * GP;              // [column][row] (FP32), rows of bd + 1
  C* sst = sinv + bd * (bd + 1);                 // [slot][k][row of the site] (FP32), rows of d + 1
  __shared__ unsigned char srhs[SC_T / 2 * SC_R];  // live right-hand sides of the tile (r0 + this): number k is the
  __shared__ int scount;                           // (k / ng)-th of group k % ng.  Bytes: 8 FP64 CTAs fit an SM
  const int tid = threadIdx.x;
  const int nbx = Ls / bs, half = nbx / 2;
  const int BT = blockIdx.x / half;
  const int BX = 2 * (blockIdx.x - BT * half) + ((BT + color) & 1);
  const int t0 = BT * bs, x0 = BX * bs, r0 = blockIdx.y * sh.G;
  const size_t n = (size_t)Ls * Ls * d;
  const C* I = inv + (size_t)(BT * nbx + BX) * bd * bd;
  // slot: the -x, +x neighbours by row, then the -t, +t neighbours by column; the block's site and direction of each
  auto slot_site = [&](int s) {
    const int e = s / bs, i = s - e * bs;
    return e < 2 ? i * bs + (e ? bs - 1 : 0) : (e == 3 ? (bs - 1) * bs : 0) + i;
  };
  auto slot_dir = [&](int s) { const int e = s / bs; return e == 0 ? 2 : e == 1 ? 1 : e == 2 ? 4 : 3; };
  auto site_of = [&](int j) { return (t0 + j / bs) * Ls + x0 + j % bs; };
  if (STAGE) {
    for (int e = tid; e < bd * bd; e += SC_T) cp_async_elem(sinv + (e % bd) * (bd + 1) + e / bd, I + e);
    if (!zero)
      for (int e = tid; e < sh.nslot * dd; e += SC_T) {
        const int s = e / dd, r = e - s * dd;
        cp_async_elem(sst + (s * d + r % d) * (d + 1) + r / d,
                      st + ((size_t)site_of(slot_site(s)) * 5 + slot_dir(s)) * dd + r);
      }
  }
  if (tid < 32) {
    int k = 0;
    for (int b = 0; b < sh.G; b += 32) {
      const int rhs = r0 + b + tid;
      const bool on = b + tid < sh.G && rhs < nrhs && !(active && !active[rhs]);
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (on) srhs[k + __popc(m & ((1u << tid) - 1))] = (unsigned char)(b + tid);
      k += __popc(m);
    }
    if (tid == 0) scount = k;
  }
  __syncthreads();
  const int cnt = scount;
  if (!zero) {
    for (int q = tid; q < sh.nslot * cnt * d; q += SC_T) {
      const int k = q % d, g = (q / d) % cnt, s = q / (d * cnt);
      cp_async_elem(sx + (s * d + k) * GP + (g % ng) * SC_R + g / ng,
                    x + (r0 + srhs[g]) * n + (size_t)nbr_site(site_of(slot_site(s)), slot_dir(s), Ls) * d + k);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int row = tid % bd, grp = tid / bd, j = row / d, i = row - j * d;
  const bool mine = grp < ng;
  const int site = site_of(j);
  const int own = mine ? (cnt - grp + ng - 1) / ng : 0;         // right-hand sides of this thread
  const int most = __reduce_max_sync(0xffffffffu, own);         // and of its warp: blocks below 32 rows share one
  auto each = [&](auto&& f) {  // with the number of right-hand sides of the warp at compile time
    if (most == 1) f(std::integral_constant<int, 1>());
    else if (most == 2) f(std::integral_constant<int, 2>());
    else if (most == 3) f(std::integral_constant<int, 3>());
    else if (most == 4) f(std::integral_constant<int, 4>());
  };
  C fv[SC_R];
#pragma unroll
  for (int b = 0; b < SC_R; ++b)
    fv[b] = b < own ? f[(r0 + srhs[grp + b * ng]) * n + (size_t)site * d + i] : czero<C>();
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  each([&](auto nb) {
    constexpr int NB = decltype(nb)::value;
    if (!zero && mine) {
      const int jt = j / bs, jx = j % bs;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (!(e == 0 ? jx == 0 : e == 1 ? jx == bs - 1 : e == 2 ? jt == 0 : jt == bs - 1)) continue;
        const int s = e * bs + (e < 2 ? jt : jx);
        const C* w = STAGE ? sst + s * d * (d + 1) + i : st + ((size_t)site * 5 + slot_dir(s)) * dd + (size_t)i * d;
        const C* xv = sx + s * d * GP + grp * SC_R;
#pragma unroll 8
        for (int k = 0; k < d; ++k) {
          const C m = cneg(STAGE ? w[k * (d + 1)] : w[k]);
#pragma unroll
          for (int b = 0; b < NB; ++b) fv[b] = cfma(m, xv[k * GP + b], fv[b]);
        }
      }
    }
    if (mine)
#pragma unroll
      for (int b = 0; b < NB; ++b) sres[row * GP + grp * SC_R + b] = fv[b];
  });
  __syncthreads();
  if (!mine) return;
  each([&](auto nb) {
    constexpr int NB = decltype(nb)::value;
    C acc[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] = czero<C>();
    const C* rv = sres + grp * SC_R;
#pragma unroll 8
    for (int c = 0; c < bd; ++c) {
      const C m = STAGE ? sinv[c * (bd + 1) + row] : __ldg(I + (size_t)row * bd + c);
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[b] = cfma(m, rv[c * GP + b], acc[b]);
    }
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (b < own) x[(r0 + srhs[grp + b * ng]) * n + (size_t)site * d + i] = acc[b];
  });
}

template <typename R>
void sap_half_coarse(cudaStream_t stm, const typename CT<R>::T* st, int Ls, int d, int bs,
                     const typename CT<R>::T* inv, const typename CT<R>::T* f, typename CT<R>::T* x, int color,
                     int nrhs, const int* active, bool zero) {
  typedef typename CT<R>::T C;
  if (nrhs <= 0) return;
  const SapCoarseShape sh(bs, d);
  MG_CHECK_ARG(sh.bd <= 64, "coarse SAP blocks have at most 64 unknowns");
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      const size_t n = (size_t)Ls * Ls * d;
      sap_half_coarse<R>(stm, st, Ls, d, bs, inv, f + r * n, x + r * n, color, k, act, zero);
    }
    return;
  }
  const size_t sm = sizeof(C) * (size_t)sh.complexes(sizeof(R) == 4);
  const int nb = (Ls / bs) * (Ls / bs) / 2;
  const double cs = sizeof(C), ar = act_rhs(nrhs), ext = zero ? 0.0 : sh.nslot * (double)d * d;
  const double bytes = nb * (ar * (zero ? 2.0 : 3.0) * sh.bd * cs + ((double)sh.bd * sh.bd + ext) * cs);
  const double flops = nb * ar * 8.0 * (ext + (double)sh.bd * sh.bd);
  const dim3 grid(nb, cdiv(nrhs, sh.G));
  auto go = [&](auto bsc, auto dc) {
    constexpr int BS = decltype(bsc)::value, DT = decltype(dc)::value;
    ensure_max_smem((const void*)k_sap_coarse<R, BS, DT>, 120 * 1024);
    MG_LAUNCH_W(bytes, flops, (k_sap_coarse<R, BS, DT>), grid, SC_T, sm, stm, st, Ls, d, bs, inv, f, x, color, nrhs, zero,
                active);
  };
  typedef std::integral_constant<int, 2> I2;
  typedef std::integral_constant<int, 0> I0;
  // 2 x 2 blocks of 2, 4 and 8 test vectors per chirality at compile time: with 4 (L = 512, level 1, 1 and 64 FP32
  // right-hand sides) the index divisions of the runtime form made a sweep 42 and 350 us instead of 24 and 210
  if (bs == 2 && d == 16) go(I2(), std::integral_constant<int, 16>());
  else if (bs == 2 && d == 8) go(I2(), std::integral_constant<int, 8>());
  else if (bs == 2 && d == 4) go(I2(), std::integral_constant<int, 4>());
  else go(I0(), I0());
}
template void sap_half_coarse<float>(cudaStream_t, const float2*, int, int, int, const float2*, const float2*,
                                     float2*, int, int, const int*, bool);
template void sap_half_coarse<double>(cudaStream_t, const double2*, int, int, int, const double2*,
                                      const double2*, double2*, int, int, const int*, bool);

// ---- restriction / prolongation ---------------------------------------------------
// Aggregate (T, X) of agg x agg sites; block of chirality c has rows
// j = js * hd + k' (js = jt * agg + jx local site, hd = d / 2 dof per chirality)
// mapping to fine dof (site(js)) * d + c * hd + k'.  One CTA per aggregate, its P blocks
// in shared memory, rhs in groups.  DT / AT / NT = d / agg / ntv at compile time (0: runtime).
template <typename R, int DT, int AT, int NT>
__global__ void __launch_bounds__(256) k_restrict(const typename CT<R>::T* __restrict__ P, int Ls, int d_, int agg_,
                                                  int ntv_, const typename CT<R>::T* __restrict__ xf,
                                                  typename CT<R>::T* __restrict__ xc, int nrhs,
                                                  const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  const int d = DT ? DT : d_, agg = AT ? AT : agg_, ntv = NT ? NT : ntv_;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int hd = d / 2, na = agg * agg, bsz = na * hd, dc = 2 * ntv, fa = na * d;
  const int G = max(1, 256 / dc);
  C* sP = reinterpret_cast<C*>(smem_raw);  // [c][j][m]
  C* sx = sP + 2 * bsz * ntv;              // [g][js * d + k]
  const int Lc = Ls / agg;
  const int a = blockIdx.x, T = a / Lc, X = a - T * Lc;
  const C* Pa = P + (size_t)a * 2 * bsz * ntv;
  for (int e = threadIdx.x; e < 2 * bsz * ntv; e += 256) sP[e] = Pa[e];
  const size_t n = (size_t)Ls * Ls * d, nc = (size_t)Lc * Lc * dc;
  for (int r0 = 0; r0 < nrhs; r0 += G) {
    __syncthreads();
    for (int q = threadIdx.x; q < G * fa; q += 256) {
      const int g = q / fa, rem = q - g * fa, js = rem / d, k = rem - js * d;
      const int rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) {
        const int jt = js / agg, jx = js - jt * agg;
        const size_t site = (size_t)(agg * T + jt) * Ls + agg * X + jx;
        sx[q] = __ldg(xf + rhs * n + site * d + k);
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < G * dc; q += 256) {
      const int g = q / dc, o = q - g * dc, c = o / ntv, m = o - c * ntv;
      const int rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) {
        C acc = czero<C>();
        const C* pc = sP + (size_t)c * bsz * ntv + m;
        const C* xv = sx + g * fa + c * hd;
#pragma unroll 16
        for (int j = 0; j < bsz; ++j) {
          const int js = j / hd, kp = j - js * hd;
          acc = cfmac(pc[j * ntv], xv[js * d + kp], acc);
        }
        xc[rhs * nc + (size_t)a * dc + o] = acc;
      }
    }
  }
}

template <typename R, bool ADD>
__global__ void __launch_bounds__(256) k_prolong(const typename CT<R>::T* __restrict__ P, int Ls, int d, int agg,
                                                 int ntv, const typename CT<R>::T* __restrict__ xc,
                                                 typename CT<R>::T* __restrict__ xf,
                                                 unsigned short* __restrict__ xf16, int bf, int nrhs,
                                                 const int* __restrict__ active) {
  typedef typename CT<R>::T C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int hd = d / 2, na = agg * agg, bsz = na * hd, dc = 2 * ntv, fa = na * d;
  const int G = max(1, 256 / fa);
  C* sP = reinterpret_cast<C*>(smem_raw);  // [c][m][j] (transposed)
  C* sc = sP + 2 * bsz * ntv;              // [g][dc]
  const int Lc = Ls / agg;
  const int a = blockIdx.x, T = a / Lc, X = a - T * Lc;
  const C* Pa = P + (size_t)a * 2 * bsz * ntv;
  for (int e = threadIdx.x; e < 2 * bsz * ntv; e += 256) {
    const int c = e / (bsz * ntv), r = e - c * bsz * ntv, j = r / ntv, m = r - j * ntv;
    sP[(c * ntv + m) * bsz + j] = Pa[e];
  }
  const size_t n = (size_t)Ls * Ls * d, nc = (size_t)Lc * Lc * dc;
  for (int r0 = 0; r0 < nrhs; r0 += G) {
    __syncthreads();
    for (int q = threadIdx.x; q < G * dc; q += 256) {
      const int g = q / dc, o = q - g * dc;
      const int rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) sc[q] = __ldg(xc + rhs * nc + (size_t)a * dc + o);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < G * fa; q += 256) {
      const int g = q / fa, rem = q - g * fa, js = rem / d, k = rem - js * d;
      const int rhs = r0 + g;
      if (rhs < nrhs && !(active && !active[rhs])) {
        const int c = k / hd, kp = k - c * hd, j = js * hd + kp;
        C acc = czero<C>();
        const C* pc = sP + (size_t)c * ntv * bsz + j;
        const C* cv = sc + g * dc + c * ntv;
#pragma unroll 8
        for (int m = 0; m < ntv; ++m) acc = cfma(pc[m * bsz], cv[m], acc);
        const int jt = js / agg, jx = js - jt * agg;
        const size_t site = (size_t)(agg * T + jt) * Ls + agg * X + jx;
        C* p = xf + rhs * n + site * d + k;
        const C v = ADD ? cadd(*p, acc) : acc;
        *p = v;
        if constexpr (sizeof(R) == 4) {
          if (xf16) {  // planar 16-bit copy of an FP32 coarse vector: Re parts of the site's d dofs, then Im
            unsigned short* p16 = xf16 + 2 * (rhs * n + site * d) + k;
            p16[0] = bf == 2 ? __half_as_ushort(__float2half_rn(v.x)) : __bfloat16_as_ushort(__float2bfloat16_rn(v.x));
            p16[d] = bf == 2 ? __half_as_ushort(__float2half_rn(v.y)) : __bfloat16_as_ushort(__float2bfloat16_rn(v.y));
          }
        }
      }
    }
  }
}

// The default hierarchy (4 x 4 aggregates, 8 test vectors per chirality: fine d = 2, coarse d = 16) has kernels of its
// own below: register tiles instead of one result per thread (whose two shared-memory reads per multiply-add and two
// barriers per 16 right-hand sides were the time), the sums in the same order.

// xc = P^H xf from a coarse level: 16 outputs x RG right-hand sides per CTA, MM x RR of them per thread, 256 products
// each.  half: xf is zero on the 2 x 2 blocks of colour 1 (and not read there).
template <typename R, int RG, int MM, int RR>
__global__ void __launch_bounds__(16 / MM * (RG / RR))
    k_restrict16(const typename CT<R>::T* __restrict__ P, int Ls, const typename CT<R>::T* xf,
                 typename CT<R>::T* __restrict__ xc, bool half, int nrhs, const int* active) {
  pdl_begin();
  typedef typename CT<R>::T C;
  constexpr int T = 16 / MM * (RG / RR), XP = 256 + 16 / (int)sizeof(C);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sP = reinterpret_cast<C*>(smem_raw);  // [chirality][row][vector]
  C* sx = sP + 2048;                       // [rhs][site][dof]
  const int Lc = Ls / 4, a = blockIdx.x, AT = a / Lc, AX = a - AT * Lc, r0 = blockIdx.y * RG, tid = threadIdx.x;
  const size_t n = (size_t)Ls * Ls * 16, nc = (size_t)Lc * Lc * 16;
  const char* Pa = reinterpret_cast<const char*>(P + (size_t)a * 2048);
  constexpr int CPS = 16 * (int)sizeof(C) / 16;  // 16-byte chunks of a site
  for (int q = tid; q < 2048 * (int)sizeof(C) / 16; q += T)
    cp_async16(reinterpret_cast<char*>(sP) + q * 16, Pa + q * 16);
  for (int q = tid; q < RG * 16 * CPS; q += T) {
    const int c = q % CPS, js = (q / CPS) & 15, g = q / (16 * CPS), rhs = r0 + g;
    if (rhs < nrhs && !(active && !active[rhs]) && !(half && (((js >> 3) + (js >> 1)) & 1))) {
      const size_t site = (size_t)(4 * AT + (js >> 2)) * Ls + 4 * AX + (js & 3);
      cp_async16(reinterpret_cast<char*>(sx + g * XP + js * 16) + c * 16,
                  reinterpret_cast<const char*>(xf + rhs * n + site * 16) + c * 16);
    }
  }
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  const int op = tid % (16 / MM), o = op * MM, c = o >> 3, m = o & 7, g0 = tid / (16 / MM) * RR;
  if (r0 + g0 >= nrhs) return;  // the rest of the last tile: whole warps but one
  C acc[MM][RR];
#pragma unroll
  for (int u = 0; u < MM; ++u)
#pragma unroll
    for (int b = 0; b < RR; ++b) acc[u][b] = czero<C>();
  for (int js = 0; js < 16; ++js) {
    if (half && (((js >> 3) + (js >> 1)) & 1)) continue;
    const C* p = sP + (c * 128 + js * 8) * 8 + m;
    const C* v = sx + g0 * XP + js * 16 + c * 8;
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int u = 0; u < MM; ++u) {
        const C pv = p[k * 8 + u];
#pragma unroll
        for (int b = 0; b < RR; ++b) acc[u][b] = cfmac(pv, v[b * XP + k], acc[u][b]);
      }
  }
#pragma unroll
  for (int b = 0; b < RR; ++b) {
    const int rhs = r0 + g0 + b;
    if (rhs < nrhs && !(active && !active[rhs]))
#pragma unroll
      for (int u = 0; u < MM; ++u) xc[rhs * nc + (size_t)a * 16 + o + u] = acc[u][b];
  }
}

// xf (+)= P xc.  A thread keeps the rows of P of its two consecutive dofs in registers (D = 16: one chirality; D = 2:
// both spins of a site; FP64 with D = 2 of one dof, so that a warp has one right-hand side and an odd one costs no more)
// and takes right-hand sides of the tile in turn, up to the last one; xc comes from shared memory.
// D = 2: a row of P serves the 8 threads of its site, so P goes through shared memory too (rows padded: their 16-byte
// reads fall into different banks); reading it from global memory in every thread was 16 loads for one or two results.
// L = 512 with 1, 8, 32 right-hand sides: FP32 20, 66, 108 -> 19, 22, 57 us, FP64 60, 226, 882 -> 33, 224, 876.
// D = 16 with xf16: the planar 16-bit copy is written alongside.
template <typename R, bool ADD, int D, int RG>
__global__ void __launch_bounds__(128) k_prolong2(const typename CT<R>::T* __restrict__ P, int Ls,
                                                  const typename CT<R>::T* xc,
                                                  typename CT<R>::T* xf, unsigned short* __restrict__ xf16,
                                                  int bf, int nrhs, const int* active) {
  pdl_begin();
  typedef typename CT<R>::T C;
  constexpr int DPT = D == 2 && sizeof(R) == 8 ? 1 : 2;  // dofs per thread
  constexpr int TPR = 16 * D / DPT, RS = 128 / TPR;      // threads per rhs, rhs taken at once
  constexpr int ROWS = 8 * D;                            // rows of a chirality block
  constexpr int PP = 8 + 16 / (int)sizeof(C);            // padded row of P
  __shared__ __align__(16) C sc[RG][16];
  __shared__ __align__(16) C sp[D == 2 ? 32 * PP : 1];
  const int Lc = Ls / 4, a = blockIdx.x, AT = a / Lc, AX = a - AT * Lc, r0 = blockIdx.y * RG, tid = threadIdx.x;
  const int cnt = min(RG, nrhs - r0);
  const size_t n = (size_t)Ls * Ls * D, nc = (size_t)Lc * Lc * 16;
  const C* Pa = P + (size_t)a * 2 * ROWS * 8;
  if constexpr (D == 2) {
    constexpr int CPR = 8 * (int)sizeof(C) / 16;  // 16-byte chunks of a row
    for (int q = tid; q < 32 * CPR; q += 128)
      cp_async16(reinterpret_cast<char*>(sp + q / CPR * PP) + q % CPR * 16, reinterpret_cast<const char*>(Pa) + q * 16);
  }
  for (int q = tid; q < cnt * 16; q += 128) {
    const int rhs = r0 + (q >> 4);
    if (!(active && !active[rhs])) cp_async_elem(&sc[q >> 4][q & 15], xc + rhs * nc + (size_t)a * 16 + (q & 15));
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int dof = DPT * (tid % TPR), js = dof / D, k = dof % D, rs = tid / TPR;  // first dof of the thread
  const int c0 = D == 2 ? k : k >> 3;                                            // its chirality
  constexpr int CS = D == 2 ? 1 : 0;                                             // step of the chirality to the next
  C w[DPT][8];
  if constexpr (D == 16) {
#pragma unroll
    for (int u = 0; u < DPT; ++u)
#pragma unroll
      for (int m = 0; m < 8; m += 2) load2(Pa + (c0 * ROWS + js * 8 + (k & 7) + u) * 8 + m, w[u] + m);
  }
  const size_t off = ((size_t)(4 * AT + (js >> 2)) * Ls + 4 * AX + (js & 3)) * D + k;
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if constexpr (D == 2) {
#pragma unroll
    for (int u = 0; u < DPT; ++u)
#pragma unroll
      for (int m = 0; m < 8; m += 2) load2(sp + ((c0 + u) * 16 + js) * PP + m, w[u] + m);
  }
#pragma unroll 4
  for (int g = rs; g < cnt; g += RS) {
    const int rhs = r0 + g;
    if (active && !active[rhs]) continue;
    C* px = xf + rhs * n + off;
    C v[DPT], acc[DPT];
    if constexpr (ADD && DPT == 2) load2(px, v);
    if constexpr (ADD && DPT == 1) v[0] = px[0];
#pragma unroll
    for (int u = 0; u < DPT; ++u) acc[u] = czero<C>();
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int u = 0; u < DPT; ++u) acc[u] = cfma(w[u][m], sc[g][(c0 + u * CS) * 8 + m], acc[u]);
#pragma unroll
    for (int u = 0; u < DPT; ++u) v[u] = ADD ? cadd(v[u], acc[u]) : acc[u];
    if constexpr (DPT == 2)
      store2(px, v);
    else
      px[0] = v[0];
    if constexpr (sizeof(R) == 4 && D == 16) {
      if (xf16) {  // Re parts of the site's 16 dofs, then the Im parts
        unsigned* p16 = reinterpret_cast<unsigned*>(xf16 + 2 * (rhs * n + off - k) + k);
        auto pack = [&](float x, float y) {
          auto b16 = [&](float f) -> unsigned {
            return bf == 2 ? __half_as_ushort(__float2half_rn(f)) : __bfloat16_as_ushort(__float2bfloat16_rn(f));
          };
          return b16(x) | b16(y) << 16;
        };
        p16[0] = pack(v[0].x, v[1].x);
        p16[8] = pack(v[0].y, v[1].y);
      }
    }
  }
}

// right-hand sides on the fullest SM where every aggregate has a CTA per tile of rg of them
static long fullest_sm(int aggs, int nrhs, int rg, int nsm) {
  return (long)cdiv((long)aggs * (nrhs / rg), nsm) * rg + (long)cdiv(aggs, nsm) * (nrhs % rg);
}

template <typename R>
void restrict_op(cudaStream_t stm, const typename CT<R>::T* P, int Ls, int d, int agg, int ntv,
                 const typename CT<R>::T* xf, typename CT<R>::T* xc, int nrhs, const int* active, bool half) {
  typedef typename CT<R>::T C;
  if (nrhs <= 0) return;
  const int na = agg * agg, bsz = na * d / 2, dc = 2 * ntv;
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      const size_t nf = (size_t)Ls * Ls * d;
      restrict_op<R>(stm, P, Ls, d, agg, ntv, xf + r * nf, xc + r * (nf / (na * d) * dc), k, act, half);
    }
    return;
  }
  const int Lc = Ls / agg;
  const double nag = (double)Lc * Lc, cs = sizeof(C), ar = act_rhs(nrhs);
  const double bytes = nag * (ar * (na * d * (half ? 0.5 : 1.0) + dc) * cs + 2.0 * bsz * ntv * cs);
  const double flops = nag * ar * 8.0 * 2.0 * bsz * ntv * (half ? 0.5 : 1.0);
  const bool aligned = ((uintptr_t)xf & 15) == 0;  // 16-byte copies; other vectors take the general kernel
  if (agg == 4 && ntv == 8 && d == 16 && aligned) {
    // FP32 2 x 2 results a thread (two 16-byte and two 8-byte reads for 16 FMAs), FP64 one (its units are the bound);
    // up to 4 right-hand sides in a tile of their own, whose shared memory lets twice the CTAs in (L = 512, level 1,
    // one right-hand side: FP32 14.6 -> 5.3 us, FP64 117 -> 41 us).
    auto go = [&](auto rg, auto mm) {
      constexpr int RG = decltype(rg)::value, MM = decltype(mm)::value;
      constexpr int T = 16 / MM * (RG / MM), sm = (int)sizeof(C) * (2048 + RG * (256 + 16 / (int)sizeof(C)));
      ensure_max_smem((const void*)k_restrict16<R, RG, MM, MM>, sm);
      MG_LAUNCH_PE(early_launch<R>(bytes, flops), bytes, flops, (k_restrict16<R, RG, MM, MM>),
                   dim3(Lc * Lc, cdiv(nrhs, RG)), T, sm, stm, P, Ls, xf, xc, half, nrhs, active);
    };
    // FP64 with few aggregates: the tile whose fullest SM has the fewer right-hand sides (64 aggregates with 32, 48, 64:
    // 37, 52, 72 us in tiles of 4, 8, 4; 51, 52, 72 before)
    const int aggs = Lc * Lc, nsm = sm_count();
    const bool small = nrhs <= 4 || (sizeof(R) == 8 && aggs * cdiv(nrhs, 8) < 4 * nsm &&
                                     fullest_sm(aggs, nrhs, 4, nsm) < fullest_sm(aggs, nrhs, 8, nsm));
    typedef std::integral_constant<int, 1> I1;
    if (small)
      go(std::integral_constant<int, 4>(), I1());
    else if constexpr (sizeof(R) == 4)
      go(std::integral_constant<int, 16>(), std::integral_constant<int, 2>());
    else
      go(std::integral_constant<int, 8>(), I1());
    return;
  }
  MG_CHECK_ARG(!half, "half restriction: 4 x 4 aggregates of 16 dof, aligned vectors");
  const int G = std::max(1, 256 / dc);
  const size_t sm = sizeof(C) * ((size_t)2 * bsz * ntv + (size_t)G * na * d);
  if (agg == 4 && ntv == 8 && d == 2) {
    set_smem_attr(k_restrict<R, 2, 4, 8>);
    MG_LAUNCH_W(bytes, flops, (k_restrict<R, 2, 4, 8>), Lc * Lc, 256, sm, stm, P, Ls, d, agg, ntv, xf, xc, nrhs,
                active);
  } else {
    set_smem_attr(k_restrict<R, 0, 0, 0>);
    MG_LAUNCH_W(bytes, flops, (k_restrict<R, 0, 0, 0>), Lc * Lc, 256, sm, stm, P, Ls, d, agg, ntv, xf, xc, nrhs,
                active);
  }
}

template <typename R, bool ADD>
static void prolong_launch(cudaStream_t stm, const typename CT<R>::T* P, int Ls, int d, int agg, int ntv,
                           const typename CT<R>::T* xc, typename CT<R>::T* xf, unsigned short* xf16, int bf,
                           int nrhs, const int* active, double bytes, double flops) {
  typedef typename CT<R>::T C;
  const int Lc = Ls / agg;
  auto go = [&](auto dd, auto rg) {
    constexpr int D = decltype(dd)::value, RG = decltype(rg)::value;
    MG_LAUNCH_PE(early_launch<R>(bytes, flops), bytes, flops, (k_prolong2<R, ADD, D, RG>),
                 dim3(Lc * Lc, cdiv(nrhs, RG)), 128, 0, stm, P, Ls, xc, xf, xf16, bf, nrhs, active);
  };
  typedef std::integral_constant<int, 8> I8;
  typedef std::integral_constant<int, 32> I32;
  const bool aligned = ((uintptr_t)xf & 15) == 0;  // 16-byte accesses; other vectors take the general kernel
  const int aggs = Lc * Lc, nsm = sm_count();
  // tiles of 8 or 32: FP64 the one whose fullest SM has the fewer right-hand sides (8 while that leaves SMs without a
  // tile; of equals 8 for even numbers of whole tiles: 256 fine aggregates with 16, 24 right-hand sides 10.5, 18.1 us in
  // tiles of 8 and 13.9, 14.2 in tiles of 32); FP32 8 for few aggregates, which spreads a batch over more CTAs
  const long f8 = fullest_sm(aggs, nrhs, 8, nsm), f32 = fullest_sm(aggs, nrhs, 32, nsm);
  const bool tile8 = nrhs <= 8 || (sizeof(R) == 4 ? d == 16 && aggs * cdiv(nrhs, 32) < 4 * nsm
                                                  : aggs * cdiv(nrhs, 8) <= nsm || f8 < f32 || (f8 == f32 && nrhs % 16 == 0));
  if (agg == 4 && ntv == 8 && d == 2 && aligned) {
    tile8 ? go(std::integral_constant<int, 2>(), I8()) : go(std::integral_constant<int, 2>(), I32());
  } else if (agg == 4 && ntv == 8 && d == 16 && aligned) {
    tile8 ? go(std::integral_constant<int, 16>(), I8()) : go(std::integral_constant<int, 16>(), I32());
  } else {
    const int na = agg * agg, bsz = na * d / 2, dc = 2 * ntv, G = std::max(1, 256 / (na * d));
    const size_t sm = sizeof(C) * ((size_t)2 * bsz * ntv + (size_t)G * dc);
    set_smem_attr(k_prolong<R, ADD>);
    MG_LAUNCH_W(bytes, flops, (k_prolong<R, ADD>), Lc * Lc, 256, sm, stm, P, Ls, d, agg, ntv, xc, xf,
                xf16, bf, nrhs, active);
  }
}

template <typename R>
void prolong_op(cudaStream_t stm, const typename CT<R>::T* P, int Ls, int d, int agg, int ntv,
                const typename CT<R>::T* xc, typename CT<R>::T* xf, bool add, int nrhs, const int* active,
                void* xf16, int bf) {
  MG_CHECK_ARG(!xf16 || (sizeof(R) == 4 && (bf == 1 || bf == 2)), "16-bit copy: FP32 vectors, BF16 or FP16");
  typedef typename CT<R>::T C;
  if (nrhs <= 0) return;
  const int na = agg * agg, bsz = na * d / 2, dc = 2 * ntv, fa = na * d;
  if (nrhs > RHS_SLICE) {
    for (int r = 0; r < nrhs; r += RHS_SLICE) {
      const int k = std::min(RHS_SLICE, nrhs - r);
      const int* act = active ? active + r : nullptr;
      const size_t nf = (size_t)Ls * Ls * d;
      prolong_op<R>(stm, P, Ls, d, agg, ntv, xc + r * (nf / fa * dc), xf + r * nf, add, k, act,
                    xf16 ? (unsigned short*)xf16 + 2 * r * nf : nullptr, bf);
    }
    return;
  }
  const int Lc = Ls / agg;
  const double nag = (double)Lc * Lc, cs = sizeof(C), ar = act_rhs(nrhs);
  const double bytes = nag * (ar * ((add ? 2.0 : 1.0) * fa + dc) * cs + 2.0 * bsz * ntv * cs) +
                       (xf16 ? nag * ar * fa * 4.0 : 0.0);
  const double flops = nag * ar * 8.0 * 2.0 * bsz * ntv;
  unsigned short* x16 = (unsigned short*)xf16;
  if (add)
    prolong_launch<R, true>(stm, P, Ls, d, agg, ntv, xc, xf, x16, bf, nrhs, active, bytes, flops);
  else
    prolong_launch<R, false>(stm, P, Ls, d, agg, ntv, xc, xf, x16, bf, nrhs, active, bytes, flops);
}
template void restrict_op<float>(cudaStream_t, const float2*, int, int, int, int, const float2*, float2*, int,
                                 const int*, bool);
template void restrict_op<double>(cudaStream_t, const double2*, int, int, int, int, const double2*, double2*, int,
                                  const int*, bool);
template void prolong_op<float>(cudaStream_t, const float2*, int, int, int, int, const float2*, float2*, bool, int,
                                const int*, void*, int);
template void prolong_op<double>(cudaStream_t, const double2*, int, int, int, int, const double2*, double2*, bool,
                                 int, const int*, void*, int);

// ---- test vectors -> prolongator blocks --------------------------------------------
__global__ void k_gather_tv(const double2* __restrict__ V, int Ls, int d, int agg, int ntv, double2* __restrict__ P) {
  const int hd = d / 2, na = agg * agg, bsz = na * hd;
  const int Lc = Ls / agg;
  const size_t total = (size_t)Lc * Lc * 2 * bsz * ntv;
  const size_t n = (size_t)Ls * Ls * d;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int m = e % ntv;
    const size_t r = e / ntv;
    const int j = r % bsz;
    const size_t r2 = r / bsz;
    const int c = r2 % 2;
    const int a = (int)(r2 / 2), T = a / Lc, X = a % Lc;
    const int js = j / hd, kp = j % hd;
    const size_t site = (size_t)(agg * T + js / agg) * Ls + agg * X + js % agg;
    P[e] = V[m * n + site * d + c * hd + kp];
  }
}

void gather_tv_blocks(cudaStream_t stm, const double2* V, int Ls, int d, int agg, int ntv, double2* P) {
  MG_LAUNCH(k_gather_tv, 1024, 256, 0, stm, V, Ls, d, agg, ntv, P);
}

// Modified Gram-Schmidt with one re-orthogonalisation pass, one warp per block:
// Q has orthonormal columns and R a real positive diagonal (the QR normalisation
// of the oracle), FP64.
__global__ void k_orthonormalise(double2* __restrict__ P, int nblocks, int bsz, int ntv, int* fail) {
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (w >= nblocks) return;
  double2* B = P + (size_t)w * bsz * ntv;  // B[j][m]
  for (int m = 0; m < ntv; ++m) {
    for (int pass = 0; pass < 2; ++pass) {
      for (int i = 0; i < m; ++i) {
        double2 acc = make_double2(0, 0);
        for (int j = lane; j < bsz; j += 32) acc = cfmac(B[j * ntv + i], B[j * ntv + m], acc);
        for (int o = 16; o; o >>= 1) {
          acc.x += __shfl_xor_sync(0xffffffff, acc.x, o);
          acc.y += __shfl_xor_sync(0xffffffff, acc.y, o);
        }
        for (int j = lane; j < bsz; j += 32) B[j * ntv + m] = csub(B[j * ntv + m], cmul(B[j * ntv + i], acc));
        __syncwarp();
      }
    }
    double nr = 0;
    for (int j = lane; j < bsz; j += 32) {
      double2 v = B[j * ntv + m];
      nr += v.x * v.x + v.y * v.y;
    }
    for (int o = 16; o; o >>= 1) nr += __shfl_xor_sync(0xffffffff, nr, o);
    if (!(nr > 0.0)) {
      if (lane == 0) atomicExch(fail, 1);
      return;
    }
    const double inv = 1.0 / sqrt(nr);
    for (int j = lane; j < bsz; j += 32) B[j * ntv + m] = cscale(B[j * ntv + m], inv);
    __syncwarp();
  }
}

// The same for NTV columns with the block in registers: LPB lanes hold four rows each (LPB = bsz / 4: 4 on the fine
// level, 32 above), so a warp works on 32 / LPB blocks and a dot product takes 16 FMAs and log2(LPB) shuffles of all
// of them (with one block per warp the FP64 additions of the shuffles were the work: 3.1 ms of the set-up at L = 512).
template <int NTV, int LPB>
__global__ void __launch_bounds__(128) k_orthonormalise_reg(double2* __restrict__ P, int nblocks, int* fail) {
  constexpr int BSZ = 4 * LPB;
  const int t = blockIdx.x * 128 + threadIdx.x, blk = t / LPB, l = t % LPB;
  const bool on = blk < nblocks;
  double2* B = P + (size_t)(on ? blk : 0) * BSZ * NTV;
  double2 v[NTV][4];  // rows l, l + LPB, ..
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int m = 0; m < NTV; ++m) v[m][r] = B[(l + r * LPB) * NTV + m];
  auto sum = [](double s) {
#pragma unroll
    for (int o = LPB / 2; o; o >>= 1) s += __shfl_xor_sync(0xffffffff, s, o);
    return s;
  };
  bool bad = false;
#pragma unroll
  for (int m = 0; m < NTV; ++m) {
#pragma unroll
    for (int pass = 0; pass < 2; ++pass)
#pragma unroll
      for (int i = 0; i < m; ++i) {
        double2 a = make_double2(0, 0);
#pragma unroll
        for (int r = 0; r < 4; ++r) a = cfmac(v[i][r], v[m][r], a);
        a.x = -sum(a.x);
        a.y = -sum(a.y);
#pragma unroll
        for (int r = 0; r < 4; ++r) v[m][r] = cfma(v[i][r], a, v[m][r]);
      }
    double nr = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) nr = fma(v[m][r].x, v[m][r].x, fma(v[m][r].y, v[m][r].y, nr));
    nr = sum(nr);
    bad |= !(nr > 0.0);
    const double inv = 1.0 / sqrt(nr);
#pragma unroll
    for (int r = 0; r < 4; ++r) v[m][r] = cscale(v[m][r], inv);
  }
  if (!on) return;
  if (bad && l == 0) atomicExch(fail, 1);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int m = 0; m < NTV; ++m) B[(l + r * LPB) * NTV + m] = v[m][r];
}

void orthonormalise_blocks(cudaStream_t stm, double2* P, int nblocks, int bsz, int ntv, int* fail) {
  if (ntv == 8 && bsz == 16)
    MG_LAUNCH((k_orthonormalise_reg<8, 4>), cdiv(nblocks * 4L, 128), 128, 0, stm, P, nblocks, fail);
  else if (ntv == 8 && bsz == 128)
    MG_LAUNCH((k_orthonormalise_reg<8, 32>), cdiv(nblocks * 32L, 128), 128, 0, stm, P, nblocks, fail);
  else
    MG_LAUNCH(k_orthonormalise, cdiv(nblocks, 4), 128, 0, stm, P, nblocks, bsz, ntv, fail);
}

// ---- Galerkin coarse operator ------------------------------------------------------
// D_{l+1} = P^H D_l P (Section 3.1), one CTA per coarse site B, block by block: for every fine
// site s of aggregate B and stencil direction f, with s' the f-neighbour of s,
//   D_{l+1}[B, f or self] += P(s)^H D_l(s, f) P(s'),
// where P(s) (d x dc) is block diagonal in chirality and s' lies in B itself or in the aggregate
// adjacent to B in direction f (a fine hop crosses only the aggregate face it points to).  The products
// D_l(s, f) P(s') of the directions that stay in B are summed before P(s)^H multiplies them, so a site of a 4 x 4
// aggregate takes two products with P^H on average instead of five (FP64 is bound by its two FMAs a clock and SM).
__device__ __forceinline__ void wilson_hop(const double2* __restrict__ lk, double diag, int L, int s, int f,
                                           double2* M) {
  double2 w;
  switch (f) {
    case 0:
      M[0] = make_double2(diag, 0); M[1] = make_double2(0, 0);
      M[2] = make_double2(0, 0); M[3] = make_double2(diag, 0);
      return;
    case 1:  // +x: (1 - sigma_1) W_0(s)
      w = lk[2 * s];
      M[0] = w; M[1] = cneg(w); M[2] = cneg(w); M[3] = w;
      return;
    case 2:  // -x: (1 + sigma_1) conj(W_0(s - x))
      w = cconj(lk[2 * nbr_site(s, 2, L)]);
      M[0] = w; M[1] = w; M[2] = w; M[3] = w;
      return;
    case 3:  // +t: (1 - sigma_2) W_1(s)
      w = lk[2 * s + 1];
      M[0] = w; M[1] = cmuli(w); M[2] = cmulmi(w); M[3] = w;
      return;
    default:  // -t: (1 + sigma_2) conj(W_1(s - t))
      w = cconj(lk[2 * nbr_site(s, 4, L) + 1]);
      M[0] = w; M[1] = cmulmi(w); M[2] = cmuli(w); M[3] = w;
      return;
  }
}

constexpr int GAL_T = 256;   // threads per coarse site
constexpr int GAL_E = 4;     // coarse block entries per thread (dc <= 32)

template <bool WILSON>
__global__ void __launch_bounds__(GAL_T) k_galerkin(const double2* __restrict__ A, double diag, int Ls, int d,
                                                    int agg, int ntv, const double2* __restrict__ P,
                                                    double2* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int hd = d / 2, na = agg * agg, bsz = na * hd, dc = 2 * ntv, Lc = Ls / agg;
  const int dd = d * d, ddc = d * dc, dcc = dc * dc;
  double2* sA = reinterpret_cast<double2*>(smem_raw);  // [f][r][k]   D_l(s, f)
  double2* sT = sA + 5 * dd;                            // [c][r][j]   D_l(s, f) P(s'_f): c = 0 sum inside B, else f = c
  __shared__ int s_nb[5], s_js[5];                      // aggregate and local site of s'_f
  const int B = blockIdx.x, BT = B / Lc, BX = B % Lc;
  const size_t pblk = (size_t)2 * bsz * ntv;
  const double2* PB = P + (size_t)B * pblk;
  double2 acc[5][GAL_E];
#pragma unroll
  for (int c = 0; c < 5; ++c)
#pragma unroll
    for (int q = 0; q < GAL_E; ++q) acc[c][q] = make_double2(0, 0);
  for (int js = 0; js < na; ++js) {
    const int s = (BT * agg + js / agg) * Ls + BX * agg + js % agg;
    bool inside[5];  // s'_f in B: the f contribution goes to the self block
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const int s2 = nbr_site(s, f, Ls), t2 = s2 / Ls, x2 = s2 % Ls;
      inside[f] = (t2 / agg) * Lc + x2 / agg == B;
    }
    __syncthreads();  // the previous site's sA / sT / s_nb / s_js are consumed
    if (threadIdx.x < 5) {
      const int s2 = nbr_site(s, threadIdx.x, Ls), t2 = s2 / Ls, x2 = s2 % Ls;
      s_nb[threadIdx.x] = (t2 / agg) * Lc + x2 / agg;
      s_js[threadIdx.x] = (t2 % agg) * agg + x2 % agg;
    }
    if (WILSON) {
      if (threadIdx.x < 5) wilson_hop(A, diag, Ls, s, threadIdx.x, sA + threadIdx.x * 4);
    } else {
      const double2* As = A + (size_t)s * 5 * dd;
      for (int e = threadIdx.x; e < 5 * dd; e += GAL_T) sA[e] = __ldg(As + e);
    }
    __syncthreads();
    if (WILSON) {  // few products per site: the five directions in parallel, then the sum
      for (int e5 = threadIdx.x; e5 < 5 * ddc; e5 += GAL_T) {
        const int f = e5 / ddc, e = e5 - f * ddc, r = e / dc, j = e % dc, cj = j / ntv, m = j % ntv;
        const double2* p = P + (size_t)s_nb[f] * pblk + ((size_t)cj * bsz + s_js[f]) * ntv + m;
        sT[e5] = cmul(sA[f * dd + r * d + cj], __ldg(p));
      }
      __syncthreads();
      for (int e = threadIdx.x; e < ddc; e += GAL_T) {
        double2 self = sT[e];
#pragma unroll
        for (int f = 1; f < 5; ++f)
          if (inside[f]) self = cadd(self, sT[f * ddc + e]);
        sT[e] = self;
      }
    } else {
      for (int e = threadIdx.x; e < ddc; e += GAL_T) {
        const int r = e / dc, j = e % dc, cj = j / ntv, m = j % ntv;
        double2 self = make_double2(0, 0);
#pragma unroll
        for (int f = 0; f < 5; ++f) {
          const double2* p = P + (size_t)s_nb[f] * pblk + ((size_t)cj * bsz + s_js[f] * hd) * ntv + m;
          const double2* a = sA + f * dd + r * d + cj * hd;
          double2 t = inside[f] ? self : make_double2(0, 0);
          for (int k = 0; k < hd; ++k) t = cfma(a[k], __ldg(p + (size_t)k * ntv), t);
          if (inside[f])
            self = t;
          else
            sT[f * ddc + e] = t;
        }
        sT[e] = self;
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < GAL_E; ++q) {
      const int e = threadIdx.x + q * GAL_T;
      if (e < dcc) {
        const int i = e / dc, j = e % dc, ci = i / ntv, mi = i % ntv;
        const double2* p = PB + ((size_t)ci * bsz + js * hd) * ntv + mi;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          if (c && inside[c]) continue;
          const double2* t = sT + c * ddc + (ci * hd) * dc + j;
          for (int k = 0; k < hd; ++k) acc[c][q] = cfmac(__ldg(p + (size_t)k * ntv), t[k * dc], acc[c][q]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < GAL_E; ++q) {
    const int e = threadIdx.x + q * GAL_T;
    if (e < dcc)
#pragma unroll
      for (int c = 0; c < 5; ++c) out[((size_t)B * 5 + c) * dcc + e] = acc[c][q];
  }
}

// The fine level with 4 x 4 aggregates and dc = 16 (one dof per chirality and site, 256 entries of a block): all 16
// sites of the aggregate at once, one thread per (site, spin, column) of D P and then one per entry of the blocks.  A
// site by site pass has 32 such products for 256 threads.  sT[site][c][spin][j]: c = 0 the hops that stay in B, 1 the
// x hop and 2 the t hop that leave it (a site has at most one of each).
__global__ void __launch_bounds__(256) k_galerkin_fine4(const double2* __restrict__ lk, double diag, int Ls,
                                                        const double2* __restrict__ P, double2* __restrict__ out) {
  constexpr int NTV = 8, DC = 16, BSZ = 16;
  __shared__ double2 sT[16][3][2][DC];
  const int Lc = Ls / 4, B = blockIdx.x, BT = B / Lc, BX = B % Lc, tid = threadIdx.x;
  constexpr size_t PB = (size_t)2 * BSZ * NTV;
  const int nb[5] = {B, BT * Lc + (BX + 1 == Lc ? 0 : BX + 1), BT * Lc + (BX == 0 ? Lc - 1 : BX - 1),
                     (BT + 1 == Lc ? 0 : BT + 1) * Lc + BX, (BT == 0 ? Lc - 1 : BT - 1) * Lc + BX};
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * 256, js = e >> 5, r = (e >> 4) & 1, j = e & 15, cj = j >> 3, m = j & 7;
    const int jt = js >> 2, jx = js & 3, s = (4 * BT + jt) * Ls + 4 * BX + jx;
    double2 self = make_double2(0, 0), ox = self, ot = self;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      double2 M[4];
      wilson_hop(lk, diag, Ls, s, f, M);
      const int js2 = f == 0 ? js : f == 1 ? (jx == 3 ? js - 3 : js + 1) : f == 2 ? (jx == 0 ? js + 3 : js - 1)
                    : f == 3 ? (js + 4) & 15 : (js + 12) & 15;
      const bool in = f == 0 || (f == 1 ? jx < 3 : f == 2 ? jx > 0 : f == 3 ? jt < 3 : jt > 0);
      const double2 p = __ldg(P + (size_t)(in ? B : nb[f]) * PB + (cj * BSZ + js2) * NTV + m);
      const double2 a = r ? (cj ? M[3] : M[2]) : (cj ? M[1] : M[0]);
      if (in)
        self = cfma(a, p, self);
      else if (f <= 2)
        ox = cfma(a, p, ox);
      else
        ot = cfma(a, p, ot);
    }
    sT[js][0][r][j] = self;
    sT[js][1][r][j] = ox;
    sT[js][2][r][j] = ot;
  }
  __syncthreads();
  const int i = tid >> 4, j = tid & 15, ci = i >> 3, mi = i & 7;
  const double2* p = P + (size_t)B * PB + ci * BSZ * NTV + mi;
  double2 acc[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) acc[c] = make_double2(0, 0);
#pragma unroll
  for (int js = 0; js < 16; ++js) {
    const double2 pc = __ldg(p + js * NTV);
    acc[0] = cfmac(pc, sT[js][0][ci][j], acc[0]);
    if ((js & 3) == 3) acc[1] = cfmac(pc, sT[js][1][ci][j], acc[1]);
    if ((js & 3) == 0) acc[2] = cfmac(pc, sT[js][1][ci][j], acc[2]);
    if ((js >> 2) == 3) acc[3] = cfmac(pc, sT[js][2][ci][j], acc[3]);
    if ((js >> 2) == 0) acc[4] = cfmac(pc, sT[js][2][ci][j], acc[4]);
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) out[((size_t)B * 5 + c) * 256 + tid] = acc[c];
}

void galerkin(cudaStream_t stm, const double2* A, bool wilson, double diag, int Ls, int d, int agg, int ntv,
              const double2* P, double2* out) {
  const int dc = 2 * ntv, Lc = Ls / agg;
  MG_CHECK_ARG(dc * dc <= GAL_E * GAL_T && d % 2 == 0 && (!wilson || d == 2), "Galerkin block sizes");
  const size_t sm = sizeof(double2) * 5 * ((size_t)d * d + (size_t)d * dc);
  MG_CHECK_ARG(sm <= 200 * 1024, "Galerkin blocks too large for shared memory");
  const double na = agg * agg, hd = d / 2;
  const double flops = (double)Lc * Lc * 8.0 * hd * (na * 5.0 * d * dc + (na + 4.0 * agg) * (double)dc * dc);
  const double bytes = (double)Lc * Lc * (na * (wilson ? 32.0 : 5.0 * d * d * 16.0) + 5.0 * dc * dc * 16.0 +
                                          2.0 * na * hd * ntv * 16.0);
  if (wilson && agg == 4 && ntv == 8) {
    MG_LAUNCH_W(bytes, flops, k_galerkin_fine4, Lc * Lc, 256, 0, stm, A, diag, Ls, P, out);
  } else if (wilson) {
    ensure_max_smem((const void*)k_galerkin<true>, 200 * 1024);
    MG_LAUNCH_W(bytes, flops, k_galerkin<true>, Lc * Lc, GAL_T, sm, stm, A, diag, Ls, d, agg, ntv, P, out);
  } else {
    ensure_max_smem((const void*)k_galerkin<false>, 200 * 1024);
    MG_LAUNCH_W(bytes, flops, k_galerkin<false>, Lc * Lc, GAL_T, sm, stm, A, diag, Ls, d, agg, ntv, P, out);
  }
}

// ---- coarsest level as a dense matrix -------------------------------------------------
__global__ void k_dense_from_stencil(const double2* __restrict__ st, int Ls, int d, double2* __restrict__ A) {
  const int nsite = Ls * Ls;
  const size_t N = (size_t)nsite * d;
  const size_t total = (size_t)nsite * d * d;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int j = e % d, i = (e / d) % d, s = (int)(e / ((size_t)d * d));
    for (int dir = 0; dir < 5; ++dir) {
      const int nb = nbr_site(s, dir, Ls);
      double2* a = A + ((size_t)s * d + i) * N + (size_t)nb * d + j;
      *a = cadd(*a, st[((size_t)s * 5 + dir) * d * d + i * d + j]);
    }
  }
}

void dense_from_stencil(cudaStream_t stm, const double2* st, int Ls, int d, double2* A) {
  const size_t N = (size_t)Ls * Ls * d;
  MG_CUDA(cudaMemsetAsync(A, 0, N * N * sizeof(double2), stm));
  // one thread per (site, i, j): the five neighbour columns are distinct for Ls >= 3
  MG_LAUNCH(k_dense_from_stencil, 512, 256, 0, stm, st, Ls, d, A);
}

}  // namespace mg
