// FP64 solve-side kernels:
//  * implicit operator (paper eq. 11) and the solves with K_reg used by d
//    (eq. 7) and the primal recovery (eq. 5): supernodal forward / backward
//    substitution with L_i, one subdomain per CTA, the subdomain vector held
//    in shared memory;
//  * the coarse problem G^T G (G = B R, eqs. 6-8): deterministic assembly,
//    blocked Cholesky and explicit inverse built from 64 x 64 FP64 tile GEMMs;
//  * the projector P = I - G (G^T G)^{-1} G^T and the PCPG vector updates of
//    Algorithm 1 (M = I), with dot products reduced in a fixed order.
#include "cluster.cuh"
#include "common.cuh"
#include "kernels.h"

namespace feti {
namespace {

constexpr int kW = 32;

__device__ __forceinline__ int pop_item_s(int* queue) {
  __shared__ int item;
  __syncthreads();
  if (threadIdx.x == 0) item = atomicAdd(queue, 1);
  __syncthreads();
  return item;
}

constexpr int kWF = 128;  // largest front handled by one warp (needs w <= 32)

// Entry of a child's update vector: another CTA of the cluster may have written it (CL), so not from L1 then.
template <bool CL>
__device__ __forceinline__ double ld_upd(const double* p) {
  if constexpr (CL) return __ldcg(p);
  else return *p;
}

// The implicit solves use L in unit-lower form, L = Lu D (D = diag of L),
// written by unit_scale_kernel after the assembly: the panel holds Lu below
// the diagonal and zeros on and above it, and d2[j] = 1 / L_jj^2.  Then
// K_reg^{-1} y = Lu^{-T} D^{-2} Lu^{-1} y: the forward sweep needs no pivot
// and its own entries are scaled by d2 once, the backward sweep none.

// One warp: forward step of a small supernode (w <= 32, w + r <= kWF).  Lane
// l keeps the front entries l + 32 q in registers; per column j, z_j comes
// from lane j and every front row takes its update in one FMA (the zeros of
// Lu on and above the diagonal leave the rows <= j unchanged).
template <bool CL>
__device__ __forceinline__ void fwd_warp(const DevPlan& P, const SubInfo& S, int gs, const double* d2,
                                         double* ubuf, double* y, double* v, int lane) {
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  for (int i = lane; i < f_; i += 32) v[i] = i < w ? y[c0 + i] : 0.0;
  __syncwarp();
  for (int c = P.ch_off[gs]; c < P.ch_off[gs + 1]; ++c) {
    const int gc = S.sn0 + P.ch_list[c];
    const int rc = P.sn_r[gc];
    const double* U = ubuf + P.uofs[gc];
    const int* rl = P.rel + P.rel_off[gc];
    for (int k = lane; k < rc; k += 32) v[rl[k]] += ld_upd<CL>(U + k);
    __syncwarp();
  }
  const int nq = (f_ + 31) / 32;  // warp-uniform
  double a[kWF / 32];
#pragma unroll
  for (int q = 0; q < kWF / 32; ++q) {
    const int i = lane + 32 * q;
    a[q] = (q < nq && i < f_) ? v[i] : 0.0;
  }
  // columns in groups of 4: the group's loads are issued together, so one
  // global-memory latency is paid per group instead of per column
  constexpr int kU = 4;
  for (int j0 = 0; j0 < w; j0 += kU) {
    double lc[kU][kWF / 32];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int j = j0 + u;
      const double* col = Ls + (int64_t)j * f_;
#pragma unroll
      for (int q = 0; q < kWF / 32; ++q) {
        const int i = lane + 32 * q;
        lc[u][q] = (j < w && q < nq && i < f_) ? col[i] : 0.0;
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int j = j0 + u;
      if (j >= w) break;
      const double zj = __shfl_sync(0xffffffffu, a[0], j);
#pragma unroll
      for (int q = 0; q < kWF / 32; ++q)
        if (q < nq) a[q] = fma(-lc[u][q], zj, a[q]);
    }
  }
  if (lane < w) y[c0 + lane] = a[0] * d2[c0 + lane];
  double* Us = ubuf + P.uofs[gs];
#pragma unroll
  for (int q = 0; q < kWF / 32; ++q) {
    const int i = lane + 32 * q;
    if (i >= w && i < f_) Us[i - w] = a[q];
  }
  __syncwarp();
}

// One warp: backward step of a small supernode.  The rows part
// t_l = sum_i L21[i][l] x_rows[i] is split over G = 32 / 2^ceil(log2 w)
// row groups per column (lane = l + wp g), reduced with shuffles; then lane
// l owns x_l through the triangular sweep.
__device__ __forceinline__ void bwd_warp(const DevPlan& P, const SubInfo& S, int gs, double* y, double* v,
                                         int lane) {
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  const int* rows = P.rows + P.sn_rows[gs];
  for (int i = lane; i < r; i += 32) v[i] = y[rows[i]];
  __syncwarp();
  int wp = 1;
  while (wp < w) wp <<= 1;
  const int G = 32 / wp, l = lane % wp, g = lane / wp;
  double t = 0.0;
  if (l < w) {
    const double* col = Ls + (int64_t)l * f_ + w;
#pragma unroll 4
    for (int i = g; i < r; i += G) t = fma(col[i], v[i], t);
  }
  for (int o = wp; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  double x = lane < w ? y[c0 + lane] - t : 0.0;
  for (int j0 = w - 1; j0 >= 0; j0 -= 4) {
    double lr[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 - u;
      lr[u] = (j >= 0 && lane < j) ? Ls[(int64_t)lane * f_ + j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 - u;
      if (j < 0) break;
      const double xj = __shfl_sync(0xffffffffu, x, j);
      x = fma(-lr[u], xj, x);
    }
  }
  if (lane < w) y[c0 + lane] = x;
  __syncwarp();
}

// Barrier of the 256 threads that share a supernode: the CTA, or team `team` of a wide CTA.
template <bool TEAM>
__device__ __forceinline__ void cta_sync(int team) {
  if constexpr (TEAM) asm volatile("bar.sync %0, 256;" ::"r"(team + 1) : "memory");
  else __syncthreads();
}

// 256 threads: forward step of a large supernode on the shared front vector.
// 32 x 32 unit-lower diagonal blocks are staged in shared memory and solved
// by warp 0; all threads apply the block's columns to the rest of the front.
template <bool TEAM = false, bool CL = false>
__device__ __forceinline__ void fwd_cta(const DevPlan& P, const SubInfo& S, int gs, const double* d2,
                                        double* ubuf, double* y, double* sf, double (*sm_blk)[kW + 1], int tid, int team = 0) {
  const int warp = tid / 32, lane = tid % 32;
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  for (int i = tid; i < f_; i += kThreads) sf[i] = i < w ? y[c0 + i] : 0.0;
  cta_sync<TEAM>(team);
  for (int c = P.ch_off[gs]; c < P.ch_off[gs + 1]; ++c) {
    const int gc = S.sn0 + P.ch_list[c];
    const int rc = P.sn_r[gc];
    const double* U = ubuf + P.uofs[gc];
    const int* rl = P.rel + P.rel_off[gc];
    for (int k = tid; k < rc; k += kThreads) sf[rl[k]] += ld_upd<CL>(U + k);
    cta_sync<TEAM>(team);
  }
  for (int kb = 0; kb < w; kb += kW) {
    const int nbk = min(kW, w - kb);
    for (int idx = tid; idx < nbk * kW; idx += kThreads) {
      const int k = idx / kW, i = idx % kW;  // column k, row i of the block
      if (i < nbk) sm_blk[i][k] = (i >= k) ? Ls[(int64_t)(kb + k) * f_ + kb + i] : 0.0;
    }
    cta_sync<TEAM>(team);
    if (warp == 0) {
      double yi = lane < nbk ? sf[kb + lane] : 0.0;
      for (int k = 0; k < nbk; ++k) {
        const double yk = __shfl_sync(0xffffffffu, yi, k);
        yi = fma(-sm_blk[lane][k], yk, yi);  // zero on and above the diagonal
      }
      if (lane < nbk) sf[kb + lane] = yi;
    }
    cta_sync<TEAM>(team);
    // rows in pairs (i, i + kThreads) per thread, so that each group of column loads has twice the bytes in
    // flight; a last unpaired row alone.  Every row's sum runs over k in the same order either way.
    int i = kb + nbk + tid;
    for (; i + kThreads < f_; i += 2 * kThreads) {
      double acc = 0.0, acc2 = 0.0;
#pragma unroll 8
      for (int k = 0; k < nbk; ++k) {
        const double* col = Ls + (int64_t)(kb + k) * f_;
        const double zk = sf[kb + k];
        acc = fma(col[i], zk, acc);
        acc2 = fma(col[i + kThreads], zk, acc2);
      }
      sf[i] -= acc;
      sf[i + kThreads] -= acc2;
    }
    if (i < f_) {
      double acc = 0.0;
#pragma unroll 8
      for (int k = 0; k < nbk; ++k) acc = fma(Ls[(int64_t)(kb + k) * f_ + i], sf[kb + k], acc);
      sf[i] -= acc;
    }
    cta_sync<TEAM>(team);
  }
  double* Us = ubuf + P.uofs[gs];
  for (int i = tid; i < f_; i += kThreads) {
    if (i < w) y[c0 + i] = sf[i] * d2[c0 + i];
    else Us[i - w] = sf[i];
  }
  cta_sync<TEAM>(team);
}

// 256 threads: backward step of a large supernode (x_rows already final).  The
// entries x_rows are gathered into sf first; then each warp takes kBC own
// columns at a time, so their column loads are in flight together (the dot
// product of each column runs over the rows in the same order as with one
// column per warp, and is reduced the same way).
constexpr int kBC = 4;
template <bool TEAM = false>
__device__ __forceinline__ void bwd_cta(const DevPlan& P, const SubInfo& S, int gs, double* y, double* sf,
                                        double (*sm_blk)[kW + 1], int tid, int team = 0) {
  const int warp = tid / 32, lane = tid % 32;
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  const int* rows = P.rows + P.sn_rows[gs];
  for (int k = tid; k < r; k += kThreads) sf[k] = y[rows[k]];
  cta_sync<TEAM>(team);
  for (int l0 = warp * kBC; l0 < w; l0 += (kThreads / 32) * kBC) {
    if (l0 + kBC <= w) {
      double acc[kBC];
      const double* col[kBC];
#pragma unroll
      for (int u = 0; u < kBC; ++u) {
        acc[u] = 0.0;
        col[u] = Ls + (int64_t)(l0 + u) * f_ + w;
      }
#pragma unroll 2
      for (int k = lane; k < r; k += 32) {
        const double xk = sf[k];
#pragma unroll
        for (int u = 0; u < kBC; ++u) acc[u] = fma(col[u][k], xk, acc[u]);
      }
#pragma unroll
      for (int u = 0; u < kBC; ++u) {
        double a = acc[u];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) y[c0 + l0 + u] -= a;
      }
    } else {
      // the last w mod kBC columns one at a time (warp-uniform branch)
      for (int l = l0; l < w; ++l) {
        const double* col = Ls + (int64_t)l * f_ + w;
        double a = 0.0;
#pragma unroll 4
        for (int k = lane; k < r; k += 32) a = fma(col[k], sf[k], a);
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) y[c0 + l] -= a;
      }
    }
  }
  cta_sync<TEAM>(team);
  for (int kb = ((w - 1) / kW) * kW; kb >= 0; kb -= kW) {
    const int nbk = min(kW, w - kb);
    if (nbk == kW) {
      // a full block: the warp's columns l = kb + warp + 8 u all at once
      constexpr int kU = kW / (kThreads / 32);
      double acc[kU];
      const double* col[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        acc[u] = 0.0;
        col[u] = Ls + (int64_t)(kb + warp + (kThreads / 32) * u) * f_;
      }
#pragma unroll 2
      for (int i = kb + nbk + lane; i < w; i += 32) {
        const double xi = y[c0 + i];
#pragma unroll
        for (int u = 0; u < kU; ++u) acc[u] = fma(col[u][i], xi, acc[u]);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        double a = acc[u];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) y[c0 + kb + warp + (kThreads / 32) * u] -= a;
      }
    } else {
      for (int l = kb + warp; l < kb + nbk; l += kThreads / 32) {
        double acc = 0.0;
#pragma unroll 4
        for (int i = kb + nbk + lane; i < w; i += 32) acc = fma(Ls[(int64_t)l * f_ + i], y[c0 + i], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) y[c0 + l] -= acc;
      }
    }
    for (int idx = tid; idx < nbk * kW; idx += kThreads) {
      const int k = idx / kW, i = idx % kW;
      if (i < nbk) sm_blk[i][k] = (i >= k) ? Ls[(int64_t)(kb + k) * f_ + kb + i] : 0.0;
    }
    cta_sync<TEAM>(team);
    if (warp == 0) {
      double yi = lane < nbk ? y[c0 + kb + lane] : 0.0;
      for (int k = nbk - 1; k >= 0; --k) {
        const double yk = __shfl_sync(0xffffffffu, yi, k);
        yi = fma(-sm_blk[k][lane], yk, yi);  // zero on and above the diagonal
      }
      if (lane < nbk) y[c0 + kb + lane] = yi;
    }
    cta_sync<TEAM>(team);
  }
}

// ---------------------------------------------------------------- one wide CTA per subdomain
//
// With at most one subdomain per SM the 256-thread CTA above leaves the SM waiting: each 32-column block of a large
// supernode was a 32-step chain in one warp, then a few column loads in flight per thread.  The wide CTA (1024
// threads) applies the block's inverse instead (inv_block_kernel keeps it above the diagonal of the block, where the
// panel holds nothing), splits the 32 columns of each update over four groups of threads, so that all of a block's
// loads are in flight at once, and issues the first of them before the block's own entries are solved.  FP64
// instructions are the scarce resource (64 clocks of a scheduler each): dot products run on eight lanes per column,
// which needs three additions per four columns to reduce.  Supernodes of moderate size (kTeamF, kTeamW) spend most of
// their time in chains of index loads, so the wide CTA's four teams of 256 threads take one each, side by side.
// A cluster of 1 to 8 wide CTAs takes a subdomain: with fewer subdomains than SMs, or uneven ones, one SM's FP64 pipe
// under the largest subdomain sets the time.  Each CTA has subtrees of its own (plan_solve_split), for which it needs
// none of the others; the few supernodes above them are dealt out level by level, update vectors go through global
// memory, and the columns that a shared supernode solves are stored into every CTA's vector.  Every front is computed as
// by one CTA, so the results do not depend on the cluster size.
// Measured per application (256 threads per subdomain -> one wide CTA -> the cluster of the dispatch's choice): 64
// elasticity subdomains of 12^3 5.7 -> 2.7 -> 1.8 ms (2 CTAs), 27 of them 2.9 -> 1.2 (4), 125 uneven 3D heat subdomains
// 9.0 -> 4.75 -> 2.1 ms (4; its largest subdomain's two sweeps of 3.5 M entries are 1.8 ms of one SM's FP64 pipe).
constexpr int kWide = 1024;
constexpr int kTeamF = 512, kTeamW = 64;  // largest front and width a team takes
constexpr int kWR = 512;  // rows of an update pass (two per thread of a group)
struct WideSmem {
  double blk[2][kW][kW + 1];  // inverses of the unit-lower diagonal blocks (strictly lower part)
  double dp[4][kW];           // partial products of a block
};
// dynamic shared memory behind the front vector: the warps' fronts (and the wide updates' partial sums) and WideSmem,
// or the four teams' fronts and diagonal blocks
constexpr int kWideBuf = kWide / 32 * kWF + (int)(sizeof(WideSmem) / 8);
static_assert(4 * (kTeamF + kW * (kW + 1)) <= kWideBuf, "the teams' buffers fit");

// (i, k) of the inverse of the unit-lower block kb, k < i, stands at row k of column i
__device__ __forceinline__ void wide_stage(const double* Ls, int f_, int kb, int nbk, double (*blk)[kW + 1], int t,
                                           int nt) {
  for (int idx = t; idx < kW * kW; idx += nt) {
    const int k = idx % kW, i = idx / kW;
    blk[i][k] = (i < nbk && k < i) ? Ls[(int64_t)(kb + i) * f_ + kb + k] : 0.0;
  }
}

template <bool CL>
__device__ __forceinline__ void fwd_wide(const DevPlan& P, const SubInfo& S, int gs, const double* d2, double* ubuf,
                                         double* y, double* sf, double* part, WideSmem& ws, int tid) {
  const int warp = tid / 32, lane = tid % 32, g = tid / 256, t = tid % 256;
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  wide_stage(Ls, f_, 0, min(kW, w), ws.blk[0], tid, kWide);
  for (int i = tid; i < f_; i += kWide) sf[i] = i < w ? y[c0 + i] : 0.0;
  __syncthreads();
  for (int c = P.ch_off[gs]; c < P.ch_off[gs + 1]; ++c) {
    const int gc = S.sn0 + P.ch_list[c];
    const int rc = P.sn_r[gc];
    const double* U = ubuf + P.uofs[gc];
    const int* rl = P.rel + P.rel_off[gc];
    for (int k = tid; k < rc; k += kWide) sf[rl[k]] += ld_upd<CL>(U + k);
    __syncthreads();
  }
  // the own rows, block by block
  for (int kb = 0, cur = 0; kb < w; kb += kW, cur ^= 1) {
    const int nbk = min(kW, w - kb);
    const int k0 = 8 * g, r0 = kb + nbk;
    const bool upd = r0 < w;  // then the block is full
    // the first rows' columns, in flight while the block is solved
    double l[8];
    if (upd) {
#pragma unroll
      for (int e = 0; e < 8; ++e) l[e] = r0 + t < w ? Ls[(int64_t)(kb + k0 + e) * f_ + r0 + t] : 0.0;
    }
    if (warp < 4) {
      double p = 0.0;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        p = fma(ws.blk[cur][lane][8 * warp + e], 8 * warp + e < nbk ? sf[kb + 8 * warp + e] : 0.0, p);
      ws.dp[warp][lane] = p;
    } else if (kb + kW < w) {
      wide_stage(Ls, f_, kb + kW, min(kW, w - kb - kW), ws.blk[cur ^ 1], tid - 128, kWide - 128);
    }
    __syncthreads();
    if (warp == 0 && lane < nbk)
      sf[kb + lane] += (ws.dp[0][lane] + ws.dp[1][lane]) + (ws.dp[2][lane] + ws.dp[3][lane]);
    __syncthreads();
    if (!upd) break;
    for (int i0 = r0, h = 0; i0 < w; i0 += 256, ++h) {
      double* pt = part + (h & 1) * 1024;
      const int i = i0 + t;
      if (h > 0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) l[e] = i < w ? Ls[(int64_t)(kb + k0 + e) * f_ + i] : 0.0;
      }
      if (i0 + (t & ~31) < w) {
        double acc = 0.0;
#pragma unroll
        for (int e = 0; e < 8; ++e) acc = fma(l[e], sf[kb + k0 + e], acc);
        pt[g * 256 + t] = acc;
      }
      __syncthreads();
      if (tid < 256 && i < w) sf[i] -= (pt[t] + pt[256 + t]) + (pt[512 + t] + pt[768 + t]);
    }
    __syncthreads();
  }
  // the rows below: each group of threads a quarter of the columns, nothing to wait for
  {
    const int kq = (w + 3) / 4, k0 = min(w, g * kq), k1 = min(w, k0 + kq);
    int h = 0;
    for (int i0 = w; i0 < f_; i0 += kWR, ++h) {
      double* pt = part + (h & 1) * 4 * kWR;
      const int i = i0 + t;
      double acc = 0.0, acc2 = 0.0;
      if (i0 + 256 + (t & ~31) < f_) {
        const int i2 = min(i + 256, f_ - 1);
#pragma unroll 8
        for (int k = k0; k < k1; ++k) {
          const double* col = Ls + (int64_t)k * f_;
          const double z = sf[k];
          acc = fma(col[i], z, acc);
          acc2 = fma(col[i2], z, acc2);
        }
      } else if (i0 + (t & ~31) < f_) {
        const int i1 = min(i, f_ - 1);
#pragma unroll 8
        for (int k = k0; k < k1; ++k) acc = fma(Ls[(int64_t)k * f_ + i1], sf[k], acc);
      }
      pt[g * kWR + t] = acc;
      pt[g * kWR + 256 + t] = acc2;
      __syncthreads();
      if (tid < kWR && i0 + tid < f_)
        sf[i0 + tid] -= (pt[tid] + pt[kWR + tid]) + (pt[2 * kWR + tid] + pt[3 * kWR + tid]);
    }
    __syncthreads();
  }
  double* Us = ubuf + P.uofs[gs];
  for (int i = tid; i < f_; i += kWide) {
    if (i < w) y[c0 + i] = sf[i] * d2[c0 + i];
    else Us[i - w] = sf[i];
  }
  __syncthreads();
}

__device__ __forceinline__ double sum8(double a) {
  a += __shfl_xor_sync(0xffffffffu, a, 4);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  return a;
}

__device__ __forceinline__ void bwd_wide(const DevPlan& P, const SubInfo& S, int gs, double* y, double* sf,
                                         WideSmem& ws, int tid) {
  const int warp = tid / 32, lane = tid % 32, c4 = lane / 8, l8 = lane % 8;
  const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs], f_ = w + r;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  const int* rows = P.rows + P.sn_rows[gs];
  for (int k = tid; k < r; k += kWide) sf[k] = y[rows[k]];
  const int kl = ((w - 1) / kW) * kW;
  wide_stage(Ls, f_, kl, w - kl, ws.blk[0], tid, kWide);
  __syncthreads();
  // the rows below: each warp four columns at a time
  for (int l0 = 4 * warp; l0 < w; l0 += 4 * (kWide / 32)) {
    const int l = l0 + c4;
    const double* col = Ls + (int64_t)min(l, w - 1) * f_ + w;
    double acc = 0.0;
#pragma unroll 8
    for (int k = l8; k < r; k += 8) acc = fma(col[k], sf[k], acc);
    acc = sum8(acc);
    if (l8 == 0 && l < w) y[c0 + l] -= acc;
  }
  __syncthreads();
  for (int kb = kl, cur = 0; kb >= 0; kb -= kW, cur ^= 1) {
    const int nbk = min(kW, w - kb);
    // the supernode's own rows below the block: columns kb + 4 (warp % 8) + c4, a quarter of the rows per warp
    {
      const int l = min(kb + 4 * (warp % 8) + c4, w - 1);
      const double* col = Ls + (int64_t)l * f_;
      double acc = 0.0;
#pragma unroll 4
      for (int i = kb + nbk + 8 * (warp / 8) + l8; i < w; i += 32) acc = fma(col[i], y[c0 + i], acc);
      acc = sum8(acc);
      if (l8 == 0) ws.dp[warp / 8][4 * (warp % 8) + c4] = acc;
    }
    __syncthreads();
    double v = 0.0;
    if (warp < 4) {
      if (lane < nbk)
        v = y[c0 + kb + lane] - ((ws.dp[0][lane] + ws.dp[1][lane]) + (ws.dp[2][lane] + ws.dp[3][lane]));
      double p = 0.0;
#pragma unroll
      for (int e = 0; e < 8; ++e)
        p = fma(ws.blk[cur][8 * warp + e][lane], __shfl_sync(0xffffffffu, v, 8 * warp + e), p);
      __syncwarp();
      asm volatile("bar.sync 2, 128;" ::: "memory");  // the four warps have read dp
      ws.dp[warp][lane] = p;
    } else if (kb > 0) {
      wide_stage(Ls, f_, kb - kW, kW, ws.blk[cur ^ 1], tid - 128, kWide - 128);
    }
    __syncthreads();
    if (warp == 0 && lane < nbk)
      y[c0 + kb + lane] = v + ((ws.dp[0][lane] + ws.dp[1][lane]) + (ws.dp[2][lane] + ws.dp[3][lane]));
    __syncthreads();
  }
}

// Inverses of the unit-lower 32 x 32 diagonal blocks of the supernodes that the wide solves take, kept above the
// diagonal of their own block ((i, k), k < i, at row k of column i).  One warp per block, lane = column.
__global__ void __launch_bounds__(128) inv_block_kernel(DevPlan P, int nsub) {
  __shared__ double B[4][kW][kW + 1];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  double(*D)[kW + 1] = B[warp];
  for (int si = blockIdx.y; si < nsub; si += gridDim.y) {
    const SubInfo& S = P.sub[si];
    for (int s = blockIdx.x; s < S.nsn; s += gridDim.x) {
      const int gs = S.sn0 + s;
      const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
      if (w <= 32 && f_ <= kWF) continue;
      double* Ls = P.L + S.L + P.Lofs[gs];
      for (int kb = kW * warp; kb < w; kb += 4 * kW) {
        const int nbk = min(kW, w - kb);
        for (int k = 0; k < kW; ++k)
          D[lane][k] = (lane < nbk && k < lane) ? Ls[(int64_t)(kb + k) * f_ + kb + lane] : 0.0;
        __syncwarp();
        double m[kW];
#pragma unroll
        for (int i = 0; i < kW; ++i) {
          double a = i == lane ? 1.0 : 0.0;
#pragma unroll
          for (int k = 0; k < i; ++k) a = fma(-D[i][k], m[k], a);
          m[i] = a;
        }
        __syncwarp();
#pragma unroll
        for (int i = 1; i < kW; ++i)
          if (i < nbk && lane < i) Ls[(int64_t)(kb + i) * f_ + kb + lane] = m[i];
      }
    }
  }
}

// The rank of the cluster that writes column col of the solution: its piece's, 0 for the shared ones.
__device__ __forceinline__ int col_owner(const DevPlan& P, const SubInfo& S, int col) {
  int owner = 0;
  for (int k = S.pc0; k < S.pc0 + S.npc; ++k) {
    const int4 pc = P.pieces[k];
    if (col >= pc.x && col < pc.y) owner = pc.z;
  }
  return owner;
}

// MODE 0: qi = B L^-T L^-1 P B^T p        (implicit apply, eq. 11)
// MODE 1: qi = B K_reg^{-1} f             (d = B K^+ f - c, eq. 7)
// MODE 2: u  = K_reg^{-1} (f - B^T lambda) (eq. 5 without R alpha)
// NT: threads of the CTA (256, or the wide 1024); CL: the wide CTAs of a cluster share a subdomain (an instantiation of
// its own: the registers that it takes cost the small problems of single CTAs 15 us of 75).
template <int MODE, int NT, bool CL>
__global__ void __launch_bounds__(NT, NT == kWide ? 1 : 4)
    implicit_kernel(DevPlan P, const int* order, int nsub, int* queue, const double* p, const double* f, double* qi,
                    double* u, double* uws, int64_t ustride, int nmax, int maxf) {
  // [nmax] subdomain vector, [maxf] front, [NT / 32 kWF] warp fronts (the wide updates' partial sums), wide: WideSmem
  extern __shared__ double y[];
  __shared__ __align__(16) uint8_t blk_raw[NT == kWide ? 16 : sizeof(double) * kW * (kW + 1)];
  double(*sm_blk)[kW + 1] = reinterpret_cast<double(*)[kW + 1]>(blk_raw);
  static_assert(kWide / 32 * kWF >= 2 * 4 * kWR, "the partial sums fit the warp fronts");
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  double* sfront = y + nmax;
  double* wbuf = sfront + maxf;
  WideSmem& wsm = *reinterpret_cast<WideSmem*>(wbuf + NT / 32 * kWF);  // NT == kWide
  static_assert(!CL || NT == kWide, "clusters of wide CTAs");
  const int rank = CL ? (int)cl_rank() : 0, C = CL ? (int)cl_size() : 1;
  __shared__ int item_s;
  double* ubuf = uws + (int64_t)(blockIdx.x / C) * ustride;
  for (;;) {
    int itx;
    if constexpr (CL) {
      cl_barrier();
      if (rank == 0 && tid == 0) {
        const int it = atomicAdd(queue, 1);
        for (int c = 0; c < C; ++c) cl_store(&item_s, c, it);
      }
      cl_barrier();
      itx = item_s;
    } else {
      itx = pop_item_s(queue);
    }
    if (itx >= nsub) return;
    const int si = order[itx];
    const SubInfo& S = P.sub[si];
    const int n = S.n;
    const double* d2 = P.dinv + S.dof;  // 1 / L_jj^2 (unit-lower form)
    for (int k = tid; k < n; k += NT) y[k] = 0.0;
    __syncthreads();
    if (MODE == 1 || MODE == 2)
      for (int k = tid; k < n; k += NT) y[P.iperm[S.diag0 + k]] = f[S.dof + k];
    __syncthreads();
    if (MODE == 0 || MODE == 2) {
      // B^T p: columns sharing a DOF are adjacent in sorted order; the first of a run sums it
      const int* sp = P.spos + S.col0;
      for (int j = tid; j < S.m; j += NT) {
        if (j > 0 && sp[j - 1] == sp[j]) continue;
        double s = 0.0;
        for (int jj = j; jj < S.m && sp[jj] == sp[j]; ++jj) s += P.qsign[S.qcol + jj] * p[P.qmap[S.qcol + jj]];
        y[sp[j]] += (MODE == 0) ? s : -s;
      }
    }
    __syncthreads();
    // Forward substitution L z = y, level by level from the leaves of the
    // supernodal tree.  Supernodes of one level are independent: each one
    // assembles its front vector from its own columns of y and the update
    // vectors of its children (in fixed order, so the result is
    // deterministic), solves with its diagonal block and writes its own
    // update vector for the parent.  Small fronts take one warp each, large
    // ones the whole CTA.  first, step: this CTA's share of the level [lo, hi).
    const int* lsn = P.lvl_sn;
    auto forward = [&](int lo, int hi, int first, int step) {
      for (int it = lo + first + step * warp; it < hi; it += step * (NT / 32)) {
        const int gs = S.sn0 + lsn[it];
        const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
        if (w > 32 || f_ > kWF) continue;
        fwd_warp<CL>(P, S, gs, d2, ubuf, y, wbuf + warp * kWF, lane);
      }
      __syncthreads();
      if constexpr (NT == kWide) {
        double* tbuf = wbuf + (tid / 256) * (kTeamF + kW * (kW + 1));
        int q = 0;
        for (int it = lo + first; it < hi; it += step) {
          const int gs = S.sn0 + lsn[it];
          const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
          if ((w <= 32 && f_ <= kWF) || w > kTeamW || f_ > kTeamF) continue;
          if ((q++ & 3) != tid / 256) continue;
          fwd_cta<true, CL>(P, S, gs, d2, ubuf, y, tbuf, reinterpret_cast<double(*)[kW + 1]>(tbuf + kTeamF), tid % 256, tid / 256);
        }
        __syncthreads();
      }
      for (int it = lo + first; it < hi; it += step) {
        const int gs = S.sn0 + lsn[it];
        const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
        if (w <= 32 && f_ <= kWF) continue;
        if (NT == kWide && w <= kTeamW && f_ <= kTeamF) continue;
        if constexpr (NT == kWide) fwd_wide<CL>(P, S, gs, d2, ubuf, y, sfront, wbuf, wsm, tid);
        else fwd_cta(P, S, gs, d2, ubuf, y, sfront, sm_blk, tid);
      }
    };
    // Backward substitution L^T x = z, level by level from the roots; every
    // supernode reads only ancestors' entries of x and writes its own columns.
    auto backward = [&](int lo, int hi, int first, int step) {
      for (int it = lo + first + step * warp; it < hi; it += step * (NT / 32)) {
        const int gs = S.sn0 + lsn[it];
        const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
        if (w > 32 || f_ > kWF) continue;
        bwd_warp(P, S, gs, y, wbuf + warp * kWF, lane);
      }
      __syncthreads();
      if constexpr (NT == kWide) {
        double* tbuf = wbuf + (tid / 256) * (kTeamF + kW * (kW + 1));
        int q = 0;
        for (int it = lo + first; it < hi; it += step) {
          const int gs = S.sn0 + lsn[it];
          const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
          if ((w <= 32 && f_ <= kWF) || w > kTeamW || f_ > kTeamF) continue;
          if ((q++ & 3) != tid / 256) continue;
          bwd_cta<true>(P, S, gs, y, tbuf, reinterpret_cast<double(*)[kW + 1]>(tbuf + kTeamF), tid % 256, tid / 256);
        }
        __syncthreads();
      }
      for (int it = lo + first; it < hi; it += step) {
        const int gs = S.sn0 + lsn[it];
        const int w = P.sn_w[gs], f_ = w + P.sn_r[gs];
        if (w <= 32 && f_ <= kWF) continue;
        if (NT == kWide && w <= kTeamW && f_ <= kTeamF) continue;
        if constexpr (NT == kWide) bwd_wide(P, S, gs, y, sfront, wsm, tid);
        else bwd_cta(P, S, gs, y, sfront, sm_blk, tid);
      }
    };
    const int nl = S.nlev;
    const int* lvo = P.lvl_off + S.lvl0;
    if constexpr (CL) {
      // own levels, then the shared ones with a barrier after each (one call site each way: the sweeps' code is long)
      const int* lvt = lvo + (1 + C) * (nl + 1);
      lvo += (1 + rank) * (nl + 1);
      for (int q = 0; q < 2 * nl; ++q) {
        const bool top = q >= nl;
        const int* lv = top ? lvt + (q - nl) : lvo + q;
        if (q == nl) cl_barrier();
        const int lo = lv[0], hi = lv[1];
        if (lo == hi) continue;
        forward(lo, hi, top ? rank : 0, top ? C : 1);
        if (top) cl_barrier();
      }
      for (int q = 2 * nl - 1; q >= 0; --q) {
        const bool top = q >= nl;
        const int* lv = top ? lvt + (q - nl) : lvo + q;
        const int lo = lv[0], hi = lv[1];
        if (lo == hi) continue;
        backward(lo, hi, top ? rank : 0, top ? C : 1);
        if (top) {
          __syncthreads();
          // the columns solved here to the other CTAs
          for (int it = lo + rank; it < hi; it += C) {
            const int gs = S.sn0 + lsn[it], c0 = P.sn_c0[gs], w = P.sn_w[gs];
            for (int c = 1; c < C; ++c)
              for (int i = tid; i < w; i += NT) cl_store(y + c0 + i, (rank + c) % C, y[c0 + i]);
          }
          cl_barrier();
        }
      }
    } else {
      for (int l = 0; l < nl; ++l) forward(lvo[l], lvo[l + 1], 0, 1);
      for (int l = nl - 1; l >= 0; --l) backward(lvo[l], lvo[l + 1], 0, 1);
    }
    __syncthreads();
    // every CTA has x in its own columns and the shared ones (which rank 0 writes)
    if (MODE == 0 || MODE == 1) {
      for (int j = tid; j < S.m_pad; j += NT) {
        const int col = j < S.m ? P.spos[S.col0 + j] : -1;
        if (!CL || col_owner(P, S, col) == rank) qi[S.qcol + j] = col >= 0 ? P.qsign[S.qcol + j] * y[col] : 0.0;
      }
    } else {
      for (int k = tid; k < n; k += NT) {
        const int col = P.iperm[S.diag0 + k];
        if (!CL || col_owner(P, S, col) == rank) u[S.dof + k] = y[col];
      }
    }
    __syncthreads();
  }
}

// Unit-lower form of every factor, for the implicit solves (after the TRSM,
// which uses L itself): column j of each panel is divided by L_jj, the
// diagonal is set to zero and d2[dof + j] = 1 / L_jj^2.
// Bound by HBM (L read and written once).  One warp per column, which needs
// nothing but its own pivot, and as many CTAs per subdomain as its columns
// fill: with one CTA per subdomain and one warp per supernode the widest
// supernode's warp set the time (27 elasticity subdomains of 12^3: 8.9 ms,
// now 0.18 ms; 64 uneven 3D heat subdomains: 16.9 ms, now 0.3 ms).
__global__ void __launch_bounds__(256) unit_scale_kernel(DevPlan P, int nsub, double* d2) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  for (int si = blockIdx.y; si < nsub; si += gridDim.y) {
    const SubInfo& S = P.sub[si];
    const int* c0s = P.sn_c0 + S.sn0;
    for (int j = blockIdx.x * 8 + warp; j < S.n; j += gridDim.x * 8) {
      // the supernode that holds column j: the last one that starts at or before it
      int lo = 0, hi = S.nsn - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (c0s[mid] <= j) lo = mid;
        else hi = mid - 1;
      }
      const int gs = S.sn0 + lo, k = j - c0s[lo], f_ = P.sn_w[gs] + P.sn_r[gs];
      double* col = P.L + S.L + P.Lofs[gs] + (int64_t)k * f_;
      const double inv = 1.0 / col[k];
      __syncwarp();
#pragma unroll 4
      for (int i = k + 1 + lane; i < f_; i += 32) col[i] *= inv;
      if (lane == 0) {
        col[k] = 0.0;
        d2[S.dof + j] = inv * inv;
      }
    }
  }
}

// q[l] = qi[c0] + qi[c1] - c[l]
__global__ void gather_minus_c_kernel(const int* c0, const int* c1, int nlam, const double* qi, const double* c,
                                      double* q) {
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < nlam; l += gridDim.x * blockDim.x) {
    const int a = c0[l], b = c1[l];
    double s = a >= 0 ? qi[a] : 0.0;
    if (b >= 0) s += qi[b];
    q[l] = s - (c ? c[l] : 0.0);
  }
}

// ---------------------------------------------------------------- G = B R

// G6[g * 6 + k] = sign_j R_i[dof_j, k] for sorted column g of subdomain i
__global__ void build_G_kernel(DevPlan P, const int* colsub, int64_t ncols, const double* R, double* G6) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ncols; g += (int64_t)gridDim.x * blockDim.x) {
    const SubInfo& S = P.sub[colsub[g]];
    const int j = (int)(g - S.qcol);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      double v = 0.0;
      if (j < S.m && k < S.d) v = P.qsign[g] * R[S.R + (int64_t)k * S.n + P.qdof[g]];
      G6[g * 6 + k] = v;
    }
  }
}

// e[alpha0 + k] = R_i[:, k]^T f_i ; one warp per (subdomain, k)
__global__ void rtf_kernel(DevPlan P, int nsub, const double* R, const double* f, double* e) {
  const int lane = threadIdx.x & 31;
  for (int wk = (blockIdx.x * blockDim.x + threadIdx.x) / 32; wk < nsub * 6; wk += gridDim.x * blockDim.x / 32) {
    const int si = wk / 6, k = wk % 6;
    const SubInfo& S = P.sub[si];
    if (k >= S.d) continue;
    double acc = 0.0;
    for (int i = lane; i < S.n; i += 32) acc += R[S.R + (int64_t)k * S.n + i] * f[S.dof + i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) e[S.alpha0 + k] = acc;
  }
}

// c[alpha0 + k] = sum_j G6[(qcol + j) * 6 + k] x[map_j]  (G^T x), warp per (subdomain, k)
__global__ void gt_kernel(DevPlan P, int nsub, const double* G6, const double* x, double* c) {
  const int lane = threadIdx.x & 31;
  for (int wk = (blockIdx.x * blockDim.x + threadIdx.x) / 32; wk < nsub * 6; wk += gridDim.x * blockDim.x / 32) {
    const int si = wk / 6, k = wk % 6;
    const SubInfo& S = P.sub[si];
    if (k >= S.d) continue;
    double acc = 0.0;
    for (int j = lane; j < S.m; j += 32) acc += G6[(S.qcol + j) * 6 + k] * x[P.qmap[S.qcol + j]];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) c[S.alpha0 + k] = acc;
  }
}

// out[l] = (x ? x[l] : 0) - sgn * (G z)[l]
__global__ void gz_kernel(DevPlan P, const int* colsub, const int* c0, const int* c1, int nlam, const double* G6,
                          const double* x, const double* z, double sgn, double* out) {
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < nlam; l += gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int g = e == 0 ? c0[l] : c1[l];
      if (g < 0) continue;
      const SubInfo& S = P.sub[colsub[g]];
      for (int k = 0; k < S.d; ++k) s += G6[(int64_t)g * 6 + k] * z[S.alpha0 + k];
    }
    out[l] = (x ? x[l] : 0.0) - sgn * s;
  }
}

// G^T G block (i, k) from the multiplier pairs shared by subdomains i and k
__global__ void gtg_kernel(const int4* pairs, int npairs, const int2* plist, const double* G6, double* A, int D) {
  for (int pi = blockIdx.x; pi < npairs; pi += gridDim.x) {
    const int4 pr = pairs[pi];  // x = offset_i, y = offset_k, z = list begin, w = list end
    const int a = threadIdx.x / 6, b = threadIdx.x % 6;
    if (threadIdx.x >= 36) continue;
    const int di = (pr.x >> 24) & 0xff, dk = (pr.y >> 24) & 0xff;
    const int oi = pr.x & 0xffffff, ok = pr.y & 0xffffff;
    if (a >= di || b >= dk) continue;
    double s = 0.0;
    for (int t = pr.z; t < pr.w; ++t) s += G6[(int64_t)plist[t].x * 6 + a] * G6[(int64_t)plist[t].y * 6 + b];
    A[(int64_t)(oi + a) * D + ok + b] = s;
    if (oi != ok) A[(int64_t)(ok + b) * D + oi + a] = s;
  }
}

// ---------------------------------------------------------------- dense FP64 tiles

// C = beta C + alpha op(A) op(B), row-major, 64 x 64 tile per CTA.
// lower: only tiles/entries with col <= row.  ktri: the K sum starts at
// max(row tile, col tile) (op(A) = W^T, op(B) = W with W lower triangular).
__global__ void __launch_bounds__(256) gemm64_kernel(int M, int N, int K, double alpha, const double* A, int lda,
                                                     int ta, const double* B, int ldb, int tb, double beta,
                                                     double* C, int ldc, int lower, int ktri) {
  __shared__ double As[16][kT + 1];
  __shared__ double Bs[16][kT + 1];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int r0 = blockIdx.y * kT, c0 = blockIdx.x * kT;
  if (lower && c0 > r0 + kT - 1) return;
  double acc[4][4] = {};
  int kstart = ktri ? (max(r0, c0) / 16) * 16 : 0;
  for (int k0 = kstart; k0 < K; k0 += 16) {
    for (int idx = tid; idx < 16 * kT; idx += 256) {
      const int k = idx / kT, x = idx % kT;
      const int gi = r0 + x, gk = k0 + k, gj = c0 + x;
      As[k][x] = (gi < M && gk < K) ? (ta ? A[(int64_t)gk * lda + gi] : A[(int64_t)gi * lda + gk]) : 0.0;
      Bs[k][x] = (gj < N && gk < K) ? (tb ? B[(int64_t)gj * ldb + gk] : B[(int64_t)gk * ldb + gj]) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      double a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = As[k][ty + 16 * u];
        b[u] = Bs[k][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = r0 + ty + 16 * u;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int j = c0 + tx + 16 * v;
      if (i < M && j < N && (!lower || j <= i)) {
        double* pc = C + (int64_t)i * ldc + j;
        *pc = (beta == 0.0 ? 0.0 : beta * *pc) + alpha * acc[u][v];
      }
    }
  }
}

// Cholesky of the n x n (n <= 64) diagonal block at A (row-major, ld lda),
// in place (lower, upper part zeroed), and the inverse of the factor into
// Dinv (64 x 64, row-major, ld 64).
__global__ void __launch_bounds__(256) potrf64_kernel(double* A, int lda, int n, double* Dinv, int* status) {
  __shared__ double a[kT][kT + 1];
  __shared__ double b[kT][kT + 1];
  __shared__ double rinv[kT];
  const int tid = threadIdx.x;
  for (int idx = tid; idx < kT * kT; idx += 256) {
    const int i = idx / kT, j = idx % kT;
    a[i][j] = (i < n && j < n && j <= i) ? A[(int64_t)i * lda + j] : 0.0;
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (tid == 0) {
      double d = a[k][k];
      if (!(d > 0.0)) {
        atomicOr(status, kStatNotSPD);
        d = 1.0;
      }
      d = sqrt(d);
      a[k][k] = d;
      rinv[k] = 1.0 / d;
    }
    __syncthreads();
    for (int i = k + 1 + tid; i < n; i += 256) a[i][k] *= rinv[k];
    __syncthreads();
    const int rem = n - k - 1;
    for (int idx = tid; idx < rem * rem; idx += 256) {
      const int i = k + 1 + idx / rem, j = k + 1 + idx % rem;
      if (j <= i) a[i][j] -= a[i][k] * a[j][k];
    }
    __syncthreads();
  }
  // inverse of the factor, column j by thread j
  if (tid < kT) {
    const int j = tid;
    for (int i = 0; i < kT; ++i) b[i][j] = 0.0;
    if (j < n) {
      b[j][j] = rinv[j];
      for (int i = j + 1; i < n; ++i) {
        double s = 0.0;
        for (int k = j; k < i; ++k) s += a[i][k] * b[k][j];
        b[i][j] = -s * rinv[i];
      }
    }
  }
  __syncthreads();
  for (int idx = tid; idx < kT * kT; idx += 256) {
    const int i = idx / kT, j = idx % kT;
    if (i < n && j < n) A[(int64_t)i * lda + j] = j <= i ? a[i][j] : 0.0;
    Dinv[i * kT + j] = b[i][j];
  }
}

__global__ void copy2d_kernel(const double* src, int lds, double* dst, int ldd, int rows, int cols, double scale) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < (int64_t)rows * cols; g += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(g / cols), j = (int)(g % cols);
    dst[(int64_t)i * ldd + j] = scale * src[(int64_t)i * lds + j];
  }
}

// ---------------------------------------------------------------- vectors

// r = d - q
__global__ void sub_kernel(const double* d, const double* q, double* r, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) r[i] = d[i] - q[i];
}

// u_i += R_i alpha_i
__global__ void add_Ralpha_kernel(DevPlan P, const int* dofsub, int64_t ndof, const double* R, const double* alpha,
                                  double* u) {
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < ndof; g += (int64_t)gridDim.x * blockDim.x) {
    const SubInfo& S = P.sub[dofsub[g]];
    const int i = (int)(g - S.dof);
    double s = 0.0;
    for (int k = 0; k < S.d; ++k) s += R[S.R + (int64_t)k * S.n + i] * alpha[S.alpha0 + k];
    u[g] += s;
  }
}

// z = A c (D x D row-major), warp per row
__global__ void gemv_kernel(const double* A, const double* c, double* z, int D, double alpha) {
  const int lane = threadIdx.x & 31;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) / 32; row < D; row += gridDim.x * blockDim.x / 32) {
    double acc = 0.0;
    for (int j = lane; j < D; j += 32) acc += A[(int64_t)row * D + j] * c[j];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) z[row] = alpha * acc;
  }
}

}  // namespace

inline int grid_for(int64_t n, int per = 256, int cap = 152 * 16) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, cap));
}

size_t implicit_smem(int nmax, int maxf, bool wide) {
  return ((size_t)nmax + maxf + (wide ? kWideBuf : kThreads / 32 * kWF)) * 8;
}

// The wide CTA takes one subdomain per SM.  With more subdomains than SMs several 256-thread CTAs per SM hide one
// another's latency better on 2D fronts, not on large 3D ones; the line at the SM count is a simple one and not the best
// (options.implicit_cluster overrides it).  Milliseconds with 256 threads / 1 / 2 / 4 wide CTAs: 576 2D heat subdomains
// of 64^2 1.34 / 2.68 / 3.56 / 5.48, 169 of them 0.94 / 1.31 / 1.33 / 1.66; 125 elasticity subdomains of 12^3 5.68 / 2.72 /
// 3.35 / 4.54, 216 of them 6.43 / 5.40 / 5.00 / 7.02; 216 uneven 3D heat subdomains 8.2 / 4.4 / 2.7 / 3.2, 512 of them 8.2 /
// 4.5 / 5.9 / 8.8.
bool implicit_wide(int nsub, int nsm, int nmax, int maxf) {
  return nsub <= nsm && implicit_smem(nmax, maxf, true) + 1024 <= 227 * 1024;
}

static cudaLaunchConfig_t cluster_launch(int ctas, int cluster, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(kWide);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  *at = {};
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)cluster;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

template <int MODE>
static void launch_implicit_mode(int cluster, const DevPlan& P, const int* order, int nsub, int* queue, const double* p,
                                 const double* f, double* qi, double* u, double* uws, int64_t ustride, int nmax,
                                 int maxf, int grid, size_t smem, cudaStream_t st) {
  if (cluster > 1) {
    auto kern = implicit_kernel<MODE, kWide, true>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaLaunchAttribute at;
    cudaLaunchConfig_t cfg = cluster_launch(grid * cluster, cluster, smem, st, &at);
    cudaLaunchKernelEx(&cfg, kern, P, order, nsub, queue, p, f, qi, u, uws, ustride, nmax, maxf);
  } else if (cluster == 1) {
    auto kern = implicit_kernel<MODE, kWide, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, kWide, smem, st>>>(P, order, nsub, queue, p, f, qi, u, uws, ustride, nmax, maxf);
  } else {
    auto kern = implicit_kernel<MODE, kThreads, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, kThreads, smem, st>>>(P, order, nsub, queue, p, f, qi, u, uws, ustride, nmax, maxf);
  }
}

void launch_implicit(int mode, int cluster, const DevPlan& P, const int* order, int nsub, int* queue, const double* p,
                     const double* f, double* qi, double* u, double* uws, int64_t ustride, int nmax, int maxf,
                     int grid, size_t smem, cudaStream_t st) {
  auto fn = mode == 0 ? launch_implicit_mode<0> : mode == 1 ? launch_implicit_mode<1> : launch_implicit_mode<2>;
  fn(cluster, P, order, nsub, queue, p, f, qi, u, uws, ustride, nmax, maxf, grid, smem, st);
}

int implicit_clusters(size_t smem, int cluster) {
  auto kern = implicit_kernel<0, kWide, true>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = cluster_launch(64 * cluster, cluster, smem, 0, &at);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

void launch_inv_blocks(const DevPlan& P, int nsub, cudaStream_t st) {
  inv_block_kernel<<<dim3(32, (unsigned)std::min(nsub, 65535)), 128, 0, st>>>(P, nsub);
}

void launch_unit_scale(const DevPlan& P, int nsub, int nmax, double* d2, cudaStream_t st) {
  // about eight waves of CTAs, one warp per column at most
  const int gx = std::max(1, std::min((nmax + 7) / 8, std::max(4, 152 * 64 / std::max(nsub, 1))));
  unit_scale_kernel<<<dim3((unsigned)gx, (unsigned)std::min(nsub, 65535)), 256, 0, st>>>(P, nsub, d2);
}

int implicit_occupancy(size_t smem) {
  int nb = 0;
  cudaFuncSetAttribute(implicit_kernel<0, kThreads, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, implicit_kernel<0, kThreads, false>, kThreads, smem);
  return std::max(nb, 1);
}

void launch_gather_minus_c(const int* c0, const int* c1, int nlam, const double* qi, const double* c, double* q,
                           cudaStream_t st) {
  gather_minus_c_kernel<<<grid_for(nlam), 256, 0, st>>>(c0, c1, nlam, qi, c, q);
}

void launch_build_G(const DevPlan& P, const int* colsub, int64_t ncols, const double* R, double* G6,
                    cudaStream_t st) {
  build_G_kernel<<<grid_for(ncols), 256, 0, st>>>(P, colsub, ncols, R, G6);
}

void launch_rtf(const DevPlan& P, int nsub, const double* R, const double* f, double* e, cudaStream_t st) {
  rtf_kernel<<<grid_for((int64_t)nsub * 6 * 32), 256, 0, st>>>(P, nsub, R, f, e);
}

void launch_gt(const DevPlan& P, int nsub, const double* G6, const double* x, double* c, cudaStream_t st) {
  gt_kernel<<<grid_for((int64_t)nsub * 6 * 32), 256, 0, st>>>(P, nsub, G6, x, c);
}

void launch_gz(const DevPlan& P, const int* colsub, const int* c0, const int* c1, int nlam, const double* G6,
               const double* x, const double* z, double sgn, double* out, cudaStream_t st) {
  gz_kernel<<<grid_for(nlam), 256, 0, st>>>(P, colsub, c0, c1, nlam, G6, x, z, sgn, out);
}

void launch_gtg(const int4* pairs, int npairs, const int2* plist, const double* G6, double* A, int D,
                cudaStream_t st) {
  if (npairs > 0) gtg_kernel<<<std::min(npairs, 152 * 32), 64, 0, st>>>(pairs, npairs, plist, G6, A, D);
}

void launch_gemm64(int M, int N, int K, double alpha, const double* A, int lda, int ta, const double* B, int ldb,
                   int tb, double beta, double* C, int ldc, int lower, int ktri, cudaStream_t st) {
  if (M <= 0 || N <= 0) return;
  dim3 grid((N + kT - 1) / kT, (M + kT - 1) / kT);
  gemm64_kernel<<<grid, 256, 0, st>>>(M, N, K, alpha, A, lda, ta, B, ldb, tb, beta, C, ldc, lower, ktri);
}

void launch_potrf64(double* A, int lda, int n, double* Dinv, int* status, cudaStream_t st) {
  potrf64_kernel<<<1, 256, 0, st>>>(A, lda, n, Dinv, status);
}

void launch_copy2d(const double* src, int lds, double* dst, int ldd, int rows, int cols, double scale,
                   cudaStream_t st) {
  if (rows > 0 && cols > 0)
    copy2d_kernel<<<grid_for((int64_t)rows * cols), 256, 0, st>>>(src, lds, dst, ldd, rows, cols, scale);
}

void launch_sub(const double* d, const double* q, double* r, int n, cudaStream_t st) {
  sub_kernel<<<grid_for(n), 256, 0, st>>>(d, q, r, n);
}

void launch_add_Ralpha(const DevPlan& P, const int* dofsub, int64_t ndof, const double* R, const double* alpha,
                       double* u, cudaStream_t st) {
  add_Ralpha_kernel<<<grid_for(ndof), 256, 0, st>>>(P, dofsub, ndof, R, alpha, u);
}

void launch_gemv(const double* A, const double* c, double* z, int D, double alpha, cudaStream_t st) {
  if (D > 0) gemv_kernel<<<grid_for((int64_t)D * 32), 256, 0, st>>>(A, c, z, D, alpha);
}

}  // namespace feti
