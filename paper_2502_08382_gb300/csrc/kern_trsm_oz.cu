// FP64 pruned forward solve X_i = L_i^{-1} P_i B_i^T of the large fronts (P.sn_big) on the tensor cores, after
// trsm_kernel has solved everything below them (its update blocks for large parents are handed over in global memory).
//
// dig_l_kernel first cuts the large panels into digits (oz.cuh), 128 columns at a time: the inverses of the 32 x 32
// diagonal blocks, the block's own rows and the rows below it.  trsm_oz_kernel then takes one block of 128 or 256
// sorted columns of one subdomain per work item (the columns are independent) up the tree of its large fronts.  The
// right-hand sides of a front are rows here, X^T (J x w): per 128 columns of the front, in steps of 32,
//   X^T_b <- A L_bb^{-T}              (K = 32, the explicit inverse, as the FP64-pipe solve uses it; cut with opposite
//                                      shifts of L's pivots' exponents, oz.cuh),
//   the block's later columns         -= X^T_b L^T (K = 32),
// and after the block the later columns of the front and its update block -= X^T L^T with K = 128.  The tiles are
// those of oz_engine.cuh.
//
// What bounds it: the staging of the digits for wide fronts, the latency of the 32-column steps for narrow ones; two
// 128-column tiles per item share that latency when there are enough items.  Measured (before: all fronts on the FP64
// pipe by trsm_kernel): 64 uneven 3D heat subdomains 78.8 ms -> 13.7 + 4.9 (small fronts) + 1.0 (digits of L), 27
// elasticity subdomains of 12^3 58.6 -> 10.0 + 1.3 + 0.7.
#include <algorithm>
#include <cuda_bf16.h>

#include "chol_common.cuh"
#include "common.cuh"
#include "kernels.h"
#include "oz_engine.cuh"

namespace feti {
namespace {

constexpr int kXDyn = 1024 + kCStages * kCStage;
constexpr int kInRows = 160;  // rows of the in-block digits: 128 and the overhang of a 64-column tile

// Digit layout of one 128-column block of a large panel (byte offsets within the block; all multiples of 512).
struct LdBlock {
  int64_t inv, invex, in, inex, piv, bel, belex, end;  // piv: the shifts of the block's columns
  int K, nck, own, ownp, botp;  // columns, chunks, own rows below the block (padded to 64), bottom rows padded to 64
};
__host__ __device__ inline LdBlock ld_block(int w, int r, int kB) {
  LdBlock b;
  b.K = w - kB < 128 ? w - kB : 128;
  b.nck = (b.K + 31) / 32;
  b.own = w - kB - b.K;
  b.ownp = (b.own + 63) / 64 * 64;
  b.botp = (r + 63) / 64 * 64;
  b.inv = 0;
  b.invex = 4 * kDig * kCB;
  b.in = b.invex + 512;
  b.inex = b.in + (int64_t)kDig * b.nck * kInRows * 64;
  b.piv = b.inex + 1024;
  b.bel = b.piv + 512;
  b.belex = b.bel + (int64_t)kDig * b.nck * (b.ownp + b.botp) * 64;
  b.end = (b.belex + (int64_t)(b.ownp + b.botp) * 4 + 511) / 512 * 512;
  return b;
}

// items: (subdomain, supernode, first column of the block, byte offset / 512 of the block in the subdomain's digits)
__global__ void __launch_bounds__(256) dig_l_kernel(DevPlan P, const int4* items, char* LD) {
  __shared__ double D[4][kNB][kNB + 1];
  const int4 it = items[blockIdx.x];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const SubInfo& S = P.sub[it.x];
  const int gs = S.sn0 + it.y, w = P.sn_w[gs], r = P.sn_r[gs], f = w + r, kB = it.z;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  const LdBlock b = ld_block(w, r, kB);
  char* out = LD + S.ld + (int64_t)it.w * 512;
  const int kE = kB + b.K;
  if (warp < 4) {
    // the inverse of diagonal block `warp`, lane = column
    const int k0 = kB + 32 * warp, nb = min(32, kE - k0);
    double(*d)[kNB + 1] = D[warp];
    const int es = lane < nb ? dig_pivot_shift(Ls[(int64_t)(k0 + lane) * f + k0 + lane]) : 0;
    reinterpret_cast<int*>(out + b.piv)[32 * warp + lane] = es;
    for (int k = 0; k < kNB; ++k)
      d[lane][k] = (lane < nb && k <= lane && k < nb) ? Ls[(int64_t)(k0 + k) * f + k0 + lane] : (lane == k ? 1.0 : 0.0);
    __syncwarp();
    double m[kNB];
#pragma unroll
    for (int i = 0; i < kNB; ++i) {
      double a = i == lane ? 1.0 : 0.0;
#pragma unroll
      for (int k = 0; k < i; ++k) a = fma(-d[i][k], m[k], a);
      m[i] = a / d[i][i];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kNB; ++i) d[i][lane] = (i < nb && lane < nb) ? m[i] : 0.0;
    __syncwarp();
    for (int i0 = 0; i0 < kNB; i0 += 8) {
      const int i = i0 + (lane >> 2), q = lane & 3;
      double v[8];
      int sh[8], mx = kKeyZero;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        v[e] = d[i][q * 8 + e];
        sh[e] = -__shfl_sync(0xffffffffu, es, q * 8 + e);
        mx = max(mx, dig_key(v[e], sh[e]));
      }
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const int ex = dig_key_exponent(mx);
      if (q == 0) reinterpret_cast<int*>(out + b.invex)[32 * warp + i] = ex;
      uint64_t c[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) c[e] = dig_cut(v[e], ex + sh[e]);
#pragma unroll
      for (int p = 0; p < kDig; ++p)
        *reinterpret_cast<uint4*>(out + b.inv + (warp * kDig + p) * kCB + i * 64 + ((q ^ ((i >> 1) & 3)) << 4)) =
            make_uint4(dig_pair(c[0], c[1], p), dig_pair(c[2], c[3], p), dig_pair(c[4], c[5], p),
                       dig_pair(c[6], c[7], p));
    }
  } else {
    dig_rows<4>(ColMajor{Ls + (int64_t)kB * f + kB, f}, b.K, b.K, 0, 128, out + b.in, b.nck, kInRows,
                reinterpret_cast<int*>(out + b.inex), warp - 4, 4);
  }
  const int np = b.ownp + b.botp;
  int* ex = reinterpret_cast<int*>(out + b.belex);
  dig_rows<4>(ColMajor{Ls + (int64_t)kB * f + kE, f}, b.own, b.K, 0, b.ownp, out + b.bel, b.nck, np, ex, warp, 8);
  dig_rows<4>(ColMajor{Ls + (int64_t)kB * f + w, f}, r, b.K, 0, b.botp, out + b.bel + (int64_t)b.ownp * 64, b.nck, np,
              ex + b.ownp, warp, 8);
}


// X^T_b = A L_bb^{-T}: rows of the item, the ncol <= 32 columns of the step
struct SolveJob {
  static constexpr int kUnits = 1;
  static constexpr bool kBSmem = false;
  const char *SA, *SB;
  const int *EX, *EXB;
  int64_t digA, digB;
  int nck, n, ncol;
  double* X;  // row 0, the step's first column
  int64_t wp;
  __device__ __forceinline__ void tile(int t, int& tm, int& tn) const {
    tm = t;
    tn = 0;
  }
  __device__ __forceinline__ const char* a(int tm, int) const { return SA + (int64_t)tm * kCM * 64; }
  __device__ __forceinline__ const char* b(int, int) const { return SB; }
  __device__ __forceinline__ int begin(int ri) const { return ri < n ? __ldcg(EX + ri) : 0; }
  __device__ __forceinline__ int load(int ri, int cb, double (&)[16]) const {
    return ri < n ? min(16, ncol - cb) : 0;
  }
  __device__ __forceinline__ int4 ec4(int c) const { return __ldg(reinterpret_cast<const int4*>(EXB + c)); }
  __device__ __forceinline__ void store4(int ri, int c, int n4, const double*, const double* t) const {
    double* p = X + (int64_t)ri * wp + c;
    if (n4 == 4) {
      st4(p, t[0], t[1], t[2], t[3]);
      return;
    }
#pragma unroll
    for (int e = 0; e < 3; ++e)
      if (e < n4) p[e] = t[e];
  }
};

// C -= X^T L^T: column c of the padded B rows is own column c (c < own) of X, or column c - ownp (< nbot) of the update
// block W
struct RectJob {
  static constexpr int kUnits = 2;
  static constexpr bool kBSmem = false;
  const char *SA, *SB;
  const int *EX, *EXB;
  int64_t digA, digB;
  int nck, n, npad, npadB, ntn, own, ownp, nbot;
  double *X, *W;  // row 0; X at the first own column
  int64_t wp, rp;
  __device__ __forceinline__ void tile(int t, int& tm, int& tn) const {
    tm = t / ntn;
    tn = t - tm * ntn;
  }
  __device__ __forceinline__ const char* a(int tm, int c) const {
    return SA + ((int64_t)c * npad + (int64_t)tm * kCM) * 64;
  }
  __device__ __forceinline__ const char* b(int tn, int c) const {
    return SB + ((int64_t)c * npadB + (int64_t)tn * 64) * 64;
  }
  __device__ __forceinline__ int begin(int ri) const { return ri < n ? __ldcg(EX + ri) : 0; }
  __device__ __forceinline__ double* at(int ri, int c) const {
    return c < ownp ? X + (int64_t)ri * wp + c : W + (int64_t)ri * rp + (c - ownp);
  }
  __device__ __forceinline__ int load(int ri, int cb, double (&cv)[16]) const {
    const int nc = ri >= n ? 0 : min(16, cb < ownp ? own - cb : ownp + nbot - cb);
    if (nc <= 0) return 0;
    const double* p = at(ri, cb);
    if (nc == 16) {
#pragma unroll
      for (int e = 0; e < 16; e += 4) ld4(p + e, cv + e);
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) cv[e] = e < nc ? __ldcg(p + e) : 0.0;
    }
    return nc;
  }
  __device__ __forceinline__ int4 ec4(int c) const { return __ldg(reinterpret_cast<const int4*>(EXB + c)); }
  __device__ __forceinline__ void store4(int ri, int c, int n4, const double* cv, const double* t) const {
    double* p = at(ri, c);
    if (n4 == 4) {
      st4(p, cv[0] - t[0], cv[1] - t[1], cv[2] - t[2], cv[3] - t[3]);
      return;
    }
#pragma unroll
    for (int e = 0; e < 3; ++e)
      if (e < n4) p[e] = cv[e] - t[e];
  }
};

// items: (subdomain, first sorted column), cw columns each (128 or 256)
__global__ void __launch_bounds__(kCT, 1)
    trsm_oz_kernel(DevPlan P, const int2* items, int nitems, int cw, int* queue, const char* LD, const double* hand,
                   double* X, double* ws, int64_t ws_stride, char* scratch, int64_t scratch_stride, int* status) {
  extern __shared__ uint8_t xo_raw[];
  __shared__ uint64_t full[kCStages], empty[kCStages], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int k = 0; k < kCStages; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&empty[k], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&accf[k], 1);
      mbar_init(&acce[k], 8);
    }
    mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    abort_s = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  CtState st{};
  st.ring = xo_raw + ((1024u - (smem_u32(xo_raw) & 1023u)) & 1023u);
  st.full = full;
  st.empty = empty;
  st.accf = accf;
  st.acce = acce;
  st.drain = &drain;
  st.abort = &abort_s;
  st.tmem = tmem_s;
  double* stack = ws + (int64_t)blockIdx.x * ws_stride;
  char* SL = scratch + (int64_t)blockIdx.x * scratch_stride;
  char* S2 = SL + (int64_t)cw * 512;
  int* EX1 = reinterpret_cast<int*>(SL + (int64_t)cw * 1024);
  int* EX2 = EX1 + cw;
  int* EX = reinterpret_cast<int*>(SL + (int64_t)cw * 2048);
  for (;;) {
    const int it = pop_item(queue);
    if (it >= nitems) break;
    const SubInfo S = P.sub[items[it].x];
    const int ca = items[it].y, cb = ca + cw;
    double* Xsub = X + S.X;
    for (int a = 0; a < S.nact; ++a) {
      const int s = P.act[S.act0 + a];
      const int gs = S.sn0 + s, bs = S.bsn0 + s;
      if (!P.sn_big[gs]) continue;
      const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs];
      const int wp = (w + 7) & ~7, rp = (r + 7) & ~7;
      const int jb = max(P.jb[bs], ca), je = min(P.je[bs], cb), jo = max(P.jo[bs], ca);
      const int J = je - jb;
      if (J <= 0) continue;
      double* Xs = Xsub + P.Xofs[bs] + (int64_t)(jb - P.jb[bs]) * wp;
      double* W = stack + P.tx_ofs[gs] * cw;  // formed where the parent reads it
      for (int64_t idx = 4 * tid; idx < (int64_t)wp * J; idx += 4 * kCT) st4(Xs + idx, 0.0, 0.0, 0.0, 0.0);
      for (int64_t idx = 4 * tid; idx < (int64_t)rp * J; idx += 4 * kCT) st4(W + idx, 0.0, 0.0, 0.0, 0.0);
      __syncthreads();
      for (int j = jo + tid; j < je; j += kCT) Xs[(int64_t)(j - jb) * wp + P.spos[S.col0 + j] - c0] = P.qsign[S.qcol + j];
      for (int c = P.ch_off[gs]; c < P.ch_off[gs + 1]; ++c) {
        const int lc = P.ch_list[c];
        const int gc = S.sn0 + lc, bc = S.bsn0 + lc;
        const int jbc = max(P.jb[bc], ca), Jc = min(P.je[bc], cb) - jbc;
        if (Jc <= 0) continue;
        const int rc = P.sn_r[gc], coff = jbc - jb;
        const bool big = P.sn_big[gc] != 0;
        const int ldc = big ? (rc + 7) & ~7 : rc;
        const double* U = big ? stack + P.tx_ofs[gc] * cw : hand + S.th + P.th_ofs[bc] + (int64_t)(jbc - P.jb[bc]) * rc;
        const int* rl = P.rel + P.rel_off[gc];
        // children own disjoint column ranges; a column per warp, kFly entries per lane in flight
        constexpr int kFly = 8;
        for (int col = warp; col < Jc; col += kCT / 32) {
          double* Xc = Xs + (int64_t)(coff + col) * wp;
          double* Wc = W + (int64_t)(coff + col) * rp - w;
          const double* Uc = U + (int64_t)col * ldc;
          for (int a0 = lane; a0 < rc; a0 += 32 * kFly) {
            double* dst[kFly];
            double v[kFly], cur[kFly];
#pragma unroll
            for (int u = 0; u < kFly; ++u) {
              const int a2 = a0 + 32 * u;
              const int ra = a2 < rc ? rl[a2] : 0;
              v[u] = a2 < rc ? __ldcg(Uc + a2) : 0.0;
              dst[u] = a2 < rc ? (ra < w ? Xc : Wc) + ra : nullptr;
            }
#pragma unroll
            for (int u = 0; u < kFly; ++u) cur[u] = dst[u] ? __ldcg(dst[u]) : 0.0;
#pragma unroll
            for (int u = 0; u < kFly; ++u)
              if (dst[u]) *dst[u] = cur[u] + v[u];
          }
        }
      }
      __syncthreads();
      const int ntm = (J + kCM - 1) / kCM, npad = ntm * kCM;
      const char* ld = LD + S.ld + P.ld_ofs[gs] * 512;
      for (int kB = 0; kB < w; kB += 128) {
        const LdBlock b = ld_block(w, r, kB);
        const int kE = kB + b.K;
        for (int kb = kB, sb = 0; kb < kE; kb += 32, ++sb) {
          const int ke = min(kE, kb + 32), nbk = ke - kb;
          dig_rows<1>(Shifted<RowMajor, false>{{Xs + kb, wp}, reinterpret_cast<const int*>(ld + b.piv) + 32 * sb}, J,
                      nbk, 0, npad, SL, 1, npad, EX1, warp, kCT / 32);
          SolveJob sj{SL, ld + b.inv + sb * kDig * kCB, EX1, reinterpret_cast<const int*>(ld + b.invex) + 32 * sb,
                      (int64_t)npad * 64, kCB, 1, J, nbk, Xs + kb, wp};
          dig_product(st, sj, 0, 1, ntm);
          if (ke < kE) {
            dig_rows<1>(RowMajor{Xs + kb, wp}, J, nbk, 0, npad, S2, 1, npad, EX2, warp, kCT / 32);
            const int own = kE - ke, ntn = (own + 63) / 64;
            RectJob rj{S2, ld + b.in + ((int64_t)sb * kInRows + (ke - kB)) * 64, EX2,
                       reinterpret_cast<const int*>(ld + b.inex) + (ke - kB), (int64_t)npad * 64,
                       (int64_t)b.nck * kInRows * 64, 1, J, npad, kInRows, ntn, own, ntn * 64, 0, Xs + ke, W, wp, rp};
            dig_product(st, rj, 0, 1, ntm * ntn);
          }
        }
        if (b.ownp + b.botp > 0) {
          dig_rows<4>(RowMajor{Xs + kB, wp}, J, b.K, 0, npad, SL, b.nck, npad, EX, warp, kCT / 32);
          const int np = b.ownp + b.botp, ntn = np / 64;
          RectJob rj{SL, ld + b.bel, EX, reinterpret_cast<const int*>(ld + b.belex), (int64_t)b.nck * npad * 64,
                     (int64_t)b.nck * np * 64, b.nck, J, npad, np, ntn, b.own, b.ownp, r, Xs + kE, W, wp, rp};
          dig_product(st, rj, 0, 1, ntm * ntn);
        }
        ld += b.end;
      }
      __syncthreads();
    }
  }
  if (tid == 0 && abort_s) atomicOr(status, kStatTimeout);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(st.tmem), "r"(512));
  }
}

}  // namespace

int64_t trsm_oz_block_bytes(int w, int r, int kB) { return ld_block(w, r, kB).end; }

int64_t trsm_oz_scratch(int cw) { return (int64_t)cw * (2048 + 512); }

void launch_dig_l(const DevPlan& P, const int4* items, int nitems, void* LD, cudaStream_t st) {
  if (nitems > 0) dig_l_kernel<<<nitems, 256, 0, st>>>(P, items, (char*)LD);
}

void launch_trsm_oz(const DevPlan& P, const int2* items, int nitems, int cw, int* queue, const void* LD,
                    const double* hand, double* X, double* ws, int64_t ws_stride, void* scratch,
                    int64_t scratch_stride, int grid, int* status, cudaStream_t st) {
  if (nitems <= 0) return;
  cudaFuncSetAttribute(trsm_oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kXDyn);
  trsm_oz_kernel<<<std::min(grid, nitems), kCT, kXDyn, st>>>(P, items, nitems, cw, queue, (const char*)LD, hand, X, ws,
                                                            ws_stride, (char*)scratch, scratch_stride, status);
}

}  // namespace feti
