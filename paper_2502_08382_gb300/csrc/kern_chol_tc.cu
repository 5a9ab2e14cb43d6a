// Tensor-core Cholesky of the large fronts (P.sn_big: the fronts at least big_f wide and their ancestors, the top of
// each supernodal tree), after chol_kernel has done everything below them.
//
// A front's w own columns go in blocks of 128, and inside a block in steps of 32:
//   pivot   the 32 x 32 block's factor L_bb and inverse on the FP64 pipe (eight warps);
//   panel   the rows below, X = A L_bb^{-T}, on the tensor cores (K = 32, N = 32), A's columns and those of the inverse
//           cut with opposite shifts of half the diagonal's exponents (oz.cuh);
//   block   the block's later columns, C -= X X^T, on the tensor cores (K = 32);
// after the block the rest of the front takes C -= X X^T with K = 128.  All products run by exact slicing of FP64
// into bf16 digits (oz.cuh); a product costs one FP64 addition per entry of C, the rest of the epilogue (sums of the
// accumulators, normalisation, rounding to nearest) is integer arithmetic, because one FP64 instruction of a warp
// takes 64 clocks of its scheduler here.
//
// A cluster of C CTAs (1, 2, 4 or 8; one CTA per SM) takes one front at a time: every CTA repeats the pivot, the rows
// of the panel and the tiles of the updates are dealt out, and barriers between the phases order the accesses (all
// shared data is in global memory).  C is as large as keeps the CTAs within the SMs (chol_tc_cluster).
//
// Measured (the kernel alone; before: 9 slices of 7 bits, 45 MMAs of N = 32 per 16-deep step, one CTA per front, the
// panel on the FP64 pipe, updates copied to the stack): 64 uneven 3D heat subdomains 50.3 -> 13.2 ms (C = 2), 27
// elasticity subdomains of 12^3 59.0 -> 9.4 ms (C = 4), 64 of them 66.0 -> 15.0 ms (C = 2), 125 uneven 3D heat
// subdomains 40.8 -> 9.3 ms (C = 1; these fronts were partly chol_kernel's before).  Of this, forming the bottom block
// in place and assembling by columns took 64 elasticity subdomains from 20.7 to 15.4 ms (assembly and copy were 36%).
// What bounds it now: on wide fronts the staging of the digits (96 KB from L2 per 2304 clocks of MMA), on fronts of a
// few hundred rows the pivot blocks (16 k clocks of FP64 work for 32 columns) and the barriers between the phases.
//
// The products run on the tiles of oz_engine.cuh.  Every mbarrier wait is bounded; a CTA that gives up keeps to the
// cluster's barriers and skips its work.
#include <algorithm>
#include <cuda_bf16.h>

#include "chol_common.cuh"
#include "cluster.cuh"
#include "common.cuh"
#include "kernels.h"
#include "oz_engine.cuh"

namespace feti {
namespace {

constexpr int kCBlk = 128;                                      // columns per block
constexpr int kCDyn = 1024 + kCStages * kCStage + kDig * kCB;  // + the digits of L_bb^{-1}

struct PivotSmem {
  double D[kNB][kNB + 1];   // the block, then L_bb
  double M[kNB][kNB + 1];   // L_bb^{-1}
  double col[2][kNB];       // the pivot column below the pivot (double-buffered)
  double cols[2][kNB];      // the same times the reciprocal pivot, which stands in the other places
};
static_assert(sizeof(PivotSmem) <= kCStage, "the pivot's buffers alias the stage ring");

// barrier of all threads of the cluster; orders their global accesses (generic and bulk copies)
__device__ __forceinline__ void cl_sync() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
  cl_barrier();
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
// The panel: Out[row, j] = (A L_bb^{-T})[row, j] for j < ncol to the front's columns kb + j, rows i0 + row.
struct PanelJob {
  static constexpr int kUnits = 1;
  static constexpr bool kBSmem = true;
  const char* SA;
  const int *EX, *EXB;
  int64_t digA, digB;
  int nck, n, ncol;
  double* out;  // row 0 of column kb
  int64_t f;
  __device__ __forceinline__ void tile(int t, int& tm, int& tn) const {
    tm = t;
    tn = 0;
  }
  __device__ __forceinline__ const char* a(int tm, int) const { return SA + (int64_t)tm * kCM * 64; }
  __device__ __forceinline__ const char* b(int, int) const { return nullptr; }
  __device__ __forceinline__ int begin(int ri) const { return ri < n ? __ldcg(EX + ri) : 0; }
  __device__ __forceinline__ int load(int ri, int cb, double (&)[16]) const {
    return ri < n ? min(16, ncol - cb) : 0;
  }
  __device__ __forceinline__ int4 ec4(int c) const { return *reinterpret_cast<const int4*>(EXB + c); }
  __device__ __forceinline__ void store4(int ri, int c, int n4, const double*, const double* t) const {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < n4) out[(int64_t)(c + e) * f + ri] = t[e];
  }
};

// C -= A A^T for the columns [i0, i0 + ncol) of the front on and below the diagonal, C in Ls (columns < w) or W;
// n = rows of A, row block tm holds min(2 (tm + 1), ntn) blocks of 64 columns.
struct UpdateJob {
  static constexpr int kUnits = 2;
  static constexpr bool kBSmem = false;
  const char* SA;
  const int* EX;
  int64_t digA, digB;
  int nck, n, npad, ntn, ncol, i0, w, r;
  double *Ls, *W;
  int64_t f;
  __device__ __forceinline__ void tile(int t, int& tm, int& tn) const {
    const int nfull = (ntn + 1) / 2;  // the row blocks before this one have fewer column blocks
    // sum_{m < tm} 2 (m + 1) = tm (tm + 1)
    tm = (int)((sqrtf(4.f * t + 1.f) - 1.f) * 0.5f);
    while ((tm + 1) * (tm + 2) <= t) ++tm;
    while (tm * (tm + 1) > t) --tm;
    if (tm >= nfull - 1) {
      const int q = t - (nfull - 1) * nfull;  // past the tiles of the first nfull - 1 row blocks
      tm = nfull - 1 + q / ntn;
      tn = q % ntn;
      return;
    }
    tn = t - tm * (tm + 1);
  }
  __device__ __forceinline__ const char* a(int tm, int c) const { return SA + ((int64_t)c * npad + (int64_t)tm * kCM) * 64; }
  __device__ __forceinline__ const char* b(int tn, int c) const { return SA + ((int64_t)c * npad + (int64_t)tn * 64) * 64; }
  __device__ __forceinline__ int begin(int ri) const { return ri < n ? __ldcg(EX + ri) : 0; }
  __device__ __forceinline__ double* at(int ri, int c) const {
    const int gi = i0 + ri, gj = i0 + c;
    return gj < w ? Ls + (int64_t)gj * f + gi : W + (int64_t)(gj - w) * r + (gi - w);
  }
  __device__ __forceinline__ int load(int ri, int cb, double (&cv)[16]) const {
    const int nc = ri < n ? min(16, min(ncol, ri + 1) - cb) : 0;
#pragma unroll
    for (int e = 0; e < 16; ++e) cv[e] = e < nc ? __ldcg(at(ri, cb + e)) : 0.0;
    return nc;
  }
  __device__ __forceinline__ int4 ec4(int c) const { return __ldcg(reinterpret_cast<const int4*>(EX + c)); }
  __device__ __forceinline__ void store4(int ri, int c, int n4, const double* cv, const double* t) const {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < n4) *at(ri, c + e) = cv[e] - t[e];
  }
};

// L_bb and L_bb^{-1} of the nbk x nbk block in sm.D by the CTA's first eight warps: lane = row, warp v holds columns
// v, v + 8, v + 16, v + 24 of the block (from the diagonal on) and of the inverse (up to the diagonal).  Elimination of
// [A | I]: step k subtracts column k (times the row k of the inverse part, whose rows are scaled by the reciprocal
// pivots at the end).  L_bb goes to sm.D, its inverse to sm.M.
__device__ __forceinline__ void pivot_block(PivotSmem& sm, int nbk, int* bad) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (warp >= 8) return;
  double a[4], m[4], rsl = 1.0;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int j = warp + 8 * u;
    a[u] = sm.D[lane][j];
    m[u] = lane == j ? 1.0 : 0.0;
  }
  for (int k = 0; k < nbk; ++k) {
    double *col = sm.col[k & 1], *cols = sm.cols[k & 1];
    const int ku = k >> 3;
    if ((k & 7) == warp) {
      double v = 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u == ku) v = a[u];
      double d = __shfl_sync(0xffffffffu, v, k);
      if (!(d > 0.0)) {  // not positive: reported, replaced by 1 so that the sweep stays finite
        if (lane == 0) *bad = 1;
        d = 1.0;
        if (lane == k) v = 1.0;
      }
      const double rs = rsqrt(d);
      v *= rs;  // lane k: the pivot d / sqrt(d)
      if (lane >= k) sm.D[lane][k] = v;
      col[lane] = lane > k ? v : 0.0;
      cols[lane] = lane > k ? v * rs : rs;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const double l = col[lane], ls = lane > k ? cols[lane] : 0.0;
    if (lane == k) rsl = cols[k];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = warp + 8 * u;
      if (j > k && j < nbk) a[u] = fma(-l, col[j], a[u]);
      if (j <= k) m[u] = fma(-ls, __shfl_sync(0xffffffffu, m[u], k), m[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int j = warp + 8 * u;
    sm.M[lane][j] = (lane < nbk && j < nbk && lane >= j) ? m[u] * rsl : 0.0;
  }
}

// The digits of L_bb^{-1} (rows j < 32, K = 32, shifts -es) into the panel's B operand in shared memory, and its row
// exponents.
__device__ __forceinline__ void dig_inverse(const PivotSmem& sm, const int* es, uint8_t* bpan, int* EXB) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, q = lane & 3;
  if (warp >= 4) return;
  const int i = warp * 8 + (lane >> 2);
  double v[8];
  int mx = kKeyZero;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    v[e] = sm.M[i][q * 8 + e];
    mx = max(mx, dig_key(v[e], -es[q * 8 + e]));
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  const int ex = dig_key_exponent(mx);
  if (q == 0) EXB[i] = ex;
  uint64_t w[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) w[e] = dig_cut(v[e], ex - es[q * 8 + e]);
#pragma unroll
  for (int p = 0; p < kDig; ++p)
    *reinterpret_cast<uint4*>(bpan + p * kCB + i * 64 + ((q ^ ((i >> 1) & 3)) << 4)) =
        make_uint4(dig_pair(w[0], w[1], p), dig_pair(w[2], w[3], p), dig_pair(w[4], w[5], p),
                   dig_pair(w[6], w[7], p));
}

// Assemble a front in global memory: the f x w panel Ls (column-major, in the factor's storage) and the r x r bottom
// block W (on and below its diagonal), from the K entries, the fixing-DOF penalty rho and the children's update blocks
// (workspace or hand-over slots), the work dealt to all warps of the cluster by columns: L2 latency bounds it, so a
// lane has kFly entries of a column in flight, and no warp meets the upper triangle or a division.
__device__ __forceinline__ void assemble_cluster(const DevPlan& P, const SubInfo& S, int s, const double* K, double* L,
                                                 double rho, double* W, const double* stack, const double* hand,
                                                 int gtid, int gthreads) {
  const int gs = S.sn0 + s;
  const int w = P.sn_w[gs], r = P.sn_r[gs], f = w + r;
  double* Ls = L + P.Lofs[gs];
  for (int64_t idx = gtid; idx < (int64_t)f * w; idx += gthreads) Ls[idx] = 0.0;
  const int gw = gtid / 32, lane = gtid % 32, nw = gthreads / 32;
  constexpr int kFly = 8;
  for (int j = gw; j < r; j += nw)
    for (int i = j + lane; i < r; i += 32) W[(int64_t)j * r + i] = 0.0;
  cl_sync();
  for (int64_t k = P.kmap_off[gs] + gtid; k < P.kmap_off[gs + 1]; k += gthreads) L[P.kmap_dst[k]] = K[P.kmap_src[k]];
  cl_sync();
  for (int k = gtid; k < S.nfix; k += gthreads)
    if (P.fix_sn[S.fix0 + k] == s) {
      double* d = L + P.fix_pos[S.fix0 + k];
      *d = __ldcg(d) + rho;
    }
  for (int c = P.ch_off[gs]; c < P.ch_off[gs + 1]; ++c) {
    const int gc = S.sn0 + P.ch_list[c];
    const int rc = P.sn_r[gc];
    const double* U = child_update(P, gc, stack, nullptr, hand);
    const int* rl = P.rel + P.rel_off[gc];
    cl_sync();
    for (int b = gw; b < rc; b += nw) {
      const int rb = rl[b];
      double* dst = rb < w ? Ls + (int64_t)rb * f : W + (int64_t)(rb - w) * r - w;
      const double* src = U + (int64_t)b * rc;
      for (int a0 = b + lane; a0 < rc; a0 += 32 * kFly) {
        int ra[kFly];
        double v[kFly], cur[kFly];
#pragma unroll
        for (int u = 0; u < kFly; ++u) {
          const int a = a0 + 32 * u;
          ra[u] = a < rc ? rl[a] : -1;
          v[u] = a < rc ? __ldcg(src + a) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kFly; ++u) cur[u] = ra[u] >= 0 ? __ldcg(dst + ra[u]) : 0.0;
#pragma unroll
        for (int u = 0; u < kFly; ++u)
          if (ra[u] >= 0) dst[ra[u]] = cur[u] + v[u];
      }
    }
  }
  cl_sync();
}

// Items: one task of the plan's split (subdomain, task, global task id, parent's global task id), children before
// parents.  The fronts' children outside the large set handed their update blocks over (chol_kernel ran first); a
// large child task's block comes from its hand-over slot after a bounded wait on the task's counter of finished large
// children (tdone), others through the cluster's stack.  Flags as in chol_kernel.
__global__ void __launch_bounds__(kCT, 1)
    chol_tc_kernel(DevPlan P, const int4* items, int nitems, int* queue, int* tdone, double* hand_all, double* ws,
                   int64_t ws_stride, char* scratch, int64_t scratch_stride, int flags, int* status) {
  extern __shared__ uint8_t ct_raw[];
  uint8_t* ring = ct_raw + ((1024u - (smem_u32(ct_raw) & 1023u)) & 1023u);
  PivotSmem& sm = *reinterpret_cast<PivotSmem*>(ring);
  __shared__ uint64_t full[kCStages], empty[kCStages], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  __shared__ int bad, item_s;
  __shared__ __align__(16) int EXB[kNB], es[kNB];  // es: the shifts of a 32-column step
  __shared__ double red[kCT / 32];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int rank = (int)cl_rank(), C = (int)cl_size(), cluster = blockIdx.x / C;
  const int gtid = rank * kCT + tid, gthreads = C * kCT;
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
  st.ring = ring;
  st.bpan = ring + kCStages * kCStage;
  st.full = full;
  st.empty = empty;
  st.accf = accf;
  st.acce = acce;
  st.drain = &drain;
  st.abort = &abort_s;
  st.tmem = tmem_s;
  double* stack = ws + (int64_t)cluster * ws_stride;
  char* SL = scratch + (int64_t)cluster * scratch_stride;
  for (;;) {
    cl_sync();
    if (rank == 0 && tid == 0) {
      int it = atomicAdd(queue, 1);
      if (it < nitems && P.task_nbig[items[it].z] > 0) {
        // the large child tasks were taken before this one and are running: wait for them (bounded)
        const int4 item = items[it];
        int ok = 0;
        for (int i = 0; i < (1 << 26); ++i) {
          if (*(volatile int*)(tdone + item.z) >= P.task_nbig[item.z]) {
            ok = 1;
            break;
          }
          __nanosleep(64);
        }
        __threadfence();
        if (!ok) {
          atomicOr(status, kStatTimeout);
          if (item.w >= 0) atomicAdd(tdone + item.w, 1);  // no cascade of waits above a failure
          it = -1;
        }
      }
      for (int c = 0; c < C; ++c) cl_store(&item_s, c, it);
    }
    if (tid == 0) bad = 0;
    cl_sync();
    const int it = item_s;
    if (it >= nitems) break;
    if (it < 0) continue;
    const int4 item = items[it];
    const int si = item.x, task = item.y;
    const SubInfo S = P.sub[si];
    const double* K = P.Kval + S.Kval;
    double* L = P.L + S.L;
    double* hand = hand_all + S.hbase;
    double mx = 0.0;  // rho = max diag K_i, as in chol_kernel
    for (int i = tid; i < S.n; i += kCT) mx = fmax(mx, K[P.diag_src[S.diag0 + i]]);
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    double rho = red[0];
    for (int k = 1; k < kCT / 32; ++k) rho = fmax(rho, red[k]);
    if (flags & kCholNoReg) rho = 0.0;
    for (int s = 0; s < S.nsn; ++s) {
      const int gs = S.sn0 + s;
      if (!P.sn_big[gs] || P.sn_task[gs] != task) continue;
      const int w = P.sn_w[gs], r = P.sn_r[gs], f = w + r;
      double* Ls = L + P.Lofs[gs];
      // the bottom block is formed where the parent reads it
      double* W = P.sn_hoff[gs] >= 0 ? hand + P.sn_hoff[gs] : stack + P.upd_ofs[gs];
      assemble_cluster(P, S, s, K, L, rho, W, stack, hand, gtid, gthreads);
      if (!((flags & kCholStopRoot) && s == S.nsn - 1)) {
        for (int kB = 0; kB < w; kB += kCBlk) {
          const int kE = min(w, kB + kCBlk);
          for (int kb = kB; kb < kE; kb += kNB) {
            const int ke = min(kE, kb + kNB), nbk = ke - kb, n = f - ke;
            const int npad = (n + kCM - 1) / kCM * kCM, ntm = npad / kCM;
            char *S1 = SL, *S2 = SL + (int64_t)npad * 512;  // the panel's digits before and after the solve
            int* EX1 = reinterpret_cast<int*>(SL + (int64_t)npad * 1024);
            int* EX2 = EX1 + npad;
            // the pivot block (every CTA), and the digits of this CTA's panel rows
            for (int idx = tid; idx < kNB * kNB; idx += kCT) {
              const int i = idx % kNB, j = idx / kNB;
              const double a = (i < nbk && j <= i) ? __ldcg(Ls + (int64_t)(kb + j) * f + kb + i) : 0.0;
              sm.D[i][j] = a;
              if (i == j) es[j] = dig_half_exponent(a);
            }
            __syncthreads();
            pivot_block(sm, nbk, &bad);
            // warps 8-11 start on the panel rows while the others factor the block
            if (warp >= 8)
              for (int tm = rank; tm < ntm; tm += C)
                dig_rows<1>(Shifted<ColMajor, false>{{Ls + (int64_t)kb * f + ke, f}, es}, n, nbk, tm * kCM,
                            tm * kCM + kCM, S1, 1, npad, EX1, warp - 8, 4);
            __syncthreads();
            dig_inverse(sm, es, st.bpan, EXB);
            double lb[3];
            for (int u = 0; u < 3; ++u) {
              const int idx = tid + u * kCT;
              lb[u] = idx < kNB * kNB ? sm.D[idx % kNB][idx / kNB] : 0.0;
            }
            PanelJob pj{S1, EX1, EXB, (int64_t)npad * 64, 0, 1, n, nbk, Ls + (int64_t)kb * f + ke, f};
            dig_product(st, pj, rank, C, ntm);
            if (ke < kE)
              for (int tm = rank; tm < ntm; tm += C)
                dig_rows<1>(ColMajor{Ls + (int64_t)kb * f + ke, f}, n, nbk, tm * kCM, tm * kCM + kCM, S2, 1, npad, EX2,
                            warp, kCT / 32);
            cl_sync();
            if (rank == 0)  // every CTA has read the block
              for (int u = 0; u < 3; ++u) {
                const int idx = tid + u * kCT, i = idx % kNB, j = idx / kNB;
                if (idx < kNB * kNB && i < nbk && j <= i) Ls[(int64_t)(kb + j) * f + kb + i] = lb[u];
              }
            if (ke < kE) {
              const int ntn = (kE - ke + 63) / 64;
              int ntile = 0;
              for (int tm = 0; tm < ntm; ++tm) ntile += min(2 * (tm + 1), ntn);
              UpdateJob uj{S2, EX2, (int64_t)npad * 64, (int64_t)npad * 64, 1, n, npad, ntn, kE - ke, ke, w, r, Ls, W, f};
              dig_product(st, uj, rank, C, ntile);
              cl_sync();
            }
          }
          if (kE < f) {
            const int n = f - kE, K2 = kE - kB, nck = (K2 + 31) / 32;
            const int npad = (n + kCM - 1) / kCM * kCM, ntm = npad / kCM, ntn = (n + 63) / 64;
            int* EX = reinterpret_cast<int*>(SL + (int64_t)npad * 64 * kDig * nck);
            for (int q = (rank * (kCT / 32) + warp) * 8; q < npad; q += C * (kCT / 32) * 8)
              dig_rows<4>(ColMajor{Ls + (int64_t)kB * f + kE, f}, n, K2, q, q + 8, SL, nck, npad, EX, 0, 1);
            cl_sync();
            int ntile = 0;
            for (int tm = 0; tm < ntm; ++tm) ntile += min(2 * (tm + 1), ntn);
            const int64_t dig = (int64_t)nck * npad * 64;
            UpdateJob uj{SL, EX, dig, dig, nck, n, npad, ntn, n, kE, w, r, Ls, W, f};
            dig_product(st, uj, rank, C, ntile);
            cl_sync();
          }
        }
      }
      cl_sync();
    }
    if (tid == 0 && bad) atomicOr(status, kStatNotSPD);
    if (rank == 0 && tid == 0 && item.w >= 0) {
      __threadfence();  // the task's factor panels and hand-over block (ordered by the barrier above) before the count
      atomicAdd(tdone + item.w, 1);
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

// CTAs per cluster for nsub subdomains with large fronts on nsm SMs
int chol_tc_cluster(int nsub, int nsm) {
  int c = 1;
  while (c < 8 && 2 * c * nsub <= nsm) c *= 2;
  return c;  // 8 is the portable limit
}

void launch_chol_tc(const DevPlan& P, const int4* items, int nitems, int* queue, int* tdone, double* hand,
                    double* ws, int64_t ws_stride, void* scratch, int64_t scratch_stride,
                    int clusters, int cluster, int* status, cudaStream_t st, int flags) {
  if (nitems <= 0) return;
  cudaFuncSetAttribute(chol_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCDyn);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(std::min(clusters, nitems) * cluster));
  cfg.blockDim = dim3(kCT);
  cfg.dynamicSmemBytes = kCDyn;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, chol_tc_kernel, P, items, nitems, queue, tdone, hand, ws, ws_stride,
                     (char*)scratch, scratch_stride, flags, status);
}

int64_t chol_tc_scratch(int fmax) {
  const int64_t npad = (fmax + kCM - 1) / kCM * kCM;
  return (npad * (2 * kDig * kCBlk + 8) + 127) / 128 * 128;
}

}  // namespace feti
