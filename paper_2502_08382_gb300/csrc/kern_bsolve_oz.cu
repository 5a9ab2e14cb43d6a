// Backward solve V <- L_u^{-T} V of the large fronts (P.sn_back, the top of the tree) for the adjoint and the TRSM-path
// assembly, on the tensor cores by exact slicing; adj_bsolve_kernel then does the supernodes below them.
//
// One work item is a block of 128 columns of one subdomain's V (n x ld row-major, rows in the factor's numbering; the
// columns are independent), which are the rows of the products, V^T.  A front's own columns go in blocks of 128 from
// the last: the rows below the block, 128 at a time, are cut into digits (gathered through the front's row list) and
//   V^T_b -= V^T_below L_below,b        (K = 128)
// runs against the digits of L^T; inside the block, in steps of 32 from the last, the step is multiplied by the inverse
// of its unit-lower block and the block's earlier columns take its rank-32 update.  dig_lt_kernel cuts L^T once per
// batch.  The tiles are those of oz_engine.cuh.  Row i of V falls with unknown i's stiffness and row i of L_u grows with
// it: the two are cut with opposite shifts of the pivot L_ii's exponent (oz.cuh), kept with the digits.
//
// What bounds it: the latency of a front's steps (cut, multiply, drain) on the narrow fronts; where the line to the
// FP64 kernel lies and why, at kBackFront.  Measured, the backward solve of one adjoint of 8 elasticity subdomains of
// 10^3: 60 ms with every front on the FP64 pipe -> 11.1 + 0.4 (digits) + 1.1 (the fronts below, FP64 pipe).
#include <algorithm>
#include <cuda_bf16.h>

#include "chol_common.cuh"
#include "common.cuh"
#include "kernels.h"
#include "oz_engine.cuh"

namespace feti {
namespace {

constexpr int kYDyn = 1024 + kCStages * kCStage;
constexpr int kTRows = 160;  // rows of the in-block digits: 128 and the overhang of a 64-column tile

// Digit layout of one 128-column block (byte offsets; multiples of 512): inverses, in-block rows, groups of 128 below,
// each with its exponents and the shifts of its inner index.
struct LtBlock {
  int64_t inv, invex, in, inex, piv, grp, end;
  int64_t grpex, grpsz;  // of a group: its 128 exponents (after the digits; then the 128 shifts), its bytes
  int K, nck, nb, ng;    // own columns, chunks, rows below the block, groups of them
  int bp;                // own columns padded to the 64 of a tile
};
__host__ __device__ inline LtBlock lt_block(int w, int r, int kB) {
  LtBlock b;
  b.K = w - kB < 128 ? w - kB : 128;
  b.nck = (b.K + 31) / 32;
  b.nb = w + r - kB - b.K;
  b.ng = (b.nb + 127) / 128;
  b.inv = 0;
  b.invex = 4 * kDig * kCB;
  b.in = b.invex + 512;
  b.inex = b.in + (int64_t)kDig * b.nck * kTRows * 64;
  b.piv = b.inex + 1024;
  b.grp = b.piv + 512;
  b.bp = (b.K + 63) / 64 * 64;
  b.grpex = (int64_t)kDig * 4 * b.bp * 64;
  b.grpsz = b.grpex + 1024;
  b.end = b.grp + b.ng * b.grpsz;
  return b;
}

// row b = column b of the panel, entries k below it; strict: only those below the (unit) diagonal
struct PanelRow {
  static constexpr bool kShift = false;
  const double* A;
  int64_t ld;
  bool strict;
  __device__ __forceinline__ void get(int i, int k, int K, double (&v)[8]) const {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = k + e < K && (!strict || k + e > i) ? A[(int64_t)i * ld + k + e] : 0.0;
  }
};

// items: (subdomain, supernode, first column of the block, byte offset / 512 of the block); base: per item's subdomain
__global__ void __launch_bounds__(256) dig_lt_kernel(DevPlan P, const int4* items, char* LT) {
  __shared__ double D[4][kNB][kNB + 1];
  __shared__ __align__(16) int es[128];
  const int4 it = items[blockIdx.x];
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const SubInfo& S = P.sub[it.x];
  const int gs = S.sn0 + it.y, w = P.sn_w[gs], r = P.sn_r[gs], f = w + r, kB = it.z;
  const double* Ls = P.L + S.L + P.Lofs[gs];
  const LtBlock b = lt_block(w, r, kB);
  char* out = LT + (int64_t)it.w * 512;
  const int kE = kB + b.K;
  const double* d2 = P.dinv + S.dof;  // 1 / L_ii^2
  auto shift = [&](int col) { return -(dig_pivot_shift(d2[col]) >> 1); };  // about the exponent of L_ii
  if (tid < 128) {
    es[tid] = tid < b.K ? shift(P.sn_c0[gs] + kB + tid) : 0;
    reinterpret_cast<int*>(out + b.piv)[tid] = es[tid];
  }
  __syncthreads();
  if (warp < 4) {
    // the inverse of the unit-lower diagonal block `warp`: lane = column k, m[i] = Linv[i][k]; row k of the operand
    const int k0 = kB + 32 * warp, nb = min(32, kE - k0);
    double(*d)[kNB + 1] = D[warp];
    for (int k = 0; k < kNB; ++k)
      d[lane][k] = (lane < nb && k < lane && k < nb) ? Ls[(int64_t)(k0 + k) * f + k0 + lane] : 0.0;
    __syncwarp();
    double m[kNB];
#pragma unroll
    for (int i = 0; i < kNB; ++i) {
      double a = i == lane ? 1.0 : 0.0;
#pragma unroll
      for (int k = 0; k < i; ++k) a = fma(-d[i][k], m[k], a);
      m[i] = a;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kNB; ++i) d[lane][i] = (i < nb && lane < nb) ? m[i] : 0.0;
    __syncwarp();
    for (int i0 = 0; i0 < kNB; i0 += 8) {
      const int i = i0 + (lane >> 2), q = lane & 3;
      const int* sh = es + 32 * warp + q * 8;
      int mx = kKeyZero;
#pragma unroll
      for (int e = 0; e < 8; ++e) mx = max(mx, dig_key(d[i][q * 8 + e], sh[e]));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const int ex = dig_key_exponent(mx);
      if (q == 0) reinterpret_cast<int*>(out + b.invex)[32 * warp + i] = ex;
      uint64_t c[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) c[e] = dig_cut(d[i][q * 8 + e], ex + sh[e]);
#pragma unroll
      for (int p = 0; p < kDig; ++p)
        *reinterpret_cast<uint4*>(out + b.inv + (warp * kDig + p) * kCB + i * 64 + ((q ^ ((i >> 1) & 3)) << 4)) =
            make_uint4(dig_pair(c[0], c[1], p), dig_pair(c[2], c[3], p), dig_pair(c[4], c[5], p),
                       dig_pair(c[6], c[7], p));
    }
  } else {
    dig_rows<4>(Shifted<PanelRow, false>{{Ls + (int64_t)kB * f + kB, f, true}, es}, b.K, b.K, 0, 128, out + b.in, b.nck,
                kTRows, reinterpret_cast<int*>(out + b.inex), warp - 4, 4);
  }
  for (int g = 0; g < b.ng; ++g) {
    char* o = out + b.grp + g * b.grpsz;
    __syncthreads();
    if (tid < 128) {
      const int i = kE + 128 * g + tid;  // row of the front
      es[tid] = 128 * g + tid < b.nb ? shift(i < w ? P.sn_c0[gs] + i : P.rows[P.sn_rows[gs] + i - w]) : 0;
      reinterpret_cast<int*>(o + b.grpex)[128 + tid] = es[tid];
    }
    __syncthreads();
    dig_rows<4>(Shifted<PanelRow, false>{{Ls + (int64_t)kB * f + kE + 128 * g, f, false}, es}, b.K,
                min(128, b.nb - 128 * g), 0, b.bp, o, 4, b.bp, reinterpret_cast<int*>(o + b.grpex), warp, 8);
  }
}

// row c = column c of V (from the item's first), entry k = front row i0 + k (own rows from c0, then the row list)
struct GatherRow {
  static constexpr bool kShift = false;
  const double* V;
  int64_t ld;
  const int* srow;
  int c0, w, i0;
  __device__ __forceinline__ void get(int i, int k, int K, double (&v)[8]) const {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int q = i0 + k + e;
      v[e] = k + e < K ? __ldcg(V + (int64_t)(q < w ? c0 + q : srow[q - w]) * ld + i) : 0.0;
    }
  }
};

// C[row c, column b] (= V[(v0 + b) ld + c]) -= A B^T, or = A B^T with SET; n rows, ncol columns
template <bool SET>
struct BackJob {
  static constexpr int kUnits = SET ? 1 : 2;
  static constexpr bool kBSmem = false;
  const char *SA, *SB;
  const int *EX, *EXB;
  int64_t digA, digB;
  int nck, n, npadB, ntn, ncol;
  double* C;
  int64_t ld;
  __device__ __forceinline__ void tile(int t, int& tm, int& tn) const {
    tm = t / ntn;
    tn = t - tm * ntn;
  }
  __device__ __forceinline__ const char* a(int, int c) const { return SA + (int64_t)c * kCM * 64; }
  __device__ __forceinline__ const char* b(int tn, int c) const {
    return SB + ((int64_t)c * npadB + (int64_t)tn * 64) * 64;
  }
  __device__ __forceinline__ int begin(int ri) const { return ri < n ? __ldcg(EX + ri) : 0; }
  __device__ __forceinline__ int load(int ri, int cb, double (&cv)[16]) const {
    const int nc = ri < n ? min(16, ncol - cb) : 0;
    if constexpr (!SET) {
#pragma unroll
      for (int e = 0; e < 16; ++e) cv[e] = e < nc ? __ldcg(C + (int64_t)(cb + e) * ld + ri) : 0.0;
    }
    return nc;
  }
  __device__ __forceinline__ int4 ec4(int c) const { return __ldg(reinterpret_cast<const int4*>(EXB + c)); }
  __device__ __forceinline__ void store4(int ri, int c, int n4, const double* cv, const double* t) const {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < n4) C[(int64_t)(c + e) * ld + ri] = SET ? t[e] : cv[e] - t[e];
  }
};

// items: (batch entry, 128-column block)
__global__ void __launch_bounds__(kCT, 1)
    bsolve_oz_kernel(DevPlan P, const AdjBatch* B, const int2* items, int nitems, int* queue, const char* LT, double* work,
                     char* scratch, int64_t scratch_stride, int* status) {
  extern __shared__ uint8_t bo_raw[];
  __shared__ uint64_t full[kCStages], empty[kCStages], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int abort_s;
  const int tid = threadIdx.x, warp = tid / 32;
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
  st.ring = bo_raw + ((1024u - (smem_u32(bo_raw) & 1023u)) & 1023u);
  st.full = full;
  st.empty = empty;
  st.accf = accf;
  st.acce = acce;
  st.drain = &drain;
  st.abort = &abort_s;
  st.tmem = tmem_s;
  char* SL = scratch + (int64_t)blockIdx.x * scratch_stride;
  int* EX = reinterpret_cast<int*>(SL + (int64_t)128 * 2048);
  for (;;) {
    const int it = pop_item(queue);
    if (it >= nitems) break;
    const AdjBatch& E = B[items[it].x];
    const SubInfo& S = P.sub[E.sub];
    const int64_t ld = (E.zonly ? 1 : 2) * (int64_t)E.m_pad;
    const int n = min(128, E.m_pad - 128 * items[it].y);  // columns of this item
    double* V = work + E.v_ofs + 128 * items[it].y;
    for (int s = S.nsn - 1; s >= 0; --s) {
      const int gs = S.sn0 + s;
      if (!P.sn_back[gs]) continue;
      const int c0 = P.sn_c0[gs], w = P.sn_w[gs], r = P.sn_r[gs];
      const int* srow = P.rows + P.sn_rows[gs];
      // the blocks' digits lie first block first
      const char* lt0 = LT + E.lt + P.lt_ofs[gs] * 512;
      for (int kB = (w - 1) / 128 * 128; kB >= 0; kB -= 128) {
        const char* lt = lt0;
        for (int k = 0; k < kB; k += 128) lt += lt_block(w, r, k).end;
        const LtBlock b = lt_block(w, r, kB);
        const int kE = kB + b.K, ntn = (b.K + 63) / 64;
        for (int g = 0; g < b.ng; ++g) {
          const int K = min(128, b.nb - 128 * g);
          const char* o = lt + b.grp + g * b.grpsz;
          const int* ex = reinterpret_cast<const int*>(o + b.grpex);
          dig_rows<4>(Shifted<GatherRow, true>{{V, ld, srow, c0, w, kE + 128 * g}, ex + 128}, n, K, 0, 128, SL, 4, 128,
                      EX, warp, kCT / 32);
          BackJob<false> bj{SL, o, EX, ex, (int64_t)4 * 128 * 64,
                            (int64_t)4 * b.bp * 64, (K + 31) / 32, n, b.bp, ntn, b.K, V + (int64_t)(c0 + kB) * ld, ld};
          dig_product(st, bj, 0, 1, ntn);
        }
        for (int sb = b.nck - 1; sb >= 0; --sb) {
          const int k0 = kB + 32 * sb, nbk = min(32, kE - k0);
          const Shifted<GatherRow, true> own{{V, ld, srow, c0, w, k0},
                                             reinterpret_cast<const int*>(lt + b.piv) + 32 * sb};
          dig_rows<1>(own, n, nbk, 0, 128, SL, 1, 128, EX, warp, kCT / 32);
          BackJob<true> sj{SL, lt + b.inv + sb * kDig * kCB, EX, reinterpret_cast<const int*>(lt + b.invex) + 32 * sb,
                           (int64_t)128 * 64, kCB, 1, n, 0, 1, nbk, V + (int64_t)(c0 + k0) * ld, ld};
          dig_product(st, sj, 0, 1, 1);
          if (sb > 0) {
            dig_rows<1>(own, n, nbk, 0, 128, SL, 1, 128, EX, warp, kCT / 32);
            const int nt = (32 * sb + 63) / 64;
            BackJob<false> uj{SL, lt + b.in + (int64_t)sb * kTRows * 64, EX, reinterpret_cast<const int*>(lt + b.inex),
                              (int64_t)128 * 64, (int64_t)b.nck * kTRows * 64, 1, n, kTRows, nt, 32 * sb,
                              V + (int64_t)(c0 + kB) * ld, ld};
            dig_product(st, uj, 0, 1, nt);
          }
        }
      }
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

int64_t bsolve_oz_block_bytes(int w, int r, int kB) { return lt_block(w, r, kB).end; }

int64_t bsolve_oz_scratch() { return 128 * (2048 + 4); }

void launch_dig_lt(const DevPlan& P, const int4* items, int nitems, void* LT, cudaStream_t st) {
  if (nitems > 0) dig_lt_kernel<<<nitems, 256, 0, st>>>(P, items, (char*)LT);
}

void launch_bsolve_oz(const DevPlan& P, const AdjBatch* B, const int2* items, int nitems, int* queue, const void* LT,
                      double* work, void* scratch, int grid, int* status, cudaStream_t st) {
  if (nitems <= 0) return;
  cudaFuncSetAttribute(bsolve_oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kYDyn);
  bsolve_oz_kernel<<<std::min(grid, nitems), kCT, kYDyn, st>>>(P, B, items, nitems, queue, (const char*)LT, work,
                                                              (char*)scratch, bsolve_oz_scratch(), status);
}

}  // namespace feti
