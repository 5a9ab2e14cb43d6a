// Tiles of digit products (oz.cuh) on the tensor cores for CTAs of 384 threads, shared by the large-front Cholesky and
// the large-front FP64 forward solve.
//
// The digits are written pre-swizzled (64-byte swizzle, 8-row atoms): [digit][32-deep chunk][row][64 bytes], so any
// 8-row-aligned run of rows of one digit and chunk is a ready operand, loaded by one bulk copy.  Tiles are 128 rows x
// 64 columns: a stage holds the 8 A digits and the digits of two blocks of 32 B columns, each with its own set of
// accumulators (256 TMEM columns), so one set is drained while the other is filled.  Warp 0 issues the MMAs, warp 1
// the copies, warps 4-11 run the epilogue.  The epilogue is integer arithmetic up to one FP64 addition per entry (a
// warp's FP64 instruction takes 64 clocks of its scheduler on this GPU).  Every mbarrier wait is bounded.
#pragma once
#include <cstdint>

#include "oz.cuh"

namespace feti {
namespace {

constexpr int kCT = 384;                                    // threads per CTA
constexpr int kCM = 128, kCH = 32;                          // rows of a tile, columns of one B block
constexpr int kCA = kCM * 64, kCB = kCH * 64;               // bytes of one digit of A / of a B block (one chunk)
constexpr int kCStage = kDig * (kCA + 2 * kCB);             // 96 KB
constexpr int kCStages = 2;

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

struct CtState {
  uint8_t* ring;
  uint8_t* bpan;      // digits of L_bb^{-1}
  uint64_t *full, *empty, *accf, *acce, *drain;
  volatile int* abort;
  uint32_t tmem;
  uint32_t chunks;    // chunks staged so far (stage and phase)
  uint32_t units;     // 32-column units multiplied so far (accumulator set and phase)
};

// Four doubles of a row, 32-byte aligned.  A lane has its own row here, so every instruction of a warp meets 32 lines
// whatever its width: the widest accesses cost the fewest.  (Written and read by the same CTA: plain loads.)
__device__ __forceinline__ void ld4(const double* p, double* v) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st4(double* p, double a, double b, double c, double d) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}

// Eight entries of a row (columns k .. k + 7, zero from K on): of a column-major matrix, and of a row-major one of this
// CTA whose rows are 32-byte aligned and padded to a multiple of 8.
struct ColMajor {
  static constexpr bool kShift = false;
  const double* A;
  int64_t ld;
  __device__ __forceinline__ void get(int i, int k, int K, double (&v)[8]) const {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = k + e < K ? __ldcg(A + (int64_t)(k + e) * ld + i) : 0.0;
  }
};
struct RowMajor {
  static constexpr bool kShift = false;
  const double* A;
  int64_t ld;
  __device__ __forceinline__ void get(int i, int k, int K, double (&v)[8]) const {
    const double* p = A + (int64_t)i * ld + k;
    if (k < K) {
      ld4(p, v);
      ld4(p + 4, v + 4);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = k + e < K ? v[e] : 0.0;
  }
};
// SRC with the shift sh[k] (NEG: -sh[k]) of column k; sh holds whole chunks of 32, 16-byte aligned
template <class SRC, bool NEG>
struct Shifted {
  static constexpr bool kShift = true;
  SRC src;
  const int* sh;
  __device__ __forceinline__ void get(int i, int k, int K, double (&v)[8]) const { src.get(i, k, K, v); }
  __device__ __forceinline__ void shifts(int k, int (&s)[8]) const {
    const int4 a = *reinterpret_cast<const int4*>(sh + k), b = *reinterpret_cast<const int4*>(sh + k + 4);
    s[0] = a.x, s[1] = a.y, s[2] = a.z, s[3] = a.w, s[4] = b.x, s[5] = b.y, s[6] = b.z, s[7] = b.w;
#pragma unroll
    for (int e = 0; e < 8; ++e) s[e] = NEG ? -s[e] : s[e];
  }
};

// Digits of the rows [r0, r1) (multiples of 8) of A (K <= 128 columns; with A's shifts where it has some): row exponents
// EX and the digits in the layout above (npad rows; rows >= n are zero).  Four lanes per row, eight of its columns each.
template <int NCK, class SRC>
__device__ __forceinline__ void dig_rows(const SRC& A, int n, int K, int r0, int r1, char* SL, int nck,
                                         int npad, int* EX, int warp, int nwarps) {
  const int lane = threadIdx.x % 32, q = lane & 3;
  for (int rb = r0 + warp * 8; rb < r1; rb += nwarps * 8) {
    const int i = rb + (lane >> 2);
    double v[NCK][8];
    int mx = SRC::kShift ? kKeyZero : 0;
#pragma unroll
    for (int c = 0; c < NCK; ++c) {
      if (i < n) {
        A.get(i, c * 32 + q * 8, K, v[c]);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[c][e] = 0.0;
      }
      if constexpr (SRC::kShift) {
        int s[8];
        A.shifts(c * 32 + q * 8, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) mx = max(mx, dig_key(v[c][e], s[e]));
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) mx = max(mx, __double2hiint(v[c][e]) & 0x7fffffff);
      }
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const int ex = SRC::kShift ? dig_key_exponent(mx) : dig_exponent((uint32_t)mx);
    if (q == 0) EX[i] = ex;
    const int64_t o = (int64_t)i * 64 + ((q ^ ((i >> 1) & 3)) << 4);
#pragma unroll
    for (int c = 0; c < NCK; ++c) {
      if (c >= nck) break;
      uint64_t w[8];
      if constexpr (SRC::kShift) {
        int s[8];
        A.shifts(c * 32 + q * 8, s);
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = dig_cut(v[c][e], ex + s[e]);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = dig_cut(v[c][e], ex);
      }
#pragma unroll
      for (int p = 0; p < kDig; ++p)
        *reinterpret_cast<uint4*>(SL + ((int64_t)(p * nck + c) * npad) * 64 + o) =
            make_uint4(dig_pair(w[0], w[1], p), dig_pair(w[2], w[3], p), dig_pair(w[4], w[5], p),
                       dig_pair(w[6], w[7], p));
    }
  }
}

// One phase of products: tiles first, first + step, ... < ntile of the job J, which provides
//   kUnits        32-column units per tile (1 or 2)
//   kBSmem        the B digits are in st.bpan (one chunk) instead of being copied
//   nck           32-deep chunks of K
//   tile(t, tm, tn)
//   a(tm, c), b(tn, c)   the operands' first digit of chunk c; digA, digB bytes between digits
//   begin(row)    the row's exponent; load(row, unit column, C[16]) valid columns; ec4(column) four exponents
//   store4(row, column, count, C, product)   up to four columns (column a multiple of 4)
template <class JOB>
__device__ __forceinline__ void dig_product(CtState& st, JOB& job, int first, int step, int ntile) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t ring = smem_u32(st.ring);
  const int mine = first < ntile ? (ntile - first + step - 1) / step : 0;
  constexpr uint32_t nu = JOB::kUnits;
  const int nck = job.nck;
  asm volatile("fence.proxy.async.global;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();  // the ring's generic use is over
  const bool live = !*st.abort;
  if (live && warp == 1 && lane == 0) {
    // ---- copies
    bool ok = true;
    uint32_t cg = st.chunks;
    for (int q = 0; q < mine && ok; ++q) {
      int tm, tn;
      job.tile(first + q * step, tm, tn);
      for (int c = 0; c < nck && ok; ++c, ++cg) {
        const uint32_t s = cg % kCStages;
        if (cg >= kCStages) ok = dig_wait(smem_u32(&st.empty[s]), ((cg / kCStages) - 1) & 1, st.abort);
        if (!ok) break;
        const uint32_t sA = ring + s * kCStage, sB = sA + kDig * kCA, bar = smem_u32(&st.full[s]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"(kDig * (kCA + (JOB::kBSmem ? 0 : (int)nu * kCB)))
                     : "memory");
        const char* a0 = job.a(tm, c);
        const char* b0 = JOB::kBSmem ? nullptr : job.b(tn, c);
#pragma unroll 1
        for (int p = 0; p < kDig; ++p) {
          bulk_copy(sA + p * kCA, a0 + p * job.digA, kCA, bar);
          if (!JOB::kBSmem) {
            bulk_copy(sB + p * kCB, b0 + p * job.digB, kCB, bar);
            if (nu == 2) bulk_copy(sB + (kDig + p) * kCB, b0 + p * job.digB + kCB, kCB, bar);
          }
        }
      }
    }
    if (!ok) {
      // the copies in flight land (bounded) before the block goes on
      for (uint32_t k = cg > kCStages ? cg - kCStages : 0; k < cg; ++k)
        mbar_wait(smem_u32(&st.full[k % kCStages]), (k / kCStages) & 1);
    }
  } else if (live && warp == 0 && lane == 0) {
    // ---- MMAs
    bool ok = true, issued = false;
    uint32_t cg = st.chunks, un = st.units;
    for (int q = 0; q < mine && ok; ++q, un += nu) {
      for (int c = 0; c < nck && ok; ++c, ++cg) {
        const uint32_t s = cg % kCStages;
        ok = dig_wait(smem_u32(&st.full[s]), (cg / kCStages) & 1, st.abort);
        const uint32_t sA = ring + s * kCStage, sB = JOB::kBSmem ? smem_u32(st.bpan) : sA + kDig * kCA;
        for (uint32_t h = 0; h < nu && ok; ++h) {
          const uint32_t u = un + h, set = u & 1;
          if (c == 0 && u >= 2) ok = dig_wait(smem_u32(&st.acce[set]), ((u >> 1) - 1) & 1, st.abort);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int p = 0; p < kDig; ++p)
              mma_f16(st.tmem + set * 256 + p * kCH, sw64_desc(sA + p * kCA + kk * 32),
                      sw64_desc(sB + h * (kDig * kCB) + kk * 32), idesc_m128(1u, (uint32_t)(kCH * (kDig - p))),
                      (c == 0 && kk == 0 && p == 0) ? 0u : 1u);
          issued = true;
          if (c == nck - 1) mma_commit(smem_u32(&st.accf[set]));
        }
        if (ok) mma_commit(smem_u32(&st.empty[s]));
      }
    }
    if (!ok && issued) {  // nothing is issued after this: every MMA is done before TMEM is released
      mma_commit(smem_u32(st.drain));
      mbar_wait(smem_u32(st.drain), 0);
    }
  } else if (live && warp >= 4) {
    // ---- epilogue: TMEM lane quarter warp % 4, 16 columns of the unit
    const int quarter = warp % 4, ch = (warp - 4) / 4;
    uint32_t un = st.units;
    int ok = 1;
    for (int q = 0; q < mine && ok; ++q) {
      int tm, tn;
      job.tile(first + q * step, tm, tn);
      const int ri = tm * kCM + quarter * 32 + lane;  // row of A
      const int ei = job.begin(ri);
      for (uint32_t h = 0; h < nu && ok; ++h, ++un) {
        const uint32_t set = un & 1;
        const int cb = (tn * (int)nu + (int)h) * kCH + ch * 16;  // first column
        // the C entries this thread subtracts from, loaded while the tile is multiplied
        double cv[16];
        const int nc = job.load(ri, cb, cv);
        if (lane == 0) ok = dig_wait(smem_u32(&st.accf[set]), (un >> 1) & 1, st.abort) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t t0 = st.tmem + ((uint32_t)(quarter * 32) << 16) + set * 256 + ch * 16;
#pragma unroll
        for (int e0 = 0; e0 < 16; e0 += 4) {
          uint32_t a[4][kDig];
          const int4 ej4 = e0 < nc ? job.ec4(cb + e0) : make_int4(0, 0, 0, 0);
#pragma unroll
          for (int d = 0; d < kDig; ++d) tmem_ld4(t0 + d * kCH + e0, a[0][d], a[1][d], a[2][d], a[3][d]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (e0 == 12) {  // the set's last columns are in registers: hand it back
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&st.acce[set]);
          }
          double t[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (e0 + e < nc) {
              long long hi = 0, lo = 0;
              dig_sum(a[e], hi, lo);
              const int ej = e == 0 ? ej4.x : e == 1 ? ej4.y : e == 2 ? ej4.z : ej4.w;
              t[e] = dig_value(hi, lo, ei + ej - 68);
              if (ei == kExpBad || ej == kExpBad) t[e] = __longlong_as_double(0x7FF8000000000000LL);
            }
          }
          if (e0 < nc) job.store4(ri, cb + e0, min(4, nc - e0), cv + e0, t);
        }
      }
    }
  }
  __syncthreads();
  if (live) {
    st.chunks += (uint32_t)(mine * nck);
    st.units += (uint32_t)mine * nu;
  }
}

}  // namespace
}  // namespace feti
