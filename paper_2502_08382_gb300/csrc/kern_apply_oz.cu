// The F-streaming part of the explicit apply for FP64 tiles (see kern_apply.cu) by exact slicing on mma.sync.
//
// With FMAs an FP64 tile costs two FP64 FMAs per entry (row and column partial) and some additions, and the FP64 pipe of
// this GPU does two a clock and SM: it bounds the stream at 2.4 TB/s (those kernels reach 1.2 to 1.75).  Here every entry is cut into eight
// balanced base-256 digits (oz.cuh; 62 bits below the largest entry of its 16 x 64 strip), the digits go as f16
// integers through mma.sync.m16n8k16 against the digits of p (N = 8: the eight digits of one vector), and the exact
// integer sums are put together in 64-bit integers; about forty FP64 instructions per tile are left.  The operands
// come out of registers and are used once, so tcgen05 (operands through shared memory, N at least 8 of one vector)
// has nothing to gain: the cutting, about 25 integer instructions an entry, sets the pace (ncu: integer ALU 50%,
// HMMA 12%, FP64 7%, twelve warps per SM).  Measured: 0.57 GB of FP64 tiles (125 uneven 3D heat subdomains) 361 us with
// the register-batch kernel -> 272 us (262 before the scales below); 48 small tiles (16 subdomains of 16^2), where one
// warp per tile is a long chain of FP64 instructions, 25 us with the fastest of the others -> 9.5 (launch included).  The other variants stay for the autotuner: they win
// where few tiles leave the stream latency-bound and for FP32 tiles.
//
// One CTA of four warps per tile at a time, its tiles copied two ahead into shared memory (one bulk copy each); warp v
// takes rows 16 v .. 16 v + 15 in A-fragment order.
//   rows:    acc_p = F_p P_col over the four 16-column blocks, P_col's digit q in column q; the digits (p, q) are
//            combined at the end (all 64 pairs);
//   columns: the fragments transposed by movmatrix, against the digits of P_row shifted by p columns, so that one
//            accumulator per 16 columns collects digit sums d = p + q <= 7 (at most 8 16 2^14 = 2^21, exact); the four
//            strips' partials are added in FP64 in a fixed order.
// Strips or vectors that hold an infinity or NaN take plain FP64 FMAs (slow_strip), so those propagate as before.
//
// Scales.  F_ij is at most sqrt(F_ii F_jj), which may differ by many decades between the rows of a strip (a stiff and a
// soft material), so the tile is cut as F_ij 2^-(s_i + s_j) with s_i half the exponent of F_ii (tile_scales_kernel,
// once per assembly) and p as p_j 2^s_j: 62 bits below the largest scaled entry are then far below what FP64 can know of
// F_ij itself, u sqrt(F_ii F_jj).  The scales only enter the exponents of the cut and of the results.
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "oz.cuh"

namespace feti {
namespace {

constexpr int kDT = 128;
constexpr int kTileBytes = kT * kT * 8;
constexpr int kDDyn = 2 * kTileBytes + 128;  // two tile buffers

// Exponent e of a strip or vector from its largest key (biased exponent less the scales, which are within kMaxScale
// each): 0 if all entries are zero, kExpBad for infinities, NaN, and entries too small or too large for the cut below.
constexpr int kMaxScale = 400;
__device__ __forceinline__ int scaled_exponent(int key, int least, int bad, bool zero) {
  return key >= least && key < bad ? key - 1022 : key < least && zero ? 0 : kExpBad;
}
constexpr int kBadF = 2047 - 2 * kMaxScale, kLeastF = 923, kLeastP = 522;  // least: so that e + s_i + s_j and e - s_j are at least -950 (zeros shift out)

// s_j of every sorted column from the diagonal of the FP64 tiles (0 for padding and for entries not positive)
__global__ void __launch_bounds__(256) tile_scales_kernel(DevPlan P, int nsub, const double* F, int* scale) {
  for (int si = blockIdx.y; si < nsub; si += gridDim.y) {
    const SubInfo& S = P.sub[si];
    for (int j = blockIdx.x * 256 + threadIdx.x; j < S.m_pad; j += gridDim.x * 256) {
      int s = 0;
      if (j < S.m) {
        const int b = j / kT, r = j % kT;
        s = dig_pivot_shift(F[S.F + tile_offset<8>(S.nb, S.vr, b, b) + diag_pos<8>(r, r)]) >> 1;
      }
      scale[S.qcol + j] = max(-kMaxScale, min(kMaxScale, s));
    }
  }
}

// The digits of x (|x| < 2^e, e >= -950) plus 128 as bytes, digit 0 in the top byte: x cut (not rounded) to 62
// fractional bits below e.  Zeros and subnormals shift out.  The shift up and the sign are multiplications: the
// integer ALU, not the FMA pipe, is what this kernel runs out of.
__device__ __forceinline__ uint64_t dig_bytes(double x, int e) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int n = min(1023 + e - (int)((hi >> 20) & 0x7FF), 63);
  const uint64_t M = (uint64_t)lo * 1024u + ((uint64_t)(((hi & 0xFFFFF) | 0x100000) * 1024u) << 32);  // [2^62, 2^63)
  const int64_t sg = (int64_t)((int32_t)hi >> 31 | 1);
  return (uint64_t)((int64_t)(M >> n) * sg) + 0x8080808080808080ULL;
}

// two bytes (digit + 128) at positions b, b + 4 of y's selection as an f16 pair of digits
__device__ __forceinline__ uint32_t bytes_f16(uint32_t y, uint32_t sel) {
  const uint32_t r = __byte_perm(y, 0x64646464u, sel);  // 1024 + byte
  uint32_t o;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o) : "r"(r), "r"(0xE480E480u));  // - 1152
  return o;
}

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t trans8(uint32_t a) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(a));
  return r;
}

// a strip in plain FP64 (lane = columns 2 l, 2 l + 1): row partials into rp[16], column partials into cs[64]
__device__ void slow_strip(const TileDesc& d, const double* F, const double* pg, int warp, int lane, double* rowpart,
                           double* cs) {
  const bool diag = (d.flags & kTileDiag) != 0;
  double c0 = 0.0, c1 = 0.0;
  const double px = pg[d.pcol + 2 * lane], py = pg[d.pcol + 2 * lane + 1];
  for (int r = 16 * warp; r < min(16 * warp + 16, d.rows); ++r) {
    const bool ok = !diag || 2 * lane <= r;
    const double* src = F + d.f_ofs + (diag ? diag_row_off<8>(r) : (int64_t)r * kT) + 2 * lane;
    const double x = ok ? src[0] : 0.0, y = ok ? src[1] : 0.0;
    const double pr = pg[d.prow + r];
    double s = ok ? fma(y, py, x * px) : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) rowpart[(int64_t)d.slot * kT + r] = s;
    if (ok && !(diag && 2 * lane >= r)) c0 = fma(x, pr, c0);
    if (ok && !(diag && 2 * lane + 1 >= r)) c1 = fma(y, pr, c1);
  }
  cs[2 * lane] = c0;
  cs[2 * lane + 1] = c1;
}

__global__ void __launch_bounds__(kDT, 3)
    apply_dig_kernel(const TileDesc* __restrict__ desc, int ntiles, const double* __restrict__ F,
                     const double* __restrict__ pg, const int* __restrict__ scale, double* rowpart, double* colpart,
                     const int* active, int* status) {
  if (active && *active == 0) return;  // the iteration this launch belongs to has stopped
  extern __shared__ uint8_t ad_raw[];
  // bytes 8 .. 15: the digits of p (column block, then row block) plus 128; bytes 0 .. 7: 128 (a zero digit)
  __shared__ __align__(16) uint8_t pd[2 * kT][16];
  __shared__ double cs[4][kT], dgs[kT];
  __shared__ int mx_s[4];
  __shared__ __align__(16) int sx[2 * kT];  // scales of the column block, then of the row block
  __shared__ uint64_t full[2];
  uint8_t* buf = ad_raw + ((128u - (smem_u32(ad_raw) & 127u)) & 127u);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, g = lane / 4, t = lane % 4;
  const int r0 = 16 * warp + g;
  if (blockIdx.x >= ntiles) return;
  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // the stored bytes of a tile are contiguous: one bulk copy, two tiles ahead
  auto fetch = [&](int tl, int b) {
    const TileDesc d = desc[tl];
    const uint32_t bytes = (uint32_t)(((d.flags & kTileDiag) ? diag_row_off<8>(d.rows) : (int64_t)d.rows * kT) * 8);
    const uint32_t bar = smem_u32(&full[b]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(buf + b * kTileBytes)),
                 "l"(F + d.f_ofs), "r"(bytes), "r"(bar)
                 : "memory");
  };
  auto pval = [&](const TileDesc& d) {
    return tid < kT ? pg[d.pcol + tid] : (tid - kT < d.rows ? pg[d.prow + tid - kT] : 0.0);
  };
  if (tid == 0) {
    fetch(blockIdx.x, 0);
    if (blockIdx.x + gridDim.x < ntiles) fetch(blockIdx.x + gridDim.x, 1);
  }
  auto sval = [&](const TileDesc& d) {
    return tid < kT ? scale[d.pcol + tid] : (tid - kT < d.rows ? scale[d.prow + tid - kT] : 0);
  };
  TileDesc dn = desc[blockIdx.x];
  double pn = pval(dn);
  int sn = sval(dn);
  int it = 0;
  bool ok_all = true;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
    const TileDesc d = dn;
    const double pv = pn;
    const int sv = sn;
    if (tile + (int)gridDim.x < ntiles) {
      dn = desc[tile + gridDim.x];
      pn = pval(dn);
      sn = sval(dn);
    }
    const bool diag = (d.flags & kTileDiag) != 0;
    // (subnormal entries, which the cut below would drop, go the slow way)
    const uint32_t ph = (uint32_t)__double2hiint(pv) & 0x7fffffffu;
    const bool tiny = ph < 0x00100000u && (ph | (uint32_t)__double2loint(pv)) != 0;
    const int pm = __reduce_max_sync(0xffffffffu, tiny ? kKeyBad : dig_key(pv, -sv));
    if (lane == 0) mx_s[warp] = pm;
    sx[tid] = sv;
    const double* Ft = reinterpret_cast<const double*>(buf + (it & 1) * kTileBytes);
    // every lane waits, so that each one sees the copied bytes
    ok_all = ok_all && mbar_wait(smem_u32(&full[it & 1]), (it >> 1) & 1);
    // f[kb][j]: row g (+ 8 for odd j), columns 16 kb + 2 t, + 1 (+ 8 for j >= 2) of the strip
    double2 f[4][4];
    if (!diag && d.rows == kT) {
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          f[kb][j] = *reinterpret_cast<const double2*>(Ft + (r0 + 8 * (j & 1)) * kT + 16 * kb + 2 * t + 8 * (j >> 1));
    } else {
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = r0 + 8 * (j & 1), c = 16 * kb + 2 * t + 8 * (j >> 1);
          const bool ok = r < d.rows && (!diag || c <= r);
          const int64_t off = diag ? diag_row_off<8>(r) : (int64_t)r * kT;
          double2 v = ok ? *reinterpret_cast<const double2*>(Ft + off + c) : make_double2(0.0, 0.0);
          if (diag && c == r) v.x = 0.0;  // the diagonal counts once: left out here, added to its row at the end
          if (diag && c + 1 == r) v.y = 0.0;
          f[kb][j] = v;
        }
    }
    if (diag && tid < kT && tid < d.rows) dgs[tid] = Ft[diag_row_off<8>(tid) + tid];
    __syncthreads();
    const int si[2] = {sx[kT + r0], sx[kT + r0 + 8]};
    // the largest scaled entry: high words less the scales, 1024 exponents up so that they stay positive
    uint32_t fm = 0;
#pragma unroll
    for (int kb = 0; kb < 4; ++kb)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int2 sj = *reinterpret_cast<const int2*>(&sx[16 * kb + 2 * t + 8 * (j >> 1)]);
        const uint32_t c = (uint32_t)(1024 - si[j & 1]) << 20;
        fm = max(fm, max(((uint32_t)__double2hiint(f[kb][j].x) & 0x7fffffffu) + c - ((uint32_t)sj.x << 20),
                         ((uint32_t)__double2hiint(f[kb][j].y) & 0x7fffffffu) + c - ((uint32_t)sj.y << 20)));
      }
    const int fkey = (int)(__reduce_max_sync(0xffffffffu, fm) >> 20) - 1024;
    bool fzero = false;
    if (fkey < kLeastF) {  // all zero, or tiny against the diagonal
      uint32_t z = 0;
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          z |= (((uint32_t)__double2hiint(f[kb][j].x) | (uint32_t)__double2hiint(f[kb][j].y)) & 0x7fffffffu) |
               (uint32_t)__double2loint(f[kb][j].x) | (uint32_t)__double2loint(f[kb][j].y);
      fzero = __reduce_or_sync(0xffffffffu, z) == 0;
    }
    const int ef = scaled_exponent(fkey, kLeastF, kBadF, fzero);
    const int kpc = max(mx_s[0], mx_s[1]), kpr = max(mx_s[2], mx_s[3]);
    const int epc = scaled_exponent(kpc, kLeastP, kKeyBad, kpc == kKeyZero);
    const int epr = scaled_exponent(kpr, kLeastP, kKeyBad, kpr == kKeyZero);
    {
      const int e = tid < kT ? epc : epr;
      const uint64_t w = e == kExpBad ? 0 : dig_bytes(pv, e - sv);
      const uint32_t hi = (uint32_t)(w >> 32), lo = (uint32_t)w;
      *reinterpret_cast<uint4*>(pd[tid]) = make_uint4(0x80808080u, 0x80808080u, __byte_perm(hi, 0, 0x0123),
                                                      __byte_perm(lo, 0, 0x0123));
    }
    __syncthreads();
    if (ef == kExpBad || epc == kExpBad || epr == kExpBad) {
      slow_strip(d, F, pg, warp, lane, rowpart, cs[warp]);
    } else {
      // digits of p: column block (digit g of entries 2 t, + 1, + 8, + 9 of each 16), row strip shifted by p digits
      uint32_t bc[4][2], br[8][2];
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = 16 * kb + 2 * t + 8 * h;
          bc[kb][h] = bytes_f16((uint32_t)pd[k][8 + g] | (uint32_t)pd[k + 1][8 + g] << 8, 0x4140);
        }
#pragma unroll
      for (int p = 0; p < kDig; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int k = kT + 16 * warp + 2 * t + 8 * h;
          br[p][h] = bytes_f16((uint32_t)pd[k][8 + g - p] | (uint32_t)pd[k + 1][8 + g - p] << 8, 0x4140);
        }
      float acc[kDig][4] = {};
#pragma unroll
      for (int kb = 0; kb < 4; ++kb) {
        uint64_t wx[4], wy[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int2 sj = *reinterpret_cast<const int2*>(&sx[16 * kb + 2 * t + 8 * (j >> 1)]);
          wx[j] = dig_bytes(f[kb][j].x, ef + si[j & 1] + sj.x);
          wy[j] = dig_bytes(f[kb][j].y, ef + si[j & 1] + sj.y);
        }
        float ca[4] = {};
#pragma unroll
        for (int p2 = 0; p2 < kDig; p2 += 2) {
          uint32_t y[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {  // bytes: digit p2 of x and y, digit p2 + 1 of x and y
            const uint32_t x4 = (uint32_t)(p2 < 4 ? wx[j] >> 32 : wx[j]), y4 = (uint32_t)(p2 < 4 ? wy[j] >> 32 : wy[j]);
            y[j] = __byte_perm(x4, y4, (p2 & 2) ? 0x4051 : 0x6273);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t a[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = bytes_f16(y[j], h ? 0x4342 : 0x4140);
            const int p = p2 + h;
            mma_16816(acc[p], a[0], a[1], a[2], a[3], bc[kb][0], bc[kb][1]);
            mma_16816(ca, trans8(a[0]), trans8(a[2]), trans8(a[1]), trans8(a[3]), br[p][0], br[p][1]);
          }
        }
        // column 16 kb + g: digit sums 2 t, 2 t + 1 in ca[0], ca[1]; column + 8: ca[2], ca[3]
        const int v0 = __float2int_rn(ca[0]) * 256 + __float2int_rn(ca[1]);
        const int v1 = __float2int_rn(ca[2]) * 256 + __float2int_rn(ca[3]);
        // lanes t = 0, 2 put column g together, t = 1, 3 column g + 8
        const int mine = (t & 1) ? v1 : v0, give = (t & 1) ? v0 : v1;
        const int got = __shfl_xor_sync(0xffffffffu, give, 1);
        const long long pr = (t & 1) ? (long long)got * 65536 + mine : (long long)mine * 65536 + got;
        const long long ot = __shfl_xor_sync(0xffffffffu, pr, 2);
        const double yv = dig_value((t & 2) ? ot : pr, (t & 2) ? pr : ot,
                                    ef + epr - 68 + sx[16 * kb + g + 8 * (t & 1)]);
        if (t < 2) cs[warp][16 * kb + g + 8 * (t & 1)] = yv;
      }
      // rows g (acc[p][0], [1]) and g + 8 (acc[p][2], [3]): digit columns q = 2 t and 2 t + 1
      double rs[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int u[9];
#pragma unroll
        for (int j = 0; j < 9; ++j)
          u[j] = (j < 8 ? __float2int_rn(acc[j][2 * h]) : 0) + (j > 0 ? __float2int_rn(acc[j - 1][2 * h + 1]) : 0);
        const long long hi = ((long long)(u[0] * 256 + u[1]) * 65536 + (u[2] * 256 + u[3])) * 256 + u[4];
        const long long lo = (long long)(u[5] * 256 + u[6]) * 65536 + (u[7] * 256 + u[8]);
        rs[h] = dig_value(hi, lo, ef + epc - 76 - 16 * t + si[h]);
      }
      // lanes t = 0, 2 add up row g, t = 1, 3 row g + 8
      double s = (t & 1) ? rs[1] : rs[0];
      s += __shfl_xor_sync(0xffffffffu, (t & 1) ? rs[0] : rs[1], 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      const int r = r0 + 8 * (t & 1);
      if (t < 2 && r < d.rows) {
        if (diag) s = fma(dgs[r], pg[d.prow + r], s);
        rowpart[(int64_t)d.slot * kT + r] = s;
      }
    }
    __syncthreads();
    if (tid == 0 && tile + 2 * (int64_t)gridDim.x < ntiles) fetch(tile + 2 * gridDim.x, it & 1);
    if (tid < kT) colpart[(int64_t)d.slot * kT + tid] = (cs[0][tid] + cs[1][tid]) + (cs[2][tid] + cs[3][tid]);
  }
  // a copy that did not land in time: reported (its tile's partials are of whatever the buffer held)
  if (!ok_all && status) atomicOr(status, kStatTimeout);
}

}  // namespace

void launch_apply_dig(int grid, cudaStream_t st, const TileDesc* desc, int ntiles, const double* F, const double* pg,
                      const int* scale, double* rowpart, double* colpart, const int* active, int* status) {
  cudaFuncSetAttribute(apply_dig_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDDyn);
  apply_dig_kernel<<<grid, kDT, kDDyn, st>>>(desc, ntiles, F, pg, scale, rowpart, colpart, active, status);
}

void launch_tile_scales(const DevPlan& P, int nsub, int m_max, const double* F, int* scale, cudaStream_t st) {
  const dim3 g((unsigned)std::max(1, std::min((m_max + kT + 255) / 256, 64)), (unsigned)std::max(1, std::min(nsub, 32768)));
  tile_scales_kernel<<<g, 256, 0, st>>>(P, nsub, F, scale);
}

int apply_dig_occupancy() {
  int nb = 0;
  cudaFuncSetAttribute(apply_dig_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDDyn);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, apply_dig_kernel, kDT, kDDyn);
  return nb;
}

}  // namespace feti
