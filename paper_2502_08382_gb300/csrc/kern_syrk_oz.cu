// FP64 SYRK F_i = X_i^T X_i on the tensor cores by exact slicing (oz.cuh), into the FP64 F tiles.
//
// The FP64 pipe of this GPU does two FMAs per SM and clock; the 36 digit products of one FP64 product take
// 36 / 4096 of a clock on the bf16 tensor cores.  Three kernels:
//   colexp_kernel   exponent of every column of X_i (one warp per column)
//   dig_x_kernel    the digits of X: per supernode block, piece (8 rows) and column 128 contiguous bytes, the
//                   eight digits one after another (16 bytes each), in place of the 64 bytes of FP64
//   syrk_oz_kernel  one CTA per SM, tiles of 128 x 64 of F_i.
//
// syrk_oz_kernel.  K runs over pieces of 8 rows of the supernodes that reach both column blocks, four pieces (32
// rows) to a chunk, whichever supernodes they belong to (so narrow supernodes are padded to 8 rows, not to 32).
// Per chunk the A digits (8 x 128 rows x 64 B) and the digits of two blocks of 32 B columns (8 x 32 x 64 B each)
// are staged by 16-byte cp.async (zero outside the supernode's columns) in the 64-byte swizzle: 96 KB, two stages.
// Each B block has its own set of eight accumulators (32 TMEM columns each, 512 in all).  After every 128 rows the
// epilogue warps add a set's accumulators into 64-bit integers while the tensor cores work on the other set.
// Warps 0-3 load, warp 4 issues the MMAs, warps 8-15 drain; registers are split 56 / 56 / 200 / 200 (the launch's
// 512 x 128).
//
// What bounds it: the staging, 96 KB from L2 for every 2304 clocks of MMA (39 bytes per SM and clock).  Measured
// (GB300, events; FP64-pipe kernel before -> the three kernels together): 64 uneven 3D heat subdomains (136 GFLOP)
// 160.7 -> 11.1 ms, 27 elasticity subdomains of 12^3 (101 GFLOP) 90.6 -> 6.2 ms, 256 2D heat subdomains of 64^2
// (1.9 GFLOP) 6.0 -> 0.93 ms, 16 of 16^2 0.31 -> 0.05 ms: it is the faster one at every size, so the FP64-pipe
// kernel is kept only for contexts whose digits do not fit the device memory.  The error against exact sums is
// about a hundredth of FP64's (host emulation on X of all three kinds of problem: 4e-18 to 1e-18 relative against
// 1e-16 to 5e-16 for FP64 sums).
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "oz.cuh"

namespace feti {
namespace {

constexpr int kOM = 128, kON = 64, kOH = 32;
constexpr int kOStages = 2;
constexpr int kOA = kOM * 64, kOB = kOH * 64;                   // bytes of one digit of A / of one B block
constexpr int kOStageBytes = kDig * (kOA + 2 * kOB);            // 96 KB
constexpr int kOPieces = 1024;                                  // piece table (window)
constexpr int kOBatch = 128;                                    // contributions scanned at a time
constexpr int kODyn = 1024 + kOStages * kOStageBytes + kOPieces * 16;
constexpr int kOThreads = 512;

struct Piece {
  long long base;  // byte offset of (column 0, this piece) in the digit array (column j at + 128 j)
  int jb, je;      // columns the block holds
};

__global__ void __launch_bounds__(256) colexp_kernel(DevPlan P, const double* X, int sub0, int* EX) {
  const int lane = threadIdx.x % 32;
  const SubInfo& S = P.sub[sub0 + blockIdx.y];
  for (int j = (blockIdx.x * blockDim.x + threadIdx.x) / 32; j < S.m; j += gridDim.x * blockDim.x / 32) {
    uint32_t mx = 0;
    for (int a0 = 0; a0 < S.nact; a0 += 32) {
      int bs = 0, gs = 0;
      bool in = false;
      if (a0 + lane < S.nact) {
        const int s = P.act[S.act0 + a0 + lane];
        bs = S.bsn0 + s;
        gs = S.sn0 + s;
        in = j >= P.jb[bs] && j < P.je[bs];
      }
      uint32_t todo = __ballot_sync(0xffffffffu, in);
      const int w_ = in ? P.sn_w[gs] : 0;
      const long long o_ = in ? P.Xofs[bs] + (long long)(j - P.jb[bs]) * ((w_ + 7) & ~7) : 0;
      while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const int w = __shfl_sync(0xffffffffu, w_, l);
        const double* x = X + S.X + __shfl_sync(0xffffffffu, o_, l);
        for (int k = lane; k < w; k += 32) mx = max(mx, (uint32_t)__double2hiint(x[k]) & 0x7fffffffu);
      }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) EX[S.qcol + j] = dig_exponent(mx);
  }
}

// items: (subdomain, supernode, first unit, units); unit = (piece, column) of the block, column fastest
__global__ void __launch_bounds__(256) dig_x_kernel(DevPlan P, const double* X, const int4* items, const int* EX,
                                                    int64_t x0, uint4* XD) {
  const int4 it = items[blockIdx.x];
  const SubInfo& S = P.sub[it.x];
  const int gs = S.sn0 + it.y, bs = S.bsn0 + it.y;
  const int wp = (P.sn_w[gs] + 7) & ~7, jb = P.jb[bs], J = P.je[bs] - jb;
  const double* Xs = X + S.X + P.Xofs[bs];
  uint4* out = XD + (S.X - x0 + P.Xofs[bs]);  // 16 bytes per value
  const int* ex = EX + S.qcol + jb;
  for (int u = it.z + threadIdx.x; u < it.z + it.w; u += 256) {
    const int q = u / J, j = u - q * J;
    const double2* src = reinterpret_cast<const double2*>(Xs + (int64_t)j * wp + 8 * q);
    const int e = ex[j];
    uint64_t c[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double2 v = src[k];
      c[2 * k] = dig_cut(v.x, e);
      c[2 * k + 1] = dig_cut(v.y, e);
    }
#pragma unroll
    for (int p = 0; p < kDig; ++p)
      out[(int64_t)u * 8 + p] = make_uint4(dig_pair(c[0], c[1], p), dig_pair(c[2], c[3], p), dig_pair(c[4], c[5], p),
                                           dig_pair(c[6], c[7], p));
  }
}

// SYRK: items (subdomain, 128-row block | 64-column block << 16, chunks, 128 x 128 tile of the contribution list), XD the
// digits of X, EX the column exponents, out F.
// DENSE: out = A B^T for the products `ents`; items (product, 128-row block | 64-column block << 16, chunks, 0), XD the
// digits of A and B per piece of 8 columns (rows contiguous), EX their row exponents.
template <bool DENSE>
__global__ void __launch_bounds__(kOThreads, 1)
    syrk_oz_kernel(DevPlan P, const DenseEnt* ents, const int4* items, int nitems, const char* XD, int64_t x0,
                   const int* EX, double* F, int* status) {
  extern __shared__ uint8_t oz_dyn[];
  __shared__ uint64_t full[kOStages], empty[kOStages], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_s;
  __shared__ volatile int s_abort;
  __shared__ int p_stop, wsum[4];
  uint8_t* smem = oz_dyn + ((1024u - (smem_u32(oz_dyn) & 1023u)) & 1023u);
  Piece* pieces = reinterpret_cast<Piece*>(smem + kOStages * kOStageBytes);
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int k = 0; k < kOStages; ++k) {
      mbar_init(&full[k], 128);
      mbar_init(&empty[k], 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&accf[h], 1);
      mbar_init(&acce[h], 8);
    }
    mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_s;
  if (warp < 4) {
    // ------------------------------------------------ loaders
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    uint32_t cg = 0;  // chunks staged so far
    bool dead = false;
    const int prow = lane & 7, pdig = lane >> 3;  // this lane's row of an 8-row atom, and digits pdig, pdig + 4
    // one chunk: warp w stages piece w, 24 atoms (16 of A, 4 + 4 of B), digits pdig and pdig + 4
    auto stage = [&](const char* srcA, int a0, int a1, const char* srcB, int b0, int b1, int ra, int rb) {
      const uint32_t st = cg % kOStages;
      if (!dead && cg >= kOStages && !dig_wait(smem_u32(&empty[st]), ((cg / kOStages) - 1) & 1, &s_abort)) dead = true;
      if (dead) return;
      const uint32_t sA = smem_u32(smem + st * kOStageBytes), sB = sA + kDig * kOA;
      const uint32_t so = prow * 64 + ((warp ^ ((prow >> 1) & 3)) << 4);
#pragma unroll 4
      for (int at = 0; at < kOM / 8; ++at) {
        const int j = ra + at * 8 + prow;
        const bool ok = j >= a0 && j < a1;
        const char* src = ok ? srcA + (long long)j * 128 + pdig * 16 : XD;
        const uint32_t dst = sA + pdig * kOA + at * 512 + so;
        cp_async16(dst, src, ok);
        cp_async16(dst + 4 * kOA, ok ? src + 64 : XD, ok);
      }
#pragma unroll 4
      for (int at = 0; at < kON / 8; ++at) {
        const int j = rb + at * 8 + prow;
        const bool ok = j >= b0 && j < b1;
        const char* src = ok ? srcB + (long long)j * 128 + pdig * 16 : XD;
        const uint32_t dst = sB + (at >> 2) * (kDig * kOB) + pdig * kOB + (at & 3) * 512 + so;
        cp_async16(dst, src, ok);
        cp_async16(dst + 4 * kOB, ok ? src + 64 : XD, ok);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&full[st]);
    };
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
      const int4 item = items[it];
      const int ra = (item.y & 0xffff) * kOM, rb = (item.y >> 16) * kON;
      if constexpr (DENSE) {
        const DenseEnt& e = ents[item.x];
        for (int ch = 0; ch < item.z; ++ch, ++cg) {
          const int q = 4 * ch + warp;
          const bool in = q < e.pieces;
          stage(XD + e.a + (long long)q * e.rows * 128, 0, in ? e.rows : 0, XD + e.b + (long long)q * e.cols * 128, 0,
                in ? e.cols : 0, ra, rb);
        }
        continue;
      }
      const SubInfo& S = P.sub[item.x];
      const int* tl = P.t2_off + S.t20;
      const int cbeg = tl[item.w], cend = tl[item.w + 1];
      for (int c0 = cbeg; c0 < cend; c0 += kOBatch) {
        // this thread's contribution, and the exclusive prefix sum of the pieces over the batch
        int np = 0, jb = 0, je = 0;
        long long base = 0;
        if (c0 + tid < cend) {
          const int s = P.t2_sn[c0 + tid];
          const int bs = S.bsn0 + s;
          np = (P.sn_w[S.sn0 + s] + 7) / 8;
          jb = P.jb[bs];
          je = P.je[bs];
          base = (S.X - x0 + P.Xofs[bs]) * 16 - (long long)jb * 128;
        }
        int inc = np;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += t;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (lane == 31) wsum[warp] = inc;
        if (tid == 0) p_stop = s_abort;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (p_stop) dead = true;  // the same value for all loaders
        int total = 0, pre = inc - np;
        for (int k = 0; k < 4; ++k) {
          if (k < warp) pre += wsum[k];
          total += wsum[k];
        }
        for (int w0 = 0; w0 < total; w0 += kOPieces) {
          const int nw = min(kOPieces, total - w0), nw4 = (nw + 3) & ~3;
          for (int q = max(0, w0 - pre); q < np && pre + q < w0 + nw; ++q)
            pieces[pre + q - w0] = Piece{base + (long long)q * (je - jb) * 128, jb, je};
          if (tid < nw4 - nw) pieces[nw + tid] = Piece{0, 0, 0};
          asm volatile("bar.sync 1, 128;" ::: "memory");
          for (int ch = 0; ch < nw4 / 4; ++ch, ++cg) {
            const Piece pc = pieces[ch * 4 + warp];
            stage(XD + pc.base, pc.jb, pc.je, XD + pc.base, pc.jb, pc.je, ra, rb);
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");
        }
      }
    }
  } else if (warp < 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 4 && lane == 0) {
      // ---------------------------------------------- MMA issue
      uint32_t cg = 0, ng = 0;  // chunks, and groups of at most four chunks (one exact accumulation), so far
      bool ok = true, issued = false;
      for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const int nch = items[it].z;
        for (int i = 0; i < nch && ok; ++i, ++cg) {
          const uint32_t st = cg % kOStages;
          const bool first = i % 4 == 0, last = i % 4 == 3 || i == nch - 1;
          ok = dig_wait(smem_u32(&full[st]), (cg / kOStages) & 1, &s_abort);
          const uint32_t sA = smem_u32(smem + st * kOStageBytes), sB = sA + kDig * kOA;
          for (int h = 0; h < 2 && ok; ++h) {
            if (first && ng >= 1) ok = dig_wait(smem_u32(&acce[h]), (ng - 1) & 1, &s_abort);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
#pragma unroll
              for (int p = 0; p < kDig; ++p)
                mma_f16(tmem + h * 256 + p * kOH, sw64_desc(sA + p * kOA + kk * 32),
                        sw64_desc(sB + h * (kDig * kOB) + kk * 32), idesc_m128(1u, (uint32_t)(kOH * (kDig - p))),
                        (first && kk == 0 && p == 0) ? 0u : 1u);
            issued = true;
            if (last) mma_commit(smem_u32(&accf[h]));
          }
          if (ok) mma_commit(smem_u32(&empty[st]));
          if (last) ++ng;
        }
      }
      if (issued) {  // every MMA is done before TMEM is released, also after a timeout
        mma_commit(smem_u32(&drain));
        if (!mbar_wait(smem_u32(&drain), 0)) s_abort = 1;
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------ epilogue: lane quarter warp % 4, columns 16 ch of each block
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    const int quarter = warp % 4, ch = (warp - 8) / 4;
    uint32_t ng = 0;
    int ok = 1;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
      const int4 item = items[it];
      const int ngr = (item.z + 3) / 4;
      long long hi[2][16], lo[2][16];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 16; ++e) hi[h][e] = lo[h][e] = 0;
      for (int g = 0; g < ngr && ok; ++g, ++ng) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (lane == 0) ok = dig_wait(smem_u32(&accf[h]), ng & 1, &s_abort) ? 1 : 0;
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t t0 = tmem + ((uint32_t)(quarter * 32) << 16) + h * 256 + ch * 16;
#pragma unroll
          for (int e0 = 0; e0 < 16; e0 += 4) {
            uint32_t a[4][kDig];
#pragma unroll
            for (int d = 0; d < kDig; ++d) tmem_ld4(t0 + d * kOH + e0, a[0][d], a[1][d], a[2][d], a[3][d]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int e = 0; e < 4; ++e) dig_sum(a[e], hi[h][e0 + e], lo[h][e0 + e]);
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[h]);
        }
      }
      if (!ok) break;
      if constexpr (DENSE) {
        const DenseEnt& e = ents[item.x];
        const int row = (item.y & 0xffff) * kOM + quarter * 32 + lane, c0 = (item.y >> 16) * kON;
        if (row < e.rows) {
          const int ei = EX[e.exa + row];
          double* out = F + e.out + (int64_t)row * e.ld + c0;
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const int c = h * kOH + ch * 16 + u;
              if (c0 + c < e.cols) {
                const int ej = EX[e.exb + c0 + c];
                const double t = fma((double)hi[h][u], 4294967296.0, (double)lo[h][u]);
                out[c] = ei == kExpBad || ej == kExpBad
                             ? __longlong_as_double(0x7FF8000000000000LL)
                             : t * dig_pow2(min(ei, 1000) - 34) * dig_pow2(min(ej, 1000) - 34);
              }
            }
        }
        continue;
      }
      const SubInfo& S = P.sub[item.x];
      const int row = (item.y & 0xffff) * kOM + quarter * 32 + lane, bj = item.y >> 16;
      const int bi = row / kT, r = row % kT;
      if (bi < S.nb && bj <= bi && r < tile_rows(S.nb, S.vr, bi)) {
        const int* ex = EX + S.qcol;
        const int ei = ex[row];
        double* Ft = F + S.F + tile_offset<8>(S.nb, S.vr, bi, bj);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            const int c = h * kOH + ch * 16 + e;
            double v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int ej = bj * kT + c + u < S.m ? ex[bj * kT + c + u] : 0;
              const double t = fma((double)hi[h][e + u], 4294967296.0, (double)lo[h][e + u]);
              v[u] = t * dig_pow2(min(ei, 1000) - 34) * dig_pow2(min(ej, 1000) - 34);
              if (ei == kExpBad || ej == kExpBad) v[u] = __longlong_as_double(0x7FF8000000000000LL);
            }
            if (bj < bi) {
              *reinterpret_cast<double2*>(Ft + tile_pos(r, c)) = make_double2(v[0], v[1]);
            } else if (c / 2 <= r / 2) {
              *reinterpret_cast<double2*>(Ft + diag_pos<8>(r, c)) = make_double2(v[0], c + 1 <= r ? v[1] : 0.0);
            }
          }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_abort && tid == 0) atomicOr(status, kStatTimeout);
  if (warp == 4) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// Row exponents and digits of the dense products' operands: A (rows x K, row-major, ld) and B^T (K x cols, row-major:
// B's row c is its column c).  blockIdx.y = product.
//
// Shifts of the inner index a (oz.cuh), A's column a 2^-s_a against B's row a 2^s_a: column a of Z falls with the
// stiffness of its multiplier's unknown as sqrt(F_aa) does, W is the caller's, so s_a takes half the difference of the
// exponents of sqrt(F_aa) and of W's largest entry in row a.  (Not of Z's own largest entry: that would depend on how
// many rows go together.)  One warp per a.
__global__ void __launch_bounds__(256) dense_shift_kernel(const DenseEnt* ents, const int* spos, const double* src, int* EX) {
  const DenseEnt e = ents[blockIdx.y];
  const int lane = threadIdx.x % 32;
  for (int a = (blockIdx.x * 256 + threadIdx.x) / 32; a < e.K; a += gridDim.x * 8) {
    const double* b = src + e.src_b + (int64_t)a * e.ldb;
    uint32_t mx = 0;
    for (int j = lane; j < e.cols; j += 32) mx = max(mx, (uint32_t)__double2hiint(b[j]) & 0x7fffffffu);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) {
      const double f = fabs(src[e.z + (int64_t)spos[e.col0 + a] * e.ld + a]);
      EX[e.exs + a] = ((dig_pivot_shift(f) >> 1) - dig_pivot_shift(__hiloint2double((int)mx, 0))) >> 1;
    }
  }
}
__global__ void __launch_bounds__(256) dense_exp_kernel(const DenseEnt* ents, const double* src, int* EX) {
  const DenseEnt e = ents[blockIdx.y];
  const int lane = threadIdx.x % 32;
  for (int i = (blockIdx.x * 256 + threadIdx.x) / 32; i < e.rows; i += gridDim.x * 8) {
    const double* a = src + e.src_a + (int64_t)i * e.ld;
    int mx = kKeyZero;
    for (int k = lane; k < e.K; k += 32) mx = max(mx, dig_key(a[k], EX[e.exs + k]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) EX[e.exa + i] = dig_key_exponent(mx);
  }
  for (int c = blockIdx.x * 256 + threadIdx.x; c < e.cols; c += gridDim.x * 256) {
    const double* b = src + e.src_b + c;
    int mx = kKeyZero;
#pragma unroll 8
    for (int k = 0; k < e.K; ++k) mx = max(mx, dig_key(b[(int64_t)k * e.ldb], -EX[e.exs + k]));
    EX[e.exb + c] = dig_key_exponent(mx);
  }
}

__device__ __forceinline__ void store_digits(uint4* out, const uint64_t (&c)[8]) {
#pragma unroll
  for (int p = 0; p < kDig; ++p)
    out[p] = make_uint4(dig_pair(c[0], c[1], p), dig_pair(c[2], c[3], p), dig_pair(c[4], c[5], p),
                        dig_pair(c[6], c[7], p));
}

__global__ void __launch_bounds__(256) dense_cut_kernel(const DenseEnt* ents, const double* src, const int* EX, char* XD) {
  const DenseEnt e = ents[blockIdx.y];
  const int64_t na = (int64_t)e.rows * e.pieces, nb = (int64_t)e.cols * e.pieces;
  for (int64_t u = blockIdx.x * 256 + threadIdx.x; u < na + nb; u += gridDim.x * 256) {
    uint64_t c[8];
    if (u < na) {  // piece fastest: a row's pieces are contiguous
      const int i = (int)(u / e.pieces), q = (int)(u - (int64_t)i * e.pieces), ex = EX[e.exa + i];
      const double* a = src + e.src_a + (int64_t)i * e.ld + 8 * q;
#pragma unroll
      for (int k = 0; k < 8; ++k) c[k] = 8 * q + k < e.K ? dig_cut(a[k], ex + EX[e.exs + 8 * q + k]) : 0;
      store_digits(reinterpret_cast<uint4*>(XD + e.a + ((int64_t)q * e.rows + i) * 128), c);
    } else {  // column fastest
      const int64_t v = u - na;
      const int q = (int)(v / e.cols), j = (int)(v - (int64_t)q * e.cols), ex = EX[e.exb + j];
      const double* b = src + e.src_b + (int64_t)8 * q * e.ldb + j;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        c[k] = 8 * q + k < e.K ? dig_cut(b[(int64_t)k * e.ldb], ex - EX[e.exs + 8 * q + k]) : 0;
      store_digits(reinterpret_cast<uint4*>(XD + e.b + ((int64_t)q * e.cols + j) * 128), c);
    }
  }
}

}  // namespace

void launch_syrk_oz(const DevPlan& P, const double* X, const OzBatch& b, const int4* ditems, const int4* items,
                    void* XD, int* EX, double* F, int nsm, int* status, cudaStream_t st) {
  cudaFuncSetAttribute(syrk_oz_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kODyn);
  if (b.nitems <= 0) return;
  for (int s0 = 0; s0 < b.nsub; s0 += 32768) {
    dim3 g((unsigned)std::max(1, std::min(64, (b.m_max + 7) / 8)), (unsigned)std::min(32768, b.nsub - s0));
    colexp_kernel<<<g, 256, 0, st>>>(P, X, b.sub0 + s0, EX);
  }
  if (b.nditems > 0) dig_x_kernel<<<b.nditems, 256, 0, st>>>(P, X, ditems + b.ditem0, EX, b.x0, (uint4*)XD);
  syrk_oz_kernel<false><<<std::min(b.nitems, nsm), kOThreads, kODyn, st>>>(P, nullptr, items + b.item0, b.nitems,
                                                                          (const char*)XD, b.x0, EX, F, status);
}

void launch_dense_oz(const DenseEnt* ents, int nent, const int4* items, int nitems, const int* spos, const double* src,
                     void* XD, int* EX, double* out, int nsm, int* status, cudaStream_t st) {
  if (nent <= 0 || nitems <= 0) return;
  const dim3 g((unsigned)std::max(1, nsm * 16 / nent), (unsigned)nent);
  dense_shift_kernel<<<g, 256, 0, st>>>(ents, spos, src, EX);
  dense_exp_kernel<<<g, 256, 0, st>>>(ents, src, EX);
  dense_cut_kernel<<<g, 256, 0, st>>>(ents, src, EX, (char*)XD);
  cudaFuncSetAttribute(syrk_oz_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kODyn);
  DevPlan P{};
  syrk_oz_kernel<true><<<std::min(nitems, nsm), kOThreads, kODyn, st>>>(P, ents, items, nitems, (const char*)XD, 0, EX,
                                                                        out, status);
}

int syrk_oz_chunks(const int* np, int n) {
  int ch = 0;
  for (int c0 = 0; c0 < n; c0 += kOBatch) {
    int total = 0;
    for (int c = c0; c < std::min(n, c0 + kOBatch); ++c) total += np[c];
    for (int w0 = 0; w0 < total; w0 += kOPieces) ch += (std::min(kOPieces, total - w0) + 3) / 4;
  }
  return ch;
}

}  // namespace feti
