// C ABI of the FETI dual-operator library: create / assemble / apply / query.
// The solver entry points (implicit apply, PCPG, recovery, adjoint) live in
// api_solve.cpp.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstring>
#include <map>
#include <numeric>
#include <queue>
#include <stdexcept>
#include <thread>
#include <unordered_map>

#include "context.h"
#include "precond.h"
#include "kernels.h"

using namespace feti;

namespace feti {
void coarse_setup_entry(feti_ctx* c);

feti_status set_error(feti_ctx* c, feti_status s, const std::string& msg) {
  if (c) {
    if (c->sticky == FETI_OK && s != FETI_ERR_NOT_CONVERGED) c->sticky = s;
    c->err = msg;
  }
  return s;
}

void* dalloc(feti_ctx* c, size_t bytes) {
  if (bytes == 0) bytes = 16;
  bytes = (bytes + 255) & ~size_t(255);
  void *p = nullptr, *base = nullptr;
  if (c->opt.dev_alloc) {
    // the kernels' widest accesses are of 32 bytes, their bulk copies of 16: a caller's allocator that aligns to less
    // than 256 bytes is asked for as much more
    constexpr size_t kAlign = 256;
    base = p = c->opt.dev_alloc(bytes, c->opt.alloc_ctx);
    if (p && (uintptr_t)p % kAlign != 0) {
      if (c->opt.dev_free) c->opt.dev_free(p, c->opt.alloc_ctx);
      bytes += kAlign;
      base = c->opt.dev_alloc(bytes, c->opt.alloc_ctx);
      p = base ? (void*)(((uintptr_t)base + kAlign - 1) / kAlign * kAlign) : nullptr;
    }
  } else {
    if (cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr;
    base = p;
  }
  if (!p) throw std::bad_alloc();
  c->bufs.push_back({p, bytes, base});
  c->device_bytes += bytes;
  return p;
}

void dfree(feti_ctx* c, void* p) {
  if (!p) return;
  for (size_t k = 0; k < c->bufs.size(); ++k)
    if (c->bufs[k].p == p) {
      if (c->opt.dev_free) c->opt.dev_free(c->bufs[k].base, c->opt.alloc_ctx);
      else if (!c->opt.dev_alloc) cudaFree(p);
      c->device_bytes -= c->bufs[k].bytes;
      c->bufs.erase(c->bufs.begin() + (long)k);
      return;
    }
}

}  // namespace feti

namespace {

struct CudaError : std::runtime_error {
  using std::runtime_error::runtime_error;
};
struct ArgError : std::runtime_error {
  using std::runtime_error::runtime_error;
};

#define CK(x)                                                                                   \
  do {                                                                                          \
    cudaError_t e_ = (x);                                                                       \
    if (e_ != cudaSuccess) throw CudaError(std::string(#x) + ": " + cudaGetErrorString(e_)); \
  } while (0)

template <typename T>
T* upload(feti_ctx* c, const std::vector<T>& v) {
  T* p = (T*)dalloc(c, v.size() * sizeof(T));
  if (!v.empty()) CK(cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, c->st));
  return p;
}

feti_status guard(feti_ctx* c) {
  if (!c) return FETI_ERR_ARG;
  if (c->sticky != FETI_OK) return FETI_ERR_STATE;
  return FETI_OK;
}

void copy_sub(const feti_subdomain& s, SubHost& h, int idx) {
  auto need = [&](bool ok, const char* what) {
    if (!ok) throw ArgError("subdomain " + std::to_string(idx) + ": " + what);
  };
  need(s.n > 0 && s.m >= 0 && s.d >= 0, "sizes must be n > 0, m >= 0, d >= 0");
  need(s.K_rowptr && s.K_col && s.K_val, "K arrays missing");
  need(s.m == 0 || (s.B_rowptr && s.B_col && s.B_val && s.B_lambda), "B arrays missing");
  need(s.nfix == s.d, "nfix must equal d (one fixing DOF per kernel vector)");
  need(s.d == 0 || (s.R && s.fix_dofs), "R / fix_dofs missing");
  need(s.f != nullptr, "f missing");
  h.n = s.n;
  h.m = s.m;
  h.d = s.d;
  h.nfix = s.nfix;
  h.rowptr.assign(s.K_rowptr, s.K_rowptr + s.n + 1);
  need(h.rowptr[0] == 0 && h.rowptr[s.n] == s.nnz, "K_rowptr must start at 0 and end at nnz");
  for (int i = 0; i < s.n; ++i) need(h.rowptr[i + 1] >= h.rowptr[i], "K_rowptr must be non-decreasing");
  h.col.assign(s.K_col, s.K_col + s.nnz);
  h.val.assign(s.K_val, s.K_val + s.nnz);
  for (int i = 0; i < s.n; ++i)
    for (int64_t k = h.rowptr[i]; k < h.rowptr[i + 1]; ++k) {
      need(h.col[k] >= 0 && h.col[k] < s.n, "K column index out of range");
      need(k == h.rowptr[i] || h.col[k] > h.col[k - 1], "K columns must be sorted and unique per row");
    }
  h.bdof.resize(s.m);
  h.bsign.resize(s.m);
  h.blam.assign(s.B_lambda, s.B_lambda + s.m);
  for (int r = 0; r < s.m; ++r) {
    need(s.B_rowptr[r + 1] - s.B_rowptr[r] == 1, "each B row must hold exactly one entry");
    int64_t k = s.B_rowptr[r];
    need(s.B_col[k] >= 0 && s.B_col[k] < s.n, "B column out of range");
    need(std::fabs(s.B_val[k]) == 1.0, "B entries must be +1 or -1");
    h.bdof[r] = s.B_col[k];
    h.bsign[r] = s.B_val[k];
    need(r == 0 || h.blam[r] > h.blam[r - 1], "B_lambda must be strictly increasing");
  }
  h.R.assign(s.R ? s.R : nullptr, s.R ? s.R + (size_t)s.n * s.d : nullptr);
  h.f.assign(s.f, s.f + s.n);
  h.fix.assign(s.fix_dofs ? s.fix_dofs : nullptr, s.fix_dofs ? s.fix_dofs + s.nfix : nullptr);
  for (int k = 0; k < s.nfix; ++k) need(h.fix[k] >= 0 && h.fix[k] < s.n, "fix DOF out of range");
  if (s.coords) h.coords.assign(s.coords, s.coords + (size_t)s.n * 3);
  h.nelem = s.nelem;
  h.edofs = s.edofs;
  if (s.nelem > 0) {
    need(s.elem_dofs && s.edofs > 0 && (s.dKe || (s.dKe_ref && s.dKe_scale)), "element data incomplete");
    need(s.edofs <= 32, "elements with more than 32 DOFs are not supported");
    const size_t ee = (size_t)s.edofs * s.edofs;
    h.elem_dofs.assign(s.elem_dofs, s.elem_dofs + (size_t)s.nelem * s.edofs);
    if (s.dKe) {
      // one derivative matrix per element
      h.dKe.assign(s.dKe, s.dKe + (size_t)s.nelem * ee);
      h.dKe_scale.assign(s.nelem, 1.0);
      h.dk_stride = (int64_t)ee;
    } else {
      // compact form: a shared reference matrix times a per-element scale
      h.dKe.assign(s.dKe_ref, s.dKe_ref + ee);
      h.dKe_scale.assign(s.dKe_scale, s.dKe_scale + s.nelem);
      h.dk_stride = 0;
    }
    for (auto v : h.elem_dofs) need(v >= 0 && v < s.n, "element DOF out of range");
  }
}

template <typename F>
void parallel_for(int n, F fn) {
  int nt = (int)std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
  nt = std::min(nt, n);
  if (nt <= 1) {
    for (int i = 0; i < n; ++i) fn(i);
    return;
  }
  std::vector<std::thread> th;
  std::vector<std::string> errs(nt);
  std::atomic<int> next{0};
  for (int t = 0; t < nt; ++t)
    th.emplace_back([&, t] {
      try {
        for (int i = next++; i < n; i = next++) fn(i);
      } catch (std::exception& e) {
        errs[t] = e.what();
      }
    });
  for (auto& x : th) x.join();
  for (auto& e : errs)
    if (!e.empty()) throw ArgError(e);
}

// FP64 SYRK on the tensor cores: batches of consecutive subdomains whose digits of X (16 bytes per value) fit
// `budget` bytes (one subdomain at least), the tiles of each batch in groups of subdomains whose digits stay in L2
// (most expensive tile first within a group), and the pieces of X to cut.
void plan_syrk_oz(feti_ctx* c, size_t budget) {
  constexpr double kGroupBytes = 64e6;  // of digits, about half of L2
  constexpr int kUnits = 2048;          // (piece, column) units per CTA of the cutting kernel
  const int ns = c->nsub;
  auto xsize = [&](int i) { return (size_t)c->bps[c->subs[i].bp].Xsize; };
  // chunks of every 128 x 128 tile of a plan (shared by the subdomains of that plan)
  std::vector<std::vector<int>> chunks(c->bps.size());
  for (size_t b = 0; b < c->bps.size(); ++b) {
    auto& B = c->bps[b];
    auto& P = c->pats[c->bp_pat[b]];
    const int nt = B.nb2 * (B.nb2 + 1) / 2;
    std::vector<int> np;
    for (int t = 0; t < nt; ++t) {
      np.clear();
      for (int k = B.t2_off[t]; k < B.t2_off[t + 1]; ++k) np.push_back((P.sn_w[B.t2_sn[k]] + 7) / 8);
      chunks[b].push_back(syrk_oz_chunks(np.data(), (int)np.size()));
    }
  }
  std::vector<int4> items, ditems;
  c->oz_batches.clear();
  size_t most = 0;
  for (int i = 0; i < ns;) {
    OzBatch o{};
    o.sub0 = i;
    o.x0 = c->info[i].X;
    o.item0 = (int)items.size();
    o.ditem0 = (int)ditems.size();
    size_t bytes = 0;
    while (i < ns && (o.nsub == 0 || bytes + 16 * xsize(i) <= budget)) {
      // one group of subdomains
      std::vector<int4> grp;
      double gb = 0;
      while (i < ns && gb < kGroupBytes && (o.nsub == 0 || bytes + 16 * xsize(i) <= budget)) {
        auto& B = c->bps[c->subs[i].bp];
        auto& P = c->pats[c->subs[i].pat];
        for (int bi = 0; bi < B.nb2; ++bi)
          for (int bj = 0; bj <= std::min(2 * bi + 1, B.nb - 1); ++bj) {
            const int t = bi * (bi + 1) / 2 + bj / 2;
            grp.push_back(make_int4(i, bi | bj << 16, chunks[c->subs[i].bp][t], t));
          }
        for (int s : B.act) {
          const int units = (P.sn_w[s] + 7) / 8 * (B.je[s] - B.jb[s]);
          for (int u = 0; u < units; u += kUnits) ditems.push_back(make_int4(i, s, u, std::min(kUnits, units - u)));
        }
        o.m_max = std::max(o.m_max, c->subs[i].m);
        bytes += 16 * xsize(i);
        gb += 16.0 * xsize(i);
        ++o.nsub;
        ++i;
      }
      std::stable_sort(grp.begin(), grp.end(), [](const int4& a, const int4& b) { return a.z > b.z; });
      items.insert(items.end(), grp.begin(), grp.end());
    }
    o.nitems = (int)items.size() - o.item0;
    o.nditems = (int)ditems.size() - o.ditem0;
    c->oz_batches.push_back(o);
    most = std::max(most, bytes);
  }
  // a recorded assembly holds the old lists
  if (c->asm_exec) CK(cudaGraphExecDestroy(c->asm_exec));
  c->asm_exec = nullptr;
  dfree(c, c->d_oz_items);
  dfree(c, c->d_oz_ditems);
  c->d_oz_items = c->d_oz_ditems = nullptr;
  c->d_oz_items = upload(c, items);
  c->d_oz_ditems = upload(c, ditems);
  CK(cudaStreamSynchronize(c->st));  // the host arrays go out of scope
  c->xd_bytes = most;
}

// The digit buffer: as many subdomains at a time as a fifth of the free memory holds (16 GB at most), one at a time if
// the allocator refuses that; false when not even one subdomain fits (the FP64-pipe kernel takes over).  The memory comes
// first and the plan after it, so a refusal leaves the plan and the recorded assembly as they are; it is not asked for
// again before that much more memory is free (recompute_X: asked for at every assembly, as X is).
bool reserve_syrk_oz(feti_ctx* c) {
  if (c->d_XD) return true;
  size_t free_b = 0, total_b = 0;
  CK(cudaMemGetInfo(&free_b, &total_b));
  size_t want = 0, least = 0;
  for (int i = 0; i < c->nsub; ++i) {
    const size_t x = 16 * (size_t)c->bps[c->subs[i].bp].Xsize;
    want += x;
    least = std::max(least, x);
  }
  if (!c->opt.recompute_X && c->xd_refused > 0 && free_b < c->xd_refused + least) return false;
  auto take = [&](size_t bytes) {
    try {
      c->d_XD = dalloc(c, bytes);
    } catch (std::bad_alloc&) {
      c->d_XD = nullptr;
    }
    return c->d_XD != nullptr;
  };
  try {
    if (!c->d_oz_ex) c->d_oz_ex = (int*)dalloc(c, (size_t)std::max<int64_t>(c->ncols, 1) * sizeof(int));
    // the plan at hand first (its buffer was released by recompute_X)
    if (!c->oz_batches.empty() && take(c->xd_bytes)) return true;
    const size_t budget = std::min(want, std::min<size_t>((size_t)16 << 30, free_b / 5));
    for (size_t b : {budget, (size_t)0})
      if (take(std::max(b, least))) {
        plan_syrk_oz(c, b);
        return true;
      }
  } catch (std::bad_alloc&) {  // of the small lists
    dfree(c, c->d_XD);
    c->d_XD = nullptr;
    c->oz_batches.clear();
  }
  c->xd_refused = std::max<size_t>(free_b, 1);
  return false;
}

// Work lists of the FP64 forward solve of the large fronts on the tensor cores, in batches of consecutive subdomains
// whose digits of L fit `budget` bytes (one subdomain at least), and the CTAs' workspaces.
void plan_trsm_oz(feti_ctx* c, size_t budget) {
  c->tx_planned = false;
  c->tx_batches.clear();
  auto ld_end = [&](int i) { return i + 1 < c->nsub ? (size_t)c->info[i + 1].ld : c->ld_bytes; };
  for (int i = 0; i < c->nsub;) {
    feti_ctx::TxBatch b;
    b.sub0 = i;
    b.ld0 = c->info[i].ld;
    do ++i;
    while (i < c->nsub && ld_end(i) - (size_t)b.ld0 <= budget);
    b.sub1 = i;
    c->tx_batches.push_back(b);
  }
  std::vector<int4> di;
  int64_t n256 = 0;
  for (int i = 0; i < c->nsub; ++i) {
    auto& P = c->pats[c->subs[i].pat];
    auto& B = c->bps[c->subs[i].bp];
    int64_t ofs = 0;
    for (int s = 0; s < P.nsn; ++s) {
      if (!P.sn_big[s]) continue;
      for (int kB = 0; kB < P.sn_w[s]; kB += 128) {
        if (B.je[s] > B.jb[s]) di.push_back(make_int4(i, s, kB, (int)(ofs / 512)));
        ofs += trsm_oz_block_bytes(P.sn_w[s], P.sn_r[s], kB);
      }
    }
    if (P.has_big) n256 += (c->subs[i].m + 255) / 256;
  }
  c->tx_cw = n256 >= 2 * (int64_t)c->nsm ? 256 : 128;
  std::vector<int2> it;
  size_t most = 0, dk = 0;
  for (auto& b : c->tx_batches) {
    std::vector<int> order;
    for (int i = b.sub0; i < b.sub1; ++i)
      if (c->pats[c->subs[i].pat].has_big && c->subs[i].m > 0) order.push_back(i);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b2) {
      return c->bps[c->subs[a].bp].trsm_flops > c->bps[c->subs[b2].bp].trsm_flops;
    });
    b.item0 = (int)it.size();
    for (int i : order)
      for (int ca = 0; ca < c->subs[i].m; ca += c->tx_cw) it.push_back(make_int2(i, ca));
    b.nitems = (int)it.size() - b.item0;
    b.ditem0 = (int)dk;  // di is in the order of the subdomains
    while (dk < di.size() && di[dk].x < b.sub1) ++dk;
    b.nditems = (int)dk - b.ditem0;
    most = std::max(most, (size_t)b.nitems);
  }
  c->tx_grid = (int)std::min<size_t>(c->nsm, std::max<size_t>(most, 1));
  // a recorded assembly holds the old lists
  if (c->asm_exec) CK(cudaGraphExecDestroy(c->asm_exec));
  c->asm_exec = nullptr;
  for (void** p : {(void**)&c->d_tx_ditems, (void**)&c->d_tx_items, (void**)&c->d_txws, (void**)&c->d_txscr}) {
    dfree(c, *p);
    *p = nullptr;
  }
  c->d_tx_ditems = upload(c, di);
  c->d_tx_items = upload(c, it);
  c->d_txws = (double*)dalloc(c, (size_t)c->tx_grid * std::max<int64_t>(c->tx_stack, 8) * c->tx_cw * 8);
  c->d_txscr = (char*)dalloc(c, (size_t)c->tx_grid * trsm_oz_scratch(c->tx_cw));
  CK(cudaStreamSynchronize(c->st));  // the host arrays go out of scope
  c->tx_none = it.empty() || di.empty();
  c->tx_planned = true;
}

// The buffers of that solve: the hand-over blocks, and the digits of as many subdomains at a time as 16 GB and, with the
// hand-over blocks, a third of the free memory hold, one at a time if the allocator refuses that; false where there are
// no large fronts or not even one subdomain fits (trsm_kernel then solves everything).  Memory first, as in
// reserve_syrk_oz, and asked for again by the same rule.
bool reserve_trsm_oz(feti_ctx* c) {
  if (c->ld_bytes == 0 || (c->tx_planned && c->tx_none)) return false;
  if (c->d_LD) return true;
  size_t free_b = 0, total_b = 0;
  CK(cudaMemGetInfo(&free_b, &total_b));
  size_t least = 0;
  for (int i = 0; i < c->nsub; ++i)
    least = std::max(least, (i + 1 < c->nsub ? (size_t)c->info[i + 1].ld : c->ld_bytes) - (size_t)c->info[i].ld);
  if (!c->opt.recompute_X && c->tx_refused > 0 && free_b < c->tx_refused + least + c->th_bytes) return false;
  auto take = [&](size_t bytes) {
    try {
      c->d_LD = dalloc(c, bytes);
      c->d_th = (double*)dalloc(c, std::max<size_t>(c->th_bytes, 8));
      return true;
    } catch (std::bad_alloc&) {
      dfree(c, c->d_LD);
      c->d_LD = nullptr;
      return false;
    }
  };
  try {
    // the plan at hand first (its buffers were released by recompute_X)
    if (c->tx_planned && take(c->tx_ld_bytes)) return true;
    if (c->th_bytes + least <= free_b / 3) {
      const size_t budget = std::min(c->ld_bytes, std::min<size_t>((size_t)16 << 30, free_b / 3 - c->th_bytes));
      for (size_t b : {budget, (size_t)0}) {
        const size_t bytes = std::max(b, least);
        if (!take(bytes)) continue;
        plan_trsm_oz(c, b);
        c->tx_ld_bytes = bytes;
        if (!c->tx_none) return true;
        break;
      }
    }
  } catch (std::bad_alloc&) {  // of the lists or the workspaces
  }
  dfree(c, c->d_LD);
  c->d_LD = nullptr;
  dfree(c, c->d_th);
  c->d_th = nullptr;
  c->tx_refused = std::max<size_t>(free_b, 1);
  return false;
}

void build(feti_ctx* c) {
  using clk = std::chrono::steady_clock;
  auto t0 = clk::now();
  const int ns = c->nsub;
  // ---- distinct patterns (with the Schur-complement route, distinct (pattern, B-touched DOFs) pairs: those
  // DOFs are ordered last, as the root supernode)
  const bool schur = c->opt.assembly_route == 1;
  std::vector<std::vector<int32_t>> tail(ns);
  if (schur)
    for (int i = 0; i < ns; ++i) {
      auto& t = tail[i];
      t.assign(c->subs[i].bdof.begin(), c->subs[i].bdof.end());
      std::sort(t.begin(), t.end());
      t.erase(std::unique(t.begin(), t.end()), t.end());
    }
  std::unordered_map<uint64_t, int> pat_of;
  std::vector<int> pat_rep;
  for (int i = 0; i < ns; ++i) {
    auto& s = c->subs[i];
    uint64_t h = hash_pattern(s.n, s.rowptr.data(), s.col.data());
    if (schur) h = hash_ints(tail[i].data(), (int64_t)tail[i].size(), h);
    auto it = pat_of.find(h);
    if (it == pat_of.end()) {
      pat_of[h] = (int)pat_rep.size();
      s.pat = (int)pat_rep.size();
      pat_rep.push_back(i);
    } else {
      s.pat = it->second;
      auto& r = c->subs[pat_rep[s.pat]];
      if (r.n != s.n || r.col.size() != s.col.size() || (schur && tail[i] != tail[pat_rep[s.pat]]))
        throw ArgError("pattern hash collision");
    }
  }
  SymbolicOptions so;
  so.leaf_dofs = c->opt.leaf_dofs > 0 ? c->opt.leaf_dofs : 16;
  so.use_coords = c->opt.use_coords != 0;
  c->pats.resize(pat_rep.size());
  parallel_for((int)pat_rep.size(), [&](int p) {
    auto& s = c->subs[pat_rep[p]];
    const auto& t = tail[pat_rep[p]];
    analyse_pattern(s.n, s.rowptr.data(), s.col.data(), s.coords.empty() ? nullptr : s.coords.data(), so,
                    c->pats[p], schur ? t.data() : nullptr, schur ? (int)t.size() : 0);
  });
  // ---- distinct RHS plans (pattern, B DOFs)
  std::map<std::pair<int, uint64_t>, int> bp_of;
  std::vector<int> bp_rep;
  for (int i = 0; i < ns; ++i) {
    auto& s = c->subs[i];
    uint64_t h = hash_ints(s.bdof.data(), s.m, (uint64_t)s.m * 1315423911ull);
    auto key = std::make_pair(s.pat, h);
    auto it = bp_of.find(key);
    if (it == bp_of.end()) {
      bp_of[key] = (int)bp_rep.size();
      s.bp = (int)bp_rep.size();
      bp_rep.push_back(i);
    } else {
      s.bp = it->second;
      auto& r = c->subs[bp_rep[s.bp]];
      if (r.m != s.m || !std::equal(r.bdof.begin(), r.bdof.end(), s.bdof.begin()))
        throw ArgError("B pattern hash collision");
    }
  }
  c->bps.resize(bp_rep.size());
  c->bp_pat.resize(bp_rep.size());
  parallel_for((int)bp_rep.size(), [&](int b) {
    auto& s = c->subs[bp_rep[b]];
    c->bp_pat[b] = s.pat;
    plan_rhs(c->pats[s.pat], s.m, s.bdof.data(), c->bps[b]);
  });
  {
    // Cholesky tasks: split heavy subtrees so that the factorisation's work units are at most about a quarter
    // of the average work per persistent CTA (large subdomains get several CTAs; uniform ones balance better)
    int dev = 0;
    CK(cudaGetDevice(&dev));
    int nsm = 0;
    CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    double total = 0;
    for (auto& sh : c->subs) total += c->pats[sh.pat].chol_flops;
    const double slots = (double)std::max(1, nsm * chol_ctas_per_sm());
    const double target = total / (4.0 * slots);
    // fronts at least 256 wide (and their ancestors) go to the tensor-core Cholesky unless switched off.  Whole
    // factorisation with 192 / 256 / 384: 27 elasticity subdomains of 12^3 15.7 / 15.1 / 17.0 ms, 64 of them 28.1 /
    // 26.7 / 29.0, 216 of them 85.2 / 82.1 / 81.8; 64 uneven 3D heat subdomains 23.6 / 27.3 / 32.4, 125 of them 24.1 /
    // 18.9 / 22.1
    if (c->opt.chol_tc < 0 || c->opt.chol_tc > 1) throw ArgError("bad chol_tc (0 tensor cores for large fronts, 1 off)");
    if (c->opt.chol_tc_front < 0) throw ArgError("bad chol_tc_front (0 default, else the narrowest front)");
    const int big_f = c->opt.chol_tc == 1 ? 0 : (c->opt.chol_tc_front > 0 ? std::max(c->opt.chol_tc_front, 128) : 256);
    for (auto& P : c->pats) plan_tasks(P, target, big_f);
    // what chol_kernel does (everything outside the large set) is cut by the same rule on its own flops
    double small = 0;
    for (auto& sh : c->subs) small += c->pats[sh.pat].sub_flops;
    for (auto& P : c->pats) plan_tasks(P, target, big_f, small / (4.0 * slots));
    // CTAs per subdomain of the implicit solves, where there is at most one subdomain per SM: the cluster size with
    // the shortest schedule (largest subdomain first) by the plans' estimates.  Milliseconds per application with
    // 1 / 2 / 4 / 8: 27 elasticity subdomains of 12^3 2.89 / 1.73 / 1.23 / 1.94, 64 of them 2.97 / 1.79 / 2.44 / 5.0;
    // 125 uneven 3D heat subdomains 5.26 / 3.12 / 2.13 / 3.6, 8 of 20^3 2.53 / 1.49 / 1.06 / 0.84; 64 2D heat subdomains
    // of 64^2 0.77 / 0.50 / 0.76 / 1.5, 64 3D ones of 6^3 0.146 / 0.141 / 0.25 / 0.6
    int nmax = 0, maxf = 0;
    for (auto& sh : c->subs) nmax = std::max(nmax, sh.n);
    for (auto& P : c->pats) maxf = std::max(maxf, P.max_f);
    const int force = c->opt.implicit_cluster;
    if (force != 0 && force != -1 && force != 1 && force != 2 && force != 4 && force != 8)
      throw ArgError("bad implicit_cluster (0 auto, -1 one 256-thread CTA, or 1, 2, 4, 8)");
    c->impl_wide = force > 0 || (force == 0 && implicit_wide(ns, nsm, nmax, maxf));
    if (force > 0 && (!implicit_wide(1, nsm, nmax, maxf) ||
                      (force > 1 && implicit_clusters(implicit_smem(nmax, maxf, true), force) < 1)))
      throw ArgError("implicit_cluster: the subdomains do not fit the shared memory of such a cluster");
    if (c->impl_wide) {
      double best = 0;
      for (int C = force > 0 ? force : 1; C <= (force > 0 ? force : 8); C *= 2) {
        const int ncl = C == 1 ? nsm : implicit_clusters(implicit_smem(nmax, maxf, true), C);
        if (ncl < 1) break;
        std::vector<SolveSplit> sp;
        for (auto& P : c->pats) sp.push_back(plan_solve_split(P, C));
        std::vector<double> cost;
        for (auto& sh : c->subs) cost.push_back(sp[sh.pat].cost);
        std::sort(cost.rbegin(), cost.rend());
        std::priority_queue<double, std::vector<double>, std::greater<double>> load;
        for (int k = 0; k < ncl; ++k) load.push(0.0);
        double t = 0;
        for (double x : cost) {
          const double y = load.top() + x;
          load.pop();
          load.push(y);
          t = std::max(t, y);
        }
        if (force > 0 || C == 1 || t < 0.95 * best) {
          best = t;
          c->impl_cluster = C;
          c->solve_splits = std::move(sp);
        }
      }
    }
  }
  c->stats.t_symbolic_ms = std::chrono::duration<double, std::milli>(clk::now() - t0).count();
  c->stats.npatterns = (int)c->pats.size();
  c->stats.nbplans = (int)c->bps.size();

  // ---- concatenate pattern tables
  std::vector<int> sn_c0, sn_w, sn_r, sn_parent, rows, ch_off, ch_list, rel, kmap_src, kmap_dst, diag_src, iperm;
  std::vector<int64_t> sn_rows, rel_off, Lofs, kmap_off, upd_ofs, uofs, usm_ofs;
  std::vector<int> sn_small, sn_task, sn_big, sn_back;
  std::vector<int64_t> sn_hoff, lh_ofs, di_ofs;
  // mixed precision: the fronts the large-front TRSM takes (a bottom block of 128 rows or more, or 256 own rows
  // or more) get a row-major bf16 hi/lo copy of their panel, pat_lh elements per pattern
  std::vector<int64_t> pat_lh(c->pats.size(), 0), pat_di(c->pats.size(), 0);
  auto lh_big = [&](const PatternPlan& P, int s) { return c->fp32 && (P.sn_r[s] >= 128 || P.sn_w[s] >= 256); };
  // FP64: the large fronts' digits and update blocks (kern_trsm_oz.cu)
  std::vector<int64_t> lt_ofs;  // the adjoint's backward solve: digits of L^T (kern_bsolve_oz.cu)
  c->pat_lt.assign(c->pats.size(), 0);
  std::vector<int64_t> ld_ofs, tx_ofs, th_ofs, pat_ld(c->pats.size(), 0), bp_th(c->bps.size(), 0);
  std::vector<int> lvl_off, lvl_sn, pat_lvl0(c->pats.size()), pat_pc0(c->pats.size());
  std::vector<int4> pieces;
  int64_t max_usize = 0;
  std::vector<int> pat_sn0(c->pats.size());
  std::vector<int64_t> pat_diag0(c->pats.size());
  for (size_t p = 0; p < c->pats.size(); ++p) {
    auto& P = c->pats[p];
    pat_sn0[p] = (int)sn_c0.size();
    int64_t rows0 = rows.size(), ch0 = ch_list.size(), rel0 = rel.size(), km0 = kmap_src.size();
    for (int s = 0; s < P.nsn; ++s) {
      sn_c0.push_back(P.sn_c0[s]);
      sn_w.push_back(P.sn_w[s]);
      sn_r.push_back(P.sn_r[s]);
      sn_parent.push_back(P.sn_parent[s]);
      sn_rows.push_back(rows0 + P.sn_rows_off[s]);
      ch_off.push_back((int)(ch0 + P.ch_off[s]));
      rel_off.push_back(rel0 + P.rel_off[s]);
      Lofs.push_back(P.Lofs[s]);
      kmap_off.push_back(km0 + P.kmap_off[s]);
      upd_ofs.push_back(P.upd_stack_ofs[s]);
      sn_small.push_back(P.sn_small[s]);
      usm_ofs.push_back(P.usm_ofs[s]);
      sn_task.push_back(P.sn_task[s]);
      sn_hoff.push_back(P.sn_hoff[s]);
      sn_big.push_back(P.sn_big[s]);
      sn_back.push_back(P.sn_back[s]);
      lh_ofs.push_back(lh_big(P, s) ? pat_lh[p] : -1);
      di_ofs.push_back(lh_big(P, s) ? pat_di[p] : -1);
      if (lh_big(P, s)) {
        pat_lh[p] += (int64_t)(P.sn_w[s] + P.sn_r[s]) * 2 * ((P.sn_w[s] + 7) & ~7);
        pat_di[p] += (int64_t)((P.sn_w[s] + 127) / 128) * 4 * 32 * 32;
      }
      uofs.push_back(P.uofs[s]);
    }
    for (int s = 0; s < P.nsn; ++s) {
      lt_ofs.push_back(P.sn_back[s] ? c->pat_lt[p] / 512 : -1);
      for (int kB = 0; P.sn_back[s] && kB < P.sn_w[s]; kB += 128)
        c->pat_lt[p] += bsolve_oz_block_bytes(P.sn_w[s], P.sn_r[s], kB);
    }
    if (!c->fp32) {
      // the digits of each 128-column block, and the update blocks of the large supernodes, each disjoint from its
      // children's
      BlockPlaces places;
      for (int s = 0; s < P.nsn; ++s) {  // postorder
        ld_ofs.push_back(P.sn_big[s] ? pat_ld[p] / 512 : -1);
        int64_t base = 0;
        if (P.sn_big[s]) {
          for (int kB = 0; kB < P.sn_w[s]; kB += 128) pat_ld[p] += trsm_oz_block_bytes(P.sn_w[s], P.sn_r[s], kB);
          const int64_t rp = (P.sn_r[s] + 7) & ~7;
          if (P.sn_parent[s] >= 0 && rp > 0) {
            base = places.take(s, rp);
            c->tx_stack = std::max(c->tx_stack, base + rp);
          }
          for (int k = P.ch_off[s]; k < P.ch_off[s + 1]; ++k) places.release(P.ch_list[k]);
        }
        tx_ofs.push_back(base);
      }
    }
    pat_lvl0[p] = (int)lvl_off.size();
    {
      const int b0 = (int)lvl_sn.size();
      for (int l = 0; l <= P.nlev; ++l) lvl_off.push_back(b0 + P.lvl_off[l]);
      lvl_sn.insert(lvl_sn.end(), P.lvl_sn.begin(), P.lvl_sn.end());
      pat_pc0[p] = (int)pieces.size();
      if (c->impl_cluster > 1) {
        const SolveSplit& sp = c->solve_splits[p];
        for (int k = 0; k <= c->impl_cluster; ++k) {
          const int b1 = (int)lvl_sn.size();
          for (int o : sp.off[k]) lvl_off.push_back(b1 + o);
          lvl_sn.insert(lvl_sn.end(), sp.own[k].begin(), sp.own[k].end());
        }
        for (auto& q : sp.pieces) pieces.push_back(make_int4(q.c0, q.c1, q.rank, 0));
      }
    }
    max_usize = std::max(max_usize, P.usize);
    c->impl_maxf = std::max(c->impl_maxf, P.max_f);
    rows.insert(rows.end(), P.rows.begin(), P.rows.end());
    ch_list.insert(ch_list.end(), P.ch_list.begin(), P.ch_list.end());
    rel.insert(rel.end(), P.rel.begin(), P.rel.end());
    kmap_src.insert(kmap_src.end(), P.kmap_src.begin(), P.kmap_src.end());
    kmap_dst.insert(kmap_dst.end(), P.kmap_dst.begin(), P.kmap_dst.end());
    pat_diag0[p] = diag_src.size();
    diag_src.insert(diag_src.end(), P.diag_src.begin(), P.diag_src.end());
    iperm.insert(iperm.end(), P.iperm.begin(), P.iperm.end());
  }
  sn_rows.push_back(rows.size());
  ch_off.push_back((int)ch_list.size());
  rel_off.push_back(rel.size());
  kmap_off.push_back(kmap_src.size());
  // ---- concatenate RHS plans
  std::vector<int> jb, je, jo, act, spos, tile_off, tile_sn, t2_off, t2_sn;
  std::vector<int> bp_t20(c->bps.size());
  std::vector<int64_t> Xofs, rhs_ofs;
  std::vector<int> bp_sn0(c->bps.size()), bp_act0(c->bps.size()), bp_col0(c->bps.size()), bp_tile0(c->bps.size());
  for (size_t b = 0; b < c->bps.size(); ++b) {
    auto& B = c->bps[b];
    bp_sn0[b] = (int)jb.size();
    bp_act0[b] = (int)act.size();
    bp_col0[b] = (int)spos.size();
    bp_tile0[b] = (int)tile_off.size();
    jb.insert(jb.end(), B.jb.begin(), B.jb.end());
    je.insert(je.end(), B.je.begin(), B.je.end());
    jo.insert(jo.end(), B.jo.begin(), B.jo.end());
    Xofs.insert(Xofs.end(), B.Xofs.begin(), B.Xofs.end());
    rhs_ofs.insert(rhs_ofs.end(), B.rhs_stack_ofs.begin(), B.rhs_stack_ofs.end());
    if (!c->fp32) {
      auto& P = c->pats[c->bp_pat[b]];
      for (int s = 0; s < P.nsn; ++s) {
        const int64_t J = B.je[s] - B.jb[s];
        const bool slot = !P.sn_big[s] && P.sn_parent[s] >= 0 && P.sn_big[P.sn_parent[s]] && J > 0;
        th_ofs.push_back(slot ? bp_th[b] : -1);
        if (slot) bp_th[b] += J * P.sn_r[s];
      }
    }
    act.insert(act.end(), B.act.begin(), B.act.end());
    spos.insert(spos.end(), B.spos.begin(), B.spos.end());
    int base = (int)tile_sn.size();
    int ntile = B.nb * (B.nb + 1) / 2;
    for (int t = 0; t < ntile; ++t) tile_off.push_back(base + B.tile_off[t]);
    tile_sn.insert(tile_sn.end(), B.tile_sn.begin(), B.tile_sn.end());
    bp_t20[b] = (int)t2_off.size();
    int base2 = (int)t2_sn.size();
    int nt2 = B.nb2 * (B.nb2 + 1) / 2;
    for (int t = 0; t < nt2; ++t) t2_off.push_back(base2 + B.t2_off[t]);
    t2_sn.insert(t2_sn.end(), B.t2_sn.begin(), B.t2_sn.end());
  }
  tile_off.push_back((int)tile_sn.size());
  t2_off.push_back((int)t2_sn.size());

  // ---- per-subdomain layout
  c->info.resize(ns);
  std::vector<int> qmap, fix_sn, colsub, colperm, qdof, dofsub, colperm_pad;
  std::vector<int> eldofs;
  std::vector<double> eldk, elsc;
  std::vector<double> qsign;
  std::vector<int64_t> fix_pos;
  int64_t Kofs = 0, Lo = 0, Xo = 0, Fo = 0, qo = 0, dofo = 0, Ro = 0, tpo = 0, hbo = 0, lho = 0, dio = 0, ldo = 0, tho = 0;
  std::vector<int2> l16_items;
  int fixo = 0, alo = 0;
  double chol = 0, trsm = 0, syrk = 0, syrke = 0, implb = 0;
  int64_t sub_chol = 0, big_chol = 0;
  int64_t max_rhs = 0, max_rf = 0, max_usm = 0, ntasks = 0;
  size_t esz = c->fp32 ? 4 : 8;
  double apply_bytes = 0, stored_bytes = 0;
  c->colperm_ofs.resize(ns);
  for (int i = 0; i < ns; ++i) {
    auto& s = c->subs[i];
    auto& P = c->pats[s.pat];
    auto& B = c->bps[s.bp];
    SubInfo& I = c->info[i];
    I.n = s.n;
    I.m = s.m;
    c->m_max = std::max(c->m_max, s.m);
    I.m_pad = B.m_pad;
    I.nb = B.nb;
    I.nsn = P.nsn;
    I.nact = (int)B.act.size();
    I.d = s.d;
    I.nfix = s.nfix;
    I.sn0 = pat_sn0[s.pat];
    I.bsn0 = bp_sn0[s.bp];
    I.act0 = bp_act0[s.bp];
    I.col0 = bp_col0[s.bp];
    I.tile0 = bp_tile0[s.bp];
    I.t20 = bp_t20[s.bp];
    I.nb2 = B.nb2;
    I.vr = B.nb > 0 ? s.m - kT * (B.nb - 1) : 0;
    I.nlev = P.nlev;
    I.lvl0 = pat_lvl0[s.pat];
    I.pc0 = pat_pc0[s.pat];
    I.npc = c->impl_cluster > 1 ? (int)c->solve_splits[s.pat].pieces.size() : 0;
    I.fix0 = fixo;
    I.alpha0 = alo;
    I.kmapb = 0;
    I.diag0 = pat_diag0[s.pat];
    I.Kval = Kofs;
    I.L = Lo;
    I.X = Xo;
    I.F = Fo;
    I.qcol = qo;
    I.trow = qo;
    I.dof = dofo;
    I.R = Ro;
    I.tpart = tpo;
    I.rpart = 0;
    I.hbase = hbo;
    hbo += P.hsize;
    I.lh = lho;
    lho += pat_lh[s.pat];
    I.ld = ldo;
    ldo += pat_ld[s.pat];
    I.th = tho;
    tho += bp_th[s.bp];
    I.di = dio;
    dio += pat_di[s.pat];
    for (int q = 0; q < P.nsn; ++q)
      if (lh_big(P, q)) l16_items.push_back(make_int2(i, q));
    int ntile = B.nb * (B.nb + 1) / 2;
    Kofs += (int64_t)s.col.size();
    Lo += P.Lsize;
    Xo += B.Xsize;
    Fo += F_size_esz((int)esz, B.nb, I.vr);
    qo += B.m_pad;
    dofo += s.n;
    Ro += (int64_t)s.n * s.d;
    tpo += (int64_t)ntile * kT;
    alo += s.d;
    for (int j = 0; j < B.m_pad; ++j) {
      if (j < s.m) {
        int r = B.colperm[j];
        qmap.push_back(s.blam[r]);
        qsign.push_back(s.bsign[r]);
        colperm.push_back(r);
        colperm_pad.push_back(r);
        qdof.push_back(s.bdof[r]);
      } else {
        qmap.push_back(-1);
        qsign.push_back(0.0);
        qdof.push_back(0);
        colperm_pad.push_back(0);
      }
      colsub.push_back(i);
    }
    c->colperm_ofs[i] = (int64_t)colperm.size() - s.m;
    for (int k = 0; k < s.nfix; ++k) {
      int nd = P.iperm[s.fix[k]];
      int sn = P.col2sn[nd];
      int loc = nd - P.sn_c0[sn];
      int f = P.sn_w[sn] + P.sn_r[sn];
      fix_sn.push_back(sn);
      fix_pos.push_back(P.Lofs[sn] + (int64_t)loc * f + loc);
    }
    fixo += s.nfix;
    for (int k = 0; k < s.n; ++k) dofsub.push_back(i);
    c->elem_ofs.push_back((int64_t)elsc.size());
    c->elem_dk_ofs.push_back((int64_t)eldk.size());
    c->elem_dofs_ofs.push_back((int64_t)eldofs.size());
    eldofs.insert(eldofs.end(), s.elem_dofs.begin(), s.elem_dofs.end());
    eldk.insert(eldk.end(), s.dKe.begin(), s.dKe.end());
    elsc.insert(elsc.end(), s.dKe_scale.begin(), s.dKe_scale.end());
    c->nmax = std::max(c->nmax, s.n);
    chol += P.chol_flops;
    trsm += B.trsm_flops;
    syrk += B.syrk_flops;
    syrke += B.syrk_exec_flops;
    implb += 2.0 * 8.0 * P.nnzL;
    ntasks += P.ntask;
    max_usm = std::max(max_usm, P.usm_size);
    sub_chol = std::max(sub_chol, P.sub_stack);
    big_chol = std::max(big_chol, P.big_stack);
    max_rhs = std::max(max_rhs, B.rhs_stack);
    max_rf = std::max(max_rf, B.rhs_front);
    apply_bytes += (double)esz * s.m * (s.m + 1) / 2.0 + (double)s.m * (4 + 8 + 8);
    stored_bytes += (double)esz * F_size_esz((int)esz, B.nb, I.vr);
  }
  apply_bytes += (double)c->nlam * 16.0;
  c->ncols = qo;
  c->dtot = alo;
  c->stats.nsub = ns;
  c->stats.n_lambda = c->nlam;
  c->stats.sum_n = dofo;
  c->stats.sum_m = 0;
  for (auto& s : c->subs) c->stats.sum_m += s.m;
  c->stats.L_doubles = Lo;
  c->stats.X_elems = Xo;
  c->stats.F_elems = Fo;
  c->stats.chol_flops = chol;
  c->stats.trsm_flops = trsm;
  c->stats.syrk_flops = syrk;
  c->stats.syrk_exec_flops = syrke;
  c->stats.apply_bytes = apply_bytes;
  c->stats.implicit_bytes = implb;

  // ---- lambda -> contributions (deterministic: subdomain order)
  std::vector<int> c0(c->nlam, -1), c1(c->nlam, -1);
  for (int i = 0; i < ns; ++i) {
    auto& I = c->info[i];
    for (int j = 0; j < I.m; ++j) {
      int lam = qmap[I.qcol + j];
      if (lam < 0 || lam >= c->nlam) throw ArgError("B_lambda out of range");
      if (c0[lam] < 0) c0[lam] = (int)(I.qcol + j);
      else if (c1[lam] < 0) c1[lam] = (int)(I.qcol + j);
      else throw ArgError("a multiplier touches more than two subdomains");
    }
  }
  // per multiplier: {tile base, (column << 8) | nb} of its first and second subdomain column (the PCPG
  // gather), and {alpha0, d} of its first and second subdomain (the projector in the update)
  std::vector<int4> lamcol(c->nlam, make_int4(0, 0, -1, 0)), lamg(c->nlam, make_int4(0, 0, 0, 0));
  for (int l = 0; l < c->nlam; ++l) {
    const int g[2] = {c0[l], c1[l]};
    int v[4] = {0, 0, -1, 0}, a[4] = {0, 0, 0, 0};
    for (int e = 0; e < 2; ++e) {
      if (g[e] < 0) continue;
      const auto& J = c->info[colsub[g[e]]];
      if (J.nb > 255) throw ArgError("a subdomain has more than 255 64-wide blocks of multipliers");
      v[2 * e] = (int)(J.tpart / kT);
      v[2 * e + 1] = (int)((g[e] - J.qcol) << 8) | J.nb;
      a[2 * e] = J.alpha0;
      a[2 * e + 1] = J.d;
    }
    lamcol[l] = make_int4(v[0], v[1], v[2], v[3]);
    lamg[l] = make_int4(a[0], a[1], a[2], a[3]);
  }

  // ---- coarse problem pairs: (i, k) blocks of G^T G and the sorted columns they pair
  {
    std::map<std::pair<int, int>, std::vector<int2>> pm;
    for (int i = 0; i < ns; ++i) {
      auto& I = c->info[i];
      if (I.d == 0) continue;
      auto& v = pm[{i, i}];
      for (int j = 0; j < I.m; ++j) v.push_back(make_int2((int)(I.qcol + j), (int)(I.qcol + j)));
    }
    for (int l = 0; l < c->nlam; ++l) {
      if (c0[l] < 0 || c1[l] < 0) continue;
      int i = colsub[c0[l]], k = colsub[c1[l]];
      if (c->info[i].d == 0 || c->info[k].d == 0) continue;
      if (i < k) pm[{i, k}].push_back(make_int2(c0[l], c1[l]));
      else pm[{k, i}].push_back(make_int2(c1[l], c0[l]));
    }
    std::vector<int4> pairs;
    std::vector<int2> plist;
    for (auto& kv : pm) {
      auto& Ii = c->info[kv.first.first];
      auto& Ik = c->info[kv.first.second];
      int b = (int)plist.size();
      plist.insert(plist.end(), kv.second.begin(), kv.second.end());
      pairs.push_back(make_int4(Ii.alpha0 | (Ii.d << 24), Ik.alpha0 | (Ik.d << 24), b, (int)plist.size()));
    }
    c->npairs = (int)pairs.size();
    c->d_pairs = upload(c, pairs);
    c->d_plist = upload(c, plist);
  }
  for (auto& I : c->info)
    if (I.d > 6) throw ArgError("kernel dimension d > 6 is not supported");

  // ---- work orders
  std::vector<int> order(ns);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return c->pats[c->subs[a].pat].chol_flops > c->pats[c->subs[b].pat].chol_flops;
  });
  std::vector<int> order_t(order);
  std::stable_sort(order_t.begin(), order_t.end(), [&](int a, int b) {
    return c->bps[c->subs[a].bp].trsm_flops > c->bps[c->subs[b].bp].trsm_flops;
  });
  std::vector<int> order_i(order);
  std::stable_sort(order_i.begin(), order_i.end(), [&](int a, int b) {
    return c->pats[c->subs[a].pat].nnzL > c->pats[c->subs[b].pat].nnzL;
  });
  std::vector<std::pair<double, int2>> sy;
  std::vector<TileDesc> tdesc;
  for (int i = 0; i < ns; ++i) {
    auto& B = c->bps[c->subs[i].bp];
    auto& P = c->pats[c->subs[i].pat];
    auto& I = c->info[i];
    int ntile = B.nb * (B.nb + 1) / 2;
    for (int t = 0; t < ntile; ++t) {
      double cost = 1.0;
      for (int k = B.tile_off[t]; k < B.tile_off[t + 1]; ++k) cost += P.sn_w[B.tile_sn[k]];
      sy.push_back({cost, make_int2(i, t)});
    }
    // one descriptor per tile, in tile order (tile t of the list owns partial slot t)
    for (int b = 0; b < B.nb; ++b)
      for (int bj = 0; bj <= b; ++bj) {
        TileDesc d{};
        d.f_ofs = I.F + (c->fp32 ? tile_offset<4>(B.nb, I.vr, b, bj) : tile_offset<8>(B.nb, I.vr, b, bj));
        d.rows = tile_rows(B.nb, I.vr, b);
        d.flags = bj == b ? kTileDiag : 0;
        d.prow = (int)(I.qcol + (int64_t)b * kT);
        d.pcol = (int)(I.qcol + (int64_t)bj * kT);
        d.slot = (int)tdesc.size();
        tdesc.push_back(d);
      }
  }
  {
    // subdomain-major copy (the TRSM-path assembly writes each subdomain's tiles)
    std::vector<int> t0(ns, 0);
    for (int i = 1; i < ns; ++i) t0[i] = t0[i - 1] + c->bps[c->subs[i - 1].bp].nb * (c->bps[c->subs[i - 1].bp].nb + 1) / 2;
    c->d_tdesc_sub = upload(c, tdesc);
    c->d_tile0 = upload(c, t0);
  }
  // the tile kernels give warp g the descriptors g, g + N, g + 2N, ...: with the largest tiles first, the
  // k-th tiles of all warps are alike in size and the last round holds the smallest ones (ragged slivers)
  std::stable_sort(tdesc.begin(), tdesc.end(), [&](const TileDesc& a, const TileDesc& b) {
    auto bytes = [&](const TileDesc& d) {
      const int64_t e = (d.flags & kTileDiag) ? (c->fp32 ? diag_row_off<4>(d.rows) : diag_row_off<8>(d.rows))
                                               : (int64_t)d.rows * kT;
      return e;
    };
    return bytes(a) > bytes(b);
  });
  c->napply = (int)tdesc.size();
  std::vector<std::pair<double, int2>> sy2;
  for (int i = 0; i < ns; ++i) {
    auto& B = c->bps[c->subs[i].bp];
    auto& P = c->pats[c->subs[i].pat];
    int nt2 = B.nb2 * (B.nb2 + 1) / 2;
    for (int t = 0; t < nt2; ++t) {
      double cost = 1.0;
      for (int k = B.t2_off[t]; k < B.t2_off[t + 1]; ++k) cost += P.sn_w[B.t2_sn[k]];
      sy2.push_back({cost, make_int2(i, t)});
    }
  }
  std::stable_sort(sy2.begin(), sy2.end(), [](auto& a, auto& b) { return a.first > b.first; });
  std::vector<int2> sy2i;
  for (auto& x : sy2) sy2i.push_back(x.second);
  c->nsyrk2 = (int)sy2i.size();
  std::stable_sort(sy.begin(), sy.end(), [](auto& a, auto& b) { return a.first > b.first; });
  std::vector<int2> syi;
  for (auto& x : sy) syi.push_back(x.second);
  std::vector<int2> blocks;
  for (int i = 0; i < ns; ++i)
    for (int b = 0; b < c->bps[c->subs[i].bp].nb; ++b) blocks.push_back(make_int2(i, b));
  c->nblocks = (int)blocks.size();
  c->nsyrk = (int)syi.size();

  // ---- persistent grids and workspace
  int dev = 0;
  CK(cudaGetDevice(&dev));
  cudaDeviceProp prop;
  CK(cudaGetDeviceProperties(&prop, dev));
  c->nsm = prop.multiProcessorCount;
  c->grid_chol = std::min(ns, c->nsm * chol_ctas_per_sm());
  {
    int64_t max_items = 0;  // the finest TRSM work split (64 columns per item)
    for (auto& sh : c->subs) max_items += std::max(1, (sh.m + 63) / 64);
    c->grid_trsm = (int)std::min<int64_t>(max_items, c->nsm * 3);
    // the mixed TRSM holds the tensor-core stage ring in shared memory: fewer resident CTAs
    c->grid_trsm32 = (int)std::min<int64_t>(c->grid_trsm, (int64_t)c->nsm * trsm_ctas_per_sm(true, 2));
  }
  c->rhs_front = max_rf;
  // one buffer for three kernels that run one after another: the TRSM's fronts and stacks per CTA or the tensor-core
  // Cholesky's update blocks per cluster (ws_stride), or chol_kernel's update blocks per CTA (sub_stride)
  c->ws_stride = std::max<int64_t>((std::max(big_chol, max_rf + max_rhs) + 31) / 32 * 32, 32);
  c->sub_stack = sub_chol;
  c->sub_stride = std::max<int64_t>((sub_chol + max_usm + 31) / 32 * 32, 32);
  {
    // it may take at most 40% of the free device memory: large fronts (the Schur-complement route's dense root) get
    // fewer CTAs
    size_t free_b = 0, total_b = 0;
    CK(cudaMemGetInfo(&free_b, &total_b));
    const int64_t cap = std::max<int64_t>(1, (int64_t)(0.4 * (double)free_b) / (c->ws_stride * 8));
    c->grid_ws = (int)std::max<int64_t>(1, std::min<int64_t>(c->grid_chol, cap));
    c->grid_trsm = (int)std::max<int64_t>(1, std::min<int64_t>(c->grid_trsm, cap));
    c->grid_trsm32 = std::max(1, std::min(c->grid_trsm32, c->grid_trsm));
    c->grid_ws = std::max(c->grid_ws, c->grid_trsm);
    // chol_kernel's tasks outnumber the subdomains (with one CTA per subdomain 64 subdomains left half the SMs idle)
    const int64_t cap_c = std::max<int64_t>(1, (int64_t)(0.4 * (double)free_b) / (c->sub_stride * 8));
    c->grid_chol = (int)std::min<int64_t>(std::min<int64_t>((int64_t)c->nsm * chol_ctas_per_sm(), cap_c),
                                          std::max<int64_t>(ntasks, 1));
  }
  const int64_t ws_doubles = std::max((int64_t)c->grid_ws * c->ws_stride, (int64_t)c->grid_chol * c->sub_stride);

  // ---- device uploads
  DevPlan& D = c->P;
  D.sn_c0 = upload(c, sn_c0);
  D.sn_w = upload(c, sn_w);
  D.sn_r = upload(c, sn_r);
  D.sn_parent = upload(c, sn_parent);
  D.sn_rows = upload(c, sn_rows);
  D.rows = upload(c, rows);
  D.ch_off = upload(c, ch_off);
  D.ch_list = upload(c, ch_list);
  D.rel_off = upload(c, rel_off);
  D.rel = upload(c, rel);
  D.Lofs = upload(c, Lofs);
  D.kmap_off = upload(c, kmap_off);
  D.kmap_src = upload(c, kmap_src);
  D.kmap_dst = upload(c, kmap_dst);
  D.diag_src = upload(c, diag_src);
  D.upd_ofs = upload(c, upd_ofs);
  D.lvl_off = upload(c, lvl_off);
  D.pieces = upload(c, pieces);
  D.lvl_sn = upload(c, lvl_sn);
  D.uofs = upload(c, uofs);
  D.sn_small = upload(c, sn_small);
  D.usm_ofs = upload(c, usm_ofs);
  D.sn_task = upload(c, sn_task);
  D.sn_big = upload(c, sn_big);
  D.sn_back = upload(c, sn_back);
  D.sn_hoff = upload(c, sn_hoff);
  D.lh_ofs = upload(c, lh_ofs);
  D.di_ofs = upload(c, di_ofs);
  D.lt_ofs = upload(c, lt_ofs);
  D.ld_ofs = upload(c, ld_ofs);
  D.tx_ofs = upload(c, tx_ofs);
  D.th_ofs = upload(c, th_ofs);
  c->ld_bytes = (size_t)ldo;
  c->th_bytes = (size_t)tho * 8;
  if (c->fp32) {
    D.LH = (uint16_t*)dalloc(c, (size_t)std::max<int64_t>(lho, 8) * 2);
    D.DI = (float*)dalloc(c, (size_t)std::max<int64_t>(dio, 8) * 4);
    c->d_l16_items = upload(c, l16_items);
    c->n_l16 = (int)l16_items.size();
  }
  c->d_hand = (double*)dalloc(c, (size_t)std::max<int64_t>(hbo, 1) * 8);
  D.jb = upload(c, jb);
  D.je = upload(c, je);
  D.jo = upload(c, jo);
  D.Xofs = upload(c, Xofs);
  D.rhs_ofs = upload(c, rhs_ofs);
  D.act = upload(c, act);
  D.spos = upload(c, spos);
  D.tile_off = upload(c, tile_off);
  D.tile_sn = upload(c, tile_sn);
  D.t2_off = upload(c, t2_off);
  D.t2_sn = upload(c, t2_sn);
  D.qmap = upload(c, qmap);
  D.qsign = upload(c, qsign);
  D.fix_sn = upload(c, fix_sn);
  D.iperm = upload(c, iperm);
  D.qdof = upload(c, qdof);
  D.colperm = upload(c, colperm_pad);
  c->nelem_total = (int64_t)elsc.size();
  {
    std::vector<int> ident(ns);
    std::iota(ident.begin(), ident.end(), 0);
    c->d_ident = upload(c, ident);
  }
  if (!elsc.empty()) {
    c->d_eldofs = upload(c, eldofs);
    c->d_eldk = upload(c, eldk);
    c->d_elsc = upload(c, elsc);
  }
  c->d_dofsub = upload(c, dofsub);
  c->ndof = (int64_t)dofsub.size();
  D.fix_pos = upload(c, fix_pos);
  D.sub = upload(c, c->info);
  std::vector<double> kv;
  kv.reserve(Kofs);
  std::vector<double> Rall, fall;
  for (auto& s : c->subs) {
    kv.insert(kv.end(), s.val.begin(), s.val.end());
    Rall.insert(Rall.end(), s.R.begin(), s.R.end());
    fall.insert(fall.end(), s.f.begin(), s.f.end());
  }
  c->d_Kval = upload(c, kv);
  D.Kval = c->d_Kval;
  c->d_L = (double*)dalloc(c, (size_t)Lo * 8);
  D.L = c->d_L;
  if (c->fp32) c->d_L32 = (float*)dalloc(c, (size_t)std::max<int64_t>(Lo, 1) * 4);
  D.dinv = (double*)dalloc(c, (size_t)std::max<int64_t>(c->ndof, 1) * 8);
  D.rho = (double*)dalloc(c, (size_t)ns * 8);
  c->d_X = dalloc(c, (size_t)Xo * esz);
  c->d_F = dalloc(c, (size_t)Fo * esz);
  c->d_ws = (double*)dalloc(c, (size_t)ws_doubles * 8);
  c->d_trow = (double*)dalloc(c, (size_t)qo * 8);
  c->d_tpart = (double*)dalloc(c, (size_t)std::max<int64_t>(tpo, 1) * 8);
  c->d_rowpart = dalloc(c, (size_t)std::max<int64_t>(tpo, 1) * 8);
  c->d_pg = dalloc(c, (size_t)qo * 8);
  c->d_qi = (double*)dalloc(c, (size_t)qo * 8);
  c->d_colsub = upload(c, colsub);
  D.colsub = c->d_colsub;
  c->d_c0 = upload(c, c0);
  c->d_c1 = upload(c, c1);
  c->d_lamcol = upload(c, lamcol);
  if (c->opt.precond == 2 && c->opt.assembly_route != 1)
    throw ArgError("the Dirichlet preconditioner needs assembly_route = 1 (its S_i is the root front of that "
                   "ordering)");
  if (c->opt.precond == 1 || c->opt.precond == 2) {
    LumpedPlan lp;
    plan_lumped(c, lp);
    c->precond = true;
    c->precond_kind = c->opt.precond;
    c->d_w_off = upload(c, lp.w_off);
    c->d_w_col = upload(c, lp.w_col);
    c->d_w_val = upload(c, lp.w_val);
  }
  if (c->opt.precond == 2) {
    // S_i from a second factorisation of K (no penalty) that stops at the root front; M_i tiles as F_i
    c->P2 = D;
    c->P2.L = (double*)dalloc(c, (size_t)Lo * 8);
    c->P2.rho = (double*)dalloc(c, (size_t)ns * 8);
    c->d_M = dalloc(c, (size_t)std::max<int64_t>(Fo, 1) * esz);
    c->d_pg2 = dalloc(c, (size_t)qo * esz);
    CK(cudaMemsetAsync(c->d_pg2, 0, (size_t)qo * esz, c->st));  // padding columns stay zero
  }
  if (c->opt.precond == 1) {
    LumpedPlan lp;
    plan_lumped(c, lp);
    c->d_m_off = upload(c, lp.m_off);
    c->d_m_col = upload(c, lp.m_col);
    c->m_nnz = (int64_t)lp.m_col.size();
    c->d_m_val = (double*)dalloc(c, (size_t)std::max<int64_t>(c->m_nnz, 1) * 8);
    c->d_mc_off = upload(c, lp.c_off);
    c->d_mc_kidx = upload(c, lp.c_kidx);
    c->d_mc_sign = upload(c, lp.c_sign);
  }
  c->d_lamg = upload(c, lamg);
  c->d_qcol = (double*)dalloc(c, (size_t)qo * 8);
  c->d_queue = (int*)dalloc(c, 64 * sizeof(int));
  c->d_status = (int*)dalloc(c, sizeof(int));
  c->d_chol_order = upload(c, order);
  {
    // Cholesky work items: whole subdomains (cost order), and the tasks of the split, children before
    // parents (by task height), heavier first
    std::vector<int4> whole;
    for (int si : order) whole.push_back(make_int4(si, 0, 0, -1));
    std::vector<std::pair<std::pair<int, double>, int4>> tk, tkb;
    std::vector<int> nchild, nbig;
    int base = 0;
    for (int i = 0; i < ns; ++i) {
      const auto& P = c->pats[c->subs[i].pat];
      for (int t = 0; t < P.ntask; ++t) {
        nchild.push_back(P.task_nchild[t]);
        nbig.push_back(P.task_nbig[t]);
        const int4 item = make_int4(i, t, base + t, P.task_parent[t] >= 0 ? base + P.task_parent[t] : -1);
        // the large fronts' tasks are the tensor-core kernel's items
        (P.task_big[t] ? tkb : tk).push_back({{P.task_height[t], -P.task_cost[t]}, item});
      }
      base += P.ntask;
    }
    std::stable_sort(tk.begin(), tk.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    std::stable_sort(tkb.begin(), tkb.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    std::vector<int4> split;
    for (auto& x : tk) split.push_back(x.second);
    c->d_chol_items[0] = upload(c, whole);
    c->d_chol_items[1] = upload(c, split);
    c->chol_nitems[0] = (int)whole.size();
    c->chol_nitems[1] = (int)split.size();
    c->ntask_total = base;
    D.task_nchild = upload(c, nchild);
    c->P2.task_nchild = D.task_nchild;
    D.task_nbig = upload(c, nbig);
    c->P2.task_nbig = D.task_nbig;
    c->d_tdone = (int*)dalloc(c, (size_t)std::max(base, 1) * sizeof(int));
    // the tensor-core Cholesky's items: the large tasks, children first; its scratch per cluster: the bf16 digits and
    // a row exponent for every row of the largest such front
    {
      int fmax = 0;
      for (int i = 0; i < ns; ++i) {
        const auto& P = c->pats[c->subs[i].pat];
        for (int q = 0; q < P.nsn; ++q)
          if (P.sn_big[q]) fmax = std::max(fmax, P.sn_w[q] + P.sn_r[q]);
      }
      std::vector<int4> tci;
      for (auto& x : tkb) tci.push_back(x.second);
      c->n_tc_items = (int)tci.size();
      if (c->n_tc_items > 0) {
        c->d_tc_items = upload(c, tci);
        int nbig_sub = 0;
        for (int i = 0; i < ns; ++i) nbig_sub += c->pats[c->subs[i].pat].has_big ? 1 : 0;
        c->tc_cluster = chol_tc_cluster(nbig_sub, c->nsm);
        c->grid_tc = std::max(1, std::min(c->nsm / c->tc_cluster, std::min(c->n_tc_items, c->grid_ws)));
        c->slice_stride = chol_tc_scratch(fmax);
        c->d_slices = (char*)dalloc(c, (size_t)c->grid_tc * c->slice_stride);
      }
    }
    // nothing to split: the whole-subdomain items only
    if (c->opt.chol_split < 0 || c->opt.chol_split > 2) throw ArgError("bad chol_split (0 auto, 1 whole, 2 tasks)");
    c->chol_pick = c->opt.chol_split == 2 ? 1 : 0;
    c->chol_tuned = c->opt.chol_split != 0 || (int)split.size() == ns;
    if (c->opt.syrk_kernel < 0 || c->opt.syrk_kernel > 3) throw ArgError("bad syrk_kernel (0 auto, 1-3 a kernel)");
    if (c->opt.syrk_kernel > 0) {
      c->syrk_variant = c->opt.syrk_kernel - 1;
      c->syrk_tuned = true;
      c->stats.syrk_variant = c->syrk_variant;
    }
  }
  c->d_trsm_order = upload(c, order_t);
  {
    // TRSM work items: a whole subdomain per CTA, or blocks of cw sorted columns (the columns of X are
    // independent); the autotuner times each at the first assembly
    for (int cw : {0, 1024, 512, 256, 128, 64}) {
      if (cw > 0 && cw >= c->m_max) continue;
      std::vector<int2> it;
      for (int si : order_t) {
        const int m = c->subs[si].m;
        if (cw == 0 || m <= cw) it.push_back(make_int2(si, 0));
        else
          for (int ca = 0; ca < m; ca += cw) it.push_back(make_int2(si, ca));
      }
      c->trsm_cands.push_back({cw, upload(c, it), (int)it.size(), 0.0});
    }
  }
  c->d_impl_order = upload(c, order_i);
  c->d_syrk_items = upload(c, syi);
  {
    // the apply deals tiles to warps round-robin; candidates of the autotuner:
    // every variant of the tile kernel at its full occupancy (capped at one tile per warp)
    c->d_tdesc = upload(c, tdesc);
    if (!c->fp32) {
      c->d_fscale = (int*)dalloc(c, (size_t)std::max<int64_t>(c->ncols, 1) * sizeof(int));
      if (c->precond_kind == 2) c->d_mscale = (int*)dalloc(c, (size_t)std::max<int64_t>(c->ncols, 1) * sizeof(int));
    }
    for (int v = 0; v < apply_variants(); ++v) {
      const int wpc = apply_warps_per_cta(v);
      const int occ = apply_max_ctas_per_sm(c->fp32, v);
      if (occ <= 0) continue;
      const int G = std::max(1, std::min((c->napply + wpc - 1) / wpc, c->nsm * occ));
      c->apply_cands.push_back({v, G, 0.0});
    }
    if (c->apply_cands.empty()) throw CudaError("no launchable configuration of the apply kernel");
    c->apply_pick = (int)c->apply_cands.size() - 1;
    if (c->opt.apply_kernel < 0 || c->opt.apply_kernel > apply_variants())
      throw ArgError("bad apply_kernel (0 auto, else feti_stats.apply_variant + 1)");
    if (c->opt.apply_kernel > 0) {
      for (size_t k = 0; k < c->apply_cands.size(); ++k)
        if (c->apply_cands[k].variant == c->opt.apply_kernel - 1) {
          c->apply_pick = (int)k;
          c->apply_tuned = true;
        }
      if (!c->apply_tuned) throw ArgError("apply_kernel: not for this precision");
      c->stats.apply_variant = c->apply_cands[c->apply_pick].variant;
      c->stats.apply_grid = c->apply_cands[c->apply_pick].grid;
    }
  }
  c->d_syrk2_items = upload(c, sy2i);
  c->d_blocks = upload(c, blocks);
  c->d_colperm = upload(c, colperm);
  c->d_R = upload(c, Rall);
  c->d_f = upload(c, fall);
  c->d_c = upload(c, c->c_host);
  {
    const int D2 = std::max(c->dtot, 1);
    const int nblk = (D2 + kT - 1) / kT;
    c->d_G6 = (double*)dalloc(c, (size_t)qo * 6 * 8);
    c->d_A = (double*)dalloc(c, (size_t)D2 * D2 * 8);
    c->d_Ainv = (double*)dalloc(c, (size_t)D2 * D2 * 8);
    c->d_Linv = (double*)dalloc(c, (size_t)D2 * D2 * 8);
    c->d_Dinv = (double*)dalloc(c, (size_t)nblk * kT * kT * 8);
    c->d_Tp = (double*)dalloc(c, (size_t)D2 * kT * 8);
    c->d_Tb = (double*)dalloc(c, (size_t)D2 * kT * 8);
    c->d_vec = (double*)dalloc(c, (size_t)std::max(c->nlam, 1) * 12 * 8);
    c->d_cv = (double*)dalloc(c, (size_t)D2 * 7 * 8);
    c->d_sc = (double*)dalloc(c, 16 * 8);
    c->d_part = (double*)dalloc(c, 2 * kPcgMaxBlocks * 8);
    CK(cudaMallocHost((void**)&c->h_sc, 16 * 8));
    c->d_ctrl = (PcgCtrl*)dalloc(c, sizeof(PcgCtrl));
    CK(cudaMallocHost((void**)&c->h_ctrl, 2 * sizeof(PcgCtrl)));
    launch_build_G(D, c->d_colsub, qo, c->d_R, c->d_G6, c->st);
    CK(cudaGetLastError());
    size_t sm = implicit_smem(c->nmax, c->impl_maxf, c->impl_wide);
    if (sm > 227 * 1024) throw ArgError("subdomain too large for the shared-memory implicit solve");
    c->impl_smem = sm;
    c->grid_impl =
        c->impl_wide ? std::min(ns, c->impl_cluster > 1 ? implicit_clusters(sm, c->impl_cluster) : c->nsm)
                     : std::min(ns, c->nsm * implicit_occupancy(sm));
    c->ustride = std::max<int64_t>((max_usize + 31) / 32 * 32, 32);
    c->d_uws = (double*)dalloc(c, (size_t)c->grid_impl * c->ustride * 8);
  }
  CK(cudaMemsetAsync(c->d_status, 0, sizeof(int), c->st));
  CK(cudaMemsetAsync(c->d_tpart, 0, (size_t)std::max<int64_t>(tpo, 1) * 8, c->st));
  c->stats.workspace_bytes = ws_doubles * 8;
  c->stats.implicit_cluster = c->impl_wide ? c->impl_cluster : -1;
  for (auto& e : c->ev) CK(cudaEventCreate(&e));
  CK(cudaStreamSynchronize(c->st));
  c->stats.device_bytes = (int64_t)c->device_bytes;
}

}  // namespace

#define API_BEGIN try {
#define API_END                                                           \
  }                                                                       \
  catch (ArgError & e) {                                                  \
    return set_error(ctx, FETI_ERR_ARG, e.what());                        \
  }                                                                       \
  catch (CudaError & e) {                                                 \
    return set_error(ctx, FETI_ERR_CUDA, e.what());                       \
  }                                                                       \
  catch (std::bad_alloc&) {                                               \
    return set_error(ctx, FETI_ERR_ALLOC, "device or host allocation failed"); \
  }                                                                       \
  catch (std::exception & e) {                                            \
    return set_error(ctx, FETI_ERR_ARG, e.what());                        \
  }

extern "C" {

const char* feti_version(void) { return "feti-gb300 0.1 (sm_103a)"; }

feti_status feti_create(const feti_problem* prob, const feti_options* opt, feti_ctx** out) {
  if (!prob || !out || prob->nsub <= 0 || !prob->sub || prob->n_lambda < 0) return FETI_ERR_ARG;
  *out = nullptr;
  feti_ctx* ctx = new feti_ctx();
  API_BEGIN
  if (opt) ctx->opt = *opt;
  else {
    ctx->opt.prec = FETI_PREC_FP64;
    ctx->opt.tol = 1e-10;
    ctx->opt.maxit = 1000;
    ctx->opt.use_coords = 1;
  }
  if (ctx->opt.prec < FETI_PREC_FP64 || ctx->opt.prec > FETI_PREC_SPLIT_BF16) throw ArgError("bad precision");
  if (ctx->opt.precond < 0 || ctx->opt.precond > 2)
    throw ArgError("bad preconditioner (0 none, 1 lumped, 2 Dirichlet)");
  if (ctx->opt.assembly_route < 0 || ctx->opt.assembly_route > 3)
    throw ArgError("bad assembly route (0 SYRK path, 1 Schur complement, 2 TRSM path, 3 autotuned 0 / 2)");
  ctx->st = (cudaStream_t)ctx->opt.stream;
  ctx->fp32 = ctx->opt.prec != FETI_PREC_FP64;
  ctx->nsub = prob->nsub;
  ctx->nlam = prob->n_lambda;
  if (prob->n_lambda > 0 && !prob->c) throw ArgError("c missing");
  ctx->c_host.assign(prob->c ? prob->c : nullptr, prob->c ? prob->c + prob->n_lambda : nullptr);
  ctx->subs.resize(prob->nsub);
  for (int i = 0; i < prob->nsub; ++i) copy_sub(prob->sub[i], ctx->subs[i], i);
  build(ctx);
  *out = ctx;
  return FETI_OK;
  }
  catch (ArgError& e) {
    set_error(ctx, FETI_ERR_ARG, e.what());
  }
  catch (CudaError& e) {
    set_error(ctx, FETI_ERR_CUDA, e.what());
  }
  catch (std::bad_alloc&) {
    set_error(ctx, FETI_ERR_ALLOC, "device or host allocation failed");
  }
  catch (std::exception& e) {
    set_error(ctx, FETI_ERR_ARG, e.what());
  }
  *out = ctx;  // keep the context so feti_last_error can report; caller destroys it
  return ctx->sticky;
}

feti_status feti_update_values(feti_ctx* ctx, int32_t sub, const double* K_val) {
  feti_status g = guard(ctx);
  if (g != FETI_OK) return g;
  API_BEGIN
  if (sub < 0 || sub >= ctx->nsub || !K_val) throw ArgError("feti_update_values: bad subdomain or values");
  // through a ring of pinned slots: one host copy, and no wait for the stream unless the ring is full (a time step
  // updates every subdomain in turn; a copy from pageable memory and a synchronisation each took 40 us a subdomain)
  const size_t n = ctx->subs[sub].col.size();
  if (!ctx->h_kslots) {
    for (auto& e : ctx->kslot_ev)
      if (!e) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    size_t most = 1;
    for (auto& s : ctx->subs) most = std::max(most, s.col.size());
    if (cudaMallocHost((void**)&ctx->h_kslots, most * 8 * feti_ctx::kSlots) != cudaSuccess) {
      // no pinned memory left: copied from the caller's array, which must not change until the copy is done
      (void)cudaGetLastError();
      ctx->h_kslots = nullptr;
      CK(cudaMemcpyAsync(ctx->d_Kval + ctx->info[sub].Kval, K_val, n * 8, cudaMemcpyHostToDevice, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
      ctx->assembled = false;
      return FETI_OK;
    }
    ctx->kslot_len = most;
  }
  const int slot = (int)(ctx->kslot_next++ % feti_ctx::kSlots);
  double* h = ctx->h_kslots + (size_t)slot * ctx->kslot_len;
  CK(cudaEventSynchronize(ctx->kslot_ev[slot]));
  std::memcpy(h, K_val, n * 8);
  CK(cudaMemcpyAsync(ctx->d_Kval + ctx->info[sub].Kval, h, n * 8, cudaMemcpyHostToDevice, ctx->st));
  CK(cudaEventRecord(ctx->kslot_ev[slot], ctx->st));
  ctx->assembled = false;
  return FETI_OK;
  API_END
}

feti_status feti_assemble(feti_ctx* ctx) {
  feti_status g = guard(ctx);
  if (g != FETI_OK) return g;
  API_BEGIN
  cudaStream_t st = ctx->st;
  if ((ctx->nsyrk2 > 0 && !ctx->d_syrk2_items) || (ctx->nsyrk > 0 && !ctx->d_syrk_items) || !ctx->d_tdesc ||
      !ctx->d_blocks || ctx->apply_cands.empty())
    throw CudaError("internal: a work list of the assembly or apply is missing");
  if (!ctx->d_X)  // released after the previous assembly (recompute_X)
    ctx->d_X = dalloc(ctx, (size_t)std::max<int64_t>(ctx->stats.X_elems, 1) * (ctx->fp32 ? 4 : 8));
  const bool split = ctx->fp32 && ctx->opt.prec == FETI_PREC_SPLIT_BF16;
  if (ctx->fp32 && !ctx->d_X2)  // the bf16 hi/lo copy of X (GEMM operand of the large fronts; split-bf16 SYRK)
    ctx->d_X2 = (uint16_t*)dalloc(ctx, (size_t)std::max<int64_t>(ctx->stats.X_elems, 1) * 4);
  // mixed precision: the TRSM panel updates run on the tensor cores in split-bf16 in both mixed modes
  // (about 16 operand bits, FP32 accumulation), so that X_i is FP32-accurate and the TF32 mode's extra
  // error is that of its SYRK alone; in the TF32 mode X_i is rounded to TF32 for that SYRK
  const int tcmode = ctx->fp32 ? 2 : 0;
  const int tf32_out = ctx->fp32 && ctx->opt.prec == FETI_PREC_TF32 ? 1 : 0;
  // FP64: the forward solve of the large fronts by exact slicing on the tensor cores (not on the TRSM path)
  const bool path2 = ctx->opt.assembly_route == 2 || (ctx->opt.assembly_route == 3 && ctx->route_tuned && ctx->route == 2);
  const bool tx = !ctx->fp32 && !path2 && reserve_trsm_oz(ctx);
  ctx->stats.trsm_grid = ctx->fp32 ? ctx->grid_trsm32 : ctx->grid_trsm;
  auto run_trsm = [&](const feti_ctx::TrsmCand& tc, cudaStream_t s2) {
    CK(cudaMemsetAsync(ctx->d_queue + 16, 0, sizeof(int), s2));
    launch_trsm(ctx->P, tc.d_items, tc.nitems, tc.cw, ctx->d_queue + 16, ctx->d_X, ctx->fp32, ctx->d_ws,
                ctx->ws_stride, ctx->rhs_front, std::min(ctx->fp32 ? ctx->grid_trsm32 : ctx->grid_trsm, tc.nitems),
                tcmode, tf32_out,
                ctx->d_status, s2, 0, ctx->d_X2, ctx->d_L32, split ? 1 : 0, tx ? ctx->d_th : nullptr);
  };
  // FP64: the SYRK by exact slicing on the tensor cores
  const bool oz = !ctx->fp32 && !path2 && ctx->stats.syrk_flops > 0 && reserve_syrk_oz(ctx);
  // the numeric phase as one sequence of launches (recorded once into a CUDA graph, see below); r2: the
  // TRSM-path route (F_i = B_i P^T L^{-T} X_i in host-driven batches, not captured)
  auto enqueue = [&](cudaStream_t s2, unsigned evf, bool r2) {
    CK(cudaMemsetAsync(ctx->d_queue, 0, 64 * sizeof(int), s2));
    CK(cudaMemsetAsync(ctx->d_status, 0, sizeof(int), s2));
    if (ctx->precond_kind == 1)
      // the lumped preconditioner's values from the current K (they change with feti_update_values)
      launch_lumped_values(ctx->m_nnz, ctx->d_mc_off, ctx->d_mc_kidx, ctx->d_mc_sign, ctx->d_Kval, ctx->d_m_val,
                           s2);
    auto run_chol = [&](int v, const DevPlan& P, int qslot, int flags, bool mark = false) {
      CK(cudaMemsetAsync(ctx->d_queue + qslot, 0, sizeof(int), s2));
      if (v) CK(cudaMemsetAsync(ctx->d_tdone, 0, (size_t)std::max(ctx->ntask_total, 1) * sizeof(int), s2));
      const int fl = flags | (ctx->n_tc_items > 0 ? kCholSkipBig : 0);
      launch_chol(P, ctx->d_chol_items[v], ctx->chol_nitems[v], v, ctx->d_queue + qslot, ctx->d_tdone, ctx->d_hand,
                  ctx->d_ws, ctx->sub_stride, ctx->sub_stack,
                  std::min(ctx->grid_chol, ctx->chol_nitems[v]), ctx->d_status, s2, fl);
      if (ctx->n_tc_items > 0) {
        // the large fronts on the tensor cores, after everything below them
        if (mark) CK(cudaEventRecordWithFlags(ctx->ev[7], s2, evf));
        CK(cudaMemsetAsync(ctx->d_queue + qslot + 1, 0, sizeof(int), s2));
        CK(cudaMemsetAsync(ctx->d_tdone, 0, (size_t)std::max(ctx->ntask_total, 1) * sizeof(int), s2));
        launch_chol_tc(P, ctx->d_tc_items, ctx->n_tc_items, ctx->d_queue + qslot + 1, ctx->d_tdone, ctx->d_hand,
                       ctx->d_ws, ctx->ws_stride, ctx->d_slices, ctx->slice_stride, ctx->grid_tc,
                       ctx->tc_cluster, ctx->d_status, s2, flags);
      }
    };
    if (!ctx->chol_tuned) {
      // autotuner: whole subdomains per CTA against the subtree tasks (the same factor bitwise), faster kept
      float ms[2] = {0, 0};
      run_chol(0, ctx->P, 0, 0);  // untimed: module loading and first-touch costs stay out of the comparison
      for (int v = 0; v < 2; ++v) {
        CK(cudaEventRecord(ctx->ev[5], s2));
        run_chol(v, ctx->P, 0, 0);
        CK(cudaEventRecord(ctx->ev[6], s2));
        CK(cudaEventSynchronize(ctx->ev[6]));
        CK(cudaEventElapsedTime(&ms[v], ctx->ev[5], ctx->ev[6]));
      }
      ctx->chol_pick = ms[1] < ms[0] ? 1 : 0;
      ctx->chol_tuned = true;
    }
    ctx->stats.chol_tasks = ctx->chol_pick ? ctx->chol_nitems[1] : ctx->chol_nitems[0];
    CK(cudaEventRecordWithFlags(ctx->ev[0], s2, evf));
    run_chol(ctx->chol_pick, ctx->P, 0, 0, true);
    CK(cudaEventRecordWithFlags(ctx->ev[1], s2, evf));
    if (r2) {
      launch_unit_scale(ctx->P, ctx->nsub, ctx->nmax, ctx->P.dinv, s2);
      if (ctx->impl_wide) launch_inv_blocks(ctx->P, ctx->nsub, s2);
      CK(cudaEventRecordWithFlags(ctx->ev[2], s2, evf));
      trsm_path_entry(ctx);
      CK(cudaEventRecordWithFlags(ctx->ev[3], s2, evf));
      return;
    }
    if (ctx->fp32) {
      // the mixed TRSM reads an FP32 copy of the factor, and its large fronts a row-major bf16 hi/lo copy
      launch_l32(ctx->P.L, ctx->d_L32, ctx->stats.L_doubles, ctx->nsm * 8, s2);
      launch_l16(ctx->P, ctx->d_l16_items, ctx->n_l16, ctx->d_L32, ctx->P.LH, ctx->P.DI, ctx->nsm * 6, s2);
    }
    if (!ctx->trsm_tuned) {
      // autotuner: time every work split of the TRSM on this problem (X is the same bitwise for all)
      for (auto& tc : ctx->trsm_cands) {
        CK(cudaEventRecord(ctx->ev[5], s2));
        run_trsm(tc, s2);
        CK(cudaEventRecord(ctx->ev[6], s2));
        CK(cudaEventSynchronize(ctx->ev[6]));
        float ms = 0;
        CK(cudaEventElapsedTime(&ms, ctx->ev[5], ctx->ev[6]));
        tc.ms = ms;
      }
      ctx->trsm_pick = 0;
      for (size_t k = 1; k < ctx->trsm_cands.size(); ++k)
        if (ctx->trsm_cands[k].ms < ctx->trsm_cands[ctx->trsm_pick].ms) ctx->trsm_pick = (int)k;
      ctx->trsm_tuned = true;
      ctx->stats.trsm_cols = ctx->trsm_cands[ctx->trsm_pick].cw;
      CK(cudaEventRecord(ctx->ev[1], s2));
    }
    run_trsm(ctx->trsm_cands[ctx->trsm_pick], s2);
    for (size_t k = 0; tx && k < ctx->tx_batches.size(); ++k) {
      const auto& b = ctx->tx_batches[k];
      if (b.nitems == 0) continue;
      char* LD = (char*)ctx->d_LD - b.ld0;  // the subdomains' offsets count from the first subdomain's
      launch_dig_l(ctx->P, ctx->d_tx_ditems + b.ditem0, b.nditems, LD, s2);
      CK(cudaMemsetAsync(ctx->d_queue + 17, 0, sizeof(int), s2));
      launch_trsm_oz(ctx->P, ctx->d_tx_items + b.item0, b.nitems, ctx->tx_cw, ctx->d_queue + 17, LD, ctx->d_th,
                     (double*)ctx->d_X, ctx->d_txws, std::max<int64_t>(ctx->tx_stack, 8) * ctx->tx_cw, ctx->d_txscr, trsm_oz_scratch(ctx->tx_cw), ctx->tx_grid,
                     ctx->d_status, s2);
    }
    // the implicit solves take L in unit-lower form; the TRSM above was its last user as L
    launch_unit_scale(ctx->P, ctx->nsub, ctx->nmax, ctx->P.dinv, s2);
    if (ctx->impl_wide) launch_inv_blocks(ctx->P, ctx->nsub, s2);
    CK(cudaEventRecordWithFlags(ctx->ev[2], s2, evf));
    if (ctx->fp32) {
      auto run_syrk = [&](int variant) {
        launch_syrk_tc(ctx->P, ctx->d_syrk2_items, ctx->nsyrk2, (const float*)ctx->d_X, ctx->d_X2, (float*)ctx->d_F,
                       std::max(1, std::min(ctx->nsyrk2, ctx->nsm * (split && variant != 2 ? 1 : 2))), split ? 1 : 0,
                       ctx->d_status, s2, variant);
      };
      if (split && !ctx->syrk_tuned) {
        // autotuner: the three split-bf16 SYRK kernels on this problem (the same F bitwise), the fastest kept
        float ms[3] = {0, 0, 0};
        for (int v = 0; v < 3; ++v) {
          CK(cudaEventRecord(ctx->ev[5], s2));
          run_syrk(v);
          CK(cudaEventRecord(ctx->ev[6], s2));
          CK(cudaEventSynchronize(ctx->ev[6]));
          CK(cudaEventElapsedTime(&ms[v], ctx->ev[5], ctx->ev[6]));
        }
        ctx->syrk_variant = 0;
        for (int v = 1; v < 3; ++v)
          if (ms[v] < ms[ctx->syrk_variant]) ctx->syrk_variant = v;
        ctx->syrk_tuned = true;
        ctx->stats.syrk_variant = ctx->syrk_variant;
        CK(cudaEventRecord(ctx->ev[2], s2));
      }
      run_syrk(ctx->syrk_variant);
      ctx->stats.syrk_variant = ctx->syrk_variant;
    } else {
      if (oz)
        for (const auto& b : ctx->oz_batches)
          launch_syrk_oz(ctx->P, (const double*)ctx->d_X, b, ctx->d_oz_ditems, ctx->d_oz_items, ctx->d_XD,
                         ctx->d_oz_ex, (double*)ctx->d_F, ctx->nsm, ctx->d_status, s2);
      else
        launch_syrk_f64(ctx->P, ctx->d_syrk_items, ctx->nsyrk, (const double*)ctx->d_X, (double*)ctx->d_F,
                      std::min(ctx->nsyrk, ctx->nsm * 8), s2);
    }
    if (ctx->precond_kind == 2) {
      // Dirichlet preconditioner: K (no penalty) eliminated up to the root front, which then holds S_i
      run_chol(ctx->chol_pick, ctx->P2, 8, kCholNoReg | kCholStopRoot);
      launch_schur_tiles(ctx->P2, ctx->d_tdesc, ctx->napply, ctx->fp32, ctx->d_M,
                         std::max(1, std::min(ctx->napply, ctx->nsm * 8)), s2);
    }
    CK(cudaEventRecordWithFlags(ctx->ev[3], s2, evf));
  };
  // Cholesky, pruned TRSM, unit-lower scaling, SYRK (+ lumped values, or the Dirichlet factorisation and tiles)
  ctx->stats.launches += 4 + (ctx->precond_kind == 1 ? 1 : ctx->precond_kind == 2 ? 2 : 0);
  if (tx)
    for (const auto& b : ctx->tx_batches) ctx->stats.launches += b.nitems > 0 ? 2 : 0;
  if (oz) ctx->stats.launches += 3 * (int64_t)ctx->oz_batches.size() - 1;
  const int want = ctx->opt.assembly_route;
  if (path2) {
    ctx->route = 2;
    if (!ctx->trsm_tuned) {  // the unit-lower TRSM of this route takes whole subdomains
      ctx->trsm_pick = 0;
      ctx->trsm_tuned = true;
      ctx->stats.trsm_cols = ctx->trsm_cands[0].cw;
    }
    enqueue(st, cudaEventRecordDefault, true);
    CK(cudaGetLastError());
  } else if (ctx->asm_exec && ctx->asm_X == ctx->d_X && ctx->asm_X2 == ctx->d_X2 && ctx->asm_XD == ctx->d_XD &&
             ctx->asm_LD == ctx->d_LD && ctx->asm_th == ctx->d_th) {
    CK(cudaGraphLaunch(ctx->asm_exec, st));
  } else {
    ctx->route = want == 1 ? 1 : 0;
    enqueue(st, cudaEventRecordDefault, false);
    CK(cudaGetLastError());
    if (want == 3 && !ctx->route_tuned) {
      // autotuner between the SYRK path and the TRSM path (Sec. IV, Table I): time the TRSM and SYRK of the
      // call above against the TRSM path on the same factor; the faster one assembles from now on (the
      // TRSM path ran last, so when it wins the F tiles are already its own)
      float a1 = 0, a2 = 0;
      CK(cudaEventSynchronize(ctx->ev[3]));
      CK(cudaEventElapsedTime(&a1, ctx->ev[1], ctx->ev[3]));
      CK(cudaEventRecord(ctx->ev[5], st));
      trsm_path_entry(ctx);
      CK(cudaEventRecord(ctx->ev[6], st));
      CK(cudaEventSynchronize(ctx->ev[6]));
      CK(cudaEventElapsedTime(&a2, ctx->ev[5], ctx->ev[6]));
      ctx->route_ms[0] = a1;
      ctx->route_ms[2] = a2;
      ctx->route_tuned = true;
      if (a2 < a1) {
        ctx->route = 2;
      } else {
        // the SYRK path keeps its F: run it once more (the TRSM path overwrote the tiles)
        enqueue(st, cudaEventRecordDefault, false);
        CK(cudaGetLastError());
      }
    }
    if (ctx->trsm_tuned && ctx->route != 2) {
      // later assemblies replay the same launches from a CUDA graph, captured on a private stream (the
      // events become record nodes, so the phase times stay measured); a new X buffer needs a new graph
      if (ctx->asm_exec) CK(cudaGraphExecDestroy(ctx->asm_exec));
      ctx->asm_exec = nullptr;
      if (!ctx->cap_st) CK(cudaStreamCreateWithFlags(&ctx->cap_st, cudaStreamNonBlocking));
      cudaGraph_t gr = nullptr;
      CK(cudaStreamBeginCapture(ctx->cap_st, cudaStreamCaptureModeThreadLocal));
      enqueue(ctx->cap_st, cudaEventRecordExternal, false);
      CK(cudaStreamEndCapture(ctx->cap_st, &gr));
      cudaError_t e = cudaGraphInstantiate(&ctx->asm_exec, gr, 0);
      cudaGraphDestroy(gr);
      if (e != cudaSuccess) throw CudaError(std::string("assembly graph: ") + cudaGetErrorString(e));
      ctx->asm_X = ctx->d_X;
      ctx->asm_X2 = ctx->d_X2;
      ctx->asm_XD = ctx->d_XD;
      ctx->asm_LD = ctx->d_LD;
      ctx->asm_th = ctx->d_th;
    }
  }
  if (!ctx->fp32) {
    launch_tile_scales(ctx->P, ctx->nsub, ctx->m_max, (const double*)ctx->d_F, ctx->d_fscale, st);
    if (ctx->precond_kind == 2)
      launch_tile_scales(ctx->P, ctx->nsub, ctx->m_max, (const double*)ctx->d_M, ctx->d_mscale, st);
    ctx->stats.launches += ctx->precond_kind == 2 ? 2 : 1;
  }
  CK(cudaGetLastError());
  ctx->stats.assembly_route = ctx->route;
  ctx->stats.digit_kernels = ctx->route == 2 ? 0 : (oz ? 1 : 0) | (tx ? 2 : 0);
  for (int k = 0; k < 3; ++k) ctx->stats.route_ms[k] = ctx->route_ms[k];
  if (!ctx->coarse_ready) {
    // G = B R does not depend on the values of K: the coarse problem is set up once
    coarse_setup_entry(ctx);
    CK(cudaGetLastError());
  }
  CK(cudaEventRecord(ctx->ev[4], st));
  CK(cudaStreamSynchronize(st));
  if (ctx->opt.recompute_X) {
    // X_i is an intermediate of the assembly: with recompute_X its memory goes back to the allocator
    dfree(ctx, ctx->d_X);
    ctx->d_X = nullptr;
    dfree(ctx, ctx->d_X2);
    ctx->d_X2 = nullptr;
  }
  if (ctx->opt.recompute_X || ctx->route == 2) {  // (the TRSM path has no use for the digits its rival was timed with)
    dfree(ctx, ctx->d_XD);
    ctx->d_XD = nullptr;
    dfree(ctx, ctx->d_LD);
    ctx->d_LD = nullptr;
    dfree(ctx, ctx->d_th);
    ctx->d_th = nullptr;
  }
  float a, b, cc, d;
  CK(cudaEventElapsedTime(&a, ctx->ev[0], ctx->ev[1]));
  CK(cudaEventElapsedTime(&b, ctx->ev[1], ctx->ev[2]));
  CK(cudaEventElapsedTime(&cc, ctx->ev[2], ctx->ev[3]));
  CK(cudaEventElapsedTime(&d, ctx->ev[0], ctx->ev[4]));
  ctx->stats.t_chol_ms = a;
  ctx->stats.t_chol_tc_ms = 0;
  if (ctx->n_tc_items > 0 && ctx->route != 2) {
    float tcm = 0;
    CK(cudaEventElapsedTime(&tcm, ctx->ev[7], ctx->ev[1]));
    ctx->stats.t_chol_tc_ms = tcm;
  }
  ctx->stats.t_trsm_ms = b;
  ctx->stats.t_syrk_ms = cc;
  float e34;
  CK(cudaEventElapsedTime(&e34, ctx->ev[3], ctx->ev[4]));
  if (!ctx->coarse_ready) ctx->stats.t_coarse_ms = e34;
  ctx->coarse_ready = true;
  ctx->stats.t_assemble_ms = d;
  if (!ctx->apply_tuned) {
    // autotuner: time every variant of the apply tile kernel on this problem, keep the fastest
    double* pz = ctx->d_vec + (size_t)5 * ctx->nlam;
    double* qz = ctx->d_vec + (size_t)6 * ctx->nlam;
    CK(cudaMemsetAsync(pz, 0, (size_t)ctx->nlam * 8, st));
    for (size_t k = 0; k < ctx->apply_cands.size(); ++k) {
      auto& c2 = ctx->apply_cands[k];
      for (int rep = 0; rep < 7; ++rep) {
        if (rep == 2) CK(cudaEventRecord(ctx->ev[5], st));
        launch_apply(ctx->P, ctx->fp32, ctx->d_tdesc, ctx->napply, ctx->d_F, ctx->P.qmap, ctx->ncols, pz,
                     ctx->d_pg, ctx->d_rowpart, ctx->d_tpart, ctx->d_blocks, ctx->nblocks, ctx->d_qi, ctx->d_c0,
                     ctx->d_c1, ctx->nlam, qz, c2.grid, c2.variant, ctx->d_fscale, ctx->d_status, st);
      }
      CK(cudaEventRecord(ctx->ev[6], st));
      CK(cudaEventSynchronize(ctx->ev[6]));
      float ms = 0;
      CK(cudaEventElapsedTime(&ms, ctx->ev[5], ctx->ev[6]));
      c2.ms = ms / 5;
    }
    ctx->apply_pick = 0;
    for (size_t k = 1; k < ctx->apply_cands.size(); ++k)
      if (ctx->apply_cands[k].ms < ctx->apply_cands[ctx->apply_pick].ms) ctx->apply_pick = (int)k;
    ctx->apply_tuned = true;
    ctx->stats.apply_variant = ctx->apply_cands[ctx->apply_pick].variant;
    ctx->stats.apply_grid = ctx->apply_cands[ctx->apply_pick].grid;
  }
  int status = 0;
  CK(cudaMemcpy(&status, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  if (status & kStatNotSPD) return set_error(ctx, FETI_ERR_NOT_SPD, "a Cholesky pivot was not positive");
  if (status & kStatTimeout) return set_error(ctx, FETI_ERR_TIMEOUT, "a bounded device wait gave up");
  ctx->assembled = true;
  return FETI_OK;
  API_END
}

feti_status feti_apply(feti_ctx* ctx, const double* p_dev, double* q_dev) {
  feti_status g = guard(ctx);
  if (g != FETI_OK) return g;
  if (!ctx->assembled) return set_error(ctx, FETI_ERR_STATE, "feti_apply before feti_assemble");
  API_BEGIN
  cudaStream_t st = ctx->st;
  const auto& cand = ctx->apply_cands[ctx->apply_pick];
  int grid = cand.grid;
  feti_ctx::EvPair ev{};
  if (ctx->prof) {
    ev = {ctx->take_event(), ctx->take_event(), ctx->take_event(), ctx->take_event(), 0};
    CK(cudaEventRecord(ev.a, st));
  }
  launch_apply(ctx->P, ctx->fp32, ctx->d_tdesc, ctx->napply, ctx->d_F, ctx->P.qmap, ctx->ncols, p_dev, ctx->d_pg,
               ctx->d_rowpart, ctx->d_tpart, ctx->d_blocks, ctx->nblocks, ctx->d_qi, ctx->d_c0, ctx->d_c1, ctx->nlam,
               q_dev, grid, cand.variant, ctx->d_fscale, ctx->d_status, st, ev.b, ev.c);
  ctx->stats.launches += 3;
  ctx->stats.apply_calls += 1;
  if (ctx->prof) {
    CK(cudaEventRecord(ev.d, st));
    ctx->ev_pending.push_back(ev);
  }
  CK(cudaGetLastError());
  return FETI_OK;
  API_END
}

feti_status feti_get_F(feti_ctx* ctx, int32_t sub, double* out_host) {
  feti_status g = guard(ctx);
  if (g != FETI_OK) return g;
  if (!ctx->assembled) return set_error(ctx, FETI_ERR_STATE, "feti_get_F before feti_assemble");
  API_BEGIN
  if (sub < 0 || sub >= ctx->nsub || !out_host) throw ArgError("feti_get_F: bad arguments");
  const SubInfo& I = ctx->info[sub];
  size_t bytes = (size_t)I.m * I.m * 8;
  double* tmp = nullptr;
  CK(cudaMallocAsync((void**)&tmp, std::max<size_t>(bytes, 8), ctx->st));
  size_t esz = ctx->fp32 ? 4 : 8;
  const char* Fsub = (const char*)ctx->d_F + I.F * esz;
  launch_unpack_F(Fsub, ctx->fp32, I.m, I.nb, I.vr, ctx->d_colperm + ctx->colperm_ofs[sub], tmp, ctx->st);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(out_host, tmp, bytes, cudaMemcpyDeviceToHost, ctx->st));
  CK(cudaFreeAsync(tmp, ctx->st));
  CK(cudaStreamSynchronize(ctx->st));
  return FETI_OK;
  API_END
}

feti_status feti_set_profiling(feti_ctx* ctx, int32_t enable) {
  if (!ctx) return FETI_ERR_ARG;
  cudaStreamSynchronize(ctx->st);
  for (auto& e : ctx->ev_pending) {
    for (cudaEvent_t x : {e.a, e.b, e.c, e.d})
      if (x) ctx->ev_pool.push_back(x);
  }
  ctx->ev_pending.clear();
  ctx->prof = enable != 0;
  ctx->stats.launches = 0;
  ctx->stats.apply_calls = 0;
  ctx->stats.apply_ms = 0;
  ctx->stats.apply_tiles_ms = 0;
  ctx->stats.implicit_calls = 0;
  ctx->stats.implicit_ms = 0;
  return FETI_OK;
}

feti_status feti_get_stats(feti_ctx* ctx, feti_stats* out) {
  if (!ctx || !out) return FETI_ERR_ARG;
  if (!ctx->ev_pending.empty()) {
    if (cudaStreamSynchronize(ctx->st) != cudaSuccess) return set_error(ctx, FETI_ERR_CUDA, "stream sync failed");
    for (auto& e : ctx->ev_pending) {
      float t = 0;
      if (e.kind == 0) {
        cudaEventElapsedTime(&t, e.a, e.d);
        ctx->stats.apply_ms += t;
        cudaEventElapsedTime(&t, e.b, e.c);
        ctx->stats.apply_tiles_ms += t;
      } else {
        cudaEventElapsedTime(&t, e.a, e.b);
        ctx->stats.implicit_ms += t;
      }
      for (cudaEvent_t x : {e.a, e.b, e.c, e.d})
        if (x) ctx->ev_pool.push_back(x);
    }
    ctx->ev_pending.clear();
  }
  *out = ctx->stats;
  return FETI_OK;
}

const char* feti_last_error(feti_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

void feti_destroy(feti_ctx* ctx) {
  if (!ctx) return;
  if (ctx->st || true) cudaStreamSynchronize(ctx->st);
  for (auto& e : ctx->ev)
    if (e) cudaEventDestroy(e);
  for (auto& e : ctx->ev_pending)
    for (cudaEvent_t x : {e.a, e.b, e.c, e.d})
      if (x) cudaEventDestroy(x);
  for (auto& e : ctx->ev_pool) cudaEventDestroy(e);
  if (ctx->h_sc) cudaFreeHost(ctx->h_sc);
  if (ctx->h_ctrl) cudaFreeHost(ctx->h_ctrl);
  if (ctx->h_kslots) cudaFreeHost(ctx->h_kslots);
  for (auto e : ctx->kslot_ev)
    if (e) cudaEventDestroy(e);
  if (ctx->pcg_exec) cudaGraphExecDestroy(ctx->pcg_exec);
  if (ctx->asm_exec) cudaGraphExecDestroy(ctx->asm_exec);
  for (auto e : ctx->pcg_ev) cudaEventDestroy(e);
  for (auto e : ctx->ctrl_ev)
    if (e) cudaEventDestroy(e);
  if (ctx->cap_st) cudaStreamDestroy(ctx->cap_st);
  for (auto& b : ctx->bufs) {
    if (ctx->opt.dev_free) ctx->opt.dev_free(b.base, ctx->opt.alloc_ctx);
    else if (!ctx->opt.dev_alloc) cudaFree(b.p);
  }
  delete ctx;
}

feti_status feti_analyse(const feti_subdomain* sub, const feti_options* opt, double* info, int32_t* perm_out,
                         int32_t* sn_out) {
  feti_ctx* ctx = nullptr;
  if (!sub || !info) return FETI_ERR_ARG;
  try {
    SubHost h;
    copy_sub(*sub, h, 0);
    SymbolicOptions so;
    if (opt) {
      so.leaf_dofs = opt->leaf_dofs > 0 ? opt->leaf_dofs : 16;
      so.use_coords = opt->use_coords != 0;
    }
    PatternPlan P;
    std::vector<int32_t> tail;
    if (opt && opt->assembly_route == 1) {
      tail.assign(h.bdof.begin(), h.bdof.end());
      std::sort(tail.begin(), tail.end());
      tail.erase(std::unique(tail.begin(), tail.end()), tail.end());
    }
    analyse_pattern(h.n, h.rowptr.data(), h.col.data(), h.coords.empty() ? nullptr : h.coords.data(), so, P,
                    tail.empty() ? nullptr : tail.data(), (int)tail.size());
    BPlan B;
    plan_rhs(P, h.m, h.bdof.data(), B);
    int roots = 0;
    for (int s = 0; s < P.nsn; ++s) roots += P.sn_parent[s] < 0;
    double v[16] = {(double)P.n, (double)P.nsn, (double)P.max_f, (double)P.max_w, P.nnzL, P.chol_flops,
                    (double)P.Lsize, (double)B.m, (double)B.Xsize, B.trsm_flops, B.syrk_flops,
                    (double)B.tile_sn.size(), (double)P.chol_stack, (double)B.rhs_stack, (double)roots,
                    (double)P.nlast};
    std::memcpy(info, v, sizeof(v));
    if (perm_out) std::copy(P.perm.begin(), P.perm.end(), perm_out);
    if (sn_out) {
      std::copy(P.sn_c0.begin(), P.sn_c0.end(), sn_out);
      std::copy(P.sn_w.begin(), P.sn_w.end(), sn_out + P.nsn);
      std::copy(P.sn_parent.begin(), P.sn_parent.end(), sn_out + 2 * P.nsn);
      std::copy(P.sn_r.begin(), P.sn_r.end(), sn_out + 3 * P.nsn);
    }
    return FETI_OK;
  } catch (std::exception& e) {
    (void)ctx;
    return FETI_ERR_ARG;
  }
}

feti_status feti_analyse_lumped(const feti_problem* prob, int64_t* sizes, int32_t* w_off, int32_t* w_col,
                                double* w_val, int32_t* m_off, int32_t* m_col, int64_t* c_off, int64_t* c_kidx,
                                double* c_sign) {
  if (!prob || !sizes || prob->nsub <= 0 || prob->n_lambda < 0) return FETI_ERR_ARG;
  feti_ctx tmp;  // host fields only: no device memory is touched
  try {
    tmp.nsub = prob->nsub;
    tmp.nlam = prob->n_lambda;
    tmp.subs.resize(prob->nsub);
    tmp.info.resize(prob->nsub);
    int64_t kofs = 0;
    for (int i = 0; i < prob->nsub; ++i) {
      copy_sub(prob->sub[i], tmp.subs[i], i);
      for (int32_t l : tmp.subs[i].blam)
        if (l < 0 || l >= prob->n_lambda) throw ArgError("B_lambda out of range");
      tmp.info[i].Kval = kofs;
      kofs += (int64_t)tmp.subs[i].col.size();
    }
    LumpedPlan lp;
    plan_lumped(&tmp, lp);
    sizes[0] = (int64_t)lp.w_col.size();
    sizes[1] = (int64_t)lp.m_col.size();
    sizes[2] = (int64_t)lp.c_kidx.size();
    if (w_off) std::copy(lp.w_off.begin(), lp.w_off.end(), w_off);
    if (w_col) std::copy(lp.w_col.begin(), lp.w_col.end(), w_col);
    if (w_val) std::copy(lp.w_val.begin(), lp.w_val.end(), w_val);
    if (m_off) std::copy(lp.m_off.begin(), lp.m_off.end(), m_off);
    if (m_col) std::copy(lp.m_col.begin(), lp.m_col.end(), m_col);
    if (c_off) std::copy(lp.c_off.begin(), lp.c_off.end(), c_off);
    if (c_kidx) std::copy(lp.c_kidx.begin(), lp.c_kidx.end(), c_kidx);
    if (c_sign) std::copy(lp.c_sign.begin(), lp.c_sign.end(), c_sign);
    return FETI_OK;
  } catch (std::exception&) {
    return FETI_ERR_ARG;
  }
}

}  // extern "C"
