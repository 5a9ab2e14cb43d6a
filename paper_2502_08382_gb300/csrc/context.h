// Internal definition of feti_ctx (host runtime state).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "feti.h"
#include "common.cuh"
#include "symbolic.h"

namespace feti {

struct SubHost {
  int n = 0, m = 0, d = 0, nfix = 0, nelem = 0, edofs = 0;
  std::vector<int64_t> rowptr;
  std::vector<int32_t> col;
  std::vector<double> val;
  std::vector<int32_t> bdof, blam;
  std::vector<double> bsign;
  std::vector<double> R, f, coords;
  std::vector<int32_t> fix;
  std::vector<int32_t> elem_dofs;
  std::vector<double> dKe, dKe_scale;  // per element (dk_stride = edofs^2) or one shared matrix (0)
  int64_t dk_stride = 0;
  int pat = -1, bp = -1;
};

// a device buffer owned by the context
struct DBuf {
  void* p = nullptr;
  size_t bytes = 0;
  void* base = nullptr;  // what the allocator returned
};

}  // namespace feti

struct feti_ctx {
  feti_options opt{};
  cudaStream_t st = nullptr;
  std::string err;
  feti_status sticky = FETI_OK;
  int nsub = 0, nlam = 0, nsm = 0;
  bool fp32 = false;
  bool assembled = false;
  std::vector<double> c_host;
  std::vector<feti::SubHost> subs;
  std::vector<feti::PatternPlan> pats;
  std::vector<feti::SolveSplit> solve_splits;  // per pattern, for impl_cluster CTAs
  std::vector<feti::BPlan> bps;
  std::vector<int> bp_pat;
  std::vector<feti::SubInfo> info;
  feti::DevPlan P{};
  std::vector<feti::DBuf> bufs;
  size_t device_bytes = 0;
  // pinned staging ring of feti_update_values
  static constexpr int kSlots = 8;
  double* h_kslots = nullptr;
  size_t kslot_len = 0, kslot_next = 0;
  cudaEvent_t kslot_ev[kSlots] = {};
  // device arrays not in DevPlan
  double* d_Kval = nullptr;
  double* d_L = nullptr;
  void* d_X = nullptr;
  void* d_F = nullptr;
  double* d_ws = nullptr;
  int grid_ws = 0;            // CTAs' workspaces of ws_stride doubles
  int64_t sub_stride = 0, sub_stack = 0;  // chol_kernel's workspace per CTA (same buffer)
  int64_t ws_stride = 0, rhs_front = 0;
  double* d_trow = nullptr;
  double* d_tpart = nullptr;
  double* d_qi = nullptr;
  int* d_colsub = nullptr;
  int* d_c0 = nullptr;
  int* d_c1 = nullptr;
  int* d_queue = nullptr;     // [8] work-queue counters
  int* d_status = nullptr;    // [1]
  int* d_chol_order = nullptr;
  int* d_trsm_order = nullptr;
  struct TrsmCand {
    int cw;           // columns per work item (0: a whole subdomain)
    int2* d_items;    // (subdomain, first column), subdomains by decreasing TRSM cost
    int nitems;
    double ms;
  };
  std::vector<TrsmCand> trsm_cands;  // autotuner candidates of the pruned TRSM
  int trsm_pick = 0;
  bool trsm_tuned = false;
  int4* d_chol_items[2] = {nullptr, nullptr};  // Cholesky items: whole subdomains / subtree tasks
  int chol_nitems[2] = {0, 0};
  int chol_pick = 0;                 // the autotuner's choice of the two
  bool chol_tuned = false;
  int ntask_total = 0;
  int* d_tdone = nullptr;            // per global task: child tasks finished
  double* d_hand = nullptr;          // hand-over slots of split subtree roots
  int4* d_tc_items = nullptr;        // the large fronts' tasks (the tensor-core Cholesky's items)
  int n_tc_items = 0, grid_tc = 0, tc_cluster = 1;  // items, clusters and CTAs per cluster
  char* d_slices = nullptr;          // its per-cluster scratch (bf16 digits and row exponents)
  int64_t slice_stride = 0;
  int2* d_l16_items = nullptr;       // (subdomain, supernode) of the panels with a row-major hi/lo copy
  int n_l16 = 0;
  int syrk_variant = 0;              // split-bf16 SYRK kernel picked by the autotuner
  bool syrk_tuned = false;
  int* d_impl_order = nullptr;
  int2* d_syrk_items = nullptr;
  // FP64 forward solve of the large fronts on the tensor cores
  bool tx_planned = false, tx_none = false;  // tx_none: no items
  size_t tx_refused = 0;             // free memory when the digits of L were last refused (0: never)
  int4* d_tx_ditems = nullptr;       // 128-column blocks of the large panels to cut
  int2* d_tx_items = nullptr;        // (subdomain, first column) of the solve
  // batches of consecutive subdomains whose digits of L are cut and used in turn
  struct TxBatch {
    int sub0 = 0, sub1 = 0, ditem0 = 0, nditems = 0, item0 = 0, nitems = 0;
    int64_t ld0 = 0;
  };
  std::vector<TxBatch> tx_batches;
  size_t tx_ld_bytes = 0;
  int tx_cw = 128, tx_grid = 0;
  size_t ld_bytes = 0, th_bytes = 0;
  int64_t tx_stack = 0;  // doubles per column
  void* d_LD = nullptr;              // digits of the large panels
  double* d_th = nullptr;            // update blocks handed over
  double* d_txws = nullptr;          // fronts and stacks
  char* d_txscr = nullptr;           // digits of X per CTA
  // FP64 SYRK on the tensor cores: batches of subdomains, their tiles and X pieces, digits and column exponents
  std::vector<feti::OzBatch> oz_batches;
  int4* d_oz_items = nullptr;
  int4* d_oz_ditems = nullptr;
  void* d_XD = nullptr;
  size_t xd_bytes = 0;       // of the plan's largest batch
  size_t xd_refused = 0;     // free memory when the digits were last refused (0: never)
  int* d_oz_ex = nullptr;
  feti::TileDesc* d_tdesc = nullptr;
  int *d_fscale = nullptr, *d_mscale = nullptr;  // FP64: scales of the F tiles (and of the Dirichlet M tiles)
  struct ApplyCand {
    int variant, grid;  // tile-kernel variant (load batch) and grid
    double ms;
  };
  std::vector<ApplyCand> apply_cands;  // autotuner candidates of the apply
  int apply_pick = 0;
  bool apply_tuned = false;
  void* d_pg = nullptr;
  void* d_rowpart = nullptr;
  int2* d_syrk2_items = nullptr;
  int2* d_blocks = nullptr;
  int nblocks = 0;
  int nsyrk2 = 0;
  int* d_colperm = nullptr;   // per subdomain sorted column -> B row (for get_F)
  std::vector<int64_t> colperm_ofs;
  int nsyrk = 0, napply = 0;
  int64_t ncols = 0;
  int grid_chol = 0, grid_trsm = 0, grid_impl = 0;
  int grid_trsm32 = 0;  // CTAs of the mixed-precision TRSM (its occupancy with the tensor-core stage ring)
  size_t impl_smem = 0;
  bool impl_wide = false;   // 1024-thread CTAs,
  int impl_cluster = 0;     // this many per subdomain (0: 256-thread ones)
  double* d_uws = nullptr;  // update vectors of the implicit solve, ustride doubles per CTA
  int64_t ustride = 0;
  int impl_maxf = 0;
  // solve-side data
  bool coarse_ready = false;
  int npairs = 0;
  int4* d_pairs = nullptr;
  int2* d_plist = nullptr;
  double* d_G6 = nullptr;      // [ncols * 6] G = B R per sorted column
  double* d_A = nullptr;       // D x D coarse matrix, then its factor
  double* d_Ainv = nullptr;    // (G^T G)^{-1}
  double* d_Linv = nullptr;
  double* d_Dinv = nullptr;    // inverses of the 64 x 64 diagonal factor blocks
  double* d_Tp = nullptr;      // D x 64 panel scratch
  double* d_Tb = nullptr;      // 64 x D row-block scratch
  int4* d_lamcol = nullptr;    // per multiplier: tile bases and columns of its subdomain columns (PCPG gather)
  int4* d_lamg = nullptr;      // per multiplier: alpha0 and d of its subdomains (PCPG update)
  double* d_qcol = nullptr;    // per B column: q of its multiplier (PCPG G^T q)
  int m_max = 0;               // widest subdomain (B rows)
  // lumped preconditioner M = W M_core W (options.precond = 1), see precond.cpp
  bool precond = false;
  int precond_kind = 0;        // 0 none, 1 lumped, 2 Dirichlet
  feti::DevPlan P2{};          // Dirichlet: the plan with its own L (K factored up to the root front) and rho
  void* d_M = nullptr;         // Dirichlet: M_i = B_i S_i B_i^T tiles (layout of F)
  void* d_pg2 = nullptr;       // Dirichlet: W w gathered per sorted column (tile precision)
  int* d_w_off = nullptr;
  int* d_w_col = nullptr;
  double* d_w_val = nullptr;
  int* d_m_off = nullptr;
  int* d_m_col = nullptr;
  double* d_m_val = nullptr;
  int64_t* d_mc_off = nullptr;
  int64_t* d_mc_kidx = nullptr;
  double* d_mc_sign = nullptr;
  int64_t m_nnz = 0;
  double* d_vec = nullptr;     // PCPG vectors (12 x n_lambda)
  double* d_cv = nullptr;      // coarse vectors (7 x D)
  double* d_sc = nullptr;      // scalars
  double* d_part = nullptr;    // block partials of the PCPG reductions (2 x kPcgMaxBlocks)
  double* h_sc = nullptr;      // pinned host scalars
  feti::PcgCtrl* d_ctrl = nullptr;  // PCPG control block
  feti::PcgCtrl* h_ctrl = nullptr;  // pinned host copy
  cudaStream_t cap_st = nullptr;     // private stream on which CUDA graphs are captured
  cudaGraphExec_t asm_exec = nullptr;  // the numeric assembly (Cholesky, TRSM, scaling, SYRK), replayed on st
  void* asm_X = nullptr;             // the X buffers the assembly graph was captured with
  void* asm_X2 = nullptr;
  void* asm_XD = nullptr;
  void* asm_LD = nullptr;
  void* asm_th = nullptr;
  uint16_t* d_X2 = nullptr;          // bf16 hi/lo copy of X (split-bf16 SYRK operands)
  float* d_L32 = nullptr;            // FP32 copy of L for the mixed TRSM
  cudaGraphExec_t pcg_exec = nullptr;  // captured chunk of iterations (replayed on st)
  int pcg_chunk = 0;
  bool pcg_prof = false;             // the captured chunk records events
  cudaEvent_t ctrl_ev[2] = {nullptr, nullptr};  // control-block copies of chunks enqueued ahead
  std::vector<cudaEvent_t> pcg_ev;  // 4 events per captured iteration (apply timing)
  int* d_dofsub = nullptr;
  // adjoint (element data and dense work buffers, allocated on first use)
  std::vector<int64_t> elem_ofs, elem_dk_ofs, elem_dofs_ofs;
  int* d_ident = nullptr;
  int64_t nelem_total = 0;
  int* d_eldofs = nullptr;
  double* d_eldk = nullptr;
  double* d_elsc = nullptr;
  double* d_Xu = nullptr;          // FP64 X_u = L_u^{-1} P B^T of every subdomain (adjoint)
  double* d_adj_work = nullptr;    // batch work arrays of the adjoint (V and sorted W)
  int64_t adj_work_bytes = 0;
  std::vector<int64_t> pat_lt;     // per pattern: bytes of the large fronts' digits of L^T
  void* d_adj_lt = nullptr;        // those digits of one batch, and the backward solve's scratch
  int64_t adj_lt_bytes = 0;
  char* d_adj_bscr = nullptr;
  int4* d_adj_lit = nullptr;
  int2* d_adj_bit = nullptr;
  int64_t adj_lit_cap = 0, adj_bit_cap = 0;
  void* d_adj_dig = nullptr;       // digits of Z and W (the adjoint's Y = Z W)
  int64_t adj_dig_bytes = 0;
  feti::DenseEnt* d_adj_ent = nullptr;
  int4* d_adj_dit = nullptr;
  int* d_adj_dex = nullptr;
  int64_t adj_ent_cap = 0, adj_dit_cap = 0, adj_dex_cap = 0;
  feti::AdjBatch* d_adj_batch = nullptr;
  int64_t adj_batch_cap = 0;
  int4* d_adj_items4 = nullptr;
  int64_t adj_items4_cap = 0;
  int2* d_adj_items2 = nullptr;
  feti::TileDesc* d_tdesc_sub = nullptr;  // the apply's tile descriptors in subdomain-major order
  int* d_tile0 = nullptr;                 // first tile of each subdomain in d_tdesc_sub
  int route = 0;                          // assembly route in use (0 SYRK path, 1 Schur, 2 TRSM path)
  bool route_tuned = false;
  double route_ms[3] = {0, 0, 0};
  int64_t adj_items2_cap = 0;
  int64_t* d_woff = nullptr;       // per subdomain offset of W_i (weighted trace)
  double* d_wt_part = nullptr;     // per tile partials of the weighted trace
  int64_t ndof = 0;
  int nmax = 0;
  double* d_R = nullptr;       // concatenated R_i (column-major n x d)
  double* d_f = nullptr;       // concatenated f_i
  double* d_c = nullptr;       // c
  int dtot = 0;
  // stats and measurement
  feti_stats stats{};
  bool prof = false;
  struct EvPair {
    cudaEvent_t a, b, c, d;
    int kind;  // 0 apply (a..d whole, b..c tiles), 1 implicit (a..b)
  };
  std::vector<EvPair> ev_pending;
  std::vector<cudaEvent_t> ev_pool;
  cudaEvent_t take_event() {
    if (ev_pool.empty()) {
      cudaEvent_t e;
      cudaEventCreate(&e);
      return e;
    }
    cudaEvent_t e = ev_pool.back();
    ev_pool.pop_back();
    return e;
  }
  cudaEvent_t ev[8]{};
};

namespace feti {
feti_status set_error(feti_ctx* c, feti_status s, const std::string& msg);
void trsm_path_entry(feti_ctx* c);  // the TRSM-path assembly of the F_i tiles (api_solve.cpp)
void* dalloc(feti_ctx* c, size_t bytes);
void dfree(feti_ctx* c, void* p);  // release a buffer from dalloc (no-op for nullptr)
}  // namespace feti
