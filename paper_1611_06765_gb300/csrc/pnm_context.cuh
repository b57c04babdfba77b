// pnm_context.cuh -- the opaque pnm_ctx behind the C ABI.
#pragma once
#include <map>
#include <vector>

#include "pnm_internal.cuh"

struct MixedState;  // mixed-precision operand arenas (mixed.cu)
struct MlpState;    // learned warm start (mlp.cu)
struct PhItem;      // work item of the ph term (ph.cu)

// Kernel ids of the per-kernel profiler.
enum {
  KID_TSTATS = 0, KID_DCHI, KID_PH64, KID_PP64, KID_UPDATE, KID_FINALIZE,
  KID_PP_TC, KID_PH32, KID_TSTATS32, KID_UPDATE_MIX, KID_PACK, KID_DCHI32, KID_PH_F2, KID_PP_F2, PNM_NKERNELS
};
extern const char* const pnm_kernel_names[PNM_NKERNELS];

// Octaves of the interaction's fall above which the FP64 ladder checks its results (iterate.cu); with
// protons, whose channels lie up to three octaves below the scale of their digits and mix three Gaussians,
// errors of 2^-48 are reached at 47 octaves already.
constexpr double PP_STEEP = 60.0, PP_STEEP_PROTONS = 40.0;

struct pnm_ctx {
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<SysInfo> sys;
  DevState d{};
  std::vector<void*> owned;  // device allocations released by pnm_destroy

  // sizes
  int nsp_total = 0, nch = 0, nx = 0, nrows = 0, n_hh_pairs = 0, n_pp_pairs = 0;
  long nt = 0, nvhh = 0, nxt = 0, nxc = 0;
  long ns = 0;  // elements of the ladder layout (n_hh x n_lad over the channels with V_pppp)
  int max_npp = 0, max_nlad = 0;
  // (channel, ij) rows of the channels with V_pppp (digits of the ladder amplitudes): first those
  // the updates compute, then the others
  int2* lad_rows = nullptr;
  int n_lad_rows = 0, n_lad_rep = 0;

  // host copies of the channel metadata
  std::vector<int> h_ch_sys, h_key, h_nhh, h_npp, h_hh_off, h_pp_off, h_vpp;
  std::vector<long> h_t_off, h_vhh_off, h_x_t_off, h_x_c_off;
  std::vector<int> h_nlad;               // ladder basis size per channel (0: no V_pppp block)
  std::vector<long> h_s_off, h_vd_off;   // ladder-layout and ladder-V offsets per channel
  long nvdig = 0, ntdig = 0;             // digit words of the ladder V, room for those of the amplitudes
  std::vector<int2> h_rows;
  std::vector<int> h_x_nph, h_x_nhp, h_x_ph_off, h_x_hp_off, h_x_sys;
  std::vector<int> h_x_cls;  // spin-flip class of each cross channel (+1, 0, -1)
  std::vector<int> h_n_urow;    // per channel the rows the updates compute
  std::vector<int> h_row_mode;  // per row (h_rows): 2/1 computed by the updates, 0 a flip

  // work lists
  // pp ladder: items for the rows the updates compute, and (made on first use) for every row
  PPItem *pp_items = nullptr, *pp_items_all = nullptr;
  int n_pp_items = 0, n_pp_all = 0, nsm = 148;
  int4* upd_items = nullptr;  // (channel, ij, first pp column), 128 columns each (the learned start)
  int n_upd_items = 0;
  int *upd_lo_d = nullptr, *upd_hi_d = nullptr;  // per system ranges of these items
  UpdItem* upd_chunks = nullptr;  // of the updates: chunks of 32 amplitudes, and the amplitudes
  int* upd_z = nullptr;
  int n_upd_ctas = 0, upd_per_warp = 1;
  // ph term: work items (pnm_need_ph_items): n_ph_large + n_ph_cta channels that take a CTA, then
  // n_ph_warp of the warp path, the last n_ph_tiny (n_ph_tiny64 with FP64 results) of them tiny
  PhItem* ph_items = nullptr;
  int n_ph_items = 0, n_ph_large = 0, n_ph_cta = 0, n_ph_warp = 0, n_ph_tiny = 0, n_ph_tiny64 = 0;
  size_t ph32_smem = 0, ph32_warp_smem = 0;  // shared memory per CTA and per warp, FP32
  // the digit ph term (made on first use, pnm_need_phdig): source indices, W fragments, <kb|v|cj>
  long ph_sizes[4] = {0, 0, 0, 0};
  int2* ph_exps = nullptr;
  int* ph_src = nullptr;
  uint4* ph_wf = nullptr;
  long long* ph_v1 = nullptr;
  double* ph_fixed64 = nullptr;
  f2* ph_fixed_f2 = nullptr;  // the fixed operands of the smallest channels as element values
  size_t ph_large_smem = 0, ph_dig_smem = 0, ph_warp_smem = 0;
  f2* t_pair = nullptr;                          // FP32-pair copy of the current amplitudes
  int *grp_lo_d = nullptr, *grp_hi_d = nullptr;  // per system ranges of the update items
  int max_nhh = 1;
  int4* stat_items = nullptr;  // warps of the stats kernel
  int n_stat = 0;

  // loop control
  int *row_lo_d = nullptr, *row_hi_d = nullptr, *lut_off_d = nullptr;  // per system
  LoopCtl* ctl = nullptr;     // device
  double* small = nullptr;    // device scratch for single-value queries
  double* mbpt3_buf = nullptr;   // per-CTA partials and per-system results of pnm_mbpt3
  double* s64 = nullptr;         // the amplitudes in the ladder layout (FP64 ladders that check their results)
  double* expand_buf = nullptr;  // the pp ladder or ph term in the amplitude layout (operator calls)
  SysCtl* sysctl = nullptr;   // device, one per system
  int* blocks_done = nullptr; // device, one per system
  double* hist = nullptr;     // device, (hist_cap) per system
  int hist_cap = 0;
  int last_iters_host = 0;

  // graphs, one per precision mode
  std::map<int, cudaGraphExec_t> graphs;
  std::map<int, cudaGraph_t> graph_defs;
  // whole-solve graphs (start, iteration loop, refinement loop, settling, read-back), one per
  // solve configuration; their run-time parameters and results pass through pinned host memory
  std::map<int, cudaGraphExec_t> solve_graphs;
  std::map<int, cudaGraph_t> solve_graph_defs;
  void* h_pinned = nullptr;      // one block: h_par, h_ctl, h_sc[nsys], h_mlp_err
  SolveParams* h_par = nullptr;
  LoopCtl* h_ctl = nullptr;
  SysCtl* h_sc = nullptr;
  int* h_mlp_err = nullptr;
  SolveParams* d_par = nullptr;
  double* d_tol = nullptr;       // per-system tolerance of the energy test
  std::vector<double> tol_host;  // the values d_tol holds

  MixedState* mixed = nullptr;
  MlpState* mlp = nullptr;
  f2* vpphh_f2 = nullptr;  // FP32-pair copy of V_pphh (made on first use by the FP32-pair sweeps)
  // work list of the ladder-basis V (channel, first row, interaction table and its size) and the
  // shared memory of its kernel; the V itself is built on first use (pnm_need_vdig)
  int4* vl_items = nullptr;
  int n_vl_items = 0;
  size_t vl_smem = 0;
  double hbar2_2m = 0.0;
  double fall = 0.0;   // octaves by which a system's interaction falls over its model space, at most
  std::vector<int> h_steep;  // per system: its interaction falls by more than PP_STEEP octaves over the model space
  int mlp_fallback = 0;  // 1 when the last learned start was replaced by the MBPT2 start

  // side streams for the independent parts of an update (ph term, pp ladder), joined by events
  cudaStream_t side[2] = {nullptr, nullptr};
  cudaEvent_t ev_fork = nullptr, ev_join[2] = {nullptr, nullptr};
  bool serial_sched[3] = {false, false, false};  // per mode (0 FP64, 1 mixed, 2 FP32-pair refinement): one stream only
  bool sched_tuned[3] = {false, false, false};
  bool sched_ended[3] = {false, false, false};  // the timed updates diverged: left untuned
  int mixed_order = 0;  // of a concurrent mixed update: what waits for the t tiles of the ladder (pnm_enqueue_body_mixed)
  int cur_mode = 0;

  // per-kernel CUDA-event profiling of host-driven solves (never active during capture)
  bool prof_on = false, prof_live = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_ev;
  std::vector<int> prof_pending;  // kernel id per used event pair
  double prof_ms[PNM_NKERNELS] = {};
  int prof_n[PNM_NKERNELS] = {};

  // timings (ms)
  double t_setup = 0, t_mbpt2 = 0, t_solve = 0, t_mixed = 0, t_refine = 0, t_mbpt3 = 0;
  // host wall time (ms) of the last solve's one-time preparation: pair and FP32 copies, schedule
  // tuning, and the capture and instantiation of its graphs (t_graph_host accumulates the latter)
  double t_prepare = 0, t_graph_host = 0;
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
};

// Autotuner cache key: device and, of every system, what fixes its channels (the density only rescales
// values): neutrons, protons, n2max, and whether it is twisted.  Twists move channels about but leave
// their sizes alike, so the systems of a twist average share an entry.
inline std::string pnm_shape_key(const pnm_ctx* ctx) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::string k = "dev" + std::to_string(dev);
  for (const SysInfo& S : ctx->sys) {
    k += ";" + std::to_string(S.N - S.Z) + "," + std::to_string(S.Z) + "," + std::to_string(S.n2max);
    if (S.phi[0] != 0.0 || S.phi[1] != 0.0 || S.phi[2] != 0.0) k += "t";
  }
  return k;
}

// Device memory of contexts: stream-ordered allocations from one memory pool per device, owned
// by the library, whose freed blocks stay cached for the next context (a create/solve/destroy
// loop then maps no new memory).  pnm_pool_alloc throws PNM_ENOMEM.
void* pnm_pool_alloc(cudaStream_t s, size_t bytes);
void pnm_pool_free(cudaStream_t s, void* p);
// Raise a kernel's dynamic shared-memory limit (a property of the function, shared by every
// context of the process) to at least `bytes`; never lowers it, so a context built later with
// smaller channels cannot break the launches of an earlier one.
void pnm_smem_at_least(const void* func, size_t bytes);
template <typename F>
void smem_at_least(F* func, size_t bytes) {
  pnm_smem_at_least((const void*)func, bytes);
}
// An allocation on the context stream recorded in ctx->owned (released by pnm_destroy).
void* pnm_ctx_alloc(pnm_ctx* ctx, size_t bytes);
template <typename T>
T* ctx_alloc(pnm_ctx* ctx, size_t n) {
  return (T*)pnm_ctx_alloc(ctx, (n ? n : 1) * sizeof(T));
}
void pnm_build(pnm_ctx* ctx, int nsys, const int* Ns, const int* Zs, const double* rhos,
               const int* n2maxs, const double* thetas, const pnm_minnesota& P);
void pnm_prepare_iteration(pnm_ctx* ctx);
void pnm_eref_all(pnm_ctx* ctx);
void pnm_mbpt2_all(pnm_ctx* ctx, double* out);
int pnm_solve(pnm_ctx* ctx, const pnm_solve_opts& o, double* dE, int* iters, double* resid);
void pnm_free_mixed(pnm_ctx* ctx);
void pnm_enqueue_body(pnm_ctx* ctx, int mode, int use_cond, cudaGraphConditionalHandle h);
void pnm_enqueue_loop_body(pnm_ctx* ctx, int mode, bool refine, cudaGraphConditionalHandle h);
void pnm_prepare_terms(pnm_ctx* ctx, int terms);
void pnm_mbpt3_all(pnm_ctx* ctx, double* out);
// The pp ladder from its ladder layout (planes summed) into host memory in the amplitude layout.
void pnm_lad_expand(pnm_ctx* ctx, const float* rs, int planes, long pstride);
void pnm_lad_expand(pnm_ctx* ctx, const double* rs, int planes, long pstride);
void pnm_lad_expand(pnm_ctx* ctx, const f2* rs, int planes, long pstride);
// alpha / eps_ij^ab of the current mixed solve (the step of the mixed and refinement updates)
const double* pnm_mixed_aw(const pnm_ctx* ctx);
void pnm_enqueue_body_mixed(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h);
void pnm_prepare_mixed(pnm_ctx* ctx);
void pnm_start(pnm_ctx* ctx, int init, const std::vector<double>& tol);
int pnm_run_loop(pnm_ctx* ctx, int mode, int max_iter, int min_iter, int host_loop, double alpha,
                 int* iter_out = nullptr);
void pnm_reopen(pnm_ctx* ctx);
void pnm_settle_amplitudes(pnm_ctx* ctx);
void pnm_mlp_start(pnm_ctx* ctx);
void pnm_mlp_prepare(pnm_ctx* ctx);
void pnm_need_vdig(pnm_ctx* ctx);
void pnm_need_pp_lists(pnm_ctx* ctx);
void pnm_mlp_enqueue(pnm_ctx* ctx);
void pnm_drop_solve_graphs(pnm_ctx* ctx);
void pnm_set_node_priorities(cudaGraph_t body);
void pnm_solve_begin(pnm_ctx* ctx);
void pnm_start_device(pnm_ctx* ctx, int init);
void pnm_loop_begin(pnm_ctx* ctx, int mode);
void pnm_refine_gate(pnm_ctx* ctx, cudaGraphConditionalHandle h);
void pnm_loop_end_settle(pnm_ctx* ctx);
void pnm_flip_copy_device(pnm_ctx* ctx);
void pnm_mixed_pack_t(pnm_ctx* ctx);
void pnm_mixed_set_alpha(pnm_ctx* ctx, double alpha);
void pnm_free_mlp(pnm_ctx* ctx);
int* pnm_mlp_err(pnm_ctx* ctx);
void prof_begin(pnm_ctx* ctx, int kid);
void prof_end(pnm_ctx* ctx);
void prof_collect(pnm_ctx* ctx);
FinArgs fin_args(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h);
void pnm_enqueue_stats(pnm_ctx* ctx, bool mixed, bool pair = false);
void pnm_launch_pp(pnm_ctx* ctx, cudaStream_t s, bool rep_only, bool pair);
void launch_ph_f2(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny);
void pnm_need_phdig(pnm_ctx* ctx);
void pnm_need_digits(pnm_ctx* ctx);
void pnm_split_f2(const double* a, f2* b, long n, cudaStream_t s);
void pnm_prepare_f2(pnm_ctx* ctx);
void pnm_split_cur(pnm_ctx* ctx, cudaStream_t s);
void pnm_mixed_pack_initial(pnm_ctx* ctx, double alpha);
void pnm_fork(pnm_ctx* ctx);
void pnm_join(pnm_ctx* ctx);
void pnm_launch_mbpt2_into(const pnm_ctx* ctx, double* partials, double* results);
void pnm_apply_ph(pnm_ctx* ctx, int sys, int precision, const double* t, double* r, size_t n);
void pnm_apply_pp(pnm_ctx* ctx, int sys, int precision, const double* t, double* r, size_t n);
void launch_ph64(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny, bool linear);
void pnm_flip_symmetrise(pnm_ctx* ctx, double* t, cudaStream_t s);
void pnm_flip_copy(pnm_ctx* ctx, double* t, cudaStream_t s);
void pnm_flip_copy_current(pnm_ctx* ctx, int iter);
void launch_ph_mix(pnm_ctx* ctx, const float* xt, const float* xw, const float* xv1, float* xq, cudaStream_t s,
                   cudaStream_t s_tiny);
void pnm_ph_pack32(pnm_ctx* ctx, float* xw, float* xv1);
void pnm_need_ph_items(pnm_ctx* ctx);
bool pnm_is_ph_kernel(const void* f);
void launch_update64(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h, bool pair = false);
void launch_update_mix(pnm_ctx* ctx, const float* rpp, const float* xq, const double* aw, float* xt, int use_cond,
                       cudaGraphConditionalHandle h, int nplanes, long pstride);
void pnm_alpha_inv(pnm_ctx* ctx, double alpha, double* aw);
void pnm_mixed_tuning(const pnm_ctx* ctx, int* ksplit, int* stages, float* us, int* serial_mask);
bool pnm_concurrent(const pnm_ctx* ctx);
void pnm_tune_schedule(pnm_ctx* ctx, int mode, double alpha);
void pnm_selftest_wait(pnm_ctx* ctx);
