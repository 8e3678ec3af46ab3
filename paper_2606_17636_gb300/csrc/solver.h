// Batched per-mode multigrid solver on the device (host-side orchestration).
#pragma once
#include <string>
#include <vector>

#include "kernels.h"

namespace ps {

// Device memory owner with optional user allocation hooks.
struct Arena {
  void* (*alloc_fn)(size_t, void*) = nullptr;
  void (*free_fn)(void*, void*) = nullptr;
  void* user = nullptr;
  std::vector<void*> blocks;
  size_t bytes = 0;
  bool failed = false;   // a needed request was refused: whoever made it stops before its next launch
  void* get(size_t n, bool optional = false);
  void give_back(void* p);
  void release_all();
};

struct MGOptions {
  int precision = 1;   // 0 FP64, 1 mixed (FP32 V-cycles inside FP64 refinement)
  int nu1 = 2, nu2 = 2, n_sor = 2;
  int nu1f = 0, nu2f = 0;   // smoothing cycles of the fused (shared-memory) levels; 0: nu1 / nu2
  Tiles tiles;         // tile shapes of the level-wide smoothing passes
  int max_cycles = 100;
  int stagnation = 0;  // retire planes whose residual stops falling
  int coarsest_size = 1;   // coarsest-level rule (psolve_desc.coarsest_size; 1: small)
};

// Shared-memory layout of the cluster-resident tail (k_tail.cu) for levels of
// nr[l] x nt[l] cells and n_sor SOR sweeps: fills t's cluster size, rows per
// CTA, offsets and table layout; returns the bytes per CTA, or 0 when the
// plan does not allow the tail (a coarsest level without the separable form,
// cluster slabs that do not divide the levels, radial lines above 256 cells
// (or below 16 on a smoothed level),
// polar segments above 24 cells, or more than kTailSmemMax bytes).
constexpr size_t kTailSmemMax = 224 * 1024;
size_t tail_layout(const std::vector<int>& nr, const std::vector<int>& nt, int n_sor, bool separable,
                   TailArgs& t);
size_t tail_tables(const std::vector<int>& nr, const std::vector<int>& nt, TailArgs& t);

class MGSolver {
 public:
  // fine: plane geometry; modes[s]: azimuthal mode number of slot s;
  // plane_slot (size max_planes, may be empty = identity); neumann: inner
  // radial face carries a prescribed flux (zero coefficient on all levels).
  bool init(Arena& A, const PlaneGeo& fine, bool neumann, const std::vector<int>& modes,
            const std::vector<int>& plane_slot, int max_planes, const MGOptions& o,
            std::string& err);
  // What a solve can do without, asked for last (false: a CUDA call failed).
  bool optional_buffers(Arena& A, std::string& err);
  // Solve L u = f for all planes (u holds the initial guess).  Enqueued on
  // st; with cond_handle (use_cond) the loop is a graph WHILE body; in eager
  // mode the host reads the continue flag each iteration.
  void init_loop(cudaStream_t st);
  void loop_body(const double2* f, double2* u, double tol, cudaStream_t st, int use_cond,
                 unsigned long long cond, bool few);
  // A solve's phases: iterations with the level-wide passes while more than
  // few_planes planes remain (none when the batch is no larger), then
  // iterations with the window passes.
  bool many_phase() const { return few_planes < batch.max_planes; }
  bool few_phase() const { return few_planes > 0; }
  int eager_solve(const double2* f, double2* u, double tol, cudaStream_t st, std::string& err);
  // One V-cycle; with u, the refinement's update u += e rides on the last
  // smoothing pass when the schedule post-smooths level 0 with the
  // level-wide passes (returns true then; else the caller updates).
  bool vcycle(cudaStream_t st, double2* u = nullptr);
  void vcycle_few(cudaStream_t st, double2* u);
  // Change the smoothing schedule and tile shapes of later V-cycles (a
  // captured solve must be captured again).
  void set_schedule(int nu1, int nu2, int n_sor, Tiles tiles, int nu1f, int nu2f);
  // results (device arrays, per plane)
  int* d_cycles = nullptr;
  int* d_status = nullptr;
  double2* d_nf2 = nullptr;
  double2* d_nr2 = nullptr;
  int* d_iter = nullptr;
  int* d_cont = nullptr;
  // continue flags of the eager loop's iterations in flight (pinned, written by
  // the residual) and the events behind those residuals
  static constexpr int kFlags = 2;
  int* h_cont = nullptr;
  cudaEvent_t flag_at[kFlags] = {};
  void release_host();
  Hierarchy H;
  std::vector<LevelDev> lv;
  Batch batch{};
  MGOptions opt;
  int max_planes = 0;
  // level buffers (T2 of the precision): e[l], f[l]
  std::vector<void*> e, f;
  void* tmp = nullptr;             // ping-pong buffer of the global-memory smoother
  int first = 0;                   // first level the shared-memory kernel can take
  // the level from which a solve's V-cycle runs it, and its arguments there
  int base = 0;
  VSmemArgs vsb{};
  // window passes (k_tile.cu, mixed path) for the last few_planes planes of a
  // solve (0: none): per level below base the launches before and after the
  // coarse correction; e2[l] takes level l's result after it, tmp2 is a second
  // scratch buffer
  int few_planes = 0;
  std::vector<std::vector<TileStep>> t_down, t_up;
  std::vector<void*> e2;
  void* tmp2 = nullptr;
  void plan_tiles();
  int zero_guess = 0;              // the next solve starts from u = 0 (set by the caller)
  VSmemArgs vs{};
  // stage helpers on explicit buffers
  // u: the last pass adds e to u instead of storing it (see launch_smooth)
  void smooth(int level, void* e, const void* f, int cycles, bool zero_init, cudaStream_t st,
              double2* u = nullptr);
  void restrict_(int level, const void* e, const void* f, void* fc, cudaStream_t st);
  void prolong(int level, void* e, const void* ec, cudaStream_t st);
  // levels lo .. coarsest in shared memory, with v built for lo
  void fused(int lo, const VSmemArgs& v, cudaStream_t st);
  bool build_vsmem(Arena& A, int lo, int n_modes, VSmemArgs& v, std::string& err);
  // hand_over: the continue flag becomes 2 once at most that many planes remain
  void residual(const double2* f, const double2* u, double tol, cudaStream_t st, int use_cond,
                unsigned long long cond, int hand_over, int* host = nullptr);
  // the defect alone into r (tolerance 0: no plane retires)
  void residual_to(const double2* f, const double2* u, void* r, cudaStream_t st);
  int* d_act = nullptr;
  int* d_nact = nullptr;
  int* d_slot = nullptr;
  int* d_mode = nullptr;
  double* d_s2 = nullptr;
  float* d_s2f = nullptr;
  double* d_inv = nullptr;
  double* d_blk = nullptr;
  double* d_sep = nullptr;
  float* d_sepf = nullptr;
  double* d_ctab = nullptr;   // level-0 per-cell FP64 products [4][nt][nr]
  double* d_dtab = nullptr;   // level-0 diagonal of each mode slot [slots][nt][nr]
  SqPart* d_part = nullptr;
  Sum4* d_psum = nullptr;
  int* d_cnt = nullptr;
  int* d_gcnt = nullptr;
  double* d_fmax2 = nullptr;
  RetireState S{};
  // cluster-resident tail (k_tail.cu): the last tail_planes active planes
  // (0: disabled) are finished by one launch, one cluster per plane
  TailArgs tl{};
  float* d_tail_tabs = nullptr;   // per-slot packed FP32 tables of every level
  int tail_planes = 0;
  int tail_cap = -1;              // -1: as many as can be resident; 0: off; n: at most n
  bool prepare_tail();            // layout for the current schedule; false when unsupported
  void tail(const double2* f, double2* u, double tol, cudaStream_t st);
  int precision_of_buffers = 1;
  size_t vbytes() const { return opt.precision ? sizeof(float2) : sizeof(double2); }
};

}  // namespace ps
