// qed_internal.h -- structures shared by the library's translation units (not part of the ABI).
#pragma once

#include <stdint.h>

#include <string>
#include <vector>

#include "qed.h"

// The host-only translation units do not include the CUDA runtime headers; this is the same
// declaration the runtime makes.
struct CUstream_st;
typedef struct CUstream_st* cudaStream_t;

namespace qedlib {

// ------------------------------------------------------------------ host table image
struct TableHost {
  qed_table_params p{};
  std::vector<double> ln_h, g, zeta_lo, zeta_hi, P, Q, ln_T, Pf;
  void resize(const qed_table_params& prm);
};
bool validate_table_params(const qed_table_params& p, std::string& err);
bool build_tables_host(const qed_table_params& p, TableHost& out, std::string& err);

// ------------------------------------------------------------------ device structures
// Look-up tables in precision R (device pointers + grid scalars).
template <typename R>
struct TabDev {
  const R* ln_h;     // [n_eta]
  const R* ln_T;     // [n_chi]
  // the inverse CDFs as an event reads them: one 16- or 32-byte head per eta row, the nodes in pairs
  // (value, next value), and per row a guide (kGuide entries) from the draw to its bracket
  const R* head;     // [n_eta * 4]  P_chi's first node, 1 - P_chi's last, zeta_lo, zeta_hi
  const R* P2;       // [n_eta * n_xi * 2]
  const R* Q2;       // [n_eta * n_xi * 2]
  const R* F2;       // [n_chi * n_f * 2]
  const uint32_t* gP;  // [n_eta * kGuide]  draws U in [0, 1/2]
  const uint32_t* gQ;  // [n_eta * kGuide]  draws 1 - U in [0, 1/2]
  const uint32_t* gF;  // [n_chi * kGuide]  draws V in [0, 1]
  int n_eta, n_xi, n_chi, n_f;
  R ln_eta_min, inv_d_eta, eta_min;
  R ln_chi_min, inv_d_chi, chi_min, chi_max, T_at_chi_max;
};

constexpr int kGuide = 256;  // guide entries per row: first bracket | last bracket << 16 of an equal share of the draws

// Per-species counters in device memory.
struct DevCounters {
  uint32_t n;        // particles held, including converted photons awaiting compaction
  uint32_t next_id;  // id given to the next particle created
  uint32_t n_app;    // particles appended to this species' append region during the step
  uint32_t n_dead;   // converted photons held
  uint32_t err;      // latched error bits (QED_ERR_* as 1u << code)
  // event counts (SpeciesDev::fine, coarse) are double-buffered: a step counts in buffer `phase`,
  // which is all zero when the step starts; its finalisation clears the entries the step before
  // used in the other one (ext, in fine groups) and then switches
  uint32_t phase;
  uint32_t ext[2];
  uint32_t win_n;    // photons the current window has advanced (the first win_n, a multiple of 1024)
  uint32_t pad[3];
};

// Photon windows: steps a window spans at most (a converted photon's step is a bit of `wflag`).
constexpr int kWinMax = 16;

// A parent's rank among its species' parents of children is summed from three levels: whole
// coarse groups, whole fine groups in its coarse group, whole mask words in its fine group.
constexpr int kFineShift = 5;    // 32 mask words (1024 parents) per fine group
constexpr int kCoarseShift = 5;  // 32 fine groups (32768 parents) per coarse group
#ifdef __CUDACC__
#define QED_HD __host__ __device__
#else
#define QED_HD
#endif
QED_HD constexpr uint32_t event_words(size_t cap) { return (uint32_t)(((cap >> 5) + 1 + 31) & ~size_t(31)); }
QED_HD constexpr uint32_t event_fines(size_t cap) { return ((event_words(cap) >> kFineShift) + 31u) & ~31u; }
QED_HD constexpr uint32_t event_coarses(size_t cap) { return ((event_fines(cap) >> kCoarseShift) + 31u) & ~31u; }
constexpr int kLedgerN = 15;

// Species arrays in precision R plus the scratch used by one step.
template <typename R>
struct SpeciesDev {
  R *x, *y, *z, *ux, *uy, *uz;
  double* tau;
  uint32_t* id;
  uint32_t cap;
  DevCounters* cnt;
  // as a parent: which lanes of each 32-particle chunk created children this step, and their
  // number per fine and coarse group (integer atomics; two buffers each, see DevCounters::phase)
  uint32_t* evmask;   // [event_words(cap)]
  uint32_t* fine;     // [2 * event_fines(cap)]
  uint32_t* coarse;   // [2 * event_coarses(cap)]
  uint32_t* cprefix;  // [event_coarses(cap)] exclusive prefix of coarse (batches)
  // photon windows: the photons a window found to convert (one bit each) and, per fine group, at
  // which of its steps (bit s); the groups' words are zero between windows
  uint32_t* cmask;    // [event_words(cap)]
  uint32_t* wflag;    // [event_fines(cap)]
  // as a destination: particles created for this species during the step
  R *ax, *ay, *az, *aux, *auy, *auz;
  double* atau;
  uint32_t* aparent;  // parent index | (parent is a positron) << 31
  uint32_t acap;
  // macroparticle weights (NULL: every particle has weight 1); children inherit their parent's
  R* w;   // [cap]
  R* aw;  // [acap]
};

// What a step's merge needs to know.  finalize_kernel's blocks each make their own (of the stored one
// they use the ticket); in batches the plan kernel stores it for the scatter.
struct FinalizePlan {
  uint32_t n_old[3];        // destination counts before the merge (e-, e+, photon destination)
  uint32_t next_id_old[3];
  uint32_t m[3];            // particles merged into each destination
  uint32_t from_electrons;  // photon children whose parents are electrons (ranked first)
  uint32_t phase[3];        // event-count buffer each parent species used
  uint32_t ticket;          // finalisation blocks done (the last one sets the counters)
};

// Analytic field parameters (Sec. 3.2 stand-in for the PIC gather).
struct FieldDev {
  int kind;
  double E[3], B[3];
  double E0, omega, phase0, phi_start, phi_len;
  // QED_FIELD_GRID: six Yee-staggered components (species precision), nodes, shape, geometry
  const void* grid;
  int n[3];
  int shape;
  double origin[3], spacing[3];
  // the grid packed by cells for this call (see pack_grid_kernel), and whether it was; NULL: not
  void* cells;
  uint32_t* packed;
};
// Cells of a packed grid component, and the bytes of a whole packed grid.
QED_HD constexpr size_t grid_cells(const int n[3]) { return ((size_t)n[0] + 1) * ((size_t)n[1] + 1) * ((size_t)n[2] + 1); }

// Whether a run of `steps` steps over that many particles gains by packing its grid (see pack_grid_kernel).
QED_HD constexpr bool packing_pays(uint64_t particles, uint64_t steps, uint64_t cells) {
  return particles * (steps < (1u << 20) ? steps : 1u << 20) >= cells / 3u;
}

// Host: descriptor -> device form, and its validation (shared by every entry point that steps).
FieldDev field_dev(const qed_field_desc& f);
qed_status check_field(const qed_field_desc& f, const char* who);

template <typename R>
struct StepArgs {
  SpeciesDev<R> sp[4];  // e-, e+, photons, drain (photon destination when draining)
  TabDev<R> tab;
  FieldDev field;
  double dt, t0, win_x0, win_v;
  R dt_r, win_v_r;  // dt and the window velocity in the working precision (set on the host)
  uint64_t seed, scenario, step;
  int emit, pairs, drain, recoil_energy;
  double* ledger_part;  // [gridDim.x * kLedgerN]
  double* ledger;       // [kLedgerN]
  FinalizePlan* plan;
  unsigned long long* work;  // [6] cumulative e+- pushes, photon pushes, particles created, the e+- and
                             // photon pushes made by multi-step passes (part of [0], [1]), and the
                             // per-step photon pushes in a field
  int want;                  // somebody can read this step's ledger: keep its sums
  int win_s;                 // step of the photon window this step belongs to (-1: none)
  uint32_t* counter;         // allocation-free step: the caller's photon counter (else NULL)
};

// What one batch step does with a slot, written by the tile schedule at the start of the step:
// the slot's tiles (256 particles, FP64 128) occupy [tile_base, tile_base + T[0] + .. + T[3]) of the batch
// step's tile space (species in order e-, e+, photons, then T[3]); n are the particles held (the step's
// parents).  Inside a photon window the photon tiles start at photon win_n, and T[3] tiles without
// particles follow, which share the conversions that the window found.
struct SlotPlan {
  uint32_t live;
  uint32_t tile_base;
  uint32_t T[4];
  uint32_t n[3];
  uint32_t win_n;
};
constexpr int kBatchTotals = 4;  // [tiles, the group of steps under way is the call's last, spare]

// Place of a batch step, or of the end of a photon window, in its call: inside; the last of a group
// of steps (a captured graph), which tot[1] says is the call's last or not; the last of its call.
enum BatchEnd { kBatchInside = 0, kBatchGroupEnd = 1, kBatchCallEnd = 2 };

// Many independent scenarios ("slots") stepped together: per-slot arguments live in device
// memory.  The per-step path puts the tiles of all live slots in one tile space that a
// persistent grid strides through; the multi-step passes give every live slot a share of the
// blocks proportional to its tiles.
template <typename R>
struct BatchCtl {
  StepArgs<R>* args;     // [S] per-slot arguments (their step field is the next step to take)
  uint32_t* remaining;   // [S] steps left per slot (0: idle)
  uint32_t* live;        // [S] slot takes part in the current batch step (set by the schedule)
  uint32_t* blocks;      // [S+1] exclusive prefix of the step-kernel blocks per slot (multi-step)
  SlotPlan* splan;       // [S] tile layout of the current batch step
  void* scal;            // [S] per-slot field scalars of the current step (StepScalars<R>)
  uint32_t* tot;         // [kBatchTotals] sizes of the current batch step's spaces
  void* wscal;           // [S * kWinMax] field scalars of the current photon window's steps (mixed path)
  TabDev<R> tab;         // the batch's tables (shared by every slot)
  int S;                 // slots
  int target_blocks;     // step-kernel grid (blocks striding through the tile space)
  int max_parts;         // ledger partials available per slot
  int grid_fields;       // some slot gathers its fields from a grid (selects that instantiation)
  uint32_t* first_event; // [S] multi-step probe result per slot
  uint32_t* tried;       // [S] stretch the slot's probe tried this batch step (0: not probed)
  uint32_t* skip;        // [S] batch steps the slot waits before probing again
  uint32_t* span;        // [S] stretch the slot's next probe tries (adapts to what probes find)
  int fuse_k;            // multi-step stretch per batch step (0: per-step only)
};

// Packs a.field's grid into a.field.cells if the run of `steps` steps has particles enough to gain by
// it, and writes to a.field.packed whether it has.
void launch_pack_grid(const StepArgs<float>& a, uint64_t steps, cudaStream_t s);
template <typename R>
void launch_step(const StepArgs<R>& a, int grid, int block, size_t smem, cudaStream_t s);
template <typename R>
void launch_batch_step(const BatchCtl<R>& c, int n_eta, int n_chi, BatchEnd end, int win_w, BatchEnd win_end, int win_s,
                       cudaStream_t s);
// A photon window of up to W steps in every slot (see window_kernel); the W batch steps that follow
// are launched with win_w = W, win_end = end and win_s = 0 .. W - 1.  The call's last step belongs to
// no window: a window that ends with it is one step shorter.
void launch_batch_window(const BatchCtl<float>& c, int n_chi, int W, BatchEnd end, cudaStream_t s);
size_t step_scalars_bytes(int precision);
// Advances the photons held, but for the last n mod 1024, by K <= kWinMax steps from a.step on (see
// window_kernel).
void launch_window(const StepArgs<float>& a, int K, cudaStream_t s);
// Merges the step's children into place and sets the counters; `step_grid` ledger partials are
// reduced when a.want is set.
template <typename R>
void launch_finalize(const StepArgs<R>& a, int step_grid, cudaStream_t s);
// Reduces `parts` ledger partials (after a multi-step commit).
template <typename R>
void launch_ledger(const StepArgs<R>& a, int parts, cudaStream_t s);
// Multi-step pass over K <= fuse_max_steps() steps: the probe (commit = false) sets
// *first_event to the first step with an event (K if none); the commit advances K event-free
// steps and writes the ledger partials of the last.  Returns the grid (ledger partials) used.
template <typename R>
int launch_fused(const StepArgs<R>& a, int K, bool commit, uint32_t* first_event, int max_parts, cudaStream_t s);
int fuse_max_steps();
void launch_selftest_wait(uint32_t polls, uint32_t* bits, cudaStream_t s);
template <typename R>
void launch_init_tau(const SpeciesDev<R>& sp, int kind, uint64_t seed, uint64_t scenario, cudaStream_t s);
template <typename R>
void launch_eval(const TabDev<R>& tab, const FieldDev& f, int kind, double t, double wx0, double wv, size_t n,
                 const double* x, const double* y, const double* z, const double* ux, const double* uy,
                 const double* uz, double* oE, double* oB, double* oparam, double* oenergy, double* orate,
                 cudaStream_t s);
template <typename R>
void launch_sample(const TabDev<R>& tab, int which, size_t n, const double* param, const double* U, double* out,
                   int32_t* ok, cudaStream_t s);
void launch_philox(size_t n, const uint64_t* ctr, uint64_t k0, uint64_t k1, uint64_t* out, cudaStream_t s);
template <typename R>
void launch_compact(const SpeciesDev<R>& sp, const SpeciesDev<R>& out, uint32_t* seg_count, uint32_t* seg_prefix,
                    cudaStream_t s);

void launch_tau_convert(int precision, double* tau, size_t n, bool to_double, cudaStream_t s);

// Macroparticle weights: fill, physical totals, photon merging (see qed_species_merge).
template <typename R>
void launch_fill(R* p, size_t n, R v, cudaStream_t s);
template <typename R>
void launch_totals(const SpeciesDev<R>& sp, int massless, double* partials, int blocks, cudaStream_t s);
struct MergeDev {
  double origin[3], cell[3];
  int n_cells[3], n_face, n_sub, min_group;
  uint64_t n_dir, n_en;  // direction and energy bins
  uint64_t none;         // cells * n_dir * n_en: the key of a photon that is not merged
  int bits;              // of the keys 0 .. none
  float inv_cell[3];     // 1/cell (the FP32 filter of the keys)
};
// Two buffers of n keys (32 or 64 bits, as M.bits needs) and indices; 256 counts per 4096 photons
// and 256 totals; two zeroed counters.
struct MergeScratch {
  void* keys[2];
  uint32_t* idx[2];
  uint32_t *hist, *totals, *count;
};
template <typename R>
void launch_merge(const SpeciesDev<R>& sp, const MergeDev& m, const MergeScratch& w, uint32_t n, int massless,
                  unsigned long long* groups, cudaStream_t s);

// Device images of a table set (defined with qed_tables in qed_api.cu).
struct TablesDev {
  TabDev<double> d64;
  TabDev<float> d32;
  template <typename R> const TabDev<R>& get() const;
};
template <> inline const TabDev<double>& TablesDev::get<double>() const { return d64; }
template <> inline const TabDev<float>& TablesDev::get<float>() const { return d32; }
TablesDev tables_dev(const qed_tables* t);
// Records the calling thread's error message (qed_last_error) and returns st.
qed_status set_error(qed_status st, const std::string& msg);
int step_grid_size(int precision);
void count_launch(int n = 1);

}  // namespace qedlib
