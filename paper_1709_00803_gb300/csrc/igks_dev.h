// igks_dev.h -- device data layout and launch entry points shared by the translation
// units of libigks (not part of the public ABI).
//
// Layout: every solve of a context is concatenated into one set of structure-of-arrays
// buffers in HBM. Cell ranges of consecutive solves start on multiples of CELL_ALIGN so
// that every block of the per-cell kernels belongs to exactly one solve (deterministic
// per-solve reductions without atomics on floating-point sums). Cells past a solve's end
// inside its aligned range are padding (cell_solve = -1) and are skipped everywhere.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "igks_norm.cuh"

namespace igks {

constexpr int KDOF = 3;                                  // internal degrees of freedom (Eq. 2)
constexpr double GAMMA = (KDOF + 4.0) / (KDOF + 2.0);    // 1.4
constexpr int CELL_ALIGN = 256;
// Block of the per-cell kernels: they are bound by the FP64 pipe of an SM, so a small mesh
// wants its cells on as many SMs as it has warps for (20,480 cells: 80 blocks of 256 threads
// left half of the 152 SMs idle; 64 threads make 320). Large meshes do not care.
constexpr int CELL_BLOCK = 64;
static_assert(CELL_BLOCK == NORM_CELLS, "a block of the residual kernel gives one partial norm");

// Spalart-Allmaras (SA-noft2 with the 2012 S-tilde clipping)
constexpr double SA_CB1 = 0.1355, SA_CB2 = 0.622, SA_SIGMA = 2.0 / 3.0, SA_KAPPA = 0.41;
constexpr double SA_CW1 = SA_CB1 / (SA_KAPPA * SA_KAPPA) + (1.0 + SA_CB2) / SA_SIGMA;
constexpr double SA_CW2 = 0.3, SA_CW3 = 2.0, SA_CV1 = 7.1, SA_CV2 = 0.7, SA_CV3 = 0.9;

struct DevFlow {
  double mach, re, prandtl, s_star, lam_inf, mu_inf, nut_inf, p_inf;
  double Winf[5];
  double cfl_exp, cfl_init, cfl_min, cfl_max, res_target, venkat_k, c_num, eq40_target;
  double pr_fix;   // 1/Pr - 1, the factor of the Prandtl-number fix
  double tr_h, visc_c;   // T/T_inf = tr_h h; Sutherland: mu = visc_c h^(3/2) / (tr_h h + s_star)
  int sa_on, limiter, visc_sr, scheme;
};

// per-solve iteration state, updated only on the device during iterations
constexpr int PF_E = 3;              // stencil entries held per sweep record

// Records of the narrow sweeps, one per sweep position and direction, brought into shared
// memory by bulk copies.
// Static part (uploaded once): cell, kind (entry count, and the flags below), the cell's
// backward position (forward records), what the cell itself stores to global memory (spill,
// the flags below), and per entry where the neighbour's increments are: a slot of the
// shared-memory ring, from ring_slots on a side slot (a neighbour that left the ring,
// fetched again ahead of its level), ZERO_SLOT (no entry: reads zeros, and its coefficients
// stay zero), SLOT_GLOBAL (read from global memory) or SLOT_GHOST (a wall or symmetry ghost
// after an interior neighbour, whose mean-flow terms the forward sweep leaves in the entry's
// coefficients).
// Per iteration (T = double, float or double-float): m = residual M (forward) or forward
// increment dW* (backward), state (r, mx, my), 1/D, 1/a_ii, u, v, H, per entry (sx, sy,
// s lambda, SA coefficient), and the backward sum's start (the ghosts that come first;
// start[4] in pad0[0]). The static part, the head (m to pad0) and two entries (8-byte types:
// one) are whole 32-byte sectors, so the pre-pass leaves few sectors partly written (with
// 176-byte records it took 377 us on a batch of 623,000 cells, with these 135 us), and four
// consecutive records start on distinct 32-byte bank groups.
constexpr int INC_STRIDE = 8;        // floats of a cell in the FP32 increment arrays (five used)
constexpr int SLOT_GLOBAL = -1, SLOT_GHOST = -2;
constexpr int KIND_COUNT = 7;        // entries
constexpr int KIND_THIRD = 8;        // a third entry, all three in ring or side slots
constexpr int KIND_RARE = 16;        // a ghost, or a neighbour in global memory
constexpr int KIND_SIDE = 32;        // a side slot (not in a cluster)
constexpr int KIND_CSR = 64;         // more than PF_E entries: the CSR stencil (KIND_RARE too)
constexpr int SPILL_READ = 1;        // a later cell reads this cell's increments from global memory
constexpr int SPILL_OWN = 2;         // the level and the next do not fit the ring: no store warp takes it
struct alignas(16) SweepStat { int i, kind, pb, spill; int slot[PF_E], pad; };
struct alignas(16) SweepJ { int j[PF_E], pad; };            // the entries' cells, -1 - face for a ghost
template <class T>
struct alignas(16) SweepRec {
  SweepStat st;
  T m[5], w[3], c[5];
  T pad0[3];
  T co[PF_E][4];
  T start[4];
};
static_assert(sizeof(SweepStat) == 32 && sizeof(SweepJ) == 16, "static record size");
static_assert(sizeof(SweepRec<float>) == 160 && sizeof(SweepRec<double>) == 288, "record size");

struct SolveState {
  double icfl;    // 1 / cfl
  double dt, cfl, res_inf, res_l2, res_l2_first, res_inf_prev, eq40;
  int iter;
  int state;      // 0 running, 1 converged, <0 error; read by every kernel of an iteration
  int pending;    // state to take at the end of the current iteration
  int blk_begin, blk_end;      // per-cell-kernel blocks of this solve that hold cells
  int cell_begin, cell_end;    // [begin, end) real cells
};

struct Dev {
  int n_solves;
  int nc_pad;               // total (padded) cells
  int nf;                   // total faces
  int nbf;                  // total boundary faces
  // nodes
  const double* xy;         // [2][nn]
  int nn;
  // cells
  const int* cell_solve;    // [nc_pad], -1 for padding
  const int* cf_ptr;        // [nc_pad+1] cell -> face CSR (ascending uploaded face order)
  const int* cf_face;
  const int* cn_ptr;        // [nc_pad+1] cell -> node CSR
  const int* cn_node;
  double* area; double* cx; double* cy; double* wall_d;
  double* W;                // [5][nc_pad]
  double* grad;             // [8][nc_pad] unlimited least-squares gradients, index 2v+{x,y}
  double* phi;              // [4][nc_pad]
  double* omega;            // [nc_pad] vorticity magnitude (SA)
  double* mu_l; double* mu_t;
  double* pu; double* pv; double* pc;   // [nc_pad] velocity and sound speed of every cell (k_prep)
  double* lsq;              // [4][nc_pad] least-squares normal matrix A00, A01, A11 and 1/det (geometry)
  double* Lam;              // [nc_pad] sum over faces of (Lambda_c)_ij
  double* M;                // [5][nc_pad]
  double* nul;              // [nc_pad] laminar kinematic viscosity (k_prep)
  double* lgrad;            // [8][nc_pad] limited gradients of solves with a limiter, from k_gradient
                            // to k_flux (the memory of sw_st, which the pre-pass writes later)
  double* sa_diag;          // [nc_pad] SA diagonal without the Omega/dt_imp term
  void* dWs;                // increments, T = sweep type: FP32 [nc_pad][INC_STRIDE], else [5][nc_pad]
  void* dW;                 // the same
  void* dF;                 // [8][nc_pad] of T: increments of the x and y Euler fluxes
  // faces
  const int* fL; const int* fR; const int* fbc; const int* fsolve;
  const int* fnode;         // [2][nf] face end nodes
  const int* bface;         // [nbf] boundary face ids
  double* fS; double* fnx; double* fny; double* fmx; double* fmy;
  double* fcx; double* fcy; // centre across the face (neighbour or ghost)
  double* fidL; double* fidR; double* fdn; // reciprocal normal distances centre->face; centre->centre
  double* lam_f;            // [nf]
  double* F;                // [6][nf]
  double* sa_a;             // [4][nf]: aLR, aRL, diag L, diag R
  double* G;                // [5][nf] ghost state (boundary faces)
  double* Gmu;              // [2][nf] ghost mu_l, mu_t
  // wall faces per solve (wall distance)
  const int* wall_face; const int* wall_ptr;   // wall_ptr[n_solves+1]
  // sweep schedule
  const int* fwd_order; const int* fwd_lvl;    // cell ids in level order; level offsets
  const int* bwd_order; const int* bwd_lvl;
  const int* lvl_solve_ptr;                     // [n_solves+1] into fwd_lvl (levels per solve)
  const int* blvl_solve_ptr;                    // [n_solves+1] into bwd_lvl
  // sweep pre-pass results (type T of the sweep precision)
  void* sw_cell;                 // [5][nc_pad]: 1/D, 1/a_ii (SA), u, v, E + p
  void* sw_st;                   // [4][nnz]: signed hS nx, hS ny, hS lambda, SA coefficient
  int* sw_j;                     // [nnz] neighbour across each cell-face entry, -1 on a boundary
  int nnz;                       // entries of the cell -> face CSR
  // narrow schedule: stencils in sweep-position order (positions index fwd_order /
  // bwd_order). Forward entries are the lower neighbours, backward entries the upper
  // neighbours plus wall/symmetry ghosts (j = -1 - face). slot >= 0: the neighbour's
  // increments are still in the block's shared-memory ring at that slot.
  const int* fs_ptr; const int* fs_j; const int* fs_slot; const int* cf_to_fs;
  const int* bs_ptr; const int* bs_j; const int* bs_slot; const int* cf_to_bs;
  void* sc_f; void* sc_b;        // [4][entries] coefficients (T), written by the pre-pass
  int nfs, nbs;                  // entry counts
  // narrow schedule, per sweep position p (P = npos = all real cells): one record per
  // position and direction, array-of-structures so that consecutive records are one
  // contiguous range (one bulk copy); the static part (cell, entry count, neighbours,
  // ring slots) is uploaded once, the per-iteration part written by the pre-pass. Up to
  // PF_E stencil entries per record (cnt < 0: more than that, use the CSR stencil above).
  int npos;
  const int* pos_f; const int* pos_b;            // [nc_pad] position of a cell (-1 padding)
  const SweepJ* fj; const SweepJ* bj;            // [P]
  void* frec; void* brec;                        // [P] SweepRec<T>
  const int* fside_ptr; const int* bside_ptr;    // per level (indexed as fwd_lvl / bwd_lvl): the cells
  const int* fside_j; const int* bside_j;        // whose increments go to the level's side slots
  const int* gent_ptr;                           // [n_solves+1] cells with wall or symmetry ghosts
  const int* gent_pos;                           // their backward positions (records, not CSR stencils)
  int ring;                                      // slots of the shared-memory ring
  void* gprim;                                   // [6][nf] T: ghost r, mx, my, u, v, H of wall/symmetry faces
  const int* cf_to_ef; const int* cf_to_eb;      // [nnz] p * PF_E + e, or -1 (not an entry)
  int wait_limit;                // spins of a device wait before it gives up (IGKS_TIMEOUT)
  int starve_test;               // test hook: the forward sweep never stages its second chunk of records
  int* tmo;                      // [n_solves] a sweep wait of the solve ran out this iteration
  // wide schedule: cells of each level of all solves
  int wide;                      // 1: one launch per level; 0: one block per solve
  int sweep_cluster;             // narrow schedule: blocks (a thread-block cluster) per solve
  const int* broad;              // [n_solves] levels of more than BROAD_LEVEL cells on average
  int n_broad;                   // broad solves of the group that clusters sweep while one block each
                                 // sweeps the others (0 with sweep_cluster > 1: all in clusters)
  const int* wfwd_cells; const int* wbwd_cells;
  const int* h_wfwd_ptr; const int* h_wbwd_ptr;   // HOST arrays of level offsets (launch sizes)
  int n_wfwd, n_wbwd;
  // per solve
  const DevFlow* flow;
  SolveState* st;
  unsigned long long* dt_bits;   // [n_solves] atomic min of the explicit time step
  unsigned long long* eq40_bits; // [n_solves] atomic max of the Eq. 40 ratio
  int* bad;                      // [n_solves] divergence flag of the current update
  double* part;                  // [2][n_blocks] residual norm partials per cell block
  double* hist;                  // [n_solves][HIST][2] residual norms of the last HIST iterations
  int n_cell_blocks;
  int flux_block;                // threads per block of the flux kernel (<= 128)
  int* err;                      // [4] device error flags (mesh orientation, area)
  // The range one launch of an iteration kernel covers: a group of consecutive solves
  // (the whole context unless the solves are split into groups that run on streams of
  // their own). Per-cell kernels take blocks [g_blk0, g_blk0 + g_nblk) of CELL_BLOCK
  // cells, per-face kernels faces [g_face0, g_face0 + g_nface), per-solve kernels and the
  // narrow sweeps solves [g_solve0, g_solve0 + g_nsolve).
  int g_blk0, g_nblk, g_face0, g_nface, g_solve0, g_nsolve;
  int sweeps;                    // 0: every solve of the group is explicit, the sweeps are not launched
  int chained;                   // launch_chained: one group, no events between the kernels
};

// ---- launches (igks_kernels.cu / igks_flux.cu) ----
void launch_geometry(const Dev& d, cudaStream_t s);
void launch_wall_distance(const Dev& d, cudaStream_t s);
void launch_init_state(const Dev& d, int solve, cudaStream_t s);
void launch_prep(const Dev& d, cudaStream_t s);
void launch_ghost(const Dev& d, cudaStream_t s);
void launch_gradient(const Dev& d, cudaStream_t s);
cudaError_t upload_flux_table(cudaStream_t s);   // the table of the FP64 and double-float solves' flux
void launch_flux(const Dev& d, int precision, cudaStream_t s);
void launch_residual(const Dev& d, cudaStream_t s);
void launch_norms(const Dev& d, cudaStream_t s);
void setup_sweeps();   // kernel attributes (shared-memory ring size), once per build
void launch_sweep_prep(const Dev& d, int precision, cudaStream_t s);
void launch_sweep_fwd(const Dev& d, int precision, int threads, cudaStream_t s);
void launch_sweep_bwd(const Dev& d, int precision, int threads, cudaStream_t s);
void launch_update(const Dev& d, int precision, cudaStream_t s);
void launch_end_iter(const Dev& d, cudaStream_t s);
// check a staged [5][nc_pad] state per solve (bad[s] = 1: non-physical) and copy the
// solves that pass into W
void launch_set_state(const Dev& d, const double* staged, int* bad, cudaStream_t s);
// Launches of an iteration are chained (programmatic dependent launch): once all blocks of a
// kernel run, the blocks of the next one in the stream may take free places, and every thread
// waits for the end of the kernel before (chain_wait, the first thing in a kernel) and so for
// all before that. It hides part of the launch latency, 0.5 us a kernel: cavity of 10,000 cells
// 82.4 -> 79.5 us an explicit iteration, 133 -> 128 with multicolour sweeps (two levels), 1,470 polygons
// 235 -> 219 (ten levels). Not chained: several groups, which fill the GPU by themselves; the
// narrow sweeps, which have too few blocks to gain; the residual, whose waiting blocks slow
// the flux's last wave and the sweeps after it (20,480 cells in mixed precision 493 -> 515 us).
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... P, class... A>
inline void launch_chained(bool chained, void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s, A... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, P(a)...);
}
constexpr int N_KERNEL_KINDS = 11;   // kernels of one iteration (the wide sweeps launch per level)
// shared-memory ring of the narrow sweeps (cells) for a sweep type of t bytes: 13 values a
// cell, 104 KiB either way (a power of two: any cluster size divides it)
constexpr int ring_slots(int t) { return t == 4 ? 2048 : 1024; }
constexpr int SIDE = 32;             // side slots of a level (two sets, by the level's parity)
constexpr int zero_slot(int t) { return ring_slots(t) + 2 * SIDE; }
// Solves of few broad levels are swept by a cluster of blocks each, also where the others have one
// block: what counts in a level is then the cells that work at once, not the time between two
// barriers. Forward + backward, one block -> eight (one thread a cell in one block before): 10,000
// multicoloured quads (two levels) FP32 234 + 241 -> 65 + 57 us (87 + 76), FP64 500 + 506 -> 96 + 90
// (268 + 274); 6,504 polygons (levels of 650) double-float 496 + 524 -> 153 + 147 (348 + 375).
// The line lies where one block lost to what it was before; levels of 250-500 cells are faster in
// one block than then (490,000 quads as given, levels of 350: FP64 17.9 + 18.3 ms, 19.8 + 21.1).
constexpr int BROAD_LEVEL = 512, BROAD_CLUSTER = 8;
constexpr int NARROW_THREADS = 256;  // cell threads of the narrow sweeps at most (two per cell of a level)
constexpr int DEFAULT_WAIT_LIMIT = 1 << 24;   // spins of a device wait (about a second)
constexpr int MAX_BATCH_GRAPH_ITERS = 64;     // iterations captured in one whole-batch graph at most
constexpr int WIDE_MAX_LEVELS = 64;  // automatic choice: wide schedule up to this many levels
constexpr int HIST = 1024;           // iterations of residual history kept per solve

}  // namespace igks
