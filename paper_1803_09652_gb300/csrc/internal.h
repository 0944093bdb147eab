// Internal interfaces between the host library and the kernel translation units.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "gbremd.h"

namespace gbk {

typedef unsigned long long u64;

// Everything the O(N^2) pair passes read and write.
struct PairArgs {
    const int64_t* atom_off;   // [M+1]
    const float4* xyzq;        // x, y, z, q
    const float2* rad;         // rho, S
    const float2* Rh;          // R, 1/(2R)          (pass 2)
    const float* cc;           // chain factor c_i   (pass 3)
    float offset;
    float tau_ke;              // (1/eps_in - 1/eps_out) k_e
    float ke_out, kappa;       // k_e / eps_out and the salt's inverse Debye length (EF_SALT)
    float kc;                  // k_e / eps_in
    float en_a, en_b, en_g;    // blocks of EnergyW: set_energy_factors
    float salt_l2;             // log2(eps_in / eps_out)
    float rep_k, rep_sigma;    // soft repulsion (rep_k == 0: off)
    float rgbmax;              // Born-radius cutoff (EF_CUT kernels of the Born and chain passes)
    float cut2;                // pair cutoff squared (EF_CUT kernels of the energy pass)
    float e_range2;            // energy-pass block range squared: max(cut, rep_sigma)^2
    u64* I_acc;                // [N]   Born integrals, 2^40 fixed point
    u64* dR_acc;               // [N]   R dE/dR pair part, 2^32
    u64* phi_acc;              // [N]   dE/dq pair part, 2^32
    u64* F_acc;                // [3N]  forces x | y | z, 2^32
    u64* E_acc;                // [M*4] E_GB, E_Coul, E_rep, spare, 2^32
    int64_t N;
    float4* boxes;             // [2 * tiles] bounding boxes of 32-atom tiles (nullable)
    const int* tile_off;       // [M+1] first tile of each replica
    int* err;                  // device error word (non-finite input, nullable)
};

// Replicas of up to this many 32-atom tiles (12,800 atoms) run 64 x 32 blocks
// only (walk_task in pairs_impl.cuh).  A pair costs less in 128 x 32 blocks, but a
// pass of them ends later: the line is where a GPU with few replicas breaks even.
// us, 64 x 32 / 128 x 32, of an MD step (with soft repulsion) and of a force call:
//   1 x 8000   162 / 184, 149 / 164      5 x 9000 to 4500   465 / 563, 452 / 539
//   1 x 9700   213 / 239, 202 / 213      5 x 9700 to 1212   315 / 373, 303 / 343
//   1 x 12000  297 / 318, 286 / 292      5 x 12000 to 6000  730 / 815, 728 / 788
//   1 x 14000  386 / 402, 374 / 370      5 x 14000          1614 / 1572, -
//   1 x 16000  467 / 487, 453 / 451      5 x 16000          2080 / 1988, -
// Full batches break even earlier (force calls): 16 x 6700 1255 / 1297, 16 x 8192
// 1824 / 1837, 16 x 9000 2177 / 2132, 16 x 10007 2628 / 2420, 8 x 12000 1896 / 1815.
constexpr int SMALL_TILES = 400;

// One warp task: replica, row pair and rows (4 P + 1, 2 or 3: atoms
// 128P .. 128P+63, the 64 after them, or both), first tile J (atoms
// 32J .. 32J+31, J >= 4P) and number of tiles of that row pair.
struct TaskList {
    int4* d_tasks = nullptr;
    int n_tasks = 0;
    bool small = false;        // every replica has at most SMALL_TILES tiles
    // register cap of each pass's kernel (Born, energy, chain), as 256-thread
    // blocks per SM: 1 (at most 128 registers), 3 (80) or 4 (64)
    int cap[3] = {1, 1, 1};
};

enum PassKind { PASS_BORN = 0, PASS_ENERGY = 1, PASS_CHAIN = 2 };

// flags for the energy pass; EF_CUT for any pass: the kernel applies the
// pass's cutoff (Born and chain passes: rgbmax; energy pass: cut) to a task
// list of in-range blocks (launch_pairs_list).  EF_STRADDLE is internal to
// the walker: the block has pairs on both sides of the cutoff and tests each
// pair.
enum { EF_ENERGY = 1, EF_PHI = 2, EF_REP = 4, EF_SALT = 8, EF_CUT = 16, EF_STRADDLE = 32 };

cudaError_t launch_pairs(int pass, int flags, const PairArgs& a, const TaskList& t,
                         int warps_per_block, cudaStream_t s);
// Cutoff passes (pairs_cut.cu).  launch_block_list clears the LIST_CTRS
// counters and builds the block neighbour lists from the tile boxes: list_b
// (Born-radius cutoff, when want_b) and list_e (pair cutoff, when want_e),
// each with room for both rows of every column of the batch; win_off [M+1] holds the first
// list-building warp of each replica (ceil(nb/4) * ceil(nb/32) warps per
// replica of nb tiles), columns the batch's columns.  launch_pairs_list runs pass `pass` with EF_CUT over
// a device-built task list whose length is ctr[0] (Born, chain) or ctr[1]
// (energy), taking tasks from the queue head ctr[2 + pass].
constexpr int LIST_CTRS = 5;
cudaError_t launch_block_list(const PairArgs& a, const int* win_off, int M, int total_warps, int64_t columns,
                              int4* list_b, int4* list_e, int* ctr, int want_b, int want_e, cudaStream_t s);
cudaError_t launch_pairs_list(int pass, int flags, const PairArgs& a, const int4* list, int* ctr, int cap,
                              int warps_per_block, cudaStream_t s);

// Uniform factors of the distant energy blocks: with W = k_c q_i q_j / f^3
// (times tF / k_c with salt, tau k_e / k_c folded into them without) the pair
// adds W (en_a exp(-D) + en_b) to -(de/dr)/r and en_g W exp(-D) (1 + D) R_i R_j
// to R de/dR.
inline void set_energy_factors(PairArgs& a, const gb_params& p) {
    const double tau = p.kappa != 0.0f ? 0.5 : 0.5 * (1.0 - (double)p.eps_in / (double)p.eps_out);
    a.en_a = (float)(0.5 * tau);
    a.en_b = (float)(-2.0 * tau);
    a.en_g = (float)tau;
    a.salt_l2 = (float)std::log2((double)p.eps_in / (double)p.eps_out);
}
// Cutoff fields of the pair arguments, and the EF_CUT flag of each pass.
inline void set_cutoffs(PairArgs& a, const gb_params& p) {
    a.rgbmax = p.rgbmax;
    a.cut2 = p.cut * p.cut;
    const float er = (p.rep_k != 0.0f && p.rep_sigma > p.cut) ? p.rep_sigma : p.cut;
    a.e_range2 = er * er;
}
inline int cut_flag(int pass, const gb_params& p) {
    return (pass == PASS_ENERGY ? p.cut > 0.0f : p.rgbmax > 0.0f) ? EF_CUT : 0;
}
// Parameter checks shared by every entry point that takes gb_params.
inline bool params_ok(const gb_params& p) {
    return p.offset >= 0.0f && p.eps_in > 0.0f && p.eps_out > 0.0f && p.rep_k >= 0.0f &&
           p.rep_sigma >= 0.0f && p.kappa >= 0.0f && p.kappa < 1.0e3f && p.rgbmax >= 0.0f &&
           p.rgbmax < 1.0e6f && p.cut >= 0.0f && p.cut < 1.0e6f;
}

// Columns (32-atom tiles against 128-atom row pairs) of an n-atom replica.
int64_t pair_columns(int64_t n);
// Bounding boxes of all tiles (PairArgs::boxes, tile_off); no-op when boxes is null.
cudaError_t launch_tile_boxes(const PairArgs& a, int M, int total_tiles, cudaStream_t s);

// O(N) kernels --------------------------------------------------------------

struct AtomArgs {
    const int64_t* atom_off;
    int32_t M;
    int32_t max_n;             // largest replica
    const float4* xyzq;
    const float2* rad;
    float alpha, beta, gamma, offset;
    double tau_ke;
    double kc, ke_out, kappa;  // k_e / eps_in, k_e / eps_out, salt (self terms)
    u64* I_acc;
    u64* dR_acc;
    u64* phi_acc;
    u64* F_acc;
    u64* E_acc;
    float2* Rh;
    float* cfac;               // a_i dR_i/dpsi_i
    float* cc;                 // c_i = dE/dR_i * cfac_i
    int* err;
    int64_t N;
};

cudaError_t launch_born_finalize(const AtomArgs& a, float* R_out, cudaStream_t s);
// bond_k != 0 adds the chain-bond forces (MD) to the force accumulators.
cudaError_t launch_energy_finalize(const AtomArgs& a, int want_energy, double* phi_out, cudaStream_t s,
                                   float bond_k = 0.0f, float bond_r0 = 0.0f);
cudaError_t launch_forces_out(const AtomArgs& a, int64_t* F_fixed, float* F_out, double* E_out,
                              cudaStream_t s);

struct MDArgs {
    float4* xyzq;
    float4* vel;
    float4* force;
    const u64* ctr;            // [0] step base, [1] exchange attempt base
    float h;                   // dt / 2
    float inv_m;               // ACCEL / mass
    float c1, c2;              // exp(-gamma dt), sqrt((1 - c1^2) kT ACCEL / m)
    float bond_k, bond_r0;
    u64 seed;
    u64 rep_base;              // global index of replica 0 in the Philox counters
};

// MD half steps between force evaluations (k_md_step): MD_CLOSE stores the
// evaluated force (MD_KICK: and applies the closing half kick), MD_OPEN runs
// B A O A of the next step and rebuilds the tile boxes (boxes may be null).
enum { MD_CLOSE = 1, MD_KICK = 2, MD_OPEN = 4 };
cudaError_t launch_md_step(const AtomArgs& a, const MDArgs& m, float4* boxes, const int* tile_off,
                           int step_in_block, int mode, cudaStream_t s);
cudaError_t launch_set_counters(u64* ctr, u64 step, u64 attempt, cudaStream_t s);
cudaError_t launch_advance_counters(u64* ctr, u64 steps, u64 attempts, cudaStream_t s);

// Monte Carlo: site rows are summed over MC_CHUNK-atom slices of a replica.
constexpr int MC_MAX_SITE_ATOMS = 128;
constexpr int MC_CHUNK = 256;

struct MCArgs {
    const int64_t* atom_off;
    const int32_t* site_off;
    const int32_t* site_kind;
    const int32_t* site_nstates;
    const int32_t* site_atom_off;
    const int32_t* site_atom_idx;
    const int32_t* site_state_off;
    const int32_t* site_q_off;
    const float* q_state;
    const double* G_ref;
    const int32_t* n_H;
    const int32_t* n_e;
    const double* pKa_ref;
    const double* E0_ref;
    float4* xyzq;
    const float* R;            // Born radii (stride 1) ...
    const float2* Rh;          // ... or (R, 1/(2R)) pairs when R == nullptr
    const double* pH;
    const double* E;
    double kT;
    double tau_ke, kc;
    double ke_out, kappa;      // salt screening of the solvent term (kappa 0: none)
    float cut2;                // pair cutoff squared (0: none)
    u64 seed;
    u64 step;
    u64 rep_base;              // global index of replica 0 in the Philox counters
    const u64* ctr;            // when non-null the step is ctr[0] + step
    int32_t kind;
    int32_t* state;
    double* dG_out;
    uint8_t* acc_out;
    double* phi_part;          // [M][n_parts][MC_MAX_SITE_ATOMS] slice partials (workspace;
                               // [M][n_parts][SWEEP_MAX_SITE_ATOMS] for sweeps)
    int32_t n_parts;           // slices of the largest replica
    int* err;                  // device error word (sweeps over their limits)
};

// Per-residue sweeps (Sec. III.A.2): limits per replica and kind.
constexpr int SWEEP_MAX_SITE_ATOMS = 1024;
constexpr int SWEEP_MAX_SITES = 256;
cudaError_t launch_mc_sweep(const MCArgs& a, int32_t M, cudaStream_t s);

cudaError_t launch_mc(const MCArgs& a, int32_t M, cudaStream_t s);

struct ExArgs {
    int32_t n_ladders, len, ladder_stride, slot_stride;
    const double* values;
    int32_t* rep_at_slot;
    const int32_t* n_count;
    int32_t dim;
    u64 attempt;
    const u64* ctr;            // when non-null the attempt is ctr[1] + attempt
    u64 seed;
    double kT;
    int32_t wrap;
    double* value_of_rep;
    double* delta_out;
    uint8_t* acc_out;
};

cudaError_t launch_exchange(const ExArgs& a, cudaStream_t s);

// Two-dimensional grid exchange used by the MD driver: the dimension of
// attempt k is E when (k / 2) is even and pH otherwise (or fixed by ex_dim).
struct GridExArgs {
    int32_t n_pH, n_E;
    const double* E_ladder;
    const double* pH_ladder;
    int32_t* grid;
    const int32_t* site_off;
    const int32_t* site_kind;
    const int32_t* site_nstates;
    const int32_t* site_state_off;
    const int32_t* n_H;
    const int32_t* n_e;
    const int32_t* state;
    const u64* ctr;
    int* err;                  // GB_ERR_INVALID_ARG on a state outside its site's range
    u64* ex_count;             // nullable [2 dims][attempts, acceptances][n_pH * n_E]
    int32_t ex_dim;            // 0 E only, 1 pH only, 2 alternate
    int32_t wrap;
    u64 seed;
    double kT;
    double* E_rep;
    double* pH_rep;
};

cudaError_t launch_grid_exchange(const GridExArgs& a, cudaStream_t s);

// State occupancy counts after a Monte Carlo halt: for every site of replica
// r, occ[g * stride + (local index of its current state)] += 1, with g the
// grid slot holding r (r itself without a grid).
struct OccArgs {
    const int32_t* site_off;
    const int32_t* site_nstates;
    const int32_t* site_state_off;
    const int32_t* state;
    const int32_t* grid;       // nullable: slot -> replica
    int32_t M, n_sites, stride;
    u64* occ;
    int* err;                  // GB_ERR_INVALID_ARG: a replica's layout or a state out of range
};
cudaError_t launch_occupancy(const OccArgs& a, cudaStream_t s);

// Persistent MD kernel (persist.cu): nsteps MD steps of the whole batch in one
// launch, as a queue of warp items with per-(phase, replica) completion counts.
struct PersistArgs {
    PairArgs pa;
    AtomArgs aa;
    MDArgs md;
    const int4* tasks;         // pair tasks of every replica, replica after replica
    const int* task_off;       // [M+1] first task of each replica
    const int* phase_off;      // [6][M+1] first item of each replica within a phase
    const int* count;          // [6][M] items of each replica per phase
    int phase_base[7];         // first item of each phase within a step; [6] = items per step
    int M;
    int nsteps;                // MD steps in this launch
    int step0;                 // index of the first of them in the enqueued block
    float* R_out;              // Born radii of the last step (nullable)
    unsigned* head;            // queue head, followed by the 6 x M completion counters
    unsigned* done;
    int* err;
    unsigned spin_limit;       // polls before a dependency wait gives up (GB_ERR_TIMEOUT)
};
cudaError_t persist_occupancy(int rep, bool small, int* blocks_per_sm);
cudaError_t launch_persist(const PersistArgs& a, int rep, bool small, int grid, cudaStream_t s);

// Small batches in one launch (fused.cu).
constexpr int FUSED_WARPS = 8;     // warps of a thread block
struct FusedArgs {
    PairArgs pa;
    AtomArgs aa;
    MDArgs md;                 // nsteps > 0
    const int4* tasks;         // pair tasks (one block each) of every replica, replica after replica
    const int* task_off;       // [M+1] first task of each replica
    int blocks;                // thread blocks of every replica's cluster: 1, 2, 4, 8 or 16
    int M;
    int nsteps;                // MD steps (0: one force evaluation of given coordinates)
    int step0;                 // index of the first of them in the enqueued block
    int born_only;             // nsteps == 0: stop after the Born radii
    float* R_out;              // nullable
    int64_t* F_fixed;          // nullable, nsteps == 0
    float* F_out;              // nullable, nsteps == 0
};
// Clusters of that many blocks the device holds at once.
cudaError_t fused_resident(int flags, int blocks, int* clusters);
cudaError_t launch_fused(const FusedArgs& a, int flags, cudaStream_t s);

cudaError_t launch_count(const int32_t* site_off, const int32_t* site_kind, const int32_t* site_nstates,
                         const int32_t* site_state_off, const int32_t* n_H,
                         const int32_t* n_e, const int32_t* state, int32_t kind, int32_t M,
                         int32_t* out, cudaStream_t s);

}  // namespace gbk
