// Launch interface between the C ABI (mcc_abi.cu) and the kernel translation units.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "mcc_device.cuh"

namespace mcc {

enum Mode { kFused = 0, kPair = 1, kScatter = 2, kCorrect = 3, kFusedSmall = 4, kModes = 5 };
constexpr int kSmallCells = 320;  // largest cell of kFusedSmall (mcc_cell.cu)

// Per-interaction constants, precomputed on the host in FP64 (and rounded once for the mixed path).
struct InterConst {
    int32_t a, b;
    double kappa_mu2;  // q_a^2 q_b^2 lnL_ab dt / (4 pi eps0^2 dV) / mu^2: s = kappa_mu2 w_max N_min / u^3
    double kappa;      // same without 1/mu^2 (relativistic: s = kappa w_max N_min / (|p*|^2 v_rel*))
    double mu_ma, mu_mb, inv_ma, inv_mb;
    float kappa_mu2_f, kappa_f, mu_ma_f, mu_mb_f;
};

// Tables of the FP64 pair kinematics (mcc_pair64.cuh; sizes and entries: mcc_tables.h).
struct F64Tab {
    const double2* n97;
    const double2* turn;
    const double2* ln;
};

struct StepArgs {
    const int64_t* offsets;
    int32_t n_cells, S;
    int64_t n_total;
    void* vx;
    void* vy;
    void* vz;
    const double* w;
    double m[kMaxSpecies];
    float m_f[kMaxSpecies];
    float m_lo[kMaxSpecies];  // m - m_f rounded to float: (m_f, m_lo) is m as float-float
    double ma[kMaxSpecies];  // species masses for the relativistic kinematics
    float ma_f[kMaxSpecies];
    InterConst ic[kMaxInter];
    int32_t n_inter;
    int32_t inter_base;  // counter index of ic[0] (unfused calls: the interaction's index in the step)
    int32_t method, fail_policy, sort_by_weight, max_corr_passes, correct;
    int32_t weighting;  // 0: w_max N_min in s; 1: duplicity weighting (w_max / D_ij) N_max for inter-species pairs
    int32_t pairing;    // 0: order-N pairs; 1: all N x N pairs (fused step only)
    double c, fE;
    float c_f, fE_f;
    float fE_lo;              // fE - fE_f: (fE_f, fE_lo) is fE as float-float
    float gm1p_f, gm1p_lo;    // sqrt(1 - fE) - 1 as float-float (a capped energy pair that loses energy)
    float gm1n_f, gm1n_lo;    // sqrt(1 + fE) - 1 as float-float (a capped energy pair that gains energy)
    float c2inv_f, c2inv_lo;  // 1 / c^2 as float-float
    RngKey rng;
    const uint64_t* step_dev;  // step index in device memory (null: rng.step); step = *step_dev + step_add
    uint32_t step_add;
    F64Tab t64;            // tables of the FP64 pairs
    const float* n97_f32;  // N97 table of the float pairs (see mcc_device.cuh)
    const float* n97_dh32;
    // unfused input / output
    int32_t* pair_i;
    int32_t* pair_j;
    uint8_t* pair_flags;
    void* backup;
    int32_t* corr_pairs;
    int32_t* fail_count;
    // control
    int32_t* status;
    int32_t* queue;
    const int32_t* order;  // processing order of the cells (null: index order)
    int32_t cap;        // particles per cell staged in shared memory
    int32_t above;      // cells of at most this many particles belong to another launch (-1: none do)
    int32_t more;       // cells above cap belong to another launch (else they latch kErrBounds)
    char* slab;         // per-CTA global slabs for larger cells (may be null)
    int64_t slab_stride;
    int32_t slab_cap;
    const int32_t* order_range;  // one-CTA kernel: [begin, end) of `order` to take cells from (null: every cell)
    // group kernels (mcc_group.cuh)
    const int32_t* class_off;  // [2 * kOrderClasses]: begin / end of each size class in `order`
    int32_t* queues;           // [kOrderClasses] work-queue counters, one per class
    int32_t gcls;              // size class of the launch
    int32_t gcap;              // particles one group stages on chip in this class
    int32_t max_cell;          // the caller's bound on particles per cell (larger cells latch kErrBounds)
    double* resid;             // [2 * n_cells] or null: per-cell |dP| / sum m w |v| and |dE| / E of the exact state
    unsigned long long* phase_clk;  // [8 * kGroupClasses] cycles per phase and class (phase-timing builds)
};

constexpr int kGroupClasses = 5;  // group sizes 32, 64, 128, 256, 512 threads
// Beside them in the order of the cells: the cells above every class (the one-CTA kernel's), and the cells of class 0 below
// kHalfCells particles, run two to a warp if there are enough. A visit of a small cell takes nearly the same time
// whatever its size (serial phases, few lanes busy), so two at once nearly halve it. Measured
// per step, three species, one / two to a warp: 40000 cells of 30: 1.62 / 1.05 ms, of 90: 1.65 / 1.26, of 120: 1.74 / 1.62;
// 2e5 of 30: 7.23 / 4.12; relativistic beam of 65536 cells 7.54 / 6.25. At 128 particles a warp's two tiles still fit its
// share of the shared memory; lines at 160 and 224, where fewer warps are resident, take 1.09 and 1.31 ms at 30 particles.
constexpr int kRestClass = kGroupClasses, kHalfClass = kGroupClasses + 1, kOrderClasses = kGroupClasses + 2;
constexpr int kHalfCells = 128;  // a multiple of an eighth of its octave (the order's steps)
// Threads of a group of class cls.
constexpr int group_threads(int cls) { return cls == kHalfClass ? 16 : 32 << cls; }
#ifndef MCC_GROUP_WARPS_PER_SM
#define MCC_GROUP_WARPS_PER_SM 16
#endif
// Warps of the group kernels resident per SM: their register budget (launch bounds) and the automatic capacity
// (shared memory per warp) are both set for this many.
constexpr int kGroupWarpsPerSm = MCC_GROUP_WARPS_PER_SM;
// Warps of one CTA of the group kernels; its groups run in lockstep (mcc_group.cuh). Two CTAs of eight warps per SM
// overlap one's barrier waits with the other's work; the relativistic code is larger and gains more from fetching once for
// all sixteen warps (three-species step of 1.34e8 particles: 27.4 / 28.5 ms with 8 / 16 warps, four were 30% slower than
// eight; relativistic beam of 1.16e7: 6.7 / 5.9 ms).
constexpr int group_cta_warps(bool rel) { return rel ? 16 : 8; }

// Bytes per particle of the cell tile (keys, weights, velocities, pre-scatter copy, permutation, weight order).
__host__ __device__ inline size_t tile_bytes_per_particle(bool f32) { return 8 + 8 + (f32 ? 6 * 4 : 6 * 8) + 4 + 4; }

// Shared-memory bytes per particle of the group kernels' cell tile (state, weight, scratch, two orders).
constexpr size_t kGroupBytesPerParticle = 44;

// Shared memory of one group: its shared variables (shared_bytes, see group_shared_bytes) and a tile of cap particles.
__host__ __device__ inline size_t group_smem(size_t shared_bytes, int cap)
{
    return (shared_bytes + (size_t)cap * kGroupBytesPerParticle + 15) & ~(size_t)15;
}

// Kernel launches (defined in mcc_cell.cu / mcc_bin.cu).
// after: the launch before it on the stream is the same unfused call's, and this one may overlap it
cudaError_t launch_cell(bool f32, bool rel, int mode, const StepArgs& a, int grid, size_t smem, bool after, cudaStream_t st);
cudaError_t launch_step_advance(uint64_t* step, uint64_t by, cudaStream_t st);
// Cells ordered by group size class (largest class first; class kGroupClasses = cells above every class), largest
// first within a class; class_off receives each class's [begin, end) in `order`.
// half_min: class kHalfClass takes class 0's cells below kHalfCells
// if they are at least so many (0: never). hist: group_order_hist_bytes() of zeroed
// device memory.
size_t group_order_hist_bytes();
cudaError_t launch_group_order(const int64_t* offsets, int32_t n_cells, int32_t S, const int32_t* caps,
                               int32_t half_min, int32_t* order, int32_t* class_off, int32_t* hist, int64_t* launches, cudaStream_t st);
// Group kernels (mcc_group_*.cu): class cls runs groups of group_threads(cls) threads.
const void* group_kernel(bool f32, bool rel, int cls);
size_t group_shared_bytes(int cls);  // shared variables of one group
// groups: groups (cells at a time) of one CTA; after: the launch before it on the stream is a class of the same step, and
// this one may overlap it
cudaError_t launch_group(bool f32, bool rel, int cls, const StepArgs& a, int grid, int groups, size_t smem, bool after,
                         cudaStream_t st);
int cell_kernel_blocks_per_sm(bool f32, bool rel, int mode, size_t smem);
cudaError_t set_cell_smem_limit(bool f32, bool rel, int mode, size_t smem);
size_t cell_kernel_static_smem(bool f32, bool rel, int mode);

cudaError_t launch_bin(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells, int32_t n_species,
                       int32_t* perm, int64_t* offsets, void* ws, int32_t* status, cudaStream_t st, int64_t* launches);
size_t bin_workspace_bytes(int64_t n, int64_t n_keys);
cudaError_t launch_bin_weighted(const int32_t* cell, const int32_t* species, const double* w, int64_t n,
                                int32_t n_cells, int32_t n_species, int32_t* perm, int64_t* offsets, void* ws,
                                int32_t* status, cudaStream_t st, int64_t* launches);
size_t bin_weighted_workspace_bytes(int64_t n, int64_t n_keys);
cudaError_t launch_bin_static(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells,
                              int32_t n_species, int32_t* perm, int64_t* offsets, cudaStream_t st);
int64_t static_bin_max_keys();
// Adjoint of one interaction (mcc_adjoint.cu).
size_t adjoint_slab_bytes(int32_t max_cell, int32_t max_epairs, bool on_chip);
size_t adjoint_work_bytes(int32_t max_cell);  // working arrays of one cell
size_t adjoint_static_smem();
int adjoint_ctas_per_sm();
cudaError_t set_adjoint_smem_limit(size_t smem);
cudaError_t launch_adjoint(const StepArgs& a, double lnL, double* ox, double* oy, double* oz, double* gx, double* gy,
                           double* gz, double* gw, double* glnL, char* slab, int32_t max_cell, int32_t max_epairs,
                           int32_t tape, bool on_chip, int grid, cudaStream_t st);
cudaError_t launch_gather(const void* in, const int32_t* perm, int64_t n, int elem_bytes, void* out, cudaStream_t st);

// Species masses for the per-species moments (mcc_species_moments).
struct SpeciesConst {
    double m[kMaxSpecies];
};
cudaError_t launch_species_moments(bool f32, const void* vx, const void* vy, const void* vz, const double* w,
                                   const int64_t* offsets, int32_t n_cells, int32_t S, const SpeciesConst& sc,
                                   int rel, double c, const int32_t* fail_count, double* out, int num_sms,
                                   cudaStream_t st);

}  // namespace mcc
