// C ABI of the collision step (declarations and contracts in include/mcc.h).
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include <nvtx3/nvToolsExt.h>

#include "../../include/mcc.h"
#include "mcc_kernels.h"
#include "mcc_tables.h"
#include "mcc_pic.h"

static_assert(mcc::kGroupClasses == MCC_GROUP_CLASSES, "size classes of the ABI and the kernels");

// NVTX range over one entry point (header-only NVTX v3: a no-op unless a profiler injects itself), so that a timeline
// shows each library call on the host thread that issued it.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

struct mcc_ctx {
    int device;
    int32_t* dbuf;  // [0] status word, [1] and [2] work-queue counters, [4..7] debug record, then the tables
    int64_t launches;
    int num_sms;
    size_t smem_optin;
    size_t smem_per_sm;
    int32_t tile_cap;  // particles staged on chip per cell by the one-CTA kernel; 0 = automatic
    int32_t group_cap; // particles per warp of the group kernels' size classes; 0 = automatic
    int32_t group_tuned;  // the automatic capacity, tuned; 0 = from the shared memory
    int32_t group_top; // upper bound of the largest class; 0 = what one CTA's shared memory holds
    size_t smem_reserved;  // shared memory the system reserves per CTA
    // Attributes of the kernels, looked up once (each look-up costs about a microsecond of every call), and the last
    // occupancy of each (an unfused call has two shapes): launch shape << 8 | CTAs per SM in one word, so threads may share a
    // context.
    size_t cell_static[2][2][mcc::kModes];  // [float][relativistic][mode]
    size_t group_static[2][mcc::kOrderClasses];
    size_t adjoint_static;
    std::atomic<uint64_t> cell_occ[2][2][2][mcc::kModes], group_occ[2][mcc::kOrderClasses];
};

namespace mcc {

// Bytes per particle of the pairing mode's tile (defined with its kernel, mcc_cell.cu).
size_t pair_tile_bytes_per_particle();

}  // namespace mcc

namespace {

using mcc::StepArgs;

constexpr size_t kTabOffset = 64;  // bytes into the context buffer where the tables start: FP64 pairs, then float pairs
constexpr size_t kTab64Bytes = mcc::kF64TabDoubles * sizeof(double);
constexpr size_t kTab32Floats = 2 * (mcc::kN97Nodes + 1);
constexpr size_t kClkOffset = (kTabOffset + kTab64Bytes + kTab32Floats * sizeof(float) + 63) & ~63;
constexpr size_t kClkWords = 8 * mcc::kGroupClasses;  // phase cycles of the group kernels (phase-timing builds)
constexpr size_t kCtxBytes = kClkOffset + kClkWords * sizeof(unsigned long long);

constexpr size_t kStaticSmemReserve = 1024;  // margin above the cell kernel's static shared memory
#ifndef MCC_AUTO_CTAS
#define MCC_AUTO_CTAS 4
#endif
constexpr int kAutoCtasPerSm = MCC_AUTO_CTAS;  // automatic tile: this many CTAs share one SM's shared memory
constexpr int kMaxCtasPerSm = 2048 / mcc::kThreads;

cudaStream_t S(mcc_stream s) { return reinterpret_cast<cudaStream_t>(s); }

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

int cuda_status(cudaError_t e) { return e == cudaSuccess ? MCC_OK : MCC_ERR_CUDA; }

bool valid_params(const mcc_params* p)
{
    if (!p) return false;
    if (p->method != MCC_TA77 && p->method != MCC_N97) return false;
    if (!(p->dt > 0) || !(p->dV > 0) || !(p->eps0 > 0) || !(p->fE > 0) || !(p->fE < 1)) return false;
    if (p->relativistic && !(p->c > 0)) return false;
    if (p->max_corr_passes < 0 || p->fail_policy < 0 || p->fail_policy > 2) return false;
    if (p->weighting != 0 && p->weighting != 1) return false;
    if (p->pairing != 0 && p->pairing != 1) return false;
    return true;
}

// Fill the species / interaction constants of a launch (host FP64; one rounding to float for the mixed path).
int fill_args(StepArgs& a, const mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells,
              int32_t n_species, const mcc_species* sp, const double* lnL, const int32_t* inter, int32_t n_inter,
              int32_t inter_base, const mcc_params* p)
{
    std::memset(&a, 0, sizeof a);
    if (n_species < 1 || n_species > mcc::kMaxSpecies || n_cells < 0 || n_inter < 1 || n_inter > mcc::kMaxInter)
        return MCC_ERR_INVALID_ARG;
    a.offsets = offsets;
    a.n_cells = n_cells;
    a.S = n_species;
    if (P) {
        a.vx = P->vx;
        a.vy = P->vy;
        a.vz = P->vz;
        a.w = P->w;
        a.n_total = P->n;
    }
    if (sp) {
        for (int s = 0; s < n_species; ++s) {
            if (!(sp[s].m > 0)) return MCC_ERR_INVALID_ARG;
            a.m[s] = sp[s].m;
            a.m_f[s] = (float)sp[s].m;
            a.m_lo[s] = (float)(sp[s].m - (double)a.m_f[s]);
            a.ma[s] = sp[s].m;
            a.ma_f[s] = (float)sp[s].m;
        }
    }
    for (int k = 0; k < n_inter; ++k) {
        const int ia = inter[2 * k], ib = inter[2 * k + 1];
        if (ia < 0 || ib < ia || ib >= n_species) return MCC_ERR_INVALID_ARG;
        mcc::InterConst& ic = a.ic[k];
        ic.a = ia;
        ic.b = ib;
        if (sp && lnL && p) {
            const double qa = sp[ia].q, qb = sp[ib].q, ma = sp[ia].m, mb = sp[ib].m;
            const double mu = ma * mb / (ma + mb);
            const double L = lnL[ia * n_species + ib];
            const double kappa = qa * qa * qb * qb * L * p->dt / (4.0 * M_PI * p->eps0 * p->eps0 * p->dV);
            ic.kappa = kappa;
            ic.kappa_mu2 = kappa / (mu * mu);
            ic.mu_ma = mu / ma;
            ic.mu_mb = mu / mb;
            ic.inv_ma = 1.0 / ma;
            ic.inv_mb = 1.0 / mb;
            ic.kappa_f = (float)ic.kappa;
            ic.kappa_mu2_f = (float)ic.kappa_mu2;
            ic.mu_ma_f = (float)ic.mu_ma;
            ic.mu_mb_f = (float)ic.mu_mb;
        }
    }
    a.n_inter = n_inter;
    a.inter_base = inter_base;
    a.above = -1;
    if (p) {
        a.method = p->method;
        a.fail_policy = p->fail_policy;
        a.sort_by_weight = p->sort_by_weight;
        a.max_corr_passes = p->max_corr_passes;
        a.correct = p->correct;
        a.c = p->c;
        a.fE = p->fE;
        a.c_f = (float)p->c;
        a.fE_f = (float)p->fE;
        auto split = [](double x, float& hi, float& lo) {
            hi = (float)x;
            lo = (float)(x - (double)hi);
        };
        split(p->fE, a.fE_f, a.fE_lo);
        split(-p->fE / (1.0 + std::sqrt(1.0 - p->fE)), a.gm1p_f, a.gm1p_lo);
        split(p->fE / (1.0 + std::sqrt(1.0 + p->fE)), a.gm1n_f, a.gm1n_lo);
        split(p->c > 0 ? 1.0 / (p->c * p->c) : 0.0, a.c2inv_f, a.c2inv_lo);
        a.rng.k0 = (uint32_t)p->seed;
        a.rng.k1 = (uint32_t)(p->seed >> 32);
        a.rng.step = (uint32_t)p->step;
        a.rng.cell_base = p->cell_base;
        a.weighting = p->weighting;
        a.pairing = p->pairing;
    }
    a.status = ctx->dbuf;
    a.queue = ctx->dbuf + 1;
    const char* base = reinterpret_cast<const char*>(ctx->dbuf) + kTabOffset;
    a.t64.n97 = reinterpret_cast<const double2*>(base);
    a.t64.turn = a.t64.n97 + 12 * mcc::kF64N97;
    a.t64.ln = a.t64.turn + mcc::kF64Turn;
    a.n97_f32 = reinterpret_cast<const float*>(base + kTab64Bytes);
    a.n97_dh32 = a.n97_f32 + (mcc::kN97Nodes + 1);
    a.phase_clk = reinterpret_cast<unsigned long long*>(reinterpret_cast<char*>(ctx->dbuf) + kClkOffset);
    return MCC_OK;
}

// Largest on-chip tile (particles) one CTA can stage: the opt-in shared memory minus the kernel's static part.
size_t max_tile_particles(const mcc_ctx* ctx, bool f32)
{
    const size_t fixed = ctx->cell_static[f32][1][mcc::kFused] + kStaticSmemReserve;
    const size_t avail = ctx->smem_optin > fixed ? ctx->smem_optin - fixed : 0;
    return avail / mcc::tile_bytes_per_particle(f32);
}

// Largest cell of the pairing mode (its compact tile in one CTA's shared memory; the tile layout and its bytes per
// particle are defined with the kernel, in mcc_cell.cu).
size_t max_pair_tile_particles(const mcc_ctx* ctx)
{
    const size_t fixed = ctx->cell_static[0][0][mcc::kPair] + kStaticSmemReserve;
    const size_t avail = ctx->smem_optin > fixed ? ctx->smem_optin - fixed : 0;
    return avail / mcc::pair_tile_bytes_per_particle();
}

// Automatic tile: the largest that still lets kAutoCtasPerSm CTAs share an SM's shared memory.
int auto_tile(const mcc_ctx* ctx, bool f32)
{
    const size_t fixed = ctx->cell_static[f32][1][mcc::kFused] + 1024;
    const size_t per_cta = ctx->smem_per_sm / kAutoCtasPerSm;
    const size_t t = per_cta > fixed ? (per_cta - fixed) / mcc::tile_bytes_per_particle(f32) : 64;
    const size_t capmax = max_tile_particles(ctx, f32);
    return (int)(t < capmax ? t : capmax);
}

// CTAs per SM of a kernel in the launch shape `shape` (what its shared memory and threads follow from), from the cache if the
// last look-up was for the same.
template <class F>
int cached_occupancy(std::atomic<uint64_t>& slot, uint64_t shape, F look_up)
{
    const uint64_t c = slot.load(std::memory_order_relaxed);
    if (c != 0 && (c >> 8) == shape) return (int)(c & 255u);
    const int b = look_up();
    if (b > 0) slot.store((shape << 8) | (uint64_t)b, std::memory_order_relaxed);
    return b;
}

// Launch one cell-kernel pass over every cell, with a persistent grid of at most max_grid CTAs that take cells from a.queue (zero
// before). pass: 0, or 1 for the second launch of an unfused call, which may overlap the first.
int launch_cells(mcc_ctx* ctx, StepArgs& a, bool f32, bool rel, int mode, int cap, cudaStream_t st, int max_grid, int pass)
{
    const size_t per = mode == mcc::kPair ? mcc::pair_tile_bytes_per_particle() : mcc::tile_bytes_per_particle(f32);
    const size_t smem = (size_t)cap * per;
    const int bps = cached_occupancy(ctx->cell_occ[pass][f32][rel][mode], smem,
                                     [&] { return mcc::cell_kernel_blocks_per_sm(f32, rel, mode, smem); });
    if (bps < 1) return MCC_ERR_CUDA;
    int grid = ctx->num_sms * bps;
    if (grid > max_grid) grid = max_grid;
    if (a.n_cells < grid) grid = a.n_cells > 0 ? a.n_cells : 1;
    a.cap = cap;
    const cudaError_t e = mcc::launch_cell(f32, rel, mode, a, grid, smem, pass > 0, st);
    ctx->launches += 1;
    return cuda_status(e);
}

// The same with its queue reset before.
int run_cells(mcc_ctx* ctx, StepArgs& a, bool f32, bool rel, int mode, int cap, cudaStream_t st, int max_grid)
{
    if (cudaMemsetAsync(ctx->dbuf + 1, 0, sizeof(int32_t), st) != cudaSuccess) return MCC_ERR_CUDA;
    return launch_cells(ctx, a, f32, rel, mode, cap, st, max_grid, 0);
}

// An unfused call (one mode of the cell kernel over every cell). The caller gives no bound on its cells, and a tile for the
// largest cell leaves one CTA per SM; so the cells that fit the tile of four CTAs per SM go first, with that tile, and the
// larger ones in a second launch with the largest. 1000 cells of 400 particles, three interactions: 1.72 -> 1.16 ms. With no
// more cells than SMs one launch with the largest tile holds them all; with more, one reset serves both queues and the second
// launch overlaps the first. mcc_scatter, two launches one after another / so, us per call: FP64, 20 cells of 400 38 / 31, 1000 of
// 400 110 / 107; float, 20 of 400 36 / 29, 100 of 2800 59 / 53, 200 of 1500 63 / 58, 500 of 1500 111 / 106 (one launch with the
// largest tile for all cells: 43, 53, 58, 105; 1000 of 400 73 against 33).
int run_split(mcc_ctx* ctx, StepArgs& a, bool f32, bool rel, int mode, cudaStream_t st)
{
    const int cap = (int)(mode == mcc::kPair ? max_pair_tile_particles(ctx) : max_tile_particles(ctx, f32));
    int small = auto_tile(ctx, f32);
    if (mode == mcc::kPair)
        small = (int)((size_t)small * mcc::tile_bytes_per_particle(f32) / mcc::pair_tile_bytes_per_particle());
    if (small >= cap || a.n_cells <= ctx->num_sms) return run_cells(ctx, a, f32, rel, mode, cap, st, 1 << 30);
    if (cudaMemsetAsync(ctx->dbuf + 1, 0, 2 * sizeof(int32_t), st) != cudaSuccess) return MCC_ERR_CUDA;
    a.more = 1;
    const int rc = launch_cells(ctx, a, f32, rel, mode, small, st, 1 << 30, 0);
    if (rc != MCC_OK) return rc;
    a.more = 0;
    a.above = small;
    a.queue = ctx->dbuf + 2;
    return launch_cells(ctx, a, f32, rel, mode, cap, st, 1 << 30, 1);
}

// Whether the adjoint's working arrays for cells of max_cell particles fit one CTA's shared memory.
bool adjoint_on_chip(const mcc_ctx* ctx, int32_t max_cell)
{
    return mcc::adjoint_work_bytes(max_cell) + ctx->adjoint_static <= ctx->smem_optin;
}

// Grid of the adjoint kernel: one CTA per cell, at most as many as are resident. slab: bytes each CTA holds of the
// workspace (0: the slabs are per cell); more than two CTAs per SM only while they hold less than 1 GiB in all.
int adjoint_grid(const mcc_ctx* ctx, int32_t n_cells, int32_t max_cell, size_t slab)
{
    const size_t cta = ctx->adjoint_static + ctx->smem_reserved +
                       (adjoint_on_chip(ctx, max_cell) ? mcc::adjoint_work_bytes(max_cell) : 0);
    int per_sm = mcc::adjoint_ctas_per_sm();
    while (per_sm > 1 && cta * (size_t)per_sm > ctx->smem_per_sm) --per_sm;
    while (per_sm > 2 && slab * (size_t)per_sm * (size_t)ctx->num_sms > ((size_t)1 << 30)) --per_sm;
    const int g = ctx->num_sms * per_sm;
    return n_cells < g ? (n_cells > 0 ? n_cells : 1) : g;
}

}  // namespace

extern "C" {

int mcc_create(mcc_ctx** out, int device)
{
    if (!out) return MCC_ERR_INVALID_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(device);
    mcc_ctx* c = new (std::nothrow) mcc_ctx();
    if (!c) return MCC_ERR_CUDA;
    c->device = device;
    c->launches = 0;
    c->tile_cap = 0;
    c->group_cap = 0;
    c->group_top = 0;
    c->group_tuned = 0;
    int optin = 0, sms = 0, per_sm = 0, reserved = 0;
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device);
    c->smem_reserved = (size_t)reserved;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device);
    c->smem_per_sm = (size_t)per_sm;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    c->smem_optin = (size_t)optin;
    c->num_sms = sms;
    // kernels' static shared memory; each may take all the rest as dynamic shared memory
    cudaError_t attr = cudaSuccess;
    for (int f32 = 0; f32 < 2; ++f32)
        for (int rel = 0; rel < 2; ++rel)
            for (int mode = 0; mode < mcc::kModes; ++mode) {
                c->cell_static[f32][rel][mode] = mcc::cell_kernel_static_smem(f32, rel, mode);
                for (int pass = 0; pass < 2; ++pass) c->cell_occ[pass][f32][rel][mode] = 0;
                const cudaError_t e =
                    mcc::set_cell_smem_limit(f32, rel, mode, c->smem_optin - c->cell_static[f32][rel][mode]);
                if (e != cudaSuccess) attr = e;
            }
    for (int rel = 0; rel < 2; ++rel)
        for (int cls = 0; cls < mcc::kOrderClasses; ++cls) {
            if (cls == mcc::kRestClass) continue;
            cudaFuncAttributes fa;
            cudaError_t e = cudaFuncGetAttributes(&fa, mcc::group_kernel(true, rel, cls));
            if (e == cudaSuccess) {
                c->group_static[rel][cls] = fa.sharedSizeBytes;
                e = cudaFuncSetAttribute(mcc::group_kernel(true, rel, cls), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(c->smem_optin - fa.sharedSizeBytes));
            }
            c->group_occ[rel][cls] = 0;
            if (e != cudaSuccess) attr = e;
        }
    c->adjoint_static = mcc::adjoint_static_smem();
    const cudaError_t ea = mcc::set_adjoint_smem_limit(c->smem_optin - c->adjoint_static);
    if (attr != cudaSuccess || ea != cudaSuccess) {
        delete c;
        return MCC_ERR_CUDA;
    }
    // status word, queue counter and the tables, computed here once
    static double tab[mcc::kF64TabDoubles];
    static float tab32[kTab32Floats];
    static std::once_flag once;
    std::call_once(once, [] {
        mcc::f64_tables(tab);
        mcc::n97_table(tab32, tab32 + (mcc::kN97Nodes + 1));
    });
    if (cudaMalloc(&c->dbuf, kCtxBytes) != cudaSuccess || cudaMemset(c->dbuf, 0, kCtxBytes) != cudaSuccess ||
        cudaMemcpy(reinterpret_cast<char*>(c->dbuf) + kTabOffset, tab, sizeof tab, cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(reinterpret_cast<char*>(c->dbuf) + kTabOffset + sizeof tab, tab32, sizeof tab32,
                   cudaMemcpyHostToDevice) != cudaSuccess) {
        if (c->dbuf) cudaFree(c->dbuf);
        delete c;
        return MCC_ERR_CUDA;
    }
    *out = c;
    return MCC_OK;
}

void mcc_destroy(mcc_ctx* ctx)
{
    if (!ctx) return;
    DeviceGuard g(ctx->device);
    cudaFree(ctx->dbuf);
    delete ctx;
}

int mcc_bin_workspace_size(int64_t n, int32_t n_cells, int32_t n_species, size_t* bytes)
{
    if (!bytes || n < 0 || n_cells <= 0 || n_species <= 0) return MCC_ERR_INVALID_ARG;
    *bytes = mcc::bin_workspace_bytes(n, (int64_t)n_cells * n_species);
    return MCC_OK;
}

int mcc_bin(mcc_ctx* ctx, const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells,
            int32_t n_species, int32_t* perm_out, int64_t* offsets_out, void* ws, size_t ws_bytes, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_bin");
    if (!ctx || n < 0 || n_cells <= 0 || n_species <= 0 || !offsets_out) return MCC_ERR_INVALID_ARG;
    if (n > 0 && (!cell || !species || !perm_out)) return MCC_ERR_INVALID_ARG;
    if (n > INT32_MAX) return MCC_ERR_TOO_LARGE;
    if (!ws || ws_bytes < mcc::bin_workspace_bytes(n, (int64_t)n_cells * n_species)) return MCC_ERR_WORKSPACE;
    DeviceGuard g(ctx->device);
    return cuda_status(mcc::launch_bin(cell, species, n, n_cells, n_species, perm_out, offsets_out, ws, ctx->dbuf,
                                       S(stream), &ctx->launches));
}

int mcc_bin_weighted_workspace_size(int64_t n, int32_t n_cells, int32_t n_species, size_t* bytes)
{
    if (!bytes || n < 0 || n_cells <= 0 || n_species <= 0) return MCC_ERR_INVALID_ARG;
    *bytes = mcc::bin_weighted_workspace_bytes(n, (int64_t)n_cells * n_species);
    return MCC_OK;
}

int mcc_bin_weighted(mcc_ctx* ctx, const int32_t* cell, const int32_t* species, const double* w, int64_t n,
                     int32_t n_cells, int32_t n_species, int32_t* perm_out, int64_t* offsets_out, void* ws,
                     size_t ws_bytes, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_bin_weighted");
    if (!ctx || n < 0 || n_cells <= 0 || n_species <= 0 || !offsets_out) return MCC_ERR_INVALID_ARG;
    if (n > 0 && (!cell || !species || !w || !perm_out)) return MCC_ERR_INVALID_ARG;
    if (n > INT32_MAX) return MCC_ERR_TOO_LARGE;
    if (!ws || ws_bytes < mcc::bin_weighted_workspace_bytes(n, (int64_t)n_cells * n_species))
        return MCC_ERR_WORKSPACE;
    DeviceGuard g(ctx->device);
    return cuda_status(mcc::launch_bin_weighted(cell, species, w, n, n_cells, n_species, perm_out, offsets_out, ws,
                                                ctx->dbuf, S(stream), &ctx->launches));
}

int mcc_bin_static(const int32_t* cell, const int32_t* species, int64_t n, int32_t n_cells, int32_t n_species,
                   int32_t* perm_out, int64_t* offsets_out, mcc_stream stream)
{
    if (n < 0 || n_cells <= 0 || n_species <= 0 || !offsets_out) return MCC_ERR_INVALID_ARG;
    if (n > 0 && (!cell || !species || !perm_out)) return MCC_ERR_INVALID_ARG;
    if (n > INT32_MAX || (int64_t)n_cells * n_species > mcc::static_bin_max_keys()) return MCC_ERR_TOO_LARGE;
    if (stream) {  // the counters' address is the current device's: the stream must run there
        int sdev = -1, cur = -1;
        if (cudaStreamGetDevice(S(stream), &sdev) != cudaSuccess || cudaGetDevice(&cur) != cudaSuccess)
            return MCC_ERR_CUDA;
        if (sdev != cur) return MCC_ERR_INVALID_ARG;
    }
    return cuda_status(mcc::launch_bin_static(cell, species, n, n_cells, n_species, perm_out, offsets_out,
                                              S(stream)));
}

int mcc_species_moments(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells,
                        int32_t n_species, const mcc_species* sp, int32_t relativistic, double c,
                        const int32_t* fail_count, double* out, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_species_moments");
    if (!ctx || !P || !offsets || !sp || !out || n_cells < 0 || n_species < 1 || n_species > MCC_MAX_SPECIES)
        return MCC_ERR_INVALID_ARG;
    if (P->prec != MCC_F64 && P->prec != MCC_F32_MIXED) return MCC_ERR_INVALID_ARG;
    if (P->n > 0 && (!P->vx || !P->vy || !P->vz || !P->w)) return MCC_ERR_INVALID_ARG;
    if (relativistic && !(c > 0.0 && std::isfinite(c))) return MCC_ERR_INVALID_ARG;
    mcc::SpeciesConst sc;
    for (int s = 0; s < MCC_MAX_SPECIES; ++s) sc.m[s] = 0.0;
    for (int s = 0; s < n_species; ++s) {
        if (!(sp[s].m > 0.0) || !std::isfinite(sp[s].m)) return MCC_ERR_INVALID_ARG;
        sc.m[s] = sp[s].m;
    }
    DeviceGuard g(ctx->device);
    const cudaError_t e = mcc::launch_species_moments(P->prec == MCC_F32_MIXED, P->vx, P->vy, P->vz, P->w, offsets,
                                                      n_cells, n_species, sc, relativistic != 0, c, fail_count, out,
                                                      ctx->num_sms, S(stream));
    ctx->launches += 1;
    return cuda_status(e);
}

int mcc_gather(const void* in, const int32_t* perm, int64_t n, int32_t elem_bytes, void* out, mcc_stream stream)
{
    if (n < 0 || (elem_bytes != 4 && elem_bytes != 8) || (n > 0 && (!in || !perm || !out))) return MCC_ERR_INVALID_ARG;
    return cuda_status(mcc::launch_gather(in, perm, n, elem_bytes, out, S(stream)));
}

int mcc_gather_n(const void* const* in, void* const* out, const int32_t* elem_bytes, int32_t n_arrays,
                 const int32_t* perm, int64_t n, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_gather_n");
    if (n < 0 || n_arrays < 1 || n_arrays > MCC_MAX_GATHER || !in || !out || !elem_bytes) return MCC_ERR_INVALID_ARG;
    for (int j = 0; j < n_arrays; ++j) {
        if (elem_bytes[j] != 4 && elem_bytes[j] != 8) return MCC_ERR_INVALID_ARG;
        if (n > 0 && (!in[j] || !out[j])) return MCC_ERR_INVALID_ARG;
    }
    if (n > 0 && !perm) return MCC_ERR_INVALID_ARG;
    return cuda_status(mcc::launch_gather_n(in, out, elem_bytes, n_arrays, perm, n, S(stream)));
}

int mcc_push(const mcc_particles* P, void* x, void* y, void* z, const mcc_grid* grid, double dt,
             int32_t relativistic, double c, int32_t* cell_out, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_push");
    if (!P || !grid || P->n < 0 || (P->prec != MCC_F64 && P->prec != MCC_F32_MIXED)) return MCC_ERR_INVALID_ARG;
    if (relativistic != 0 && relativistic != 1) return MCC_ERR_INVALID_ARG;
    const int32_t nc[3] = {grid->nx, grid->ny, grid->nz};
    const double l[3] = {grid->lx, grid->ly, grid->lz};
    int64_t cells = 1;
    for (int d = 0; d < 3; ++d) {
        if (nc[d] < 1 || !(l[d] > 0.0) || !std::isfinite(l[d])) return MCC_ERR_INVALID_ARG;
        cells *= nc[d];
        if (cells > INT32_MAX) return MCC_ERR_INVALID_ARG;
    }
    if (!std::isfinite(dt) || (relativistic && !(c > 0.0 && std::isfinite(c)))) return MCC_ERR_INVALID_ARG;
    if (P->n == 0) return MCC_OK;
    if (!P->vx || !P->vy || !P->vz || !x || !y || !z || !cell_out) return MCC_ERR_INVALID_ARG;
    mcc::PushGrid g;
    for (int d = 0; d < 3; ++d) {
        g.n[d] = nc[d];
        g.l[d] = l[d];
    }
    return cuda_status(mcc::launch_push(P->prec == MCC_F32_MIXED, relativistic != 0, x, y, z, P->vx, P->vy, P->vz,
                                        P->n, g, dt, c, cell_out, S(stream)));
}

int mcc_pair(mcc_ctx* ctx, const int64_t* offsets, int32_t n_cells, int32_t n_species, int32_t sa, int32_t sb,
             int32_t inter, uint64_t seed, uint64_t step, int32_t* pair_i, int32_t* pair_j, uint8_t* pair_flags,
             mcc_stream stream)
{
    NvtxRange nvtx_("mcc_pair");
    if (!ctx || !offsets || !pair_i || !pair_j || !pair_flags || inter < 0 || inter > 0xFFFFFF)
        return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    StepArgs a;
    const int32_t ab[2] = {sa, sb};
    mcc_params p;
    std::memset(&p, 0, sizeof p);
    p.seed = seed;
    p.step = step;
    int rc = fill_args(a, ctx, nullptr, offsets, n_cells, n_species, nullptr, nullptr, ab, 1, inter, &p);
    if (rc != MCC_OK) return rc;
    if (n_cells == 0) return MCC_OK;
    a.pair_i = pair_i;
    a.pair_j = pair_j;
    a.pair_flags = pair_flags;
    return run_split(ctx, a, false, false, mcc::kPair, S(stream));
}

int mcc_scatter(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells, int32_t n_species,
                const mcc_species* sp, const double* lnL, int32_t sa, int32_t sb, int32_t inter, const int32_t* pair_i,
                const int32_t* pair_j, const uint8_t* pair_flags, const mcc_params* p, void* backup,
                mcc_stream stream)
{
    NvtxRange nvtx_("mcc_scatter");
    if (!ctx || !P || !offsets || !sp || !lnL || !pair_i || !pair_j || !pair_flags || !backup || !valid_params(p) ||
        inter < 0 || inter > 0xFFFFFF || p->pairing != 0)
        return MCC_ERR_INVALID_ARG;
    if (P->prec != MCC_F64 && P->prec != MCC_F32_MIXED) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    StepArgs a;
    const int32_t ab[2] = {sa, sb};
    int rc = fill_args(a, ctx, P, offsets, n_cells, n_species, sp, lnL, ab, 1, inter, p);
    if (rc != MCC_OK) return rc;
    if (n_cells == 0) return MCC_OK;
    a.pair_i = const_cast<int32_t*>(pair_i);
    a.pair_j = const_cast<int32_t*>(pair_j);
    a.pair_flags = const_cast<uint8_t*>(pair_flags);
    a.backup = backup;
    return run_split(ctx, a, P->prec == MCC_F32_MIXED, p->relativistic != 0, mcc::kScatter, S(stream));
}

int mcc_correct(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells, int32_t n_species,
                const mcc_species* sp, int32_t sa, int32_t sb, int32_t inter, const mcc_params* p,
                const void* backup, int32_t* corr_pairs_out, int32_t* fail_flags_out, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_correct");
    if (!ctx || !P || !offsets || !sp || !backup || !valid_params(p) || inter < 0 || inter > 0xFFFFFF)
        return MCC_ERR_INVALID_ARG;
    if (P->prec != MCC_F64 && P->prec != MCC_F32_MIXED) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    StepArgs a;
    const int32_t ab[2] = {sa, sb};
    int rc = fill_args(a, ctx, P, offsets, n_cells, n_species, sp, nullptr, ab, 1, inter, p);
    if (rc != MCC_OK) return rc;
    if (n_cells == 0) return MCC_OK;
    a.backup = const_cast<void*>(backup);
    a.corr_pairs = corr_pairs_out;
    a.fail_count = fail_flags_out;
    return run_split(ctx, a, P->prec == MCC_F32_MIXED, p->relativistic != 0, mcc::kCorrect, S(stream));
}

namespace {
// Workspace of mcc_step_fused: the cell order (n_cells int32), the class bounds and queue counters of the group
// kernels, then, when some cell exceeds the largest group class, one slab per resident CTA of the one-CTA kernel.
size_t order_bytes(int32_t n_cells) { return ((size_t)n_cells * sizeof(int32_t) + 255) & ~(size_t)255; }
// class_off [2 kOrderClasses], queues [kOrderClasses] and the order's bins, int32
constexpr size_t kCtrlHist = 256;
size_t ctrl_bytes() { return kCtrlHist + ((mcc::group_order_hist_bytes() + 255) & ~(size_t)255); }

int tile_of(const mcc_ctx* ctx, bool f32)
{
    const size_t capmax = max_tile_particles(ctx, f32);
    return ctx->tile_cap > 0 ? (int)((size_t)ctx->tile_cap < capmax ? (size_t)ctx->tile_cap : capmax)
                             : auto_tile(ctx, f32);
}

size_t slab_stride_of(int32_t max_cell, bool f32)
{
    return ((size_t)max_cell * mcc::tile_bytes_per_particle(f32) + 255) & ~(size_t)255;
}

size_t group_static_smem(const mcc_ctx* ctx, bool f32, bool rel, int cls) { return f32 ? ctx->group_static[rel][cls] : 0; }

// Shared memory one CTA of the group kernels may take for its groups: its share of the SM (kGroupWarpsPerSm warps in CTAs
// of group_cta_warps).
size_t group_budget(const mcc_ctx* ctx, bool f32, bool rel, int cls)
{
    size_t b = ctx->smem_per_sm / (mcc::kGroupWarpsPerSm / mcc::group_cta_warps(rel));
    b = b > ctx->smem_reserved ? b - ctx->smem_reserved : 0;
    if (b > ctx->smem_optin) b = ctx->smem_optin;
    const size_t st = group_static_smem(ctx, f32, rel, cls);
    return b > st ? b - st : 0;
}

// Groups of one CTA of class cls with tiles of cap particles: group_cta_warps warps, or as many groups as fit.
int groups_per_cta(const mcc_ctx* ctx, bool f32, bool rel, int cls, int cap)
{
    const int most = 32 * mcc::group_cta_warps(rel) / mcc::group_threads(cls);
    const int fit = (int)(group_budget(ctx, f32, rel, cls) / mcc::group_smem(mcc::group_shared_bytes(cls), cap));
    const int g = fit < most ? fit : most;
    return g > 1 ? g : 1;
}

// Capacity (particles) of each group size class. Class k runs 32 << k threads and holds cells of up to
// per_warp << k particles, so that the shared memory per thread is the same in every class; the largest class
// takes up to what one CTA's shared memory holds, unless the capacity is set explicitly.
void group_caps(const mcc_ctx* ctx, bool f32, bool rel, int32_t caps[mcc::kGroupClasses])
{
    if (!f32) {  // FP64: every cell on the one-CTA kernel
        for (int k = 0; k < mcc::kGroupClasses; ++k) caps[k] = 0;
        return;
    }
    size_t per_warp;
    if (ctx->group_cap > 0) {
        per_warp = (size_t)ctx->group_cap;
    } else if (ctx->group_tuned > 0) {
        per_warp = (size_t)ctx->group_tuned;
    } else {
        const size_t share = (group_budget(ctx, f32, rel, 0) / mcc::group_cta_warps(rel)) & ~(size_t)15;
        const size_t fixed = mcc::group_shared_bytes(0);
        per_warp = share > fixed ? (share - fixed) / mcc::kGroupBytesPerParticle : 32;
    }
    for (int k = 0; k < mcc::kGroupClasses; ++k) {
        const size_t st = group_static_smem(ctx, f32, rel, k) + mcc::group_shared_bytes(k);
        const size_t maxp = ctx->smem_optin > st ? (ctx->smem_optin - st) / mcc::kGroupBytesPerParticle : 0;
        size_t cap = per_warp << k;
        if (k == mcc::kGroupClasses - 1) cap = ctx->group_top > 0 ? (size_t)ctx->group_top : maxp;
        if (cap > maxp) cap = maxp;
        if (cap > 65535) cap = 65535;  // cell-local indices are 16-bit
        caps[k] = (int32_t)cap;
    }
}
static_assert(MCC_SMALL_CELL == mcc::kHalfCells, "the header's small cells are those of the half warps");
// A call with few cells runs them on larger groups, as long as every warp is still resident: one visit is then shorter, and
// one launch serves what would be several (the classes run one after another). Cells go up to class 3; class k is taken
// while n_cells groups of it fit the GPU. Measured per step, 152 SMs, two species (us by group size 64 / 128 / 256 / 512):
// 100 cells of 300: 43.6 / 35.2 / 32.8 / 36.2; 100 of 1000: 84.8 / 54.6 / 42.9 / 43.3; 600 of 300: 47.4 / 44.3 / 68 / 134;
// 1200 of 300: 56.7 / 85 / 130 / 262. Not on more threads than half the largest cell's particles: 500 three-species
// cells of 50 take 133 us per call with one-warp groups and 142 with 128 threads.
void few_cells_caps(const mcc_ctx* ctx, int32_t n_cells, int32_t max_cell, int32_t caps[mcc::kGroupClasses])
{
    int k = 0;
    while (k < 3 && ((int64_t)n_cells << (k + 1)) <= (int64_t)mcc::kGroupWarpsPerSm * ctx->num_sms && (128 << k) <= max_cell)
        ++k;
    for (int j = 0; j < k; ++j) caps[j] = -1;  // not even empty cells
}
}  // namespace

int mcc_step_workspace_size(mcc_ctx* ctx, int32_t prec, int32_t n_cells, int32_t max_cell, size_t* bytes)
{
    if (!ctx || !bytes || max_cell < 0 || n_cells < 0 || (prec != MCC_F64 && prec != MCC_F32_MIXED))
        return MCC_ERR_INVALID_ARG;
    if (max_cell > MCC_MAX_SEGMENT) return MCC_ERR_TOO_LARGE;
    const bool f32 = prec == MCC_F32_MIXED;
    int32_t caps[mcc::kGroupClasses];
    group_caps(ctx, f32, false, caps);
    int32_t caps_rel[mcc::kGroupClasses];
    group_caps(ctx, f32, true, caps_rel);
    const int32_t top = caps[mcc::kGroupClasses - 1] < caps_rel[mcc::kGroupClasses - 1]
                            ? caps[mcc::kGroupClasses - 1]
                            : caps_rel[mcc::kGroupClasses - 1];
    size_t total = order_bytes(n_cells) + ctrl_bytes();
    if (max_cell > top && max_cell > tile_of(ctx, f32))
        total += slab_stride_of(max_cell, f32) * (size_t)ctx->num_sms * kMaxCtasPerSm;
    *bytes = total;
    return MCC_OK;
}

int mcc_set_group_capacity(mcc_ctx* ctx, int32_t particles_per_warp, int32_t largest)
{
    if (!ctx || particles_per_warp < 0 || largest < 0) return MCC_ERR_INVALID_ARG;
    ctx->group_cap = particles_per_warp;
    ctx->group_top = largest;
    ctx->group_tuned = 0;
    return MCC_OK;
}

int mcc_tune_group_capacity(mcc_ctx* ctx, int32_t particles_per_warp)
{
    if (!ctx || particles_per_warp < 0) return MCC_ERR_INVALID_ARG;
    ctx->group_cap = 0;
    ctx->group_top = 0;
    ctx->group_tuned = particles_per_warp;
    return MCC_OK;
}

int mcc_group_capacities(mcc_ctx* ctx, int32_t prec, int32_t relativistic, int32_t* caps_out)
{
    if (!ctx || !caps_out || (prec != MCC_F64 && prec != MCC_F32_MIXED)) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    group_caps(ctx, prec == MCC_F32_MIXED, relativistic != 0, caps_out);
    return MCC_OK;
}

int mcc_step_fused(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells, int32_t n_species,
                   const mcc_species* sp, const double* lnL, const int32_t* interactions, int32_t n_inter,
                   const mcc_params* p, int32_t n_steps, int32_t max_cell, int32_t* corr_pairs, int32_t* fail_count,
                   void* ws, size_t ws_bytes, mcc_stream stream)
{
    return mcc_step_fused_part(ctx, P, offsets, n_cells, n_species, sp, lnL, interactions, n_inter, p, n_steps, max_cell,
                               corr_pairs, fail_count, ws, ws_bytes, 0, 0, stream);
}

int mcc_step_fused_part(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells, int32_t n_species,
                        const mcc_species* sp, const double* lnL, const int32_t* interactions, int32_t n_inter,
                        const mcc_params* p, int32_t n_steps, int32_t max_cell, int32_t* corr_pairs, int32_t* fail_count,
                        void* ws, size_t ws_bytes, int32_t whole_cells, int32_t whole_small, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_step_fused");
    if (!ctx || !P || !offsets || !sp || !lnL || !interactions || !valid_params(p) || n_steps < 0 || max_cell < 0)
        return MCC_ERR_INVALID_ARG;
    if (P->prec != MCC_F64 && P->prec != MCC_F32_MIXED) return MCC_ERR_INVALID_ARG;
    if (max_cell > MCC_MAX_SEGMENT) return MCC_ERR_TOO_LARGE;  // in-cell indices are 20-bit key fields
    const bool part = whole_cells != 0;
    if (part && (whole_cells < n_cells || whole_small < 0 || whole_small > whole_cells)) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    StepArgs a;
    int rc = fill_args(a, ctx, P, offsets, n_cells, n_species, sp, lnL, interactions, n_inter, 0, p);
    if (rc != MCC_OK) return rc;
    if (n_cells == 0 || n_steps == 0) return MCC_OK;
    // cells by whose number the call picks its groups
    const int32_t pick_cells = part ? whole_cells : n_cells;
    a.corr_pairs = corr_pairs;
    a.fail_count = fail_count;
    a.resid = p->residual;
    a.max_cell = max_cell;
    const bool f32 = P->prec == MCC_F32_MIXED;
    const bool rel = p->relativistic != 0;
    size_t need = 0;
    mcc_step_workspace_size(ctx, P->prec, n_cells, max_cell, &need);
    if (!ws || ws_bytes < need) return MCC_ERR_WORKSPACE;
    int32_t caps[mcc::kGroupClasses];
    group_caps(ctx, f32, rel, caps);
    if (ctx->group_cap == 0) few_cells_caps(ctx, pick_cells, max_cell, caps);
    // two small cells to a warp, with automatic capacities, if they fill every warp's halves (a launch of its own costs the
    // time of a visit, 0.1 ms)
    int32_t half_min = 2 * mcc::kGroupWarpsPerSm * ctx->num_sms;
    if (!f32 || ctx->group_cap > 0 || caps[0] < mcc::kHalfCells || pick_cells < half_min) half_min = 0;
    // (the device counts the small cells of a whole problem; for a part the caller has)
    if (part && half_min > 0) half_min = whole_small >= half_min ? 1 : 0;
    // the group kernels serve the mixed path; the FP64 path runs every cell on the one-CTA kernel
    const bool fallback = !f32 || max_cell > caps[mcc::kGroupClasses - 1];
    int32_t* order = reinterpret_cast<int32_t*>(ws);
    int32_t* class_off = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(ws) + order_bytes(n_cells));
    int32_t* queues = class_off + 2 * mcc::kOrderClasses;
    // cells by size class, largest first (the order is the same for every step of the call)
    int32_t* hist = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(class_off) + kCtrlHist);
    if (cudaMemsetAsync(class_off, 0, kCtrlHist + mcc::group_order_hist_bytes(), S(stream)) != cudaSuccess)
        return MCC_ERR_CUDA;
    if (mcc::launch_group_order(offsets, n_cells, n_species, caps, half_min, order, class_off, hist, &ctx->launches, S(stream)) !=
        cudaSuccess)
        return MCC_ERR_CUDA;
    a.order = order;
    a.class_off = class_off;
    a.queues = queues;
    a.step_dev = p->step_device;
    // the one-CTA kernel takes the cells above every class from the order's first range
    const int tile = tile_of(ctx, f32);
    int max_grid = 1 << 30;
    StepArgs big = a;
    if (fallback) {
        big.order_range = class_off + 2 * mcc::kGroupClasses;
        if (max_cell > tile) {
            big.slab = reinterpret_cast<char*>(ws) + order_bytes(n_cells) + ctrl_bytes();
            big.slab_stride = (int64_t)slab_stride_of(max_cell, f32);
            big.slab_cap = max_cell;
            max_grid = (int)((ws_bytes - order_bytes(n_cells) - ctrl_bytes()) / (size_t)big.slab_stride);
        }
    }
    // under stream capture the marks become event-record nodes of the graph, so that a replay records them too
    unsigned rec_flags = cudaEventRecordDefault;
    if (p->launch_events) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(S(stream), &cs) != cudaSuccess) return MCC_ERR_CUDA;
        if (cs == cudaStreamCaptureStatusActive) rec_flags = cudaEventRecordExternal;
    }
    // one launch of a size class with tiles of cap particles
    bool after = false;  // the launch before is a class of this step
    auto run_class = [&](int cls, int32_t cap) -> int {
        // Fewer cells than groups: spread them over the SMs. Up to four groups per SM get a CTA each: so few warps fetch little,
        // and in lockstep each waits for the slowest (us per call, in a CTA per SM / a CTA each: 600 relativistic beam cells
        // 368 / 315, 500 three-species cells of 100 126 / 121; 1200 cells of 50, eight per SM, 152 / 205).
        const int per_sm = (n_cells + ctx->num_sms - 1) / ctx->num_sms;
        int groups = groups_per_cta(ctx, f32, rel, cls, cap);
        if (groups > per_sm) groups = per_sm;
        if (per_sm <= 4) groups = 1;
        const size_t smem = (size_t)groups * mcc::group_smem(mcc::group_shared_bytes(cls), cap);
        const int bps = cached_occupancy(ctx->group_occ[rel][cls], ((uint64_t)smem << 6) | (uint64_t)groups, [&] {
            int b = 0;
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, mcc::group_kernel(f32, rel, cls),
                                                                 groups * mcc::group_threads(cls), smem) == cudaSuccess
                       ? b
                       : 0;
        });
        if (bps < 1) return MCC_ERR_CUDA;
        int grid = bps * ctx->num_sms;
        if (grid > n_cells) grid = n_cells;
        a.gcls = cls;
        a.gcap = cap;
        const cudaError_t e = mcc::launch_group(f32, rel, cls, a, grid, groups, smem, after, S(stream));
        after = !p->launch_events;  // (an event between two kernels orders them)
        ctx->launches += 1;
        return e == cudaSuccess ? MCC_OK : MCC_ERR_CUDA;
    };
    for (int32_t t = 0; t < n_steps; ++t) {
        a.rng.step = (uint32_t)(p->step + (uint64_t)t);
        a.step_add = (uint32_t)t;
        // (the first step's queues are zero)
        if (t > 0 && cudaMemsetAsync(queues, 0, sizeof(int32_t) * mcc::kOrderClasses, S(stream)) != cudaSuccess)
            return MCC_ERR_CUDA;
        cudaEvent_t* ev = (p->launch_events && t == n_steps - 1) ? reinterpret_cast<cudaEvent_t*>(p->launch_events)
                                                                   : nullptr;
        auto mark = [&](int k, int end) {
            if (ev) cudaEventRecordWithFlags(ev[2 * k + end], S(stream), rec_flags);
        };
        mark(mcc::kGroupClasses, 0);
        if (fallback) {
            big.rng.step = a.rng.step;
            big.step_add = a.step_add;
            const int cap = max_cell <= tile ? max_cell : tile;
            const bool small = !f32 && max_cell <= mcc::kSmallCells && pick_cells > 4 * ctx->num_sms;
            rc = run_cells(ctx, big, f32, rel, small ? mcc::kFusedSmall : mcc::kFused, cap, S(stream), max_grid);
            if (rc != MCC_OK) return rc;
        }
        mark(mcc::kGroupClasses, 1);
        after = false;
        for (int cls = mcc::kGroupClasses - 1; cls >= 0; --cls) {
            mark(cls, 0);
            // no cell can be in this class
            if (!f32 || caps[cls] < 0 || (cls > 0 && caps[cls - 1] >= max_cell)) {
                mark(cls, 1);
                continue;
            }
            rc = run_class(cls, caps[cls]);
            if (rc == MCC_OK && cls == 0 && half_min > 0)
                rc = run_class(mcc::kHalfClass, max_cell < mcc::kHalfCells ? max_cell : mcc::kHalfCells);
            if (rc != MCC_OK) return rc;
            mark(cls, 1);
        }
    }
    if (p->step_device) {
        if (mcc::launch_step_advance(p->step_device, (uint64_t)n_steps, S(stream)) != cudaSuccess) return MCC_ERR_CUDA;
        ctx->launches += 1;
    }
    return MCC_OK;
}

int mcc_adjoint_workspace_size(mcc_ctx* ctx, int32_t n_cells, int32_t max_cell, int32_t max_corr_passes,
                               size_t* bytes)
{
    if (!ctx || !bytes || n_cells < 0 || max_cell < 0 || max_corr_passes < 0) return MCC_ERR_INVALID_ARG;
    if (max_cell > MCC_MAX_SEGMENT) return MCC_ERR_TOO_LARGE;
    const int32_t mc = max_cell > 0 ? max_cell : 1;
    const int32_t ep = max_corr_passes * (mc / 2 + 1) + 1;
    const size_t slab = mcc::adjoint_slab_bytes(mc, ep, adjoint_on_chip(ctx, mc));
    *bytes = slab * (size_t)adjoint_grid(ctx, n_cells, mc, slab);
    return MCC_OK;
}

int mcc_adjoint_tape_size(mcc_ctx* ctx, int32_t n_cells, int32_t max_cell, int32_t max_corr_passes, size_t* bytes)
{
    if (!ctx || !bytes || n_cells < 0 || max_cell < 0 || max_corr_passes < 0) return MCC_ERR_INVALID_ARG;
    if (max_cell > MCC_MAX_SEGMENT) return MCC_ERR_TOO_LARGE;
    const int32_t mc = max_cell > 0 ? max_cell : 1;
    const int32_t ep = max_corr_passes * (mc / 2 + 1) + 1;
    *bytes = mcc::adjoint_slab_bytes(mc, ep, adjoint_on_chip(ctx, mc)) * (size_t)(n_cells > 0 ? n_cells : 1);
    return MCC_OK;
}

int mcc_adjoint(mcc_ctx* ctx, const mcc_particles* P, const int64_t* offsets, int32_t n_cells, int32_t n_species,
                const mcc_species* sp, const double* lnL, int32_t sa, int32_t sb, int32_t inter, const mcc_params* p,
                int32_t max_cell, double* vx_out, double* vy_out, double* vz_out, double* gvx, double* gvy,
                double* gvz, double* gw, double* glnL, int32_t tape, void* ws, size_t ws_bytes, mcc_stream stream)
{
    NvtxRange nvtx_("mcc_adjoint");
    if (!ctx || !P || !offsets || !sp || !lnL || !valid_params(p) || inter < 0 || inter > 0xFFFFFF || max_cell < 0)
        return MCC_ERR_INVALID_ARG;
    if (max_cell > MCC_MAX_SEGMENT) return MCC_ERR_TOO_LARGE;
    if (P->prec != MCC_F64 || p->relativistic || p->weighting != 0 || p->pairing != 0) return MCC_ERR_INVALID_ARG;
    const bool fwd = vx_out || vy_out || vz_out, rev = gvx || gvy || gvz;
    if (fwd && !(vx_out && vy_out && vz_out)) return MCC_ERR_INVALID_ARG;
    if (rev && !(gvx && gvy && gvz && gw && glnL)) return MCC_ERR_INVALID_ARG;
    if (tape < MCC_ADJOINT_RECOMPUTE || tape > MCC_ADJOINT_REPLAY || (tape == MCC_ADJOINT_REPLAY && fwd))
        return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    StepArgs a;
    const int32_t ab[2] = {sa, sb};
    int rc = fill_args(a, ctx, P, offsets, n_cells, n_species, sp, lnL, ab, 1, inter, p);
    if (rc != MCC_OK) return rc;
    if (n_cells == 0 || (!fwd && !rev)) return MCC_OK;
    size_t need = 0;
    if (tape == MCC_ADJOINT_RECOMPUTE) mcc_adjoint_workspace_size(ctx, n_cells, max_cell, p->max_corr_passes, &need);
    else mcc_adjoint_tape_size(ctx, n_cells, max_cell, p->max_corr_passes, &need);
    if (!ws || ws_bytes < need) return MCC_ERR_WORKSPACE;
    const int32_t mc = max_cell > 0 ? max_cell : 1;
    const int32_t ep = p->max_corr_passes * (mc / 2 + 1) + 1;
    const bool on_chip = adjoint_on_chip(ctx, mc);
    const size_t slab = tape == MCC_ADJOINT_RECOMPUTE ? mcc::adjoint_slab_bytes(mc, ep, on_chip) : 0;
    const cudaError_t e = mcc::launch_adjoint(a, lnL[sa * n_species + sb], vx_out, vy_out, vz_out, gvx, gvy, gvz, gw,
                                              glnL, reinterpret_cast<char*>(ws), mc, ep, tape, on_chip,
                                              adjoint_grid(ctx, n_cells, mc, slab), S(stream));
    ctx->launches += 1;
    return cuda_status(e);
}

int mcc_sync_status(mcc_ctx* ctx, mcc_stream stream)
{
    if (!ctx) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    if (cudaStreamSynchronize(S(stream)) != cudaSuccess) return MCC_ERR_CUDA;
    int32_t st = 0;
    if (cudaMemcpy(&st, ctx->dbuf, sizeof st, cudaMemcpyDeviceToHost) != cudaSuccess) return MCC_ERR_CUDA;
    if (cudaMemset(ctx->dbuf, 0, sizeof(int32_t)) != cudaSuccess) return MCC_ERR_CUDA;
    return st;
}

int64_t mcc_launch_count(mcc_ctx* ctx) { return ctx ? ctx->launches : -1; }

int mcc_debug_record(mcc_ctx* ctx, mcc_stream stream, int32_t* out)
{
    if (!ctx || !out) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    if (cudaStreamSynchronize(S(stream)) != cudaSuccess) return MCC_ERR_CUDA;
    if (cudaMemcpy(out, ctx->dbuf + 4, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess) return MCC_ERR_CUDA;
    if (cudaMemset(ctx->dbuf + 4, 0, 4 * sizeof(int32_t)) != cudaSuccess) return MCC_ERR_CUDA;
    return MCC_OK;
}

int mcc_phase_clocks(mcc_ctx* ctx, mcc_stream stream, uint64_t* out)
{
    if (!ctx || !out) return MCC_ERR_INVALID_ARG;
    DeviceGuard g(ctx->device);
    if (cudaStreamSynchronize(S(stream)) != cudaSuccess) return MCC_ERR_CUDA;
    char* p = reinterpret_cast<char*>(ctx->dbuf) + kClkOffset;
    if (cudaMemcpy(out, p, kClkWords * sizeof(uint64_t), cudaMemcpyDeviceToHost) != cudaSuccess) return MCC_ERR_CUDA;
    if (cudaMemset(p, 0, kClkWords * sizeof(uint64_t)) != cudaSuccess) return MCC_ERR_CUDA;
    return MCC_OK;
}

int mcc_phase_clocks_build(void)
{
#ifdef MCC_PHASE_CLOCKS
    return 1;
#else
    return 0;
#endif
}

int mcc_debug_bounds_build(void)
{
#ifdef MCC_DEBUG_BOUNDS
    return 1;
#else
    return 0;
#endif
}

int mcc_set_tile_cap(mcc_ctx* ctx, int32_t cap)
{
    if (!ctx || cap < 0) return MCC_ERR_INVALID_ARG;
    ctx->tile_cap = cap;
    return MCC_OK;
}

const char* mcc_status_string(int status)
{
    switch (status) {
    case MCC_OK: return "ok";
    case MCC_ERR_INVALID_ARG: return "invalid argument";
    case MCC_ERR_CUDA: return "CUDA error";
    case MCC_ERR_WORKSPACE: return "workspace missing or too small";
    case MCC_ERR_TIMEOUT: return "bounded wait timed out";
    case MCC_ERR_CORRECTION_FAILED: return "energy correction could not absorb the violation";
    case MCC_ERR_BOUNDS: return "index or cell size out of bounds";
    case MCC_ERR_TOO_LARGE: return "segment larger than supported";
    default: return "unknown status";
    }
}

}  // extern "C"
