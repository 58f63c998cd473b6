// cg_internal.cuh -- internal declarations of the GB300 coupling library.
//
// Shared by the .cu files of the library only (never by the oracle).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>
#include <vector>

#include "../../include/cg.h"

namespace cg {

// One-time settings that the CUDA runtime keeps per device (kernel
// attributes such as the dynamic shared-memory limit): f runs once on each
// device, the first time a call is made with that device current, under a
// lock; a failure is returned and retried on the next call.
struct PerDeviceOnce {
    std::mutex mu;
    bool done[64] = {};
};

template <typename F>
inline cg_status once_per_device(PerDeviceOnce& o, F f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return CG_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(o.mu);
    if (o.done[dev]) return CG_OK;
    const cg_status s = f();
    if (s == CG_OK) o.done[dev] = true;
    return s;
}

// ----------------------------------------------------------------------
// Sizes
// ----------------------------------------------------------------------
constexpr int kSortThreads = 512;                   // threads of a sort tile
constexpr int kSortItems = 8;                       // items per thread
constexpr int kSortTile = kSortThreads * kSortItems; // 4096 particles per tile
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxDigitBits = 11;                   // widest radix digit of one pass
constexpr int kMaxPasses = 3;
constexpr int kMaxBulkBits = 2 * kMaxDigitBits;     // two passes -> 2^22 cells
constexpr int kScanItems = 4096;                    // elements per scan block
// per-cell sort
constexpr int kKeyThreads = 256;                    // threads of its key kernel
constexpr int kKeyItems = 4;                        // particles per thread of the key kernel
constexpr int kPlaceItems = 4;                      // particles per thread of the placement
constexpr int kSegSortWarps = 8;                    // warps of a per-cell sort CTA
constexpr int kGroupCells = 8;                      // consecutive cells a warp takes at a time
constexpr int kWarpStage = 1024;                    // ids of a group staged in the warp's shared memory
constexpr int kSegWarpMax = 256;                    // largest cell a warp sorts in registers
// Split of a key of `bits` bits into the fewest passes of at most `digits`
// bits (at most kMaxPasses; wider only when the key needs it), the low
// digits first.  digits 0 takes the default: narrow digits (8) for grids of
// 2^20 cells and more, whose particles are usually far from cell order and
// whose scatters then profit from long digit runs (three passes measured
// faster on the 32M-particle clustered bed), wide ones (10) below (two
// passes measured faster on the 4M-particle packed bed).  Returns the passes.
inline int split_passes(int bits, int (&pb)[kMaxPasses], int digits = 0) {
    const int D = digits > 0 ? digits : (bits >= 20 ? 8 : 10);
    int np = (bits + D - 1) / D;
    np = np < 1 ? 1 : (np > kMaxPasses ? kMaxPasses : np);
    for (int i = 0; i < kMaxPasses; ++i) pb[i] = i < np ? bits / np + (i < bits % np ? 1 : 0) : 0;
    return np;
}

// cg_grid_desc.sort_digits: automatic, per-cell sort, or a digit width.
inline bool sort_choice_valid(int v) { return v == CG_SORT_AUTO || v == CG_SORT_CELLS || (v >= 6 && v <= kMaxDigitBits); }
// The per-cell sort serves a call of n particles over nbulk cells.
inline bool use_cell_sort(int v, long long n, long long nbulk) {
    return v == CG_SORT_CELLS ||
           (v == CG_SORT_AUTO && n <= CG_SORT_CELLS_AUTO_MAX && n <= (long long)CG_SORT_CELLS_AUTO_DENSITY * nbulk);
}

// Dynamic shared memory of a sort scatter pass with 2^bits digits: the
// per-warp counters, or the staged tile (key, id, diameter of T), whichever
// is larger, plus two [2^bits] int arrays.
__host__ __device__ constexpr size_t scatter_smem_bytes(int bits, size_t tsize) {
    return ((size_t)kSortWarps * sizeof(int) << bits) > (size_t)kSortTile * (8 + tsize)
               ? (((size_t)kSortWarps * sizeof(int) << bits) + (2 * sizeof(int) << bits))
               : ((size_t)kSortTile * (8 + tsize) + (2 * sizeof(int) << bits));
}
constexpr int kNumSlots = 16;                       // status counters

// Status word slots (unsigned long long each).
enum { ST_FLAGS = 0, ST_OUTSIDE = 1, ST_NONFINITE = 2, ST_CLAMPED = 3, ST_TIMEOUT = 4, ST_FALLBACK = 5 };

// Partial-sum regions of the conservation sums.
// The projection's region holds six columns: sum S_f V_f (3), then sum S_B
// V_B (3) of the source it reads.
enum { PS_VOL = 0, PS_DRAG = 1, PS_PROJ = 2, PS_NREG = 3 };
constexpr int kDragLaneSums = 8;              // V_p, F(3), |F|, m u (3)
constexpr int kDragSums = kDragLaneSums + 1;   // + the clamped count

// ----------------------------------------------------------------------
// Device-side view of the grid geometry (passed by value to kernels)
// ----------------------------------------------------------------------
struct GridDev {
    int nb[3];          // bulk cells per axis
    int nf[3];          // fine cells per axis
    int r;              // coarsening ratio
    long long nbulk, nfine;
    double x0[3];       // origin
    double xhi[3];      // origin + extent
    double H[3];        // bulk spacing (L / nb, rounded to double)
    double invH[3];     // 1 / H (double)
    double VB, invVB, Vf;
    // float versions for the FP32 path
    float x0f[3];       // (float)x0
    float xhif[3];      // (float)xhi
    float invHf[3];     // (float)(1/H)
    float binh[3];      // 1/2 - 2^-21 |x0 / H| - 2^-24: how near a cell's middle the float bin rule decides (bin_axis_fast)
    float vch, vcl;     // pi / (6 V_B) as float-float: a sphere's volume over V_B is this times d^3
    double vcd;         // pi / (6 V_B)
    float x0h[3], x0l[3];   // x0 as float-float
    float ihh[3], ihl[3];   // 1/H as float-float
    float xbh[3], xbl[3];   // -(x0 / H + 1/2) as float-float: the lattice coordinate is x / H + xb
    float topf[3];      // n_b - 2
    float invVBf, VBf, Vff;
    float VBh, VBl, Vfh, Vfl;   // V_B, V_f as float-float
    // physics
    int law, interp;
    double rho_f, mu_f, rho_p, eps_switch, eps_min, g[3];
};

// ----------------------------------------------------------------------
// Handle
// ----------------------------------------------------------------------
struct ProfSlot {
    std::string name;
    long long launches = 0;
    double total_ms = 0.0;
};

struct PendingEv {
    int slot;
    int ev;   // index into the event pool (start = 2 ev, stop = 2 ev + 1)
};

struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
};

// Device staging of one host-buffer step: inputs, outputs, and the events
// that order its copies and compute against the next use of the same set.
struct HostStage {
    DevBuf pos, vel, ufine, eps, ub, var, Sb, F, Sf, epsf, sums, cell, perm, cs;
    cudaEvent_t in_done = nullptr, comp_done = nullptr, out_done = nullptr;
    bool used = false;
};

}  // namespace cg

struct cg_grids {
    cg_grid_desc desc;
    cg::GridDev gd;
    int fp64 = 0;
    size_t tsize = 4;          // bytes of T
    cudaStream_t stream = nullptr;
    int device = 0;
    int num_sms = 148;
    int bulk_bits = 0, pass_bits[cg::kMaxPasses] = {0, 0, 0}, npasses = 1;

    // binning state
    long long n_binned = -1;
    long long cap = -1;        // particle capacity of the particle buffers

    // particle-sized buffers
    int32_t* key = nullptr;        // [cap] cell per particle (caller order)
    int32_t* key1 = nullptr;       // [cap] keys after pass 1
    int32_t* val1 = nullptr;       // [cap] particle ids after pass 1
    int32_t* key2 = nullptr;       // [cap] keys after pass 2 of three
    int32_t* val2 = nullptr;       // [cap] particle ids after pass 2 of three
    int32_t* perm = nullptr;       // [cap] particle ids in cell order
    int32_t* key_sorted = nullptr; // [cap] cell of each slot of the sorted order
    int32_t* inv_perm = nullptr;   // [cap] sorted slot of each particle
    void* vol = nullptr;           // [cap] T particle diameter, caller order (for the volume deposit)
    void* vol_sorted = nullptr;    // [cap] T particle diameter, sorted order
    void* Fs = nullptr;            // [cap] T4 drag force, sorted order
    bool key_valid = false;        // key holds the binning's caller-order cells (see copy_cells)
    bool bin_ident = false;        // the binning of this call took the identity hint, which leaves inv_perm out
    bool ident_seen = false;       // some binning of this handle did, called or captured (see ensure_inverse)
    // incremental rebinning (rebin.cu): a binning of hint_n particles held in
    // perm / key_sorted / cell_start is where the next binning of the same
    // count starts; hint_ident is the particle array the last sorted step
    // wrote in that binning's order (so its particle i sat at old slot i)
    long long hint_n = -1;
    const void* hint_ident = nullptr;
    int32_t* rb_rid = nullptr;     // [cap] per old slot: its particle id (the caller's order kept)
    int32_t* rb_rkn = nullptr;     // [cap] per old slot: the new cell, complemented for a mover
    int4* rb_mov = nullptr;        // [rb_nblk * kRebinTile] movers, each block of old slots its own part:
                                   // (id, new cell, next mover of that cell + 1, arrival rank)
    int32_t* rb_small = nullptr;   // per-cell and per-block counts, starts, list heads; counters (rebin_ptrs)
    long long rb_nblk = 0;
    int32_t* hist = nullptr;       // [2^digit * ntiles]
    int32_t* scan_part = nullptr;  // scan block partials
    long long hist_cap = 0, scan_cap = 0;

    // bulk-sized buffers
    int32_t* cell_start = nullptr; // [nbulk + 1]
    void* bulk4 = nullptr;         // [nbulk] T4: eps, u_x, u_y, u_z
    void* eps_t = nullptr;         // [nbulk] T: porosity in the path precision
    unsigned long long* vol_acc = nullptr;   // [5 nbulk] volume accumulators (see volume_add_row)
    void* partials = nullptr;      // conservation-sum block partials: (s, c) pairs of T
    long long part_off[cg::PS_NREG] = {0, 0, 0};
    long long part_blocks[cg::PS_NREG] = {0, 0, 0};
    long long part_cap = 0;
    unsigned long long* status = nullptr;   // [kNumSlots]

    // host-buffer entries: two staging sets used in turn, and the copy
    // streams (inputs in, outputs out) that overlap consecutive steps
    cg::HostStage hs[2];
    int hs_next = 0;
    cudaStream_t h2d = nullptr, d2h = nullptr;
    // the last host step that advanced its particles in place: the event
    // after their copies back and the host arrays they went to (a later
    // host step reading those arrays waits for them)
    cudaEvent_t part_out = nullptr;
    const void* part_pos = nullptr;
    const void* part_vel = nullptr;
    cg::DevBuf fresh4;   // [nbulk] T4: (phi, u) of the fresh field of cg_mlp_features
    cg::DevBuf Bs;       // [cap] T4: (beta, beta u) in sorted order, for the semi-implicit coefficients

    // second stream of the step: fine-grid work that does not depend on the
    // particle path runs beside it (fork / join through events)
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_avg = nullptr, ev_pack = nullptr, ev_epsf = nullptr;

    // launch accounting / profiling
    long long launches = 0;
    bool prof = false;
    std::vector<cg::ProfSlot> slots;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<cg::PendingEv> pending;
    int ev_used = 0;
};

namespace cg {

// ----------------------------------------------------------------------
// Launch plumbing (api.cu)
// ----------------------------------------------------------------------
int prof_slot(cg_grids* g, const char* name);
void prof_begin(cg_grids* g, int slot, int* ev);
void prof_end(cg_grids* g, int slot, int ev);
bool injected_launch_failure();   // cg_debug_fail_launch_after

// Launch a kernel on the handle's stream, count it, time it when profiling,
// and turn a launch error into CG_ERR_CUDA.
// Launches are programmatic dependent launches: the next kernel on the
// stream may be scheduled while this one drains, and every kernel launched
// here starts with pdl_wait(), which returns once the kernels it depends on
// have completed and their memory is visible (so each kernel still sees all
// earlier work; only the launch latency overlaps).
#define CG_LAUNCH(g, name, kernel, grid, block, smem, ...)                        \
    do {                                                                         \
        int slot_ = -1, ev_ = -1;                                                \
        if ((g)->prof) {                                                         \
            slot_ = cg::prof_slot((g), (name));                                  \
            cg::prof_begin((g), slot_, &ev_);                                    \
        }                                                                        \
        cudaLaunchAttribute a_[1];                                               \
        a_[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;           \
        a_[0].val.programmaticStreamSerializationAllowed = 1;                    \
        cudaLaunchConfig_t c_ = {};                                              \
        c_.gridDim = dim3(grid);                                                 \
        c_.blockDim = dim3((unsigned)(block));                                   \
        c_.dynamicSmemBytes = (size_t)(smem);                                    \
        c_.stream = (g)->stream;                                                 \
        c_.attrs = a_;                                                           \
        c_.numAttrs = 1;                                                         \
        cudaError_t e_ = cg::injected_launch_failure() ? cudaErrorLaunchFailure  \
                                                       : cudaLaunchKernelEx(&c_, kernel, __VA_ARGS__); \
        (g)->launches++;                                                         \
        if (e_ == cudaSuccess) e_ = cudaGetLastError();                          \
        if ((g)->prof) cg::prof_end((g), slot_, ev_);                            \
        if (e_ != cudaSuccess) return CG_ERR_CUDA;                               \
    } while (0)

#define CG_CUDA(call)                                   \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return CG_ERR_CUDA;      \
    } while (0)

#define CG_TRY(call)                                    \
    do {                                                \
        cg_status s_ = (call);                          \
        if (s_ != CG_OK) return s_;                     \
    } while (0)

// ----------------------------------------------------------------------
// Step launchers (one .cu each)
// ----------------------------------------------------------------------
// Up to two independent arrays are scanned by one pair of launches: blocks
// [0, n0) cover array 0, the others array 1.
constexpr int kScanArrays = 2;
struct ScanJob {
    const int32_t* in[kScanArrays] = {};
    int32_t* out[kScanArrays] = {};
    long long m[kScanArrays] = {};
    long long nblk[kScanArrays] = {};
};

// Column map of the conservation-sum reduction: sum k merges cnt[k]
// compensated pairs starting at pair off[k] of the partials.
struct SumsMap {
    long long off[CG_NSUMS];     // first pair of the partial column, -1 = not computed
    long long cnt[CG_NSUMS];     // number of partials
};

cg_status ensure_particle_capacity(cg_grids* g, long long n);
// What the last kernel of a rebinning clears for the next one: the per-cell
// arrays (in int4) and the tile totals.
struct RebinClear {
    int4* a;
    long long na;
    int32_t* part;
    long long npart;
};
// The last kernel of a rebinning: the ids of the crowded cells, placed in val1
// from the cell starts cs, in order; cs to cs_copy; the clear.
cg_status launch_rebin_finish(cg_grids* g, const int32_t* cs, int32_t* ctr, const int4* crowd, int32_t* cs_copy,
                              int32_t* inv_perm, const RebinClear& clear);
// Incremental rebinning (rebin.cu).
// Counters: entries of the crowded cells' list, movers, finished blocks of the last
// kernel, which clears these three; whether inv_perm is not the inverse of perm, and the
// finished blocks of the kernel that makes it so.
enum { RB_CROWD = 0, RB_MOVERS = 1, RB_DONE = 2, RB_INV_STALE = 3, RB_INV_DONE = 4 };
constexpr int kRebinThreads = 256;
constexpr int kRebinItems = 4;
constexpr int kRebinTile = kRebinThreads * kRebinItems;   // old slots per block
constexpr int kRebinScan = 1024;                           // elements per block of its scans
// Arrivals of a cell whose list is walked; a cell of more is crowded.  (The bed of
// 977 per cell, 2% leaving: 4 293, 8 298, 16 312, 32 349 us; 500,000 particles in
// another order 149, 180, 258, 382 with one warp for the movers of 1024 slots; few
// movers per cell: no difference.)
constexpr int kRebinMaxArrivals = 4;
constexpr int kCrowdPart = 4096;                           // ids of a crowded cell that a warp merges
constexpr long long kRebinMaxParticles = 1LL << 30;        // the marking kernel's 32-bit slots (a longer list is sorted)
constexpr int kRebinCounters = 8;
// The small rebinning arrays each start on a 256-byte boundary (the scan reads
// them as int4): the counts (n_b + 1), the departures per block (nblk + 1), the
// arrivals with the list heads (2 (n_b + 1)), the departures per cell, the
// counters, the scans' block totals.
inline long long rebin_pad(long long ints) { return (ints + 63) / 64 * 64; }
inline long long rebin_tiles(long long m) { return (m + kRebinScan - 1) / kRebinScan; }
// Cells per thread of the pass over the cells: one, the shortest chain, except
// on larger FP64 grids, where the block's compensated sum costs more than the
// cells (128,000 cells: 17 us against 23).  Its blocks (with the end of the
// last cell).
inline int cell_items(long long nbulk, bool fp64) { return fp64 && nbulk >= (1 << 16) ? kRebinScan / 256 : 1; }
inline long long cell_blocks(long long nbulk, bool fp64) {
    const long long per = 256LL * cell_items(nbulk, fp64);
    return (nbulk + per) / per;
}
inline long long rebin_small_ints(long long nbulk, long long nblk) {
    return 4 * rebin_pad(nbulk + 1) + rebin_pad(nblk + 1) + rebin_pad(kRebinCounters) + 2 * rebin_tiles(nbulk + 1) +
           rebin_tiles(nblk + 1);
}
// Where a step wants its porosity (EpsOut), formed while binning when the
// binning is incremental; sums: also the deposited volume's partials.
struct StepEps {
    double* eps = nullptr;
    void* rec = nullptr;
    void* eps_t = nullptr;
    void* S = nullptr;
    bool sums = false;
    bool formed = false;             // set by the binning when it formed the porosity
    cudaEvent_t ready = nullptr;     // recorded (nullable) once the porosity is formed
};
// The binning of n particles from the handle's last binning of n; ident:
// the particles are that binning's sorted output (particle i at old slot i).
cg_status launch_rebin(cg_grids* g, long long n, const void* pos_d, bool ident, StepEps* eps);
// The caller-order cells of the last binning into cell_out.
cg_status copy_cells(cg_grids* g, long long n, int32_t* cell_out);
// inv_perm of the last binning.  The identity-hint rebinning leaves it out, and
// whether it did is a word on the device: what ran last may have been a
// replayed graph, which the host does not see.  A handle that never took that
// path, by a call or a capture, launches nothing.
cg_status ensure_inverse(cg_grids* g, long long n);
cg_status ensure_partials(cg_grids* g, long long n);

cg_status launch_bin(cg_grids* g, long long n, const void* pos_d, StepEps* eps = nullptr);
// Porosity of the binned particles: from the sorted diameters of a binning
// from scratch (pos_d null), or gathered from pos_d [n] T4.
cg_status launch_deposit_volume(cg_grids* g, long long n, const void* pos_d, StepEps* eps);
// Slots per chunk of the segmented sums: 256, and fewer for small particle
// counts, whose few chunks would be a chain of eight rounds on a few SMs
// (10,000 particles, FP64: the reaction 18 -> 10 us).  Chunks of 160 at 500,000
// particles would take 2 us of 23 off the sorted drag, and add a quarter to the
// reaction of a batch of such instances (52 -> 65 us).  By the particle count
// alone, so that every path over the same particles cuts them alike and gives
// the same sums.
__host__ __device__ inline int seg_chunk(long long n) {
    return n >= (1 << 17) ? 256 : n >= (1 << 16) ? 128 : n >= (1 << 15) ? 64 : 32;
}
// Threads per block of the kernels over chunks: few chunks take smaller blocks, so that
// they reach every SM (10,000 particles, FP64, blocks of 256 -> 32: 47 -> 19 us).
inline unsigned seg_threads(const cg_grids* g, long long n) {
    const long long per_sm = (n + seg_chunk(n) - 1) / seg_chunk(n) / g->num_sms;
    return per_sm < 8 ? 32 : per_sm < 16 ? 64 : per_sm < 32 ? 128 : 256;
}
// cleared: S_bulk is zero already.
cg_status launch_deposit_sorted_force(cg_grids* g, long long n, void* S_bulk, bool cleared);
// Gather the particle records into the binned order (cg_reorder_particles).
cg_status launch_reorder(cg_grids* g, long long n, const void* pos_d, const void* vel, void* pos_out, void* vel_out);
// Semi-implicit coefficients [4][n_b] (A, b) from the drag's sorted (beta, beta u) records.
cg_status launch_deposit_implicit(cg_grids* g, long long n, void* coef_bulk);
cg_status launch_deposit_momentum(cg_grids* g, long long n, const void* force_soa, void* S_bulk);
// rec (nullable): also write the mean velocity into the drag record's u part.
cg_status launch_average(cg_grids* g, const void* u_fine, void* u_bulk, void* var_bulk, void* rec = nullptr);
cg_status launch_pack(cg_grids* g, const double* eps, const void* u_bulk, bool want_eps_t);
// pos_out, vel_out (nullable, needs S_bulk): the particles, advanced when
// dt > 0, are written to these arrays in the order of the binning.
// perm_out (nullable): also gets the binning's permutation.  S_cleared: S_bulk
// is zero already.  Without pos_out, S_bulk needs inv_perm (ensure_inverse).
cg_status launch_drag(cg_grids* g, long long n, const void* pos_d, const void* vel, void* force, void* S_bulk,
                      bool sums, double dt, bool S_cleared = false, void* coef_bulk = nullptr, void* pos_out = nullptr,
                      void* vel_out = nullptr, int32_t* perm_out = nullptr);
// Learned drag (FP32 only): bulk4 must hold (phi of this step, stale u); S_bulk needs inv_perm.
cg_status launch_drag_learned(cg_grids* g, const cg_mlp* m, long long n, void* pos_d, void* vel,
                              const void* var_stale, const void* u_fine, int32_t age, void* force, void* S_bulk,
                              double dt, bool S_cleared = false);
cg_status grow_buf(DevBuf& b, size_t bytes);
// The closure's feature box (CG_MLP_NFEAT values each).
cg_status mlp_feature_box(const cg_mlp* m, float* lo, float* hi);
// The stale variance field, fine velocity and record age bound to a closure by cg_mlp_bind.
cg_status mlp_bound_inputs(const cg_mlp* m, const void** var_stale, const void** u_fine, int32_t* age);
cg_status launch_project(cg_grids* g, int ncomp, const void* const* in, void* const* out, bool sums);
// Lanes of a warp that share a bulk cell in the average: one per plane for
// FP32 r = 2 and 4, fewer values per lane where a plane would not fit the
// registers (r = 8, 64 values) or where FP64 doubles them; 1 otherwise.
__host__ __device__ constexpr int average_lanes(int r, bool fp64) {
    return r == 2 ? 2 : r == 4 ? (fp64 ? 8 : 4) : r == 8 ? (fp64 ? 32 : 16) : 1;
}
// Layers a thread of the projection walks, and its blocks of
// project_block threads per component.
int project_depth(const GridDev& g, int ncomp, bool fp64);
int project_block(const GridDev& g, int ncomp, bool fp64, int num_sms);
long long project_threads(const GridDev& g, int depth);
long long project_blocks(const GridDev& g, int ncomp, bool fp64, int num_sms);
cg_status launch_sums(cg_grids* g, double* sums);
// Sum columns of the partial regions (offsets in pairs; blocks < 0: region not formed).
SumsMap sums_map(const long long* part_off, const long long* part_blocks);
// First element (in units of T) of the partial region r.
inline void* part_ptr(cg_grids* g, int r) { return (char*)g->partials + 2 * g->tsize * g->part_off[r]; }

}  // namespace cg

// ----------------------------------------------------------------------
// Device helpers
// ----------------------------------------------------------------------
namespace cg {

template <typename T> struct V4;
template <> struct V4<float> {
    float x, y, z, w;
};
template <> struct V4<double> {
    double x, y, z, w;
};

__device__ __forceinline__ V4<float> ld4(const float* __restrict__ p, long long i) {
    float4 v = __ldg(reinterpret_cast<const float4*>(p) + i);
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ V4<double> ld4(const double* __restrict__ p, long long i) {
    const double2* q = reinterpret_cast<const double2*>(p) + 2 * i;
    double2 a = __ldg(q), b = __ldg(q + 1);
    return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void st4(float* p, long long i, float x, float y, float z, float w) {
    reinterpret_cast<float4*>(p)[i] = make_float4(x, y, z, w);
}
__device__ __forceinline__ void st4(double* p, long long i, double x, double y, double z, double w) {
    double2* q = reinterpret_cast<double2*>(p) + 2 * i;
    q[0] = make_double2(x, y);
    q[1] = make_double2(z, w);
}

// Knuth's TwoSum: s + e == a + b exactly.
template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T& s, T& e) {
    s = a + b;
    T z = s - a;
    e = (a - (s - z)) + (b - z);
}

// Compensated accumulator (TwoSum cascade, Neumaier-equivalent).
template <typename T>
struct CSum {
    T s = T(0), c = T(0);
    __device__ __forceinline__ void add(T x) {
        T t, e;
        two_sum(s, x, t, e);
        s = t;
        c += e;
    }
    __device__ __forceinline__ void merge(const CSum& o) {
        add(o.s);
        c += o.c;
    }
    __device__ __forceinline__ T get() const { return s + c; }
};

// Warp-level fixed-tree reduction of a compensated sum (deterministic).
template <typename T>
__device__ __forceinline__ CSum<T> warp_reduce(CSum<T> v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        CSum<T> o;
        o.s = __shfl_xor_sync(0xffffffffu, v.s, off);
        o.c = __shfl_xor_sync(0xffffffffu, v.c, off);
        v.merge(o);
    }
    return v;
}

// Block coordinates of a kernel body: the launch's own (blockIdx.x,
// gridDim.x) for one instance, or a virtual block of one instance inside a
// batched launch over many instances.
struct Blk {
    long long id;   // block index within the instance's work
    long long n;    // number of blocks of the instance's work
};
__device__ __forceinline__ Blk launch_blk() { return {(long long)blockIdx.x, (long long)gridDim.x}; }

// Warp sums of K (a power of two) values in one pass over the lanes: at each
// of the first log2 K steps a lane hands half of its sums to its partner and
// keeps the others, so a step merges K/2, K/4, ... sums instead of K (for eight
// values 9 merges instead of 40, of 8 FP64 operations each: the drag's were
// an eighth of its FP64 time over 1M particles, half over 10,000).  Value k ends
// on lane 32 / K * k, in a fixed order.
template <typename T, int K>
__device__ __forceinline__ CSum<T> warp_reduce_many(CSum<T> (&v)[K]) {
    static_assert(K == 1 || K == 2 || K == 4 || K == 8, "a power of two");
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int m = K / 2; m > 0; m >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int j = 0; j < m; ++j) {
            const CSum<T> a = up ? v[m + j] : v[j], b = up ? v[j] : v[m + j];
            CSum<T> o;
            o.s = __shfl_xor_sync(0xffffffffu, b.s, off);
            o.c = __shfl_xor_sync(0xffffffffu, b.c, off);
            v[j] = a;
            v[j].merge(o);
        }
    }
    for (; off > 0; off >>= 1) {
        CSum<T> o;
        o.s = __shfl_xor_sync(0xffffffffu, v[0].s, off);
        o.c = __shfl_xor_sync(0xffffffffu, v[0].c, off);
        v[0].merge(o);
    }
    return v[0];
}

// Block-level deterministic reduction of K compensated sums.  The pair (s, c)
// of sum k goes to part[2 * (k * stride + bid)]: partials stay in the path
// precision as compensated pairs, so no FP64 arithmetic runs per block (GB300's
// FP64 rate is a small fraction of FP32).
template <typename T, int K>
__device__ __forceinline__ void block_sums(CSum<T> (&v)[K], T* __restrict__ part, long long stride, long long bid) {
    __shared__ T sh_s[K][32];
    __shared__ T sh_c[K][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const CSum<T> r = warp_reduce_many<T, K>(v);
    if ((lane & (32 / K - 1)) == 0) {
        const int k = lane / (32 / K);
        sh_s[k][warp] = r.s;
        sh_c[k][warp] = r.c;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        const int k = threadIdx.x;
        CSum<T> a;
        a.s = sh_s[k][0];
        a.c = sh_c[k][0];
        for (int w = 1; w < nw; ++w) {
            CSum<T> o;
            o.s = sh_s[k][w];
            o.c = sh_c[k][w];
            a.merge(o);
        }
        T* dst = part + 2 * ((long long)k * stride + bid);
        dst[0] = a.s;
        dst[1] = a.c;
    }
}

// The block's sum of a count held once per warp (on every lane), as such a pair.
template <typename T>
__device__ __forceinline__ void block_count(int warp_count, T* __restrict__ dst) {
    __shared__ int sh[32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = warp_count;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long c = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) c += sh[w];
        dst[0] = (T)c;
        dst[1] = (T)(c - (long long)dst[0]);
    }
}

// Block-wide exclusive scan of one int per thread (total in `total`); every
// thread of the block must call it.
__device__ __forceinline__ int block_exclusive_scan(int v, int* sh_warp, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) sh_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (int)(blockDim.x >> 5) ? sh_warp[lane] : 0;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += y;
        }
        sh_warp[lane] = w;   // inclusive warp totals
    }
    __syncthreads();
    int wbase = warp ? sh_warp[warp - 1] : 0;
    total = sh_warp[(blockDim.x >> 5) - 1];
    __syncthreads();
    return wbase + x - v;
}

// Length of the run of equal values starting at this lane, or 0 if the lane
// is not the first of its run (runs of consecutive lanes with equal v).
__device__ __forceinline__ int run_head_length(int v, bool valid) {
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(0xffffffffu, v, 1);
    const bool head = valid && (lane == 0 || prev != v);
    const unsigned heads = __ballot_sync(0xffffffffu, head) | __ballot_sync(0xffffffffu, !valid);
    if (!head) return 0;
    const unsigned later = heads & ~((2u << lane) - 1u);
    const int next = lane == 31 ? 32 : (later ? __ffs(later) - 1 : 32);
    return next - lane;
}

// Programmatic dependent launch: wait until the grids this one depends on
// have completed and flushed their memory (returns at once for a kernel not
// launched as a dependent).  First statement of every kernel of the
// library (required of those launched through CG_LAUNCH).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// ----------------------------------------------------------------------
// (a0) bin index, shared by the binning and the cell-value gather.
// ----------------------------------------------------------------------
// a / b correctly rounded, from y = 1 / b correctly rounded: q1 is within one
// unit in the last place of a / b, so its remainder is exact and q1 + r y
// rounds to the quotient (Markstein's theorem).  Six FP64 operations on a GPU
// that issues FP64 at 1/64 of the FP32 rate, about half of a division.  Where
// a product could leave the exponent range (or a is not finite) it divides.
__device__ __forceinline__ double quotient_rn(double a, double b, double y) {
    const double q0 = __dmul_rn(a, y);
    const double q1 = __fma_rn(__fma_rn(-q0, b, a), y, q0);
    const double q = __fma_rn(__fma_rn(-q1, b, a), y, q1);
    // exponents of a within 2^-767 .. 2^752 and of b within 2^-511 .. 2^496; or a = +0
    const unsigned ea = (unsigned)__double2hiint(a) & 0x7ff00000u, eb = (unsigned)__double2hiint(b) & 0x7ff00000u;
    const bool zero = ((unsigned)__double2hiint(a) | (unsigned)__double2loint(a)) == 0u;
    return (ea - 0x10000000u < 0x5f000000u || zero) && eb - 0x20000000u < 0x3f000000u ? q : __ddiv_rn(a, b);
}

__device__ __forceinline__ int bin_axis_exact(double x, double x0, double H, double invH, int nb, int& outside) {
    const double q = quotient_rn(__dsub_rn(x, x0), H, invH);
    int i = __double2int_rd(q);
    if (__double2hiint(q) >= 0 && (unsigned)i < (unsigned)nb) return i;   // the quotient is not negative, nor NaN with i in range
    if (!(q >= 0.0)) i = 0;
    else if (q >= (double)nb) i = nb - 1;
    else i = (int)floor(q);
    if (!(q >= 0.0 && q <= (double)nb)) outside = 1;
    return i;
}

// |q32 - q64| <= 4 u (|q| + |x0/H|), u = 2^-24, for
// q32 = (x - fl(x0)) * fl(1/H) in round-to-nearest float, and <= 5 u (|q| +
// |x0/H|) when x is a double cut to float; the margin below is 8 u (|q| +
// |x0/H|).  Outside the margin floor(q32) == floor(q64).  True when the cell
// is decided and inside the grid.
// The floor by adding 2^23 rounded down, whose low bits are then the integer:
// no conversions, whose unit issues at a quarter of the others' rate (marking
// 8M particles: 201 -> 192 instructions per row, half of that unit's, 57.8 ->
// 55.1 us).  Below 0 and from 2^23 on those bits are out of range.
// With k the floor, q - (k + 1/2) is exact for k >= 1 and within 2^-26 for k = 0, as
// is the bound on its size; 2^-24 in the bound covers the three roundings.
__device__ __forceinline__ bool bin_axis_fast(float x, const GridDev& g, int a, int& i) {
    const float q = __fmul_rn(__fsub_rn(x, g.x0f[a]), g.invHf[a]);
    const float y = __fadd_rd(q, 8388608.0f);
    i = __float_as_int(y) - 0x4b000000;
    const float d = __fsub_rn(q, __fsub_rn(y, 8388607.5f));
    return fabsf(d) < __fmaf_rn(q, -4.76837158203125e-7f, g.binh[a]) && (unsigned)i < (unsigned)g.nb[a];
}

// A double cut (toward zero) to float with integer operations: no conversion
// on the FP64 pipe, which GB300 runs at 1/64 of the FP32 rate.  Below 2^-126: 0,
// from 2^128 on, infinities and NaN: an infinity, which no fast path takes.
__device__ __forceinline__ float f64_cut_f32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    if (e < 897u) return __uint_as_float(sign);
    if (e > 1150u) return __uint_as_float(sign | 0x7f800000u);
    return __uint_as_float(sign | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}
__device__ __forceinline__ float bin_float(float x) { return x; }
__device__ __forceinline__ float bin_float(double x) { return f64_cut_f32(x); }

// Bulk cell of a point by the exact rule (bin_axis_exact), decided in float
// away from the cell faces.
template <typename T>
__device__ __forceinline__ int cell_of(const V4<T>& v, const GridDev& g, int& outside, int& nonfinite) {
    int i, j, k;   // outside, nonfinite: counted up
    const bool a = bin_axis_fast(bin_float(v.x), g, 0, i), b = bin_axis_fast(bin_float(v.y), g, 1, j);
    const bool c = bin_axis_fast(bin_float(v.z), g, 2, k);
    if (!(a && b && c)) {   // near a face, outside, or not finite
        int out = 0;
        if (!a) i = bin_axis_exact((double)v.x, g.x0[0], g.H[0], g.invH[0], g.nb[0], out);
        if (!b) j = bin_axis_exact((double)v.y, g.x0[1], g.H[1], g.invH[1], g.nb[1], out);
        if (!c) k = bin_axis_exact((double)v.z, g.x0[2], g.H[2], g.invH[2], g.nb[2], out);
        outside += out;
        if (!(isfinite(v.x) && isfinite(v.y) && isfinite(v.z))) ++nonfinite;
    }
    return i + g.nb[0] * (j + g.nb[1] * k);
}

__device__ __forceinline__ int cell_of_f(float x, float y, float z, const GridDev& g) {
    int o = 0, f = 0;
    return cell_of(V4<float>{x, y, z, 0.f}, g, o, f);
}
__device__ __forceinline__ int cell_of_d(double x, double y, double z, const GridDev& g) {
    int o = 0, f = 0;
    return cell_of(V4<double>{x, y, z, 0.0}, g, o, f);
}

// ----------------------------------------------------------------------
// Segmented reductions over the sorted particle order.
//
// The sorted order is cut into chunks of seg_chunk(n) slots; warp w owns the
// segments (cells) that START in its chunks and runs past a chunk's end to
// finish its last segment, so every segment is reduced by exactly one warp
// and the work follows the particles, not the cells (a dense bed occupying
// a few percent of the cells still spreads over every SM).  The warp reduces
// its range in rounds of 32 slots, one per lane, with a segmented shuffle
// scan.  The rounds start at the range's first slot, so the summation order
// depends only on the chunk's slots, never on the launch shape.
// ----------------------------------------------------------------------
// Range [s, t) of sorted slots owned by the chunk starting at `base`.
__device__ __forceinline__ void seg_chunk_range(long long base, long long n, const int32_t* __restrict__ key_sorted,
                                                const int32_t* __restrict__ cs, long long& s, long long& t) {
    const int len = seg_chunk(n);
    const long long last = (base + len < n ? base + len : n) - 1;
    s = base;
    if (base > 0) {
        const int k0 = __ldg(key_sorted + base);
        if (__ldg(key_sorted + base - 1) == k0) s = __ldg(cs + k0 + 1);
    }
    t = __ldg(cs + __ldg(key_sorted + last) + 1);
    if (s > last) t = s;   // the whole chunk lies inside a segment owned earlier
}

// One round of the segmented sum of K (<= 4) values per slot over a chunk's
// slots: 32 consecutive slots, one per lane (key -1: none), with `next31` the key
// of the next round's first slot (-1 past the chunk's end).  Inside the round a
// plain inclusive shuffle scan, or, where the round holds one cell, a tree (at
// most five roundings either way; the tree: FP64, 1M packed particles, 62 ->
// 53 us, the sorted drag of 32M 710 -> 701); the segment that goes on from
// round to round is a compensated sum.  That sum is held once per warp, value k
// on lane k, so that its additions cost one instruction for all K values (held
// by every lane, they were 40% of the reaction's FP32 and two thirds of its FP64
// instructions: FP64, 1M particles 137 -> 68 us; FP32, which the shuffles bound,
// 4M particles 32 -> 29, 32M 190 -> 170).
// emit(key, k, total) is called once per segment and value, each value by
// one lane.
template <typename T, int K>
struct SegCarry {
    CSum<T> a;      // lane k: value k of the segment of `key`
    int key = -1;
};
template <typename T, int K, typename Emit>
__device__ __forceinline__ void seg_round(T (&v)[K], int key, int next31, SegCarry<T, K>& carry, Emit emit) {
    static_assert(K <= 4, "one lane per value");
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(full, key, 1);
    const unsigned heads = __ballot_sync(full, lane == 0 || prev != key);
    if (heads == 1u) {
        // one cell: a tree over the lanes in which a lane hands half of its values
        // on at the first two steps (six additions for up to four values)
        const int first = __shfl_sync(full, key, 0);
        T w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = k < K ? v[k < K ? k : 0] : T(0);
        const bool up = lane & 16, up2 = lane & 8;
        const T a0 = (up ? w[2] : w[0]) + __shfl_xor_sync(full, up ? w[0] : w[2], 16);
        const T a1 = (up ? w[3] : w[1]) + __shfl_xor_sync(full, up ? w[1] : w[3], 16);
        T x = (up2 ? a1 : a0) + __shfl_xor_sync(full, up2 ? a0 : a1, 8);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) x += __shfl_xor_sync(full, x, off);
        x = __shfl_sync(full, x, (lane & 2) * 8 + (lane & 1) * 8);   // value k on lane k
        if (first == carry.key) {
            carry.a.add(x);
        } else {
            carry.a = CSum<T>();
            carry.a.s = x;
            carry.key = first;
        }
        if (first >= 0 && next31 != first && lane < K) emit(first, lane, carry.a.get());
        return;
    }
    const int head = 31 - __clz(heads & ((2u << lane) - 1u));   // first lane of this lane's segment
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const T o = __shfl_up_sync(full, v[k], off);
            if (lane - off >= head) v[k] += o;
        }
    }
    auto to_lanes = [&](int src) {   // value k of lane src, on lane k
        T x = __shfl_sync(full, v[0], src);
#pragma unroll
        for (int k = 1; k < K; ++k) {
            const T y = __shfl_sync(full, v[k], src);
            if (lane == k) x = y;
        }
        return x;
    };
    const int first = __shfl_sync(full, key, 0), last = __shfl_sync(full, key, 31);
    const unsigned endm = (heads >> 1) | (next31 != last ? 0x80000000u : 0u);   // last lanes of their segments
    const bool ends = key >= 0 && (endm >> lane & 1u);
    const bool cont = first >= 0 && first == carry.key;   // the round goes on with the carried segment
    if (cont) {
        const unsigned later = heads & ~1u;
        const int e = later ? __ffs(later) - 2 : 31;      // its last lane in this round
        carry.a.add(to_lanes(e));
        if ((endm >> e & 1u) && lane < K) emit(first, lane, carry.a.get());
    }
    if (ends && !(cont && key == first))
#pragma unroll
        for (int k = 0; k < K; ++k) emit(key, k, v[k]);
    if (last != carry.key) {
        carry.a = CSum<T>();
        carry.a.s = to_lanes(31);
        carry.key = last;
    }
}

// Segmented sum of K values per slot over the slots [s, t) of one chunk by
// one warp, in rounds of 32 slots.  load(i, v) fills the K values of slot i.
// Four rounds are loaded ahead of the reduction.
template <typename T, int K, typename Load, typename Emit>
__device__ __forceinline__ void seg_rounds(long long s, long long t, const int32_t* __restrict__ key_sorted,
                                           Load load, Emit emit) {
    constexpr int B = 4;   // rounds loaded ahead of the reduction
    const int lane = threadIdx.x & 31;
    SegCarry<T, K> carry;
    for (long long r0 = s; r0 < t; r0 += 32 * B) {
        int key[B + 1];
        T v[B][K];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long i = r0 + 32 * j + lane;
            key[j] = -1;
#pragma unroll
            for (int k = 0; k < K; ++k) v[j][k] = T(0);
            if (i < t) {
                key[j] = __ldg(key_sorted + i);
                load(i, v[j]);
            }
        }
        {
            const long long i = r0 + 32 * B + lane;
            key[B] = (lane == 0 && i < t) ? __ldg(key_sorted + i) : -1;   // first key after the batch
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if (r0 + 32 * j >= t) break;   // warp-uniform
            seg_round<T, K>(v[j], key[j], __shfl_sync(0xffffffffu, key[j + 1], 0), carry, emit);
        }
    }
}

// Component k of the reaction of one cell from its force sum: S_B =
// -(1/V_B) sum F (Eq. UFP: F_fpi is the fluid-side reaction to F_drag), written
// to S ([3][n_b]).  The conservation sum of S_B V_B is formed by the
// projection, which reads every S_B.
template <typename T>
__device__ __forceinline__ void reaction_emit(const GridDev& g, T* __restrict__ S, int key, int k, T sum) {
    S[k * g.nbulk + key] = -sum * (sizeof(T) == 4 ? (T)g.invVBf : (T)g.invVB);
}

// ----------------------------------------------------------------------
// Porosity (Table 1: sum of the particle volumes of a cell over V_B).
//
// Each sphere's volume over V_B is rounded once to a multiple of 2^-84 and the
// cells add whole numbers, so the sum is exact and the same in any order:
// particles can be added where their cell is first known, with one set of
// atomics per run of equal cells in a warp, and every path (binning from
// scratch, incremental, batched) gives the same bits.
//
// A volume is cut into 27-bit pieces: w[0] the multiples of 2^-57 below 2^-30,
// w[1] the multiples of 2^-30, w[2] those of 2^-84 below 2^-57.  The last one
// keeps small spheres as exact as large ones (their sums against the sums of
// their volumes: with 2^-57 alone a sphere of 0.001 H was off by up to 6e-9,
// and spheres below 2e-6 H were not deposited).  FP32 volumes have 46 bits, so
// they do without from 2^-12 of a cell (0.08 H) on, and rows of such spheres skip
// it; FP64 volumes have 53 and nearly always fill it.
//
// A cell's accumulator: acc[2 c] the sum of the w[0], acc[2 c + 1] of the w[1],
// acc[2 n_b + c] of the w[2].  Spheres of 2 V_B and more also add the multiples
// of 2 V_B to acc[3 n_b + c], those of 2^32 V_B and more, and non-finite ones, go
// into a double at acc[4 n_b + c]; bit 62 of acc[2 c] marks either, and, in FP32,
// bit 61 the third pieces (most cells have none and save the read).  Each sphere
// adds less than 2^31 to a word, so 2^31 spheres do not overflow one.  The
// accumulators are zero between steps: whoever forms the porosity of a cell
// clears them.
// ----------------------------------------------------------------------
constexpr unsigned kVolMask = (1u << 27) - 1u;
constexpr unsigned long long kVolMark = 1ULL << 62, kVolThird = 1ULL << 61;

// The pieces of m 2^(s - 84), m below 2^53 and the result below 1, rounded.
__device__ __forceinline__ void volume_pieces(unsigned long long m, int s, unsigned (&w)[3]) {
    if (s < 0) {   // below 2^-31
        m = s > -64 ? (m + (1ULL << (-s - 1))) >> -s : 0ULL;
        s = 0;
    }
    const unsigned long long low = m << s;
    w[2] = (unsigned)low & kVolMask;
    w[0] = (unsigned)(low >> 27) & kVolMask;
    w[1] = (unsigned)(m >> (54 - s));
}

// Pieces of pi d^3 / (6 V_B); false when it is not in [0, 1) (the slow path's).
// FP32: the product as a pair hi + lo by FMA (relative error about 2^-46), put
// into one integer with shifts: the conversions to 64-bit integers issue on the
// FP64 pipe at 1/64 of the FP32 rate (two of them per row of 32 particles took
// over half of the marking kernel's time).
__device__ __forceinline__ void sphere_pair(float d, const GridDev& g, float& hi, float& lo) {
    const float p = __fmul_rn(d, d), pe = __fmaf_rn(d, d, -p);   // d^2 = p + pe exactly
    const float q = __fmul_rn(p, d), qe = __fmaf_rn(p, d, -q);   // p d = q + qe exactly
    const float r = __fmaf_rn(pe, d, qe);                        // d^3 = q + r (to 2^-48)
    hi = __fmul_rn(g.vch, q);
    lo = __fmaf_rn(g.vch, r, __fmaf_rn(g.vcl, q, __fmaf_rn(g.vch, q, -hi)));
}
// The pair, hi = m 2^(E - 150) with a 24-bit m and lo below 2^-22 hi, as an
// integer of 46 bits in units of 2^(E - 172).
__device__ __forceinline__ unsigned long long sphere_int(float hi, float lo, float unit) {
    const unsigned m = (__float_as_uint(hi) & 0x7fffffu) | 0x800000u;
    return ((unsigned long long)m << 22) + (long long)__float2int_rn(__fmul_rn(lo, unit));
}
// Plain spheres, from 2^-12 of a cell (0.08 H) to 1/8: multiples of 2^-57, so the
// third piece is zero.
__device__ __forceinline__ bool sphere_plain(float hi) {
    return __float_as_uint(hi) - (115u << 23) < (9u << 23);
}
__device__ __forceinline__ void sphere_pieces_plain(float hi, float lo, unsigned& w0, unsigned& w1) {
    const unsigned e = __float_as_uint(hi) & 0x7f800000u;
    const unsigned long long t = sphere_int(hi, lo, __uint_as_float((299u << 23) - e)) << ((e >> 23) - 115u & 63u);
    w0 = (unsigned)t & kVolMask;
    w1 = (unsigned)(t >> 27);
}
// Any other (2^(172 - E) is a float down to E = 45, a volume of 2^-82).
__device__ __forceinline__ bool sphere_pieces_other(float hi, float lo, unsigned (&w)[3]) {
    const unsigned u = __float_as_uint(hi);
    const int E = (int)(u >> 23);
    const bool in = u < 0x3f800000u;   // 0 <= hi < 1, not NaN
    volume_pieces(sphere_int(hi, lo, __uint_as_float(E >= 45 ? (unsigned)(299 - E) << 23 : 0u)), in ? E - 88 : -64, w);
    return in;
}
__device__ __forceinline__ bool sphere_pieces(double d, const GridDev& g, unsigned (&w)[3]) {
    const double v = __dmul_rn(__dmul_rn(__dmul_rn(g.vcd, d), d), d);   // m 2^(E - 1075)
    const unsigned hi = (unsigned)__double2hiint(v);
    const bool in = hi < 0x3ff00000u;   // 0 <= v < 1, compared as integers
    const unsigned long long m = (unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(v);
    volume_pieces(m, in ? (int)(hi >> 20) - 991 : -64, w);
    return in;
}

// One sphere outside that range: a large one, or a diameter that is negative
// or not finite.
__device__ __forceinline__ void volume_add_third(unsigned long long w2, int cell, long long nbulk, bool fp32,
                                                 unsigned long long* __restrict__ acc) {
    atomicAdd(acc + 2 * nbulk + cell, w2);
    if (fp32) atomicOr(acc + 2 * (size_t)cell, kVolThird);
}
static __device__ __noinline__ void volume_add_slow(double d, int cell, const double vcd, long long nbulk,
                                                    unsigned long long* __restrict__ acc) {
    const double t = vcd * d * d * d;
    if (fabs(t) < 4294967296.0) {
        const double x = t * 1073741824.0, f = floor(x);                        // 2^30
        const double y = (x - f) * 134217728.0, e = floor(y);                   // 2^27
        const long long h = (long long)f;
        atomicAdd(acc + 2 * (size_t)cell, (unsigned long long)e);
        atomicAdd(acc + 2 * (size_t)cell + 1, (unsigned long long)(h & 0x7fffffffLL));
        volume_add_third(__double2ull_rn((y - e) * 134217728.0), cell, nbulk, true, acc);
        if (h >> 31) {
            atomicAdd(acc + 3 * nbulk + cell, (unsigned long long)(h >> 31));
            atomicOr(acc + 2 * (size_t)cell, kVolMark);
        }
    } else {
        atomicAdd((double*)(acc + 4 * nbulk) + cell, isfinite(t) ? t : __longlong_as_double(0x7ff8000000000000LL));
        atomicOr(acc + 2 * (size_t)cell, kVolMark);
    }
}

// The first lanes of the runs of equal cells among a row's valid lanes.
__device__ __forceinline__ unsigned run_heads(bool valid, int cell) {
    const int c = valid ? cell : -1;
    const int prev = __shfl_up_sync(0xffffffffu, c, 1);
    return __ballot_sync(0xffffffffu, (threadIdx.x & 31) == 0 || prev != c);
}
// Sums of N values (of at most 27 bits, which cannot overflow 32 bits over 32
// lanes) over the runs that begin at the lanes `heads`: one or two runs by
// warp reductions, more by a segmented scan.  True on the lane that holds its
// run's sums.
template <int N>
__device__ __forceinline__ bool volume_runs(unsigned* w, unsigned heads) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    if (__popc(heads) <= 2) {
        const unsigned later = heads & ~1u;
        const bool first = lane < (later ? __ffs(later) - 1 : 32);   // of the first run, or of the second
        unsigned a[N];
#pragma unroll
        for (int k = 0; k < N; ++k) a[k] = __reduce_add_sync(full, first ? w[k] : 0u);
        if (later)
#pragma unroll
            for (int k = 0; k < N; ++k) w[k] = __reduce_add_sync(full, first ? 0u : w[k]);
        if (first)
#pragma unroll
            for (int k = 0; k < N; ++k) w[k] = a[k];
        return heads >> lane & 1u;
    }
    const int head = 31 - __clz(heads & ((2u << lane) - 1u));
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        unsigned x[N];
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = __shfl_up_sync(full, w[k], off);
        if (lane - off >= head)
#pragma unroll
            for (int k = 0; k < N; ++k) w[k] += x[k];
    }
    return lane == 31 || (heads >> (lane + 1) & 1u);
}
__device__ __forceinline__ void volume_atomics(unsigned w0, unsigned w1, int cell, unsigned long long* __restrict__ acc) {
    atomicAdd(acc + 2 * (size_t)cell, (unsigned long long)w0);
    atomicAdd(acc + 2 * (size_t)cell + 1, (unsigned long long)w1);
}
// A sphere that is not to go into its run's sums: one of 1/8 of a cell or more
// (its pieces w, when it is in their range).
__device__ __forceinline__ bool volume_alone(bool in, const unsigned (&w)[3], double d, int cell, double vcd, long long nbulk,
                                             bool fp32, unsigned long long* __restrict__ acc) {
    if (in && w[1] <= kVolMask) return false;
    if (in) {
        volume_atomics(w[0], w[1], cell, acc);
        if (w[2]) volume_add_third(w[2], cell, nbulk, fp32, acc);
    } else {
        volume_add_slow(d, cell, vcd, nbulk, acc);
    }
    return true;
}

// FP32 rows with spheres that are not plain: the first two pieces of such a lane
// for its run's sums (the second in the upper half; zero for one added alone);
// the third pieces of up to four lanes go to their cells by themselves, those of
// more through sums of their own.  Out of line, so that the marking kernel's
// registers are those of the plain rows.  (32M log-normal spheres, of whose rows
// 7% hold another sphere: 207 us; with the whole row in three pieces then 223,
// with every such sphere added alone 230.  700,001 spheres of 0.08 H, some below
// 2^-12: 16 us; as rows of other spheres 18.7.)
static __device__ __noinline__ unsigned long long volume_other(bool other, int cell, float hi, float lo, float d, double vcd,
                                                               long long nbulk, unsigned heads,
                                                               unsigned long long* __restrict__ acc) {
    unsigned w[3] = {0u, 0u, 0u};
    if (other) {
        const bool in = sphere_pieces_other(hi, lo, w);
        if (volume_alone(in, w, (double)d, cell, vcd, nbulk, true, acc)) w[0] = w[1] = w[2] = 0u;
    }
    unsigned third = w[2];
    const int lanes = __popc(__ballot_sync(0xffffffffu, third != 0u));
    const bool sum = lanes <= 4 || volume_runs<1>(&third, heads);
    if (sum && third) volume_add_third(third, cell, nbulk, true, acc);
    return (unsigned long long)w[1] << 32 | w[0];
}

// Add 32 spheres, one per lane (valid lanes), to their cells: equal cells on
// consecutive lanes are summed first.  Called by the whole warp.
__device__ __forceinline__ void volume_add_row(bool valid, int cell, float d, const GridDev& g,
                                               unsigned long long* __restrict__ acc) {
    const unsigned heads = run_heads(valid, cell);
    float hi, lo;
    sphere_pair(d, g, hi, lo);
    unsigned w[2];
    sphere_pieces_plain(hi, lo, w[0], w[1]);
    if (!valid) w[0] = w[1] = 0u;
    const bool other = valid && !sphere_plain(hi);
    if (__any_sync(0xffffffffu, other)) {
        const unsigned long long o = volume_other(other, cell, hi, lo, d, g.vcd, g.nbulk, heads, acc);
        if (other) {
            w[0] = (unsigned)o;
            w[1] = (unsigned)(o >> 32);
        }
    }
    if (volume_runs<2>(w, heads) && valid) volume_atomics(w[0], w[1], cell, acc);
}
__device__ __forceinline__ void volume_add_row(bool valid, int cell, double d, const GridDev& g,
                                               unsigned long long* __restrict__ acc) {
    unsigned w[3];
    const bool in = sphere_pieces(d, g, w);
    if (!valid || volume_alone(in, w, d, cell, g.vcd, g.nbulk, false, acc)) w[0] = w[1] = w[2] = 0u;
    if (volume_runs<3>(w, run_heads(valid, cell)) && valid) {
        volume_atomics(w[0], w[1], cell, acc);
        if (w[2]) volume_add_third(w[2], cell, g.nbulk, false, acc);
    }
}
// The same in line, for kernels with registers to spare: the pieces of spheres from
// 2^-39 of a cell (1.5e-4 H) to one in a few shifts (the same pieces), and a row
// with such spheres sums three pieces at once; the others out of line.  4M spheres
// in the caller's order: packed 60 us either way, log-normal 58 -> 56, of 0.05 H 65 ->
// 59; the deposit of a batch of mostly small ones 31 -> 27.  (In the sorted step's
// marking kernel, which has 48 registers, 207 -> 221 us for the 32M log-normal ones.)
__device__ __forceinline__ bool sphere_pieces_mid(float hi, float lo, unsigned (&w)[3]) {
    const unsigned e = __float_as_uint(hi) & 0x7f800000u, s = ((e >> 23) - 88u) & 63u;
    const unsigned long long m = sphere_int(hi, lo, __uint_as_float((299u << 23) - e)), low = m << s;
    w[2] = (unsigned)low & kVolMask;
    w[0] = (unsigned)(low >> 27) & kVolMask;
    w[1] = (unsigned)(m >> ((54u - s) & 63u));
    return __float_as_uint(hi) - (88u << 23) < (39u << 23);
}
static __device__ __noinline__ void volume_add_odd(int cell, float hi, float lo, float d, double vcd, long long nbulk,
                                                   unsigned long long* __restrict__ acc) {
    unsigned w[3];
    if (sphere_pieces_other(hi, lo, w)) {
        volume_atomics(w[0], w[1], cell, acc);
        if (w[2]) volume_add_third(w[2], cell, nbulk, true, acc);
    } else {
        volume_add_slow((double)d, cell, vcd, nbulk, acc);
    }
}
__device__ __forceinline__ void volume_add_row_wide(bool valid, int cell, float d, const GridDev& g,
                                                    unsigned long long* __restrict__ acc) {
    const unsigned heads = run_heads(valid, cell);
    float hi, lo;
    sphere_pair(d, g, hi, lo);
    unsigned w[3];
    sphere_pieces_plain(hi, lo, w[0], w[1]);
    w[2] = 0u;
    const bool other = valid && !sphere_plain(hi);
    const bool mixed = __any_sync(0xffffffffu, other);
    bool out = !valid;
    if (other) {
        const bool in = sphere_pieces_mid(hi, lo, w);
        if (!in) {
            volume_add_odd(cell, hi, lo, d, g.vcd, g.nbulk, acc);
            out = true;
        } else if (w[1] > kVolMask) {   // 1/8 and more
            volume_atomics(w[0], w[1], cell, acc);
            if (w[2]) volume_add_third(w[2], cell, g.nbulk, true, acc);
            out = true;
        }
    }
    if (out) w[0] = w[1] = w[2] = 0u;
    if ((mixed ? volume_runs<3>(w, heads) : volume_runs<2>(w, heads)) && valid) {
        volume_atomics(w[0], w[1], cell, acc);
        if (mixed && w[2]) volume_add_third(w[2], cell, g.nbulk, true, acc);
    }
}
__device__ __forceinline__ void volume_add_row_wide(bool valid, int cell, double d, const GridDev& g,
                                                    unsigned long long* __restrict__ acc) {
    volume_add_row(valid, cell, d, g, acc);
}

// Where a step's porosity goes: double, and (nullable) the porosity of the
// drag's record, its copy in the path precision, and the reaction source to
// clear (cells without particles keep the zero).
template <typename T>
struct EpsOut {
    unsigned long long* acc;
    double* eps;
    T* rec;
    T* eps_t;
    T* S;
};

// Accumulators of n_b cells, and zeroes into them on stream s: of a new handle,
// and after a launch between the spheres and the cells' porosity failed.
inline size_t vol_acc_bytes(long long nbulk) { return 5 * sizeof(unsigned long long) * nbulk; }
inline cudaError_t clear_volumes(cg_grids* g, cudaStream_t s) {
    return cudaMemsetAsync(g->vol_acc, 0, vol_acc_bytes(g->gd.nbulk), s);
}

// The accumulators of the handle with a step's (or no) outputs.
template <typename T>
inline EpsOut<T> eps_out(cg_grids* g, const StepEps* e) {
    return {g->vol_acc, e ? e->eps : nullptr, e ? (T*)e->rec : nullptr,
            e ? (T*)e->eps_t : nullptr, e ? (T*)e->S : nullptr};
}

__device__ __forceinline__ void eps_round(long long e57, double, float& et) {
    et = __ll2float_rn(e57) * 6.938893903907228e-18f;
}
__device__ __forceinline__ void eps_round(long long, double e, double& et) { et = e; }
// A cell's volume (p57 2^-57 + r 2^-84) V_B into a sum.  FP32: a pair of 48 bits.
__device__ __forceinline__ void deposited_volume(long long p57, unsigned r, const GridDev& g, CSum<float>& tot) {
    const float ph = __ll2float_rn(p57);
    const float pl = __ll2float_rn((p57 - __float2ll_rn(ph)) * (1LL << 27) + r) * 5.1698788284564230e-26f;   // 2^-84
    const float p = ph * 6.938893903907228e-18f;
    const float hi = p * g.VBh;
    const float lo = fmaf(pl, g.VBh, fmaf(p, g.VBl, fmaf(p, g.VBh, -hi)));
    tot.add(hi);
    tot.c += lo;
}
__device__ __forceinline__ void deposited_volume(long long p57, unsigned r, const GridDev& g, CSum<double>& tot) {
    tot.add(fma((double)r, 5.1698788284564230e-26, (double)p57 * 6.938893903907228e-18) * g.VB);
}

// The volume (over V_B) of a cell beyond the ordinary range, or with a marked
// accumulator (out of line: such cells are rare).
static __device__ __noinline__ double volume_far(long long h, unsigned l, unsigned r, bool marked, unsigned long long* fine,
                                                 long long nbulk) {
    double phi = (double)h * 9.313225746154785e-10 +
                 ((double)l * 6.938893903907228e-18 + (double)r * 5.1698788284564230e-26);   // 2^-30, 2^-57, 2^-84
    if (marked) {
        long long* const top = (long long*)fine + nbulk;
        double* const big = (double*)fine + 2 * nbulk;
        phi += 2.0 * (double)*top + *big;
        *top = 0;
        *big = 0.0;
    }
    return phi;
}

// The porosity of one cell from its accumulator, which is cleared; its
// deposited volume goes into tot with SUMS.
template <typename T, bool SUMS>
__device__ __forceinline__ void eps_finish(long long c, const GridDev& g, const EpsOut<T>& o, CSum<T>& tot) {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(o.acc + 2 * c);
    unsigned long long* const fine = o.acc + 2 * g.nbulk + c;
    const unsigned long long b = sizeof(T) == 8 || (a.x & kVolThird) ? *fine : 0ULL;
    double e = 1.0;
    T et = T(1);
    if (a.x | a.y | b) {
        *reinterpret_cast<ulonglong2*>(o.acc + 2 * c) = make_ulonglong2(0, 0);
        if (b) *fine = 0;
        const bool marked = a.x & kVolMark;
        const unsigned long long low = (a.x & ~(kVolMark | kVolThird)) + (b >> 27);
        const long long h = (long long)a.y + (long long)(low >> 27);
        const unsigned l = (unsigned)low & kVolMask, r = (unsigned)b & kVolMask;
        if (!marked && h >= 0 && h < (1LL << 33)) {
            const long long p57 = (h << 27) | l;
            const long long e57 = (1LL << 57) - p57 - (r >> 26);   // 1 - sum, to 2^-58
            e = __ll2double_rn(e57) * 6.938893903907228e-18;
            eps_round(e57, e, et);
            if (SUMS) deposited_volume(p57, r, g, tot);
        } else {
            const double phi = volume_far(h, l, r, marked, fine, g.nbulk);
            e = 1.0 - phi;
            et = (T)e;
            if (SUMS) tot.add((T)(phi * g.VB));
        }
    }
    o.eps[c] = e;
    if (o.rec) o.rec[4 * c] = et;
    if (o.eps_t) o.eps_t[c] = et;
    if (o.S)
#pragma unroll
        for (int k = 0; k < 3; ++k) o.S[k * g.nbulk + c] = T(0);
}

}  // namespace cg
