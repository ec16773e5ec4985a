// Internal declarations of the KLB library: host geometry tables, device
// memory plan and kernel launchers.  Not part of the public ABI (include/klb.h).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "klb.h"

namespace klb {

constexpr int kMaxFaces = 4;   // fluid/solid faces of one cross-section cell (+-y, +-z)
constexpr int kBlockX = 128;   // threads per block along x (one x per thread)
constexpr int kObsBlocks = 4 * 152;  // resident blocks of the observation pass (FP32 arithmetic)
// Rows are padded to a multiple of kRowAlign elements.  RowInfo::src counts
// in these units, so a 32-bit entry reaches 2^31 * 32 elements of a class
// buffer; offsets within one direction plane (row * nxp + x) stay 32-bit.
constexpr int kRowAlign = 32;

// Row classes: a row is one cross-section cell together with all its x.
// Water lives on fluid rows; electrons and phonons share the solid rows.
enum RowClass { kFluid = 0, kSolid = 1 };

// Per-row table: a warp's threads share a row (with FP64 and in the field and
// initialisation passes a block's).
struct RowInfo {
    int32_t src[19];            // (dir' * n_rows + row') * nxp / kRowAlign: first element,
                                // in kRowAlign units, of the row direction i is pulled from
    uint32_t xm;                // bit i: pull direction i from x - 1
    uint32_t xp;                // bit i: pull direction i from x + 1
    int32_t slot;               // interface slot of this row, -1 if none
    int32_t nface;              // number of fluid/solid faces
    int32_t partner[kMaxFaces]; // interface slots of the rows across those faces
    float d2;                   // fluid rows: squared distance to centre plane / axis
    int32_t flags;              // bit 0 in the slip fit, bit 1 wall row (fluid rows);
                                // bit 2: some direction with c_x != 0 bounces back
    int32_t cs;                 // cross-section cell y + ny z (cell x + nx cs of the box)
    int32_t pad[2];
};
static_assert(sizeof(RowInfo) == 128, "RowInfo is one 128-byte line");

enum RowFlags { kFitRow = 1, kWallRow = 2, kXBounce = 4 };

// Indices of the FP64 sums of the observation pass.
enum SumIndex {
    kSumUxFluid = 0,   // sum of u_x over fluid cells
    kSumFitU,          // sum of u_x and of u_x d^2 over the slip fit's cells
    kSumFitUD2,
    kSumWallU,         // sum of u_x over the wall rows
    kSumUxE,           // electron / phonon sum u_x
    kSumUxP,
    kSumMomW,          // sum rho u_x per species
    kSumMomE,
    kSumMomP,
    kSumMassW,         // sum (rho - rho0) per species
    kSumMassE,
    kSumMassP,
    kSumNonfinite,     // count of non-finite rho/u values
    kSumResidual,      // max |u_x(n) - u_x(n-1)| (a max, not a sum)
    kSumClipped,       // 16-bit storage: species-cells with a saturated population
    kNumSums
};

// Host geometry of one lattice (built from the description only).
struct Geometry {
    int Q = 0, nx = 0, ny = 0, nz = 0, nxp = 0;
    int periodic_y = 0, periodic_z = 0;
    std::vector<uint8_t> cs_type;          // ny*nz, index y + ny*z
    std::vector<int> rows[2];              // cross-section index of each row
    std::vector<int> row_of_cs[2];         // row of a cross-section cell, -1 if none
    std::vector<RowInfo> info[2];
    std::vector<int> slot_row[2];          // row of each interface slot
    int max_faces[2] = {0, 0};
    double d_wall = 0.0;
    bool has_fit = false;
    double fit_n = 0, fit_d2 = 0, fit_d4 = 0, wall_n = 0;  // cells of the slip fit with sums of d^2, d^4; wall-row cells
};

// Builds the geometry and its streaming / interface tables.  Returns false
// with a message on an invalid description.
bool build_geometry(const klb_desc &d, Geometry &g, std::string &err);

// Offsets (bytes from the caller's buffer) of every device region.
struct MemoryPlan {
    size_t pop[2][3];      // [buffer][species]
    size_t pop_bytes[3];
    size_t U[3][2];        // [time slot][row class]
    size_t U_bytes[2];
    size_t rows[2];
    size_t partials, sums, field;
    size_t field_bytes;
    size_t ref_enc[2][3], ref_dec[2][3];  // [generation][species], reduced storage only
    size_t ref_bytes[3];
    size_t acc, acc_bytes;
    size_t bounds;         // error word of debug builds (KLB_BOUNDS)
    size_t total;
    int nblocks_w, nblocks_s, nchunk, bx;  // one cell per thread (observe, field, init)
    bool fine;                             // step kernel: small-lattice form of the solid rows (step_ep, fp64_split),
    int sbx, snblocks;                     // threads per block, blocks
    int static_blocks;                     // row chunks that klb_observables_static bounds
    int oblocks, oblocks_s;                // observation with FP32 arithmetic: blocks of kBlockX, of which solid
};
MemoryPlan plan_memory(const Geometry &g, int storage);

// Reduced-precision storage: floats per row in the reference tables (Q
// used, padded to a multiple of four), steps between reference refreshes,
// and the power-of-two scale of FP16 differences (keeps them out of the
// subnormal range).
constexpr int kRefStride = 20;
constexpr int kRefEvery = 32;
constexpr float kFp16Scale = 1048576.0f;  // 2^20

// FP64 lattices of so few cells that a species-cell per thread in one-warp
// blocks leaves SMs idle: one warp per block, and solid rows one species per
// block.  The FP64 pipe takes 16 cycles per warp instruction on every SM, so
// a step lasts as long as its busiest SM computes.
inline long long fp64_warps(int nx, long long rows_w, long long rows_s) { return (rows_w + 2 * rows_s) * ((nx + 31) / 32); }
inline bool fp64_split(int nx, int rows_w, int rows_s) { return fp64_warps(nx, rows_w, rows_s) <= 152; }

// Whether the members of a batch (warps: fp64_warps of all) keep that form:
// while all of them find a place on the chip (16 warps on each of 152 SMs).
// Beyond, the second species streamed and collided for nothing is what the
// FP64 pipe waits for.  Step times with -> without, GB300: 24 slabs of 64x40
// (2304 warps) 24.3 -> 27.9 us, 36 (3456) 34.1 -> 33.4, 100 75.5 -> 70.6, 400
// 273 -> 242; 400 slabs of 16x20 (10400) 87.3 -> 77.8.
inline bool fp64_batch_split(long long warps) { return warps <= 152 * 16; }

// Blocks of sbx threads of one step launch: FP64 one block per row chunk of
// sbx cells (with `fine` a solid one per species, fp64_split); FP32 arithmetic
// one warp per item (`fine`: species pairs, step_ep).
inline long long step_items(int nx, long long rows_w, long long rows_s, bool ep);
inline int step_blocks(int nx, int rows_w, int rows_s, int sbx, int storage, bool fine)
{
    if (storage == KLB_FP64) return (rows_w + rows_s + (fine ? rows_s : 0)) * ((nx + sbx - 1) / sbx);
    return (int)((step_items(nx, rows_w, rows_s, fine) + sbx / 32 - 1) / (sbx / 32));
}

// Items of one launch of the FP32-arithmetic step on a lattice's rows: 64
// cells of a row; with ep solid items are 32 cells, one per lane, electrons
// and phonons as the pair.
inline long long step_items(int nx, long long rows_w, long long rows_s, bool ep)
{
    return rows_w * ((nx + 63) / 64) + rows_s * (ep ? (nx + 31) / 32 : (nx + 63) / 64);
}

// Which form the solid items take: ep where latency counts (the items find a
// place on the chip at about the same time): the species are pulled once, in
// one round of loads.  Two cells and two pulls of the phonons where
// throughput counts.  Step times with cell pairs -> with species pairs,
// GB300, FP32: pipe R 8, nx 8 (384 items) 5.6 -> 3.8 us, nx 200 7.7 -> 5.5,
// nx 400 (3792 items) 9.5 -> 7.7; 128x64x64 (5552 items) 8.5 -> 8.8; R 48,
// nx 8 (9176 items) 11.0 -> 11.3; 512x128x128 134.9 -> 140.9.
// FP16: 384 items 5.9 -> 4.2 us, 3160 9.4 -> 7.0, 3576 8.6 -> 7.4, 3812 7.3 ->
// 7.6.
inline bool step_ep(long long ep_items) { return ep_items <= 4000; }

// The same with thermal noise, whose water cells take most of the time: on
// D3Q19 while nearly all items find a place at once (16 warps of 128 registers
// on each of 152 SMs), on D2Q9 never.  Cell pairs -> species pairs: 764 items
// 9.0 -> 6.8 us, 2424 10.0 -> 7.8, 2612 10.4 -> 9.0, 2780 9.6 -> 9.7, 2872 10.0
// -> 9.9, 3024 9.3 -> 10.8, 3232 10.1 -> 9.9, 3576 9.5 -> 11.2; D2Q9 48 to 420
// items equal, 1100 5.1 -> 5.5, 1600 4.9 -> 5.7.
inline bool noise_ep(int Q, long long ep_items) { return Q == 19 && ep_items <= 2900; }

// Threads per step block with FP32 arithmetic: four warps, or one where the
// launch's items are few, which spreads them over all SMs (20 warps of cell
// pairs, 16 of species pairs find a place on each of 152 SMs).  For species
// pairs the width matters little: four -> one, FP32 1616 items 5.70 -> 5.62 us,
// 2592 6.25 -> 6.24, 3160 6.69 -> 6.81; FP16 5.54 -> 5.58, 6.48 -> 6.51, 6.95 ->
// 7.07.
inline int step_width(long long items) { return items <= 152 * 20 ? 32 : kBlockX; }

inline bool reduced_storage(int storage) { return storage == KLB_FP16_DEV || storage == KLB_BF16_DEV; }
inline size_t storage_bytes(int storage)
{
    return storage == KLB_FP64 ? 8 : (storage == KLB_FP32 ? 4 : 2);
}

// Distance, in rows, of the step's L2 requests (prefetch_rows); 0: none.
// They pay once the state buffers (all_bytes, of every lattice in the launch)
// exceed the 129 MB L2, so that the populations have left it by the next
// step: step times without -> with, GB300, FP32 at 108 MB 17.4 -> 18.6 us,
// 162 MB 33.1 -> 32.4, 270 MB 51.3 -> 47.7, 865 MB 134.9 -> 130.4, 2.9 GB
// 437.8 -> 428.2; FP16 at 108 MB 32.2 -> 32.2, 135 MB 47.9 -> 46.7, 433 MB
// 114.8 -> 109.3, 1.5 GB 366.6 -> 347.0.  FP32 is best at 2 MB of populations
// (4 MB: 131.8 us at 865 MB, 10 MB: 141.7), 16 bits at 4 MB (2 MB: 355.0 us
// at 1.5 GB, 10 MB: 352.8).
constexpr size_t kL2Bytes = 129000000;
inline int step_ahead(int Q, int storage, int nxp, size_t all_bytes)
{
    if (storage == KLB_FP64 || all_bytes <= kL2Bytes) return 0;
    const size_t ahead = reduced_storage(storage) ? 4u << 20 : 2u << 20, row = (size_t)Q * nxp * storage_bytes(storage);
    return (int)((ahead + row - 1) / row);
}

// Collision constants of one relaxation rate om (fo = 1 - om/2) per weight
// class (rest, axis, edge directions), as the pairs that the packed
// instructions take: from the kernel's parameters they need no moves and no
// arithmetic in the kernel (512x128x128 FP16 108.1 -> 106.0 us, 768x192x192
// FP16 344.1 -> 338.7, 12-channel sweep FP16 410 -> 401, FP32 456 -> 453).
struct CollideK {
    float2 om1, omw[3], fow[3], tow[3], tfw[3];  // 1 - om, om w, fo w, 3 om w, 3 fo w
};
inline __host__ __device__ CollideK collide_k(int Q, float om)
{
    const float w[3] = {Q == 19 ? float(1.0 / 3.0) : float(4.0 / 9.0), Q == 19 ? float(1.0 / 18.0) : float(1.0 / 9.0),
                        float(1.0 / 36.0)};
    const float om1 = 1.f - om, fo = 1.f - 0.5f * om;
    CollideK c;
    c.om1 = make_float2(om1, om1);
    for (int k = 0; k < 3; ++k) {
        const float v[4] = {om * w[k], fo * w[k], 3.f * om * w[k], 3.f * fo * w[k]};
        c.omw[k] = make_float2(v[0], v[0]);
        c.fow[k] = make_float2(v[1], v[1]);
        c.tow[k] = make_float2(v[2], v[2]);
        c.tfw[k] = make_float2(v[3], v[3]);
    }
    return c;
}

// The constants of a lattice's three species.
struct alignas(16) CollideSet {
    CollideK s[3];
};

// What a step reads of its lattice: the record that a batch keeps per phase
// and member.  T is the arithmetic type (float or double); the populations
// are stored as T, or as FP16/BF16 against per-row references.
template <typename T>
struct alignas(16) StepRecord {
    const void *in[3];     // current state, per species
    void *out[3];          // next state (step and init modes)
    const RowInfo *rows[2];
    const T *U1[2], *U2[2];  // lagged velocities u(n-1), u(n-2)
    T *U0[2];                // u(n) written here (step mode)
    int nx, nxp;
    int snchunk, split;              // FP64 step: x chunks of blockDim.x per row; one species per solid block
    int nseg64;                      // 64-wide x segments per row
    uint32_t seg_mul, seg_shift;     // n / nseg64 = n seg_mul >> seg_shift for 0 <= n < 2^31
    int sseg;                        // the same for the solid rows: segments of 64, or 32 with step_ep
    uint32_t sseg_mul, sseg_shift;
    int nch32, nseg_w;               // 32-wide x segments per row; water segments
    int n_rows[2], n_slots[2];
    T rho0, om[3], G[3];
    T g_we, g_wp, g_ep, g_ec, g_pc;
    T q_p;                 // phonons: 1 second-order equilibrium, 0 linear (damped waves, Sec. 3.4)
    // reduced-precision storage only (null otherwise)
    const float *dec_in[3];   // references of pulled populations
    const float *enc_out[3];  // references of stored populations
    float scale, inv_scale;
    float *acc;            // x-sums of g* per 32-wide segment [segment][2Q]
    // thermal fluctuations of the water (step with noise only)
    T noise_amp;           // sqrt(3 rho0 kT omega (2 - omega))
    uint32_t key[2];       // generator key (seed)
    uint32_t step_lo, step_hi;  // the step being taken
    // batches: the record is of a period's phase, replayed; the step taken is
    // step_lo + *step_reps * step_period (low 32 bits), step_reps counting the
    // periods completed since the tables were built (null for one lattice)
    const uint32_t *step_reps;
    int step_period;
    int ahead;             // rows ahead whose populations the step asks L2 for (step_ahead; 0: none)
    unsigned *bounds_err;  // debug builds: first out-of-range index site
};

// Kernel arguments: the record, what is the same in every step of a lattice
// and formed from it, and what the other passes read.
template <typename T>
struct alignas(16) StepArgs : StepRecord<T> {
    CollideSet ck;           // FP32 arithmetic: collision constants
    const void *in_prev[3];  // observe mode: previous state and its references (residual),
    const float *dec_prev[3];
    const T *U3[2];          // u(n-3),
    double *partials;        // [block][kNumSums],
    int obs_solid;           // with FP32 arithmetic the blocks that take the solid rows
    int residual_valid;
    int nchunk, nbw;         // observe, field and init modes: x chunks of blockDim.x per row, water blocks
    T *field;                // field / init mode: per species [4][n_rows][nxp]
};

enum Mode {
    kModeStep = 0,
    kModeObserve = 1,
    kModeField = 2,
    kModeStepAcc = 3,  // step that also writes the x-sums for a refresh
    kModeInit = 4,
    kModeInitAcc = 5,  // x-sums of the initial equilibria, nothing stored
    kModeStepNoise = 6, // step with thermal fluctuations of the water
    kModeEp = 8         // added to a step mode: solid items of one cell per thread (step_ep)
};

// Launchers (return the launch error, if any).
cudaError_t launch(int Q, int storage, const void *args, int mode, int nblocks, int bx,
                   cudaStream_t s);
// Reference refresh from args.acc into the tables enc[s], dec[s].
cudaError_t launch_ref(int Q, int storage, const void *args, float *const enc[3],
                       float *const dec[3], cudaStream_t s);
// Final sums of an observation pass from its blocks' partial sums.
cudaError_t launch_finalize(const double *partials, int nblocks, double *sums, cudaStream_t s);
// One more period completed by a batch (StepArgs::step_reps).
cudaError_t launch_count_period(uint32_t *reps, cudaStream_t s);
// One step of many lattices: argument records and first block of each lattice
// (prefix[n] = total blocks), and the collision constants.
// Up to kBatchParams records go as kernel parameters (32 KB in all).  More
// lattices take several such launches, or one over device copies of the
// records (batch_by_table).  A launch waits for the one before it, so several
// pay only when each fills the chip (20 warps on each of 152 SMs) some times
// over: kGroupItems items (warps) in each.  One launch -> several, us per
// step, GB300, FP32 / FP16, by items per launch: 1333 (400 D2Q9 slabs 64x40)
// 24.2 -> 56.4 / 70.5 -> 102; 4466 (400 pipes R 4-5, nx 3) 141 -> 166 / 223 ->
// 243; 4824 (72 of them) 24.8 -> 26.1 / 36.3 -> 38.8; 7020 (40 pipes R 6-9, nx
// 8) 34.8 -> 35.0 / 41.5 -> 42.9; 9065 (40 sweep channels at a quarter) 44.0 ->
// 43.1 / 48.6 -> 49.2; 11700 (100 pipes R 6-9) 85.6 -> 82.6 / 115 -> 112;
// 61200 (40 channels at half) 232 -> 214 / 234 -> 218.  FP64, which the FP64
// pipe bounds, takes one launch throughout (9065: 428 -> 451).
constexpr int kBatchParams = 36;
constexpr long long kGroupItems = 8000;
inline int batch_groups(int n) { return (n + kBatchParams - 1) / kBatchParams; }
inline bool batch_by_table(int n, int storage, long long items)
{
    return n > kBatchParams && (storage == KLB_FP64 || items < kGroupItems * batch_groups(n));
}
struct BatchLaunch {
    const void *table, *dev_table;
    const int *prefix, *dev_prefix;
    const CollideSet *ck, *dev_ck;
    int n, width;
    bool acc, ep, by_table;  // ep: species pairs (FP32 arithmetic)
};
cudaError_t launch_batch(int Q, int storage, const BatchLaunch &b, cudaStream_t s);

// Device bytes of the argument tables of a batch of n lattices with this
// storage (the layout klb_batch_create uses).
size_t batch_table_bytes(int storage, int n);

// Observation pass of a lattice enqueued on its stream, its kNumSums sums copied
// to host_sums (pinned host memory; valid after the stream synchronises),
// and the observables computed from them (klb_observables in two halves).
cudaError_t observe_enqueue(klb_lattice *L, double *host_sums);
klb_status observe_finish(klb_lattice *L, const double *host_sums, klb_obs *out);

// Static scratch of klb_observables_static (klb_static.cu): device addresses
// of its partial-sum rows and final sums on the current device.
cudaError_t static_scratch(double **partials, double **sums, size_t *max_blocks);

}  // namespace klb
