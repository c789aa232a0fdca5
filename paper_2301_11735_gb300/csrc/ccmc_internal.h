// ccmc_internal.h -- library-internal types shared by the host API and the
// kernels (plain C++, no device code).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "../../include/ccmc.h"

struct ccmc_lattice;
struct ccmc_batch;

namespace ccmc {

constexpr uint32_t TAG_SCHED = 1u;    // phase schedule
constexpr uint32_t TAG_MOVE = 2u;     // per 8 pairs: a 16-bit field a pair
constexpr uint32_t TAG_SLOW = 3u;     // per pair: acceptance word, choice fallback
constexpr uint32_t TAG_FEISTEL = 4u;  // initial placement
constexpr uint32_t TAG_SIGN = 5u;     // initial spin signs

constexpr int kDB = 20;                 // |dBV|, |dBJ| <= 20 when Lx, Ly >= 4
constexpr int kNB = 2 * kDB + 1;        // 41
constexpr int kTableN = 3 * kNB * kNB;  // dQ in {-2, 0, 2}: 5043 thresholds

// Control block of a lattice (int64 words in device memory).
enum CtlSlot : int {
  kCtlPhaseBase = 0,  // global phase index of the next phase with offset 0
  kCtlObsCount = 1,   // records written to the ring so far
  kCtlTicket = 2,     // arrival counter of the recount's last-block reduction
  kCtlStatus = 3,     // device-side error flag (no sweep kernel has a wait that could set it)
  kCtlLatest = 4,     // 8 words: the last recount record
  kCtlWords = 16
};

// Lattice geometry as seen by the kernels.
struct Geo {
  uint32_t *words;  // 16 classes x Cy rows x W words
  int64_t *ctl;     // control block
  int Lx, Ly, Cx, Cy, W;
  int64_t cstride;  // Cy * W words per class
  uint32_t k0, k1;  // Philox key = seed
  uint64_t rej;     // 2^64 mod (Lx Ly): Lemire rejection bound
};

// The device's threshold tables hold only the energy changes a coupled pair
// can make, in three segments; every move stays in the segment of its kind, so
// that its index is an affine function of the neighbour sums:
//   one unit of charge moves or a +- pair appears or vanishes (|dS| = 1):
//     |dBV|, |dBJ| <= 9, dQ in {-2, 0, 2}: 3 x 19 x 19 entries
//     [(dQ + 2) / 2][dBV + 9][dBJ + 9];
//   the two charges of a +- pair change places (|dS| = 2, no spin involved):
//     41 entries [dBV + 20];
//   spins flip (dS = 0): 41 entries [dBJ + 20].
// 1165 of the 5043 entries of the full dQ x dBV x dBJ table: 2.3 KB of levels
// instead of 10 KB, so that a CTA's prologue copies 5.4 KB, not 13.2 KB, and
// many small CTAs fit an SM.
constexpr int kSegR = 9;                      // |dBV|, |dBJ| of the first segment
constexpr int kSegW = 2 * kSegR + 1;          // 19
constexpr int kSegSwap = 3 * kSegW * kSegW;   // first entry of the second segment: 1083
constexpr int kSegFlip = kSegSwap + kNB;      // and of the third: 1124
constexpr int kDevN = kSegFlip + kNB;         // 1165
constexpr int kDevPad = (kDevN + 3) / 4 * 4;  // thr32 padded to 16 bytes

// Per-lattice parameter tables in device memory (built on the host).
struct DevTables {
  uint16_t *thrT;   // kThrT: threshold levels T = floor(5461 thr / 2^32), 5461 for
                    // thr = 0xFFFFFFFF (fast path)
  uint32_t *trans;  // kMoveN x 2 words: move entries (see kMoveN), directly after thrT
  uint32_t *thr32;  // kDevPad: full thresholds (exact path), directly after trans
};

// The fast path's threshold level of a 32-bit threshold: a field's w = v / 12
// (in [0, 5461)) below it accepts, above it rejects, equal to it is a tie.
__host__ __device__ inline uint16_t threshold_level(uint32_t thr) {
  return thr == 0xFFFFFFFFu ? (uint16_t)5461 : (uint16_t)(((uint64_t)thr * 5461u) >> 32);
}

// Move entries: one uint2 per (r, near, pc), entry (2 r + near) * 16 + (pc ^ r), i.e.
// at byte offset 256 r + 128 near + 8 (pc ^ r) -- r the pair's choice field mod 12
// (12 is a multiple of both q-set sizes, 4 and 6), near whether the partner is a
// nearest neighbour, pc = 4 code_a + code_b the pair state.
constexpr int kTransN = 16 * 12;     // entries of one kind (far or near)
constexpr int kMoveN = 2 * kTransN;  // both kinds
constexpr int kThrT = (kDevN + 7) / 8 * 8;  // 16-bit levels, padded to 16 bytes

struct LaunchCfg {
  int phase_grid_cap = 152 * 4;  // one resident wave of phase_kernel (set at create)
};

// One lattice of a resident launch (ccmc_resident.cu): held in the shared memory
// of one CTA or of a cluster, each CTA owning `rows` rows of every class.
struct ResJob {
  Geo g;                  // the lattice in global memory
  const uint16_t *thrT;   // its tables (levels, moves, full thresholds: one block)
  int nsweeps;            // sweeps to run in this launch, at most kResMaxSweeps
  int64_t *ring;          // observable ring (records every obs_every sweeps)
  int64_t ring_cap;
  int64_t *hist;          // histograms (nullptr: none)
  int nbins;
  int obs_every;
  int rows;
  alignas(16) uint32_t rk[20];  // Philox round keys: round r's at 2 r, 2 r + 1
};

// Launch shape of a resident launch: CTAs a lattice, rows of each class a CTA,
// threads a word, workers a CTA and all its threads, dynamic shared memory.
struct ResShape {
  int cluster = 0, rows = 0, tpw = 1, workers = 0, threads = 0;
  int64_t smem = 0;
};

constexpr int kResMaxWorkers = 512;
constexpr int kResQuadWords = 96;     // words a CTA that may have four threads each
constexpr int kResMaxThreads = 608;  // 96 registers a thread
static_assert(kResMaxWorkers + 32 <= kResMaxThreads && 6 * kResQuadWords + 32 <= kResMaxThreads,
              "workers, draw threads and the auxiliary warp");
constexpr int kResMaxCluster = 16;
constexpr int kResClusterWords = 128;  // lattices of fewer a-words a phase take one CTA
constexpr int kResMinWords = 16;       // a-words a CTA of a cluster at least
constexpr int kResMaxSweeps = 1 << 14;
constexpr int kResMaxSmem = 224 << 10;

// One lattice of a lock-step multi-lattice phase launch: CTAs
// [cta_begin, cta_begin + cta_count) of the grid work on it.
struct MultiJob {
  Geo g;
  const uint16_t *thrT;
  const uint32_t *thr32;
  uint32_t mw;  // row_magic
  int cta_begin, cta_count;
};

// ccmc_batch_config takes resident limits of at most four sites for every word of a
// CTA's shared memory but these and 64 (219,024 sites, 55 KB of packed words, on a
// GB300): a quarter of what one CTA holds, a limit that callers know.
constexpr int kConfigTableWords = 3292;

// Host-side table builders (ccmc_tables.cpp): the full table of
// ccmc_threshold_table (kTableN entries) and the device's (kDevN).
void build_thresholds(double beta, double Delta, double V, double J, uint32_t *thr32);
void build_device_thresholds(double beta, double Delta, double V, double J, uint32_t *thr32);
// Returns false if some entry could index outside its segment of the device's
// threshold table.
bool build_transitions(uint32_t *trans);

// Launchers (ccmc_kernels.cu).
cudaError_t launch_init(const Geo &g, int h, int64_t n_plus, int64_t n_minus, cudaStream_t s);
cudaError_t launch_phase(const Geo &g, const DevTables &t, int64_t p_off, const LaunchCfg &cfg,
                         cudaStream_t s);
int recount_grid(const Geo &g);
// CTAs of phase_kernel that fit the device at once (one wave).
int phase_resident_grid(bool aligned);
// One colour phase of every lattice in d_jobs (all aligned or all not).
cudaError_t launch_phase_multi(const MultiJob *d_jobs, int njobs, int grid, bool aligned,
                               int64_t p_off, cudaStream_t s);
// What the lock-step kernel's MultiJob::mw is for a lattice.
uint32_t row_magic(const Geo &g);
cudaError_t launch_recount(const Geo &g, int64_t *partials, int64_t *ring, int64_t ring_cap,
                           int64_t *hist, int nbins, int64_t sweep_off, cudaStream_t s);
cudaError_t launch_advance(int64_t *ctl, int64_t phases, cudaStream_t s);
cudaError_t launch_set_ctl(int64_t *ctl, int64_t phase_base, cudaStream_t s);
cudaError_t launch_gather_status(int64_t *const *ctls, int n, int64_t *out, cudaStream_t s);
cudaError_t launch_unpack(const Geo &g, uint8_t *out, cudaStream_t s);
cudaError_t launch_pack(const Geo &g, const uint8_t *in, int *bad, cudaStream_t s);
// Resident sweeps (ccmc_resident.cu): the most CTAs in a cluster (16, 8, 4, 2 or 1)
// that the current device places for any shape of the kernels, 0 when they cannot run
// there (raises the kernels' limits once per device; call outside a capture); a CTA's
// shared memory for `rows` rows of every class; and the launch of `one` lattice or
// of the njobs lattices of d_jobs (in device memory), all of one shape.
int resident_cluster_limit();
int64_t resident_smem(const Geo &g, int rows);
// The launch shape of a lattice that may take `ctas` CTAs of the GPU (at least
// one), clusters of max_cluster at most, while `load` a-words a phase run on an
// average SM, with at most max_threads workers a CTA and max_tpw threads a word.
ResShape resident_shape(const Geo &g, int max_cluster, double ctas, double load, int max_threads,
                        int max_tpw);
// Whether the lattice fits shared memory in some shape.
bool resident_possible(const Geo &g, int max_cluster);
// The shape for n such lattices in one launch: another one when their clusters
// would not all fit the GPU at once.
ResShape resident_fit(const Geo &g, int max_cluster, const ResShape &shape, bool aligned, int n);
cudaError_t launch_resident_sweep(const ResJob *one, const ResJob *d_jobs, int njobs,
                                  const ResShape &shape, bool aligned, cudaStream_t s);
cudaError_t launch_philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                          uint32_t k1, int64_t count, uint32_t *out, cudaStream_t s);

// ccmc_lattice_create without the final wait (wait false): the lattice's
// memory, tables and zeroed state are queued on its stream.
int lattice_new(int Lx, int Ly, void *cuda_stream, int64_t obs_capacity, bool wait,
                ccmc_lattice **out);

// ccmc_init_counts / ccmc_init_constrained without the final wait.
int init_counts_async(ccmc_lattice *h, uint64_t seed, int64_t n_plus, int64_t n_minus);
int init_constrained_async(ccmc_lattice *h, uint64_t seed, double n, double charged_frac);

// What a finished simulation reports, copied to pinned host memory by work
// queued on its stream (then `ready` recorded there): rec (8 int64), the
// latest exact recount (its word 0 is replaced by the sweeps done); status,
// the device-side error flag; count and ring (8 int64 a record, ring_cap
// records), the observable ring, when ring is not null; state (Lx Ly bytes),
// the site codes, when state is not null.
int export_async(ccmc_lattice *h, int64_t *rec, int64_t *status, int64_t *count, int64_t *ring,
                 uint8_t *state, cudaEvent_t ready);
// The observables of a record exported by export_async (its E from the
// lattice's parameters), and the records of an exported ring, oldest first.
void obs_of_record(const ccmc_lattice *h, const int64_t *rec, ccmc_obs *out);
int64_t series_of_ring(const ccmc_lattice *h, const int64_t *ring, int64_t count, ccmc_obs *out,
                       int64_t cap);
int64_t ring_capacity(const ccmc_lattice *h);
cudaStream_t lattice_stream(const ccmc_lattice *h);

// A batch with no fixed members, room for `cap` lattices, on `stream`.
int batch_new(int cap, cudaStream_t stream, ccmc_batch **out);

// Sweep a list of lattices (at most the batch's capacity) with per-lattice
// sweeps, parameters and observable intervals through the batch machinery.
// lockstep: large lattices at the same position may share phase launches
// (the launches are captured once per group and replayed, so the list should
// be the same on every call).
int batch_run(ccmc_batch *b, const std::vector<ccmc_lattice *> &lats, const int64_t *nsweeps,
              const double *beta, const double *Delta, const double *V, const double *J,
              const int *obs_every, bool lockstep);

}  // namespace ccmc
