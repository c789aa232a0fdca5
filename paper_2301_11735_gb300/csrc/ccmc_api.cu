// ccmc_api.cu -- the C ABI of libccmc (declared in include/ccmc.h): handle
// lifecycle, parameter tables, the sweep driver and state transfer.  Host code
// only; the kernels live in ccmc_kernels.cu.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "../../include/ccmc.h"
#include "ccmc_fault.h"
#include "ccmc_internal.h"
#include "ccmc_map.h"
#include "ccmc_state.h"
#include "ccmc_trace.h"

using namespace ccmc;

#define CK(call)                                \
  do {                                          \
    cudaError_t e_ = (call);                    \
    if (e_ != cudaSuccess) return CCMC_E_CUDA;  \
  } while (0)

namespace {

// A sweep of the graph path is captured as a chunk of `sweeps` sweeps; with
// obs_every in [1, 16] the chunk holds a recount after every obs_every-th
// sweep and is replayed only when the run is aligned to obs_every.
struct GraphEntry {
  int sweeps = 0;
  int obs_every = 0;
  cudaGraphExec_t exec = nullptr;
};

constexpr int kChunk = 16;
// Lock-step groups: at least kLockstepMin lattices, each with fewer than
// kLockstepMaxWords a-words per phase.  Measured on GB300, us a phase of all, lock
// step against their own streams, whose phases fill each other's tails: 8 of 1536^2
// (9216 words) 4.7 against 4.0, 16 6.8 against 7.4, 32 11.4 against 13.5; 16 of 1200^2
// 6.5 against 6.9, 40 11.7 against 16.5; 16 of 1980^2 (15345 words) 10.9 against 9.5,
// 64 33.1 against 32.0.
constexpr int kLockstepMin = 12;
constexpr int64_t kLockstepMaxWords = 12288;

// Lattice memory comes from a library-owned pool per device, kept cached:
// creating and destroying lattices never synchronises the device, which a server
// admitting and retiring simulations while others run depends on.  Everything is
// allocated and freed on one stream of the library's own, which carries nothing
// else: an allocation is complete when the call returns (any stream may use it),
// and a free follows the owner's last work, for which the caller has waited.
// (Allocating on every lattice's own stream made the pool grow by a chunk a
// stream: 0.2 to 0.8 ms a lattice when 512 were created, or read back for the
// first time; now 0.02.)
constexpr int kMaxDevices = 64;
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  cudaStream_t stream = nullptr;
};
std::mutex g_pool_mu;
DevicePool g_pool[kMaxDevices] = {};

// The device's pool (made on first use), nullptr when that fails.
const DevicePool *device_pool(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool &d = g_pool[dev];
  if (!d.stream && cudaStreamCreateWithFlags(&d.stream, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    d.stream = nullptr;
    return nullptr;
  }
  if (!d.pool) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    d.pool = p;
  }
  return &d;
}

// bytes of device memory of device dev, usable at once on any stream
bool dalloc(void **p, size_t bytes, int dev) {
  const DevicePool *d = device_pool(dev);
  *p = nullptr;
  if (!d || cudaMallocFromPoolAsync(p, bytes, d->pool, d->stream) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return false;
  }
  if (cudaStreamSynchronize(d->stream) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeAsync(*p, d->stream);
    *p = nullptr;
    return false;
  }
  return true;
}

// the caller has waited for the last work that uses p
void dfree(void *p, int dev) {
  const DevicePool *d = p ? device_pool(dev) : nullptr;
  if (d) cudaFreeAsync(p, d->stream);
}

// Pinned host buffers through which short results reach the caller: a copy or a
// kernel writes the buffer, one synchronisation, then a host copy (a copy to
// pageable memory stages and waits inside the driver: 15.5 us for a 16 KB state
// instead of 12.1).  At most kStages of kStageBytes for the process, lent for the
// length of one call; a caller that finds none takes the pageable path.
constexpr size_t kStageBytes = (size_t)1 << 20;
constexpr size_t kDirectBytes = (size_t)64 << 10;  // lattice states (see read_state)
constexpr size_t kStateBytes = (size_t)256 << 10;  // and those that nothing waits for
constexpr int kStages = 8;
std::mutex g_stage_mu;
std::vector<void *> g_stage_free;
int g_stage_made = 0;

class Stage {
 public:
  explicit Stage(size_t bytes) {
    if (bytes > kStageBytes) return;
    std::lock_guard<std::mutex> lock(g_stage_mu);
    if (!g_stage_free.empty()) {
      p_ = g_stage_free.back();
      g_stage_free.pop_back();
    } else if (g_stage_made < kStages &&
               cudaHostAlloc(&p_, kStageBytes, cudaHostAllocPortable) == cudaSuccess) {
      ++g_stage_made;
    } else {
      p_ = nullptr;
      cudaGetLastError();
    }
  }
  ~Stage() {
    if (!p_) return;
    std::lock_guard<std::mutex> lock(g_stage_mu);
    g_stage_free.push_back(p_);
  }
  Stage(const Stage &) = delete;
  Stage &operator=(const Stage &) = delete;
  explicit operator bool() const { return p_ != nullptr; }
  template <class T>
  T *as(size_t offset = 0) const {
    return reinterpret_cast<T *>(static_cast<char *>(p_) + offset);
  }

 private:
  void *p_ = nullptr;
};

}  // namespace

struct ccmc_lattice {
  Geo g{};
  int h = 1;  // Feistel half width: 4^h >= N
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int device = 0;
  void *d_slab = nullptr;  // one allocation: the members down to the flag
  uint32_t *d_words = nullptr;
  int64_t *d_ctl = nullptr;
  int64_t *d_partials = nullptr;
  int64_t *d_ring = nullptr;
  int64_t ring_cap = 0;
  DevTables t{};
  int *d_flag = nullptr;
  int64_t *d_hist = nullptr;
  int nbins = 0;
  uint8_t *d_bytes = nullptr;
  bool queued = true;  // work may be queued on `stream` that no call has waited for
  bool initialised = false;
  uint64_t seed = 0;
  int64_t phases_done = 0;  // global phase index of the next phase
  bool have_params = false;
  double params[4] = {0, 0, 0, 0};  // beta, Delta, V, J
  LaunchCfg cfg{};
  int max_cluster = 0;    // largest cluster its resident launches may take (0: none runs)
  bool resident = false;  // swept by the resident kernel
  std::vector<GraphEntry> graphs;
  int32_t *d_maps = nullptr;  // paper-map mode: uploaded pairs
  int64_t map_cap = 0;        // int32 entries held by d_maps
  cudaEvent_t map_ev = nullptr;
};

namespace {

// Lattices that the resident kernel sweeps unless the caller says otherwise: up
// to 4608 a-words a phase (1024^2 has 4096), 288 a CTA of a cluster of 16; a little
// further on a launch of a phase's own is as fast (us a sweep resident and with a
// launch a phase: 64^2 3.5, 16.9; 256^2 7.5, 18.3; 1000^2, ragged, 17.9, 23.6; 1024^2
// 15.0, 21.4; 1200^2 22.6, 23.4; 1280^2 22.5, 22.1; 1536^2 33.3, 22.9).
bool resident_default(const Geo &g, int max_cluster) {
  return g.cstride <= 4608 && resident_possible(g, max_cluster);
}

// How ccmc_sweep launches a lattice it holds in shared memory.
ResShape resident_alone(const Geo &g, int max_cluster) {
  return resident_shape(g, max_cluster, max_cluster, 0.0, kResMaxWorkers, 4);
}

// The move table, the same for every lattice (built and checked once: 25 us).
struct MoveTable {
  uint32_t words[2 * kMoveN];
  bool ok;
};

const MoveTable &move_table() {
  static const MoveTable t = [] {
    MoveTable m;
    m.ok = build_transitions(m.words);
    return m;
  }();
  return t;
}

int validate_shape(int Lx, int Ly) {
  if (Lx < 4 || Ly < 4 || (Lx & 3) || (Ly & 3)) return CCMC_E_INVAL;
  if ((int64_t)Lx * (int64_t)Ly > ((int64_t)1 << 30)) return CCMC_E_INVAL;
  // the phase kernels' byte offsets are 32-bit: 64 bytes a row of a class and block of
  // 16 columns, at most 2^32 of the sites above (Lx = 4)
  if (64 * (int64_t)(Ly / 4) * ((Lx / 4 + 15) / 16) > ((int64_t)1 << 32)) return CCMC_E_INVAL;
  return CCMC_OK;
}

Geo geometry(int Lx, int Ly) {
  Geo g{};
  g.Lx = Lx;
  g.Ly = Ly;
  g.Cx = Lx / 4;
  g.Cy = Ly / 4;
  g.W = (g.Cx + 15) / 16;
  g.cstride = (int64_t)g.Cy * g.W;
  const uint64_t N = (uint64_t)Lx * (uint64_t)Ly;
  g.rej = (0 - N) % N;
  return g;
}

// (a graph that is still running is freed when it has ended)
void drop_graphs(ccmc_lattice *h) {
  for (auto &e : h->graphs)
    if (e.exec) cudaGraphExecDestroy(e.exec);
  h->graphs.clear();
}

void set_seed(ccmc_lattice *h, uint64_t seed) {
  if (seed != h->seed) drop_graphs(h);  // captured phases hold the seed's Philox keys
  h->seed = seed;
  h->g.k0 = (uint32_t)(seed & 0xFFFFFFFFu);
  h->g.k1 = (uint32_t)(seed >> 32);
}

int upload_params_on(ccmc_lattice *h, double beta, double Delta, double V, double J,
                     cudaStream_t st) {
  if (h->have_params && h->params[0] == beta && h->params[1] == Delta && h->params[2] == V &&
      h->params[3] == J)
    return CCMC_OK;
  uint32_t thr32[kDevPad] = {};
  uint16_t thrT[kThrT] = {};
  build_device_thresholds(beta, Delta, V, J, thr32);
  for (int i = 0; i < kDevN; ++i) thrT[i] = threshold_level(thr32[i]);
  CK(cudaMemcpyAsync(h->t.thr32, thr32, sizeof(thr32), cudaMemcpyHostToDevice, st));
  CK(cudaMemcpyAsync(h->t.thrT, thrT, sizeof(thrT), cudaMemcpyHostToDevice, st));
  // pageable sources: the copies are staged before the calls return
  h->have_params = true;
  h->params[0] = beta;
  h->params[1] = Delta;
  h->params[2] = V;
  h->params[3] = J;
  return CCMC_OK;
}

int upload_params(ccmc_lattice *h, double beta, double Delta, double V, double J) {
  return upload_params_on(h, beta, Delta, V, J, h->stream);
}

// Queue `sweeps` sweeps starting at phase offset 0 of the control block's base;
// obs_every > 0: a recount after every obs_every-th of them (the caller aligns).
int enqueue_chunk(ccmc_lattice *h, int sweeps, int obs_every) {
  for (int s = 0; s < sweeps; ++s) {
    for (int p = 0; p < 8; ++p) CK(launch_phase(h->g, h->t, 8LL * s + p, h->cfg, h->stream));
    if (obs_every > 0 && (s + 1) % obs_every == 0)
      CK(launch_recount(h->g, h->d_partials, h->d_ring, h->ring_cap, h->d_hist, h->nbins, s + 1,
                        h->stream));
  }
  CK(launch_advance(h->d_ctl, 8LL * sweeps, h->stream));
  return CCMC_OK;
}

int run_graph(ccmc_lattice *h, int sweeps, int obs_every) {
  GraphEntry *hit = nullptr;
  for (auto &e : h->graphs)
    if (e.sweeps == sweeps && e.obs_every == obs_every) hit = &e;
  if (!hit) {
    cudaGraph_t graph = nullptr;
    CK(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    const int rc = enqueue_chunk(h, sweeps, obs_every);
    const cudaError_t ce = cudaStreamEndCapture(h->stream, &graph);
    if (rc != CCMC_OK || ce != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      return CCMC_E_CUDA;
    }
    GraphEntry e;
    e.sweeps = sweeps;
    e.obs_every = obs_every;
    const cudaError_t ie = cudaGraphInstantiate(&e.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess) return CCMC_E_CUDA;
    h->graphs.push_back(e);
    hit = &h->graphs.back();
  }
  CK(cudaGraphLaunch(hit->exec, h->stream));
  return CCMC_OK;
}

ResJob resident_job(const ccmc_lattice *h, int64_t nsweeps, int obs_every, int rows) {
  ResJob j{};
  j.g = h->g;
  j.thrT = h->t.thrT;
  j.nsweeps = (int)nsweeps;
  j.ring = h->d_ring;
  j.ring_cap = h->ring_cap;
  j.hist = h->d_hist;
  j.nbins = h->nbins;
  j.obs_every = obs_every;
  j.rows = rows;
  for (uint32_t r = 0; r < 10; ++r) {
    j.rk[2 * r] = h->g.k0 + r * 0x9E3779B9u;
    j.rk[2 * r + 1] = h->g.k1 + r * 0xBB67AE85u;
  }
  return j;
}

// Sweep one lattice by the resident kernel, a bounded number of sweeps a launch.
int resident_sweeps(ccmc_lattice *h, int64_t nsweeps, int obs_every) {
  const ResShape sh = resident_alone(h->g, h->max_cluster);
  for (int64_t s = 0; s < nsweeps; s += kResMaxSweeps) {
    const ResJob j =
        resident_job(h, std::min<int64_t>(nsweeps - s, kResMaxSweeps), obs_every, sh.rows);
    CK(launch_resident_sweep(&j, nullptr, 1, sh, (h->g.Cx & 15) == 0, h->stream));
  }
  return CCMC_OK;
}

// Drives nsweeps sweeps from absolute sweep index sweeps_done: replayable
// chunks of G sweeps (chunk(G, obs): G a multiple of obs when 0 < obs <= 16,
// started aligned to obs) where possible, single directly launched sweeps
// (single(obs_due)) to align or finish.
template <typename Chunk, typename Single>
int drive_sweeps(int64_t sweeps_done, int64_t nsweeps, int obs_every, Chunk chunk, Single single) {
  int64_t s = 0;
  while (s < nsweeps) {
    const int64_t abs_sweep = sweeps_done + s;
    const int64_t remaining = nsweeps - s;
    if (obs_every > 0 && obs_every <= kChunk) {
      const int g = obs_every * (kChunk / obs_every);
      if (abs_sweep % obs_every == 0 && remaining >= g) {
        const int rc = chunk(g, obs_every);
        if (rc) return rc;
        s += g;
        continue;
      }
    } else {
      const int64_t dist = obs_every > 0 ? obs_every - abs_sweep % obs_every : INT64_MAX;
      if (remaining >= kChunk && dist > kChunk) {
        const int rc = chunk(kChunk, 0);
        if (rc) return rc;
        s += kChunk;
        continue;
      }
    }
    const int rc = single(obs_every > 0 && (abs_sweep + 1) % obs_every == 0);
    if (rc) return rc;
    s += 1;
  }
  return CCMC_OK;
}

int write_recount_latest(ccmc_lattice *h) {
  CK(launch_recount(h->g, h->d_partials, nullptr, 0, nullptr, 0, 0, h->stream));
  return CCMC_OK;
}

void fill_obs(const ccmc_lattice *h, const int64_t *rec, ccmc_obs *o) {
  o->sweeps_done = rec[0];
  o->Nc = rec[1];
  o->BV = rec[2];
  o->BJ = rec[3];
  o->M = rec[4];
  o->M_stag = rec[5];
  o->S_sum = rec[6];
  o->S_stag = rec[7];
  const double Delta = h->params[1], V = h->params[2], J = h->params[3];
  o->E = Delta * (double)rec[1] + V * (double)rec[2] + (0.25 * J) * (double)rec[3];
}

// The control block's words as they are behind the work queued on the lattice's
// stream (synchronises it).
int read_ctl(ccmc_lattice *h, int64_t ctl[kCtlWords]) {
  const size_t n = sizeof(int64_t) * kCtlWords;
  Stage st(n);
  int64_t *to = st ? st.as<int64_t>() : ctl;
  CK(cudaMemcpyAsync(to, h->d_ctl, n, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  h->queued = false;
  if (st) std::memcpy(ctl, to, n);
  return CCMC_OK;
}

int check_status(ccmc_lattice *h) {
  int64_t ctl[kCtlWords];
  const int rc = read_ctl(h, ctl);
  if (rc) return rc;
  return ctl[kCtlStatus] == 0 ? CCMC_OK : CCMC_E_TIMEOUT;
}

}  // namespace

int ccmc::lattice_new(int Lx, int Ly, void *cuda_stream, int64_t obs_capacity, bool wait,
                      ccmc_lattice **out) {
  if (!out) return CCMC_E_INVAL;
  *out = nullptr;
  int rc = validate_shape(Lx, Ly);
  if (rc) return rc;
  if (fault_injected("alloc")) return CCMC_E_NOMEM;
  ccmc_lattice *h = new (std::nothrow) ccmc_lattice();
  if (!h) return CCMC_E_NOMEM;
  Geo &g = h->g;
  g = geometry(Lx, Ly);
  const uint64_t N = (uint64_t)Lx * (uint64_t)Ly;
  h->cfg.phase_grid_cap = phase_resident_grid((g.Cx & 15) == 0);
  // CCMC_TILE_GRID=n (tests): at most n CTAs a phase, so that small lattices take
  // several rounds of words a CTA
  if (const char *e = std::getenv("CCMC_TILE_GRID"))
    if (const int n = std::atoi(e); n > 0) h->cfg.phase_grid_cap = std::min(n, h->cfg.phase_grid_cap);
  // any of these variables (tests) keeps the lattice on the phase kernels
  h->max_cluster = resident_cluster_limit();
  if (h->max_cluster > 1 && fault_injected("cluster")) h->max_cluster = 1;
  h->resident = resident_default(g, h->max_cluster) && !std::getenv("CCMC_NO_TILE") &&
                !std::getenv("CCMC_TILE_GRID") && !std::getenv("CCMC_NO_RESIDENT");
  while (((int64_t)1 << (2 * h->h)) < (int64_t)N) ++h->h;
  h->ring_cap = obs_capacity > 0 ? obs_capacity : 4096;
  cudaGetDevice(&h->device);
  auto fail = [&](int code) {
    ccmc_lattice_destroy(h);
    return code;
  };
  if (cuda_stream) {
    h->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess)
      return fail(CCMC_E_CUDA);
    h->own_stream = true;
  }
  const int np = recount_grid(g);
  const int dev = h->device;
  // the threshold levels, the move table and the full thresholds one after another
  // (multiples of 16 bytes from a 256-byte aligned base): the kernels copy the first
  // two, or all three, into shared memory as one block
  size_t at = 0;
  auto part = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) & ~(size_t)255;
    return o;
  };
  const size_t o_words = part(sizeof(uint32_t) * 16 * g.cstride);
  const size_t o_tables =
      part(sizeof(uint16_t) * kThrT + sizeof(uint32_t) * (2 * kMoveN + kDevPad));
  const size_t o_ctl = part(sizeof(int64_t) * kCtlWords);
  const size_t o_partials = part(sizeof(int64_t) * 7 * np);
  const size_t o_flag = part(sizeof(int));
  const size_t o_ring = part(sizeof(int64_t) * 8 * h->ring_cap);
  if (!dalloc(&h->d_slab, at, dev)) return fail(CCMC_E_NOMEM);
  char *p = (char *)h->d_slab;
  h->d_words = (uint32_t *)(p + o_words);
  h->d_ctl = (int64_t *)(p + o_ctl);
  h->d_partials = (int64_t *)(p + o_partials);
  h->d_flag = (int *)(p + o_flag);
  h->d_ring = (int64_t *)(p + o_ring);
  p += o_tables;
  h->t.thrT = (uint16_t *)p;
  p += sizeof(uint16_t) * kThrT;
  h->t.trans = (uint32_t *)p;
  p += sizeof(uint32_t) * 2 * kMoveN;
  h->t.thr32 = (uint32_t *)p;
  g.words = h->d_words;
  g.ctl = h->d_ctl;
  const MoveTable &moves = move_table();
  if (!moves.ok) return fail(CCMC_E_INVAL);
  if (cudaMemcpyAsync(h->t.trans, moves.words, sizeof(moves.words), cudaMemcpyHostToDevice,
                      h->stream) != cudaSuccess ||
      cudaMemsetAsync(h->d_words, 0, sizeof(uint32_t) * 16 * g.cstride, h->stream) !=
          cudaSuccess ||
      launch_set_ctl(h->d_ctl, 0, h->stream) != cudaSuccess ||
      (wait && cudaStreamSynchronize(h->stream) != cudaSuccess))
    return fail(CCMC_E_CUDA);
  *out = h;
  return CCMC_OK;
}

static int ensure_bytes(ccmc_lattice *h) {
  if (h->d_bytes) return CCMC_OK;
  const size_t N = (size_t)h->g.Lx * h->g.Ly;
  if (!dalloc((void **)&h->d_bytes, N, h->device)) return CCMC_E_NOMEM;
  return CCMC_OK;
}

int ccmc::init_counts_async(ccmc_lattice *h, uint64_t seed, int64_t n_plus, int64_t n_minus) {
  if (!h) return CCMC_E_INVAL;
  const int64_t N = (int64_t)h->g.Lx * h->g.Ly;
  if (n_plus < 0 || n_minus < 0 || n_plus + n_minus > N) return CCMC_E_INVAL;
  h->queued = true;
  set_seed(h, seed);
  CK(launch_set_ctl(h->d_ctl, 0, h->stream));
  CK(launch_init(h->g, h->h, n_plus, n_minus, h->stream));
  if (h->d_hist) CK(cudaMemsetAsync(h->d_hist, 0, sizeof(int64_t) * 3 * h->nbins, h->stream));
  h->phases_done = 0;
  h->initialised = true;
  return CCMC_OK;
}

int ccmc::init_constrained_async(ccmc_lattice *h, uint64_t seed, double n, double charged_frac) {
  if (!h) return CCMC_E_INVAL;
  if (!std::isfinite(n)) return CCMC_E_INVAL;
  if (charged_frac < 0.0) charged_frac = 0.3;
  if (!std::isfinite(charged_frac)) return CCMC_E_INVAL;
  const int64_t N = (int64_t)h->g.Lx * h->g.Ly;
  const int64_t Q = std::llround(n * (double)N);
  int64_t C = std::llround(charged_frac * (double)N);
  const int64_t aQ = Q < 0 ? -Q : Q;
  if (C < aQ) C = aQ;
  if ((C - Q) & 1) C += 1;
  if (C > N) return CCMC_E_INVAL;
  return init_counts_async(h, seed, (C + Q) / 2, (C - Q) / 2);
}

int ccmc::export_async(ccmc_lattice *h, int64_t *rec, int64_t *status, int64_t *count,
                       int64_t *ring, uint8_t *state, cudaEvent_t ready) {
  if (!h || !rec || !status || !h->initialised) return CCMC_E_INVAL;
  h->queued = true;
  int rc = write_recount_latest(h);
  if (rc) return rc;
  CK(cudaMemcpyAsync(rec, h->d_ctl + kCtlLatest, sizeof(int64_t) * 8, cudaMemcpyDeviceToHost,
                     h->stream));
  CK(cudaMemcpyAsync(status, h->d_ctl + kCtlStatus, sizeof(int64_t), cudaMemcpyDeviceToHost,
                     h->stream));
  if (ring) {
    if (!count) return CCMC_E_INVAL;
    CK(cudaMemcpyAsync(count, h->d_ctl + kCtlObsCount, sizeof(int64_t), cudaMemcpyDeviceToHost,
                       h->stream));
    CK(cudaMemcpyAsync(ring, h->d_ring, sizeof(int64_t) * 8 * h->ring_cap,
                       cudaMemcpyDeviceToHost, h->stream));
  }
  if (state && (size_t)h->g.Lx * h->g.Ly <= (h->g.Lx % 16 ? 4096 : kStateBytes)) {
    CK(launch_unpack(h->g, state, h->stream));  // straight into the pinned buffer
  } else if (state) {
    rc = ensure_bytes(h);
    if (rc) return rc;
    CK(launch_unpack(h->g, h->d_bytes, h->stream));
    CK(cudaMemcpyAsync(state, h->d_bytes, (size_t)h->g.Lx * h->g.Ly, cudaMemcpyDeviceToHost,
                       h->stream));
  }
  CK(cudaEventRecord(ready, h->stream));
  return CCMC_OK;
}

void ccmc::obs_of_record(const ccmc_lattice *h, const int64_t *rec, ccmc_obs *out) {
  int64_t r[8];
  std::memcpy(r, rec, sizeof(r));
  r[0] = h->phases_done / 8;
  fill_obs(h, r, out);
}

int64_t ccmc::series_of_ring(const ccmc_lattice *h, const int64_t *ring, int64_t count,
                             ccmc_obs *out, int64_t cap) {
  const int64_t held = count < h->ring_cap ? count : h->ring_cap;
  int64_t n = 0;
  for (int64_t r = count - held; r < count && n < cap; ++r, ++n)
    fill_obs(h, ring + 8 * (r % h->ring_cap), out + n);
  return n;
}

int64_t ccmc::ring_capacity(const ccmc_lattice *h) { return h->ring_cap; }

cudaStream_t ccmc::lattice_stream(const ccmc_lattice *h) { return h->stream; }

extern "C" {

const char *ccmc_strerror(int code) {
  switch (code) {
    case CCMC_OK: return "ok";
    case CCMC_E_INVAL: return "invalid argument";
    case CCMC_E_NOMEM: return "out of memory";
    case CCMC_E_CUDA: return "CUDA error";
    case CCMC_E_TIMEOUT: return "device wait timed out";
    case CCMC_E_BUDGET: return "memory budget exhausted";
    case CCMC_E_STATE: return "call out of order";
    case CCMC_E_NOTFOUND: return "not found";
    default: return "unknown error";
  }
}

int ccmc_threshold_table(double beta, double Delta, double V, double J, uint32_t *out) {
  if (!out || !(beta >= 0.0) || !std::isfinite(Delta) || !std::isfinite(V) ||
      !std::isfinite(J))
    return CCMC_E_INVAL;
  build_thresholds(beta, Delta, V, J, out);
  return CCMC_OK;
}

int ccmc_resident_plan(int Lx, int Ly, int max_cluster, int64_t *plan) {
  if (!plan || max_cluster < 0 || max_cluster > kResMaxCluster ||
      (max_cluster & (max_cluster - 1)) || validate_shape(Lx, Ly) != CCMC_OK)
    return CCMC_E_INVAL;
  const Geo g = geometry(Lx, Ly);
  const ResShape sh =
      resident_default(g, max_cluster) ? resident_alone(g, max_cluster) : ResShape{};
  plan[0] = sh.cluster;
  plan[1] = sh.rows;
  plan[2] = sh.cluster ? sh.tpw : 0;
  plan[3] = sh.smem;
  return CCMC_OK;
}

int ccmc_lattice_create(int Lx, int Ly, void *cuda_stream, int64_t obs_capacity,
                        ccmc_lattice **out) {
  return lattice_new(Lx, Ly, cuda_stream, obs_capacity, true, out);
}

int ccmc_lattice_destroy(ccmc_lattice *h) {
  if (!h) return CCMC_E_INVAL;
  if (h->stream) cudaStreamSynchronize(h->stream);  // this lattice's work only
  drop_graphs(h);
  dfree(h->d_slab, h->device);
  dfree(h->d_hist, h->device);
  dfree(h->d_bytes, h->device);
  dfree(h->d_maps, h->device);
  if (h->map_ev) cudaEventDestroy(h->map_ev);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
  return CCMC_OK;
}

int ccmc_init_counts(ccmc_lattice *h, uint64_t seed, int64_t n_plus, int64_t n_minus) {
  const int rc = init_counts_async(h, seed, n_plus, n_minus);
  if (rc) return rc;
  CK(cudaStreamSynchronize(h->stream));
  h->queued = false;
  return CCMC_OK;
}

int ccmc_init_constrained(ccmc_lattice *h, uint64_t seed, double n, double charged_frac) {
  const int rc = init_constrained_async(h, seed, n, charged_frac);
  if (rc) return rc;
  CK(cudaStreamSynchronize(h->stream));
  h->queued = false;
  return CCMC_OK;
}

int ccmc_sweep(ccmc_lattice *h, int64_t nsweeps, double beta, double Delta, double V, double J,
               int obs_every) {
  if (!h || nsweeps < 0) return CCMC_E_INVAL;
  if (!(beta >= 0.0) || !std::isfinite(Delta) || !std::isfinite(V) || !std::isfinite(J))
    return CCMC_E_INVAL;
  if (!h->initialised) return CCMC_E_STATE;
  if (fault_injected("launch")) return CCMC_E_CUDA;
  TraceRange trace("ccmc_sweep");
  h->queued = true;
  int rc = upload_params(h, beta, Delta, V, J);
  if (rc) return rc;
  if (nsweeps > 0 && h->phases_done % 8) {
    // finish the sweep that ccmc_phases left open; it counts as the first one
    const int64_t rest = 8 - h->phases_done % 8;
    rc = ccmc_phases(h, rest, beta, Delta, V, J);
    if (rc) return rc;
    if (obs_every > 0 && (h->phases_done / 8) % obs_every == 0)
      CK(launch_recount(h->g, h->d_partials, h->d_ring, h->ring_cap, h->d_hist, h->nbins, 0,
                        h->stream));
    --nsweeps;
  }
  if (h->resident) {
    rc = resident_sweeps(h, nsweeps, obs_every);
    if (rc) return rc;
    h->phases_done += 8 * nsweeps;
    return CCMC_OK;
  }
  rc = drive_sweeps(
      h->phases_done / 8, nsweeps, obs_every,
      [&](int g, int obs) { return run_graph(h, g, obs); },
      [&](bool obs_due) {
        for (int p = 0; p < 8; ++p) CK(launch_phase(h->g, h->t, p, h->cfg, h->stream));
        if (obs_due)
          CK(launch_recount(h->g, h->d_partials, h->d_ring, h->ring_cap, h->d_hist, h->nbins, 1,
                            h->stream));
        CK(launch_advance(h->d_ctl, 8, h->stream));
        return CCMC_OK;
      });
  if (rc) return rc;
  h->phases_done += 8 * nsweeps;
  return CCMC_OK;
}

int ccmc_phases(ccmc_lattice *h, int64_t nphases, double beta, double Delta, double V,
                double J) {
  if (!h || nphases < 0) return CCMC_E_INVAL;
  if (!(beta >= 0.0) || !std::isfinite(Delta) || !std::isfinite(V) || !std::isfinite(J))
    return CCMC_E_INVAL;
  if (!h->initialised) return CCMC_E_STATE;
  if (fault_injected("launch")) return CCMC_E_CUDA;
  h->queued = true;
  int rc = upload_params(h, beta, Delta, V, J);
  if (rc) return rc;
  for (int64_t p = 0; p < nphases; ++p) {
    CK(launch_phase(h->g, h->t, 0, h->cfg, h->stream));
    CK(launch_advance(h->d_ctl, 1, h->stream));
  }
  h->phases_done += nphases;
  return CCMC_OK;
}

int ccmc_sync(ccmc_lattice *h) {
  if (!h) return CCMC_E_INVAL;
  return check_status(h);
}

int ccmc_map_apply(ccmc_lattice *h, const int32_t *pairs, int64_t map0, int64_t nmaps,
                   double beta, double Delta, double V, double J) {
  if (!h || map0 < 0 || nmaps < 0 || (nmaps > 0 && !pairs) || !(beta >= 0.0) ||
      !std::isfinite(Delta) || !std::isfinite(V) || !std::isfinite(J))
    return CCMC_E_INVAL;
  if (!h->initialised) return CCMC_E_STATE;
  if (nmaps == 0) return CCMC_OK;
  const int64_t P = ccmc_map_size(h->g.Lx, h->g.Ly);
  const int64_t N = (int64_t)h->g.Lx * h->g.Ly;
  if (nmaps > ((int64_t)1 << 40) / (2 * P)) return CCMC_E_INVAL;
  const int64_t n = 2 * P * nmaps;
  h->queued = true;
  // the kernel addresses the lattice with these indices: reject any outside it
  for (int64_t i = 0; i < n; ++i)
    if (pairs[i] < 0 || pairs[i] >= N) return CCMC_E_INVAL;
  if (!h->map_ev && cudaEventCreateWithFlags(&h->map_ev, cudaEventDisableTiming) != cudaSuccess)
    return CCMC_E_CUDA;
  if (n > h->map_cap) {
    if (h->d_maps) CK(cudaStreamSynchronize(h->stream));  // the earlier maps' work
    dfree(h->d_maps, h->device);
    h->d_maps = nullptr;
    h->map_cap = 0;
    if (!dalloc((void **)&h->d_maps, sizeof(int32_t) * n, h->device))
      return CCMC_E_NOMEM;
    h->map_cap = n;
  }
  int rc = upload_params(h, beta, Delta, V, J);
  if (rc) return rc;
  CK(cudaMemcpyAsync(h->d_maps, pairs, sizeof(int32_t) * n, cudaMemcpyHostToDevice, h->stream));
  CK(cudaEventRecord(h->map_ev, h->stream));
  for (int64_t k = 0; k < nmaps; ++k)
    CK(launch_map(h->g, h->d_maps + 2 * P * k, P, (uint64_t)(map0 + k), h->t, h->stream));
  // the caller may reuse `pairs` once the copy has run
  CK(cudaEventSynchronize(h->map_ev));
  return CCMC_OK;
}

int ccmc_observables(ccmc_lattice *h, ccmc_obs *out) {
  if (!h || !out) return CCMC_E_INVAL;
  if (!h->initialised) return CCMC_E_STATE;
  h->queued = true;
  int rc = write_recount_latest(h);
  if (rc) return rc;
  int64_t ctl[kCtlWords];
  rc = read_ctl(h, ctl);
  if (rc) return rc;
  int64_t *rec = ctl + kCtlLatest;
  rec[0] = h->phases_done / 8;
  fill_obs(h, rec, out);
  return ctl[kCtlStatus] == 0 ? CCMC_OK : CCMC_E_TIMEOUT;
}

int ccmc_obs_series(ccmc_lattice *h, ccmc_obs *out, int64_t cap, int64_t *n_written) {
  if (!h || !n_written || cap < 0 || (cap > 0 && !out)) return CCMC_E_INVAL;
  const size_t head = sizeof(int64_t) * kCtlWords, bytes = sizeof(int64_t) * 8 * h->ring_cap;
  Stage st(head + bytes);
  int64_t ctl[kCtlWords];
  std::vector<int64_t> own;
  const int64_t *ring = nullptr;
  if (st) {  // control block and ring behind one synchronisation
    CK(cudaMemcpyAsync(st.as<char>(), h->d_ctl, head, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaMemcpyAsync(st.as<char>(head), h->d_ring, bytes, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    h->queued = false;
    std::memcpy(ctl, st.as<char>(), head);
    ring = st.as<int64_t>(head);
  } else {
    const int rc = read_ctl(h, ctl);
    if (rc) return rc;
    own.resize((size_t)(8 * h->ring_cap));
    CK(cudaMemcpyAsync(own.data(), h->d_ring, bytes, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    ring = own.data();
  }
  *n_written = series_of_ring(h, ring, ctl[kCtlObsCount], out, cap);
  return CCMC_OK;
}

int ccmc_hist_enable(ccmc_lattice *h, int nbins) {
  if (!h || nbins < 1 || nbins > (1 << 20)) return CCMC_E_INVAL;
  CK(cudaStreamSynchronize(h->stream));
  drop_graphs(h);  // captured recounts hold the old histogram pointer
  dfree(h->d_hist, h->device);
  h->d_hist = nullptr;
  h->nbins = 0;
  if (!dalloc((void **)&h->d_hist, sizeof(int64_t) * 3 * nbins, h->device))
    return CCMC_E_NOMEM;
  h->nbins = nbins;
  h->queued = true;
  CK(cudaMemsetAsync(h->d_hist, 0, sizeof(int64_t) * 3 * nbins, h->stream));
  return CCMC_OK;
}

int ccmc_hist_get(ccmc_lattice *h, int64_t *out) {
  if (!h || !out) return CCMC_E_INVAL;
  if (!h->d_hist) return CCMC_E_STATE;
  CK(cudaMemcpyAsync(out, h->d_hist, sizeof(int64_t) * 3 * h->nbins, cudaMemcpyDeviceToHost,
                     h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return CCMC_OK;
}


}  // extern "C"

// Hands `n` bytes of state made by `make(device pointer)` to the caller: at most
// `direct` of them through a pinned buffer that the kernel writes itself, longer ones by
// a copy from device memory, which the driver stages.  (us a call, written into a pinned
// buffer and copied by the driver: 4 KB 11.4 and 15.2, 64 KB 15.2 and 15.6, 96 KB 17.2 and
// 17.1, 256 KB 26.5 and 17.3; packed rows written in single bytes 12 KB 16.4 and 17.5,
// 16 KB 17.7 and 18.5, 24 KB 19.4 and 17.3, 64 KB 24.2 and 17.4.  A copy to the pinned
// buffer and another on the host is never the fastest.)
template <typename Make>
static int read_state(ccmc_lattice *h, uint8_t *host_out, size_t n, size_t direct, Make make) {
  if (!h || !host_out) return CCMC_E_INVAL;
  if (!h->initialised) return CCMC_E_STATE;
  Stage st(n <= direct ? n : kStageBytes + 1);
  if (st) {
    CK(make(st.as<uint8_t>()));
    CK(cudaStreamSynchronize(h->stream));
    std::memcpy(host_out, st.as<uint8_t>(), n);
  } else {
    const int rc = ensure_bytes(h);
    if (rc) return rc;
    CK(make(h->d_bytes));
    CK(cudaMemcpyAsync(host_out, h->d_bytes, n, cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
  }
  h->queued = false;
  return CCMC_OK;
}

extern "C" {

int ccmc_get_state(ccmc_lattice *h, uint8_t *host_out) {
  return read_state(h, host_out, h ? (size_t)h->g.Lx * h->g.Ly : 0, kDirectBytes,
                    [&](uint8_t *to) { return launch_unpack(h->g, to, h->stream); });
}

int ccmc_get_state_packed(ccmc_lattice *h, uint8_t *host_out) {
  return read_state(h, host_out, h ? (size_t)h->g.Lx * h->g.Ly / 4 : 0,
                    h && h->g.Lx % 64 ? kDirectBytes / 4 : kDirectBytes,
                    [&](uint8_t *to) { return launch_unpack2(h->g, to, h->stream); });
}

int ccmc_set_state_packed(ccmc_lattice *h, const uint8_t *host_in, uint64_t seed,
                          int64_t sweeps_done) {
  if (!h || !host_in || sweeps_done < 0 || sweeps_done > ((int64_t)1 << 59)) return CCMC_E_INVAL;
  h->queued = true;
  int rc = ensure_bytes(h);
  if (rc) return rc;
  const size_t nb = (size_t)h->g.Lx * h->g.Ly / 4;
  // every 2-bit code is a state: nothing to validate, nothing to wait for
  CK(cudaMemcpyAsync(h->d_bytes, host_in, nb, cudaMemcpyHostToDevice, h->stream));
  set_seed(h, seed);
  CK(launch_pack2(h->g, h->d_bytes, h->stream));
  CK(launch_set_ctl(h->d_ctl, 8 * sweeps_done, h->stream));
  if (h->d_hist) CK(cudaMemsetAsync(h->d_hist, 0, sizeof(int64_t) * 3 * h->nbins, h->stream));
  h->phases_done = 8 * sweeps_done;
  h->initialised = true;
  return CCMC_OK;
}

int ccmc_set_state(ccmc_lattice *h, const uint8_t *host_in, uint64_t seed, int64_t sweeps_done) {
  if (!h || !host_in || sweeps_done < 0) return CCMC_E_INVAL;
  h->queued = true;
  int rc = ensure_bytes(h);
  if (rc) return rc;
  const size_t N = (size_t)h->g.Lx * h->g.Ly;
  int zero = 0, bad = 0;
  CK(cudaMemcpyAsync(h->d_flag, &zero, sizeof(int), cudaMemcpyHostToDevice, h->stream));
  CK(cudaMemcpyAsync(h->d_bytes, host_in, N, cudaMemcpyHostToDevice, h->stream));
  set_seed(h, seed);
  CK(launch_pack(h->g, h->d_bytes, h->d_flag, h->stream));
  CK(launch_set_ctl(h->d_ctl, 8 * sweeps_done, h->stream));
  if (h->d_hist) CK(cudaMemsetAsync(h->d_hist, 0, sizeof(int64_t) * 3 * h->nbins, h->stream));
  CK(cudaMemcpyAsync(&bad, h->d_flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (bad) {
    h->initialised = false;
    return CCMC_E_INVAL;
  }
  h->phases_done = 8 * sweeps_done;
  h->initialised = true;
  return CCMC_OK;
}

}  // extern "C"

// ----------------------------------------------------------------------------
// Batches: many lattices swept together.  Lattices up to the resident limit run in
// shared memory, one resident_sweep_kernel launch a shape, side by side on streams
// that fork from the batch stream and join it; larger ones run the per-phase path
// on their own streams, or in lock step, at the same time.
struct ccmc_batch {
  std::vector<ccmc_lattice *> lats;
  int cap = 0;  // largest number of lattices one launch may hold
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  int device = 0;
  void *d_slab = nullptr;    // one allocation: the next two and d_multi
  ResJob *d_jobs = nullptr;  // resident lattices
  int64_t **d_ctls = nullptr;  // the members' control blocks (a batch with fixed members)
  int threads = kResMaxWorkers;
  int64_t resident_max_sites = -1;  // -1: the lattices that ccmc_sweep holds resident
  int ctas_per_sm = 1;
  int max_tpw = 4;
  int sms = 152;
  cudaEvent_t ev = nullptr;
  std::vector<cudaEvent_t> lat_ev;
  std::vector<cudaStream_t> side;   // resident launches of different shapes run side by side
  std::vector<cudaEvent_t> side_ev;
  MultiJob *d_multi = nullptr;  // lock-step groups of large lattices
  struct MultiGraph {
    std::vector<ccmc_lattice *> members;
    int sweeps, obs_every;
    int64_t off;
    cudaGraphExec_t exec;
    std::vector<std::pair<int64_t *, int>> hists;  // the members', held by its recounts
  };
  std::vector<MultiGraph> graphs;
};

namespace {

// Whether a batch holds a lattice in shared memory: below the configured limit, or
// what ccmc_sweep would hold.
bool batch_resident(const ccmc_batch *b, const ccmc_lattice *h) {
  if (b->resident_max_sites < 0) return h->resident;
  return h->max_cluster > 0 && 16 * h->g.cstride * 16 <= b->resident_max_sites;
}

// A resident launch of a batch: lattices of one shape.
struct ResGroup {
  ResShape shape;
  bool aligned;
  double cost;             // of its longest lattice
  std::vector<ResJob> jobs;
};

constexpr int kSideStreams = 8;

int side_streams(ccmc_batch *b, int n) {
  while ((int)b->side.size() < n) {
    cudaStream_t s = nullptr;
    cudaEvent_t e = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return CCMC_E_CUDA;
    b->side.push_back(s);
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return CCMC_E_CUDA;
    b->side_ev.push_back(e);
  }
  return CCMC_OK;
}

// Queue the resident launches of lats[which] (ordered after the batch stream's
// work; the batch stream waits for them).
int run_resident(ccmc_batch *b, const std::vector<ccmc_lattice *> &lats,
                 const std::vector<int> &which, const int64_t *nsweeps, const int *obs_every) {
  // every lattice's share of the CTAs the GPU holds, by its work in this launch (a
  // lattice with many sweeps left gets more, so that it does not end alone)
  double words = 0, work = 0;
  for (int i : which) {
    words += (double)lats[i]->g.cstride;
    work += (double)lats[i]->g.cstride * (double)nsweeps[i];
  }
  const double ctas = (double)b->sms * b->ctas_per_sm;
  struct Plan {
    int i;
    ResShape shape;
    bool aligned;
  };
  std::vector<Plan> plans;
  for (int i : which) {
    const Geo &g = lats[i]->g;
    plans.push_back({i,
                     resident_shape(g, lats[i]->max_cluster,
                                    ctas * (double)g.cstride * (double)nsweeps[i] / work,
                                    words / b->sms, b->threads, b->max_tpw),
                     (g.Cx & 15) == 0});
  }
  auto same = [](const ResShape &x, const ResShape &y) {
    return x.cluster == y.cluster && x.tpw == y.tpw && x.workers == y.workers;
  };
  std::vector<ResGroup> groups;
  for (const Plan &p : plans) {
    const ccmc_lattice *h = lats[p.i];
    ResShape sh = p.shape;
    if (sh.cluster > 1) {
      int n = 0;
      for (const Plan &o : plans) n += same(o.shape, p.shape);
      sh = resident_fit(h->g, h->max_cluster, sh, p.aligned, n);
    }
    ResGroup *hit = nullptr;
    for (ResGroup &G : groups)
      if (same(G.shape, sh) && G.aligned == p.aligned) hit = &G;
    if (!hit) {
      groups.push_back(ResGroup{sh, p.aligned, 0.0, {}});
      hit = &groups.back();
    }
    hit->shape.smem = std::max(hit->shape.smem, sh.smem);
    hit->cost = std::max(hit->cost, (double)sh.rows * h->g.W * (double)nsweeps[p.i]);
    hit->jobs.push_back(resident_job(h, nsweeps[p.i], obs_every[p.i], sh.rows));
  }
  // the longest first, in every launch and over the launches
  std::sort(groups.begin(), groups.end(),
            [](const ResGroup &x, const ResGroup &y) { return x.cost > y.cost; });
  std::vector<ResJob> jobs;
  for (ResGroup &G : groups) {
    std::stable_sort(G.jobs.begin(), G.jobs.end(), [](const ResJob &x, const ResJob &y) {
      return (double)x.rows * x.g.W * x.nsweeps > (double)y.rows * y.g.W * y.nsweeps;
    });
    jobs.insert(jobs.end(), G.jobs.begin(), G.jobs.end());
  }
  CK(cudaMemcpyAsync(b->d_jobs, jobs.data(), sizeof(ResJob) * jobs.size(), cudaMemcpyHostToDevice,
                     b->stream));
  const int n = (int)groups.size(), side = std::min(n - 1, kSideStreams);
  const int rc = side_streams(b, side);
  if (rc) return rc;
  if (side > 0) CK(cudaEventRecord(b->ev, b->stream));
  for (int k = 0; k < side; ++k) CK(cudaStreamWaitEvent(b->side[k], b->ev, 0));
  int64_t off = 0;
  for (int k = 0; k < n; ++k) {
    const ResGroup &G = groups[k];
    const int on = k % (side + 1);
    if (k == 1 && fault_injected("group")) return CCMC_E_CUDA;
    CK(launch_resident_sweep(nullptr, b->d_jobs + off, (int)G.jobs.size(), G.shape, G.aligned,
                             on == 0 ? b->stream : b->side[on - 1]));
    off += (int64_t)G.jobs.size();
  }
  for (int k = 0; k < side; ++k) {
    CK(cudaEventRecord(b->side_ev[k], b->side[k]));
    CK(cudaStreamWaitEvent(b->stream, b->side_ev[k], 0));
  }
  return CCMC_OK;
}

}  // namespace

namespace {

struct MultiGroup {
  std::vector<ccmc_lattice *> m;
  int64_t off;  // first slot in d_multi
  int grid;
  bool aligned;
};

int enqueue_multi_chunk(ccmc_batch *b, const MultiGroup &G, int sweeps, int obs_every) {
  for (int s = 0; s < sweeps; ++s) {
    for (int p = 0; p < 8; ++p)
      CK(launch_phase_multi(b->d_multi + G.off, (int)G.m.size(), G.grid, G.aligned,
                                      8LL * s + p, b->stream));
    if (obs_every > 0 && (s + 1) % obs_every == 0)
      for (ccmc_lattice *h : G.m)
        CK(launch_recount(h->g, h->d_partials, h->d_ring, h->ring_cap, h->d_hist, h->nbins,
                          s + 1, b->stream));
  }
  for (ccmc_lattice *h : G.m) CK(launch_advance(h->d_ctl, 8LL * sweeps, b->stream));
  return CCMC_OK;
}

int run_multi_graph(ccmc_batch *b, const MultiGroup &G, int sweeps, int obs_every) {
  std::vector<std::pair<int64_t *, int>> hists;
  for (const ccmc_lattice *h : G.m) hists.emplace_back(h->d_hist, h->nbins);
  for (size_t i = 0; i < b->graphs.size(); ++i) {
    ccmc_batch::MultiGraph &e = b->graphs[i];
    if (e.members != G.m || e.sweeps != sweeps || e.obs_every != obs_every || e.off != G.off)
      continue;
    if (e.hists == hists) {
      CK(cudaGraphLaunch(e.exec, b->stream));
      return CCMC_OK;
    }
    // a member's histograms were enabled since: its captured recounts hold the old ones
    cudaGraphExecDestroy(e.exec);
    b->graphs.erase(b->graphs.begin() + (ptrdiff_t)i);
    break;
  }
  cudaGraph_t graph = nullptr;
  CK(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
  const int rc = enqueue_multi_chunk(b, G, sweeps, obs_every);
  const cudaError_t ce = cudaStreamEndCapture(b->stream, &graph);
  if (rc != CCMC_OK || ce != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return CCMC_E_CUDA;
  }
  ccmc_batch::MultiGraph e{G.m, sweeps, obs_every, G.off, nullptr, hists};
  const cudaError_t ie = cudaGraphInstantiate(&e.exec, graph, 0);
  cudaGraphDestroy(graph);
  if (ie != cudaSuccess) return CCMC_E_CUDA;
  b->graphs.push_back(e);
  CK(cudaGraphLaunch(e.exec, b->stream));
  return CCMC_OK;
}

// Sweep a lock-step group (same position, sweeps, observable interval and
// alignment) with one phase launch per phase for all of them.
int run_multi(ccmc_batch *b, MultiGroup &G, int64_t nsweeps, int obs_every) {
  int64_t words = 0;
  for (ccmc_lattice *h : G.m) words += (int64_t)h->g.Cy * h->g.W;
  const int wave = G.m[0]->cfg.phase_grid_cap;  // the same for all of one alignment
  std::vector<MultiJob> jobs;
  int begin = 0;
  for (ccmc_lattice *h : G.m) {
    const int64_t w = (int64_t)h->g.Cy * h->g.W;
    int share = (int)((double)wave * (double)w / (double)words);
    const int64_t need = (w + 255) / 256;  // more CTAs than a word each would idle
    if (share > need) share = (int)need;
    if (share < 1) share = 1;
    MultiJob j{};
    j.g = h->g;
    j.thrT = h->t.thrT;
    j.thr32 = h->t.thr32;
    j.mw = row_magic(h->g);
    j.cta_begin = begin;
    j.cta_count = share;
    begin += share;
    jobs.push_back(j);
  }
  G.grid = begin;
  CK(cudaMemcpyAsync(b->d_multi + G.off, jobs.data(), sizeof(MultiJob) * jobs.size(),
                     cudaMemcpyHostToDevice, b->stream));
  const int rc = drive_sweeps(
      G.m[0]->phases_done / 8, nsweeps, obs_every,
      [&](int g, int obs) { return run_multi_graph(b, G, g, obs); },
      [&](bool obs_due) {
        for (int p = 0; p < 8; ++p)
          CK(launch_phase_multi(b->d_multi + G.off, (int)G.m.size(), G.grid, G.aligned,
                                          p, b->stream));
        if (obs_due)
          for (ccmc_lattice *h : G.m)
            CK(launch_recount(h->g, h->d_partials, h->d_ring, h->ring_cap, h->d_hist, h->nbins,
                              1, b->stream));
        for (ccmc_lattice *h : G.m) CK(launch_advance(h->d_ctl, 8, b->stream));
        return CCMC_OK;
      });
  if (rc) return rc;
  for (ccmc_lattice *h : G.m) h->phases_done += 8 * nsweeps;
  return CCMC_OK;
}

// Queues the sweeps of lattices that batch_run has checked.
int batch_queue(ccmc_batch *b, const std::vector<ccmc_lattice *> &lats, const int64_t *nsweeps,
                const double *beta, const double *Delta, const double *V, const double *J,
                const int *obs_every, bool lockstep) {
  const int n = (int)lats.size();
  std::vector<int> resident;
  for (int i = 0; i < n; ++i) {
    ccmc_lattice *h = lats[i];
    if (nsweeps[i] == 0 || !batch_resident(b, h)) continue;
    // order the batch stream after work already queued on this lattice's stream (a
    // stream of the library's own that a call has waited for carries none)
    if (h->stream != b->stream && (h->queued || !h->own_stream)) {
      CK(cudaEventRecord(b->lat_ev[i], h->stream));
      CK(cudaStreamWaitEvent(b->stream, b->lat_ev[i], 0));
    }
    int rc = upload_params_on(h, beta[i], Delta[i], V[i], J[i], b->stream);
    if (rc) return rc;
    resident.push_back(i);
  }
  if (!resident.empty()) {
    // a bounded number of sweeps a launch
    std::vector<int64_t> left(nsweeps, nsweeps + n), now(n);
    for (std::vector<int> go = resident; !go.empty();) {
      for (int i : go) left[i] -= now[i] = std::min<int64_t>(left[i], kResMaxSweeps);
      const int rc = run_resident(b, lats, go, now.data(), obs_every);
      if (rc) return rc;
      go.erase(std::remove_if(go.begin(), go.end(), [&](int i) { return left[i] == 0; }),
               go.end());
    }
    CK(cudaEventRecord(b->ev, b->stream));
    for (int i : resident) {
      ccmc_lattice *h = lats[i];
      h->phases_done += 8 * nsweeps[i];
      h->queued = true;
      if (h->stream != b->stream) CK(cudaStreamWaitEvent(h->stream, b->ev, 0));
    }
  }
  // The large lattices: those at the same position with the same sweeps,
  // observable interval and alignment advance in lock-step with one phase
  // launch for all of them (on the batch stream); the others run the per-phase
  // path on their own streams.  Both overlap the resident launch.
  std::vector<char> used(n, 0);
  int64_t off = 0;
  for (int i = 0; i < n; ++i) {
    ccmc_lattice *h = lats[i];
    if (used[i] || nsweeps[i] == 0 || batch_resident(b, h)) continue;
    MultiGroup G{{h}, off, 0, (h->g.Cx & 15) == 0};
    used[i] = 1;
    auto small = [](const ccmc_lattice *x) { return (int64_t)x->g.Cy * x->g.W < kLockstepMaxWords; };
    for (int k = i + 1; k < n && lockstep && small(h); ++k) {
      ccmc_lattice *o = lats[k];
      if (used[k] || nsweeps[k] != nsweeps[i] || obs_every[k] != obs_every[i] ||
          o->phases_done != h->phases_done || ((o->g.Cx & 15) == 0) != G.aligned ||
          !small(o) || batch_resident(b, o))
        continue;
      G.m.push_back(o);
      used[k] = 1;
    }
    // Few or large lattices run on their own streams (see kLockstepMin).
    if ((int)G.m.size() < kLockstepMin) {
      for (ccmc_lattice *o : G.m) {
        const int k = (int)(std::find(lats.begin(), lats.end(), o) - lats.begin());
        const int rc = ccmc_sweep(o, nsweeps[k], beta[k], Delta[k], V[k], J[k], obs_every[k]);
        if (rc) return rc;
      }
      continue;
    }
    for (ccmc_lattice *o : G.m) {
      const int k = (int)(std::find(lats.begin(), lats.end(), o) - lats.begin());
      if (o->stream != b->stream) {
        CK(cudaEventRecord(b->lat_ev[k], o->stream));
        CK(cudaStreamWaitEvent(b->stream, b->lat_ev[k], 0));
      }
      const int rc = upload_params_on(o, beta[k], Delta[k], V[k], J[k], b->stream);
      if (rc) return rc;
    }
    const int rc = run_multi(b, G, nsweeps[i], obs_every[i]);
    if (rc) return rc;
    off += (int64_t)G.m.size();
    CK(cudaEventRecord(b->ev, b->stream));
    for (ccmc_lattice *o : G.m) {
      o->queued = true;
      if (o->stream != b->stream) CK(cudaStreamWaitEvent(o->stream, b->ev, 0));
    }
  }
  return CCMC_OK;
}

}  // namespace

namespace ccmc {

int batch_run(ccmc_batch *b, const std::vector<ccmc_lattice *> &lats, const int64_t *nsweeps,
              const double *beta, const double *Delta, const double *V, const double *J,
              const int *obs_every, bool lockstep) {
  const int n = (int)lats.size();
  if (n > b->cap) return CCMC_E_INVAL;
  TraceRange trace("ccmc_batch_run");
  for (int i = 0; i < n; ++i) {
    if (nsweeps[i] < 0 || !(beta[i] >= 0.0) || !std::isfinite(Delta[i]) ||
        !std::isfinite(V[i]) || !std::isfinite(J[i]))
      return CCMC_E_INVAL;
    ccmc_lattice *h = lats[i];
    if (!h || !h->initialised || h->phases_done % 8) return CCMC_E_STATE;
    for (int k = 0; k < i; ++k)
      if (lats[k] == h) return CCMC_E_INVAL;  // a lattice may appear once
  }
  const int rc = batch_queue(b, lats, nsweeps, beta, Delta, V, J, obs_every, lockstep);
  if (rc != CCMC_OK) {
    // some launches may be queued that no lattice's stream waits for: they end before
    // the caller may destroy a lattice and its memory goes to another
    cudaStreamSynchronize(b->stream);
    for (cudaStream_t x : b->side) cudaStreamSynchronize(x);
  }
  return rc;
}

}  // namespace ccmc

extern "C" {

int ccmc_batch_create(int count, ccmc_lattice *const *lattices, void *cuda_stream,
                      ccmc_batch **out) {
  if (!out || count < 1 || !lattices) return CCMC_E_INVAL;
  *out = nullptr;
  for (int i = 0; i < count; ++i)
    if (!lattices[i]) return CCMC_E_INVAL;
  if (ccmc::fault_injected("alloc")) return CCMC_E_NOMEM;
  const int rc = ccmc::batch_new(count, (cudaStream_t)cuda_stream, out);
  if (rc != CCMC_OK) return rc;
  (*out)->lats.assign(lattices, lattices + count);
  std::vector<int64_t *> ctls;
  for (int i = 0; i < count; ++i) ctls.push_back(lattices[i]->d_ctl);
  if (cudaMemcpyAsync((*out)->d_ctls, ctls.data(), sizeof(int64_t *) * count,
                      cudaMemcpyHostToDevice, (*out)->stream) != cudaSuccess) {
    ccmc_batch_destroy(*out);
    *out = nullptr;
    return CCMC_E_CUDA;
  }
  return CCMC_OK;
}

}  // extern "C"

int ccmc::batch_new(int cap, cudaStream_t stream, ccmc_batch **out) {
  if (!out || cap < 1) return CCMC_E_INVAL;
  *out = nullptr;
  ccmc_batch *b = new (std::nothrow) ccmc_batch();
  if (!b) return CCMC_E_NOMEM;
  b->cap = cap;
  const int count = cap;
  void *cuda_stream = (void *)stream;
  auto fail = [&](int code) {
    ccmc_batch_destroy(b);
    return code;
  };
  if (cuda_stream) {
    b->stream = (cudaStream_t)cuda_stream;
  } else {
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess)
      return fail(CCMC_E_CUDA);
    b->own_stream = true;
  }
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev);
  b->device = dev;
  const size_t o_multi = (sizeof(ResJob) * count + 255) & ~(size_t)255;
  const size_t o_ctls = o_multi + ((sizeof(MultiJob) * count + 255) & ~(size_t)255);
  if (!dalloc(&b->d_slab, o_ctls + sizeof(int64_t *) * count, dev)) return fail(CCMC_E_NOMEM);
  b->d_jobs = (ResJob *)b->d_slab;
  b->d_multi = (MultiJob *)((char *)b->d_slab + o_multi);
  b->d_ctls = (int64_t **)((char *)b->d_slab + o_ctls);
  if (cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) != cudaSuccess)
    return fail(CCMC_E_CUDA);
  b->lat_ev.assign(count, nullptr);
  for (auto &e : b->lat_ev)
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess)
      return fail(CCMC_E_CUDA);
  *out = b;
  return CCMC_OK;
}

extern "C" {

int ccmc_batch_destroy(ccmc_batch *b) {
  if (!b) return CCMC_E_INVAL;
  if (b->stream) cudaStreamSynchronize(b->stream);
  for (auto &e : b->graphs)
    if (e.exec) cudaGraphExecDestroy(e.exec);
  for (cudaStream_t x : b->side) cudaStreamSynchronize(x);
  dfree(b->d_slab, b->device);
  for (cudaStream_t x : b->side) cudaStreamDestroy(x);
  for (cudaEvent_t e : b->side_ev) cudaEventDestroy(e);
  if (b->ev) cudaEventDestroy(b->ev);
  for (auto e : b->lat_ev)
    if (e) cudaEventDestroy(e);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
  delete b;
  return CCMC_OK;
}

int ccmc_batch_config(ccmc_batch *b, int resident_threads, int64_t resident_max_sites,
                      int ctas_per_sm, int max_threads_per_word) {
  if (!b) return CCMC_E_INVAL;
  if (resident_threads != 64 && resident_threads != 128 && resident_threads != 256 &&
      resident_threads != 512)
    return CCMC_E_INVAL;
  if (max_threads_per_word != 1 && max_threads_per_word != 2 && max_threads_per_word != 4)
    return CCMC_E_INVAL;
  if (resident_max_sites < 0 || ctas_per_sm < 1 || ctas_per_sm > 32) return CCMC_E_INVAL;
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int64_t max_words = optin / 4 - kConfigTableWords - 64;
  if (resident_max_sites / 4 > max_words) return CCMC_E_INVAL;
  b->threads = resident_threads;
  b->resident_max_sites = resident_max_sites;
  b->ctas_per_sm = ctas_per_sm;
  b->max_tpw = max_threads_per_word;
  return CCMC_OK;
}

int ccmc_batch_sweep(ccmc_batch *b, const int64_t *nsweeps, const double *beta,
                     const double *Delta, const double *V, const double *J, int obs_every) {
  if (!b || !nsweeps || !beta || !Delta || !V || !J) return CCMC_E_INVAL;
  if (ccmc::fault_injected("launch")) return CCMC_E_CUDA;
  std::vector<int> every(b->lats.size(), obs_every);
  return ccmc::batch_run(b, b->lats, nsweeps, beta, Delta, V, J, every.data(), true);
}

int ccmc_batch_sync(ccmc_batch *b) {
  if (!b) return CCMC_E_INVAL;
  CK(cudaStreamSynchronize(b->stream));
  const int n = (int)b->lats.size();
  const size_t bytes = sizeof(int64_t) * n;
  Stage st(bytes);
  if (!st) {
    for (ccmc_lattice *h : b->lats) {
      const int rc = check_status(h);
      if (rc) return rc;
    }
    return CCMC_OK;
  }
  // every member's stream, then all their status words at once
  for (ccmc_lattice *h : b->lats) {
    CK(cudaStreamSynchronize(h->stream));
    h->queued = false;
  }
  CK(launch_gather_status(b->d_ctls, n, st.as<int64_t>(), b->stream));
  CK(cudaStreamSynchronize(b->stream));
  for (int i = 0; i < n; ++i)
    if (st.as<int64_t>()[i]) return CCMC_E_TIMEOUT;
  return CCMC_OK;
}

int ccmc_selftest_wait(uint32_t polls) {
  if (polls == 0 || polls > (1u << 24)) return CCMC_E_INVAL;
  int *d = nullptr;
  if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return CCMC_E_NOMEM;
  int status = 0;
  int rc = CCMC_OK;
  if (cudaMemset(d, 0, sizeof(int)) != cudaSuccess ||
      ccmc::launch_wait_selftest(polls, d, 0) != cudaSuccess ||
      cudaMemcpy(&status, d, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = CCMC_E_CUDA;
  cudaFree(d);
  if (rc) return rc;
  return status ? CCMC_E_TIMEOUT : CCMC_OK;
}

int ccmc_philox_device(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                       uint32_t k1, int64_t count, uint32_t *out) {
  if (!out || count < 0 || count > ((int64_t)1 << 28)) return CCMC_E_INVAL;
  if (count == 0) return CCMC_OK;
  uint32_t *d = nullptr;
  if (cudaMalloc(&d, sizeof(uint32_t) * 4 * count) != cudaSuccess) return CCMC_E_NOMEM;
  int rc = CCMC_OK;
  if (launch_philox(c0, c1, c2, c3, k0, k1, count, d, 0) != cudaSuccess ||
      cudaMemcpy(out, d, sizeof(uint32_t) * 4 * count, cudaMemcpyDeviceToHost) != cudaSuccess)
    rc = CCMC_E_CUDA;
  cudaFree(d);
  return rc;
}

}  // extern "C"
