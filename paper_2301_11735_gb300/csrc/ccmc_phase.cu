// ccmc_phase.cu -- the colour-phase kernels of the coupled-pair Metropolis
// sweep for sm_103a (one lattice per launch: direct and tile-staged; several
// lattices in lock step) and their launchers (declared in ccmc_internal.h).  The
// resident kernel, whole sweeps of lattices that fit shared memory, is in
// ccmc_resident.cu.
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "ccmc_device.cuh"
#include "ccmc_internal.h"
#include "ccmc_launch.cuh"
#include "ccmc_word.cuh"

namespace ccmc {

// ============================================================================
// One colour phase (Sec. 3.1-3.2).  A word of the a-class holds 16 pairs
// (a, a + r), site t of the word at bits 2t..2t+1.  Its pairs are read as the
// a word, the four neighbour windows of a, the b window and the four neighbour
// windows of b; every pair's move is evaluated; the a word is stored and the
// changed b sites are XORed back.
//
// Random fields: pair t takes the 16-bit half (t mod 2) of word (t / 4) mod 4
// of MOVE call c = (t / 2) mod 2 of its word, i.e. call c serves the pair
// groups k = 2c (low halves) and k = 2c + 1 (high halves), group k being the
// sites k, k + 4, k + 8, k + 12 (lane q = site / 4).  Per pair, with pc =
// 4 code_a + code_b and its field v:
//   w      = floor(v / 12), the choice class v - 12 w (v < 65532 = 12 x 5461)
//   entry  = trans[v - 12 w][near][pc] -> base, byte coefficients, pc XOR npc
//   offset = dp4a(coefficients, (2 n1_a, n0_a, 2 n1_b, n0_b), base), n1 and n0 the
//            neighbours with bit 1, bit 0 set (byte offset of the level)
//   accept = w < T(offset), with T = floor(5461 thr / 2^32) (5461 when thr is
//            0xFFFFFFFF): w < T implies w 2^32 + s < 5461 thr for every 32-bit
//            s, w > T the opposite
// A tie (w == T) or a field v >= 65532 (about one pair in 4000, rejected by the
// fast decision) is decided exactly, with the pair's SLOW random words.
struct PhaseSmem {
  alignas(16) uint16_t thrT[kThrT];
  uint2 trans[kMoveN];  // directly after thrT, as in device memory
  PhaseD u;
  uint64_t P;
};

__device__ __forceinline__ int wrap(int v, int n) { return v >= n ? v - n : (v < 0 ? v + n : v); }

// The direct path's view of a word: row j, word w of the classes in global memory
// (class offsets in words), rows of whole words (kAl) or of any width.
template <bool kAl>
struct DirectView {
  const Geo &g;
  const PhaseD &u;
  int j, w;

  // sites of the window from one class row
  __device__ __forceinline__ uint32_t window(const uint32_t *row, const Win &x) const {
    uint32_t v = __funnelshift_r(row[x.lo], row[x.hi], x.sh);
    if constexpr (!kAl) {
      if (x.n1 < 16)  // the row ends inside the window: go on at its start
        v = (v & ((1u << (2 * x.n1)) - 1u)) | (row[0] << (2 * x.n1));
    }
    return v;
  }
  __device__ __forceinline__ WordIn gather() const {
    WordIn in;
    const SideD &a = u.side[0], &b = u.side[1];
    const int jb = turn(j + b.qy, g.Cy);
    const uint32_t *rb = g.words + (int64_t)jb * g.W,
                   *ry = g.words + (int64_t)turn(jb + b.ys, g.Cy) * g.W;
    const Win win = window_at<kAl>(g, w, b.qx);
    in.B = window(rb + b.c, win);
    in.nb = neighbour_planes(window(rb + b.m, win), window(rb + b.r, win), window(ry + b.y, win),
                             window(rb + b.x, window_at<kAl>(g, w, b.offX)));
    const uint32_t *ra = g.words + (int64_t)j * g.W;
    in.A = ra[a.c + w];
    in.na = neighbour_planes(ra[a.m + w], ra[a.r + w],
                             g.words[a.y + (int64_t)turn(j + a.ys, g.Cy) * g.W + w],
                             window(ra + a.x, window_at<kAl>(g, w, a.offX)));
    return in;
  }
  // a's word by a plain read-modify-write (kOwn: its thread's own) or by atomic XOR;
  // the b sites by atomic XOR (their words are shared with the partners of
  // neighbouring words)
  template <bool kOwn>
  __device__ __forceinline__ void change(int jj, int ww, uint32_t dA, uint32_t dB) const {
    const SideD &a = u.side[0], &b = u.side[1];
    if constexpr (!kAl) {
      const int n = g.Cx - (ww << 4);
      if (n < 16) {  // pairs past the end of the row do not exist
        const uint32_t valid = (1u << (2 * n)) - 1u;
        dA &= valid;
        dB &= valid;
      }
    }
    if (dA) {
      uint32_t *pa = g.words + a.c + (int64_t)jj * g.W + ww;
      if constexpr (kOwn)
        *pa ^= dA;
      else
        atomicXor(pa, dA);
    }
    if (dB) {
      uint32_t *row = g.words + b.c + (int64_t)turn(jj + b.qy, g.Cy) * g.W;
      const Win x = window_at<kAl>(g, ww, b.qx);
      uint32_t d1 = dB;
      if constexpr (!kAl) {
        if (x.n1 < 16) {
          d1 = dB & ((1u << (2 * x.n1)) - 1u);
          const uint32_t d2 = dB >> (2 * x.n1);
          if (d2) atomicXor(row, d2);
        }
      }
      const uint32_t lo = d1 << x.sh, hi = __funnelshift_l(d1, 0u, x.sh);
      if (lo) atomicXor(row + x.lo, lo);
      if (hi) atomicXor(row + x.hi, hi);
    }
  }
  __device__ __forceinline__ void apply(uint32_t dA, uint32_t dB) const {
    change<true>(j, w, dA, dB);
  }
  __device__ __forceinline__ void apply_other(int oj, int ow, uint32_t dA, uint32_t dB) const {
    change<false>(oj, ow, dA, dB);
  }
};

// One word's pairs by one lane, with all 32 lanes of the warp calling
// together (inactive lanes: active false): the fast decisions are applied;
// then, for every lane with rare calls (about one word in 250), the warp
// decides that word's rare pairs together, one pair a lane, from the owner's
// inputs.  The rare pairs were rejected by the fast path, and no other pair of
// the phase touches their sites or neighbours, so the order does not matter.
// view: how the word is read and changed; j: its row in the class (keys the random
// streams), w its place in the row; near128: 128 if the phase's partners are
// nearest neighbours, else 0; keys: the source of the Philox keys (SeedKeys or
// TableKeys of the lattice's seed).
template <class View, class Keys>
__device__ __forceinline__ void warp_word(const Geo &g, const View &view, const uint2 *trans,
                                          const uint16_t *thrT, const uint32_t *thr32, int j,
                                          int w, uint64_t P, uint32_t near128, const Keys &keys,
                                          bool active = true) {
  WordIn in{};
  uint32_t rz = 0u;
  if (active) {
    in = view.gather();
    const uint32_t gbase = (uint32_t)j * (uint32_t)(2 * g.W) + (uint32_t)(2 * w);
    const uint3 d = fast_moves<1, false>(trans, thrT, 0, in, near128, [&](int c) {
      return keys(gbase + (uint32_t)c, (uint32_t)P, (uint32_t)(P >> 32), TAG_MOVE);
    });
    view.apply(d.x, d.y);
    rz = d.z;
  }
  unsigned ball = __ballot_sync(0xFFFFFFFFu, rz != 0u);
  if (ball) {
    const int lane = threadIdx.x & 31;
    __syncwarp();  // the fast moves of every lane are in memory
#pragma unroll 1
    while (ball) {
      const int src = __ffs(ball) - 1;
      ball &= ball - 1u;
      const uint32_t orz = __shfl_sync(0xFFFFFFFFu, rz, src);
      WordIn o;
      o.A = __shfl_sync(0xFFFFFFFFu, in.A, src);
      o.B = __shfl_sync(0xFFFFFFFFu, in.B, src);
      o.na.O = __shfl_sync(0xFFFFFFFFu, in.na.O, src);
      o.na.T = __shfl_sync(0xFFFFFFFFu, in.na.T, src);
      o.na.F = __shfl_sync(0xFFFFFFFFu, in.na.F, src);
      o.nb.O = __shfl_sync(0xFFFFFFFFu, in.nb.O, src);
      o.nb.T = __shfl_sync(0xFFFFFFFFu, in.nb.T, src);
      o.nb.F = __shfl_sync(0xFFFFFFFFu, in.nb.F, src);
      const int oj = __shfl_sync(0xFFFFFFFFu, j, src), ow = __shfl_sync(0xFFFFFFFFu, w, src);
      // the owner's pairs, one a lane: half h of call c, word lane & 3 of it
      const int c = (lane >> 3) & 1, h = (lane >> 2) & 1;
      const int t = 2 * c + h + 4 * (lane & 3);
      if (lane < 16 && ((orz >> c) & 1u) && 16 * ow + t < g.Cx) {
        const uint32_t x = exact_move(g, trans, thrT, thr32, oj, ow, t, o, P, near128);
        if (x) view.apply_other(oj, ow, (x >> 2) << (2 * t), (x & 3u) << (2 * t));
      }
    }
  }
}

// One phase on the direct path.  The prologue (tables, and for a launch after the
// first of a chain the phase index and its schedule) runs before the kernel waits
// for its predecessor, as in the tile kernels.  Small lattices take small CTAs: a
// thread's chain is what they wait for, and it is shorter on an SM of its own.
template <bool kAligned>
__global__ void __launch_bounds__(256, 4) phase_kernel(Geo g, const uint16_t *thrT,
                                                       const uint32_t *thr32, int64_t p_off,
                                                       const __grid_constant__ RoundKeys rk) {
  __shared__ PhaseSmem sm;
  // The tables come from host uploads that precede the whole launch chain.
  for (int t = threadIdx.x; t < (int)((2u * kThrT + 8u * kMoveN) / 16u); t += blockDim.x)
    reinterpret_cast<uint4 *>(sm.thrT)[t] = reinterpret_cast<const uint4 *>(thrT)[t];
  auto prologue = [&] {
    if (threadIdx.x < 32) {
      const uint64_t P = (uint64_t)(g.ctl[kCtlPhaseBase] + p_off);
      const Sched s = draw_schedule(g, P);
      if (threadIdx.x == 0) {
        sm.u = phase_desc(g, s, (uint32_t)g.cstride);
        sm.P = P;
      }
    }
  };
  const bool pre = p_off > 0;  // the counter's base is two launches old (see tile_phase)
  if (pre) prologue();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // The next kernel may launch now: with one resident wave its blocks only take
  // the slots of blocks that finish, and it waits for this whole grid before
  // touching the lattice.
  asm volatile("griddepcontrol.launch_dependents;");
  if (!pre) prologue();
  __syncthreads();
  const PhaseD &u = sm.u;
  const uint64_t P = sm.P;
  const uint32_t near128 = u.near128;
  const int nw = g.Cy * g.W;
  const int stride = gridDim.x * blockDim.x;
  for (int base = blockIdx.x * blockDim.x; base < nw; base += stride) {
    const int wid = base + threadIdx.x;
    const bool act = wid < nw;
    const int j = act ? wid / g.W : 0, w = act ? wid - j * g.W : 0;
    warp_word(g, DirectView<kAligned>{g, u, j, w}, sm.trans, sm.thrT, thr32, j, w, P, near128,
              TableKeys{&rk}, act);
  }
}

// ----------------------------------------------------------------------------
// Tile-staged phase (lattices whose class rows are W words with W dividing 256
// and a multiple of 4, and Cy a multiple of R = 256 / W).  A tile is R
// consecutive rows of the a-class (256 words, one per thread).  CTA c takes
// tiles c, c + grid, ... c + (kBufs - 1) grid first, then claims tiles beyond
// kBufs grid one at a time from a counter in the lattice's control block, so
// that CTAs which start late (placed on an SM whose previous CTA finished
// last) take fewer tiles instead of ending the phase late.  The claim for a
// buffer is made when the buffer is refilled, kBufs - 1 tiles ahead of its
// use, so its latency is hidden.  Phase P claims from slot P mod 2; its kernel
// tags slot (P + 1) mod 2 for phase P + 1 (with P + 1 in the high word) once
// phase P - 1 is done with it; a slot whose tag is not the phase's own (the
// previous phase ran on another path, or the phase counter was just set: that
// zeroes both slots) makes every CTA of the phase keep to the fixed order c +
// t grid.  A tile's ten row bands -- the a rows,
// the b rows and the rows of all eight neighbour classes, each band R full
// rows -- arrive in shared memory by bulk asynchronous copies (one band per
// lane of the staging warp) that complete on the buffer's `full` mbarrier.
// The threads evaluate their words from shared memory.  The last warp to
// finish a tile (counted on the buffer's arrival counter) sends its a and b
// bands back to global memory with plain vector stores and stages the tile
// kBufs later into the same buffer, so every buffer is refilled as soon as it
// is free, kBufs - 1 tiles ahead of its use, and no warp waits for another
// warp except on a tile's data.  (A fixed staging thread that first evaluated
// its own word trailed the slowest warp every tile; the other warps' polls
// then starved it of issue slots: first tiles landed 2.6 to 19 us after a
// phase started.)  Waits suspend in hardware (try_wait with a time hint)
// instead of spinning.  No two tiles of a phase write the same rows (each b
// row is the partner row of exactly one a row), and no tile reads a row
// another tile writes (the pairs of a phase do not interact), so global memory
// sees no atomics and staging may run ahead of the write-back.
constexpr int kTileWords = 256;
constexpr int kBands = 10;
constexpr int kTileBufs = 3;
constexpr uint32_t kTileBytes = kBands * kTileWords * 4;
constexpr uint32_t kWaitSpins = 1u << 24;              // bounded mbarrier waits:
constexpr unsigned long long kWaitNs = 1000000000ull;  // at most 2^24 polls or 1 s
constexpr uint32_t kSuspendNs = 20000;                 // suspend-time hint of a poll

// The lattice's threshold levels and the move table, contiguous in device
// memory (thrT, trans), staged with one bulk copy.
constexpr uint32_t kStagedTableBytes = 2u * kThrT + 8u * kMoveN;
static_assert(kStagedTableBytes % 16 == 0, "bulk copies move multiples of 16 bytes");

// Row band: R rows of one class starting at row j0 + dy of the tile's first a
// row j0 (periodic in Cy).
struct Band {
  const uint32_t *cls;
  int dy;
};

// The tile phase's column uniforms.  Each side is staged as five bands: the class
// itself, the column neighbour in the same columns, the one xs = -1, 0 or 1 sites
// further, and the two row neighbours, whose band starts at the right row (a side's
// neighbours differ in no other way: see the resident kernel's SideD).
enum BandOf { kA = 0, kAm, kAx, kAr, kAy, kB, kBm, kBx, kBr, kBy };
struct TileCols {
  int xA;          // a's further column neighbour
  int qx, offX;    // b's columns and its further column neighbour's
};

// The tile path's view of a word: its byte offsets in a band, the same in every
// tile of a phase, so that all sixteen loads are a base, one of seven offsets and
// the band's constant.  (Taking every window's words from its own column offset,
// with class pointers, cost 60 more instructions a word.)
struct TileView {
  char *band;  // the tile's bands in shared memory
  uint32_t own, alo, ahi, blo, bhi, xlo, xhi;
  int ash, bsh, xsh;

  __device__ __forceinline__ TileView(const TileCols &c, int W, int jr, int w) {
    const int m = W - 1;  // W is a power of two
    const uint32_t row = 4u * (uint32_t)(jr * W);
    auto at = [&](int i) { return row + 4u * (uint32_t)(i & m); };
    band = nullptr;
    own = at(w);
    alo = c.xA < 0 ? at(w - 1) : own;
    ahi = c.xA > 0 ? at(w + 1) : own;
    ash = 2 * c.xA & 31;
    blo = at(w + (c.qx >> 4));
    bhi = at(w + (c.qx >> 4) + 1);
    bsh = 2 * (c.qx & 15);
    xlo = at(w + (c.offX >> 4));
    xhi = at(w + (c.offX >> 4) + 1);
    xsh = 2 * (c.offX & 15);
  }
  __device__ __forceinline__ uint32_t &word(int k, uint32_t off) const {
    return *reinterpret_cast<uint32_t *>(band + off + (uint32_t)(k * kTileWords * 4));
  }
  __device__ __forceinline__ uint32_t window(int k) const {
    return __funnelshift_r(word(k, blo), word(k, bhi), bsh);
  }
  __device__ __forceinline__ WordIn gather() const {
    WordIn in;
    in.A = word(kA, own);
    in.B = window(kB);
    in.na = neighbour_planes(word(kAm, own), word(kAr, own), word(kAy, own),
                             __funnelshift_r(word(kAx, alo), word(kAx, ahi), ash));
    in.nb = neighbour_planes(window(kBm), window(kBr), window(kBy),
                             __funnelshift_r(word(kBx, xlo), word(kBx, xhi), xsh));
    return in;
  }
  __device__ __forceinline__ void apply_b(uint32_t dB) const {
    if (dB) {
      atomicXor(&word(kB, blo), dB << bsh);
      const uint32_t hi = __funnelshift_l(dB, 0u, bsh);  // dB >> (32 - bsh), 0 for 0
      if (hi) atomicXor(&word(kB, bhi), hi);
    }
  }
  __device__ __forceinline__ void apply(uint32_t dA, uint32_t dB) const {
    if (dA) word(kA, own) ^= dA;
    apply_b(dB);
  }
};

// A tile's words seen by the warp's exact path: another lane's word from its place.
struct TileWord {
  const TileView &v;
  const TileCols &c;
  int W, j0;

  __device__ __forceinline__ WordIn gather() const { return v.gather(); }
  __device__ __forceinline__ void apply(uint32_t dA, uint32_t dB) const { v.apply(dA, dB); }
  __device__ __forceinline__ void apply_other(int oj, int ow, uint32_t dA, uint32_t dB) const {
    TileView o(c, W, oj - j0, ow);
    o.band = v.band;
    if (dA) atomicXor(&o.word(kA, o.own), dA);
    o.apply_b(dB);
  }
};

// kBufs: band buffers (three for the pipelined tile loop, one for a CTA that
// takes a single tile).
template <int kBufs = kTileBufs>
struct TileSmem {
  alignas(128) uint16_t thrT[kThrT];
  uint2 trans[kMoveN];  // directly after thrT, as in device memory
  alignas(128) uint32_t band[kBufs][kBands][kTileWords];
  alignas(8) unsigned long long full[kBufs];  // bands landed (transaction count)
  alignas(8) unsigned long long tables;       // the tables landed
  int done[kBufs];     // warps finished with the buffer's tile
  int armed[kBufs];    // times the buffer's `full` barrier was armed
  int tile[kBufs];     // the tile staged in the buffer, -1: no more tiles
  Band bands[kBands];
  TileCols cols;
  uint32_t near128;
  int err;
  int busy0, busy1;  // classes the previous phase writes (early staging waits for them)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for the phase of parity `parity` of the mbarrier at `bar` to complete:
// true when it did, false after kWaitSpins polls or kWaitNs nanoseconds.  Each
// poll may suspend the thread (up to kSuspendNs) until the phase completes.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (uint32_t i = 0; i < kWaitSpins; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(kSuspendNs)
        : "memory");
    if (ok) return true;
    if ((i & 63u) == 0) {
      const unsigned long long t = global_ns();
      if (i == 0)
        t0 = t;
      else if (t - t0 > kWaitNs)
        return false;
    }
  }
  return false;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      :
      : "r"(dst), "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// One tile-staged phase of lattice g by CTA `cta` of the `ncta` CTAs that
// work on it; keys: the source of its Philox keys.
// kSingle: every CTA takes at most one tile (ncta == tiles): one band buffer.
template <bool kSingle, class Keys>
__device__ __forceinline__ void tile_phase(const Geo &g, const uint16_t *thrT,
                                           const uint32_t *thr32, int64_t p_off, int cta,
                                           int ncta, const Keys &keys) {
  extern __shared__ __align__(128) unsigned char tile_smem[];
  constexpr int kBufs = kSingle ? 1 : kTileBufs;
  constexpr int kWarps = kTileWords / 32;
  using Smem = TileSmem<kBufs>;
  Smem &sm = *reinterpret_cast<Smem *>(tile_smem);
  static_assert(offsetof(Smem, trans) == 2 * kThrT, "tables staged as one block");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sm.err = 0;
    for (int b = 0; b < kBufs; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.full[b])));
      sm.done[b] = 0;
      sm.armed[b] = 0;
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.tables)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // The tables come from host uploads that precede the whole launch chain:
    // their copy may start before the previous kernel of the stream finishes.
    const uint32_t bar = smem_u32(&sm.tables);
    mbar_expect(bar, kStagedTableBytes);
    bulk_load(smem_u32(sm.thrT), thrT, kStagedTableBytes, bar);
  }
  // The phase index.  A launch after the first of a chain (p_off > 0) reads the
  // counter base, draws its schedule and places its bands before it waits for
  // its predecessor: the base was written by a kernel at least two launches
  // back (the chain's counter advance), which the predecessor's
  // griddepcontrol.wait has already waited for.  With several tiles a CTA it
  // then stages the bands of its first tiles that lie in classes the
  // predecessor (phase P - 1, whose schedule it draws too) does not write,
  // while that phase is still finishing, and the other bands once it has
  // finished.  Only lattices whose phases give every CTA several tiles do
  // this: for smaller ones it measured slower when several lattices share the
  // GPU on their own streams.
  const bool pre = p_off > 0;
  const bool early = !kSingle && pre && g.Cy / (kTileWords / g.W) > ncta;
  if (!pre) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
  }
  const uint64_t P = (uint64_t)(g.ctl[kCtlPhaseBase] + p_off);
  if (warp == 0) {
    const Sched sc = draw_schedule(g, P);
    if (early) {
      const Sched pv = draw_schedule(g, P - 1u);
      if (lane == 0) {
        sm.busy0 = pv.a0y * 4 + pv.a0x;
        sm.busy1 = ((pv.a0y + pv.ry) & 3) * 4 + ((pv.a0x + pv.rx) & 3);
      }
    }
    if (lane == 0) {
      sm.near128 = sc.near ? 128u : 0u;
      const int bx = sc.a0x + sc.rx, by = sc.a0y + sc.ry;
      const int qx = (bx >> 2) % g.Cx, qy = (by >> 2) % g.Cy;
      auto cls = [&](int x, int y) {
        return g.words + (int64_t)((y & 3) * 4 + (x & 3)) * g.cstride;
      };
      // bands k .. k + 4 of the side at class (cx, cy), dy rows below the a rows;
      // returns where its further column neighbour lies
      auto side = [&](int k, int cx, int cy, int dy) {
        const int dx = cx == 3 ? 1 : -1, dr = cy == 3 ? 1 : -1;
        sm.bands[k + kA] = {cls(cx, cy), dy};
        sm.bands[k + kAm] = {cls(cx - dx, cy), dy};
        sm.bands[k + kAx] = {cls(cx + dx, cy), dy};
        sm.bands[k + kAr] = {cls(cx, cy - dr), dy};
        sm.bands[k + kAy] = {cls(cx, cy + dr), dy + (cy == 0 ? -1 : cy == 3 ? 1 : 0)};
        return cx == 0 ? -1 : cx == 3 ? 1 : 0;
      };
      sm.cols.xA = side(kA, sc.a0x, sc.a0y, 0);
      const int xB = side(kB, bx & 3, by & 3, qy);
      sm.cols.qx = qx;
      sm.cols.offX = wrap(qx + xB, g.Cx);
    }
  }
  __syncthreads();
  const uint32_t near128 = sm.near128;
  const int W = g.W, R = kTileWords / W, Cy = g.Cy;
  const int ntiles = Cy / R;
  const uint32_t row_bytes = (uint32_t)W * 4u;

  // lane `lane` (< kBands) of the calling warp: the bulk loads of band `lane`
  // of tile `tile` into buffer b, if `mask` selects it
  auto stage_band = [&](int tile, int b, unsigned mask) {
    if (lane < kBands && ((mask >> lane) & 1u)) {
      const Band bd = sm.bands[lane];
      const int j0 = tile * R;
      int r0 = j0 + bd.dy;  // in [-Cy, 2 Cy)
      r0 = r0 < 0 ? r0 + Cy : (r0 >= Cy ? r0 - Cy : r0);
      const int n1 = min(R, Cy - r0);
      const uint32_t bar = smem_u32(&sm.full[b]);
      const uint32_t dst = smem_u32(&sm.band[b][lane][0]);
      bulk_load(dst, bd.cls + (int64_t)r0 * W, (uint32_t)n1 * row_bytes, bar);
      if (n1 < R)
        bulk_load(dst + (uint32_t)n1 * row_bytes, bd.cls, (uint32_t)(R - n1) * row_bytes, bar);
    }
  };
  // lane 0 of the calling warp arms buffer b for tile `tile` (its ten bands'
  // bytes), or marks it empty (tile < 0: the barrier completes at once)
  auto arm = [&](int tile, int b) {
    if (lane == 0) {
      ++sm.armed[b];
      sm.tile[b] = tile;
      if (tile >= 0)
        mbar_expect(smem_u32(&sm.full[b]), kTileBytes);
      else
        mbar_arrive(smem_u32(&sm.full[b]));
    }
    __syncwarp();
  };
  // the first kBufs tiles are fixed (cta + i ncta), staged by warp 0
  auto first_tile = [&](int i) { return cta + i * ncta < ntiles ? cta + i * ncta : -1; };
  if (early) {
    unsigned busy = 0u;  // bands in the classes the previous phase writes
    for (int k = 0; k < kBands; ++k)
      if (sm.bands[k].cls == g.words + (int64_t)sm.busy0 * g.cstride ||
          sm.bands[k].cls == g.words + (int64_t)sm.busy1 * g.cstride)
        busy |= 1u << k;
    if (warp == 0) {
      for (int i = 0; i < kBufs; ++i) {
        arm(first_tile(i), i);
        if (first_tile(i) >= 0) stage_band(first_tile(i), i, ~busy & ((1u << kBands) - 1u));
      }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    if (warp == 0)
      for (int i = 0; i < kBufs; ++i)
        if (first_tile(i) >= 0) stage_band(first_tile(i), i, busy);
  } else {
    if (pre) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      asm volatile("griddepcontrol.launch_dependents;");
    }
    if (warp == 0)
      for (int i = 0; i < kBufs; ++i) {
        arm(first_tile(i), i);
        if (first_tile(i) >= 0) stage_band(first_tile(i), i, (1u << kBands) - 1u);
      }
  }
  // phase P - 1 is done (griddepcontrol.wait): tag the claim slot of phase P + 1
  if (!kSingle && cta == 0 && threadIdx.x == 0)
    *reinterpret_cast<volatile unsigned long long *>(g.ctl + kCtlTileClaim + ((P + 1u) & 1u)) =
        (unsigned long long)(uint32_t)(P + 1u) << 32;
  if (!mbar_wait(smem_u32(&sm.tables), 0u)) sm.err = 1;

  const int lw = __ffs(W) - 1;  // W is a power of two
  const int jr = (int)threadIdx.x >> lw, w = (int)threadIdx.x & (W - 1);  // word of the tile
  TileView view(sm.cols, W, jr, w);
  int b = 0;
  for (int t = 0;; ++t) {
    // (1) evaluate this thread's word of the tile in buffer b, if any
    if (!mbar_wait(smem_u32(&sm.full[b]), (uint32_t)(t / kBufs) & 1u)) {
      sm.err = 1;
      break;
    }
    const int tile = sm.tile[b];
    if (tile < 0) break;
    view.band = reinterpret_cast<char *>(sm.band[b][0]);
    warp_word(g, TileWord{view, sm.cols, W, tile * R}, sm.trans, sm.thrT, thr32, tile * R + jr, w,
              P, near128, keys);
    // (2) this warp is done with the tile: its shared-memory writes are ordered
    // before the async copies that will refill the buffer, and before the
    // last warp's reads
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    int last = 0;
    if (lane == 0) {
      __threadfence_block();
      last = atomicAdd(&sm.done[b], 1) == kWarps - 1;
      if (last) __threadfence_block();
    }
    last = __shfl_sync(0xFFFFFFFFu, last, 0);
    __syncwarp();
    if (last) {
      // (3) the last warp: write the a and b bands back, then refill the buffer
      if (*(volatile int *)&sm.err == 0) {
        const int j0 = tile * R;
        const uint4 *sa = reinterpret_cast<const uint4 *>(sm.band[b][0]);
        const uint4 *sb = reinterpret_cast<const uint4 *>(sm.band[b][kB]);
        uint4 *ga = reinterpret_cast<uint4 *>(const_cast<uint32_t *>(sm.bands[kA].cls) +
                                              (int64_t)j0 * W);
        int rb = j0 + sm.bands[kB].dy;
        rb = rb >= Cy ? rb - Cy : rb;
        const int split = min(R, Cy - rb) * W / 4;  // uint4 before the band wraps
        uint4 *gb = reinterpret_cast<uint4 *>(const_cast<uint32_t *>(sm.bands[kB].cls));
        const int64_t gb1 = (int64_t)rb * W / 4;  // in uint4
#pragma unroll
        for (int q = lane; q < kTileWords / 4; q += 32) {
          ga[q] = sa[q];
          gb[q < split ? gb1 + q : (int64_t)(q - split)] = sb[q];
        }
      }
      __syncwarp();
      if constexpr (!kSingle) {
        // the buffer's next tile: claimed, or in the fixed order when the
        // claim slot is not this phase's
        int next = 0;
        if (lane == 0) {
          sm.done[b] = 0;
          const unsigned long long old = atomicAdd(
              reinterpret_cast<unsigned long long *>(g.ctl + kCtlTileClaim + (P & 1u)), 1ull);
          next = (uint32_t)(old >> 32) == (uint32_t)P ? kBufs * ncta + (int)(uint32_t)old
                                                      : cta + (t + kBufs) * ncta;
          if (next >= ntiles || *(volatile int *)&sm.err != 0) next = -1;
        }
        next = __shfl_sync(0xFFFFFFFFu, next, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        arm(next, b);
        if (next >= 0) stage_band(next, b, (1u << kBands) - 1u);
      }
    }
    if constexpr (kSingle) break;  // one tile per CTA
    b = b == kBufs - 1 ? 0 : b + 1;
    // leave together: the warp's lanes meet in __syncwarp every tile
    if (__any_sync(0xFFFFFFFFu, *(volatile int *)&sm.err != 0)) break;
  }
  __syncthreads();
  if (threadIdx.x == 0 && sm.err) {
    // give loads still in flight a bounded chance to land before exiting: the
    // last staging of every buffer (phases complete in order)
    mbar_wait(smem_u32(&sm.tables), 0u);
    for (int q = 0; q < kBufs; ++q)
      if (sm.armed[q] > 0) mbar_wait(smem_u32(&sm.full[q]), (uint32_t)(sm.armed[q] - 1) & 1u);
    g.ctl[kCtlStatus] = 1;
  }
}

// kMinBlocks, kSingle: four CTAs per SM with the pipelined tile loop (the
// large-lattice kernel), or five CTAs per SM, one tile per CTA and one band
// buffer (the compact kernel for lattices whose phase fits one wave: more CTAs
// resident for several lattices on their own streams, at 48 registers).
template <int kMinBlocks, bool kSingle>
__global__ void __launch_bounds__(kTileWords, kMinBlocks) phase_tile_kernel(
    Geo g, const uint16_t *thrT, const uint32_t *thr32, int64_t p_off,
    const __grid_constant__ RoundKeys rk) {
  tile_phase<kSingle>(g, thrT, thr32, p_off, (int)blockIdx.x, (int)gridDim.x,
                            TableKeys{&rk});
}

// Lock-step tile-staged phase of several lattices in one launch: CTAs
// [cta_begin, cta_begin + cta_count) of the grid work on job j, each lattice
// with its own tables, phase counter and schedule.
__global__ void __launch_bounds__(256, 4) phase_tile_multi_kernel(const MultiJob *__restrict__ jobs,
                                                                  int njobs, int64_t p_off) {
  int j = 0;
  while (j + 1 < njobs && (int)blockIdx.x >= jobs[j + 1].cta_begin) ++j;
  const MultiJob &J = jobs[j];
  const Geo g = J.g;
  tile_phase<false>(g, J.thrT, J.thr32, p_off, (int)blockIdx.x - J.cta_begin, J.cta_count,
                       SeedKeys{g.k0, g.k1});
}

// Lock-step phase of several lattices in one launch: each CTA works on one
// lattice (its share of the grid is proportional to the lattice's words), with
// that lattice's tables, phase counter and schedule.
template <bool kAligned>
__global__ void __launch_bounds__(256, 4) phase_multi_kernel(const MultiJob *__restrict__ jobs,
                                                             int njobs, int64_t p_off) {
  __shared__ PhaseSmem sm;
  __shared__ int s_job;
  if (threadIdx.x == 0) {
    int j = 0;
    while (j + 1 < njobs && (int)blockIdx.x >= jobs[j + 1].cta_begin) ++j;
    s_job = j;
  }
  __syncthreads();
  const MultiJob &J = jobs[s_job];
  const Geo g = J.g;
  for (int t = threadIdx.x; t < (int)((2u * kThrT + 8u * kMoveN) / 16u); t += blockDim.x)
    reinterpret_cast<uint4 *>(sm.thrT)[t] = reinterpret_cast<const uint4 *>(J.thrT)[t];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  const uint64_t P = (uint64_t)(g.ctl[kCtlPhaseBase] + p_off);
  if (threadIdx.x < 32) {
    const Sched sc = draw_schedule(g, P);
    if (threadIdx.x == 0) sm.u = phase_desc(g, sc, (uint32_t)g.cstride);
  }
  __syncthreads();
  const PhaseD &u = sm.u;
  const uint32_t near128 = u.near128;
  const int nw = g.Cy * g.W;
  const int stride = J.cta_count * blockDim.x;
  for (int base = ((int)blockIdx.x - J.cta_begin) * blockDim.x; base < nw; base += stride) {
    const int wid = base + threadIdx.x;
    const bool act = wid < nw;
    const int j = act ? wid / g.W : 0, w = act ? wid - j * g.W : 0;
    warp_word(g, DirectView<kAligned>{g, u, j, w}, sm.trans, sm.thrT, J.thr32, j, w, P, near128,
              SeedKeys{g.k0, g.k1}, act);
  }
}

// ============================================================================
// Launchers.
int phase_resident_grid(bool aligned) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const cudaError_t e =
      aligned ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, phase_kernel<true>, 256, 0)
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, phase_kernel<false>, 256, 0);
  if (e != cudaSuccess || per_sm < 1 || sms < 1) return 152 * 3;
  return per_sm * sms;
}

int tile_count(const Geo &g) { return g.Cy / (kTileWords / g.W); }

bool tile_path_ok(const Geo &g) {
  return (g.Cx & 15) == 0 && (g.W & 3) == 0 && g.W <= kTileWords && kTileWords % g.W == 0 &&
         g.Cy % (kTileWords / g.W) == 0;
}

// Also raises the tile kernel's dynamic shared memory limit on the current
// device (outside any stream capture: called when a lattice is created).  0
// when that fails: the lattice then takes the direct path.
int tile_resident_grid() {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  constexpr int bytes = (int)sizeof(TileSmem<>);
  if (cudaFuncSetAttribute(phase_tile_kernel<4, false>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      cudaFuncSetAttribute(phase_tile_multi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           bytes) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, phase_tile_kernel<4, false>, 256,
                                                    bytes) != cudaSuccess ||
      per_sm < 1 || sms < 1) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * sms;
}

// The single-tile kernel: five CTAs per SM (48 registers; six at 40 registers
// spilled more and measured slower).
constexpr int kSmallMinB = 5;

int tile_resident_grid_small() {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  constexpr int bytes = (int)sizeof(TileSmem<1>);
  if (cudaFuncSetAttribute(phase_tile_kernel<kSmallMinB, true>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &per_sm, phase_tile_kernel<kSmallMinB, true>, 256, bytes) !=
          cudaSuccess ||
      per_sm < 1 || sms < 1) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * sms;
}

// a-words up to which the direct path takes CTAs of 64 and 128 threads: two and
// four warps on each of the 152 SMs.
constexpr int64_t kDirectSmall64 = 152 * 64, kDirectSmall128 = 152 * 128;

cudaError_t launch_phase(const Geo &g, const DevTables &t, int64_t p_off, const LaunchCfg &cfg,
                         cudaStream_t s) {
  const int64_t nw = (int64_t)g.Cy * g.W;
  if (cfg.tile_grid > 0) {
    const int64_t tiles = nw / kTileWords;
    if (reinterpret_cast<const char *>(t.trans) !=
            reinterpret_cast<const char *>(t.thrT) + 2 * kThrT ||
        (reinterpret_cast<uintptr_t>(t.thrT) & 15u))
      return cudaErrorInvalidValue;  // the tables must be one staged block
    // A phase that fits one wave of the compact kernel (one tile per CTA)
    // takes it: measured faster for several such lattices on their own streams.
    if (cfg.tile_grid_small > 0 && tiles <= cfg.tile_grid_small)
      return launch_pdl_smem(phase_tile_kernel<kSmallMinB, true>, (int)tiles,
                             256, sizeof(TileSmem<1>), s, g,
                             (const uint16_t *)t.thrT, t.thr32, p_off, round_keys(g.k0, g.k1));
    const int grid = (int)(tiles < cfg.tile_grid ? tiles : cfg.tile_grid);
    return launch_pdl_smem(phase_tile_kernel<4, false>, grid, 256, sizeof(TileSmem<>),
                           s, g, (const uint16_t *)t.thrT, t.thr32, p_off,
                           round_keys(g.k0, g.k1));
  }
  const int block = nw <= kDirectSmall64 ? 64 : nw <= kDirectSmall128 ? 128 : 256;
  const int grid = grid_for(nw, block, cfg.phase_grid_cap);
  return launch_pdl((g.Cx & 15) == 0 ? phase_kernel<true> : phase_kernel<false>, grid, block, s, g,
                    (const uint16_t *)t.thrT, t.thr32, p_off, round_keys(g.k0, g.k1));
}

cudaError_t launch_phase_tile_multi(const MultiJob *d_jobs, int njobs, int grid, int64_t p_off,
                                    cudaStream_t s) {
  return launch_pdl_smem(phase_tile_multi_kernel, grid, 256, sizeof(TileSmem<>), s,
                         d_jobs, njobs, p_off);
}

cudaError_t launch_phase_multi(const MultiJob *d_jobs, int njobs, int grid, bool aligned,
                               int64_t p_off, cudaStream_t s) {
  if (aligned) return launch_pdl(phase_multi_kernel<true>, grid, 256, s, d_jobs, njobs, p_off);
  return launch_pdl(phase_multi_kernel<false>, grid, 256, s, d_jobs, njobs, p_off);
}

}  // namespace ccmc
