// ccmc_phase.cu -- the colour-phase kernels of the coupled-pair Metropolis
// sweep for sm_103a (one phase of one lattice a launch; of several
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

// The direct path's view of a word: row j, word w of the classes in global memory,
// rows of whole words (kAl) or of any width.  Addresses are 32-bit byte offsets from
// the lattice's base: its words take at most 2^32 bytes (validate_shape), which a
// lattice of 4 x 2^28 sites does, with one site a word.
template <bool kAl>
struct DirectView {
  const Geo &g;
  const PhaseD &u;  // class offsets in bytes
  int j, w;

  __device__ __forceinline__ uint32_t *at(uint32_t off) const {
    return reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(g.words) + off);
  }
  __device__ __forceinline__ uint32_t row(int jj) const {
    return (uint32_t)jj * (4u * (uint32_t)g.W);
  }
  // sites of the window from one class row
  __device__ __forceinline__ uint32_t window(uint32_t r, const Win &x) const {
    uint32_t v = __funnelshift_r(*at(r + 4u * (uint32_t)x.lo), *at(r + 4u * (uint32_t)x.hi), x.sh);
    if constexpr (!kAl) {
      if (x.n1 < 16)  // the row ends inside the window: go on at its start
        v = (v & ((1u << (2 * x.n1)) - 1u)) | (*at(r) << (2 * x.n1));
    }
    return v;
  }
  __device__ __forceinline__ WordIn gather() const {
    WordIn in;
    const SideD &a = u.side[0], &b = u.side[1];
    const int jb = turn(j + b.qy, g.Cy);
    const uint32_t rb = row(jb), ry = row(turn(jb + b.ys, g.Cy));
    const Win win = window_at<kAl>(g, w, b.qx);
    in.B = window(rb + b.c, win);
    in.nb = neighbour_planes(window(rb + b.m, win), window(rb + b.r, win), window(ry + b.y, win),
                             window(rb + b.x, window_at<kAl>(g, w, b.offX)));
    const uint32_t ra = row(j), own = ra + 4u * (uint32_t)w;
    in.A = *at(a.c + own);
    in.na = neighbour_planes(*at(a.m + own), *at(a.r + own),
                             *at(a.y + row(turn(j + a.ys, g.Cy)) + 4u * (uint32_t)w),
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
      uint32_t *pa = at(a.c + row(jj) + 4u * (uint32_t)ww);
      if constexpr (kOwn)
        *pa ^= dA;
      else
        atomicXor(pa, dA);
    }
    if (dB) {
      const uint32_t r = b.c + row(turn(jj + b.qy, g.Cy));
      const Win x = window_at<kAl>(g, ww, b.qx);
      uint32_t d1 = dB;
      if constexpr (!kAl) {
        if (x.n1 < 16) {
          d1 = dB & ((1u << (2 * x.n1)) - 1u);
          const uint32_t d2 = dB >> (2 * x.n1);
          if (d2) atomicXor(at(r), d2);
        }
      }
      const uint32_t lo = d1 << x.sh, hi = __funnelshift_l(d1, 0u, x.sh);
      if (lo) atomicXor(at(r + 4u * (uint32_t)x.lo), lo);
      if (hi) atomicXor(at(r + 4u * (uint32_t)x.hi), hi);
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

// A CTA's levels and move table, one block in device memory as here (they come from
// host uploads that precede the whole launch chain).
__device__ __forceinline__ void load_tables(PhaseSmem &sm, const uint16_t *thrT) {
  static_assert((2u * kThrT + 8u * kMoveN) % 16u == 0 &&
                    offsetof(PhaseSmem, trans) == 2u * kThrT,
                "copied 16 bytes at a time as one block");
  for (int t = threadIdx.x; t < (int)((2u * kThrT + 8u * kMoveN) / 16u); t += blockDim.x)
    reinterpret_cast<uint4 *>(sm.thrT)[t] = reinterpret_cast<const uint4 *>(thrT)[t];
}

// The phase index and its uniforms, by the first warp.  A launch after the first of
// a chain (p_off > 0) does this before it waits for its predecessor: the counter was
// written by a kernel at least two launches back (the chain's counter advance), which
// the predecessor's griddepcontrol.wait has already waited for.
__device__ __forceinline__ void draw_uniforms(PhaseSmem &sm, const Geo &g, int64_t p_off) {
  if (threadIdx.x < 32) {
    const uint64_t P = (uint64_t)(g.ctl[kCtlPhaseBase] + p_off);
    const Sched s = draw_schedule(g, P);
    if (threadIdx.x == 0) {
      sm.u = phase_desc(g, s, 4u * (uint32_t)g.cstride);
      sm.P = P;
    }
  }
}

// Word wid (of nw; beyond them the lane only joins its warp) of the phase.
// mw: ceil(2^32 / W) where its product's high half is wid / W, else 0.
template <bool kAligned, class Keys>
__device__ __forceinline__ void phase_word(const Geo &g, const PhaseSmem &sm,
                                           const uint32_t *thr32, uint32_t mw, int wid, int nw,
                                           const Keys &keys) {
  const bool act = wid < nw;
  const int j = !act ? 0 : mw ? (int)__umulhi((uint32_t)wid, mw) : wid / g.W;
  const int w = act ? wid - j * g.W : 0;
  warp_word(g, DirectView<kAligned>{g, sm.u, j, w}, sm.trans, sm.thrT, thr32, j, w, sm.P,
            sm.u.near128, keys, act);
}

// One phase of one lattice.  Its windows come straight from L2: the loads of a word
// are in flight together, and 32 warps an SM hide them behind the integer work that
// bounds the phase.  (Staging tiles of class rows into shared memory by bulk copies,
// with the last warp of a tile writing it back, held that rate too, but a phase then
// began and ended with a tile's latency on every SM: 16384^2 28.5 us against 26.6
// here, 4096^2 5.1 against 4.1, 2048^2 4.1 against 3.0.)  Four CTAs of 64 registers an
// SM: with 48 registers and five 16384^2 takes 28.0 us, with 56 and nine of 128 threads
// 28.1, with 384-thread CTAs 27.0.  The prologue (tables, and
// for a launch after the first of a chain the phase index and its schedule) runs
// before the kernel waits for its predecessor.  Small lattices take small CTAs: a
// thread's chain is what they wait for, and it is shorter on an SM of its own
// (1100^2: 4.4 us a phase before, 3.0 now).
template <bool kAligned>
__global__ void __launch_bounds__(256, 4) phase_kernel(Geo g, const uint16_t *thrT,
                                                       const uint32_t *thr32, int64_t p_off,
                                                       uint32_t mw,
                                                       const __grid_constant__ RoundKeys rk) {
  __shared__ PhaseSmem sm;
  load_tables(sm, thrT);
  if (p_off > 0) draw_uniforms(sm, g, p_off);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // The next kernel may launch now: with one resident wave its blocks only take
  // the slots of blocks that finish, and it waits for this whole grid before
  // touching the lattice.
  asm volatile("griddepcontrol.launch_dependents;");
  if (p_off == 0) draw_uniforms(sm, g, p_off);
  __syncthreads();
  const int nw = g.Cy * g.W, stride = gridDim.x * blockDim.x;
  for (int base = blockIdx.x * blockDim.x; base < nw; base += stride)
    phase_word<kAligned>(g, sm, thr32, mw, base + (int)threadIdx.x, nw, TableKeys{&rk});
}

// Lock-step phase of several lattices in one launch: each CTA works on one
// lattice (its share of the grid is proportional to the lattice's words), with
// that lattice's tables, phase counter and schedule; the prologue as phase_kernel's.
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
  load_tables(sm, J.thrT);
  if (p_off > 0) draw_uniforms(sm, g, p_off);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  if (p_off == 0) draw_uniforms(sm, g, p_off);
  __syncthreads();
  const int nw = g.Cy * g.W, stride = J.cta_count * blockDim.x;
  for (int base = ((int)blockIdx.x - J.cta_begin) * blockDim.x; base < nw; base += stride)
    phase_word<kAligned>(g, sm, J.thr32, J.mw, base + (int)threadIdx.x, nw,
                         SeedKeys{g.k0, g.k1});
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
  if (e != cudaSuccess || per_sm < 1 || sms < 1) return 152 * 4;
  return per_sm * sms;
}

// ceil(2^32 / W) when its product's high half is wid / W for every word of a phase
// (the excess stays below one: wid times at most W - 1 is below 2^32), else 0.
uint32_t row_magic(const Geo &g) {
  if (g.W < 2 || (uint64_t)g.cstride * (uint64_t)g.W >= (1ull << 32)) return 0u;
  return 0xFFFFFFFFu / (uint32_t)g.W + 1u;
}

// a-words up to which the direct path takes CTAs of 64 and 128 threads: two and
// four warps on each of the 152 SMs.
constexpr int64_t kDirectSmall64 = 152 * 64, kDirectSmall128 = 152 * 128;

cudaError_t launch_phase(const Geo &g, const DevTables &t, int64_t p_off, const LaunchCfg &cfg,
                         cudaStream_t s) {
  const int64_t nw = (int64_t)g.Cy * g.W;
  const int block = nw <= kDirectSmall64 ? 64 : nw <= kDirectSmall128 ? 128 : 256;
  const int grid = grid_for(nw, block, cfg.phase_grid_cap);
  return launch_pdl((g.Cx & 15) == 0 ? phase_kernel<true> : phase_kernel<false>, grid, block, s, g,
                    (const uint16_t *)t.thrT, t.thr32, p_off, row_magic(g),
                    round_keys(g.k0, g.k1));
}

cudaError_t launch_phase_multi(const MultiJob *d_jobs, int njobs, int grid, bool aligned,
                               int64_t p_off, cudaStream_t s) {
  if (aligned) return launch_pdl(phase_multi_kernel<true>, grid, 256, s, d_jobs, njobs, p_off);
  return launch_pdl(phase_multi_kernel<false>, grid, 256, s, d_jobs, njobs, p_off);
}

}  // namespace ccmc
