// ccmc_resident.cu -- the resident kernel: all sweeps of a lattice in one launch,
// the lattice held in the shared memory of one CTA or of a cluster of CTAs.
//
// A CTA (or every CTA of a cluster of C) owns `rows` consecutive rows of each of
// the 16 residue classes; its worker threads evaluate the a-class words of those
// rows in every phase, one, two or four threads a word, and one more warp, the
// auxiliary warp, draws the phase schedules two phases ahead (double Philox
// and divisions off the workers' chain) and writes the observable records.
// The a side of a word is the CTA's own; the b side (the partner rows) may
// belong to another CTA of the cluster and is read and changed through
// distributed shared memory.  One barrier a phase (of the CTA, or the
// cluster's hardware barrier, which cannot deadlock: a cluster's CTAs are
// scheduled together): no two pairs of a phase interact, so a phase's reads and
// writes need no order among themselves.  A worker draws the random words of its
// first word of the next phase before it waits.
//
// What bounds it: a small lattice's phase is one chain of dependent operations a
// thread (windows, counts, two table lookups, atomic write-back, barrier);
// larger ones are bound by integer issue on their CTAs' SMs.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "ccmc_device.cuh"
#include "ccmc_internal.h"
#include "ccmc_word.cuh"

namespace ccmc {

namespace {

constexpr uint32_t kTableBytes = 2u * kThrT + 8u * kMoveN;
static_assert(kTableBytes % 16 == 0, "the lattice words start on 16 bytes");

// One phase's uniforms: classes as byte offsets into a CTA's words, column
// offsets in sites.  Of a site's two column neighbours at most one lies in
// another column block, and of its two row neighbours at most one in another
// row: the neighbour sums do not care which is which, so each side has its own
// class, one column neighbour read at the side's own column (cAm, cBm) and one
// at a column xA, xB sites further (cAx, cBx: -1, 0 or 1; for b as the offset
// offX), one row neighbour in its own row (cAr, cBr) and one yA, yB rows further
// (cAy, cBy).
struct alignas(16) PhaseD {
  uint32_t cA, cAm, cAx, cAr, cAy;
  uint32_t cB, cBm, cBx, cBr, cBy;
  int xA, yA, yB, qx, qy, offX;
  uint32_t near128;
};

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Loads and XORs of lattice words by shared-memory address; kCl: an address in
// the cluster's shared memory (this CTA's or another's).  Volatile: they stay
// between the barriers and the write-backs around them.
template <bool kCl>
__device__ __forceinline__ uint32_t ld_word(uint32_t addr) {
  uint32_t v;
  if constexpr (kCl)
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  else
    asm volatile("ld.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// (nothing to do for 0: predicated, no branch)
template <bool kCl>
__device__ __forceinline__ void xor_word(uint32_t addr, uint32_t v) {
  if constexpr (kCl)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "@p red.relaxed.cluster.shared::cluster.xor.b32 [%0], %1;\n\t}" ::"r"(addr),
        "r"(v)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "@p red.relaxed.cta.shared::cta.xor.b32 [%0], %1;\n\t}" ::"r"(addr),
        "r"(v)
        : "memory");
}

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

template <bool kCl>
__device__ __forceinline__ void bar_arrive() {
  if constexpr (kCl) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
}
template <bool kCl>
__device__ __forceinline__ void bar_wait() {
  if constexpr (kCl) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

__device__ __forceinline__ int wrap_row(int v, int n) {
  return v >= n ? v - n : (v < 0 ? v + n : v);
}

// The phase's uniforms from its schedule, for classes of cls_bytes bytes.
__device__ __forceinline__ PhaseD phase_desc(const Geo &g, const Sched &sc, uint32_t cls_bytes) {
  PhaseD u;
  auto cls = [&](int cx, int cy) { return (uint32_t)((cy & 3) * 4 + (cx & 3)) * cls_bytes; };
  // -1 when the left (upper) neighbours lie in the block (row) before, +1 when the
  // right (lower) ones lie in the next
  auto shift = [](int c) { return c == 0 ? -1 : c == 3 ? 1 : 0; };
  auto side = [&](int cx, int cy, uint32_t &c, uint32_t &m, uint32_t &x, uint32_t &r,
                  uint32_t &y) {
    const int dx = cx == 3 ? 1 : -1, dy = cy == 3 ? 1 : -1;  // the further ones
    c = cls(cx, cy);
    m = cls(cx - dx, cy);
    x = cls(cx + dx, cy);
    r = cls(cx, cy - dy);
    y = cls(cx, cy + dy);
  };
  const int ax = sc.a0x, ay = sc.a0y;
  const int bx = ax + sc.rx, by = ay + sc.ry, cbx = bx & 3, cby = by & 3;
  side(ax, ay, u.cA, u.cAm, u.cAx, u.cAr, u.cAy);
  side(cbx, cby, u.cB, u.cBm, u.cBx, u.cBr, u.cBy);
  u.xA = shift(ax);
  u.yA = shift(ay);
  u.yB = shift(cby);
  int qx = bx >> 2, qy = by >> 2;  // rx < Lx: at most one turn
  if (qx >= g.Cx) qx -= g.Cx;
  if (qy >= g.Cy) qy -= g.Cy;
  u.qx = qx;
  u.qy = qy;
  u.offX = wrap_row(qx + shift(cbx), g.Cx);
  u.near128 = sc.near ? 128u : 0u;
  return u;
}

// The words and shift of the window of 16 sites at column 16 w + off (mod Cx) of
// a row; n1: sites before the row's end (rows of whole words: never cut).
struct Win {
  uint32_t lo, hi;  // byte offsets of its two words
  int sh, n1;
};

template <bool kAl>
__device__ __forceinline__ Win window_at(const Geo &g, int w, int off) {
  Win x;
  if constexpr (kAl) {
    int wl = w + (off >> 4);
    wl = wl >= g.W ? wl - g.W : wl;
    x.lo = 4u * (uint32_t)wl;
    x.hi = wl + 1 == g.W ? 0u : x.lo + 4u;
    x.sh = 2 * (off & 15);
    x.n1 = 16;
  } else {
    int s = 16 * w + off;
    s = s >= g.Cx ? s - g.Cx : s;
    const int wl = s >> 4;
    x.lo = 4u * (uint32_t)wl;
    x.hi = wl + 1 == g.W ? 0u : x.lo + 4u;
    x.sh = 2 * (s & 15);
    x.n1 = g.Cx - s;
  }
  return x;
}

template <bool kCl, bool kAl>
__device__ __forceinline__ uint32_t read_window(uint32_t row, const Win &x) {
  uint32_t v = __funnelshift_r(ld_word<kCl>(row + x.lo), ld_word<kCl>(row + x.hi), x.sh);
  if constexpr (!kAl) {
    if (x.n1 < 16)  // the row ends inside the window: go on at its start
      v = (v & ((1u << (2 * x.n1)) - 1u)) | (ld_word<kCl>(row) << (2 * x.n1));
  }
  return v;
}

// XOR the first n sites of D into the window's words.
template <bool kCl, bool kAl>
__device__ __forceinline__ void xor_window(uint32_t row, const Win &x, uint32_t D) {
  uint32_t d1 = D;
  if constexpr (!kAl) {
    if (x.n1 < 16) {
      d1 = D & ((1u << (2 * x.n1)) - 1u);
      xor_word<kCl>(row, D >> (2 * x.n1));
    }
  }
  xor_word<kCl>(row + x.lo, d1 << x.sh);
  xor_word<kCl>(row + x.hi, __funnelshift_l(d1, 0u, x.sh));  // d1 >> (32 - sh), 0 for sh = 0
}

// Where a CTA's rows lie.
struct Place {
  uint32_t base;  // shared-memory address of this CTA's words
  uint32_t row_bytes;
  uint32_t mrows;  // ceil(2^32 / rows)
  int rows, row0;  // rows a CTA of the cluster, this CTA's first
};

// Address (class offset not added) of class row j: this CTA's or, in a cluster,
// its owner's.
template <bool kCl>
__device__ __forceinline__ uint32_t row_addr(const Place &pl, int j) {
  if constexpr (kCl) {
    const uint32_t rank = pl.rows == 1 ? (uint32_t)j : __umulhi((uint32_t)j, pl.mrows);
    return map_rank(pl.base, rank) + (uint32_t)(j - (int)rank * pl.rows) * pl.row_bytes;
  } else {
    return pl.base + (uint32_t)j * pl.row_bytes;
  }
}

// What a thread keeps of a word's place: its row in the CTA, column, byte offset
// in a class, and where the words left and right of it lie from it.
struct Spot {
  int l, w;
  uint32_t off;
  int left, right;
};

__device__ __forceinline__ Spot spot_of(const Geo &g, const Place &pl, int l, int w) {
  return Spot{l, w, (uint32_t)l * pl.row_bytes + 4u * (uint32_t)w,
              w == 0 ? 4 * (g.W - 1) : -4, w == g.W - 1 ? -4 * (g.W - 1) : 4};
}

// Window of the word at `addr` one site further left (x = -1), right (x = 1)
// or the word itself (x = 0).
template <bool kAl>
__device__ __forceinline__ uint32_t side_window(const Geo &g, const Spot &p, uint32_t addr,
                                                int x) {
  uint32_t lo = ld_word<false>(addr + (uint32_t)(x < 0 ? p.left : 0));
  uint32_t hi = ld_word<false>(addr + (uint32_t)(x > 0 ? p.right : 0));
  if constexpr (!kAl) {  // the row's last word holds tail < 16 sites, zeros above them
    const int tail = g.Cx - 16 * (g.W - 1);
    if (p.w == 0 && x < 0) lo <<= 32 - 2 * tail;
    if (p.w == g.W - 1 && x > 0 && tail < 16) lo |= hi << (2 * tail);
  }
  return __funnelshift_r(lo, hi, 2 * x);  // the shift counts modulo 32
}

template <bool kCl, bool kAl>
__device__ __forceinline__ WordIn gather_word(const Geo &g, const PhaseD &u, const Place &pl,
                                              const Spot &p) {
  WordIn in;
  const int j = pl.row0 + p.l;
  int jb = j + u.qy;
  jb = jb >= g.Cy ? jb - g.Cy : jb;
  const uint32_t rb = row_addr<kCl>(pl, jb);
  const uint32_t ry = u.yB ? row_addr<kCl>(pl, wrap_row(jb + u.yB, g.Cy)) : rb;
  const Win wb = window_at<kAl>(g, p.w, u.qx);
  in.B = read_window<kCl, kAl>(rb + u.cB, wb);
  const uint32_t bm = read_window<kCl, kAl>(rb + u.cBm, wb);
  const uint32_t br = read_window<kCl, kAl>(rb + u.cBr, wb);
  const uint32_t bx = read_window<kCl, kAl>(rb + u.cBx, window_at<kAl>(g, p.w, u.offX));
  const uint32_t by = read_window<kCl, kAl>(ry + u.cBy, wb);
  const uint32_t own = pl.base + p.off;
  in.A = ld_word<false>(own + u.cA);
  const uint32_t am = ld_word<false>(own + u.cAm);
  const uint32_t ar = ld_word<false>(own + u.cAr);
  const uint32_t ax = side_window<kAl>(g, p, own + u.cAx, u.xA);
  uint32_t ay;
  if constexpr (kCl) {
    ay = u.yA ? ld_word<true>(row_addr<true>(pl, wrap_row(j + u.yA, g.Cy)) + u.cAy +
                              4u * (uint32_t)p.w)
              : ld_word<false>(own + u.cAy);
  } else {
    const int jy = wrap_row(j + u.yA, g.Cy);
    ay = ld_word<false>(own + u.cAy + (uint32_t)(jy - j) * pl.row_bytes);
  }
  in.na = neighbour_planes(am, ar, ax, ay);
  in.nb = neighbour_planes(bm, br, bx, by);
  return in;
}

// Apply the moves (dA, dB) of a word; n: its sites.
template <bool kCl, bool kAl>
__device__ __forceinline__ void apply_word(const Geo &g, const PhaseD &u, const Place &pl,
                                           const Spot &p, int n, uint32_t dA, uint32_t dB) {
  if constexpr (!kAl) {
    if (n < 16) {  // pairs past the end of the row do not exist
      const uint32_t valid = (1u << (2 * n)) - 1u;
      dA &= valid;
      dB &= valid;
    }
  }
  xor_word<false>(pl.base + p.off + u.cA, dA);
  int jb = pl.row0 + p.l + u.qy;
  jb = jb >= g.Cy ? jb - g.Cy : jb;
  xor_window<kCl, kAl>(row_addr<kCl>(pl, jb) + u.cB, window_at<kAl>(g, p.w, u.qx), dB);
}

// The rare pairs of a warp's words, warp-cooperatively: for every lane with
// flagged calls, 16 / kTPW lanes each decide one of its pairs from its inputs
// (see the phase kernels' warp_word).
template <bool kCl, bool kAl, int kTPW>
__device__ __forceinline__ void rare_pairs(const Geo &g, const PhaseD &u, const Place &pl,
                                        const uint2 *trans, const uint16_t *thrT,
                                        const uint32_t *thr32, unsigned ball, uint32_t rz,
                                        const WordIn &in, const Spot &p, int n, int sub,
                                        uint64_t P) {
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
    const int ol = __shfl_sync(0xFFFFFFFFu, p.l, src), ow = __shfl_sync(0xFFFFFFFFu, p.w, src),
              on = __shfl_sync(0xFFFFFFFFu, n, src), osub = __shfl_sync(0xFFFFFFFFu, sub, src);
    const int c = kTPW == 1 ? (lane >> 3) & 1 : kTPW == 2 ? osub : osub >> 1;
    const int h = kTPW == 4 ? osub & 1 : (lane >> 2) & 1;
    const int t = 2 * c + h + 4 * (lane & 3);
    if (lane < 16 / kTPW && ((orz >> c) & 1u) && t < on) {
      const uint32_t x = exact_move(g, trans, thrT, thr32, pl.row0 + ol, ow, c, h, lane & 3, o, P,
                                    u.near128);
      if (x)
        apply_word<kCl, kAl>(g, u, pl, spot_of(g, pl, ol, ow), on, (x >> 2) << (2 * t),
                             (x & 3u) << (2 * t));
    }
  }
}

// Observables of this CTA's words by definition, as sums over bit products of
// the linear code (S = b1 - b0, sigma = 1 - b1 - b0): a site's bits against its
// right and down neighbours', like bits (n[0]) and unlike ones (n[1]); the
// sites' b1, b0 and both (n[2..4]); b1 and b0 with the staggered sign (n[5], n[6]).
template <bool kCl, bool kAl>
__device__ __forceinline__ void count_words(const Geo &g, const Place &pl, int nr,
                                            uint32_t cls_bytes, int tid, int nthreads, int n[7]) {
  const int nw = nr * g.W;
  if (nw == 0) return;
  const uint32_t mw = 0xFFFFFFFFu / (uint32_t)g.W + 1u, mn = 0xFFFFFFFFu / (uint32_t)nw + 1u;
  for (int i = tid; i < 16 * nw; i += nthreads) {
    const int cls = nw == 1 ? i : (int)__umulhi((uint32_t)i, mn);
    const int wid = i - cls * nw;
    const int l = g.W == 1 ? wid : (int)__umulhi((uint32_t)wid, mw), w = wid - l * g.W;
    const int cx = cls & 3, cy = cls >> 2;
    const uint32_t row = pl.base + (uint32_t)l * pl.row_bytes;
    uint32_t X = ld_word<false>(row + (uint32_t)cls * cls_bytes + 4u * (uint32_t)w);
    if constexpr (!kAl) {
      const int ns = min(16, g.Cx - 16 * w);
      if (ns < 16) X &= (1u << (2 * ns)) - 1u;
    }
    const uint32_t Yr = read_window<false, kAl>(
        row + (uint32_t)(cy * 4 + ((cx + 1) & 3)) * cls_bytes,
        window_at<kAl>(g, w, cx == 3 && g.Cx > 1 ? 1 : 0));
    const uint32_t dcls = (uint32_t)(((cy + 1) & 3) * 4 + cx) * cls_bytes + 4u * (uint32_t)w;
    const uint32_t Yd =
        cy == 3 ? ld_word<kCl>(row_addr<kCl>(pl, wrap_row(pl.row0 + l + 1, g.Cy)) + dcls)
                : ld_word<false>(row + dcls);
    const uint32_t odd = X & 0xAAAAAAAAu, even = X & 0x55555555u;
    const uint32_t Xs = (odd >> 1) | (even << 1);
    n[0] += __popc(X & Yr) + __popc(X & Yd);
    n[1] += __popc(Xs & Yr) + __popc(Xs & Yd);
    const int k1 = __popc(odd), k0 = __popc(even);
    n[2] += k1;
    n[3] += k0;
    n[4] += __popc(odd & Xs);
    const bool minus = (cx + cy) & 1;
    n[5] += minus ? -k1 : k1;
    n[6] += minus ? -k0 : k0;
  }
}

}  // namespace

template <bool kCl, bool kAl, int kTPW>
__global__ void __launch_bounds__(kResMaxThreads, 1)
    resident_sweep_kernel(const __grid_constant__ ResJob one, const ResJob *__restrict__ jobs,
                    int cluster) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  __shared__ PhaseD s_d[4];   // phase P's uniforms in slot P mod 4
  __shared__ int s_obs[2][8]; // the counts of even and odd records
  uint16_t *thrT = reinterpret_cast<uint16_t *>(res_smem);
  uint2 *trans = reinterpret_cast<uint2 *>(res_smem + 2 * kThrT);
  __shared__ ResJob s_job;  // read where used: its fields would fill the registers
  const int tid = threadIdx.x, lane = tid & 31;
  const int nworkers = (int)blockDim.x - 32;
  const bool aux = tid >= nworkers;
  {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(
        jobs ? jobs + (kCl ? blockIdx.x / cluster : blockIdx.x) : &one);
    for (int t = tid; t < (int)(sizeof(ResJob) / 4); t += blockDim.x)
      reinterpret_cast<uint32_t *>(&s_job)[t] = src[t];
    __syncthreads();
  }
  const ResJob &J = s_job;
  const Geo &g = s_job.g;
  Place pl;
  uint32_t rank = 0;
  if constexpr (kCl) asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  pl.base = smem_addr(res_smem) + kTableBytes;
  pl.row_bytes = 4u * (uint32_t)g.W;
  pl.rows = J.rows;
  pl.mrows = J.rows > 1 ? 0xFFFFFFFFu / (uint32_t)J.rows + 1u : 0u;
  pl.row0 = (int)rank * J.rows;
  const int nr = max(0, min(J.rows, g.Cy - pl.row0));  // rows of this CTA
  const uint32_t cls_bytes = (uint32_t)J.rows * pl.row_bytes;
  const uint32_t mw = g.W > 1 ? 0xFFFFFFFFu / (uint32_t)g.W + 1u : 0u;
  // tables and words in
  {
    const uint4 *src = reinterpret_cast<const uint4 *>(J.thrT);  // levels, then moves
    uint4 *dst = reinterpret_cast<uint4 *>(res_smem);
    for (int t = tid; t < (int)(kTableBytes / 16); t += blockDim.x) dst[t] = src[t];
    uint32_t *words = reinterpret_cast<uint32_t *>(res_smem + kTableBytes);
    const int nw = nr * g.W;
#pragma unroll 4
    for (int cls = 0; cls < 16; ++cls)
      for (int t = tid; t < nw; t += blockDim.x)
        words[cls * J.rows * g.W + t] =
            g.words[(int64_t)cls * g.cstride + (int64_t)pl.row0 * g.W + t];
    if (tid < 16) s_obs[tid >> 3][tid & 7] = 0;
  }
  const int64_t P0 = g.ctl[kCtlPhaseBase];
  const int obs_every = J.obs_every;
  auto describe = [&](uint64_t P) {  // the auxiliary warp
    const Sched sc = draw_schedule(g, P);
    if (lane == 0) s_d[P & 3u] = phase_desc(g, sc, cls_bytes);
  };
  // sweeps until the next record, and the record writer's ring position
  int until = obs_every > 0 ? obs_every - (int)((P0 / 8) % obs_every) : 0;
  int64_t obs_cnt = 0, obs_slot = 0;
  if (aux) {
    describe((uint64_t)P0);
    describe((uint64_t)P0 + 1u);
    if (obs_every > 0 && rank == 0 && lane == 0) {
      obs_cnt = g.ctl[kCtlObsCount];
      obs_slot = obs_cnt % J.ring_cap;
    }
  }
  // this thread's place in every phase's first pass, and that pass's random words
  const int items = kTPW * nr * g.W;
  constexpr int kCalls = kTPW == 1 ? 2 : 1;
  auto place = [&](int i) {
    const int wid = i / kTPW;
    const int l = g.W > 1 ? (int)__umulhi((uint32_t)wid, mw) : wid;
    return spot_of(g, pl, l, wid - l * g.W);
  };
  auto call_of = [&](const Spot &p, int c, uint64_t P) {
    const uint32_t gbase = (uint32_t)(pl.row0 + p.l) * (uint32_t)(2 * g.W) + (uint32_t)(2 * p.w);
    return philox(gbase + (uint32_t)c, (uint32_t)P, (uint32_t)(P >> 32), TAG_MOVE, g.k0, g.k1);
  };
  const Spot p0 = place(aux ? 0 : tid);
  const int sub = tid % kTPW;
  U4 rn[kCalls];
  auto draw_first = [&](uint64_t P) {
#pragma unroll
    for (int ci = 0; ci < kCalls; ++ci)
      rn[ci] = call_of(p0, kTPW == 1 ? ci : kTPW == 2 ? sub : sub >> 1, P);
  };
  draw_first((uint64_t)P0);
  bar_arrive<kCl>();
  bar_wait<kCl>();
  int obs_buf = 0;
  const int nphases = 8 * J.nsweeps;
  for (int q = 0; q < nphases; ++q) {
    const uint64_t P = (uint64_t)(P0 + q);
    if (!aux) {
      const PhaseD &u = s_d[P & 3u];
      for (int base = tid - lane; base < items; base += nworkers) {  // uniform over the warp
        const bool act = base + lane < items;
        const bool first = base < nworkers;
        Spot p = p0;
        if (!first) p = place(base + lane);
        const int n = !act ? 0 : kAl ? 16 : min(16, g.Cx - (p.w << 4));
        WordIn in{};
        uint32_t rz = 0u;
        if (act) {
          in = gather_word<kCl, kAl>(g, u, pl, p);
          const uint3 d = fast_moves<kTPW>(trans, thrT, sub, in, u.near128, [&](int c) {
            return first ? rn[kTPW == 1 ? c : 0] : call_of(p, c, P);
          });
          apply_word<kCl, kAl>(g, u, pl, p, n, d.x, d.y);
          rz = d.z;
        }
        const unsigned ball = __ballot_sync(0xFFFFFFFFu, rz != 0u);
        if (ball)
          rare_pairs<kCl, kAl, kTPW>(g, u, pl, trans, thrT, J.thr32, ball, rz, in, p, n, sub, P);
      }
    }
    bar_arrive<kCl>();
    if (aux)
      describe(P + 2u);
    else
      draw_first(P + 1u);
    bar_wait<kCl>();
    if (obs_every > 0 && (q & 7) == 7 && --until == 0) {
      until = obs_every;
      int n[7] = {0, 0, 0, 0, 0, 0, 0};
      if (!aux) count_words<kCl, kAl>(g, pl, nr, cls_bytes, tid, nworkers, n);
      if (!aux) {
        uint32_t dst = smem_addr(s_obs[obs_buf]);
        if constexpr (kCl) dst = map_rank(dst, 0u);
#pragma unroll
        for (int k = 0; k < 7; ++k) {
          const int v = __reduce_add_sync(0xFFFFFFFFu, n[k]);
          if (lane == 0) {
            if constexpr (kCl)
              asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(
                               dst + 4u * k),
                           "r"(v)
                           : "memory");
            else
              atomicAdd(&s_obs[obs_buf][k], v);
          }
        }
      }
      // the counts are complete, and no word changes before all are counted
      bar_arrive<kCl>();
      bar_wait<kCl>();
      if (aux && rank == 0 && lane == 0) {
        volatile int *c = s_obs[obs_buf];
        const int64_t like = c[0], unlike = c[1], b1 = c[2], b0 = c[3], both = c[4], s1 = c[5],
                      s0 = c[6];
        for (int k = 0; k < 7; ++k) c[k] = 0;  // for the record after the next
        const int64_t N = (int64_t)g.Lx * g.Ly;
        const int64_t rec[8] = {(int64_t)(P + 1u) / 8, b1 + b0 - 2 * both, like - unlike,
                                2 * N - 4 * (b1 + b0) + like + unlike, N - b1 - b0,
                                -s1 - s0, b1 - b0, s1 - s0};
        int64_t *dst = J.ring + obs_slot * 8;
        for (int k = 0; k < 8; ++k) {
          g.ctl[kCtlLatest + k] = rec[k];
          dst[k] = rec[k];
        }
        g.ctl[kCtlObsCount] = ++obs_cnt;
        if (++obs_slot == J.ring_cap) obs_slot = 0;
        if (J.hist) {  // reductions: no load to wait for
          const int64_t vals[3] = {rec[4], rec[5], rec[7]};
          for (int h = 0; h < 3; ++h)
            atomicAdd(reinterpret_cast<unsigned long long *>(
                          J.hist + h * J.nbins + (vals[h] + N) * J.nbins / (2 * N + 1)),
                      1ull);
        }
      }
      obs_buf ^= 1;
    }
  }
  // words out; in a cluster nobody leaves while others may still read (the last
  // barrier was passed by all, and nothing is read after it)
  {
    const uint32_t *words = reinterpret_cast<const uint32_t *>(res_smem + kTableBytes);
    const int nw = nr * g.W;
    for (int cls = 0; cls < 16; ++cls)
      for (int t = tid; t < nw; t += blockDim.x)
        g.words[(int64_t)cls * g.cstride + (int64_t)pl.row0 * g.W + t] =
            words[cls * J.rows * g.W + t];
    if (rank == 0 && tid == 0) g.ctl[kCtlPhaseBase] = P0 + nphases;
  }
}

namespace {

using Kernel = void (*)(const ResJob, const ResJob *, int);

Kernel kernel_of(bool cluster, bool aligned, int tpw) {
  static const Kernel k[2][2][3] = {
      {{resident_sweep_kernel<false, false, 1>, resident_sweep_kernel<false, false, 2>,
        resident_sweep_kernel<false, false, 4>},
       {resident_sweep_kernel<false, true, 1>, resident_sweep_kernel<false, true, 2>,
        resident_sweep_kernel<false, true, 4>}},
      {{resident_sweep_kernel<true, false, 1>, resident_sweep_kernel<true, false, 2>,
        resident_sweep_kernel<true, false, 4>},
       {resident_sweep_kernel<true, true, 1>, resident_sweep_kernel<true, true, 2>,
        resident_sweep_kernel<true, true, 4>}}};
  return k[cluster][aligned][tpw == 4 ? 2 : tpw == 2 ? 1 : 0];
}

constexpr int kMaxDevices = 64;
std::mutex g_mu;
bool g_ready[kMaxDevices] = {};

// Raises every instance's shared-memory limit and allows clusters of 16, once
// per device (outside any capture: called when a lattice or a batch is created).
bool prepare_device(int dev) {
  if (dev < 0 || dev >= kMaxDevices) return false;
  std::lock_guard<std::mutex> lock(g_mu);
  if (g_ready[dev]) return true;
  for (int c = 0; c < 2; ++c)
    for (int a = 0; a < 2; ++a)
      for (int t : {1, 2, 4}) {
        const void *f = reinterpret_cast<const void *>(kernel_of(c, a, t));
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kResMaxSmem) !=
                cudaSuccess ||
            (c && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                      cudaSuccess)) {
          cudaGetLastError();
          return false;
        }
      }
  g_ready[dev] = true;
  return true;
}

}  // namespace

bool resident_ready() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && prepare_device(dev);
}

int64_t resident_smem(const Geo &g, int rows) {
  return (int64_t)kTableBytes + 64ll * rows * g.W;
}

// Shapes, measured on GB300 (us a sweep, records off).  A cluster's barrier and
// remote windows cost 0.7 us a phase, which only pays for lattices of enough
// words: 256^2 (256 words a phase) 15.0 on one CTA, 12.4 on four, 11.5 on sixteen;
// 1024^2 51.8 on four, 33.1 on eight, 26.1 on sixteen; 128 lattices of 128^2 12.6
// on one CTA each, 16.6 on two.  Four threads a word shorten the chain while few
// words share an SM (64^2: 5.7, 6.3 with two, 10.1 with one), two up to 256; with
// more, the work repeated for threads that share a word costs more than it hides
// (512 replicas: 22.9 with one, 25.8 with two, 30.8 with four).
ResShape resident_shape(const Geo &g, double ctas, double load, int max_threads, int max_tpw) {
  ResShape sh;
  int C = 1;
  if (g.cstride >= kResClusterWords)
    while (C < kResMaxCluster && 2 * C <= ctas && g.cstride >= 2 * C * kResMinWords) C *= 2;
  while (C < kResMaxCluster && resident_smem(g, (g.Cy + C - 1) / C) > kResMaxSmem) C *= 2;
  sh.rows = (g.Cy + C - 1) / C;
  sh.cluster = C;
  const int words = sh.rows * g.W;
  const double busy = words > load ? words : load;
  sh.tpw = max_tpw >= 4 && busy <= 24 ? 4 : max_tpw >= 2 && busy <= 256 ? 2 : 1;
  while (sh.tpw > 1 && sh.tpw * words > max_threads) sh.tpw /= 2;
  int workers = 32;
  while (workers < sh.tpw * words && workers < max_threads) workers *= 2;
  sh.threads = workers + 32;
  sh.smem = resident_smem(g, sh.rows);
  return sh;
}

cudaError_t launch_resident_sweep(const ResJob *one, const ResJob *d_jobs, int njobs,
                            const ResShape &shape, bool aligned, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(njobs * shape.cluster));
  cfg.blockDim = dim3((unsigned)shape.threads);
  cfg.dynamicSmemBytes = (size_t)shape.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)shape.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = shape.cluster > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel_of(shape.cluster > 1, aligned, shape.tpw),
                            one ? *one : ResJob{}, one ? nullptr : d_jobs, shape.cluster);
}

}  // namespace ccmc
