// ccmc_resident.cu -- the resident kernel: all sweeps of a lattice in one launch,
// the lattice held in the shared memory of one CTA or of a cluster of CTAs.
//
// A CTA (or every CTA of a cluster of C) owns `rows` consecutive rows of each of
// the 16 residue classes; its worker threads evaluate the a-class words of those
// rows in every phase, one, two or four threads a word, and one more warp, the
// auxiliary warp, draws the next sweep's eight phase schedules side by side (Philox
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

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "ccmc_device.cuh"
#include "ccmc_internal.h"
#include "ccmc_word.cuh"

namespace ccmc {

namespace {

// Levels, moves and full thresholds (the rare pairs' path must not wait for
// global memory while the CTA waits at the barrier).
constexpr uint32_t kFastBytes = 2u * kThrT + 8u * kMoveN;
constexpr uint32_t kTableBytes = kFastBytes + 4u * kDevPad;
static_assert(kFastBytes % 16 == 0 && kTableBytes % 16 == 0, "copied 16 bytes at a time");

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

// v, or the word at addr if p: a predicated load, no branch.
__device__ __forceinline__ uint32_t ld_remote_if(bool p, uint32_t addr, uint32_t v) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t"
      "@q ld.shared::cluster.u32 %0, [%1];\n\t}"
      : "+r"(v)
      : "r"(addr), "r"((uint32_t)p));
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

// The uniforms of phases P .. P + 7 by one warp: four lanes a phase, each trying
// attempts lane mod 4, + 4, ... (draw_schedule's: the first allowed one of at most
// 64 wins, then the fixed offset); one round settles a phase with probability 0.99.
__device__ __forceinline__ void describe_sweep(const Geo &g, uint64_t P, uint32_t cls_bytes,
                                               PhaseD *s_d) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t p = P + (lane >> 2), N = (uint64_t)g.Lx * (uint64_t)g.Ly;
  bool done = false;
#pragma unroll 1
  for (uint32_t round = 0; round < 16u; ++round) {
    const U4 w = philox(4u * round + (lane & 3u), (uint32_t)p, (uint32_t)(p >> 32), TAG_SCHED,
                        g.k0, g.k1);
    const uint64_t x = ((uint64_t)w.z << 32) | (uint64_t)w.y;
    const uint32_t idx = (uint32_t)__umul64hi(x, N);
    Sched s;
    s.a0x = (int)(w.x & 3u);
    s.a0y = (int)((w.x >> 2) & 3u);
    s.ry = (int)(idx / (uint32_t)g.Lx);
    s.rx = (int)(idx - (uint32_t)s.ry * (uint32_t)g.Lx);
    s.near = is_near(g, s.rx, s.ry);
    const bool ok = !done && x * N >= g.rej && offset_allowed(g.Lx, g.Ly, s.rx, s.ry);
    const uint32_t m = (__ballot_sync(0xFFFFFFFFu, ok) >> (lane & ~3u)) & 15u;
    if (m && (lane & 3u) == (uint32_t)__ffs((int)m) - 1u) s_d[p & 15u] = phase_desc(g, s, cls_bytes);
    done = done || m;
    if (__all_sync(0xFFFFFFFFu, done)) return;
  }
  if (!done && (lane & 3u) == 0)
    s_d[p & 15u] = phase_desc(g, Sched{0, 0, 2, 2, is_near(g, 2, 2)}, cls_bytes);
}

template <bool kCl, bool kAl>
__device__ __forceinline__ uint32_t read_window(uint32_t row, const Win &x) {
  uint32_t v = __funnelshift_r(ld_word<kCl>(row + 4u * (uint32_t)x.lo),
                               ld_word<kCl>(row + 4u * (uint32_t)x.hi), x.sh);
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
  xor_word<kCl>(row + 4u * (uint32_t)x.lo, d1 << x.sh);
  xor_word<kCl>(row + 4u * (uint32_t)x.hi, __funnelshift_l(d1, 0u, x.sh));  // d1 >> (32 - sh), 0 for sh = 0
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
    const uint32_t rank = __umulhi((uint32_t)j, pl.mrows);  // clusters have rows >= 2
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

// Row jb of a side's sites for the a sites' row l of this CTA.
__device__ __forceinline__ int side_row(const Geo &g, const Place &pl, const SideD &d, int l) {
  return turn(pl.row0 + l + d.qy, g.Cy);
}

// One side of a word read the general way (rows anywhere in the cluster): the
// 16 sites and their neighbours' counts.
struct SideIn {
  uint32_t X;
  Planes n;
};

template <bool kCl, bool kAl>
__device__ __forceinline__ SideIn gather_side(const Geo &g, const SideD &d, const Place &pl,
                                              int l, const Win &win, uint32_t row, int w) {
  SideIn in;
  const uint32_t ry = row_addr<kCl>(pl, turn(side_row(g, pl, d, l) + d.ys, g.Cy));
  in.X = read_window<kCl, kAl>(row + d.c, win);
  const uint32_t m = read_window<kCl, kAl>(row + d.m, win);
  const uint32_t r = read_window<kCl, kAl>(row + d.r, win);
  const uint32_t x = read_window<kCl, kAl>(row + d.x, window_at<kAl>(g, w, d.offX));
  const uint32_t y = read_window<kCl, kAl>(ry + d.y, win);
  in.n = neighbour_planes(m, r, x, y);
  return in;
}

// The b side of the words of a whole warp in a cluster (kTPW lanes a word), as
// gather_side: a window's second word is the first word of the lane that holds the
// next word of the row, so it comes from that lane; only lanes without such a
// neighbour (the warp's last, a ragged row's turn) load it.  Remote shared memory
// delivers 10 to 13 bytes a cycle to an SM: this halves its share of a phase.
template <bool kAl, int kTPW>
__device__ __forceinline__ SideIn gather_remote(const Geo &g, const SideD &d, const Place &pl,
                                                int l, int w) {
  const int lane = threadIdx.x & 31;
  const int next = w + 1 < g.W ? lane + kTPW : lane + kTPW * (1 - g.W);
  const int src = next >= 0 && next < 32 ? next : lane;
  const int jb = side_row(g, pl, d, l);
  const uint32_t row = row_addr<true>(pl, jb), ry = row_addr<true>(pl, turn(jb + d.ys, g.Cy));
  const Win win = window_at<kAl>(g, w, d.qx), wx = window_at<kAl>(g, w, d.offX);
  const bool near = __shfl_sync(0xFFFFFFFFu, row + 4u * (uint32_t)win.lo, src) == row + 4u * (uint32_t)win.hi;
  const bool nearx = __shfl_sync(0xFFFFFFFFu, row + 4u * (uint32_t)wx.lo, src) == row + 4u * (uint32_t)wx.hi;
  const uint32_t at[5] = {row + d.c, row + d.m, row + d.r, ry + d.y, row + d.x};
  uint32_t lo[5], v[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) lo[k] = ld_word<true>(at[k] + 4u * (uint32_t)(k < 4 ? win.lo : wx.lo));
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const Win &x = k < 4 ? win : wx;
    const uint32_t hi = ld_remote_if(!(k < 4 ? near : nearx), at[k] + 4u * (uint32_t)x.hi,
                                     __shfl_sync(0xFFFFFFFFu, lo[k], src));
    v[k] = __funnelshift_r(lo[k], hi, x.sh);
    if constexpr (!kAl) {
      if (x.n1 < 16)
        v[k] = (v[k] & ((1u << (2 * x.n1)) - 1u)) | (ld_word<true>(at[k]) << (2 * x.n1));
    }
  }
  SideIn in;
  in.X = v[0];
  in.n = neighbour_planes(v[1], v[2], v[3], v[4]);
  return in;
}

// Both sides of a word, the a side (this CTA's rows, whole words) read directly.
// kTPW: all lanes of the warp call, with so many lanes a word.
template <bool kCl, bool kAl, int kTPW>
__device__ __forceinline__ WordIn gather_word(const Geo &g, const PhaseD &u, const Place &pl,
                                              const Spot &p) {
  WordIn in;
  const SideD &a = u.side[0], &b = u.side[1];
  if constexpr (kCl) {
    const SideIn s = gather_remote<kAl, kTPW>(g, b, pl, p.l, p.w);
    in.B = s.X;
    in.nb = s.n;
  } else {
    const uint32_t row = row_addr<kCl>(pl, side_row(g, pl, b, p.l));
    const SideIn s =
        gather_side<kCl, kAl>(g, b, pl, p.l, window_at<kAl>(g, p.w, b.qx), row, p.w);
    in.B = s.X;
    in.nb = s.n;
  }
  const int j = pl.row0 + p.l;
  const uint32_t own = pl.base + p.off;
  in.A = ld_word<false>(own + a.c);
  const uint32_t am = ld_word<false>(own + a.m);
  const uint32_t ar = ld_word<false>(own + a.r);
  const uint32_t ax = side_window<kAl>(g, p, own + a.x, a.xs);
  const int jy = turn(j + a.ys, g.Cy);
  uint32_t ay;
  if constexpr (kCl)
    ay = ld_word<true>(row_addr<true>(pl, jy) + a.y + 4u * (uint32_t)p.w);
  else
    ay = ld_word<false>(own + a.y + (uint32_t)(jy - j) * pl.row_bytes);
  in.na = neighbour_planes(am, ar, ax, ay);
  return in;
}

// Apply the moves (dA, dB) of a word's sites.
template <bool kCl, bool kAl>
__device__ __forceinline__ void apply_word(const Geo &g, const PhaseD &u, const Place &pl,
                                           const Spot &p, uint32_t dA, uint32_t dB) {
  xor_word<false>(pl.base + p.off + u.side[0].c, dA);
  const SideD &b = u.side[1];
  xor_window<kCl, kAl>(row_addr<kCl>(pl, side_row(g, pl, b, p.l)) + b.c,
                       window_at<kAl>(g, p.w, b.qx), dB);
}

// Bits of a word's sites that exist (the row may end in it), none for a thread
// without a word.
template <bool kAl>
__device__ __forceinline__ uint32_t valid_bits(const Geo &g, const Spot &p, bool act) {
  uint32_t v = 0xFFFFFFFFu;
  if constexpr (!kAl) {
    const int n = g.Cx - (p.w << 4);
    if (n < 16) v = (1u << (2 * n)) - 1u;
  }
  return act ? v : 0u;
}

// Round keys in shared memory (five 16-byte loads a call instead of twenty
// additions on the drawing thread's chain).
__device__ __forceinline__ U4 philox_keys(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                          const uint32_t *rk) {
  const uint4 *k4 = reinterpret_cast<const uint4 *>(rk);
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    const uint4 k = k4[r];
    uint32_t lo0, hi0, lo1, hi1;
    mul_wide(0xD2511F53u, c0, lo0, hi0);
    mul_wide(0xCD9E8D57u, c2, lo1, hi1);
    c0 = hi1 ^ c1 ^ k.x;
    c2 = hi0 ^ c3 ^ k.y;
    c1 = lo1;
    c3 = lo0;
    mul_wide(0xD2511F53u, c0, lo0, hi0);
    mul_wide(0xCD9E8D57u, c2, lo1, hi1);
    c0 = hi1 ^ c1 ^ k.z;
    c2 = hi0 ^ c3 ^ k.w;
    c1 = lo1;
    c3 = lo0;
  }
  return U4{c0, c1, c2, c3};
}

// ----------------------------------------------------------------------------
// Four lanes a word (lattices with few words an SM, bound by one thread's chain).
// Lane sub decides group k = sub (call sub / 2, half sub mod 2).  Lanes 0 and 1
// read the a side, lanes 2 and 3 the b side, each for its half; three exchanges
// with lane sub XOR 2 bring the other side.  The random words come from draw
// threads (two a word, one a call) one phase ahead, already divided by 12.

// A draw thread's call: for every half the four pairs' fields as wq << 16 |
// 264 r (a field >= 65532 has wq = 5461; bit 15 of the first: the call has one).
__device__ __forceinline__ void draw_call(uint32_t gbase, int c, uint64_t P, const uint32_t *rk,
                                          uint4 *out) {
  const U4 r = philox_keys(gbase + (uint32_t)c, (uint32_t)P, (uint32_t)(P >> 32), TAG_MOVE, rk);
  const uint32_t mx = __vmaxu2(__vimax3_u16x2(r.x, r.y, r.z), r.w);
  const uint32_t flag = mx >= 0xFFFC0000u || (mx & 0xFFFFu) >= 0xFFFCu ? 0x8000u : 0u;
  const uint32_t X[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t v = h ? X[q] >> 16 : X[q] & 0xFFFFu;
      const uint32_t wq = div12(v);
      f[q] = (wq << 16) + (v - 12u * wq) * 264u;
    }
    out[h] = make_uint4(f[0] | flag, f[1], f[2], f[3]);
  }
}

// One phase of a word by its four lanes (inactive lanes: valid 0): the word's
// moves applied.
template <bool kCl, bool kAl>
__device__ __forceinline__ void quad_word(const Geo &g, const PhaseD &u, const Place &pl,
                                          const uint2 *trans, const uint16_t *thrT,
                                          const uint32_t *thr32, const uint32_t *rk,
                                          const Spot &p, int sub, uint32_t valid, const uint4 &f,
                                          uint64_t P) {
  const SideD &d = u.side[sub >> 1];
  const int h2 = 2 * (sub & 1), c4 = 4 * (sub >> 1);
  const uint32_t row = row_addr<kCl>(pl, side_row(g, pl, d, p.l));
  const Win win = window_at<kAl>(g, p.w, d.qx);
  const SideIn s = gather_side<kCl, kAl>(g, d, pl, p.l, win, row, p.w);
  // this side's (2 n1, n0) of the half's pairs, two pairs a word (see half_env)
  const uint32_t O = s.n.O >> h2, T = (s.n.T >> h2) << 1, F = (s.n.F >> h2) << 2;
  const uint32_t n1 = lop3<kLutMux>(F, lop3<kLutMux>(O, T, 0x22222222u), 0x88888888u);
  const uint32_t n0 = lop3<kLutMux>(F, lop3<kLutMux>(O, T, 0x11111111u), 0x44444444u);
  const uint32_t x01 = prmt(n1, n0, 0x5140u), x23 = prmt(n1, n0, 0x7362u);
  const uint32_t o01 = __shfl_xor_sync(0xFFFFFFFFu, x01, 2);
  const uint32_t o23 = __shfl_xor_sync(0xFFFFFFFFu, x23, 2);
  const uint32_t oX = __shfl_xor_sync(0xFFFFFFFFu, s.X, 2);
  // operands (a's counts below b's): the lane's own side first or second
  const uint32_t lo = sub < 2 ? 0x5410u : 0x1054u, hi = sub < 2 ? 0x7632u : 0x3276u;
  const uint32_t ev[4] = {prmt(x01, o01, lo), prmt(x01, o01, hi), prmt(x23, o23, lo),
                          prmt(x23, o23, hi)};
  const uint32_t A = sub < 2 ? s.X : oX, B = sub < 2 ? oX : s.X;
  const uint32_t pcs = half_pc(A >> h2, B >> h2, 0);
  const uint32_t pc = __funnelshift_l(pcs, pcs, 3 - c4);
  const uint2 *moves = trans + (u.near128 >> 3);  // + 128 near bytes
  const uint32_t fs[4] = {f.x, f.y, f.z, f.w};
  uint32_t df[4], t[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint2 e = move_entry(moves, entry_offset(pc, q, fs[q] & 0x7FFFu));
    t[q] = (uint32_t)__dp4a((int)e.y, (int)((ev[q] >> c4) & kEnvMask), (int)e.x);
    df[q] = fs[q] - (level_at(thrT, t[q] & 0xFFFFu) << 16);  // negative: accept; < 2^16: a tie
  }
  const uint32_t mn = __vimin3_u32(__vimin3_u32(df[0], df[1], df[2]), df[3], df[3]);
  const uint32_t acc = prmt(prmt(df[0], df[1], 0x00FBu), prmt(df[2], df[3], 0x00FBu), 0x5410u) &
                       prmt(prmt(t[0], t[1], 0x0073u), prmt(t[2], t[3], 0x0073u), 0x5410u);
  uint32_t dB = (acc & 0x03030303u) << (2 * sub);
  uint32_t dA = ((acc >> 2) & 0x03030303u) << (2 * sub);
  // the word's moves together; one lane a side writes its sites
  uint32_t mine = sub < 2 ? dA : dB, other = sub < 2 ? dB : dA;
  mine |= __shfl_xor_sync(0xFFFFFFFFu, other, 2);
  mine |= __shfl_xor_sync(0xFFFFFFFFu, mine, 1);
  if (sub & 1) mine = 0u;
  xor_window<kCl, kAl>(row + d.c, win, mine & valid);
  // The rare pairs, which the fast path left as they were, decided exactly behind the
  // word's other moves: no lane waits at this branch before the exchange (256^2: 7.8 us
  // a sweep with it there, 7.2 here; 16^2: 4.06, 3.93).
  if ((mn < 0x10000u || (f.x & 0x8000u)) && valid) {
    uint32_t m = 0u, wq[4], e4[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      wq[q] = fs[q] >> 16;
      e4[q] = (ev[q] >> c4) & kEnvMask;
      if (df[q] < 0x10000u || wq[q] == 5461u) m |= 1u << q;
    }
    const uint32_t slow0 = (uint32_t)(pl.row0 + p.l) * (uint32_t)g.Cx + (uint32_t)(p.w << 4);
    const uint32_t x = exact_group(
        trans, thr32, m, wq, t, e4, pc, u.near128, slow0 + (uint32_t)sub, [&](uint32_t i) {
          return philox_keys(i, (uint32_t)P, (uint32_t)(P >> 32), TAG_SLOW, rk);
        });
    apply_word<kCl, kAl>(g, u, pl, p, (((x >> 2) & 0x03030303u) << (2 * sub)) & valid,
                         ((x & 0x03030303u) << (2 * sub)) & valid);
  }
}

// Observables of this CTA's words by definition, as sums over bit products of
// the linear code (S = b1 - b0, sigma = 1 - b1 - b0), added to out[0..6] (of the
// cluster's first CTA): a site's bits against its right and down neighbours', like
// bits and unlike ones; the sites' b1 and b0; both; b1 and b0 on the sites of even
// x + y.  A thread takes the four classes of a row of sites at one word place: they
// are each other's right neighbours, so nine loads serve four words and only the
// last one's window crosses into the next word.  Bits above a ragged row's end are
// zero in the words, so they count nowhere.  Two 16-bit counts share a register
// through the warp's sums (a thread takes at most seven places between them: 7 x
// 256 x 32 < 2^16).
template <bool kCl, bool kAl>
__device__ __forceinline__ void count_words(const Geo &g, const Place &pl, int nw, uint32_t mw,
                                            uint32_t mn, uint32_t cls_bytes, int tid, int nthreads,
                                            int *out) {
  constexpr uint32_t kOdd = 0xAAAAAAAAu;
  uint32_t dst = smem_addr(out);
  if constexpr (kCl) dst = map_rank(dst, 0u);
  const int lane = threadIdx.x & 31;
  for (int i = tid; i - lane < 4 * nw;) {  // uniform in the warp
    uint32_t bonds = 0u, bits = 0u, both = 0u, even = 0u;
    for (int k = 0; k < 7 && i - lane < 4 * nw; ++k, i += nthreads) {
      if (i >= 4 * nw) continue;
      const int cy = nw == 1 ? i : (int)__umulhi((uint32_t)i, mn);
      const int wid = i - cy * nw;
      const int l = g.W == 1 ? wid : (int)__umulhi((uint32_t)wid, mw);
      const Spot p = spot_of(g, pl, l, wid - l * g.W);
      const uint32_t own = pl.base + p.off + (uint32_t)(4 * cy) * cls_bytes;
      uint32_t X[4], Yr[4], Yd[4];
#pragma unroll
      for (int cx = 0; cx < 4; ++cx) X[cx] = ld_word<false>(own + (uint32_t)cx * cls_bytes);
      if (kCl && cy == 3) {
        const uint32_t down =
            row_addr<true>(pl, turn(pl.row0 + l + 1, g.Cy)) + 4u * (uint32_t)p.w;
#pragma unroll
        for (int cx = 0; cx < 4; ++cx) Yd[cx] = ld_word<true>(down + (uint32_t)cx * cls_bytes);
      } else {
        const uint32_t down = cy < 3 ? own + 4u * cls_bytes
                                     : pl.base + p.off + (uint32_t)(turn(l + 1, g.Cy) - l) * pl.row_bytes;
#pragma unroll
        for (int cx = 0; cx < 4; ++cx) Yd[cx] = ld_word<false>(down + (uint32_t)cx * cls_bytes);
      }
      Yr[0] = X[1];
      Yr[1] = X[2];
      Yr[2] = X[3];
      Yr[3] = side_window<kAl>(g, p, own, g.Cx > 1 ? 1 : 0);
      uint32_t like = 0u, unlike = 0u, B[4];
#pragma unroll
      for (int cx = 0; cx < 4; ++cx) {
        const uint32_t Xs = lop3<kLutMux>(X[cx] << 1, X[cx] >> 1, kOdd);  // b0, b1 swapped
        like += (uint32_t)(__popc(X[cx] & Yr[cx]) + __popc(X[cx] & Yd[cx]));
        unlike += (uint32_t)(__popc(Xs & Yr[cx]) + __popc(Xs & Yd[cx]));
        B[cx] = X[cx] & Xs;
      }
      bonds += like + (unlike << 16);
      // two classes of one parity share a count
      uint32_t b[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        b[h] = (uint32_t)__popc(lop3<kLutMux>(X[h], X[h + 2] >> 1, kOdd)) +
               ((uint32_t)__popc(lop3<kLutMux>(X[h] << 1, X[h + 2], kOdd)) << 16);
        both += (uint32_t)__popc(lop3<kLutMux>(B[h], B[h + 2], kOdd));
      }
      bits += b[0] + b[1];
      even += cy & 1 ? b[1] : b[0];
    }
    bonds = __reduce_add_sync(0xFFFFFFFFu, bonds);
    bits = __reduce_add_sync(0xFFFFFFFFu, bits);
    both = __reduce_add_sync(0xFFFFFFFFu, both);
    even = __reduce_add_sync(0xFFFFFFFFu, even);
    const uint32_t v = lane < 2 ? bonds : lane < 4 ? bits : lane == 4 ? both : even;
    const uint32_t add = lane == 4 ? v
                         : (lane == 1 || lane == 3 || lane == 6) ? v >> 16 : v & 0xFFFFu;
    if (lane < 7) {
      if constexpr (kCl)
        asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(
                         dst + 4u * (uint32_t)lane),
                     "r"(add)
                     : "memory");
      else
        atomicAdd(out + lane, (int)add);
    }
  }
}

}  // namespace

// Threads: `workers` (a multiple of 32), with four lanes a word then workers / 2
// draw threads (rounded up to warps), then the auxiliary warp.  The register limit
// (96 a thread, by the largest CTA) leaves hardly a spill: a spilled value read
// after a cluster barrier comes from L2, as the barrier's acquire empties L1
// (1024^2 on sixteen CTAs: 19.4 us a sweep, 23.6 at 72 registers).
template <bool kCl, bool kAl, int kTPW>
__global__ void __launch_bounds__(kResMaxThreads, 1)
    resident_sweep_kernel(const __grid_constant__ ResJob one, const ResJob *__restrict__ jobs,
                          int cluster, int workers) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  __shared__ PhaseD s_d[16];  // phase P's uniforms in slot P mod 16
  __shared__ int s_obs[2][8]; // the counts of even and odd records
  __shared__ ResJob s_job;    // read where used: its fields would fill the registers
  uint16_t *thrT = reinterpret_cast<uint16_t *>(res_smem);
  uint2 *trans = reinterpret_cast<uint2 *>(res_smem + 2 * kThrT);
  const uint32_t *thr32 = reinterpret_cast<const uint32_t *>(res_smem + kFastBytes);
  int tid;  // opaque: the compiler would read the special register again every phase
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  const int lane = tid & 31;
  {
    const uint32_t *src = reinterpret_cast<const uint32_t *>(
        jobs ? jobs + (kCl ? blockIdx.x / cluster : blockIdx.x) : &one);
    for (int t = tid; t < (int)(sizeof(ResJob) / 4); t += blockDim.x)
      reinterpret_cast<uint32_t *>(&s_job)[t] = src[t];
    __syncthreads();
  }
  const ResJob &J = s_job;
  const Geo &g = s_job.g;
  const bool aux = tid >= (int)blockDim.x - 32;
  const bool worker = tid < workers;
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
  const uint32_t mn = nr * g.W > 1 ? 0xFFFFFFFFu / (uint32_t)(nr * g.W) + 1u : 0u;
  // tables and words in
  {
    const uint4 *src = reinterpret_cast<const uint4 *>(J.thrT);  // one block in this order
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
  // sweeps until the next record, and the record writer's ring position
  int until = obs_every > 0 ? obs_every - (int)((P0 / 8) % obs_every) : 0;
  int64_t obs_cnt = 0, obs_slot = 0;
  if (aux) {
    describe_sweep(g, (uint64_t)P0, cls_bytes, s_d);
    if (obs_every > 0 && rank == 0 && lane == 0) {
      obs_cnt = g.ctl[kCtlObsCount];
      obs_slot = obs_cnt % J.ring_cap;
    }
  }
  const int items = kTPW * nr * g.W;
  auto place = [&](int wid) {
    const int l = g.W > 1 ? (int)__umulhi((uint32_t)wid, mw) : wid;
    return spot_of(g, pl, l, wid - l * g.W);
  };
  auto base_of = [&](const Spot &p) {
    return (uint32_t)(pl.row0 + p.l) * (uint32_t)(2 * g.W) + (uint32_t)(2 * p.w);
  };
  // four lanes a word: the fields of phase P in buffer P mod 2, 16 bytes a worker
  uint4 *fields =
      reinterpret_cast<uint4 *>(res_smem + kTableBytes + 16u * cls_bytes);
  const int call = tid - workers;  // a draw thread's call
  const bool drawer = kTPW == 4 && !worker && !aux && 2 * call < items;
  Spot pt = place(worker ? (tid < items ? tid / kTPW : 0) : drawer ? call >> 1 : 0);
  const int sub = tid % kTPW;
  constexpr int kCalls = kTPW == 1 ? 2 : 1;
  U4 rn[kCalls];  // one or two threads a word: the random words of the word at pt
  auto draw_next = [&](uint64_t P) {
    if constexpr (kTPW == 4) {
      if (drawer)
        draw_call(base_of(pt), call & 1, P, J.rk, fields + (P & 1u) * workers + 2 * call);
    } else {
#pragma unroll
      for (int ci = 0; ci < kCalls; ++ci)
        rn[ci] = philox_keys(base_of(pt) + (uint32_t)(kTPW == 1 ? ci : sub), (uint32_t)P,
                             (uint32_t)(P >> 32), TAG_MOVE, J.rk);
    }
  };
  if (!aux) draw_next((uint64_t)P0);
  uint32_t valid = valid_bits<kAl>(g, pt, tid < items);
  const bool warp_has = tid - lane < items;
  bar_arrive<kCl>();
  bar_wait<kCl>();
  // The barrier of a phase.  On one CTA the auxiliary warp only joins a sweep's last.
  auto phase_wait = [&](int p) {
    if (kCl || p == 7)
      bar_wait<kCl>();
    else
      asm volatile("bar.sync 1, %0;" ::"r"((int)blockDim.x - 32) : "memory");
  };
  int obs_buf = 0;
  const int nsweeps = J.nsweeps;
  for (int sweep = 0; sweep < nsweeps; ++sweep) {
    const uint64_t S = (uint64_t)P0 + 8u * (uint32_t)sweep;
    if (aux) {
      // the next sweep's schedules, into the other eight slots
      if constexpr (kCl) {
        bar_arrive<true>();
        describe_sweep(g, S + 8u, cls_bytes, s_d);
        bar_wait<true>();
        for (int p = 1; p < 8; ++p) {
          bar_arrive<true>();
          bar_wait<true>();
        }
      } else {
        describe_sweep(g, S + 8u, cls_bytes, s_d);
        __syncthreads();
      }
    } else if (kTPW == 4 && !worker) {
#pragma unroll 1
      for (int p = 0; p < 8; ++p) {
        draw_next(S + (uint32_t)p + 1u);
        bar_arrive<kCl>();
        phase_wait(p);
      }
    } else {
#pragma unroll 1
      for (int p = 0; p < 8; ++p) {
        const uint64_t P = S + (uint32_t)p;
        const PhaseD &u = s_d[P & 15u];
        if constexpr (kTPW == 4) {
          if (warp_has) {
            // lanes without a word decide word 0 on zero fields (nobody draws theirs, and
            // what the buffer holds there is no table offset); valid drops their moves
            const uint4 f =
                tid < items ? fields[(P & 1u) * workers + tid] : uint4{0u, 0u, 0u, 0u};
            quad_word<kCl, kAl>(g, u, pl, trans, thrT, thr32, J.rk, pt, sub, valid, f, P);
          }
          bar_arrive<kCl>();
        } else {
          if (!warp_has) {
            bar_arrive<kCl>();
            phase_wait(p);
            continue;
          }
          for (int base = tid - lane;;) {  // uniform in the warp
            const WordIn in = gather_word<kCl, kAl, kTPW>(g, u, pl, pt);
            uint3 d = fast_moves<kTPW, true>(trans, thrT, sub, in, u.near128,
                                             [&](int c) { return rn[kTPW == 1 ? c : 0]; });
            // rare pairs, decided by their own thread from the inputs it holds (all
            // lanes together after exchanging them took longer, and the whole cluster
            // waits at its barrier for the last warp of a phase)
            if (!valid) d.z = 0u;
#pragma unroll 1
            while (d.z) {
              const int t = __ffs((int)d.z) - 1, q = t >> 2;
              d.z &= d.z - 1u;
              uint32_t X = q == 0 ? rn[0].x : q == 1 ? rn[0].y : q == 2 ? rn[0].z : rn[0].w;
              if constexpr (kTPW == 1) {  // no indexing: rn stays in registers
                const U4 &r = rn[kCalls - 1];
                if (t & 2) X = q == 0 ? r.x : q == 1 ? r.y : q == 2 ? r.z : r.w;
              }
              const uint32_t x = rare_move(
                  trans, thr32, t, in, X,
                  (uint32_t)(pl.row0 + pt.l) * (uint32_t)g.Cx + (uint32_t)(pt.w << 4), u.near128,
                  [&](uint32_t i) {
                    return philox_keys(i, (uint32_t)P, (uint32_t)(P >> 32), TAG_SLOW, J.rk);
                  });
              d.x |= (x >> 2) << (2 * t);
              d.y |= (x & 3u) << (2 * t);
            }
            apply_word<kCl, kAl>(g, u, pl, pt, d.x & valid, d.y & valid);
            // on to the next pass, or with the phase's last to the next phase: the next
            // word's random words are drawn here, behind the arrival at the barrier
            base += workers;
            const bool last = base >= items;
            if (last) bar_arrive<kCl>();
            const int i = last ? tid : base + lane;
            if (items > workers) {
              pt = place(i < items ? i / kTPW : 0);
              valid = valid_bits<kAl>(g, pt, i < items);
            }
            draw_next(P + (last ? 1u : 0u));
            if (last) break;
          }
        }
        phase_wait(p);
      }
    }
    if (obs_every > 0 && --until == 0) {
      until = obs_every;
      if (!aux)
        count_words<kCl, kAl>(g, pl, nr * g.W, mw, mn, cls_bytes, tid, (int)blockDim.x - 32,
                              s_obs[obs_buf]);
      // the counts are complete, and no word changes before all are counted
      bar_arrive<kCl>();
      bar_wait<kCl>();
      if (aux && rank == 0 && lane == 0) {
        volatile int *c = s_obs[obs_buf];
        const int64_t like = c[0], unlike = c[1], b1 = c[2], b0 = c[3], both = c[4],
                      s1 = 2 * (int64_t)c[5] - b1, s0 = 2 * (int64_t)c[6] - b0;
        for (int k = 0; k < 7; ++k) c[k] = 0;  // for the record after the next
        const int64_t N = (int64_t)g.Lx * g.Ly;
        const int64_t rec[8] = {(int64_t)(S / 8u) + 1, b1 + b0 - 2 * both, like - unlike,
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
    if (rank == 0 && tid == 0) g.ctl[kCtlPhaseBase] = P0 + 8 * (int64_t)nsweeps;
  }
}

namespace {

using Kernel = void (*)(const ResJob, const ResJob *, int, int);

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
int g_limit[kMaxDevices] = {};  // resident_cluster_limit + 1, 0: not asked yet

void launch_config(const ResShape &shape, int njobs, cudaStream_t s, cudaLaunchConfig_t &cfg,
                   cudaLaunchAttribute *attr) {
  cfg.gridDim = dim3((unsigned)(njobs * shape.cluster));
  cfg.blockDim = dim3((unsigned)shape.threads);
  cfg.dynamicSmemBytes = (size_t)shape.smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)shape.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = shape.cluster > 1 ? 1 : 0;
}

// Raises every instance's shared-memory limit and allows clusters of 16 (outside any
// capture: called when a lattice is created), then asks for the largest cluster that
// the device places with the most threads and shared memory a CTA may have: a part of
// a GPU may have no sixteen SMs side by side, and its lattices then take smaller
// clusters or a launch a phase.  (A whole GB300 holds seven such clusters of 16.)
int cluster_limit() {
  for (int c = 0; c < 2; ++c)
    for (int a = 0; a < 2; ++a)
      for (int t : {1, 2, 4})
        if (cudaFuncSetAttribute(reinterpret_cast<const void *>(kernel_of(c, a, t)),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kResMaxSmem) != cudaSuccess) {
          cudaGetLastError();
          return 0;
        }
  for (int C = kResMaxCluster; C > 1; C /= 2) {
    bool ok = true;
    for (int a = 0; a < 2; ++a)
      for (int t : {1, 2, 4}) {
        const void *f = reinterpret_cast<const void *>(kernel_of(true, a, t));
        ResShape most;
        most.cluster = C;
        most.threads = kResMaxThreads;
        most.smem = kResMaxSmem;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute attr[1];
        launch_config(most, 1, nullptr, cfg, attr);
        int n = 0;
        ok = ok &&
             cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, C > 8) ==
                 cudaSuccess &&
             cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n > 0;
      }
    if (ok) return C;
    cudaGetLastError();
  }
  return 1;
}

}  // namespace

int resident_cluster_limit() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_limit[dev]) g_limit[dev] = cluster_limit() + 1;
  return g_limit[dev] - 1;
}

int64_t resident_smem(const Geo &g, int rows) {
  return (int64_t)kTableBytes + 64ll * rows * g.W;
}

// The shape of `rows` rows a CTA of a cluster of C.
static ResShape shape_of(const Geo &g, int C, int tpw, int max_workers) {
  ResShape sh;
  sh.cluster = C;
  sh.rows = (g.Cy + C - 1) / C;
  sh.tpw = tpw;
  const int words = sh.rows * g.W;
  // whole warps, beyond 128 in steps of 64 (fewer different shapes in a batch)
  const int step = tpw * words <= 128 ? 32 : 64;
  const int workers = std::min((tpw * words + step - 1) / step * step, max_workers);
  sh.workers = workers;
  sh.threads = workers + (tpw == 4 ? (workers / 2 + 31) / 32 * 32 : 0) + 32;
  sh.smem = resident_smem(g, sh.rows) + (tpw == 4 ? 32 * workers : 0);
  return sh;
}

// Shapes, measured on GB300 (us a sweep, records off).  A cluster's barrier and
// remote windows cost 0.4 us a phase, which pays from 128 words a phase: 128^2
// (64 words) 5.2 on one CTA, 6.1 on four; 256^2 10.6 on one, 8.7 on four, 7.2 on
// sixteen; 1024^2 37.7 on four, 21.8 on eight, 15.0 on sixteen.  Four lanes a word up
// to 96 words a CTA (64^2: 3.3, with one 6.5; 516^2, 81 words a CTA: 12.9, with two
// 13.3), of rows of whole words up to 48 (448^2, 49 words: 10.6 both; 512^2, 64: 10.9,
// with two 10.2; 576^2, 81: 12.5, 12.1); above that the work repeated for threads that
// share a word costs more than the shorter chain hides (1024^2 on sixteen: 15.0 with
// one thread, 16.8 with two), two threads paying up to 128 words.  When lattices crowd
// the SMs only the smallest keep four lanes: their four kinds of warps fall on the four
// schedulers (a lone worker warp a CTA lands on the same one every time: 128 lattices of
// 256^2 and 128 of 64^2 34 against 23; 512 replicas: 28 against 14.7), while a
// 416-thread CTA finds no room beside another (512 replicas: 18.5 with four lanes for
// their 128^2 lattices, 14.7 with one thread).
ResShape resident_shape(const Geo &g, int max_cluster, double ctas, double load, int max_threads,
                        int max_tpw) {
  int C = 1;
  if (g.cstride >= kResClusterWords)
    while (C < max_cluster && 2 * C <= ctas && g.cstride >= 2 * C * kResMinWords &&
           g.Cy >= 4 * C)  // two rows a CTA at least
      C *= 2;
  while (C < max_cluster && g.Cy >= 4 * C && resident_smem(g, (g.Cy + C - 1) / C) > kResMaxSmem)
    C *= 2;
  const int words = (g.Cy + C - 1) / C * g.W;
  const bool crowded = load > 128.0;
  const int quad = crowded ? 32 : (g.Cx & 15) == 0 ? 48 : kResQuadWords;
  int tpw = 1;
  if (max_tpw >= 4 && words <= quad)
    tpw = 4;
  else if (max_tpw >= 2 && words <= 128 && !crowded)
    tpw = 2;
  while (tpw > 1 && tpw * words > max_threads) tpw /= 2;
  return shape_of(g, C, tpw, max_threads);
}

bool resident_possible(const Geo &g, int max_cluster) {
  return max_cluster > 0 && resident_shape(g, max_cluster, max_cluster, 0.0, kResMaxWorkers, 1)
                                    .smem <= kResMaxSmem;
}

// Clusters of eight full CTAs do not all find eight free SMs of one processing
// cluster: for 16 lattices of 1024^2 two waited for the others (54 us a sweep).
// CTAs of 128 workers that take their words in several passes fit four to an SM:
// 37 us (eight CTAs of 256 workers, two to an SM: 43).
ResShape resident_fit(const Geo &g, int max_cluster, const ResShape &shape, bool aligned, int n) {
  auto fits = [&](const ResShape &sh) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    launch_config(sh, n, nullptr, cfg, attr);
    int most = 0;
    if (cudaOccupancyMaxActiveClusters(
            &most, reinterpret_cast<const void *>(kernel_of(true, aligned, sh.tpw)), &cfg) !=
        cudaSuccess) {
      cudaGetLastError();
      return true;
    }
    return n <= most;
  };
  if (shape.cluster == 1 || fits(shape)) return shape;
  if (max_cluster == kResMaxCluster && g.cstride >= kResMaxCluster * 128 &&
      g.Cy >= 2 * kResMaxCluster) {
    const ResShape wide = shape_of(g, kResMaxCluster, 1, std::min(128, shape.workers));
    if (fits(wide)) return wide;
  }
  if (shape.cluster > 2) {
    const ResShape half = shape_of(g, shape.cluster / 2, shape.tpw, shape.workers);
    if (half.smem <= kResMaxSmem &&
        (half.tpw == 1 || half.tpw * half.rows * g.W <= half.workers) && fits(half))
      return half;
  }
  return shape;
}

cudaError_t launch_resident_sweep(const ResJob *one, const ResJob *d_jobs, int njobs,
                            const ResShape &shape, bool aligned, cudaStream_t s) {
  // (a block barrier of a part of a warp would never complete)
  if (shape.workers % 32 || shape.threads % 32 || shape.threads > kResMaxThreads)
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  launch_config(shape, njobs, s, cfg, attr);
  return cudaLaunchKernelEx(&cfg, kernel_of(shape.cluster > 1, aligned, shape.tpw),
                            one ? *one : ResJob{}, one ? nullptr : d_jobs, shape.cluster,
                            shape.workers);
}

}  // namespace ccmc
