// ccmc_word.cuh -- the per-word core of a colour phase, shared by the phase
// kernels and the resident kernel: the 16 pairs of one a-class word decided from
// the word's inputs (its a word, b window and both sides' neighbour counts), and the
// phase's uniforms from which a kernel reads those inputs.  How it reads them and
// where the moves go is each kernel's own.
#pragma once

#include <cstdint>

#include "ccmc_device.cuh"
#include "ccmc_internal.h"

namespace ccmc {

// One phase's uniforms of one side (a or b): classes as offsets of a unit of the
// kernel's, column offsets in sites, row offsets.  Of a site's two column neighbours
// at most one lies in another column block, and of its two row neighbours at most
// one in another row: the neighbour sums do not care which is which, so a side
// has its own class c, one column neighbour read at the side's own column (m) and
// one xs = -1, 0 or 1 sites further (x), one row neighbour in its own row (r)
// and one 0, 1 or Cy - 1 rows further (y, ys).  The side's sites lie qx columns and
// qy rows from the a sites (0, 0 for a itself); offX = qx + xs in [0, Cx).
struct alignas(16) SideD {
  uint32_t c, m, x, r, y;
  int qx, offX, qy, ys, xs;
  int pad[2];
};
struct alignas(16) PhaseD {
  SideD side[2];
  uint32_t near128;
};

// v in [0, 2 n) modulo n: an unsigned minimum instead of a comparison and a choice.
__device__ __forceinline__ int turn(int v, int n) {
  return (int)min((uint32_t)v, (uint32_t)(v - n));
}

// The phase's uniforms from its schedule, class c at offset c * unit.
__device__ __forceinline__ PhaseD phase_desc(const Geo &g, const Sched &sc, uint32_t unit) {
  PhaseD u;
  auto cls = [&](int cx, int cy) { return (uint32_t)((cy & 3) * 4 + (cx & 3)) * unit; };
  // -1 when the left (upper) neighbours lie in the block (row) before, +1 when the
  // right (lower) ones lie in the next
  auto shift = [](int c) { return c == 0 ? -1 : c == 3 ? 1 : 0; };
  auto side = [&](SideD &d, int x, int y) {
    const int cx = x & 3, cy = y & 3;
    const int dx = cx == 3 ? 1 : -1, dy = cy == 3 ? 1 : -1;  // the further ones
    d.c = cls(cx, cy);
    d.m = cls(cx - dx, cy);
    d.x = cls(cx + dx, cy);
    d.r = cls(cx, cy - dy);
    d.y = cls(cx, cy + dy);
    d.qx = turn(x >> 2, g.Cx);  // an offset is below the size: at most one turn
    d.qy = turn(y >> 2, g.Cy);
    d.xs = shift(cx);
    const int ys = shift(cy);
    d.ys = ys < 0 ? g.Cy - 1 : ys < g.Cy ? ys : 0;
    d.offX = turn(d.qx + (d.xs < 0 ? g.Cx - 1 : d.xs), g.Cx);
  };
  side(u.side[0], sc.a0x, sc.a0y);
  side(u.side[1], sc.a0x + sc.rx, sc.a0y + sc.ry);
  u.near128 = sc.near ? 128u : 0u;
  return u;
}

// The words and shift of the window of 16 sites at column 16 w + off (mod Cx) of
// a row; n1: sites before the row's end (rows of whole words: never cut).
struct Win {
  int lo, hi;  // its two words
  int sh, n1;
};

template <bool kAl>
__device__ __forceinline__ Win window_at(const Geo &g, int w, int off) {
  Win x;
  if constexpr (kAl) {
    x.lo = turn(w + (off >> 4), g.W);
    x.sh = 2 * (off & 15);
    x.n1 = 16;
  } else {
    const int s = turn(16 * w + off, g.Cx);
    x.lo = s >> 4;
    x.sh = 2 * (s & 15);
    x.n1 = g.Cx - s;
  }
  x.hi = turn(x.lo + 1, g.W);
  return x;
}

// Move entry of choice class r (v mod 12) and r264 = 264 r + 128 near: entry
// (2 r + near) 16 + (pc XOR r) of the move table, at byte offset
// 256 r + 128 near + 8 (pc XOR r) = r264 XOR 8 pc.  The XOR spreads a warp's
// lookups over the banks: with entry (2 r + near) 16 + pc the bank pair of a
// lookup was its pair state alone, and the few common states (both sites
// magnetic) piled onto four of sixteen bank pairs.  Word 0: the level
// offset's base and, at bits 24-27, the move pc XOR npc; word 1: the signed byte
// coefficients of (2 n1_a, n0_a, 2 n1_b, n0_b).
__device__ __forceinline__ uint2 move_entry(const uint2 *trans, uint32_t off) {
  return *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(trans) + off);
}

// The threshold level at byte offset `off` (the offset is formed in bytes, so
// that it is the load's address without a shift).
__device__ __forceinline__ uint32_t level_at(const uint16_t *thrT, uint32_t off) {
  return *reinterpret_cast<const uint16_t *>(reinterpret_cast<const char *>(thrT) + off);
}

// floor(v / 12) for v < 2^16 by a multiply-high: floor(v m / 2^32) with
// m = ceil(2^32 / 12) is exact there.
__device__ __forceinline__ uint32_t div12(uint32_t v) { return __umulhi(v, 357913942u); }

// A pair's neighbour counts as dp4a's byte operands.  A word's pairs form four
// groups k (sites k, k + 4, k + 8, k + 12: one a byte); group k = 2 c + h is
// half h of MOVE call c.
constexpr uint32_t kEnvMask = 0x070E070Eu;  // 2 n1 at bits 1-3, n0 at bits 0-2 of a nibble

// The counts of half h's pairs of both calls: byte q of ev[q] .. is lane q's
// (2 n1_a, n0_a, 2 n1_b, n0_b), call 0 in the low nibbles, call 1 in the high
// ones (bits outside kEnvMask are whatever the planes hold there).  Two
// selections put a count's three bits side by side (its unwanted neighbours
// are masked with the nibble), then eight byte permutes transpose the four
// counts: 30 instructions for eight pairs, where masked additions, byte
// extraction per group and a permute per pair took about 70.
struct Env {
  uint32_t ev[4];
};

__device__ __forceinline__ Env half_env(const Planes &a, const Planes &b, int h) {
  // bits of half h's sites at the low two bits of every nibble
  const uint32_t m1 = 0x22222222u, m2 = 0x88888888u, m3 = 0x11111111u, m4 = 0x44444444u;
  const uint32_t aO = h ? a.O >> 2 : a.O, aT = h ? a.T >> 1 : a.T << 1,
                 aF = h ? a.F : a.F << 2;
  const uint32_t bO = h ? b.O >> 2 : b.O, bT = h ? b.T >> 1 : b.T << 1,
                 bF = h ? b.F : b.F << 2;
  const uint32_t a1 = lop3<kLutMux>(aF, lop3<kLutMux>(aO, aT, m1), m2);
  const uint32_t a0 = lop3<kLutMux>(aF, lop3<kLutMux>(aO, aT, m3), m4);
  const uint32_t b1 = lop3<kLutMux>(bF, lop3<kLutMux>(bO, bT, m1), m2);
  const uint32_t b0 = lop3<kLutMux>(bF, lop3<kLutMux>(bO, bT, m3), m4);
  const uint32_t x01 = prmt(a1, a0, 0x5140u), x23 = prmt(a1, a0, 0x7362u);
  const uint32_t y01 = prmt(b1, b0, 0x5140u), y23 = prmt(b1, b0, 0x7362u);
  return Env{{prmt(x01, y01, 0x5410u), prmt(x01, y01, 0x7632u), prmt(x23, y23, 0x5410u),
              prmt(x23, y23, 0x7632u)}};
}

// The inputs of a word's pairs: its a word, its b window and the neighbour
// counts of both sides.
struct WordIn {
  uint32_t A, B;
  Planes na, nb;
};

// The pair states pc (a's code above b's) of half h's pairs: lane q of call c at
// bits 8 q + 4 c .. + 3.
__device__ __forceinline__ uint32_t half_pc(uint32_t A, uint32_t B, int h) {
  return h ? lop3<kLutMux>(A, B >> 2, 0xCCCCCCCCu) : lop3<kLutMux>(A << 2, B, 0xCCCCCCCCu);
}

// 264 r + 128 near XOR 8 pc, the move entry's offset: the pair's pc at bits 3-6
// of pcs >> 8 q (of the half's pair states rotated left by 3 - 4 c).
__device__ __forceinline__ uint32_t entry_offset(uint32_t pcs, int q, uint32_t r264) {
  return lop3<kLutAndXor>(pcs >> (8 * q), 0x78u, r264);
}

// Pair t's own counts (dp4a's operand) and state (times 8), from bits 2 t and 2 t + 1
// of the word's planes and words.
__device__ __forceinline__ uint32_t pair_env(const WordIn &in, int t) {
  auto counts = [&](const Planes &p) {
    const uint32_t O = p.O >> (2 * t), T = p.T >> (2 * t), F = p.F >> (2 * t);
    return ((O & 2u) + 2u * (T & 2u) + 4u * (F & 2u)) |
           (((O & 1u) + 2u * (T & 1u) + 4u * (F & 1u)) << 8);
  };
  return counts(in.na) | (counts(in.nb) << 16);
}
__device__ __forceinline__ uint32_t pair_pc8(const WordIn &in, int t) {
  return ((((in.A >> (2 * t)) & 3u) << 2) | ((in.B >> (2 * t)) & 3u)) << 3;
}

// The exact decision against the full threshold of a pair with w = wq (5461: its choice
// class was drawn again) and SLOW word s.
__device__ __forceinline__ bool exact_accept(uint32_t thr, uint32_t wq, uint32_t s) {
  return thr == 0xFFFFFFFFu ||
         (wq != 5461u ? ((uint64_t)wq << 32) + s < 5461ull * thr : s < thr);
}

// The exact decision of pair t of word w of class row j, with its SLOW words, if it
// is rare (a tie or a field >= 65532, which the fast path rejected): the accepted
// move, else 0.
__device__ __forceinline__ uint32_t exact_move(const Geo &g, const uint2 *trans,
                                               const uint16_t *thrT, const uint32_t *thr32, int j,
                                               int w, int t, const WordIn &in, uint64_t P,
                                               uint32_t near128) {
  const int c = (t >> 1) & 1, h = t & 1, q = t >> 2;  // its MOVE call, half and word
  const uint32_t gbase = (uint32_t)j * (uint32_t)(2 * g.W) + (uint32_t)(2 * w);
  const U4 r = philox(gbase + (uint32_t)c, (uint32_t)P, (uint32_t)(P >> 32), TAG_MOVE, g.k0, g.k1);
  const uint32_t X = q == 0 ? r.x : q == 1 ? r.y : q == 2 ? r.z : r.w;
  const uint32_t v = h ? X >> 16 : X & 0xFFFFu;
  const uint32_t wq = div12(v);
  const uint32_t env = pair_env(in, t), pc8 = pair_pc8(in, t);
  uint2 e = move_entry(trans, ((v - 12u * wq) * 264u + near128) ^ pc8);
  if (v < 65532u && wq != level_at(thrT, (uint32_t)__dp4a((int)e.y, (int)env, (int)e.x) & 0xFFFFu))
    return 0u;  // not rare
  const uint32_t slow0 = (uint32_t)((uint64_t)j * g.Cx + (uint32_t)(w << 4));
  const U4 sl = philox(slow0 + (uint32_t)t, (uint32_t)P, (uint32_t)(P >> 32), TAG_SLOW, g.k0, g.k1);
  if (v >= 65532u) {
    if (sl.y >= 4294967292u) return 0u;  // keep the current configuration
    e = move_entry(trans, ((sl.y % 12u) * 264u + near128) ^ pc8);
  }
  const uint32_t thr = thr32[((uint32_t)__dp4a((int)e.y, (int)env, (int)e.x) & 0xFFFFu) >> 1];
  return exact_accept(thr, wq, sl.x) ? e.x >> 24 : 0u;
}

// The same of a pair known to be rare, with the random word X of its MOVE call at hand;
// slow0: the SLOW index of the word's pair 0, slow(i): the SLOW words of index i, which
// do not wait for the level and the exact threshold.  A resident phase waits for its
// slowest warp, and of a lattice of 256 words one has a rare pair in most phases: with
// exact_move there, 800 cycles, 1000^2 took 18.7 us a sweep, now 17.1.
template <class Slow>
__device__ __forceinline__ uint32_t rare_move(const uint2 *trans, const uint32_t *thr32, int t,
                                              const WordIn &in, uint32_t X, uint32_t slow0,
                                              uint32_t near128, const Slow &slow) {
  const uint32_t v = t & 1 ? X >> 16 : X & 0xFFFFu;
  const uint32_t wq = div12(v);
  const uint32_t env = pair_env(in, t), pc8 = pair_pc8(in, t);
  // (a field >= 65532 has v - 12 wq = 0 .. 3: an entry of the table, not the pair's)
  uint2 e = move_entry(trans, ((v - 12u * wq) * 264u + near128) ^ pc8);
  auto threshold = [&]() {
    return thr32[((uint32_t)__dp4a((int)e.y, (int)env, (int)e.x) & 0xFFFFu) >> 1];
  };
  uint32_t thr = threshold();
  const U4 sl = slow(slow0 + (uint32_t)t);
  if (v >= 65532u) {
    if (sl.y >= 4294967292u) return 0u;  // keep the current configuration
    e = move_entry(trans, ((sl.y % 12u) * 264u + near128) ^ pc8);
    thr = threshold();
  }
  return exact_accept(thr, wq, sl.x) ? e.x >> 24 : 0u;
}

// The exact decisions of a group's rare pairs (mask m of its lanes q, not empty), by
// the thread that holds the group: the accepted moves, byte q for lane q.  wq, t, ev:
// the lanes' w, level offset with the move in byte 3, and dp4a operand; pc: the pair
// states as entry_offset takes them; slow0: the SLOW index of lane 0, slow(i): the
// SLOW words of index i.  The threshold is on its way while the words are drawn.
template <class Slow>
__device__ __forceinline__ uint32_t exact_group(const uint2 *trans, const uint32_t *thr32,
                                                uint32_t m, const uint32_t (&wq)[4],
                                                const uint32_t (&t)[4], const uint32_t (&ev)[4],
                                                uint32_t pc, uint32_t near128, uint32_t slow0,
                                                const Slow &slow) {
  auto lane = [](const uint32_t (&x)[4], int q) {  // no indexing: the array stays in registers
    return q == 0 ? x[0] : q == 1 ? x[1] : q == 2 ? x[2] : x[3];
  };
  uint32_t acc = 0u;
#pragma unroll 1
  do {
    const int q = __ffs((int)m) - 1;
    m &= m - 1u;
    const uint32_t w = lane(wq, q);
    uint32_t tq = lane(t, q);
    uint32_t thr = thr32[(tq & 0xFFFFu) >> 1];
    const U4 sl = slow(slow0 + 4u * (uint32_t)q);
    const bool big = w == 5461u;  // a field >= 65532: the choice class drawn again
    if (big) {
      if (sl.y >= 4294967292u) continue;  // keep the current configuration
      const uint2 e = move_entry(trans, entry_offset(pc, q, (sl.y % 12u) * 264u + near128));
      tq = (uint32_t)__dp4a((int)e.y, (int)lane(ev, q), (int)e.x);
      thr = thr32[(tq & 0xFFFFu) >> 1];
    }
    if (exact_accept(thr, w, sl.x)) acc |= (tq >> 24) << (8 * q);
  } while (m);
  return acc;
}

// The fast path of the pairs of a word one thread evaluates: all 16 (kTPW 1), or with
// two threads a word (kTPW 2) the eight of MOVE call `sub`.  (Four lanes a word have a
// path of their own in the resident kernel.)
// rand(c): the four words of the word's MOVE call c.  Returns the (dA, dB) of the
// fast decisions and, in z, what needs the exact path (a tie or a field >= 65532,
// rejected here): bit t for every such pair t (kPairs), or bit c for every call c
// with one (fewer instructions, for a path that looks at the call's pairs anyway).  A
// call asks once for all its pairs: a branch for every four kept the groups of a call
// from being worked on together (1000^2: 0.1 us a phase).
template <int kTPW, bool kPairs, class Rand>
__device__ __forceinline__ uint3 fast_moves(const uint2 *trans, const uint16_t *thrT, int sub,
                                            const WordIn &in, uint32_t near128,
                                            const Rand &rand) {
  static_assert(kTPW == 1 || kTPW == 2, "one or two threads a word");
  constexpr int kCalls = kTPW == 1 ? 2 : 1;
  const int c0 = kTPW == 1 ? 0 : sub;
  Env env[2];
  uint32_t pcs[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    env[h] = half_env(in.na, in.nb, h);
    pcs[h] = half_pc(in.A, in.B, h);
  }
  uint32_t dA = 0u, dB = 0u, slow = 0u;
#pragma unroll
  for (int ci = 0; ci < kCalls; ++ci) {
    const int c = c0 + ci;
    const U4 r = rand(c);
    const uint32_t mx = __vmaxu2(__vimax3_u16x2(r.x, r.y, r.z), r.w);
    const bool big = mx >= 0xFFFC0000u || (mx & 0xFFFFu) >= 0xFFFCu;  // a field >= 65532
    uint32_t mn = 0xFFFFFFFFu;  // smallest w - T of the call
    uint32_t d[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 2 * c + h;
      uint32_t t[4];
      const uint32_t pc = __funnelshift_l(pcs[h], pcs[h], 3 - 4 * c);  // counts modulo 32
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t X = q == 0 ? r.x : q == 1 ? r.y : q == 2 ? r.z : r.w;
        const uint32_t v = (X >> (16 * h)) & 0xFFFFu;
        const uint32_t wq = div12(v);
        const uint2 e =
            move_entry(trans, entry_offset(pc, q, (v - 12u * wq) * 264u + near128));
        t[q] = (uint32_t)__dp4a((int)e.y, (int)((env[h].ev[q] >> (4 * c)) & kEnvMask), (int)e.x);
        d[h][q] = wq - level_at(thrT, t[q] & 0xFFFFu);  // negative: accept; zero: a tie
      }
      mn = __vimin3_u32(mn, d[h][0], d[h][1]);
      mn = __vimin3_u32(mn, d[h][2], d[h][3]);
      // byte q: the accepted move of lane q, i.e. byte 3 of t[q] under the sign
      // of d[q] (byte permutes: bit 3 of a selector replicates a byte's sign)
      const uint32_t acc =
          prmt(prmt(d[h][0], d[h][1], 0x00FBu), prmt(d[h][2], d[h][3], 0x00FBu), 0x5410u) &
          prmt(prmt(t[0], t[1], 0x0073u), prmt(t[2], t[3], 0x0073u), 0x5410u);
      // byte q of acc -> site k + 4 q: b bits to 2 (k + 4 q) of dB, a bits of dA
      dB |= (acc & 0x03030303u) << (2 * k);
      dA |= ((acc >> 2) & 0x03030303u) << (2 * k);
    }
    if (mn == 0u || big) {
      if constexpr (kPairs) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t X = q == 0 ? r.x : q == 1 ? r.y : q == 2 ? r.z : r.w;
            if (d[h][q] == 0u || ((X >> (16 * h)) & 0xFFFFu) >= 65532u)
              slow |= 1u << (2 * c + h + 4 * q);
          }
      } else {
        slow |= 1u << c;
      }
    }
  }
  return make_uint3(dA, dB, slow);
}

}  // namespace ccmc
