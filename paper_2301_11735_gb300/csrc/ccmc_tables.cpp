// ccmc_tables.cpp -- host-side parameter tables of the sweep.  Compiled with
// -ffp-contract=off so every FP64 operation rounds in the order written.
#include <cmath>
#include <cstdint>

#include "ccmc_internal.h"

namespace ccmc {

namespace {
// Site values of the four codes (Sec. 2.1): S, and sigma = 2 (1 - S^2) s.
constexpr int kS[4] = {0, 0, 1, -1};
constexpr int kSigma[4] = {1, -1, 0, 0};

// Metropolis acceptance threshold of an energy change (Sec. 3.1): the move is
// accepted iff the threshold is 0xFFFFFFFF or a uniform 32-bit word lies below
// it, i.e. with probability min(1, exp(-beta dE)) to within 2^-32.
uint32_t threshold(double beta, double Delta, double V, double J, int dQ, int dBV, int dBJ) {
  const double eQ = Delta * static_cast<double>(dQ);
  const double eV = V * static_cast<double>(dBV);
  const double eQV = eQ + eV;
  const double quarterJ = 0.25 * J;
  const double eJ = quarterJ * static_cast<double>(dBJ);
  const double dE = eQV + eJ;  // Eq. (3): Delta dQ + V dBV + (J/4) dBJ
  if (dE <= 0.0) return 0xFFFFFFFFu;
  const double p = std::exp(-beta * dE);
  if (p >= 1.0) return 0xFFFFFFFFu;
  const double scaled = std::floor(std::ldexp(p, 32));
  if (scaled >= 4294967295.0) return 0xFFFFFFFEu;
  return static_cast<uint32_t>(scaled);
}
}  // namespace

void build_thresholds(double beta, double Delta, double V, double J, uint32_t *thr32) {
  for (int dqi = 0; dqi < 3; ++dqi)
    for (int dBV = -kDB; dBV <= kDB; ++dBV)
      for (int dBJ = -kDB; dBJ <= kDB; ++dBJ)
        thr32[(dqi * kNB + dBV + kDB) * kNB + dBJ + kDB] =
            threshold(beta, Delta, V, J, 2 * dqi - 2, dBV, dBJ);
}

void build_device_thresholds(double beta, double Delta, double V, double J, uint32_t *thr32) {
  for (int dqi = 0; dqi < 3; ++dqi)
    for (int dBV = -kSegR; dBV <= kSegR; ++dBV)
      for (int dBJ = -kSegR; dBJ <= kSegR; ++dBJ)
        thr32[(dqi * kSegW + dBV + kSegR) * kSegW + dBJ + kSegR] =
            threshold(beta, Delta, V, J, 2 * dqi - 2, dBV, dBJ);
  for (int d = -kDB; d <= kDB; ++d) {
    thr32[kSegSwap + d + kDB] = threshold(beta, Delta, V, J, 0, d, 0);
    thr32[kSegFlip + d + kDB] = threshold(beta, Delta, V, J, 0, 0, d);
  }
}

// Move entries (see the phase kernel).  For choice class r = v mod 12, kind
// near (the partner is a nearest neighbour) and pair state pc = 4 a + b, the
// proposed state is the (r mod |set|)-th configuration of the pair's q-set in
// the paper's order (Sec. 3.1); frozen pairs (|q| = 2) propose themselves.  dE
// of the move:
//   dBV = dS_a sum_<a> S + dS_b sum_<b> S + m dS_a dS_b
//   dBJ = dsig_a sum_<a> sigma + dsig_b sum_<b> sigma + m dsig_a dsig_b
// with neighbour sums over old states (partner included) and m = near the number
// of a-b bonds.  With n1, n0 the numbers of a site's neighbours whose linear
// code has bit 1, bit 0 set, sum S = n1 - n0 and sum sigma = 4 - n1 - n0.  As
// dS_b = -dS_a, the byte offset of the move's 16-bit level, twice its index in
// its segment's strides (sS entries a unit of dBV, sG a unit of dBJ), is an
// affine function of 2 n1 and n0 of both sides:
//   offset = base + (sS dS_a - sG dsig_a) 2 n1_a - 2 (sS dS_a + sG dsig_a) n0_a
//                 + (sS dS_b - sG dsig_b) 2 n1_b - 2 (sS dS_b + sG dsig_b) n0_b.
// Entry (2 r + near) * 16 + (pc XOR r), pc the pair's two linear codes: word 0
// holds base in its low half and, in bits 24-27, the move pc XOR npc (both
// survive the sum, whose value stays below 2^16); word 1 the four signed byte
// coefficients.
namespace {
constexpr int kLinear[4] = {0, 3, 2, 1};  // a site code's linear form (ccmc_device.cuh)
constexpr int kSetN[3] = {4, 6, 4};  // q = +1, 0, -1
constexpr int kSets[3][6][2] = {
    {{2, 0}, {2, 1}, {0, 2}, {1, 2}, {0, 0}, {0, 0}},  // q = +1
    {{2, 3}, {3, 2}, {0, 0}, {1, 1}, {0, 1}, {1, 0}},  // q = 0
    {{3, 0}, {3, 1}, {0, 3}, {1, 3}, {0, 0}, {0, 0}},  // q = -1
};
}  // namespace

bool build_transitions(uint32_t *trans) {
  bool ok = true;
  for (int codes = 0; codes < 16; ++codes) {
    const int ca = codes >> 2, cb = codes & 3;
    const int pc = (kLinear[ca] << 2) | kLinear[cb];
    const int q = kS[ca] + kS[cb];
    for (int r = 0; r < 12; ++r) {
      int na = ca, nb = cb;
      if (q >= -1 && q <= 1) {
        const int qi = 1 - q;
        na = kSets[qi][r % kSetN[qi]][0];
        nb = kSets[qi][r % kSetN[qi]][1];
      }
      const int dQ = kS[na] * kS[na] + kS[nb] * kS[nb] - kS[ca] * kS[ca] - kS[cb] * kS[cb];
      const int dSa = kS[na] - kS[ca], dSb = kS[nb] - kS[cb];
      const int dGa = kSigma[na] - kSigma[ca], dGb = kSigma[nb] - kSigma[cb];
      // the move's segment: entries a unit of dBV and of dBJ, the entry of dBV =
      // dBJ = 0, the segment's first entry and its end
      const int kind = dSa == 0 ? 2 : (dSa == 1 || dSa == -1) ? 0 : 1;
      const int sS = kind == 0 ? kSegW : kind == 1 ? 1 : 0, sG = kind == 1 ? 0 : 1;
      const int first = kind == 0 ? (dQ + 2) / 2 * kSegW * kSegW : kind == 1 ? kSegSwap : kSegFlip;
      const int end = first + (kind == 0 ? kSegW * kSegW : kNB);
      const int zero = first + (kind == 0 ? kSegR * kSegW + kSegR : kDB);
      const int cA1 = sS * dSa - sG * dGa, cA0 = -2 * (sS * dSa + sG * dGa);
      const int cB1 = sS * dSb - sG * dGb, cB0 = -2 * (sS * dSb + sG * dGb);
      const int base = 2 * zero + 8 * sG * (dGa + dGb);
      const uint32_t x = (uint32_t)(pc ^ ((kLinear[na] << 2) | kLinear[nb]));
      const uint32_t coef = ((uint32_t)cA1 & 0xFFu) | (((uint32_t)cA0 & 0xFFu) << 8) |
                            (((uint32_t)cB1 & 0xFFu) << 16) | ((uint32_t)cB0 << 24);
      for (int near = 0; near < 2; ++near) {
        const int e = (2 * r + near) * 16 + (pc ^ r);  // bank-spread (see the phase kernel)
        const int b = base + near * 2 * (sS * dSa * dSb + sG * dGa * dGb);
        trans[2 * e] = (uint32_t)b + (x << 24);
        trans[2 * e + 1] = coef;
        // every offset the entry can form, over all neighbour counts (linear in
        // them: the corners), and both its energy terms, stay inside the segment
        for (int c = 0; c < 16; ++c) {
          const int a1 = c & 1 ? 4 : 0, a0 = c & 2 ? 4 : 0, b1 = c & 4 ? 4 : 0, b0 = c & 8 ? 4 : 0;
          const int off = b + 2 * cA1 * a1 + cA0 * a0 + 2 * cB1 * b1 + cB0 * b0;
          const int dBV = dSa * (a1 - a0) + dSb * (b1 - b0) + near * dSa * dSb;
          const int dBJ = dGa * (4 - a1 - a0) + dGb * (4 - b1 - b0) + near * dGa * dGb;
          const int reach = kind == 0 ? kSegR : kDB;
          ok = ok && off == 2 * (zero + sS * dBV + sG * dBJ);
          ok = ok && off >= 2 * first && off < 2 * end && (kind == 0 || dQ == 0);
          ok = ok && (kind == 1 ? dGa == 0 && dGb == 0 : dBJ >= -reach && dBJ <= reach);
          ok = ok && (kind == 2 ? dSb == 0 : dBV >= -reach && dBV <= reach);
        }
      }
    }
  }
  return ok;
}

}  // namespace ccmc
