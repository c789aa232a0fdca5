// ccmc_count.cuh -- observables of a packed lattice by definition (Eq. 3 and
// Eq. 2) as sums over bit products.  In the linear code S = b1 - b0 and sigma = 1 -
// b1 - b0, so with `like` the bonds' products b1 b1' + b0 b0' and `unlike` b1 b0' +
// b0 b1', summed over all 2N right and down bonds,
//   BV = like - unlike,
//   BJ = 2N - 4 (b1 + b0) + like + unlike   (every site has four bond ends),
// and Nc = b1 + b0 - 2 both, M = N - b1 - b0, S = b1 - b0 from the sites' sums; the
// staggered ones from the sums over the sites of even x + y (half of all).
// Used by the recount kernel; the resident kernel counts the same sums.
#pragma once

#include <cstdint>

#include "ccmc_device.cuh"
#include "ccmc_internal.h"

namespace ccmc {

// like, unlike, b1, b0, both, and b1, b0 over the sites of even x + y.
constexpr int kSums = 7;

// The observables Nc, BV, BJ, M, M_stag, S_sum, S_stag of the lattice's sums.
__device__ __forceinline__ void observables_of(const Geo &g, const int64_t s[kSums],
                                               int64_t obs[7]) {
  const int64_t N = (int64_t)g.Lx * g.Ly;
  const int64_t like = s[0], unlike = s[1], b1 = s[2], b0 = s[3], both = s[4];
  const int64_t d1 = 2 * s[5] - b1, d0 = 2 * s[6] - b0;  // even minus odd sites
  obs[0] = b1 + b0 - 2 * both;
  obs[1] = like - unlike;
  obs[2] = 2 * N - 4 * (b1 + b0) + like + unlike;
  obs[3] = N - b1 - b0;
  obs[4] = -d1 - d0;
  obs[5] = b1 - b0;
  obs[6] = d1 - d0;
}

// Bits b1 and b0 of every site exchanged.
__device__ __forceinline__ uint32_t swapped(uint32_t X) {
  return lop3<kLutMux>(X << 1, X >> 1, 0xAAAAAAAAu);
}

// Adds the sums of words tid, tid + nthreads, ... of class `cls`, any row width
// (bits above a row's end are zero in the words).
__device__ __forceinline__ void count_class(const Geo &g, int cls, int tid, int nthreads,
                                            int s[kSums]) {
  const int W = g.W, nw = g.Cy * W;
  const int cx = cls & 3, cy = cls >> 2;
  const uint32_t *X0 = g.words + (int64_t)cls * g.cstride;
  const uint32_t *R0 = g.words + (int64_t)(cy * 4 + ((cx + 1) & 3)) * g.cstride;
  const uint32_t *D0 = g.words + (int64_t)(((cy + 1) & 3) * 4 + cx) * g.cstride;
  int wid = tid;
  int j = wid / W, w = wid - j * W;
  const int sj = nthreads / W, sw = nthreads - sj * W;
  int k1 = 0, k0 = 0;
  for (; wid < nw; wid += nthreads) {
    const int s0 = w << 4;
    const uint32_t X = X0[wid], Xs = swapped(X);
    const uint32_t Yr = fetch_window(R0 + j * W, W, g.Cx,
                                     cx == 3 ? (s0 + 1 == g.Cx ? 0 : s0 + 1) : s0,
                                     min(16, g.Cx - s0));
    const int jd = cy == 3 ? (j + 1 == g.Cy ? 0 : j + 1) : j;
    const uint32_t Yd = D0[jd * W + w];
    s[0] += __popc(X & Yr) + __popc(X & Yd);
    s[1] += __popc(Xs & Yr) + __popc(Xs & Yd);
    k1 += __popc(X & 0xAAAAAAAAu);
    k0 += __popc(X & 0x55555555u);
    s[4] += __popc(X & Xs & 0xAAAAAAAAu);
    w += sw;
    j += sj;
    if (w >= W) {
      w -= W;
      ++j;
    }
  }
  s[2] += k1;
  s[3] += k0;
  if (!((cx + cy) & 1)) {
    s[5] += k1;
    s[6] += k0;
  }
}

// The quad path: rows of whole words (Cx a multiple of 16) with W a multiple of 4.
// A thread takes four consecutive words of the four classes of a row of sites at
// once with 16-byte loads: the classes are each other's right neighbours, so eight
// loads (and one word across the quad's end) serve sixteen words, 8.25 bytes a word
// where a class at a time took 12.  The logic pipe and the population counts (a
// quarter of its rate) share the work: a half adder joins a word's two bonds, a full
// adder three words, and two classes share the site counts: 4 counts and 15 logic
// instructions a word.

// The bond products of four words against their right and down windows.
__device__ __forceinline__ int bond_count(const uint32_t X[4], const uint32_t R[4],
                                          const uint32_t D[4]) {
  constexpr uint32_t kLutAndXor2 = 0x60;  // a & (b ^ c)
  uint32_t s[4], c[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    s[k] = lop3<kLutAndXor2>(X[k], R[k], D[k]);
    c[k] = lop3<kLutAnd3>(X[k], R[k], D[k]);
  }
  const uint32_t s1 = lop3<kLutXor3>(s[0], s[1], s[2]), t0 = lop3<kLutMaj>(s[0], s[1], s[2]);
  const uint32_t t1 = lop3<kLutXor3>(t0, c[0], c[1]), f0 = lop3<kLutMaj>(t0, c[0], c[1]);
  const uint32_t t2 = lop3<kLutXor3>(t1, c[2], c[3]), f1 = lop3<kLutMaj>(t1, c[2], c[3]);
  return __popc(s1) + __popc(s[3]) + 2 * __popc(t2) + 4 * (__popc(f0) + __popc(f1));
}

__device__ __forceinline__ void count_quads(const Geo &g, int cy, int q, int nthreads,
                                            int s[kSums]) {
  constexpr uint32_t kOdd = 0xAAAAAAAAu;
  const int W = g.W, Wq = W >> 2, nq = g.Cy * Wq, last_row = (g.Cy - 1) * Wq;
  const uint32_t *own = g.words + (int64_t)(4 * cy) * g.cstride;
  const uint32_t *below = g.words + (int64_t)(4 * ((cy + 1) & 3)) * g.cstride;
  int wq = q % Wq;
  const int sw = nthreads % Wq;
  for (; q < nq; q += nthreads) {
    const int o = 4 * q;  // word offset of the quad: row j, column 4 wq
    // the down neighbours of class row 3 lie one class row further down
    const int od = cy < 3 ? o : q < last_row ? o + W : o - last_row * 4;
    uint4 x[4], d[4];
#pragma unroll
    for (int cx = 0; cx < 4; ++cx) {
      x[cx] = *reinterpret_cast<const uint4 *>(own + cx * g.cstride + o);
      d[cx] = *reinterpret_cast<const uint4 *>(below + cx * g.cstride + od);
    }
    const uint32_t next = own[wq == Wq - 1 ? o + 4 - W : o + 4];
    wq += sw;
    if (wq >= Wq) wq -= Wq;
    uint32_t X[4][4], B[4][4];
#pragma unroll
    for (int cx = 0; cx < 4; ++cx) {
      X[cx][0] = x[cx].x;
      X[cx][1] = x[cx].y;
      X[cx][2] = x[cx].z;
      X[cx][3] = x[cx].w;
    }
#pragma unroll
    for (int cx = 0; cx < 4; ++cx) {
      const uint32_t D[4] = {d[cx].x, d[cx].y, d[cx].z, d[cx].w};
      uint32_t R[4], Xs[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // the last class's right neighbours: the first class one site further
        R[k] = cx < 3 ? X[(cx + 1) & 3][k]
                      : __funnelshift_r(X[0][k], k < 3 ? X[0][(k + 1) & 3] : next, 2);
        Xs[k] = swapped(X[cx][k]);
        B[cx][k] = X[cx][k] & Xs[k];
      }
      s[0] += bond_count(X[cx], R, D);
      s[1] += bond_count(Xs, R, D);
    }
    int b1[2] = {0, 0}, b0[2] = {0, 0};
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        b1[h] += __popc(lop3<kLutMux>(X[h][k], X[h + 2][k] >> 1, kOdd));
        b0[h] += __popc(lop3<kLutMux>(X[h][k] << 1, X[h + 2][k], kOdd));
        s[4] += __popc(lop3<kLutMux>(B[h][k], B[h + 2][k], kOdd));
      }
    s[2] += b1[0] + b1[1];
    s[3] += b0[0] + b0[1];
    s[5] += cy & 1 ? b1[1] : b1[0];
    s[6] += cy & 1 ? b0[1] : b0[0];
  }
}

__host__ __device__ inline bool quads_ok(const Geo &g) {
  return (g.Cx & 15) == 0 && (g.W & 3) == 0;
}

}  // namespace ccmc
