// ccmc_kernels.cu -- the CUDA kernels around the colour phases for sm_103a
// (initial state, observables recount, phase counter, state packing, Philox
// export) and their launchers (declared in ccmc_internal.h).  The phase
// kernels are in ccmc_phase.cu.
#include <cuda_runtime.h>

#include <cstdint>

#include "ccmc_count.cuh"
#include "ccmc_device.cuh"
#include "ccmc_fault.h"
#include "ccmc_internal.h"
#include "ccmc_launch.cuh"
#include "ccmc_state.h"

namespace ccmc {

// ============================================================================
// Initial state (Sec. 3.1, stage 1): exactly N+ sites S=+1 and N- sites S=-1.
// Site index i = y Lx + x gets rank pi(i) under a seeded four-round Feistel
// permutation of [0, 4^h) with cycle-walking into [0, N); rank < N+ -> S=+1,
// rank < N+ + N- -> S=-1, else magnetic with sign bit i of the SIGN stream.
__device__ __forceinline__ uint64_t feistel_round_trip(uint32_t k0, uint32_t k1, int h,
                                                       uint64_t x) {
  const uint64_t mask = ((uint64_t)1 << h) - 1;
  uint64_t L = x >> h, R = x & mask;
#pragma unroll
  for (uint32_t round = 0; round < 4; ++round) {
    const U4 w = philox((uint32_t)R, round, 0u, TAG_FEISTEL, k0, k1);
    const uint64_t nR = L ^ ((uint64_t)w.x & mask);
    L = R;
    R = nR;
  }
  return (L << h) | R;
}

__global__ void init_kernel(Geo g, int h, int64_t n_plus, int64_t n_minus) {
  const int64_t nwords = 16 * g.cstride;
  const uint64_t N = (uint64_t)g.Lx * (uint64_t)g.Ly;
  for (int64_t wid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; wid < nwords;
       wid += (int64_t)gridDim.x * blockDim.x) {
    const int cls = (int)(wid / g.cstride);
    const int64_t rem = wid - (int64_t)cls * g.cstride;
    const int j = (int)(rem / g.W), w = (int)(rem - (int64_t)j * g.W);
    const int cx = cls & 3, cy = cls >> 2;
    const int s0 = w << 4;
    const int n = min(16, g.Cx - s0);
    uint32_t word = 0;
    for (int t = 0; t < n; ++t) {
      const int x = 4 * (s0 + t) + cx, y = 4 * j + cy;
      const uint64_t site = (uint64_t)y * g.Lx + x;
      uint64_t r = feistel_round_trip(g.k0, g.k1, h, site);
      while (r >= N) r = feistel_round_trip(g.k0, g.k1, h, r);
      uint32_t code;
      if ((int64_t)r < n_plus) {
        code = 2u;
      } else if ((int64_t)r < n_plus + n_minus) {
        code = 3u;
      } else {
        const U4 sw = philox((uint32_t)(site >> 7), 0u, 0u, TAG_SIGN, g.k0, g.k1);
        const uint32_t q = (uint32_t)(site >> 5) & 3u;
        const uint32_t bits = q == 0 ? sw.x : q == 1 ? sw.y : q == 2 ? sw.z : sw.w;
        code = (bits >> (site & 31u)) & 1u;
      }
      word |= code << (2 * t);
    }
    g.words[wid] = linear_code(word);
  }
}

// ============================================================================
// Recount (Eq. 3 and Eq. 2 by definition): sums of bit products of the class words
// against their right and down neighbour windows (ccmc_count.cuh).  Block
// partials go to scratch; the last block to arrive sums them into a record,
// appends it to the ring and the histograms, and re-arms the ticket.
struct RecountArgs {
  int64_t *partials;    // (gridDim.x * gridDim.y) x 7 scratch
  int64_t *ring;        // cap x 8 records (nullptr: latest only)
  int64_t ring_cap;
  int64_t *hist;        // 3 x nbins (nullptr: none)
  int nbins;
  int64_t sweep_off;    // sweeps_done = phase_base / 8 + sweep_off
};

// Grid (gx, 4): grid row y counts the classes of site rows y mod 4; or (gx, 16),
// class y, for rows that are not whole quads of words.
__global__ void __launch_bounds__(1024, 1) recount_kernel(Geo g, RecountArgs a) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  int c[kSums] = {0, 0, 0, 0, 0, 0, 0};
  if (quads_ok(g))
    count_quads(g, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, c);
  else
    count_class(g, blockIdx.y, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, c);
  const unsigned nblocks = gridDim.x * gridDim.y;
  const unsigned bid = blockIdx.y * gridDim.x + blockIdx.x;
  constexpr int kRuns = 256 / kSums;  // threads that share a sum in the last block
  __shared__ int64_t red[kRuns][kSums];
  __shared__ bool last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kSums; ++k) {  // a warp counts below 2^31
    const int v = __reduce_add_sync(0xFFFFFFFFu, c[k]);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kSums) {
    int64_t v = 0;
    for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) v += red[wv][threadIdx.x];
    a.partials[bid * kSums + threadIdx.x] = v;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long prev =
        atomicAdd(reinterpret_cast<unsigned long long *>(g.ctl + kCtlTicket), 1ull);
    last = (prev == (unsigned long long)(nblocks - 1));
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // The last block's end is what the next phase waits for: consecutive threads read
  // consecutive partials (L2 loads: other blocks wrote them), then one warp writes the
  // record, a lane a word, and the three bins side by side.
  const int64_t base = g.ctl[kCtlPhaseBase], cnt = g.ctl[kCtlObsCount];
  if (threadIdx.x < kRuns * kSums) {
    int64_t v = 0;
#pragma unroll 8
    for (unsigned b = threadIdx.x; b < nblocks * kSums; b += kRuns * kSums)
      v += __ldcg(a.partials + b);
    red[threadIdx.x / kSums][threadIdx.x % kSums] = v;
  }
  __syncthreads();
  if (warp != 0) return;
  int64_t x = 0;
  if (lane < kSums) {
#pragma unroll
    for (int r = 0; r < kRuns; ++r) x += red[r][lane];
  }
  int64_t sums[kSums], rec[8];
#pragma unroll
  for (int k = 0; k < kSums; ++k) sums[k] = __shfl_sync(0xFFFFFFFFu, x, k);
  rec[0] = base / 8 + a.sweep_off;
  observables_of(g, sums, rec + 1);
  int64_t mine = rec[0];  // lane k: word k
#pragma unroll
  for (int k = 1; k < 8; ++k) mine = lane == k ? rec[k] : mine;
  if (lane < 8) g.ctl[kCtlLatest + lane] = mine;
  if (a.ring) {
    if (lane < 8) a.ring[(cnt % a.ring_cap) * 8 + lane] = mine;
    if (lane == 0) g.ctl[kCtlObsCount] = cnt + 1;
    if (a.hist && (lane == 4 || lane == 5 || lane == 7)) {  // M, M_stag, S_stag
      const int64_t N = (int64_t)g.Lx * g.Ly;
      const int64_t bin = (mine + N) * a.nbins / (2 * N + 1);
      a.hist[(lane == 7 ? 2 : lane - 4) * a.nbins + bin] += 1;
    }
  }
  if (lane == 0) g.ctl[kCtlTicket] = 0;
}

// ============================================================================
__global__ void advance_kernel(int64_t *ctl, int64_t phases) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  ctl[kCtlPhaseBase] += phases;
}

// The status words of n lattices side by side (for one copy to the host).
__global__ void gather_status_kernel(int64_t *const *ctls, int n, int64_t *out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = ctls[i][kCtlStatus];
}

cudaError_t launch_gather_status(int64_t *const *ctls, int n, int64_t *out, cudaStream_t s) {
  gather_status_kernel<<<grid_for(n, 256, 152), 256, 0, s>>>(ctls, n, out);
  return cudaGetLastError();
}

// Self-test of the bounded device waits: one CTA waits on an mbarrier that
// nothing completes, polling at most `polls` times, then records the timeout in
// *status and returns, so that the context stays usable.  (The sweep kernels wait
// only at hardware barriers of their own block or cluster, and on their predecessor.)
__global__ void wait_selftest_kernel(uint32_t polls, int *status) {
  __shared__ __align__(8) unsigned long long bar;
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(&bar);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(a));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool done = false;
  for (uint32_t i = 0; i < polls && !done; ++i) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(a)
        : "memory");
    done = r != 0;
  }
  if (!done && threadIdx.x == 0) *status = 1;
}

cudaError_t launch_wait_selftest(uint32_t polls, int *status, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(polls, status);
  return cudaGetLastError();
}

__global__ void set_ctl_kernel(int64_t *ctl, int64_t phase_base) {
  for (int k = threadIdx.x; k < kCtlWords; k += blockDim.x) ctl[k] = 0;
  __syncthreads();
  if (threadIdx.x == 0) ctl[kCtlPhaseBase] = phase_base;
}

// Logical bytes (site y Lx + x) <-> packed class words.  The four classes of a
// row of sites hold its sites in turn, so byte q of their four words of column
// block w is 16 consecutive bytes of the row: one thread per such group, the four
// words' bytes side by side in B (class cx at byte cx), site 4 i + cx of the group
// at bits 2 i of byte cx.  Memory-bound: 16-byte accesses on the byte side (4-byte
// ones on rows that are no multiple of 16), consecutive threads consecutive
// groups.  A thread a class word, with 16 byte accesses 4 bytes apart, moved
// every sector of the byte side four times (4096^2: see the launch list).
struct ByteGroup {
  int64_t word;  // of class cx = 0
  int64_t byte;  // of the group's first site
  int q, sites;  // byte of the words; sites of each class in the row (0 to 4)
};

__device__ __forceinline__ ByteGroup byte_group(const Geo &g, int64_t id) {
  const int64_t wid = id >> 2;
  const int w = (int)(wid % g.W);
  const int64_t r = wid / g.W;  // r = cy Cy + j
  const int cy = (int)(r / g.Cy), j = (int)(r - (int64_t)cy * g.Cy);
  ByteGroup b;
  b.q = (int)(id & 3);
  b.word = (int64_t)(cy * 4) * g.cstride + (int64_t)j * g.W + w;
  b.byte = (int64_t)(4 * j + cy) * g.Lx + 64 * w + 16 * b.q;
  b.sites = max(0, min(4, g.Cx - 16 * w - 4 * b.q));
  return b;
}

__global__ void unpack_kernel(Geo g, uint8_t *out) {
  const int64_t n = 16 * (int64_t)g.Cy * g.W;  // 4 rows a class row, 4 groups a word
  const bool vec = (g.Lx & 15) == 0;
  for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < n;
       id += (int64_t)gridDim.x * blockDim.x) {
    const ByteGroup b = byte_group(g, id);
    uint32_t B = 0u;
#pragma unroll
    for (int cx = 0; cx < 4; ++cx)
      B |= ((g.words[b.word + cx * g.cstride] >> (8 * b.q)) & 0xFFu) << (8 * cx);
    B = linear_code(B);
    uint32_t v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = (B >> (2 * i)) & 0x03030303u;
    if (vec && b.sites == 4) {
      *reinterpret_cast<uint4 *>(out + b.byte) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < b.sites) *reinterpret_cast<uint32_t *>(out + b.byte + 4 * i) = v[i];
    }
  }
}

__global__ void pack_kernel(Geo g, const uint8_t *in, int *bad) {
  const int64_t n = 16 * (int64_t)g.Cy * g.W;
  const bool vec = (g.Lx & 15) == 0;
  for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < n;
       id += (int64_t)gridDim.x * blockDim.x) {
    const ByteGroup b = byte_group(g, id);
    uint32_t v[4] = {0u, 0u, 0u, 0u};
    if (vec && b.sites == 4) {
      const uint4 x = *reinterpret_cast<const uint4 *>(in + b.byte);
      v[0] = x.x;
      v[1] = x.y;
      v[2] = x.z;
      v[3] = x.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < b.sites) v[i] = *reinterpret_cast<const uint32_t *>(in + b.byte + 4 * i);
    }
    if ((v[0] | v[1] | v[2] | v[3]) & 0xFCFCFCFCu) *bad = 1;
    uint32_t B = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) B |= (v[i] & 0x03030303u) << (2 * i);
    B = linear_code(B);
    uint8_t *words = reinterpret_cast<uint8_t *>(g.words);
#pragma unroll
    for (int cx = 0; cx < 4; ++cx)
      words[4 * (b.word + cx * g.cstride) + b.q] = (uint8_t)(B >> (8 * cx));
  }
}

// Compact row-major state, 2 bits a site: site i = y Lx + x at bits 2 (i mod
// 4) of byte i / 4.  As Lx is a multiple of 4, byte i of row y holds column i of
// the four classes (cx = 0..3) of class row y / 4, y mod 4: one thread builds
// (or splits) the four class words of column block w from 16 consecutive bytes.
__device__ __forceinline__ uint32_t gather_field(uint32_t q, int cx) {
  // the cx-th 2-bit field of each of q's four bytes, packed into 8 bits
  uint32_t x = (q >> (2 * cx)) & 0x03030303u;
  x = (x | (x >> 6)) & 0x000F000Fu;
  return (x | (x >> 12)) & 0xFFu;
}

__device__ __forceinline__ uint32_t scatter_field(uint32_t f, int cx) {
  // inverse of gather_field: 8 bits -> the cx-th field of four bytes
  uint32_t x = (f | (f << 12)) & 0x000F000Fu;
  x = (x | (x << 6)) & 0x03030303u;
  return x << (2 * cx);
}

__global__ void pack2_kernel(Geo g, const uint8_t *in) {
  const int64_t nthr = 4 * (int64_t)g.Cy * g.W;
  const int64_t row_bytes = g.Lx / 4;
  const bool vec = (row_bytes & 15) == 0;
  for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < nthr;
       id += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(id % g.W);
    const int64_t r = id / g.W;  // r = cy Cy + j
    const int cy = (int)(r / g.Cy), j = (int)(r - (int64_t)cy * g.Cy);
    const uint8_t *src = in + (int64_t)(4 * j + cy) * row_bytes + 16 * w;
    const int n = min(16, g.Cx - 16 * w);
    uint32_t q[4] = {0u, 0u, 0u, 0u};
    if (vec) {
      const uint4 v = *reinterpret_cast<const uint4 *>(src);
      q[0] = v.x;
      q[1] = v.y;
      q[2] = v.z;
      q[3] = v.w;
    } else {
      for (int t = 0; t < n; ++t) q[t >> 2] |= (uint32_t)src[t] << (8 * (t & 3));
    }
#pragma unroll
    for (int cx = 0; cx < 4; ++cx) {
      uint32_t word = 0u;
#pragma unroll
      for (int k = 0; k < 4; ++k) word |= gather_field(q[k], cx) << (8 * k);
      g.words[(int64_t)(cy * 4 + cx) * g.cstride + (int64_t)j * g.W + w] = linear_code(word);
    }
  }
}

__global__ void unpack2_kernel(Geo g, uint8_t *out) {
  const int64_t nthr = 4 * (int64_t)g.Cy * g.W;
  const int64_t row_bytes = g.Lx / 4;
  const bool vec = (row_bytes & 15) == 0;
  for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < nthr;
       id += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(id % g.W);
    const int64_t r = id / g.W;
    const int cy = (int)(r / g.Cy), j = (int)(r - (int64_t)cy * g.Cy);
    uint8_t *dst = out + (int64_t)(4 * j + cy) * row_bytes + 16 * w;
    const int n = min(16, g.Cx - 16 * w);
    uint32_t q[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int cx = 0; cx < 4; ++cx) {
      const uint32_t word =
          linear_code(g.words[(int64_t)(cy * 4 + cx) * g.cstride + (int64_t)j * g.W + w]);
#pragma unroll
      for (int k = 0; k < 4; ++k) q[k] |= scatter_field((word >> (8 * k)) & 0xFFu, cx);
    }
    if (vec) {
      *reinterpret_cast<uint4 *>(dst) = make_uint4(q[0], q[1], q[2], q[3]);
    } else {
      for (int t = 0; t < n; ++t) dst[t] = (uint8_t)(q[t >> 2] >> (8 * (t & 3)));
    }
  }
}

__global__ void philox_kernel(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                              uint32_t k1, int64_t count, uint32_t *out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const U4 r = philox(c0 + (uint32_t)i, c1, c2, c3, k0, k1);
    out[4 * i + 0] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
  }
}

// ============================================================================
// Launchers.
cudaError_t launch_init(const Geo &g, int h, int64_t n_plus, int64_t n_minus, cudaStream_t s) {
  init_kernel<<<grid_for(16 * g.cstride, 256, 152 * 16), 256, 0, s>>>(g, h, n_plus, n_minus);
  return cudaGetLastError();
}

// Launch of recount_kernel: one wave of 1024 threads an SM (64 registers).  A thread's
// unit is a word, or a quad of words of four classes.  A block's end (its sums, its
// fence and ticket) costs what a block of 256 counts in 4 us, so a wave that is full of
// work takes one block an SM (16384^2: 26.6 us a recount with four, 24.7; 8192^2 13.8,
// 11.1) and one that is not takes small blocks, for more SMs (4096^2: 7.5 us, 14.2 with
// blocks of 1024).  Rows that are not whole quads: four blocks an SM.
struct RecountShape {
  dim3 grid;
  int block;
};
static RecountShape recount_shape(const Geo &g) {
  const int64_t words = (int64_t)g.Cy * g.W;
  if (!quads_ok(g)) return {dim3((unsigned)grid_for(words, 256, 38), 16u), 256};
  const int block = words / 4 >= 38 * 1024 ? 1024 : 256;
  return {dim3((unsigned)grid_for(words / 4, block, 152 * 256 / block), 4u), block};
}

int recount_grid(const Geo &g) {
  const dim3 d = recount_shape(g).grid;
  return (int)(d.x * d.y);
}

cudaError_t launch_recount(const Geo &g, int64_t *partials, int64_t *ring, int64_t ring_cap,
                           int64_t *hist, int nbins, int64_t sweep_off, cudaStream_t s) {
  RecountArgs a{partials, ring, ring_cap, hist, nbins, sweep_off};
  const RecountShape sh = recount_shape(g);
  return launch_pdl(recount_kernel, sh.grid, sh.block, s, g, a);
}

cudaError_t launch_advance(int64_t *ctl, int64_t phases, cudaStream_t s) {
  return launch_pdl(advance_kernel, 1, 1, s, ctl, phases);
}

cudaError_t launch_set_ctl(int64_t *ctl, int64_t phase_base, cudaStream_t s) {
  set_ctl_kernel<<<1, 32, 0, s>>>(ctl, phase_base);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const Geo &g, uint8_t *out, cudaStream_t s) {
  unpack_kernel<<<grid_for(16 * (int64_t)g.Cy * g.W, 256, 152 * 16), 256, 0, s>>>(g, out);
  return cudaGetLastError();
}

cudaError_t launch_pack(const Geo &g, const uint8_t *in, int *bad, cudaStream_t s) {
  pack_kernel<<<grid_for(16 * (int64_t)g.Cy * g.W, 256, 152 * 16), 256, 0, s>>>(g, in, bad);
  return cudaGetLastError();
}

cudaError_t launch_pack2(const Geo &g, const uint8_t *in, cudaStream_t s) {
  pack2_kernel<<<grid_for(4 * (int64_t)g.Cy * g.W, 256, 152 * 16), 256, 0, s>>>(g, in);
  return cudaGetLastError();
}

cudaError_t launch_unpack2(const Geo &g, uint8_t *out, cudaStream_t s) {
  unpack2_kernel<<<grid_for(4 * (int64_t)g.Cy * g.W, 256, 152 * 16), 256, 0, s>>>(g, out);
  return cudaGetLastError();
}

cudaError_t launch_philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                          uint32_t k1, int64_t count, uint32_t *out, cudaStream_t s) {
  philox_kernel<<<grid_for(count, 256, 152 * 8), 256, 0, s>>>(c0, c1, c2, c3, k0, k1, count, out);
  return cudaGetLastError();
}

}  // namespace ccmc
