// cic_kernels.cuh -- particle mass deposition by Cloud-in-Cell on a periodic
// n^3 grid (paper Sec. 4, mass deposition), in FP64 or FP32.
//
// Shifted stencil: along each axis s = x n - 1/2, i0 = floor(s), f = s - i0;
// the particle gives m (wx wy wz) n^3 to the 8 cells (i0 + cx, j0 + cy,
// k0 + cz), wx = 1 - f for cx = 0 and f for cx = 1 (the `medium' stencil:
// only the 2^3 cells with non-zero weight).  The cell (i0, j0, k0) is the
// particle's source cell; particles are sorted by the Hilbert index of their
// source cell so that particles of one source cell are contiguous.
//
//   sort      source-cell Hilbert keys, then a stable LSD radix sort of
//             (key, particle) pairs, tiles of 4096 items staged through
//             shared memory so that every digit's run is written contiguously;
//             then the particle arrays are gathered into the sorted order.
//   atomic    one thread per particle; lanes of a warp that share a source
//             cell add their 8 contributions by a segmented shuffle reduction
//             and the segment's first lane issues 8 atomic adds (the paper's
//             medium kernel: warp combining + atomicAdd).
//   segment   deterministic: segment starts by a prefix sum over the sorted
//             keys; one thread per source-cell segment sums its particles'
//             8 contributions in particle order; one thread per grid cell
//             gathers the 8 segment sums that reach it, in stencil order
//             (the paper's small kernel: prefix sums and one update per
//             segment and stencil offset).  The result depends only on the
//             particles and their order, not on the launch or on timing.
//
// Every grid index is masked by n - 1 (n a power of two), so that no position,
// even a non-finite one, addresses outside the grid.
#pragma once
#include "amr_internal.cuh"
#include "cic_weights.cuh"
#include "hilbert_table.cuh"
#include "scan_kernels.cuh"

namespace amr {
namespace {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortRounds = 8;
constexpr int kSortTile = kSortThreads * kSortRounds;  // 4096 items per tile

// Grid of the deposition: n = 2^bits cells per axis; fn = n in the state type.
template <class T>
struct CicGrid {
  int n, bits;
  T fn, scale;  // scale = n^3 (mass -> density), exact
};

// floor(x 2^k) for a double 0 <= x < 1, from its bits on the integer pipe
// (GB300 runs FP64 at 1/64 of the FP32 rate, so the deposition keeps its
// FP64 instruction count low).  Out-of-range inputs give some value that the
// callers mask into the grid.
__device__ __forceinline__ int floor_scaled(double x, int k) {
  const uint64_t u = uint64_t(__double_as_longlong(x));
  const int E = int(u >> 52) & 0x7FF;
  const uint64_t M = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = 1075 - E - k;
  if (E == 0 || sh >= 64) return 0;
  if (sh <= 0) return 0x7FFFFFFF;
  return int(M >> sh);
}

// (2 i + 1) / 2 as a double, built on the integer pipe (|2 i + 1| < 2^31)
__device__ __forceinline__ double half_odd(int i) {
  const int k = 2 * i + 1;
  const uint32_t a = uint32_t(k < 0 ? -k : k);
  const int lz = __clz(a);
  const int e = 31 - lz;                              // a = 1.frac 2^e
  const uint32_t frac = e ? (a << (lz + 1)) : 0u;     // bits below the leading one, left aligned
  const uint32_t hi = (uint32_t(k < 0) << 31) | (uint32_t(1022 + e) << 20) | (frac >> 12);
  return __hiloint2double(int(hi), int(frac << 20));
}

// source cell along one axis: floor(x n - 1/2), unmasked
template <class T>
__device__ __forceinline__ int cic_cell(T x, const CicGrid<T> &g) {
  return __float2int_rd(x * g.fn - T(0.5));
}
template <>
__device__ __forceinline__ int cic_cell<double>(double x, const CicGrid<double> &g) {
  // floor(x n - 1/2) = floor((floor(2 x n) - 1) / 2)
  return (floor_scaled(x, g.bits + 1) - 1) >> 1;
}

// source cell (masked into the grid) and weights along one axis:
// s = x n - 1/2, i0 = floor(s), w1 = f = s - i0, w0 = 1 - f
template <class T>
__device__ __forceinline__ int cic_axis(T x, const CicGrid<T> &g, T &w0, T &w1) {
  const T s = x * g.fn - T(0.5);
  const T fl = floor(s);
  w1 = s - fl;
  w0 = T(1) - w1;
  return int(fl) & (g.n - 1);
}
template <>
__device__ __forceinline__ int cic_axis<double>(double x, const CicGrid<double> &g, double &w0,
                                                double &w1) {
  // x n and x n - 1/2 - i0 are exact, so one FMA gives the same f as
  // (x n - 1/2) - floor(x n - 1/2)
  const int i0 = cic_cell(x, g);
  w1 = fma(x, g.fn, -half_odd(i0));
  w0 = 1.0 - w1;
  return i0 & (g.n - 1);
}

__device__ __forceinline__ uint32_t grid_at(int n, int i, int j, int k) {
  const int m = n - 1;
  return uint32_t(i & m) + uint32_t(n) * (uint32_t(j & m) + uint32_t(n) * uint32_t(k & m));
}

// the 8 contributions ((m n^3 wx) wy) wz of one particle, corner
// c = cx + 2 cy + 4 cz; (i, j, k) its source cell
template <class T>
__device__ __forceinline__ void cic_weights(T x, T y, T z, T m, const CicGrid<T> &g, int &i, int &j,
                                            int &k, T w[8]) {
  T wx[2], wy[2], wz[2];
  i = cic_axis(x, g, wx[0], wx[1]);
  j = cic_axis(y, g, wy[0], wy[1]);
  k = cic_axis(z, g, wz[0], wz[1]);
  const T ms = m * g.scale;
  T a[2], b[4];
#pragma unroll
  for (int cx = 0; cx < 2; ++cx) a[cx] = ms * wx[cx];
#pragma unroll
  for (int q = 0; q < 4; ++q) b[q] = a[q & 1] * wy[q >> 1];
#pragma unroll
  for (int c = 0; c < 8; ++c) w[c] = b[c & 3] * wz[c >> 2];
}

// FP64: on the integer pipes, each contribution rounded once
template <>
__device__ __forceinline__ void cic_weights<double>(double x, double y, double z, double m, const CicGrid<double> &g,
                                                    int &i, int &j, int &k, double w[8]) {
  if (cic_in_range(x, y, z, m)) {
    uint64_t b[8];
    cic_weights_int(uint64_t(__double_as_longlong(x)), uint64_t(__double_as_longlong(y)),
                    uint64_t(__double_as_longlong(z)), uint64_t(__double_as_longlong(m)), g.bits, i, j, k, b);
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = __longlong_as_double((long long)b[c]);
    return;
  }
  double wx[2], wy[2], wz[2];
  i = cic_axis(x, g, wx[0], wx[1]);
  j = cic_axis(y, g, wy[0], wy[1]);
  k = cic_axis(z, g, wz[0], wz[1]);
  for (int c = 0; c < 8; ++c) w[c] = ((m * g.scale * wx[c & 1]) * wy[(c >> 1) & 1]) * wz[c >> 2];
}

// Sums of the lanes' w over runs of lanes (`runs`: bit L set where a run
// starts at lane L; bit 0 always set): a backward segmented scan that leaves
// each run's total in its first lane.  The tree depends only on the run
// lengths, so equal inputs give equal sums.
template <class T>
__device__ __forceinline__ void warp_run_sums(T w[8], unsigned runs, unsigned lane) {
  const unsigned above = runs & ~((2u << lane) - 1u);  // run starts after this lane
  const unsigned next = above ? unsigned(__ffs(above) - 1) : 32u;
  const unsigned len = ((runs >> lane) & 1u) ? next - lane : 0u;
  const unsigned maxrun = __reduce_max_sync(0xFFFFFFFFu, len);
  for (unsigned off = 1; off < maxrun; off <<= 1) {
    const bool take = lane + off < next;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const T o = __shfl_down_sync(0xFFFFFFFFu, w[c], off);
      if (take) w[c] += o;
    }
  }
}

// The 8 sums over all 32 lanes, reduce-scatter style (9 additions per lane
// instead of 40): afterwards lane L holds the total of component L >> 2.
template <class T>
__device__ __forceinline__ T warp_total_scatter(const T w[8], unsigned lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  T h[4], q[2];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const T send = b4 ? w[c] : w[c + 4];
    const T keep = b4 ? w[c + 4] : w[c];
    h[c] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 16);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const T send = b3 ? h[c] : h[c + 2];
    const T keep = b3 ? h[c + 2] : h[c];
    q[c] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 8);
  }
  T v = (b2 ? q[1] : q[0]) + __shfl_xor_sync(0xFFFFFFFFu, b2 ? q[0] : q[1], 4);
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
  return v;
}

// ---------------------------------------------------------------------------
// sort
// ---------------------------------------------------------------------------
// the source cells' Hilbert indices (hilbert_table.cuh)
__device__ const HilbertTable kHilbert = hilbert_table();

// the index of a cell with BITS bits per axis; two: kHilbert.two in shared memory
template <int BITS>
__device__ __forceinline__ uint32_t hilbert_index_u32(const uint16_t *two, uint32_t x, uint32_t y, uint32_t z) {
  uint32_t key = 0, s = 0;
  if (BITS & 1) {
    constexpr int b = BITS - 1;
    const uint32_t v = __ldg(kHilbert.one + (((x >> b) & 1) << 2 | ((y >> b) & 1) << 1 | ((z >> b) & 1)));
    key = v & 7u;
    s = v >> 6;
  }
#pragma unroll
  for (int b = (BITS & ~1) - 2; b >= 0; b -= 2) {
    const uint32_t v = two[s << 6 | ((x >> b) & 3) << 4 | ((y >> b) & 3) << 2 | ((z >> b) & 3)];
    key = key << 6 | (v & 63u);
    s = v >> 6;
  }
  return key;
}

// per-tile digit counts, tile-major: table[tile * ndig + d]; digits of up to 8 bits
constexpr int kSortBins = 256;

// the keys, and the tile's counts of the first digit
template <class T, int BITS>
__global__ void __launch_bounds__(kSortThreads) k_part_keys(int64_t np, CicGrid<T> g, const T *__restrict__ x,
                                                            const T *__restrict__ y, const T *__restrict__ z,
                                                            uint32_t *__restrict__ key, int nbits,
                                                            uint32_t *__restrict__ table) {
  __shared__ uint32_t hist[kSortBins];
  __shared__ __align__(16) uint16_t two[96 * 64];
  const int ndig = 1 << nbits;
  for (int d = threadIdx.x; d < ndig; d += kSortThreads) hist[d] = 0;
  static_assert(alignof(HilbertTable) >= alignof(uint32_t) && offsetof(HilbertTable, two) == 0, "read as 32-bit words");
  for (int q = threadIdx.x; q < 96 * 64 / 2; q += kSortThreads)
    reinterpret_cast<uint32_t *>(two)[q] = __ldg(reinterpret_cast<const uint32_t *>(kHilbert.two) + q);
  __syncthreads();
  const int64_t base = blockIdx.x * int64_t(kSortTile);
  const uint32_t m = uint32_t(g.n - 1);
#pragma unroll 4
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t t = base + r * kSortThreads + threadIdx.x;
    if (t < np) {
      const uint32_t i = uint32_t(cic_cell(x[t], g)) & m, j = uint32_t(cic_cell(y[t], g)) & m,
                     k = uint32_t(cic_cell(z[t], g)) & m;
      const uint32_t h = hilbert_index_u32<BITS>(two, i, j, k);
      key[t] = h;
      atomicAdd(&hist[h & unsigned(ndig - 1)], 1u);
    }
  }
  __syncthreads();
  for (int d = threadIdx.x; d < ndig; d += kSortThreads) table[int64_t(blockIdx.x) * ndig + d] = hist[d];
}

__global__ void __launch_bounds__(kSortThreads) k_psort_hist(const uint32_t *__restrict__ keys,
                                                             int64_t np, int shift, int nbits,
                                                             uint32_t *__restrict__ table) {
  __shared__ uint32_t hist[kSortBins];
  const int ndig = 1 << nbits;
  for (int d = threadIdx.x; d < ndig; d += kSortThreads) hist[d] = 0;
  __syncthreads();
  const int64_t base = blockIdx.x * int64_t(kSortTile);
  unsigned dk[kSortRounds];  // all loads of the tile in flight at once
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int64_t t = base + r * kSortThreads + threadIdx.x;
    dk[r] = t < np ? __ldcs(keys + t) : 0xFFFFFFFFu;
  }
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r)
    if (dk[r] != 0xFFFFFFFFu) atomicAdd(&hist[(dk[r] >> shift) & unsigned(ndig - 1)], 1u);
  __syncthreads();
  for (int d = threadIdx.x; d < ndig; d += kSortThreads) table[int64_t(blockIdx.x) * ndig + d] = hist[d];
}

// Offsets of the scatter from the tile-major counts cnt[tile][d]: per digit,
// an exclusive prefix over tiles inside chunks of kScanChunk tiles (pref),
// then the chunks' exclusive prefix per digit (base[chunk][d]), then the
// digits' bases (dbase[d]); a tile's run of digit d starts at
// pref[tile][d] + base[tile / kScanChunk][d] + dbase[d].  The counts, the
// prefixes and the scatter's reads all run along the digits (coalesced).
constexpr int kScanChunk = 32;

__global__ void k_psort_chunks(const uint32_t *__restrict__ cnt, int64_t ntiles, int ndig,
                               uint32_t *__restrict__ pref, uint32_t *__restrict__ base) {
  const int d = threadIdx.x;
  if (d >= ndig) return;
  const int64_t t0 = blockIdx.x * int64_t(kScanChunk);
  const int64_t t1 = t0 + kScanChunk < ntiles ? t0 + kScanChunk : ntiles;
  uint32_t run = 0;
  for (int64_t t = t0; t < t1; ++t) {
    const uint32_t c = cnt[t * ndig + d];
    pref[t * ndig + d] = run;
    run += c;
  }
  base[int64_t(blockIdx.x) * ndig + d] = run;  // the chunk's total, for now
}

// one block per digit: exclusive scan of the digit's chunk totals (in place)
// and the digit's total
constexpr int kScanThreads = 256;

__global__ void __launch_bounds__(kScanThreads) k_psort_digit_scan(uint32_t *__restrict__ base, int64_t nchunks,
                                                                  int ndig, uint32_t *__restrict__ dtot) {
  __shared__ uint32_t part[kScanThreads];
  const int d = blockIdx.x;
  const int64_t per = (nchunks + kScanThreads - 1) / kScanThreads;
  const int64_t c0 = threadIdx.x * per, c1 = c0 + per < nchunks ? c0 + per : nchunks;
  uint32_t sum = 0;
  for (int64_t c = c0; c < c1; ++c) sum += base[c * ndig + d];
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int off = 1; off < kScanThreads; off <<= 1) {
    const uint32_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  uint32_t run = part[threadIdx.x] - sum;
  for (int64_t c = c0; c < c1; ++c) {
    const uint32_t x = base[c * ndig + d];
    base[c * ndig + d] = run;
    run += x;
  }
  if (threadIdx.x == kScanThreads - 1) dtot[d] = part[kScanThreads - 1];
}

// one block: the digits' bases, the exclusive scan of their totals (in place)
__global__ void __launch_bounds__(kScanThreads) k_psort_digit_base(uint32_t *__restrict__ dtot, int ndig) {
  __shared__ uint32_t part[kScanThreads];
  const int d = threadIdx.x;
  const uint32_t x = d < ndig ? dtot[d] : 0u;
  part[d] = x;
  __syncthreads();
  for (int off = 1; off < kScanThreads; off <<= 1) {
    const uint32_t v = d >= off ? part[d - off] : 0u;
    __syncthreads();
    part[d] += v;
    __syncthreads();
  }
  if (d < ndig) dtot[d] = part[d] - x;
}

// Stable scatter of one tile.  Each warp ranks 256 consecutive items by itself
// (8 rounds of 32, counting per digit in its own row of wcnt), the rows are
// summed over the warps once, and the tile goes through shared memory in digit
// order, so that consecutive threads write consecutive places of a digit's run.
// A pass of 16.8 M pairs takes 101 us; 131 us with tiles of 2048 items and two
// barriers per round of the block (a digit's count kept for the block).
// FIRST: the values are the items' indices (nothing read).
template <bool FIRST>
__global__ void __launch_bounds__(kSortThreads) k_psort_scatter(
    const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint32_t *__restrict__ kout,
    uint32_t *__restrict__ vout, int64_t np, int shift, int nbits, const uint32_t *__restrict__ pref,
    const uint32_t *__restrict__ cbase, const uint32_t *__restrict__ dbase) {
  __shared__ uint32_t skey[kSortTile], sval[kSortTile];
  __shared__ uint16_t wcnt[kSortWarps * kSortBins];  // [warp][digit]; a tile's counts stay below 2^16
  __shared__ uint32_t lstart[kSortBins], goff[kSortBins], wsum[kSortBins / 32];
  const int ndig = 1 << nbits;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t base = blockIdx.x * int64_t(kSortTile);
  const int nt = int(np - base < kSortTile ? np - base : kSortTile);
  uint16_t *mine = wcnt + warp * kSortBins;
  uint32_t kr[kSortRounds], vr[kSortRounds];  // all loads of the tile in flight at once
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const int q = warp * 32 * kSortRounds + r * 32 + lane;
    kr[r] = q < nt ? __ldcs(kin + base + q) : 0u;
    vr[r] = FIRST ? uint32_t(base + q) : q < nt ? __ldcs(vin + base + q) : 0u;
  }
#pragma unroll
  for (int d = 0; d < kSortBins / 32; ++d) mine[32 * d + lane] = 0;
  __syncwarp();
  uint32_t rank[kSortRounds];
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    const bool valid = warp * 32 * kSortRounds + r * 32 + lane < nt;
    const unsigned dig = (kr[r] >> shift) & unsigned(ndig - 1);
    const unsigned peers = digit_peers(dig, nbits, valid);
    const unsigned before = mine[dig];
    rank[r] = before + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
    if (valid && (peers >> lane) == 1u) mine[dig] = uint16_t(before + __popc(peers));  // the last of the peers
    __syncwarp();
  }
  __syncthreads();
  // per digit: the warps' exclusive offsets and the tile's count; then the
  // counts' exclusive scan over the digits (one digit per thread)
  uint32_t cnt = 0;
  if (threadIdx.x < kSortBins) {
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t c = wcnt[w * kSortBins + threadIdx.x];
      wcnt[w * kSortBins + threadIdx.x] = uint16_t(cnt);
      cnt += c;
    }
  }
  uint32_t incl = cnt;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
    if (lane >= off) incl += v;
  }
  if (threadIdx.x < kSortBins && lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (threadIdx.x < kSortBins) {
    uint32_t start = incl - cnt;
    for (int w = 0; w < warp; ++w) start += wsum[w];
    lstart[threadIdx.x] = start;
    if (int(threadIdx.x) < ndig)
      goff[threadIdx.x] = pref[int64_t(blockIdx.x) * ndig + threadIdx.x] +
                          cbase[int64_t(blockIdx.x / kScanChunk) * ndig + threadIdx.x] + dbase[threadIdx.x] - start;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortRounds; ++r) {
    if (warp * 32 * kSortRounds + r * 32 + lane < nt) {
      const unsigned dig = (kr[r] >> shift) & unsigned(ndig - 1);
      const uint32_t lp = lstart[dig] + mine[dig] + rank[r];
      skey[lp] = kr[r];
      sval[lp] = vr[r];
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nt; q += kSortThreads) {
    const uint32_t k = skey[q];
    const uint32_t dst = goff[(k >> shift) & unsigned(ndig - 1)] + uint32_t(q);  // modulo 2^32: np < 2^32
    kout[dst] = k;
    vout[dst] = sval[q];
  }
}

// particle arrays into the sorted order
template <class T>
__global__ void k_part_gather(int64_t np, const uint32_t *__restrict__ perm, const T *__restrict__ x,
                              const T *__restrict__ y, const T *__restrict__ z,
                              const T *__restrict__ m, const uint32_t *__restrict__ id,
                              T *__restrict__ x2, T *__restrict__ y2, T *__restrict__ z2,
                              T *__restrict__ m2, uint32_t *__restrict__ id2) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= np) return;
  const uint32_t p = perm[t];
  x2[t] = x[p];
  y2[t] = y[p];
  z2[t] = z[p];
  m2[t] = m[p];
  id2[t] = id[p];
}

// ---------------------------------------------------------------------------
// atomic deposit (warp combining of equal source cells)
// ---------------------------------------------------------------------------
// the 8 contributions of source cell (i, j, k) added to the grid
template <class T>
__device__ __forceinline__ void add_stencil(const CicGrid<T> &g, int i, int j, int k, const T w[8], T *rho) {
#pragma unroll
  for (int c = 0; c < 8; ++c) atomicAdd(&rho[grid_at(g.n, i + (c & 1), j + ((c >> 1) & 1), k + (c >> 2))], w[c]);
}
template <class T>
__global__ void __launch_bounds__(256) k_cic_atomic(int64_t np, CicGrid<T> g, const T *__restrict__ x,
                                                    const T *__restrict__ y, const T *__restrict__ z,
                                                    const T *__restrict__ m, T *__restrict__ rho) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const unsigned lane = threadIdx.x & 31;
  const bool valid = t < np;
  T w[8];
  int i = 0, j = 0, k = 0;
  uint32_t cell = 0xFFFFFFFFu;
  if (valid) {
    cic_weights(x[t], y[t], z[t], m[t], g, i, j, k, w);
    cell = grid_at(g.n, i, j, k);
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = T(0);
  }
  // runs of equal source cells among the warp's lanes
  const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, cell, 1);
  const unsigned runs = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != cell);
  if (runs == 1u) {
    // one source cell for the whole warp (or no particle at all): lanes
    // 0, 4, .., 28 add one component each
    if (cell == 0xFFFFFFFFu) return;
    const T v = warp_total_scatter(w, lane);
    if ((lane & 3) == 0) {
      const int c = int(lane >> 2);
      atomicAdd(&rho[grid_at(g.n, i + (c & 1), j + ((c >> 1) & 1), k + (c >> 2))], v);
    }
    return;
  }
  // Partial runs: FP32 sums them before its atomics; FP64, whose additions
  // cost 1/64 of the FP32 rate on GB300, lets every particle add its own 8
  // contributions (L2 absorbs the extra atomics).
  const bool combine = sizeof(T) == 4;
  if (combine && runs != 0xFFFFFFFFu) warp_run_sums(w, runs, lane);
  if (valid && (!combine || ((runs >> lane) & 1u))) add_stencil(g, i, j, k, w, rho);
}

// ---------------------------------------------------------------------------
// deterministic deposit (segment sums)
// ---------------------------------------------------------------------------
__global__ void k_seg_heads(int64_t np, const uint32_t *__restrict__ key, uint32_t *__restrict__ flag) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= np) return;
  flag[q] = (q == 0 || key[q] != key[q - 1]) ? 1u : 0u;
}

// Per particle, in aligned groups of 32 (one warp each): the contributions
// summed over each run of equal source cells inside the group (fixed shuffle
// tree).  A run that starts segment s writes its sums to sums[c * cap + s],
// its first particle to start[s], and maps its source cell to s; the run at the start of group G that
// continues a segment from earlier groups writes them to carry[c * ngroups + G].
template <class T>
__global__ void __launch_bounds__(256) k_seg_partial(int64_t np, CicGrid<T> g, const uint32_t *__restrict__ key,
                                                     const uint32_t *__restrict__ scan, const T *__restrict__ x,
                                                     const T *__restrict__ y, const T *__restrict__ z,
                                                     const T *__restrict__ m, int64_t cap, int64_t ngroups,
                                                     T *__restrict__ sums, T *__restrict__ carry,
                                                     int32_t *__restrict__ cellmap, uint32_t *__restrict__ start,
                                                     uint32_t *__restrict__ nseg) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const unsigned lane = threadIdx.x & 31;
  const bool valid = t < np;
  T w[8];
  int i = 0, j = 0, k = 0;
  uint32_t kk = 0xFFFFFFFFu;
  bool head = false;
  if (valid) {
    cic_weights(x[t], y[t], z[t], m[t], g, i, j, k, w);
    kk = key[t];
    head = t == 0 || key[t - 1] != kk;
    if (head) start[scan[t]] = uint32_t(t);
    if (t == np - 1) {  // the number of segments; start[S] = np ends the last one
      const uint32_t S = scan[t] + (head ? 1u : 0u);
      start[S] = uint32_t(np);
      *nseg = S;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = T(0);
  }
  const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, kk, 1);
  const unsigned runs = __ballot_sync(0xFFFFFFFFu, lane == 0 || prev != kk);
  if (runs == 1u) {
    // the whole group is one run: reduce-scatter, lane 4c writes component c
    if (kk == 0xFFFFFFFFu) return;
    const T v = warp_total_scatter(w, lane);
    const bool head0 = __shfl_sync(0xFFFFFFFFu, head, 0);
    if ((lane & 3) == 0) {
      const int c = int(lane >> 2);
      if (head0)
        sums[c * cap + int64_t(scan[t - lane])] = v;
      else
        carry[c * ngroups + (t >> 5)] = v;
    }
    if (lane == 0 && head0) cellmap[grid_at(g.n, i, j, k)] = int32_t(scan[t]);
    return;
  }
  if (runs != 0xFFFFFFFFu) warp_run_sums(w, runs, lane);
  if (!valid) return;
  if (head) {
    const int64_t s = scan[t];
#pragma unroll
    for (int c = 0; c < 8; ++c) sums[c * cap + s] = w[c];
    cellmap[grid_at(g.n, i, j, k)] = int32_t(s);
  } else if (lane == 0) {
    const int64_t G = t >> 5;
#pragma unroll
    for (int c = 0; c < 8; ++c) carry[c * ngroups + G] = w[c];
  }
}

// Per segment that spans groups: add the carries of its later groups, in
// group order.
template <class T>
__global__ void k_seg_carry(const uint32_t *__restrict__ nseg, const uint32_t *__restrict__ start, int64_t cap,
                            int64_t ngroups, const T *__restrict__ carry, T *__restrict__ sums) {
  const int64_t s = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (s >= int64_t(*nseg)) return;
  const int64_t g0 = int64_t(start[s]) >> 5, g1 = (int64_t(start[s + 1]) - 1) >> 5;
  if (g1 == g0) return;
  T acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = sums[c * cap + s];
  for (int64_t G = g0 + 1; G <= g1; ++G) {
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] += carry[c * ngroups + G];
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) sums[c * cap + s] = acc[c];
}

// one thread per grid cell: rho = the sums of the (up to) 8 segments whose
// stencils reach the cell, in stencil order c = 0..7
template <class T>
__global__ void k_seg_gather(int n, int64_t cap, const int32_t *__restrict__ cellmap,
                             const T *__restrict__ sums, T *__restrict__ rho) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= int64_t(n) * n * n) return;
  const int i = int(t & (n - 1)), j = int((t / n) & (n - 1)), k = int(t / (int64_t(n) * n));
  T acc = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int32_t s = cellmap[grid_at(n, i - (c & 1), j - ((c >> 1) & 1), k - (c >> 2))];
    if (s >= 0) acc += sums[c * cap + s];
  }
  rho[t] = acc;
}

// ---------------------------------------------------------------------------
// host <-> device helpers of the particle handle
// ---------------------------------------------------------------------------

template <class T>
__global__ void k_from_double(int64_t n, const double *__restrict__ a, T *__restrict__ b) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) b[t] = T(a[t]);
}

template <class T>
__global__ void k_to_double(int64_t n, const T *__restrict__ a, double *__restrict__ b) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) b[t] = double(a[t]);
}

__global__ void k_iota(int64_t n, uint32_t *id) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) id[t] = uint32_t(t);
}

}  // namespace
}  // namespace amr
