// mg_kernels.cuh -- multigrid Poisson V-cycles on the periodic base level
// (paper Sec. 5, self-gravity).
//
//   (sum of the 6 neighbours - 6 phi) / dx^2 = fourpiG (rho - mean rho)
//
// Smoother: red-black Gauss-Seidel, colour = parity of x + y + z (the parity
// of the cell's index inside its oct).  Restriction: the residuals of the 8
// children, averaged into the coarse source.  Prolongation: trilinear, weights
// (1, 3, 3, 9, 3, 9, 9, 27)/64.  Hierarchy: the same periodic box at half the
// resolution per level, down to 2^3 cells, smoothed 8 times there.
//
// The base level lives in the mesh's oct order; the solver works on dense
// arrays [x + n (y + n z)] of every multigrid level (unit-stride x, so every
// stencil access is coalesced), gathered from and scattered back to the octs.
// On GB300 the FP64 pipe bounds these stencils on the large grids (6 FP64
// instructions per smoothed cell against 16 bytes of traffic) and the launches on
// the small ones; no step divides: the Gauss-Seidel update multiplies by the
// rounded 1/6 where the operator divides by 6 (the two differ by at most a few
// units in the last place per update; the product runs on the integer pipes),
// and the residual multiplies by 1/dx^2, which is exact (dx is a power of two).
#pragma once
#include "amr_internal.cuh"
#include "fp64_int.cuh"

namespace amr {

__device__ __forceinline__ int64_t mg_at(int n, int x, int y, int z) {
  const int m = n - 1;  // n is a power of two: periodic wrap by masking
  return int64_t(x & m) + int64_t(n) * (int64_t(y & m) + int64_t(n) * int64_t(z & m));
}

__device__ __forceinline__ double mg_nbsum(int n, const double *__restrict__ p, int x, int y, int z) {
  return ((p[mg_at(n, x - 1, y, z)] + p[mg_at(n, x + 1, y, z)]) +
          (p[mg_at(n, x, y - 1, z)] + p[mg_at(n, x, y + 1, z)])) +
         (p[mg_at(n, x, y, z - 1)] + p[mg_at(n, x, y, z + 1)]);
}

// base-level density (oct order) into the dense array; one thread per cell
template <class T>
__global__ void k_mg_gather(const T *__restrict__ U, const uint64_t *__restrict__ key, int lo,
                            int nl, int n, double *__restrict__ rho) {
  const int64_t g = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (g >= 8 * int64_t(nl)) return;
  const int o = lo + int(g >> 3), c = int(g & 7);
  const uint64_t k = key[o];
  const int x = 2 * int(ikey_x(k)) + (c & 1), y = 2 * int(ikey_y(k)) + ((c >> 1) & 1),
            z = 2 * int(ikey_z(k)) + ((c >> 2) & 1);
  rho[mg_at(n, x, y, z)] = double(U[8 * int64_t(o) + c]);
}

// block sums of a[0..m) into part[blockIdx.x] (warp shuffles, then shared
// memory); squared when sq
__global__ void k_mg_sum(const double *__restrict__ a, int64_t m, int sq, double *__restrict__ part) {
  __shared__ double ws[32];
  double s = 0.0;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < m; t += int64_t(gridDim.x) * blockDim.x)
    s += sq ? a[t] * a[t] : a[t];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

// sum of the partial sums by one warp: lane l adds parts l, l + 32, .., then a
// fixed butterfly (one thread adding up to 1024 of them in turn took 20 us)
__device__ __forceinline__ double mg_sum_parts(const double *__restrict__ part, int nparts) {
  double s = 0.0;
  for (int q = threadIdx.x; q < nparts; q += 32) s += part[q];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  return s;
}

// out = scale * (sum of the partial sums); one warp
__global__ void k_mg_total(const double *__restrict__ part, int nparts, double scale,
                           double *__restrict__ out) {
  const double s = mg_sum_parts(part, nparts);
  if (threadIdx.x == 0) *out = s * scale;
}

// f = fourpiG (rho - mean)
__global__ void k_mg_source(const double *__restrict__ rho, int64_t m, const double *__restrict__ mean,
                            double fourpiG, double *__restrict__ f) {
  const double mu = *mean;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < m; t += int64_t(gridDim.x) * blockDim.x)
    f[t] = fourpiG * (rho[t] - mu);
}

// v / 6 as v times the rounded 1/6, on the integer pipes (NaN, infinities and
// values near overflow: on the FP64 pipe)
__device__ __forceinline__ double mg_sixth(double v) {
  return below<1000>(v) ? mul_int0(v, 1.0 / 6.0) : v * (1.0 / 6.0);
}

// one colour of a red-black sweep: thread t -> (x, y, z) with x + y + z of
// the colour's parity; n = 2^b
__global__ void k_mg_smooth(int b, double dx2, const double *__restrict__ f, double *p, int colour) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= int64_t(1) << (3 * b - 1)) return;
  const int n = 1 << b;
  const int64_t yz = t >> (b - 1);
  const int y = int(yz) & (n - 1), z = int(yz >> b);
  const int x = 2 * (int(t) & (n / 2 - 1)) + ((y + z + colour) & 1);
  const int64_t i = mg_at(n, x, y, z);
  p[i] = mg_sixth(mg_nbsum(n, p, x, y, z) - dx2 * f[i]);
}

// coarse source = mean of the 8 children's residuals; coarse correction = 0.
// Three of a child's neighbours lie in the block of 8 and cancel against half
// of its diagonal when the residuals are summed: the sum needs, per child, its
// three outer neighbours less 3 p (42 FP64 operations per block, 72 with eight
// residuals).
__device__ __forceinline__ double mg_block_residual(int n, double inv_dx2, const double *__restrict__ f,
                                                    const double *__restrict__ p, int X, int Y, int Z) {
  double sf = 0.0, sp = 0.0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
    const int x = 2 * X + cx, y = 2 * Y + cy, z = 2 * Z + cz;
    const int64_t i = mg_at(n, x, y, z);
    sf += f[i];
    sp += ((p[mg_at(n, x + 2 * cx - 1, y, z)] + p[mg_at(n, x, y + 2 * cy - 1, z)]) +
           p[mg_at(n, x, y, z + 2 * cz - 1)]) - 3.0 * p[i];
  }
  return (sf - sp * inv_dx2) * 0.125;
}
__global__ void k_mg_restrict(int b, double inv_dx2, const double *__restrict__ f,
                              const double *__restrict__ p, double *__restrict__ fc, double *__restrict__ ec) {
  const int64_t T = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const int bc = b - 1, m = (1 << bc) - 1;
  if (T >= int64_t(1) << (3 * bc)) return;
  fc[T] = mg_block_residual(1 << b, inv_dx2, f, p, int(T) & m, int(T >> bc) & m, int(T >> (2 * bc)));
  ec[T] = 0.0;
}

// phi += trilinear prolongation of the coarse correction: the eight fine cells
// of coarse cell (X, Y, Z), one axis after the other (3 a + b per axis, the
// weights over 64; 46 FMAs for eight cells, against 12 operations per cell when
// each forms its own weighted sum)
__device__ __forceinline__ void mg_block_prolong(int n, const double *__restrict__ ec, double *__restrict__ p, int X,
                                                 int Y, int Z) {
  const int h = n >> 1;
  double zlo[2][2], zhi[2][2];  // [y][x] sums over z for the lower and the upper fine cells
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double a[3][2];  // [j][x]
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double c0 = ec[mg_at(h, X - 1, Y + j - 1, Z + k - 1)], c1 = ec[mg_at(h, X, Y + j - 1, Z + k - 1)],
                   c2 = ec[mg_at(h, X + 1, Y + j - 1, Z + k - 1)];
      a[j][0] = fma(3.0, c1, c0);
      a[j][1] = fma(3.0, c1, c2);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const double v[2] = {fma(3.0, a[1][x], a[0][x]), fma(3.0, a[1][x], a[2][x])};
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        if (k == 0) {
          zlo[y][x] = v[y];
        } else if (k == 1) {
          zlo[y][x] = fma(3.0, v[y], zlo[y][x]);
          zhi[y][x] = v[y];
        } else {
          zhi[y][x] = fma(3.0, zhi[y][x], v[y]);
        }
      }
    }
  }
#pragma unroll
  for (int z = 0; z < 2; ++z)
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const int64_t i = mg_at(n, 2 * X, 2 * Y + y, 2 * Z + z);
      double2 *q = reinterpret_cast<double2 *>(p + i);
      double2 w = *q;
      w.x = fma(z ? zhi[y][0] : zlo[y][0], 1.0 / 64.0, w.x);
      w.y = fma(z ? zhi[y][1] : zlo[y][1], 1.0 / 64.0, w.y);
      *q = w;
    }
}
__global__ void k_mg_prolong(int b, const double *__restrict__ ec, double *__restrict__ p) {
  const int64_t T = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  const int bc = b - 1, m = (1 << bc) - 1;
  if (T >= int64_t(1) << (3 * bc)) return;
  mg_block_prolong(1 << b, ec, p, int(T) & m, int(T >> bc) & m, int(T >> (2 * bc)));
}

// The rest of a V-cycle from a grid of n = 2^b <= 8 cells per axis down to 2^3
// and back, by one block in shared memory (21 launches otherwise; a 16^3 grid's
// FP64 work on one SM takes longer than its launches).
constexpr int kMGTail = 8;
__global__ void __launch_bounds__(256) k_mg_tail(int b, double dx2, const double *__restrict__ f, double *p, int pre,
                                                 int post, int sweeps) {
  __shared__ __align__(16) double sf[584], sp[584];  // 8^3 + 4^3 + 2^3
  const int n3 = 1 << (3 * b);
  for (int t = threadIdx.x; t < n3; t += blockDim.x) {
    sf[t] = f[t];
    sp[t] = p[t];
  }
  __syncthreads();
  auto smooth = [&](int bb, int off, double d2, int ns) {
    const int n = 1 << bb;
    for (int s = 0; s < 2 * ns; ++s) {
      for (int t = threadIdx.x; t < n * n * n / 2; t += blockDim.x) {
        const int y = (t >> (bb - 1)) & (n - 1), z = t >> (2 * bb - 1);
        const int x = 2 * (t & (n / 2 - 1)) + ((y + z + s) & 1);
        const int64_t i = mg_at(n, x, y, z);
        sp[off + i] = mg_sixth(mg_nbsum(n, sp + off, x, y, z) - d2 * sf[off + i]);
      }
      __syncthreads();
    }
  };
  int off = 0, bb = b;
  double d2 = dx2;
  while (bb > 1) {  // down
    smooth(bb, off, d2, pre);
    const int n = 1 << bb, nc = n / 2, offc = off + n * n * n;
    for (int T = threadIdx.x; T < nc * nc * nc; T += blockDim.x) {
      sf[offc + T] = mg_block_residual(n, 1.0 / d2, sf + off, sp + off, T & (nc - 1), (T >> (bb - 1)) & (nc - 1),
                                       T >> (2 * bb - 2));
      sp[offc + T] = 0.0;
    }
    __syncthreads();
    off = offc;
    --bb;
    d2 *= 4.0;
  }
  smooth(bb, off, d2, sweeps);
  while (bb < b) {  // up
    ++bb;
    const int n = 1 << bb, nc = n / 2, offc = off;
    off -= n * n * n;
    d2 *= 0.25;
    for (int T = threadIdx.x; T < nc * nc * nc; T += blockDim.x)
      mg_block_prolong(n, sp + offc, sp + off, T & (nc - 1), (T >> (bb - 1)) & (nc - 1), T >> (2 * bb - 2));
    __syncthreads();
    smooth(bb, off, d2, post);
  }
  for (int t = threadIdx.x; t < n3; t += blockDim.x) p[t] = sp[t];
}

// residual of the base level into r (for its L2 norm)
__global__ void k_mg_residual(int n, double inv_dx2, const double *__restrict__ f,
                              const double *__restrict__ p, double *__restrict__ r) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= int64_t(n) * n * n) return;
  const int x = int(t % n), y = int((t / n) % n), z = int(t / (int64_t(n) * n));
  r[t] = f[t] - (mg_nbsum(n, p, x, y, z) - 6.0 * p[t]) * inv_dx2;
}

// sqrt of the sum of the partial sums into out
__global__ void k_mg_norm(const double *__restrict__ part, int nparts, double *__restrict__ out) {
  const double s = mg_sum_parts(part, nparts);
  if (threadIdx.x == 0) *out = sqrt(s);
}

// phi - mean into the octs' cells (mesh order)
__global__ void k_mg_scatter(const double *__restrict__ p, const uint64_t *__restrict__ key, int lo,
                             int nl, int n, const double *__restrict__ mean,
                             double *__restrict__ phi_cells) {
  const int64_t g = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (g >= 8 * int64_t(nl)) return;
  const int o = lo + int(g >> 3), c = int(g & 7);
  const uint64_t k = key[o];
  const int x = 2 * int(ikey_x(k)) + (c & 1), y = 2 * int(ikey_y(k)) + ((c >> 1) & 1),
            z = 2 * int(ikey_z(k)) + ((c >> 2) & 1);
  phi_cells[g] = p[mg_at(n, x, y, z)] - *mean;
}

// ---------------------------------------------------------------------------
// Poisson on a refined level (Sec. 5, level by level): flat tables over the
// cells of each MG level (level 0: the level's cells; level k: their
// ancestors at level L-k), built on the host once per (member, level).
// Every operation is rounded as written (no contraction; a division by a power
// of two is the exact product with its reciprocal, one by 6..12 see
// mgl_over_diag), in the order of the plain definition, so the potential equals
// that of a sequential evaluation bit for bit.
//   nb[6][n]   face neighbour in the same MG level (-x,+x,-y,+y,-z,+z) or -1
//   nbnd[n]    faces to the outside (Dirichlet): the diagonal is -(6 + nbnd)
//   bsum[n]    2 sum of the faces' boundary values (MG level 0; 0 above)
//   child[8][n]   children in the MG level below (order cx, cy, cz with cz
//                 fastest) or -1; pro[8][n] the 8 coarse cells of a cell's
//                 trilinear stencil (a, b, d: 4 a + 2 b + d) or -1
// ---------------------------------------------------------------------------
__global__ void k_mgl_bsum(int64_t n, const int32_t *__restrict__ fatherg, const int32_t *__restrict__ acrossg,
                           const double *__restrict__ phil, double *__restrict__ bsum) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  const double pf = phil[fatherg[t]];
  double bs = 0.0;
  for (int k = 0; k < 6; ++k) {
    const int32_t q = acrossg[k * n + t];
    if (q >= 0) bs = __dadd_rn(bs, __dmul_rn(2.0, __dmul_rn(0.5, __dadd_rn(pf, phil[q]))));
  }
  bsum[t] = bs;
}

// source fourpiG (rho - rho_bar); rho_bar from the device when rho_bar_dev is
// set (the base level's mean, without a host round trip)
template <class T>
__global__ void k_mgl_source(int64_t n, const int32_t *__restrict__ g0, const T *__restrict__ rho, double fourpiG,
                             double rho_bar, const double *__restrict__ rho_bar_dev, double *__restrict__ f) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  const double rb = rho_bar_dev ? *rho_bar_dev : rho_bar;
  f[t] = __dmul_rn(fourpiG, __dsub_rn(double(rho[g0[t]]), rb));
}

__global__ void k_mgl_gather(int64_t n, const int32_t *__restrict__ g0, const double *__restrict__ phil,
                             double *__restrict__ e) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) e[t] = phil[g0[t]];
}

__global__ void k_mgl_scatter(int64_t n, const int32_t *__restrict__ g0, const double *__restrict__ e,
                              double *__restrict__ phil) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) phil[g0[t]] = e[t];
}

// x / (6 + b) rounded to nearest for b in 0..6, without a division: with y the
// rounded reciprocal (|1 - d y| is at most 2^-54 for these divisors), q = x y is
// within an ulp of the quotient and one step q + y (x - d q) rounds correctly
// (Markstein, IBM J. Res. Dev. 34, 1990).  Outside the range where the residual
// is exact (tiny, huge or non-finite x) the division itself.
__constant__ double kDiag[7] = {6.0, 7.0, 8.0, 9.0, 10.0, 11.0, 12.0};
__constant__ double kRcpDiag[7] = {1.0 / 6.0, 1.0 / 7.0, 1.0 / 8.0, 1.0 / 9.0, 1.0 / 10.0, 1.0 / 11.0, 1.0 / 12.0};
__device__ __forceinline__ double mgl_over_diag(double x, int b) {
  if (!within<900>(fabs(x))) return __ddiv_rn(x, kDiag[b]);
  const double d = kDiag[b], y = kRcpDiag[b], q = mul_int(x, y);
  return __fma_rn(y, __fma_rn(-d, q, x), q);
}

__device__ __forceinline__ double mgl_nbsum(int64_t n, const int32_t *__restrict__ nb, const double *e, int64_t t) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int32_t q = nb[k * n + t];
    if (q >= 0) s = __dadd_rn(s, e[q]);
  }
  return s;
}

// one colour of a red-black sweep: the cells of list[0..m)
__global__ void k_mgl_smooth(int64_t n, const int32_t *__restrict__ list, int64_t m, const int32_t *__restrict__ nb,
                             const int32_t *__restrict__ nbnd, const double *__restrict__ bsum,
                             const double *__restrict__ f, double *e, double dx2) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= m) return;
  const int64_t t = list[i];
  const double s = mgl_nbsum(n, nb, e, t);
  const double bs = bsum ? bsum[t] : 0.0;
  e[t] = mgl_over_diag(__dsub_rn(__dadd_rn(s, bs), __dmul_rn(dx2, f[t])), nbnd[t]);
}

// `sweeps` red-black sweeps of a small MG level (its even cells first in list)
// by one block: a launch per colour costs more than its few cells
constexpr int64_t kMGLBlock = 1024;
__global__ void __launch_bounds__(512) k_mgl_sweeps(int64_t n, const int32_t *__restrict__ list, int64_t nc0,
                                                    const int32_t *__restrict__ nb, const int32_t *__restrict__ nbnd,
                                                    const double *__restrict__ bsum, const double *__restrict__ f,
                                                    double *e, double dx2, int sweeps) {
  for (int s = 0; s < 2 * sweeps; ++s) {
    const int64_t i1 = (s & 1) ? n : nc0;
    for (int64_t i = ((s & 1) ? nc0 : 0) + threadIdx.x; i < i1; i += blockDim.x) {
      const int64_t t = list[i];
      const double sum = mgl_nbsum(n, nb, e, t);
      const double bs = bsum ? bsum[t] : 0.0;
      e[t] = mgl_over_diag(__dsub_rn(__dadd_rn(sum, bs), __dmul_rn(dx2, f[t])), nbnd[t]);
    }
    __syncthreads();
  }
}

__global__ void k_mgl_residual(int64_t n, const int32_t *__restrict__ nb, const int32_t *__restrict__ nbnd,
                               const double *__restrict__ bsum, const double *__restrict__ f,
                               const double *__restrict__ e, double inv_dx2, double *__restrict__ r) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  const double s = mgl_nbsum(n, nb, e, t);
  const double bs = bsum ? bsum[t] : 0.0;
  r[t] = __dsub_rn(f[t], __dmul_rn(__dsub_rn(__dadd_rn(s, bs), __dmul_rn(kDiag[nbnd[t]], e[t])), inv_dx2));
}

// coarse source = the children's residuals summed over 8; correction zeroed
__global__ void k_mgl_restrict(int64_t nc, const int32_t *__restrict__ child, const double *__restrict__ r,
                               double *__restrict__ fc, double *__restrict__ ec) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= nc) return;
  double s = 0.0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int32_t q = child[j * nc + t];
    if (q >= 0) s = __dadd_rn(s, r[q]);
  }
  fc[t] = __dmul_rn(s, 0.125);
  ec[t] = 0.0;
}

__global__ void k_mgl_prolong(int64_t nf, const int32_t *__restrict__ pro, const double *__restrict__ ec,
                              double *__restrict__ e) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= nf) return;
  double c[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int32_t q = pro[j * nf + t];
    c[j] = q >= 0 ? ec[q] : 0.0;
  }
  // c[4 a + 2 b + d]: a along x, b along y, d along z
  double v = __dmul_rn(27.0, c[0]);
  v = __dadd_rn(v, __dmul_rn(9.0, __dadd_rn(__dadd_rn(c[4], c[2]), c[1])));
  v = __dadd_rn(v, __dmul_rn(3.0, __dadd_rn(__dadd_rn(c[6], c[5]), c[3])));
  v = __dadd_rn(v, c[7]);
  e[t] = __dadd_rn(e[t], __dmul_rn(v, 1.0 / 64.0));
}

// sum of r^2 into one value per block (for the residual norm)
__global__ void k_mgl_sq(int64_t n, const double *__restrict__ r, double *__restrict__ part) {
  __shared__ double ws[8];
  double s = 0.0;
  for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < n; t += int64_t(gridDim.x) * blockDim.x)
    s += r[t] * r[t];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = 0.0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) b += ws[w];
    part[blockIdx.x] = b;
  }
}

__global__ void k_mgl_norm(const double *__restrict__ part, int nparts, double *out) {
  const double s = mg_sum_parts(part, nparts);
  if (threadIdx.x == 0) *out = sqrt(s);
}

// ---------------------------------------------------------------------------
// the tables of a refined level's hierarchy, built on the device: cells are
// keyed by (x << 2b) | (y << b) | z with b bits per axis (lexicographic in
// x, y, z, the sorted order of every table); neighbours, children and
// prolongation stencils are found by binary search in the sorted keys
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t mgl_key(int64_t x, int64_t y, int64_t z, int b) {
  return (uint64_t(x) << (2 * b)) | (uint64_t(y) << b) | uint64_t(z);
}
__device__ __forceinline__ void mgl_unkey(uint64_t k, int b, int64_t &x, int64_t &y, int64_t &z) {
  const uint64_t m = (uint64_t(1) << b) - 1;
  x = int64_t(k >> (2 * b));
  y = int64_t((k >> b) & m);
  z = int64_t(k & m);
}
// index of key c in the sorted keys[0..n), or -1 (at most log2(n) + 1 steps)
__device__ __forceinline__ int32_t mgl_find(const uint64_t *__restrict__ keys, int64_t n, uint64_t c) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (keys[mid] < c) lo = mid + 1; else hi = mid;
  }
  return (lo < n && keys[lo] == c) ? int32_t(lo) : -1;
}

// the cells of the level-L octs [lo, lo + nl): key and global cell index
__global__ void k_mgl_cells(const uint64_t *__restrict__ key, int lo, int64_t nl, int L, uint64_t *__restrict__ ck,
                            uint32_t *__restrict__ cv) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= 8 * nl) return;
  const int o = lo + int(t >> 3), c = int(t & 7);
  const uint64_t k = key[o];
  ck[t] = mgl_key(2 * int64_t(ikey_x(k)) + (c & 1), 2 * int64_t(ikey_y(k)) + ((c >> 1) & 1),
                  2 * int64_t(ikey_z(k)) + ((c >> 2) & 1), L);
  cv[t] = uint32_t(8 * int64_t(o) + c);
}

// parent keys (b bits per axis) of sorted child keys (b + 1 bits)
__global__ void k_mgl_parents(const uint64_t *__restrict__ ck, int64_t n, int b, uint64_t *__restrict__ pk,
                              uint32_t *__restrict__ pv) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  int64_t x, y, z;
  mgl_unkey(ck[t], b + 1, x, y, z);
  pk[t] = mgl_key(x >> 1, y >> 1, z >> 1, b);
  pv[t] = uint32_t(t);
}

// head flags of runs of equal keys in a sorted array
__global__ void k_mgl_heads(const uint64_t *__restrict__ k, int64_t n, uint32_t *__restrict__ head) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t < n) head[t] = (t == 0 || k[t] != k[t - 1]) ? 1u : 0u;
}

// the unique keys (pos = exclusive scan of head) and their count
__global__ void k_mgl_unique(const uint64_t *__restrict__ k, const uint32_t *__restrict__ head,
                             const uint32_t *__restrict__ pos, int64_t n, uint64_t *__restrict__ out,
                             int64_t *__restrict__ count) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  if (head[t]) out[pos[t]] = k[t];
  if (t == n - 1) *count = int64_t(pos[t] + head[t]);
}

// the six face neighbours in the MG level (-1 outside it), the count of
// faces to the outside, and the even-colour flag (parity of x + y + z)
__global__ void k_mgl_faces(const uint64_t *__restrict__ keys, int64_t n, int b, int32_t *__restrict__ nb,
                            int32_t *__restrict__ nbnd, uint32_t *__restrict__ even) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  int64_t x, y, z;
  mgl_unkey(keys[t], b, x, y, z);
  const int64_t m = (int64_t(1) << b) - 1;
  int nout = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int sg = 0; sg < 2; ++sg) {
      const int64_t dd = sg ? 1 : -1;
      const int32_t q = mgl_find(keys, n, mgl_key((x + (d == 0) * dd) & m, (y + (d == 1) * dd) & m,
                                                  (z + (d == 2) * dd) & m, b));
      nb[(2 * d + sg) * n + t] = q;
      nout += q < 0;
    }
  nbnd[t] = nout;
  even[t] = ((x + y + z) & 1) ? 0u : 1u;
}

// colour lists: even cells first, then odd, each in key order (pos = the
// exclusive scan of even; nc0 = the number of even cells)
__global__ void k_mgl_colours(const uint32_t *__restrict__ even, const uint32_t *__restrict__ pos, int64_t n,
                              int32_t *__restrict__ col, int64_t *__restrict__ nc0) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  const int64_t n0 = int64_t(pos[n - 1] + even[n - 1]);
  col[even[t] ? int64_t(pos[t]) : n0 + (t - int64_t(pos[t]))] = int32_t(t);
  if (t == 0) *nc0 = n0;
}

// children of coarse cell t (b bits) in the finer MG level (b + 1 bits),
// order (cx, cy, cz) with cz fastest
__global__ void k_mgl_children(const uint64_t *__restrict__ keys, int64_t n, int b,
                               const uint64_t *__restrict__ fkeys, int64_t nf, int32_t *__restrict__ child) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  int64_t x, y, z;
  mgl_unkey(keys[t], b, x, y, z);
  int j = 0;
  for (int cx = 0; cx < 2; ++cx)
    for (int cy = 0; cy < 2; ++cy)
      for (int cz = 0; cz < 2; ++cz, ++j)
        child[j * n + t] = mgl_find(fkeys, nf, mgl_key(2 * x + cx, 2 * y + cy, 2 * z + cz, b + 1));
}

// trilinear stencil of fine cell t (b + 1 bits) in the coarse MG level (b
// bits): entry 4a + 2b' + d for the coarse cells (X + a sx, Y + b' sy, Z + d sz)
__global__ void k_mgl_stencils(const uint64_t *__restrict__ fkeys, int64_t nf, int b,
                               const uint64_t *__restrict__ keys, int64_t n, int32_t *__restrict__ pro) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= nf) return;
  int64_t x, y, z;
  mgl_unkey(fkeys[t], b + 1, x, y, z);
  const int64_t X = x >> 1, Y = y >> 1, Z = z >> 1, m = (int64_t(1) << b) - 1;
  const int64_t sx = (x & 1) ? 1 : -1, sy = (y & 1) ? 1 : -1, sz = (z & 1) ? 1 : -1;
  for (int a = 0; a < 2; ++a)
    for (int bb = 0; bb < 2; ++bb)
      for (int d = 0; d < 2; ++d)
        pro[(4 * a + 2 * bb + d) * nf + t] =
            mgl_find(keys, n, mgl_key((X + a * sx) & m, (Y + bb * sy) & m, (Z + d * sz) & m, b));
}

// global index of the level-(L-1) cell (X, Y, Z), or -1 (no such oct)
__device__ __forceinline__ int32_t mgl_coarse_cell(HashView hv, int member, int Lc, int64_t X, int64_t Y,
                                                   int64_t Z, int N) {
  const int32_t v = hash_probe1(hv, ikey(member, Lc, uint32_t(X >> 1), uint32_t(Y >> 1), uint32_t(Z >> 1)));
  if (v < 1 || v > N) return -1;
  return 8 * (v - 1) + int32_t((X & 1) | ((Y & 1) << 1) | ((Z & 1) << 2));
}

// MG level 0: the father cell of every cell and the level-(L-1) cell across
// every face that leaves the level (-1 for the others)
__global__ void k_mgl_coarse(HashView hv, int member, int L, int N, const uint64_t *__restrict__ keys, int64_t n,
                             const int32_t *__restrict__ nb, int32_t *__restrict__ fatherg,
                             int32_t *__restrict__ acrossg, int *err) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= n) return;
  int64_t x, y, z;
  mgl_unkey(keys[t], L, x, y, z);
  const int64_t m = (int64_t(1) << L) - 1, mc = (int64_t(1) << (L - 1)) - 1;
  const int32_t f = mgl_coarse_cell(hv, member, L - 1, x >> 1, y >> 1, z >> 1, N);
  if (f < 0) atomicOr(err, kErrGrading);
  fatherg[t] = f < 0 ? 0 : f;
  for (int d = 0; d < 3; ++d)
    for (int sg = 0; sg < 2; ++sg) {
      const int k6 = 2 * d + sg;
      int32_t q = -1;
      if (nb[k6 * n + t] < 0) {
        const int64_t dd = sg ? 1 : -1;
        const int64_t X = (x + (d == 0) * dd) & m, Y = (y + (d == 1) * dd) & m, Z = (z + (d == 2) * dd) & m;
        q = mgl_coarse_cell(hv, member, L - 1, (X >> 1) & mc, (Y >> 1) & mc, (Z >> 1) & mc, N);
        if (q < 0) {
          atomicOr(err, kErrGrading);
          q = 0;
        }
      }
      acrossg[k6 * n + t] = q;
    }
}

}  // namespace amr
