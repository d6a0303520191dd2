// deposit_kernels.cuh -- Cloud-in-Cell mass deposition onto the levels of a
// mesh (paper Sec. 4, "Mass Deposition": at level l the particles of level l
// and of every finer level deposit, then the particle list is split for
// level l+1 by "host cell refined").
//
// A list holds particle indices; its length lives on the device, so the
// levels run back to back without a host round trip.  One kernel per level,
// one thread per particle of the list: the CIC weights at cell size 2^-l with
// the half-cell-shifted stencil (s = x 2^l - 1/2, i0 = floor(s), f = s - i0),
// m (wx wy) wz 2^(3l) added with one atomic per stencil cell that exists
// at level l (a cell of a real level-l oct: found in the complete base level's
// table, or in the hash table), and the particle kept for the next list when
// its host cell (the cell containing it) exists and is split.  A block's kept
// particles take one run of the next list in thread order (ballots, one atomic
// add per block): the lists are used as sets.  (Flags, a prefix sum over all
// particles and a compaction per level took seven launches and read and wrote
// every particle's flag and position four times.)
#pragma once
#include "amr_internal.cuh"
#include "cic_weights.cuh"

namespace amr {

// the source cell (i, j, k) (unmasked), the 8 contributions of a particle at
// level l and its host cell h (unmasked)
__device__ __forceinline__ void level_stencil(float x, float y, float z, float m, int l, int (&i0)[3], int (&h)[3],
                                              float (&w)[8]) {
  const float n = float(1 << l);
  const float pos[3] = {x, y, z};
  float wd[3][2];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float s = pos[d] * n - 0.5f;
    const float fl = floorf(s);
    const float f = s - fl;
    i0[d] = __float2int_rd(fl);
    h[d] = __float2int_rd(pos[d] * n);
    wd[d][0] = 1.0f - f;
    wd[d][1] = f;
  }
  const float scale = n * n * n;  // 1 / dx^3, exact
#pragma unroll
  for (int c = 0; c < 8; ++c) w[c] = (m * ((wd[0][c & 1] * wd[1][(c >> 1) & 1]) * wd[2][c >> 2])) * scale;
}
__device__ __forceinline__ void level_stencil(double x, double y, double z, double m, int l, int (&i0)[3],
                                              int (&h)[3], double (&w)[8]) {
  if (cic_in_range(x, y, z, m)) {  // on the integer pipes
    const uint64_t b[3] = {uint64_t(__double_as_longlong(x)), uint64_t(__double_as_longlong(y)),
                           uint64_t(__double_as_longlong(z))};
    uint64_t wb[8];
    cic_weights_int(b[0], b[1], b[2], uint64_t(__double_as_longlong(m)), l, i0[0], i0[1], i0[2], wb);
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = __longlong_as_double((long long)wb[c]);
#pragma unroll
    for (int d = 0; d < 3; ++d) h[d] = cic_floor_int(b[d], l);
    return;
  }
  const double n = double(1 << l);
  const double pos[3] = {x, y, z};
  double wd[3][2];
  for (int d = 0; d < 3; ++d) {
    const double s = pos[d] * n - 0.5;
    const double fl = floor(s);
    const double f = s - fl;
    i0[d] = int(int64_t(fl));
    h[d] = int(int64_t(floor(pos[d] * n)));
    wd[d][0] = 1.0 - f;
    wd[d][1] = f;
  }
  const double scale = ldexp(1.0, 3 * l);
  for (int c = 0; c < 8; ++c) w[c] = (m * ((wd[0][c & 1] * wd[1][(c >> 1) & 1]) * wd[2][c >> 2])) * scale;
}

// the base level is complete: a table from oct coordinates to oct index
// replaces the hash probes there
__global__ void k_base_table(const uint64_t *__restrict__ key, int lo, int64_t nb, int lmin, int32_t *btab) {
  const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (t >= nb) return;
  const int o = lo + int(t);
  const uint64_t k = key[o];
  const int64_t side = int64_t(1) << (lmin - 1);
  btab[(int64_t(ikey_x(k)) * side + ikey_y(k)) * side + ikey_z(k)] = o;
}

// where the octs of a level are found: by coordinates in the base table, or in
// the hash table; -1: no real oct
struct OctFinder {
  const int32_t *btab;  // the base level's table, or NULL
  HashView hv;
  int member, l, N;
  __device__ __forceinline__ int operator()(uint32_t i, uint32_t j, uint32_t k) const {
    if (btab) return __ldg(btab + (((int64_t(i) << (l - 1)) + j) << (l - 1)) + k);
    const int32_t v = hash_probe1(hv, ikey(member, l, i, j, k));
    return v >= 1 && v <= N ? v - 1 : -1;
  }
};

// deposit of a list's particles at level l (list NULL: particles 0 .. count[l] - 1)
// and, with next, the next level's list and its length count[l + 1] (zero before)
template <class T>
__global__ void __launch_bounds__(256) k_deposit_level(OctFinder find, const uint32_t *__restrict__ son,
                                                       const T *__restrict__ px, const T *__restrict__ py,
                                                       const T *__restrict__ pz, const T *__restrict__ pm,
                                                       const uint32_t *__restrict__ list, int64_t *count, T *rho,
                                                       uint32_t *__restrict__ next) {
  __shared__ int64_t run;
  __shared__ int wkeep[8];
  const int64_t n = count[find.l];
  const uint32_t mask = (1u << find.l) - 1u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t t0 = blockIdx.x * int64_t(256); t0 < n; t0 += gridDim.x * int64_t(256)) {
    const int64_t t = t0 + threadIdx.x;
    bool keep = false;
    uint32_t p = 0;
    if (t < n) {
      p = list ? list[t] : uint32_t(t);
      int i0[3], h[3];
      T w[8];
      level_stencil(px[p], py[p], pz[p], pm[p], find.l, i0, h, w);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint32_t X = uint32_t(i0[0] + (c & 1)) & mask, Y = uint32_t(i0[1] + ((c >> 1) & 1)) & mask,
                       Z = uint32_t(i0[2] + (c >> 2)) & mask;
        const int o = find(X >> 1, Y >> 1, Z >> 1);
        if (o >= 0) atomicAdd(rho + 8 * int64_t(o) + int((X & 1) + 2 * (Y & 1) + 4 * (Z & 1)), w[c]);
      }
      if (next) {
        const uint32_t X = uint32_t(h[0]) & mask, Y = uint32_t(h[1]) & mask, Z = uint32_t(h[2]) & mask;
        const int o = find(X >> 1, Y >> 1, Z >> 1);
        keep = o >= 0 && ((__ldg(son + o) >> ((X & 1) + 2 * (Y & 1) + 4 * (Z & 1))) & 1u);
      }
    }
    if (!next) continue;
    const unsigned ballot = __ballot_sync(0xFFFFFFFFu, keep);
    if (lane == 0) wkeep[warp] = __popc(ballot);
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      before += q < warp ? wkeep[q] : 0;
      all += wkeep[q];
    }
    if (threadIdx.x == 0 && all)
      run = int64_t(atomicAdd(reinterpret_cast<unsigned long long *>(count + find.l + 1), (unsigned long long)all));
    __syncthreads();
    if (keep) next[run + before + __popc(ballot & ((1u << lane) - 1u))] = p;
  }
}

}  // namespace amr
