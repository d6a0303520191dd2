// hydro_kernels.cuh -- one AMR level step of compressible Euler (paper Sec. 3:
// MUSCL-Hancock predictor-corrector with an HLLC Riemann solver and two
// ghost cells per side; Sec. 2.3 ghost octs; Table 1 stages godunov /
// set uold / upload), as non-redundant per-cell passes:
//
//   k_ghost_prim  ghost octs of the level from their father cell (minmod) and
//                 primitive variables of every real and ghost cell
//   k_predict     limited slopes and the Hancock half-step, once per cell
//   k_flux        one HLLC flux per face (owned by the cell on its minus side)
//   k_update      conservative update of leaf cells + pending reflux; father
//                 cell = mean of its 8 children; fixed-order sum of
//                 coarse-fine fluxes for the coarse cells
//
// FP32 takes three: k_prolong (ghost octs, and the previous level step's
// fixed-order sums of coarse-fine fluxes), k_predict_u (primitives formed from U
// as they are needed) and k_flux_update (flux, update, father cells).
//
// The paper's kernels gather a 6x6x6 stencil per oct and recompute the
// slopes and predictor of its ghost ring (8x work per cell at nsubgrid=1).
// On GB300 the FP64 rate is far below the memory rate, so each cell's
// predictor and each face's Riemann solve is computed exactly once and the
// intermediate states go through L2/HBM instead.
//
// Every kernel is persistent over a flattened work list of tiles, each tile
// one block's worth of items of one (member mesh, level) segment, so one
// launch advances a level of many meshes at once.
#pragma once
#include "fp64_int.cuh"
#include "hydro_args.cuh"

namespace amr {

// ---------------------------------------------------------------------------
// arithmetic helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double minmod(double a, double b) {
  // 0 for opposite signs or a zero argument, else the argument of smaller
  // magnitude; decided on the bit patterns (integer pipes, no FP64 issue):
  // the bits shifted left by one drop the sign and order the magnitudes
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  const unsigned long long ma = (unsigned long long)ia << 1, mb = (unsigned long long)ib << 1;
  if (((ia ^ ib) < 0) | (ma == 0) | (mb == 0)) return 0.0;
  return ma < mb ? a : b;
}
// FP32: the definition as written, 0 when a b <= 0 (the FP32 pipes have room)
__device__ __forceinline__ float minmod(float a, float b) {
  const float m = fabsf(a) < fabsf(b) ? a : b;
  return a * b > 0.0f ? m : 0.0f;
}
// FP64 compares, min and max decided on the bit patterns: GB300's FP64 pipe
// is 1/64 of its FP32 rate and these kernels are bound by it, while the
// integer pipes have room.  ord() maps a non-NaN double to a signed integer
// of the same order (-0 just below +0); a NaN argument propagates instead of
// being dropped (the time-step reduction reports it).
__device__ __forceinline__ long long ord(double x) {
  const long long i = __double_as_longlong(x);
  return i ^ ((i >> 63) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ double vmax(double a, double b) { return ord(a) < ord(b) ? b : a; }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double vmin(double a, double b) { return ord(b) < ord(a) ? b : a; }
__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
// x > 0
__device__ __forceinline__ bool pos(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool pos(float x) { return x > 0.0f; }
// x is neither infinite nor NaN (exponent field not all ones)
__device__ __forceinline__ bool finite_bits(double x) {
  return ((__double_as_longlong(x) >> 52) & 0x7FF) != 0x7FF;
}
__device__ __forceinline__ bool finite_bits(float x) {
  return ((__float_as_int(x) >> 23) & 0xFF) != 0xFF;
}
// a > b for a, b >= 0
__device__ __forceinline__ bool gt_nonneg(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b);
}
__device__ __forceinline__ bool gt_nonneg(float a, float b) { return __float_as_int(a) > __float_as_int(b); }

// 1/x from the hardware's approximate reciprocal r (relative error near
// 2^-20 on GB300, measured) by one third-order step of the series
// 1/x = r / (1 - e) = r (1 + e + e^2 + ...), e = 1 - x r: the error drops to
// about e^3 (2^-60), so the result is within an ulp or two of 1/x, as two
// Newton steps would give, with three FMAs instead of four (checked against
// the correctly rounded quotient by the parity tests).  Operands here are
// positive, finite and normal (densities, sums of rho |u - S|, wave-speed
// gaps), so the flush-to-zero form is safe.
__device__ __forceinline__ double rcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1/sqrt(x) from the hardware approximation y (x y^2 within about 2^-19 of
// 1, measured) by one third-order step of the binomial series
// (1 - h)^(-1/2) = 1 + h/2 + 3h^2/8 + ..., h = 1 - x y^2: the error drops to
// about h^3, double precision in five operations (two Newton steps take
// seven).  x is a positive normal number here (gamma p rho).
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = fma(-x, y * y, 1.0);
  return fma(y, h * fma(0.375, h, 0.5), y);
}
__device__ __forceinline__ float rsqrt_nr(float x) { return rsqrtf(x); }

// sqrt(c2) of the time-step reduction: c2 rsqrt(c2) in FP64 (within an ulp
// or two of the correctly rounded root; 0 for c2 = 0; NaN propagates), the
// library's sqrtf in FP32
__device__ __forceinline__ double sound_speed(double c2) { return c2 > 0.0 ? c2 * rsqrt_nr(c2) : sqrt(c2); }
__device__ __forceinline__ float sound_speed(float c2) { return sqrtf(c2); }

// FP32 image of a state component: exact for an FP32 state; for FP64 the
// bits are truncated on the integer pipes (relative error below 2^-23, no
// conversion instruction: those run on the FP64 pipe), magnitudes below
// 2^-126 give 0 and above 2^128 infinity
template <class T>
__device__ __forceinline__ float to_f32(T x) {
  return float(x);
}
template <>
__device__ __forceinline__ float to_f32<double>(double x) {
  const uint64_t b = uint64_t(__double_as_longlong(x));
  const uint32_t sign = uint32_t(b >> 32) & 0x80000000u;
  const int e = int((b >> 52) & 0x7FF);
  if (e < 1023 - 126) return __uint_as_float(sign);
  if (e > 1023 + 127) return __uint_as_float(sign | 0x7F800000u);
  return __uint_as_float(sign | (uint32_t(e - 896) << 23) | uint32_t((b >> 29) & 0x7FFFFFu));
}

// ---------------------------------------------------------------------------
// segment context: what a thread needs to know about its (member, level)
// ---------------------------------------------------------------------------
template <class T>
struct SegCtx {
  int lo, nl, clo, ncl, base, flags;
  T gamma, gm1, igm1, smallr, smallp, dtdx;  // gm1 = gamma - 1, igm1 = 1 / gm1
};

__device__ __forceinline__ double seg_dtdx(const StepArgs<double> &a, const Seg &s) {
  return a.dtdx_dev ? __ldg(a.dtdx_dev + s.member) : ldexp(a.dt_host, s.level);
}
__device__ __forceinline__ float seg_dtdx(const StepArgs<float> &a, const Seg &s) {
  // scaling by a power of two is exact, so this is float(dt 2^l)
  return a.dtdxf_dev ? __ldg(a.dtdxf_dev + s.member) : ldexpf(float(a.dt_host), s.level);
}

template <class T>
__device__ __forceinline__ SegCtx<T> seg_ctx(const StepArgs<T> &a, const Seg &s) {
  SegCtx<T> c;
  c.lo = s.lo;
  c.nl = s.nl;
  c.clo = s.clo;
  c.ncl = s.ncl;
  c.base = s.base;
  c.flags = s.flags;
  c.gamma = __ldg(a.mgamma + s.member);
  c.igm1 = __ldg(a.migm1 + 2 * s.member);
  c.gm1 = __ldg(a.migm1 + 2 * s.member + 1);
  c.smallr = __ldg(a.msmallr + s.member);
  c.smallp = __ldg(a.msmallp + s.member);
  c.dtdx = seg_dtdx(a, s);
  return c;
}

// the segment's context; false: nothing to do (a finished member)
template <class T>
__device__ __forceinline__ bool open_segment(const StepArgs<T> &a, int seg, SegCtx<T> &s) {
  const Seg sg = seg_at(a.tiles, seg);
  if (a.mact && !__ldg(a.mact + sg.member)) return false;
  s = seg_ctx(a, sg);
#ifdef AMR_CHECKED
  // the segment's local cells must fit the scratch arrays
  if (s.base < 0 || s.base + 8 * (s.nl + s.ncl) > a.LS) {
    atomicOr(a.err, kErrIndex);
    return false;
  }
#endif
  return true;
}

// persistent loop over the launch's tiles: body(ctx, item) for every thread of a
// tile's block, also beyond the segment's items (bodies work by whole warps)
template <class T, class Body>
__device__ __forceinline__ void warp_tile_loop(const StepArgs<T> &a, Body body) {
  for (int ti = blockIdx.x; ti < a.tiles.ntiles; ti += gridDim.x) {
    const Tile td = tile_at(a.tiles, ti);
    SegCtx<T> s;
    if (open_segment(a, td.seg, s)) body(s, td.start + int(threadIdx.x));
  }
}

// the same for every item of the tile that lies inside the segment's domain of
// `size(ctx)` items
template <class T, class Size, class Body>
__device__ __forceinline__ void tile_loop(const StepArgs<T> &a, Size size, Body body) {
  warp_tile_loop(a, [&](const SegCtx<T> &s, int item) {
    if (item < size(s)) body(s, item);
  });
}

// extended oct index of local oct index q, and back
template <class T>
__device__ __forceinline__ int ext_of_local(const StepArgs<T> &a, const SegCtx<T> &s, int q) {
  return q < s.nl ? s.lo + q : a.N + s.clo + (q - s.nl);
}
template <class T>
__device__ __forceinline__ int local_of_ext(const StepArgs<T> &a, const SegCtx<T> &s, int e) {
  return e < a.N ? e - s.lo : e - a.N - s.clo + s.nl;
}

// local index of the face neighbour of local cell t (extended oct e, cell c)
// along axis d on side `plus`; -1 when the neighbouring oct does not exist
template <class T>
__device__ __forceinline__ int nbr_local(const StepArgs<T> &a, const SegCtx<T> &s, int t, int e,
                                         int c, int d, int plus) {
  const int bit = 1 << d;
  if (((c >> d) & 1) != plus) return t ^ bit;
  const int32_t ne = __ldg(a.fnb + (2 * d + plus) * int64_t(a.NE) + e);
  if (ne < 0) return -1;
  // a face neighbour is in the same (member, level) segment: else "none"
  const int q = int(checked(local_of_ext(a, s, ne), 0, s.nl + s.ncl, a.err, -1));
  return q < 0 ? -1 : 8 * q + (c ^ bit);
}

template <class T>
__device__ __forceinline__ bool cell_is_split(const StepArgs<T> &a, const SegCtx<T> &s, int t) {
  const int q = t >> 3;
  if (q >= s.nl) return false;  // ghost cells are leaves
  return (__ldg(a.son + s.lo + q) >> (t & 7)) & 1u;
}

// R(X) += sum of the 24 slots of ghost oct g (X its father cell), in slot
// order (direction -x,+x,-y,+y,-z,+z seen from X, then fine face)
template <class T>
__device__ __forceinline__ void reflux_sum(const StepArgs<T> &a, int v, int g) {
  const T *cv = a.C + v * a.CS + 24 * int64_t(g);
  T *Rv = a.Rc + v * int64_t(a.NC) + g;
  constexpr int W = 16 / sizeof(T);  // 16 bytes per load: a ghost oct's slots are 192 (96) bytes in a row
  struct alignas(16) Slots {
    T x[W];
  } sl[24 / W];
#pragma unroll
  for (int k = 0; k < 24 / W; ++k) sl[k] = reinterpret_cast<const Slots *>(cv)[k];
  T acc = *Rv;
#pragma unroll
  for (int k = 0; k < 24; ++k) acc += sl[k / W].x[k % W];
  *Rv = acc;
}

// the reflux sums of a list's ghost octs; domain: 5 ncl (if kSegReflux)
template <class T>
__device__ __forceinline__ void reflux_tile(const StepArgs<T> &a, const TileList &l, int ti) {
  const Tile td = tile_at(l, ti);
  const Seg s = seg_at(l, td.seg);
  if (a.mact && !__ldg(a.mact + s.member)) return;  // finished member
  const int q = td.start + threadIdx.x;
  if (!(s.flags & kSegReflux) || q >= 5 * s.ncl) return;
  const int v = q / s.ncl;
  reflux_sum(a, v, s.clo + (q - v * s.ncl));
}
template <class T>
__global__ void k_reflux(StepArgs<T> a) {
  for (int ti = blockIdx.x; ti < a.tiles.ntiles; ti += gridDim.x) reflux_tile(a, a.tiles, ti);
}

// ---------------------------------------------------------------------------
// ghost octs: child = U_C + sum_d (+-1/4) minmod(U(C+e_d)-U(C), U(C)-U(C-e_d))
// domain: 5 * ncl (variable, ghost oct)
// ---------------------------------------------------------------------------
// pend: a list whose fluxes were solved by the previous level step and whose
// reflux sums are still to be formed (FP32: the slots are written by the last
// kernel of a level step); they touch other data, so they ride along here
template <class T>
__global__ void k_prolong(StepArgs<T> a, TileList pend) {
  for (int ti = blockIdx.x; ti < pend.ntiles; ti += gridDim.x) reflux_tile(a, pend, ti);
  tile_loop(a, [](const SegCtx<T> &s) { return 5 * s.ncl; }, [&](const SegCtx<T> &s, int q) {
    const int v = q / s.ncl;
    const int cs = s.clo + (q - v * s.ncl);
    const T *Uv = a.U + v * a.S;
    T src[7];
#pragma unroll
    for (int k = 0; k < 7; ++k)
      src[k] = Uv[checked(__ldg(a.csrc + k * int64_t(a.NC) + cs), 0, 8 * int64_t(a.NE), a.err)];
    const T uc = src[0];
    const T sx = minmod(src[2] - uc, uc - src[1]);
    const T sy = minmod(src[4] - uc, uc - src[3]);
    const T sz = minmod(src[6] - uc, uc - src[5]);
    T *dst = a.U + v * a.S + 8 * int64_t(a.N + cs);
    const T h = T(0.25);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const T hx = (c & 1) ? h : -h, hy = (c & 2) ? h : -h, hz = (c & 4) ? h : -h;
      dst[c] = ((uc + hx * sx) + hy * sy) + hz * sz;
    }
  });
}

// ---------------------------------------------------------------------------
// primitives of every real and ghost cell; domain: 8 (nl + ncl)
// ---------------------------------------------------------------------------
// The plain products of the FP64 arithmetic: every operation rounded as written,
// so that a result has the same bits in every kernel, on the FP64 pipe (MulFp64)
// or on the integer pipes (MulInt), which are otherwise idle.  mul0 is for operands that can be
// tiny or zero (a product below the normal range is zero in both).
struct MulFp64 {
  static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __device__ __forceinline__ double mul0(double a, double b) { return mul_fp64_0(a, b); }
  static __device__ __forceinline__ double half(double a) { return __dmul_rn(0.5, a); }
};
struct MulInt {
  static __device__ __forceinline__ double mul(double a, double b) { return mul_int(a, b); }
  static __device__ __forceinline__ double mul0(double a, double b) { return mul_int0(a, b); }
  static __device__ __forceinline__ double half(double a) {  // exponent - 1
    return __hiloint2double(__double2hiint(a) - (1 << 20), __double2loint(a));
  }
};

// p <- max(p, r smallp), r > 0.  FP64: when p's exponent lies two above that
// of r smallp the floor cannot act, and its product is not formed
__device__ __forceinline__ float floor_p(float p, float r, float smallp) { return vmax(p, r * smallp); }
__device__ __forceinline__ double floor_p(double p, double r, double smallp) {
  if (__double2hiint(p) <= __double2hiint(r) + (__double2hiint(smallp) - (1021 << 20))) p = vmax(p, r * smallp);
  return p;
}

// primitives (rho, u, v, w, p) of the conservative state (u0..u4), with the
// density and pressure floors
__device__ __forceinline__ void prim_of(const SegCtx<float> &s, float u0, float u1, float u2, float u3, float u4,
                                        float (&w)[5]) {
  const float r = vmax(u0, s.smallr);
  const float ir = rcp(r);
  const float vx = u1 * ir, vy = u2 * ir, vz = u3 * ir;
  const float ek = 0.5f * r * ((vx * vx + vy * vy) + vz * vz);
  w[0] = r;
  w[1] = vx;
  w[2] = vy;
  w[3] = vz;
  w[4] = vmax(s.gm1 * (u4 - ek), r * s.smallp);
}
template <class O>
__device__ __forceinline__ void prim_fp64(const SegCtx<double> &s, double r, double u1, double u2, double u3,
                                          double u4, double (&w)[5]) {
  const double ir = rcp(r);
  const double vx = O::mul0(u1, ir), vy = O::mul0(u2, ir), vz = O::mul0(u3, ir);
  const double ek = O::mul0(O::half(r), __fma_rn(vz, vz, __fma_rn(vy, vy, O::mul0(vx, vx))));
  w[0] = r;
  w[1] = vx;
  w[2] = vy;
  w[3] = vz;
  w[4] = floor_p(O::mul0(s.gm1, __dadd_rn(u4, -ek)), r, s.smallp);
}
// FP64: 6 of 12 operations are products that the integer pipes take when the
// warp's densities lie in [2^-100, 2^100), momenta below 2^150 and energies
// below 2^300 (nothing overflows then); 14 on the FP64 pipe otherwise
__device__ __forceinline__ void prim_of(const SegCtx<double> &s, double u0, double u1, double u2, double u3,
                                        double u4, double (&w)[5]) {
  const double r = vmax(u0, s.smallr);
  const bool safe = within<100>(r) && below<150>(u1) && below<150>(u2) && below<150>(u3) && below<300>(u4) &&
                    within<100>(s.gm1);
  if (__all_sync(__activemask(), safe))
    prim_fp64<MulInt>(s, r, u1, u2, u3, u4, w);
  else
    prim_fp64<MulFp64>(s, r, u1, u2, u3, u4, w);
}

template <class T>
__device__ __forceinline__ void prim_at(const StepArgs<T> &a, const SegCtx<T> &s, int t,
                                        T (&w)[5]) {
  const int g = 8 * ext_of_local(a, s, t >> 3) + (t & 7);
  prim_of(s, a.U[g], a.U[a.S + g], a.U[2 * a.S + g], a.U[3 * a.S + g], a.U[4 * a.S + g], w);
}

// FP64: ghost octs (as k_prolong) and the primitives of every real and ghost
// cell in one pass; thread per cell, an oct in 8 neighbouring lanes.  A ghost
// oct's 15 slopes (variable, axis) are formed once, two per lane, and shared by
// its cells.
__global__ void __launch_bounds__(512, 3) k_ghost_prim(StepArgs<double> a) {
  extern __shared__ double slopes[];  // [5 d + v][oct of the block], 16 bytes per thread
  const int qb = threadIdx.x >> 3, nq = blockDim.x >> 3;
  warp_tile_loop(a, [&](const SegCtx<double> &s, int t) {
    const int q = t >> 3, c = t & 7;
    const bool on = t < 8 * (s.nl + s.ncl), ghost = on && q >= s.nl;
    const int cs = s.clo + (q - s.nl);
    const int64_t g = 8 * int64_t(ext_of_local(a, s, q)) + c;
    double u[5];
    if (ghost) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = c + 8 * h;  // slope 5 d + v
        if (k < 15) {
          const int d = k / 5;
          const double *Uv = a.U + (k - 5 * d) * a.S;
          auto at = [&](int j) {
            return Uv[checked(__ldg(a.csrc + j * int64_t(a.NC) + cs), 0, 8 * int64_t(a.NE), a.err)];
          };
          const double uc = at(0), um = at(1 + 2 * d), up = at(2 + 2 * d);
          slopes[k * nq + qb] = minmod(up - uc, uc - um);
        }
      }
      const int64_t f = checked(__ldg(a.csrc + cs), 0, 8 * int64_t(a.NE), a.err);
#pragma unroll
      for (int v = 0; v < 5; ++v) u[v] = a.U[v * a.S + f];
    } else if (on) {
#pragma unroll
      for (int v = 0; v < 5; ++v) u[v] = a.U[v * a.S + g];
    }
    if (__any_sync(0xFFFFFFFFu, ghost)) {
      __syncwarp();
      if (ghost) {
        const double hx = (c & 1) ? 0.25 : -0.25, hy = (c & 2) ? 0.25 : -0.25, hz = (c & 4) ? 0.25 : -0.25;
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          u[v] = ((u[v] + hx * slopes[v * nq + qb]) + hy * slopes[(5 + v) * nq + qb]) + hz * slopes[(10 + v) * nq + qb];
          a.U[v * a.S + g] = u[v];
        }
      }
      __syncwarp();
    }
    if (on) {
      double w[5];
      prim_of(s, u[0], u[1], u[2], u[3], u[4], w);
      const int o = s.base + t;
#pragma unroll
      for (int v = 0; v < 5; ++v) a.W[v * a.LS + o] = w[v];
    }
  });
}

// ---------------------------------------------------------------------------
// limited slopes and Hancock predictor W* = W + dt/(2dx) S(W, dW)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void predictor(const SegCtx<float> &s, const float (&w)[5], const float (&dw)[3][5],
                                          float (&ws)[5]) {
  const float r = w[0], p = w[4], g = s.gamma;
  const float ir = rcp(r);
  const float gp = g * p;
  float src[5];
  src[0] = -(((w[1] * dw[0][0] + r * dw[0][1]) + (w[2] * dw[1][0] + r * dw[1][2])) +
             (w[3] * dw[2][0] + r * dw[2][3]));
#pragma unroll
  for (int k = 0; k < 3; ++k)
    src[1 + k] =
        -((w[1] * dw[0][1 + k] + w[2] * dw[1][1 + k]) + w[3] * dw[2][1 + k]) - dw[k][4] * ir;
  src[4] = -(((w[1] * dw[0][4] + gp * dw[0][1]) + (w[2] * dw[1][4] + gp * dw[1][2])) +
             (w[3] * dw[2][4] + gp * dw[2][3]));
  const float hdt = 0.5f * s.dtdx;
#pragma unroll
  for (int v = 0; v < 5; ++v) ws[v] = w[v] + hdt * src[v];
}
// FP64: the velocity divergence is formed once for the density and the
// pressure, and each source is one chain of FMAs: 31 operations (42 with the
// terms of each direction on their own), 6 of them products for the integer
// pipes
template <class O>
__device__ __forceinline__ void predictor_fp64(const SegCtx<double> &s, const double (&w)[5],
                                               const double (&dw)[3][5], double (&ws)[5]) {
  const double ir = rcp(w[0]), gp = O::mul(s.gamma, w[4]);
  const double div = __dadd_rn(__dadd_rn(dw[0][1], dw[1][2]), dw[2][3]);
  const int hd = __double2hiint(s.dtdx);  // -dt/(2dx): exponent - 1, on the integer pipe
  const double mh = (hd & 0x7FF00000) > (1 << 20)
                        ? __hiloint2double(int(uint32_t(hd - (1 << 20)) ^ 0x80000000u), __double2loint(s.dtdx))
                        : -0.5 * s.dtdx;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double adv = __fma_rn(w[3], dw[2][v], __fma_rn(w[2], dw[1][v], O::mul0(w[1], dw[0][v])));
    const double src = v == 0   ? __fma_rn(w[0], div, adv)
                       : v == 4 ? __fma_rn(gp, div, adv)
                                : __fma_rn(dw[v < 1 || v > 3 ? 0 : v - 1][4], ir, adv);
    ws[v] = __fma_rn(mh, src, w[v]);
  }
}
__device__ __forceinline__ void predictor(const SegCtx<double> &s, const double (&w)[5], const double (&dw)[3][5],
                                          double (&ws)[5]) {
  bool safe = within<100>(w[0]) && within<100>(w[4]) && below<150>(w[1]) && within<100>(s.gamma);
#pragma unroll
  for (int v = 0; v < 5; ++v) safe = safe && below<300>(dw[0][v]);
  if (__all_sync(__activemask(), safe))
    predictor_fp64<MulInt>(s, w, dw, ws);
  else
    predictor_fp64<MulFp64>(s, w, dw, ws);
}

// The predictor's results: FP64 as 20 arrays; FP32 as five arrays of four values
// each (W* without pressure; the pressure and its three slopes; the other slopes per
// axis), so that a face's side takes three loads instead of ten.
__device__ __forceinline__ void store_q(const StepArgs<double> &a, int o, const double (&ws)[5],
                                        const double (&dw)[3][5]) {
#pragma unroll
  for (int v = 0; v < 5; ++v) a.Q[v * a.LS + o] = ws[v];
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int v = 0; v < 5; ++v) a.Q[(5 + 5 * d + v) * a.LS + o] = dw[d][v];
}
__device__ __forceinline__ void store_q(const StepArgs<float> &a, int o, const float (&ws)[5],
                                        const float (&dw)[3][5]) {
  float4 *q = reinterpret_cast<float4 *>(a.Q) + o;
  q[0] = make_float4(ws[0], ws[1], ws[2], ws[3]);
  q[a.LS] = make_float4(ws[4], dw[0][4], dw[1][4], dw[2][4]);
#pragma unroll
  for (int d = 0; d < 3; ++d) q[(2 + d) * a.LS] = make_float4(dw[d][0], dw[d][1], dw[d][2], dw[d][3]);
}
// one side of a face normal to axis D: W* + h dW of local cell o (h = 1/2: its plus
// face, -1/2: its minus face).  Q is read-only while faces are solved
__device__ __forceinline__ void load_side(const StepArgs<double> &a, int o, int D, double h, double (&q)[5]) {
  const double *Q = a.Q + o, *S = Q + (5 + 5 * D) * a.LS;
#pragma unroll
  for (int v = 0; v < 5; ++v) q[v] = __ldg(Q + v * a.LS) + h * __ldg(S + v * a.LS);
}
__device__ __forceinline__ void side_of(const float4 &w, const float4 &p, const float4 &d, int D, float h,
                                        float (&q)[5]) {
  q[0] = w.x + h * d.x;
  q[1] = w.y + h * d.y;
  q[2] = w.z + h * d.z;
  q[3] = w.w + h * d.w;
  q[4] = p.x + h * (D == 0 ? p.y : D == 1 ? p.z : p.w);
}
__device__ __forceinline__ void load_side(const StepArgs<float> &a, int o, int D, float h, float (&q)[5]) {
  const float4 *Q = reinterpret_cast<const float4 *>(a.Q) + o;
  side_of(__ldg(Q), __ldg(Q + a.LS), __ldg(Q + (2 + D) * a.LS), D, h, q);
}

// FP64: one thread per cell, an oct in 8 neighbouring lanes.  Along each axis a
// cell has one neighbour inside its oct and one outside; the inner difference
// is the same number for both cells of a pair, so the pair's lanes each form it
// for half of the variables and exchange it (24 differences per cell instead
// of 30, and 15 loads instead of 30).  Bound by the FP64 pipe: 49 operations
// per cell, 72 with every difference and product on it.  Level 7 of the Sedov blast
// 196 us (87 % of the FP64 pipe; 281 with 72 operations); all indices and loads come
// first: waiting per axis, a coarse step of the 3-6 random mesh takes 208 us of it
// instead of 140.
__device__ __forceinline__ double shfl_xor_f64(unsigned mask, double x, int lanes) {
  const int lo = __shfl_xor_sync(mask, __double2loint(x), lanes), hi = __shfl_xor_sync(mask, __double2hiint(x), lanes);
  return __hiloint2double(hi, lo);
}
__global__ void k_predict(StepArgs<double> a) {
  warp_tile_loop(a, [&](const SegCtx<double> &s, int t) {  // tiles start at multiples of 8: octs are whole
    const bool on = t < 8 * (s.nl + s.ncl);
    const unsigned lanes = __ballot_sync(0xFFFFFFFFu, on);
    if (!on) return;
    const int e = ext_of_local(a, s, t >> 3);
    const int c = t & 7;
    const int o = s.base + t;
    // the three outer neighbours, or the cell itself (outer ring of a ghost oct,
    // slopes never used): all addresses before the first wait
    int out[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int to = nbr_local(a, s, t, e, c, d, (c >> d) & 1);
      out[d] = to >= 0 ? s.base + to : o;
    }
    double w[5], dw[3][5], ws[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) w[v] = a.W[v * a.LS + o];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int v = 0; v < 5; ++v) dw[d][v] = a.W[v * a.LS + out[d]];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int bit = 1 << d;
      const bool up = c & bit;  // the pair's cell on the plus side
      double in[5];             // inner differences, plus side minus minus side
#pragma unroll
      for (int v = 0; v < 4; v += 2) {  // the minus side's lane forms v, the plus side's v + 1
        const double got = shfl_xor_f64(lanes, up ? w[v] : w[v + 1], bit);
        const double mine = (up ? w[v + 1] : got) - (up ? got : w[v]);
        const double other = shfl_xor_f64(lanes, mine, bit);
        in[v] = up ? other : mine;
        in[v + 1] = up ? mine : other;
      }
      const double got = shfl_xor_f64(lanes, w[4], bit);
      in[4] = (up ? w[4] : got) - (up ? got : w[4]);
#pragma unroll
      for (int v = 0; v < 5; ++v) dw[d][v] = minmod((up ? dw[d][v] : w[v]) - (up ? w[v] : dw[d][v]), in[v]);
    }
    predictor(s, w, dw, ws);
    store_q(a, o, ws, dw);
  });
}

// FP32: primitives derived from U directly (no W array): the cell's own and its
// three outer neighbours' are formed, the three inner ones come from the lanes of
// its oct (four conversions and 20 gathered loads per cell instead of seven
// and 35).  128^3 uniform 48 us (53 at 40 registers with the neighbours one after the
// other), of which 31 are its 100 bytes per cell.
__global__ void __launch_bounds__(512, 2) k_predict_u(StepArgs<float> a) {
  warp_tile_loop(a, [&](const SegCtx<float> &s, int t) {  // tiles start at multiples of 8: octs are whole
    const bool on = t < 8 * (s.nl + s.ncl);
    const unsigned lanes = __ballot_sync(0xFFFFFFFFu, on);
    if (!on) return;
    const int e = ext_of_local(a, s, t >> 3);
    const int c = t & 7;
    // the three outer neighbours, or the cell itself (outer ring of a ghost oct, slopes
    // never used): all addresses before the first wait
    int out[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int to = nbr_local(a, s, t, e, c, d, (c >> d) & 1);
      out[d] = to >= 0 ? to : t;
    }
    float w[5], dw[3][5], ws[5];
    prim_at(a, s, t, w);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const bool up = (c >> d) & 1;  // the pair's cell on the plus side
      float wo[5];
      prim_at(a, s, out[d], wo);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const float wi = __shfl_xor_sync(lanes, w[v], 1 << d);
        dw[d][v] = minmod((up ? wo[v] : wi) - w[v], w[v] - (up ? wi : wo[v]));
      }
    }
    predictor(s, w, dw, ws);
    store_q(a, s.base + t, ws, dw);
  });
}

// ---------------------------------------------------------------------------
// HLLC flux across a face from the two sides' density r, normal velocity u,
// transverse velocities a and b, pressure p (L, R): S_L = min(u) - max(c),
// S_R = max(u) + max(c); star speed and pressure from the two-wave HLL jump
// conditions; physical flux of the state sampled at x/t = 0 (Toro's HLLC);
// transverse velocities from the upwind side K.
//
// FP64.  max(c): c^2 = gamma p / rho compared by cross-multiplication, then for
// the larger side c = a / sqrt(a rho), a = gamma p: one reciprocal square root
// (by the series of rsqrt_nr) instead of a reciprocal and a square root.  With
// these wave speeds u_L - S_L = S_R - u_R = e = max(c) + max(u_L - u_R, 0), so
//   u* = (e (rho_L u_L + rho_R u_R) + p_L - p_R) / (e (rho_L + rho_R))
//   p* = p_j -+ rho_j e (u* - u_j), the same from both sides: j is the lighter
//        one, whose terms do not cancel
// K = L when u* > 0 (S_L > 0 implies it: u* - S_L is at least max(c) (1 -
// 1/gamma)); K's star state is taken when S_L <= 0 (left) or S_R > 0 (right).
// Selected without divergent branches: the side's state and energy, then one
// star state (unused in the supersonic cases).  21 products, 27 FMAs and 8 sums
// per face (the products of rho (u - S) per side, and p* from both sides: 67
// FP64 instructions); its rounding errors against extended precision are those
// of that form (1.04-2.05 against 1.09-2.01 units of 1e-16 of the rms flux over
// smooth, rough, shock, hypersonic and density-contrast faces).
// ---------------------------------------------------------------------------
template <class O>
__device__ __forceinline__ void hllc(double rl, double ul, double al, double bl, double pl, double rr, double ur,
                                     double ar, double br, double pr, double g, double igm1, double &f0,
                                     double &fn, double &fa, double &fb, double &f4) {
  double c;
  {
    const bool lbig = gt_nonneg(O::mul(pl, rr), O::mul(pr, rl));
    const double a = O::mul(g, lbig ? pl : pr), x = O::mul(a, lbig ? rl : rr);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = __fma_rn(-x, O::mul(y, y), 1.0), t = O::mul(a, y);
    c = __fma_rn(t, O::mul0(h, __fma_rn(0.375, h, 0.5)), t);
  }
  const double du = __dadd_rn(ul, -ur);
  const double e = __dadd_rn(c, pos(du) ? du : 0.0);
  const double ie = rcp(O::mul(e, __dadd_rn(rl, rr)));
  const double us = O::mul0(__fma_rn(e, __fma_rn(rr, ur, O::mul0(rl, ul)), __dadd_rn(pl, -pr)), ie);
  const bool light = gt_nonneg(rr, rl);  // the left side is the lighter one
  const double ps = __fma_rn(O::mul(light ? rl : rr, light ? -e : e), __dadd_rn(us, -(light ? ul : ur)),
                             light ? pl : pr);
  const bool left = pos(us);
  const double rk = left ? rl : rr, uk = left ? ul : ur, ak = left ? al : ar, bk = left ? bl : br,
               pk = left ? pl : pr;
  const double se = left ? -e : e;  // S_K - u_K
  const double sk = __dadd_rn(uk, se);
  const bool star = left ? !pos(sk) : pos(sk);
  const double ds = __dadd_rn(sk, -us), id = rcp(ds);
  const double ek =
      __fma_rn(pk, igm1, O::mul0(O::half(rk), __fma_rn(bk, bk, __fma_rn(ak, ak, O::mul0(uk, uk)))));
  const double rs = O::mul(O::mul(rk, se), id);
  const double es = O::mul0(__fma_rn(ps, us, __fma_rn(-pk, uk, O::mul0(se, ek))), id);
  const double ro = star ? rs : rk, eo = star ? es : ek, uo = star ? us : uk, po = star ? ps : pk;
  f0 = O::mul0(ro, uo);
  fn = __fma_rn(f0, uo, po);
  fa = O::mul0(f0, ak);
  fb = O::mul0(f0, bk);
  f4 = O::mul0(__dadd_rn(eo, po), uo);
  // the integer products know no infinities: a vanishing S_K - u* gives NaN
  if (star && ds == 0.0) f0 = fn = fa = fb = f4 = __dmul_rn(0.0, id);
}

// HLLC flux normal to axis D from face states qL, qR (rho, u, v, w, p).
// FP64: a warp whose faces all have densities and pressures in [2^-100, 2^100)
// and velocities below 2^150 takes the products on the integer pipes: nothing
// overflows, and the operands of mul (densities, pressures, wave speeds) are
// normal with normal products.  Others take the FP64 pipe, with the same bits.
// Level 7 of the Sedov blast (2.1 M cells): 780 us with all products on the
// FP64 pipe, 497 us with them on the integer pipes, 451 us with a block per tile and
// axis (k_flux; FP64 pipe 87 %, issue slots 50 % busy).
__device__ __forceinline__ void hllc_axis(int D, const double (&qL)[5], const double (&qR)[5], double g, double igm1,
                                          double (&F)[5]) {
  const bool x = D == 0, z = D == 2;
  const double ul = x ? qL[1] : z ? qL[3] : qL[2], al = x ? qL[2] : qL[1], bl = z ? qL[2] : qL[3];
  const double ur = x ? qR[1] : z ? qR[3] : qR[2], ar = x ? qR[2] : qR[1], br = z ? qR[2] : qR[3];
  double fn, fa, fb;
  const bool safe = within<100>(qL[0]) && within<100>(qL[4]) && within<100>(qR[0]) && within<100>(qR[4]) &&
                    below<150>(ul) && below<150>(al) && below<150>(bl) && below<150>(ur) && below<150>(ar) &&
                    below<150>(br);
  if (__all_sync(__activemask(), safe))
    hllc<MulInt>(qL[0], ul, al, bl, qL[4], qR[0], ur, ar, br, qR[4], g, igm1, F[0], fn, fa, fb, F[4]);
  else
    hllc<MulFp64>(qL[0], ul, al, bl, qL[4], qR[0], ur, ar, br, qR[4], g, igm1, F[0], fn, fa, fb, F[4]);
  F[1] = x ? fn : fa;
  F[2] = x ? fa : z ? fb : fn;
  F[3] = z ? fn : fb;
}
// FP32: the definitions as written.  max(c) keeps the quotient form: a rho can
// leave float's range at the density and pressure floors (about 1e-41), a / rho
// cannot.
__device__ __forceinline__ void hllc_axis(int D, const float (&qL)[5], const float (&qR)[5], float g, float igm1,
                                          float (&F)[5]) {
  const bool x = D == 0, z = D == 2;
  const float rl = qL[0], ul = x ? qL[1] : z ? qL[3] : qL[2], pl = qL[4];
  const float rr = qR[0], ur = x ? qR[1] : z ? qR[3] : qR[2], pr = qR[4];
  const float cmax = sqrtf(fmaxf(g * pl * rcp(rl), g * pr * rcp(rr)));
  const float sl = vmin(ul, ur) - cmax;
  const float sr = vmax(ul, ur) + cmax;
  const float rcl = rl * (ul - sl), rcr = rr * (sr - ur);
  const float irc = rcp(rcl + rcr);
  const float us = ((rcr * ur + rcl * ul) + (pl - pr)) * irc;
  const float ps = ((rcr * pl + rcl * pr) + rcl * rcr * (ul - ur)) * irc;
  const bool left = pos(sl) || pos(us);
  const bool star = left ? !pos(sl) : pos(sr);
  float qk[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) qk[v] = left ? qL[v] : qR[v];
  const float rk = qk[0], uk = left ? ul : ur, pk = qk[4];
  const float ek = qk[4] * igm1 + 0.5f * qk[0] * ((qk[1] * qk[1] + qk[2] * qk[2]) + qk[3] * qk[3]);
  const float sk = left ? sl : sr;
  const float id = rcp(sk - us);
  const float rs = rk * (sk - uk) * id;
  const float es = ((sk - uk) * ek - pk * uk + ps * us) * id;
  const float ro = star ? rs : rk, eo = star ? es : ek, uo = star ? us : uk, po = star ? ps : pk;
  const float mf = ro * uo, fn = mf * uo + po;
  F[0] = mf;
  F[1] = x ? fn : mf * qk[1];
  F[2] = x || z ? mf * qk[2] : fn;
  F[3] = z ? fn : mf * qk[3];
  F[4] = (eo + po) * uo;
}

// face states W* +- dW/2 of the two cells of a face (with the floors) and
// their HLLC flux normal to axis D
template <class T>
__device__ __forceinline__ void face_flux_states(int D, const SegCtx<T> &s, T (&qL)[5], T (&qR)[5], T (&F)[5]) {
  qL[0] = vmax(qL[0], s.smallr);
  qR[0] = vmax(qR[0], s.smallr);
  qL[4] = floor_p(qL[4], qL[0], s.smallp);
  qR[4] = floor_p(qR[4], qR[0], s.smallp);
  hllc_axis(D, qL, qR, s.gamma, s.igm1, F);
}

// flux across the face normal to axis D between local cells tl (minus side) and
// tr (plus side)
template <class T>
__device__ __forceinline__ void face_flux(const StepArgs<T> &a, const SegCtx<T> &s, int D, int tl, int tr,
                                          T (&F)[5]) {
  T qL[5], qR[5];
  load_side(a, s.base + tl, D, T(0.5), qL);
  load_side(a, s.base + tr, D, T(-0.5), qR);
  face_flux_states(D, s, qL, qR, F);
}

// reflux slot of a coarse-fine face normal to axis D: ghost oct gq (local oct
// index), the direction of the face seen from the ghost's father cell X, fine
// face (a, b) of the real cell's index c in its oct
__device__ __forceinline__ int64_t reflux_slot(int D, int clo, int nl, int gq, int dirX, int c) {
  const int ab = D == 0 ? ((c >> 1) & 1) << 1 | ((c >> 2) & 1) : D == 1 ? (c & 1) << 1 | ((c >> 2) & 1)
                                                                       : (c & 1) << 1 | ((c >> 1) & 1);
  return int64_t(clo + gq - nl) * 24 + dirX * 4 + ab;
}

// One thread per real or ghost cell and axis: the flux of the cell's plus face.
// A face is needed when at least one side is a real cell and neither side is
// split; other faces carry zero.  A needed face with a ghost on one side is a
// coarse-fine face: its flux, times sigma dt/dx / 8, goes to slot (direction
// seen from the coarse cell, fine face a,b) of the ghost oct.  A tile's three
// axes are consecutive blocks: the faces of a small level are solved at once
// (one after the other they are a chain of three solves, which bounds a level
// that does not fill the GPU), and a large level finds the cells' states in L2.
__global__ void k_flux(StepArgs<double> a) {
  for (int tb = blockIdx.x; tb < 3 * a.tiles.ntiles; tb += gridDim.x) {
    const int ti = tb / 3, D = tb - 3 * ti;
    const Tile td = tile_at(a.tiles, ti);
    SegCtx<double> s;
    if (!open_segment(a, td.seg, s)) continue;
    const int t = td.start + threadIdx.x;
    if (t >= 8 * (s.nl + s.ncl)) continue;
    const int q = t >> 3, c = t & 7;
    const bool real = q < s.nl;
    double F[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const int tn = nbr_local(a, s, t, ext_of_local(a, s, q), c, D, 1);
    if (tn >= 0) {
      const bool nreal = (tn >> 3) < s.nl;
      if ((real || nreal) && !cell_is_split(a, s, t) && !cell_is_split(a, s, tn)) {
        face_flux(a, s, D, t, tn, F);
        if (a.reflux && (real != nreal)) {
          // ghost on the plus side: the coarse cell's minus face (sigma +1);
          // ghost on the minus side: its plus face (sigma -1)
          const int64_t gslot = real ? reflux_slot(D, s.clo, s.nl, tn >> 3, 2 * D, c)
                                     : reflux_slot(D, s.clo, s.nl, t >> 3, 2 * D + 1, c);
          const double sg8 = real ? 1.0 : -1.0;
#pragma unroll
          for (int v = 0; v < 5; ++v)
            a.C[v * a.CS + checked(gslot, 0, a.CS, a.err)] = (sg8 * s.dtdx) * F[v] / 8.0;
        }
      }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) a.F[(5 * D + v) * a.LS + s.base + t] = F[v];
  }
}

// sum over the axes of F(minus face) - F(plus face) of one variable.  FP64: the three
// differences on the FP64 pipe, which are exact where leading bits cancel (a pressure
// that is nearly the same on both sides must not take bits from a small difference
// along another axis), their sum on the integer pipes.  Sedov 7-10 / clustered 6-9, us
// of updates per coarse step: 385 / 256; all five additions on the FP64 pipe 478 / 397,
// none of them 405 / 258.
__device__ __forceinline__ double flux_sum(double xm, double xp, double ym, double yp, double zm, double zp) {
  return sum3_int(__dadd_rn(xm, -xp), __dadd_rn(ym, -yp), __dadd_rn(zm, -zp));
}
__device__ __forceinline__ float flux_sum(float xm, float xp, float ym, float yp, float zm, float zp) {
  return ((xm - xp) + (ym - yp)) + (zm - zp);
}

// variable v of the pending reflux R in slot rs (-1: none).  Loaded with the fluxes,
// before their sum: after it the load's latency comes on top (clustered 6-9, update
// per coarse step: 439 instead of 256 us)
template <class T>
__device__ __forceinline__ T pending(const StepArgs<T> &a, int v, int rs) {
  return rs >= 0 ? a.Rc[v * int64_t(a.NC) + rs] : T(0);
}
// new state (u + dt/dx dF) + R of variable v, dF its flux sum; R <- 0
template <class T>
__device__ __forceinline__ T new_state(const StepArgs<T> &a, const SegCtx<T> &s, int v, T u, int rs, T r, T dF) {
  u = u + s.dtdx * dF;
  if (rs >= 0) {
    u = u + r;
    a.Rc[v * int64_t(a.NC) + rs] = T(0);
  }
  return u;
}
template <class T>
__device__ __forceinline__ int reflux_of(const StepArgs<T> &a, int g) {
  return int(checked(__ldg(a.rslot + g), -1, a.NC, a.err, -1));
}

// father cell (index in its oct) of the oct with internal key k
__device__ __forceinline__ int father_cell(uint64_t k) {
  return int((ikey_x(k) & 1) | ((ikey_y(k) & 1) << 1) | ((ikey_z(k) & 1) << 2));
}

// restriction of local oct q, variable v: father cell = (sum of the 8 children's
// new states u[0..8) in child order) / 8
template <class T>
__device__ __forceinline__ void restrict_oct(const StepArgs<T> &a, const SegCtx<T> &s, int q, int v, const T *u) {
  const int o = s.lo + q;
  const int fc = father_cell(__ldg(a.key + o));
  const int f = int(checked(__ldg(a.father + o), 0, a.N, a.err));
  T sum = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) sum += u[c];
  a.U[v * a.S + 8 * int64_t(f) + fc] = sum * T(0.125);
}

// The last pass of a level step: new states of the leaf cells, the restriction of
// their octs and, beyond the cells, the reflux sums of the level's ghost octs.
// They touch disjoint data: the level's cells, the coarser level's split cells,
// the pending reflux of its leaf cells.

// FP64, a list that fills the GPU: a thread per cell, one variable after the other
// (figures at flux_sum).  The loads of the next variable ahead of the sum, or 40
// registers for more warps, gain nothing (3 % and more slower).
// domain: 8 nl, + 5 ncl (if kSegReflux)
__global__ void __launch_bounds__(512, 2) k_update(StepArgs<double> a) {
  extern __shared__ double update_smem[];  // the block's new states [5][threads]
  const int lane = threadIdx.x & 31;
  warp_tile_loop(a, [&](const SegCtx<double> &s, int t) {
    if (t < 8 * s.nl) {
      const int e = s.lo + (t >> 3), c = t & 7, g = 8 * e + c;
      const bool leaf = !cell_is_split(a, s, t);
      int mx = 0, my = 0, mz = 0, rs = -1;
      if (leaf) {
        mx = nbr_local(a, s, t, e, c, 0, 0);
        my = nbr_local(a, s, t, e, c, 1, 0);
        mz = nbr_local(a, s, t, e, c, 2, 0);
        rs = reflux_of(a, g);
      }
#pragma unroll 1
      for (int v = 0; v < 5; ++v) {
        double u = a.U[v * a.S + g];
        if (leaf) {
          const double *Fx = a.F + v * a.LS + s.base, *Fy = Fx + 5 * a.LS, *Fz = Fy + 5 * a.LS;
          const double xm = Fx[mx], xp = Fx[t], ym = Fy[my], yp = Fy[t], zm = Fz[mz], zp = Fz[t];
          const double r = pending(a, v, rs);
          u = new_state(a, s, v, u, rs, r, flux_sum(xm, xp, ym, yp, zm, zp));
          a.U[v * a.S + g] = u;
        }
        if (s.flags & kSegRestrict) update_smem[v * blockDim.x + threadIdx.x] = u;
      }
    } else if ((s.flags & kSegReflux) && t - 8 * s.nl < 5 * s.ncl) {
      const int q = t - 8 * s.nl, v = q / s.ncl;
      reflux_sum(a, v, s.clo + (q - v * s.ncl));
    }
    if (s.flags & kSegRestrict) {  // a lane per (oct, variable)
      __syncwarp();
      const int q = ((t - lane) >> 3) + (lane & 3), v = lane >> 2;
      if (v < 5 && q < s.nl)
        restrict_oct(a, s, q, v, update_smem + v * blockDim.x + (threadIdx.x - lane) + 8 * (lane & 3));
      __syncwarp();
    }
  });
}

// FP64, a short list: a thread per (cell, variable), a tile's five variables in
// consecutive blocks (five times the threads and a fifth of the chain).
// domain: 8 nl, + ncl (if kSegReflux)
__global__ void k_update_small(StepArgs<double> a) {
  extern __shared__ double update_smem[];  // the block's new states
  double *sm = update_smem;
  const int lane = threadIdx.x & 31;
  for (int tb = blockIdx.x; tb < 5 * a.tiles.ntiles; tb += gridDim.x) {
    const int ti = tb / 5, v = tb - 5 * ti;
    const Tile td = tile_at(a.tiles, ti);
    SegCtx<double> s;
    if (!open_segment(a, td.seg, s)) continue;
    const int t = td.start + threadIdx.x;
    if (t < 8 * s.nl) {
      const int e = s.lo + (t >> 3), c = t & 7, g = 8 * e + c;
      double u = a.U[v * a.S + g];
      if (!cell_is_split(a, s, t)) {
        const double *Fx = a.F + v * a.LS + s.base, *Fy = Fx + 5 * a.LS, *Fz = Fy + 5 * a.LS;
        const int mx = nbr_local(a, s, t, e, c, 0, 0), my = nbr_local(a, s, t, e, c, 1, 0),
                  mz = nbr_local(a, s, t, e, c, 2, 0);
        const int rs = reflux_of(a, g);
        const double xm = Fx[mx], xp = Fx[t], ym = Fy[my], yp = Fy[t], zm = Fz[mz], zp = Fz[t], r = pending(a, v, rs);
        u = new_state(a, s, v, u, rs, r, flux_sum(xm, xp, ym, yp, zm, zp));
        a.U[v * a.S + g] = u;
      }
      sm[threadIdx.x] = u;
    } else if ((s.flags & kSegReflux) && t - 8 * s.nl < s.ncl) {
      reflux_sum(a, v, s.clo + (t - 8 * s.nl));
    }
    if (s.flags & kSegRestrict) {
      __syncwarp();
      const int q = ((t - lane) >> 3) + lane;
      if (lane < 4 && q < s.nl) restrict_oct(a, s, q, v, sm + (threadIdx.x - lane) + 8 * lane);
      __syncwarp();
    }
  }
}

// FP32 flux and update, thread per cell of a tile.  Each leaf cell solves its plus
// faces into shared memory; a minus face belongs to the cell beyond it, and only
// where that one lies outside the tile (at most 12 of an oct's faces) it goes to a
// list that the block solves next, without idle lanes.  A tile of 512 cells of a
// refined region, 8^3 in Hilbert order, solves 3.4 faces per cell instead of both
// cells of a face solving it, and stores no flux.  Then the update and the
// restriction of the warp's octs.  Bound by instructions (issue 73 %) and the latency
// of gathered loads: the neighbours' indices are all loaded before the first is
// needed, and the state and its pending reflux before the first store, which the
// compiler would keep them behind.  us, 128^3 uniform / Sedov 7-10 / clustered 6-9 per
// coarse step: six solves per cell from 20 predictor arrays 136 / 427 / 338; plus
// faces shared 123 / 415; with four-value arrays and indices first 100 / 365 / 328;
// loads before stores and the tile size a constant 94 / 288 / 205.  At 62 registers
// 120, at 32 with spills 140.  A solve per face into memory and an update of its own,
// with more threads per cell, is no faster on short lists either (random mesh 3-6
// 0.191 against 0.190 ms, levels of 25-72 thousand cells 51 against 47 us).
// domain: 8 nl
constexpr int kFluxSmem = 15 * 4 + 10 * 4 + 2 * 6 + 2;  // bytes per thread
template <int TH>
__global__ void __launch_bounds__(TH, 1536 / TH) k_flux_update(StepArgs<float> a) {
  extern __shared__ float flux_smem[];
  // fluxes [5][TH]: plus faces along each axis, two halves of the list (at most 1.5 TH)
  float *const flux = flux_smem;
  int *const cell = reinterpret_cast<int *>(flux + 25 * TH), *const beyond = cell + TH + TH / 2;
  int *const listed = beyond + TH + TH / 2;  // list: axis and thread; the cell beyond
  const int tid = threadIdx.x, lane = tid & 31;
  warp_tile_loop(a, [&](const SegCtx<float> &s, int t) {  // the same tile for the whole block
    if (tid == 0) *listed = 0;
    __syncthreads();
    const int t0 = t - tid, e = s.lo + (t >> 3), c = t & 7, g = 8 * e + c;
    const uint32_t split = t < 8 * s.nl ? __ldg(a.son + e) : ~0u;  // of the oct's cells
    const bool leaf = !((split >> c) & 1u);
    // the neighbour in the next oct along each axis, or -1 where that is split (the
    // other neighbour is in this oct)
    int out[3] = {-1, -1, -1};
    if (leaf) {
#pragma unroll
      for (int D = 0; D < 3; ++D) out[D] = nbr_local(a, s, t, e, c, D, (c >> D) & 1);
#pragma unroll
      for (int D = 0; D < 3; ++D)
        if (out[D] >= 0 && cell_is_split(a, s, out[D])) out[D] = -1;
    }
    int from[3];  // first of the five values of each minus face's flux, -1: none
#pragma unroll
    for (int D = 0; D < 3; ++D) {
      const bool up = (c >> D) & 1;
      const int rel = up ? tid ^ (1 << D) : out[D] - t0;
      const bool none = up ? (split >> (c ^ (1 << D))) & 1u : out[D] < 0;
      from[D] = none ? -1 : 5 * D * TH + rel;
      const bool outside = leaf && !up && !none && (unsigned(rel) >= TH || (out[D] >> 3) >= s.nl);
      const unsigned add = __ballot_sync(0xFFFFFFFFu, outside);
      if (add) {
        int at = 0;
        if (lane == 0) at = atomicAdd(listed, __popc(add));
        at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(add & ((1u << lane) - 1u));
        if (outside) {
          cell[at] = D << 16 | tid;
          beyond[at] = out[D];
          from[D] = 15 * TH + at + (at >= TH ? 4 * TH : 0);
        }
      }
    }
    if (leaf) {
      const float4 *Q = reinterpret_cast<const float4 *>(a.Q) + s.base + t;
      const float4 w = __ldg(Q), p = __ldg(Q + a.LS);
#pragma unroll
      for (int D = 0; D < 3; ++D) {
        const bool up = (c >> D) & 1;
        const int tp = up ? out[D] : (split >> (c ^ (1 << D))) & 1u ? -1 : t ^ (1 << D);
        float F[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (tp >= 0) {
          float qL[5], qR[5];
          side_of(w, p, __ldg(Q + (2 + D) * a.LS), D, 0.5f, qL);
          load_side(a, s.base + tp, D, -0.5f, qR);
          face_flux_states(D, s, qL, qR, F);
          if (a.reflux && (tp >> 3) >= s.nl) {
            const int64_t gslot = reflux_slot(D, s.clo, s.nl, tp >> 3, 2 * D, c);
#pragma unroll
            for (int v = 0; v < 5; ++v)
              a.C[v * a.CS + checked(gslot, 0, a.CS, a.err)] = (1.0f * s.dtdx) * F[v] / 8.0f;
          }
        }
#pragma unroll
        for (int v = 0; v < 5; ++v) flux[(5 * D + v) * TH + tid] = F[v];
      }
    }
    __syncthreads();
    for (int i = tid; i < *listed; i += TH) {
      const int D = cell[i] >> 16, tc = t0 + (cell[i] & 0xFFFF), tb = beyond[i];
      float F[5];
      face_flux(a, s, D, tb, tc, F);
      if (a.reflux && (tb >> 3) >= s.nl) {
        const int64_t gslot = reflux_slot(D, s.clo, s.nl, tb >> 3, 2 * D + 1, tc & 7);
#pragma unroll
        for (int v = 0; v < 5; ++v)
          a.C[v * a.CS + checked(gslot, 0, a.CS, a.err)] = (-1.0f * s.dtdx) * F[v] / 8.0f;
      }
      float *m = flux + 15 * TH + i + (i >= TH ? 4 * TH : 0);
#pragma unroll
      for (int v = 0; v < 5; ++v) m[v * TH] = F[v];
    }
    const int rs = leaf ? reflux_of(a, g) : -1;
    __syncthreads();
    float u[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, r[5];
    if (t < 8 * s.nl) {
#pragma unroll
      for (int v = 0; v < 5; ++v) u[v] = a.U[v * a.S + g];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) r[v] = pending(a, v, rs);
    if (leaf) {
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const float *p = flux + v * TH + tid;
        float m[3];
#pragma unroll
        for (int D = 0; D < 3; ++D) m[D] = from[D] < 0 ? 0.0f : flux[v * TH + from[D]];
        u[v] = new_state(a, s, v, u[v], rs, r[v], flux_sum(m[0], p[0], m[1], p[5 * TH], m[2], p[10 * TH]));
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) a.U[v * a.S + g] = u[v];
    }
    __syncthreads();  // the fluxes are read
    if (s.flags & kSegRestrict) {  // the warp's octs, a lane per (oct, variable)
#pragma unroll
      for (int v = 0; v < 5; ++v) flux[v * TH + tid] = u[v];
      __syncwarp();
      const int q = ((t - lane) >> 3) + (lane & 3), v = lane >> 2;
      if (v < 5 && q < s.nl) restrict_oct(a, s, q, v, flux + v * TH + (tid - lane) + 8 * (lane & 3));
    }
  });
}

// Restriction alone (of a state that was written): father cell = (sum of the 8
// children in child order) / 8.  domain: 5 nl (if kSegRestrict)
template <class T>
__global__ void k_restrict(StepArgs<T> a) {
  tile_loop(a, [](const SegCtx<T> &s) { return (s.flags & kSegRestrict) ? 5 * s.nl : 0; },
            [&](const SegCtx<T> &s, int r) {
              const int v = r / s.nl, q = r - v * s.nl;
              restrict_oct(a, s, q, v, a.U + v * a.S + 8 * int64_t(s.lo + q));
            });
}

// ---------------------------------------------------------------------------
// CFL time step: per (member, level) max of sum_d (|u_d| + c) over leaf cells
// (cell speeds in the state's precision, the maximum and dt in FP64), by integer
// atomicMax on the bit pattern (non-negative doubles order like their bits): FP32
// once per block and segment, FP64 once per warp that formed a speed; then one
// thread per member computes its dt.
// ---------------------------------------------------------------------------
// the block's maximum over a segment: warp shuffles, then shared memory
template <class T>
__device__ __forceinline__ void cfl_flush(const CflArgs &a, double s, int seg, double *wmax) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s = fmax(s, __shfl_xor_sync(0xFFFFFFFFu, s, off));
  if (lane == 0) wmax[warp] = s;
  __syncthreads();
  if (warp == 0) {
    s = lane < int(blockDim.x >> 5) ? wmax[lane] : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s = fmax(s, __shfl_xor_sync(0xFFFFFFFFu, s, off));
    if (lane == 0 && s > 0.0) {
      const Seg sg = seg_at(a.tiles, seg);
      atomicMax(a.smax + 16 * sg.member + sg.level, (unsigned long long)__double_as_longlong(s));
    }
  }
  __syncthreads();
}

// sum_d (|u_d| + c) of a cell in the state's precision
template <class T>
__device__ __forceinline__ T cell_speed(T g, T smallr, T smallp, T u0, T u1, T u2, T u3, T u4) {
  const T r = vmax(u0, smallr);
  const T ir = rcp(r);
  const T vx = u1 * ir, vy = u2 * ir, vz = u3 * ir;
  const T ek = T(0.5) * r * ((vx * vx + vy * vy) + vz * vz);
  const T p = vmax((g - T(1)) * (u4 - ek), r * smallp);
  const T cs = sound_speed(g * p * ir);
  return ((fabs(vx) + cs) + (fabs(vy) + cs)) + (fabs(vz) + cs);
}

// FP32: each block keeps a running maximum per thread while its tiles stay in
// one segment and reduces it (one atomicMax) when the segment changes.
// The running maximum is kept in FP32 (float to double is exact and monotonic,
// so converting once per flush gives the same maximum) and the parameters are
// read in that type: no conversions per cell, which would run on the FP64 pipe.
__global__ void k_cfl_fp32(CflArgs a, const float *U) {
  __shared__ double wmax[32];
  float s = 0.0f;
  int cur = -1;
  const float *mgamma = static_cast<const float *>(a.mgamma_t), *msmallr = static_cast<const float *>(a.msmallr_t),
              *msmallp = static_cast<const float *>(a.msmallp_t);
  for (int ti = blockIdx.x; ti < a.tiles.ntiles; ti += gridDim.x) {
    const Tile td = tile_at(a.tiles, ti);
    if (td.seg != cur) {
      if (cur >= 0) cfl_flush<float>(a, double(s), cur, wmax);
      s = 0.0f;
      cur = td.seg;
    }
    const Seg sg = seg_at(a.tiles, td.seg);
    const int t = td.start + threadIdx.x;
    if (t < 8 * sg.nl && a.mrem[sg.member] != 0 &&
        !((__ldg(a.son + sg.lo + (t >> 3)) >> (t & 7)) & 1u)) {
      const int64_t gi = 8 * int64_t(sg.lo) + t;
      const float u0 = U[gi], u1 = U[a.S + gi], u2 = U[2 * a.S + gi], u3 = U[3 * a.S + gi], u4 = U[4 * a.S + gi];
      const float st = cell_speed(mgamma[sg.member], msmallr[sg.member], msmallp[sg.member], u0, u1, u2, u3, u4);
      if (!finite_bits(st) || !(finite_bits(u0) && finite_bits(u1) && finite_bits(u2) &&
                                finite_bits(u3) && finite_bits(u4))) {
        atomicOr(a.err, kErrNaN);
        atomicOr(a.merr + sg.member, kErrNaN);
      } else if (gt_nonneg(st, s)) {
        s = st;
      }
    }
  }
  if (cur >= 0) cfl_flush<float>(a, double(s), cur, wmax);
}

// FP64: the maximum needs the FP64 speed of few cells.  Each cell's speed is
// bounded from above in FP32; a warp forms the FP64 speeds (31 operations on
// the FP64 pipe, which bounded this pass) only when one of its bounds reaches
// the largest speed found so far, and publishes what it finds at once.  The
// maximum is over the same FP64 values as before: a cell passed over lies
// strictly below one of them.
//
// The bound: the FP32 images of the state are truncated (relative error below
// 2^-23), the parameters, quotients, squares and sums err by a few 2^-23 each:
// |u_d| by less than 2^-20 of itself, ek by less than 2^-19, so E - ek lies
// within 2^-18 (|E| + ek) of its FP32 value; c = sqrt(gamma p / rho) by less
// than 2^-18 of itself and sqrt(gamma smallp) for the floor.  2^-16 over the
// sum covers them and the approximate reciprocal, and 2^-60 a momentum that
// vanishes in FP32.  A cell whose density, energy, kinetic energy or gamma lies
// outside the powers of two named below (no value there over- or underflows),
// or that is not finite, always takes the FP64 test: an infinite or NaN
// momentum makes its kinetic energy so.
__global__ void __launch_bounds__(512) k_cfl_fp64(CflArgs a, const double *U) {
  const double *mgamma = a.mgamma, *msmallr = a.msmallr, *msmallp = a.msmallp;
  for (int ti = blockIdx.x; ti < a.tiles.ntiles; ti += gridDim.x) {
    const Tile td = tile_at(a.tiles, ti);
    const Seg sg = seg_at(a.tiles, td.seg);
    const int t = td.start + threadIdx.x;
    unsigned long long *out = a.smax + 16 * sg.member + sg.level;
    bool test = false;
    double u0 = 0.0, u1 = 0.0, u2 = 0.0, u3 = 0.0, u4 = 0.0;
    if (t < 8 * sg.nl && a.mrem[sg.member] != 0 &&
        !((__ldg(a.son + sg.lo + (t >> 3)) >> (t & 7)) & 1u)) {
      const unsigned long long seen = __ldcg(out);
      const int64_t gi = 8 * int64_t(sg.lo) + t;
      u0 = U[gi];
      u1 = U[a.S + gi];
      u2 = U[2 * a.S + gi];
      u3 = U[3 * a.S + gi];
      u4 = U[4 * a.S + gi];
      const float gm1 = a.mflag32[3 * sg.member], smallr = a.mflag32[3 * sg.member + 1],
                  smallp = a.mflag32[3 * sg.member + 2];
      const float g = gm1 + 1.0f;
      const float r = fmaxf(to_f32(u0), smallr), ir = rcp(r);
      const float vx = fabsf(to_f32(u1)) * ir, vy = fabsf(to_f32(u2)) * ir, vz = fabsf(to_f32(u3)) * ir;
      const float e4 = to_f32(u4), ek = 0.5f * r * ((vx * vx + vy * vy) + vz * vz);
      const float p = gm1 * ((e4 - ek) + 0x1p-18f * (fabsf(e4) + ek));
      const float c = sqrtf(g * fmaxf(p, 0.0f) * ir) + sqrtf(g * smallp);
      const float bound = (1.0f + 0x1p-16f) * ((vx + vy) + (vz + 3.0f * c)) + 0x1p-60f;
      const bool ok = r >= 0x1p-60f && r <= 0x1p60f && e4 >= 0x1p-60f && e4 <= 0x1p60f && ek <= 0x1p60f &&
                      gm1 >= 0x1p-20f && gm1 <= 0x1p20f && finite_bits(u0);
      test = !ok || !(bound < to_f32(__longlong_as_double((long long)seen)));
    }
    if (!__any_sync(0xFFFFFFFFu, test)) continue;
    double s = 0.0;
    if (test) {
      s = cell_speed(__ldg(mgamma + sg.member), __ldg(msmallr + sg.member), __ldg(msmallp + sg.member), u0, u1, u2,
                     u3, u4);
      if (!finite_bits(s) || !(finite_bits(u0) && finite_bits(u1) && finite_bits(u2) && finite_bits(u3) &&
                               finite_bits(u4))) {
        atomicOr(a.err, kErrNaN);
        atomicOr(a.merr + sg.member, kErrNaN);
        s = 0.0;
      }
    }
    // the warp's maximum: non-negative doubles order like their bits
    long long b = __double_as_longlong(s);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const long long o = __shfl_xor_sync(0xFFFFFFFFu, b, off);
      b = o > b ? o : b;
    }
    if ((threadIdx.x & 31) == 0 && b > 0) atomicMax(out, (unsigned long long)b);
  }
}

__global__ void k_dt(CflArgs a) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= a.nmembers) return;
  const int lmin = a.mlmin[m];
  double dt = __longlong_as_double(0x7FF0000000000000ll);  // +inf
  for (int l = lmin; l <= kMaxLev; ++l) {
    const unsigned long long b = a.smax[16 * m + l];
    a.smax[16 * m + l] = 0ull;
    if (b == 0ull) continue;
    const double smax = __longlong_as_double((long long)b);
    const double dtl = a.mcfl[m] * ldexp(1.0, -l) / smax;
    const double dtc = dtl * ldexp(1.0, l - lmin);
    dt = fmin(dt, dtc);
  }
  // a member with no coarse steps left keeps its state and its last dt
  const int rem = a.mrem[m];
  if (a.consume) {
    a.mact[m] = rem != 0;
    if (rem > 0) a.mrem[m] = rem - 1;
  }
  if (rem == 0) return;
  a.dt_dev[m] = dt;
  a.dtdx_dev[m] = ldexp(dt, lmin);
  a.dtdxf_dev[m] = ldexpf(float(dt), lmin);
}

// ---------------------------------------------------------------------------
// Conservation totals of one level (FP64 in both precisions, fixed order, no
// atomics): block b sums the leaf cells of [b chunk, (b+1) chunk) of the
// level's cells, thread t the cells b chunk + t + 256 k in increasing k, then
// a fixed butterfly over each warp and the 8 warp sums in warp order;
// partial[v G + b].  k_totals_sum adds a level's G partials in block order,
// scales by dx^3 (exact: a power of two) into lev[5 l + v], and with
// all_levels adds the levels' totals in ascending level order into out.
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(256) k_totals(const T *__restrict__ U, int64_t S,
                                                const uint32_t *__restrict__ son, int64_t c0,
                                                int64_t n, int64_t chunk, double *partial, int G) {
  __shared__ double ws[5][8];
  const int64_t b0 = blockIdx.x * chunk;
  const int64_t b1 = b0 + chunk < n ? b0 + chunk : n;
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t t = b0 + threadIdx.x; t < b1; t += 256) {
    const int64_t g = c0 + t;
    if ((__ldg(son + (g >> 3)) >> (g & 7)) & 1u) continue;  // split: not a leaf
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] += double(U[v * S + g]);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc[v] += __shfl_xor_sync(0xFFFFFFFFu, acc[v], off);
    if (lane == 0) ws[v][warp] = acc[v];
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    double sum = 0.0;
    for (int w = 0; w < 8; ++w) sum += ws[threadIdx.x][w];
    partial[threadIdx.x * int64_t(G) + blockIdx.x] = sum;
  }
}

__global__ void k_totals_sum(const double *partial, int G, int level, double *lev, int all_levels,
                             int lmin, int lmax, double *out) {
  const int v = threadIdx.x;
  if (v >= 5) return;
  double sum = 0.0;
  for (int b = 0; b < G; ++b) sum += partial[v * int64_t(G) + b];
  lev[5 * level + v] = ldexp(sum, -3 * level);
  if (all_levels) {
    double t = 0.0;
    for (int l = lmin; l <= lmax; ++l) t += lev[5 * l + v];
    out[v] = t;
  } else {
    out[v] = lev[5 * level + v];
  }
}

template <class T>
__global__ void k_to_double(const T *src, int64_t src_stride, int64_t count, double *dst) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= 5 * count) return;
  const int v = int(q / count);
  dst[q] = double(src[v * src_stride + q % count]);
}
// five rows of `count` doubles from src (row stride src_stride) to dst (row
// stride dst_stride), 16 bytes per thread; count and both strides even, both
// bases 16-byte aligned (the state's rows start at multiples of 8 cells)
__global__ void k_rows_copy(const double2 *__restrict__ src, int64_t src_stride2, int64_t count2,
                            double2 *__restrict__ dst, int64_t dst_stride2) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= 5 * count2) return;
  const int64_t v = q / count2, j = q - v * count2;
  dst[v * dst_stride2 + j] = __ldg(src + v * src_stride2 + j);
}

template <class T>
__global__ void k_from_double(const double *src, int64_t count, T *dst, int64_t dst_stride) {
  const int64_t q = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (q >= 5 * count) return;
  const int v = int(q / count);
  dst[v * dst_stride + q % count] = T(src[q]);
}

}  // namespace amr
