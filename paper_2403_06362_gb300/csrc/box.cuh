// box.cuh -- device physics of the two-region multigroup box, shared by the
// history-based (box.cu) and event-based (box_event.cu) schedules.
//
// Geometry: box [0,S]^3 with an inner cube [lo,hi]^3 (region 1) inside the
// outer region 0, vacuum outside.  Surface tracking: each flight samples
// d = -ln(1-u) / Sigma_t[region] and stops at the region surface if that is
// nearer.  Collisions: implicit capture, downscatter by CDF row, isotropic
// direction by Marsaglia's rejection method, then the region's weight window
// (roulette or split).  Children of a split are seeded on demand with
// S_c = hash(k, S_p) (Section 4, Eq. 5) from the parent's current state.
// Track lengths go to a group-summed mesh as int64 fixed point (2^32).
//
// T = double: every operation rounds once (this code is compiled with
// --fmad=false), matching the fp64 transport definition step for step.
// T = float: geometry and distances in fp32; a flight whose fp32 collision
// distance lies within a relative 2^-16 of the surface distance is decided
// again in fp64; uniforms, hashes and the fixed-point scaling stay exact.
#pragma once
#include <cstdint>

#include "../../include/mc.h"
#include "mc_device.cuh"
#include "slab.cuh"

namespace mcb {

constexpr int kMaxG = MC_BOX_MAX_GROUPS;

struct BoxDev {
  double side, lo, hi;
  double st[2], c[2], wl[2], wh[2], ws[2];
  double cdf[2][kMaxG][kMaxG];
  uint64_t n_hist, seed, stride_q, id_offset, key, tally_offset;
  uint32_t ng, mesh, max_split, n_batches, seeding, source;
  // derived on the device (box_prep_kernel)
  double inv_st[2], h, inv_h;
  uint32_t ih_q;  // inv_h as ih_q 2^-ih_s: the voxel lookup guess
  int ih_s;
  float side_f, lo_f, hi_f, h_f, inv_h_f;
  float inv_st_f[2], c_f[2], wl_f[2], wh_f[2], ws_f[2];
  float inv_ws_f[2];
  uint32_t f32_ok;  // extents and windows lie in the range of the fp32 decisions of the fp64 path
  uint64_t cdf_n[2][kMaxG][kMaxG];  // u < cdf  <=>  n < cdf_n for u = n 2^-53
  uint64_t seed_hash, hist_begin;
};

// A particle of the box (position, direction and its componentwise inverse,
// weight, group, region).
template <typename T>
struct Part {
  T p[3], u[3], inv[3];
  T w;
  uint32_t g, region;
};

// Record of a split child waiting in a device bank (fp64 fields; fp32
// particles store their values exactly).
struct ChildRec {
  double p[3], u[3], w;
  uint64_t rng;
  uint64_t tbase;  // tally slot row of the family (problem offset + batch row)
  uint32_t g, region, prob, pad;
};

enum BoxOutcome : int { kBoxCollide = 0, kBoxCross = 1, kBoxLeak = 2, kBoxContinue = 3, kBoxKilled = 4 };

// The uniform u = n 2^-53 in T (fp32: rounded once).
template <typename T> __device__ __forceinline__ T from_n(uint64_t n);
template <> __device__ __forceinline__ double from_n<double>(uint64_t n) {
  return mcd::u53_to_double((uint32_t)(n >> 32), (uint32_t)n);
}
template <> __device__ __forceinline__ float from_n<float>(uint64_t n) { return mcs::u53_to_float(n); }

template <typename T> __device__ __forceinline__ T sel(const double& d, const float& f);
template <> __device__ __forceinline__ double sel<double>(const double& d, const float&) { return d; }
template <> __device__ __forceinline__ float sel<float>(const double&, const float& f) { return f; }

// Comparisons: fp64 on the integer pipes (sign-magnitude order keys, equal to
// the fp64 comparisons for non-NaN values), fp32 native.
__device__ __forceinline__ bool lt(double a, double b) { return mcx::d_lt(a, b); }
__device__ __forceinline__ bool lt(float a, float b) { return a < b; }
// the same for non-negative values (fp64: the bits order them)
__device__ __forceinline__ bool ltn(double a, double b) { return mcs::nn_lt(a, b); }
__device__ __forceinline__ bool ltn(float a, float b) { return a < b; }
__device__ __forceinline__ bool eq(double a, double b) { return mcx::okey(a) == mcx::okey(b); }
__device__ __forceinline__ bool eq(float a, float b) { return a == b; }
__device__ __forceinline__ bool gt0(double a) { return mcx::d_pos(a); }
__device__ __forceinline__ bool gt0(float a) { return a > 0.0f; }
__device__ __forceinline__ bool lt0(double a) { return mcx::d_neg(a); }
__device__ __forceinline__ bool lt0(float a) { return a < 0.0f; }
__device__ __forceinline__ bool is0(double a) { return mcx::d_zero(a); }
__device__ __forceinline__ bool is0(float a) { return a == 0.0f; }

template <typename T> __device__ __forceinline__ T recip(T v);
template <> __device__ __forceinline__ double recip<double>(double v) { return mcx::recip_normal(v); }
template <> __device__ __forceinline__ float recip<float>(float v) { return __frcp_rn(v); }

// Componentwise inverse of the direction (fp64: the correctly rounded
// reciprocal on the integer pipes, fp_exact.cuh); 0 for a zero component.
// One copy of the reciprocal's code, run three times with the components
// rotated through it: an indexed loop would put the direction in local
// memory, three inlined copies cost instruction-cache misses (the fp64
// kernel's largest stall).
template <typename T>
__device__ __forceinline__ void set_inv(Part<T>& q) {
  if constexpr (sizeof(T) == 4) {  // short enough three times over
#pragma unroll
    for (int a = 0; a < 3; ++a) q.inv[a] = q.u[a] != T(0) ? recip<T>(q.u[a]) : T(0);
    return;
  }
  T u0 = q.u[0], u1 = q.u[1], u2 = q.u[2], i0 = T(0), i1 = T(0), i2 = T(0);
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    const T i = recip<T>(u0), v = is0(u0) ? T(0) : i, r = u0;  // |u0| >= 2^-78 otherwise
    u0 = u1;
    u1 = u2;
    u2 = r;
    i0 = i1;
    i1 = i2;
    i2 = v;
  }
  q.inv[0] = i0;
  q.inv[1] = i1;
  q.inv[2] = i2;
}

// v1^2 + v2^2 - 1 of a direction try in fp32, off by less than 2^-20: from
// the leading 24 bits of each draw (exact in fp32; |v| off by less than
// 2^-23).
__device__ __forceinline__ float try_s(uint64_t n1, uint64_t n2) {
  const float a = __uint2float_rn((uint32_t)(n1 >> 29)) * 0x1p-23f - 1.0f;
  const float b = __uint2float_rn((uint32_t)(n2 >> 29)) * 0x1p-23f - 1.0f;
  return a * a + b * b - 1.0f;
}

// Marsaglia (1972): v1, v2 uniform on [-1,1)^2 until v1^2 + v2^2 < 1.
// A try is decided by try_s where that is not within 2^-19 of the circle, so
// that only the accepted one's v1 and v2 are formed as the path has them
// (fp32: 2 RN(u) - 1; fp64: exact, and the fp64 unit forms s once); fp64's
// square root is the integer pipes'.
template <int M, typename T>
__device__ __forceinline__ void iso_dir(mcs::Rng<M>& r, const mcd::Lcg& l, T u[3]) {
  if constexpr (sizeof(T) == 8) {
    uint64_t n1, n2;
    for (;;) {
      n1 = r.next_n(l);
      n2 = r.next_n(l);
      const float s = try_s(n1, n2);
      if (s < -0x1p-19f) break;
      if (s > 0x1p-19f) continue;
      const double v1 = mcx::two_u_minus_1(n1), v2 = mcx::two_u_minus_1(n2);
      if (lt(v1 * v1 + v2 * v2, 1.0)) break;
    }
    const double v1 = mcx::two_u_minus_1(n1), v2 = mcx::two_u_minus_1(n2);
    const double s = v1 * v1 + v2 * v2;
    const double t = mcx::scale_pow2(mcx::sqrt_rn(1.0 - s), 1);  // (2 v) t = v (2 t): doubling is exact
    u[0] = v1 * t;
    u[1] = v2 * t;
    u[2] = __fma_rn(-2.0, s, 1.0);  // 2 s is exact: one rounding either way
  } else {
    uint64_t n1, n2;
    T v1, v2, s;
    for (;;) {
      n1 = r.next_n(l);
      n2 = r.next_n(l);
      const float c = try_s(n1, n2);
      if (c > 0x1p-19f) continue;
      v1 = T(2) * from_n<T>(n1) - T(1);
      v2 = T(2) * from_n<T>(n2) - T(1);
      s = v1 * v1 + v2 * v2;
      if (c < -0x1p-19f || lt(s, T(1))) break;
    }
    const T t = sqrt(T(1) - s);
    u[0] = T(2) * v1 * t;
    u[1] = T(2) * v2 * t;
    u[2] = T(1) - T(2) * s;
  }
}

template <typename T>
__device__ __forceinline__ uint32_t region_of(const BoxDev& b, const T p[3], const T u[3]) {
  const T lo = sel<T>(b.lo, b.lo_f), hi = sel<T>(b.hi, b.hi_f);
  for (int a = 0; a < 3; ++a) {
    const bool above = lt(lo, p[a]) || (eq(p[a], lo) && gt0(u[a]));
    const bool below = lt(p[a], hi) || (eq(p[a], hi) && lt0(u[a]));
    if (!above || !below) return 0u;
  }
  return 1u;
}

// Distance to the way out of [lo, hi]^3 from inside: per axis the face ahead
// is picked first, so that lanes flying in different directions take one
// subtraction and one product together.
template <typename T>
__device__ __forceinline__ T exit_dist(const Part<T>& q, T lo, T hi) {
  T t = T(INFINITY);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const T ta = ((gt0(q.u[a]) ? hi : lo) - q.p[a]) * q.inv[a];
    if (!is0(q.u[a]) && lt(ta, t)) t = ta;
  }
  return lt0(t) ? T(0) : t;
}

// Distance to the way into [lo, hi]^3 from outside (infinite: it misses).
// Rounding is monotone, so the face on the side the particle comes from has
// the smaller of an axis's two distances.
template <typename T>
__device__ __forceinline__ T entry_dist(const Part<T>& q, T lo, T hi) {
  T tn = T(-INFINITY), tf = T(INFINITY);
  bool miss = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool neg = lt0(q.u[a]);
    const T tmin = ((neg ? hi : lo) - q.p[a]) * q.inv[a], tmax = ((neg ? lo : hi) - q.p[a]) * q.inv[a];
    if (!is0(q.u[a])) {
      if (lt(tn, tmin)) tn = tmin;
      if (lt(tmax, tf)) tf = tmax;
    } else if (!lt(lo, q.p[a]) || !lt(q.p[a], hi)) {
      miss = true;
    }
  }
  return !miss && !lt0(tn) && lt(tn, tf) ? tn : T(INFINITY);
}

// Distance to the region surface and its kind (1: into the other region,
// 2: out of the box).  Both regions share the code of the way out.
template <typename T>
__device__ __forceinline__ T surface_of(const BoxDev& b, const Part<T>& q, int& kind) {
  const T lo = sel<T>(b.lo, b.lo_f), hi = sel<T>(b.hi, b.hi_f), side = sel<T>(b.side, b.side_f);
  const bool inner = q.region == 1u;
  T ds = exit_dist(q, inner ? lo : T(0), inner ? hi : side);
  kind = inner ? 1 : 2;
  if (!inner) {
    const T de = entry_dist(q, lo, hi);
    if (lt(de, ds)) {
      ds = de;
      kind = 1;
    }
  }
  return ds;
}

// surface_of in fp64, out of line: for the few flights that pass an edge too
// closely for surface<double>'s fp32 decision.
static __device__ __noinline__ double surface_exact(const BoxDev* b, const Part<double>* q, int* kind) {
  return surface_of<double>(*b, *q, *kind);
}

template <typename T> __device__ __forceinline__ T surface(const BoxDev& b, const Part<T>& q, int& kind);
template <> __device__ __forceinline__ float surface<float>(const BoxDev& b, const Part<float>& q, int& kind) {
  return surface_of<float>(b, q, kind);
}

// fp64: which face the flight meets is decided in fp32, and only that face's
// distance is formed in fp64 (2 operations instead of 18).  The fp32 distance
// to a face ahead on axis a is off by less than e_a = |1/u_a| side 2^-20:
// position (truncated), face and their difference are off by less than
// 2^-22 side together, 1/u_a and the product by less than 2^-22 of a distance
// that is at most |1/u_a| side.  Distances closer to each other than their
// e's, a direction with a zero component and boxes outside the fp32 range go
// to surface_exact.
template <> __device__ __forceinline__ double surface<double>(const BoxDev& b, const Part<double>& q, int& kind) {
  const bool inner = q.region == 1u;
  const float xl = inner ? b.lo_f : 0.0f, xh = inner ? b.hi_f : b.side_f, eps = b.side_f * 0x1p-20f;
  bool sure = b.f32_ok != 0u;
  float t[3], e[3], p[3], inv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    sure = sure && mcx::f32_range(q.inv[a]);
    p[a] = mcx::f32_range(q.p[a]) ? mcx::f32_trunc(q.p[a]) : 0.0f;  // (out of the range: below 2^-120)
    inv[a] = mcx::f32_trunc(q.inv[a]);
    e[a] = fabsf(inv[a]) * eps;
    t[a] = ((inv[a] < 0.0f ? xl : xh) - p[a]) * inv[a];
  }
  // the nearest face ahead, and the least the other two can be
  const bool s1 = t[1] < t[0];
  const float m1 = s1 ? t[1] : t[0], f1 = s1 ? e[1] : e[0], o1 = s1 ? t[0] - e[0] : t[1] - e[1];
  const bool s2 = t[2] < m1;
  const float m = s2 ? t[2] : m1, f = s2 ? e[2] : f1;
  const float others = fminf(o1, s2 ? m1 - f1 : t[2] - e[2]);
  int ax = s2 ? 2 : (s1 ? 1 : 0);
  bool into = false;
  bool clear = others > m + f;
  if (!inner) {
    float n[3], lo_far = INFINITY, hi_far = INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const bool neg = inv[a] < 0.0f;
      n[a] = ((neg ? b.hi_f : b.lo_f) - p[a]) * inv[a];
      const float far = ((neg ? b.lo_f : b.hi_f) - p[a]) * inv[a];
      lo_far = fminf(lo_far, far - e[a]);
      hi_far = fminf(hi_far, far + e[a]);
    }
    // the last near face, and the most the other two can be
    const bool r1 = n[1] > n[0];
    const float k1 = r1 ? n[1] : n[0], g1 = r1 ? e[1] : e[0], h1 = r1 ? n[0] + e[0] : n[1] + e[1];
    const bool r2 = n[2] > k1;
    const float k = r2 ? n[2] : k1, g = r2 ? e[2] : g1;
    const float rest = fmaxf(h1, r2 ? k1 + g1 : n[2] + e[2]);
    const float hi_near = fmaxf(rest, k + g), lo_near = k - g;
    const bool miss = hi_near < 0.0f || lo_near > hi_far;
    const bool hit = lo_near > 0.0f && rest < lo_near && hi_near < lo_far && hi_near < fminf(others, m - f);
    into = hit;
    clear = hit || (miss && clear);
    if (hit) ax = r2 ? 2 : (r1 ? 1 : 0);
  }
  if (!(sure && clear)) {
    const Part<double> c = q;
    return surface_exact(&b, &c, &kind);
  }
  kind = inner || into ? 1 : 2;
  const double pa = ax == 2 ? q.p[2] : (ax == 1 ? q.p[1] : q.p[0]);
  const double ia = ax == 2 ? q.inv[2] : (ax == 1 ? q.inv[1] : q.inv[0]);
  // the face ahead of the particle (the near one of the inner cube, the far
  // one of the region it is in)
  const bool low = lt0(ia) != into;
  const double face = inner || into ? (low ? b.lo : b.hi) : (low ? 0.0 : b.side);
  const double ds = (face - pa) * ia;
  return lt0(ds) ? 0.0 : ds;
}

__device__ __forceinline__ long long fix_of(double wl) { return mcx::fix32_nonneg(wl); }
__device__ __forceinline__ long long fix_of(float wl) { return mcs::fix32_from_float(wl); }

// Mesh plane j: RN(j h) for j < mesh, side for j = mesh.  fp64: from the
// caller's table (shared memory, one problem per launch) or computed as one
// rounding of an exact integer product (mesh <= 1024).
constexpr int kMaxPlanes = MC_BOX_MAX_MESH + 1;
__device__ __forceinline__ double plane_of(const BoxDev& b, int j) {
  return j >= (int)b.mesh ? b.side : mcx::mul_small((uint32_t)j, b.h);
}
static __device__ __noinline__ double plane_call(const BoxDev* b, int j) { return plane_of(*b, j); }
template <typename T> __device__ __forceinline__ T plane(const BoxDev& b, const double* tab, int j);
template <> __device__ __forceinline__ double plane<double>(const BoxDev& b, const double* tab, int j) {
  return tab ? tab[j] : plane_call(&b, j);
}
template <> __device__ __forceinline__ float plane<float>(const BoxDev& b, const double*, int j) {
  return j >= (int)b.mesh ? b.side_f : (float)j * b.h_f;
}

template <typename T> __device__ __forceinline__ int voxel_guess(const BoxDev& b, T p);
template <> __device__ __forceinline__ int voxel_guess<double>(const BoxDev& b, double p) {
  return lt0(p) ? -1 : (int)min(mcx::guess_floor_mul(p, b.ih_q, b.ih_s), (uint64_t)b.mesh);
}
template <> __device__ __forceinline__ int voxel_guess<float>(const BoxDev& b, float p) {
  return (int)floorf(p * b.inv_h_f);
}

// The walk of a segment p + t u, 0 <= t <= L, through the mesh: t, the start
// of the current piece; per axis the distance tn to its next plane and that
// plane's index j; the voxel's slot.  A lane can leave the walk after any
// step and take it up again (the history kernel walks in chunks).  The axes
// are scalars picked by selects: arrays indexed by the crossed axis would
// live in local memory.
template <typename T>
struct Walk {
  T t, L, tn0, tn1, tn2;
  int j0, j1, j2;
  uint32_t slot;
};

// The voxel of coordinate p on one axis, from a guess i in [0, nm), and, as
// seen by direction u, the next plane j and its distance tn.  A looked-up guess
// is within one of the right voxel, the voxel the last flight ended in mostly
// right; the exact plane comparisons correct it, and put a particle on a plane on
// the side it flies to, in a rarely taken branch.
template <typename T>
__device__ __forceinline__ int walk_axis(const BoxDev& b, const double* tab, int nm, int i, T p, T u, T inv, int& j,
                                         T& tn) {
  T lo = plane<T>(b, tab, i), hi = plane<T>(b, tab, i + 1);
  const bool neg = lt0(u);
  if ((i > 0 && !ltn(lo, p)) || (i + 1 < nm && !ltn(p, hi))) {
    while (i > 0 && lt(p, lo)) { hi = lo; lo = plane<T>(b, tab, --i); }
    while (i + 1 < nm && !lt(p, hi)) { lo = hi; hi = plane<T>(b, tab, ++i + 1); }
    if (neg && i > 0 && eq(p, lo)) lo = plane<T>(b, tab, --i);
  }
  j = neg ? i : i + 1;
  tn = ((neg ? lo : hi) - p) * inv;
  if (lt0(tn)) tn = T(0);  // p beyond the plane by a rounding: an empty piece either way
  if (is0(u)) tn = T(INFINITY);
  return i;
}

template <typename T>
__device__ __forceinline__ int guess_axis(const BoxDev& b, int nm, T p) {
  const int i = voxel_guess<T>(b, p);
  return i < 0 ? 0 : (i >= nm ? nm - 1 : i);
}

// k.j0 .. k.j2: guesses of the particle's voxel, from its position ...
template <typename T>
__device__ __forceinline__ void walk_locate(const BoxDev& b, const Part<T>& q, Walk<T>& k) {
  const int nm = (int)b.mesh;
  k.j0 = guess_axis<T>(b, nm, q.p[0]);
  k.j1 = guess_axis<T>(b, nm, q.p[1]);
  k.j2 = guess_axis<T>(b, nm, q.p[2]);
}

// ... or, at the end of a walk in direction u, from its next planes.
template <typename T>
__device__ __forceinline__ void walk_leave(const BoxDev& b, const Part<T>& q, Walk<T>& k) {
  const int top = (int)b.mesh - 1;
  k.j0 = max(0, min(top, k.j0 - (lt0(q.u[0]) ? 0 : 1)));
  k.j1 = max(0, min(top, k.j1 - (lt0(q.u[1]) ? 0 : 1)));
  k.j2 = max(0, min(top, k.j2 - (lt0(q.u[2]) ? 0 : 1)));
}

template <typename T>
__device__ __forceinline__ void walk_begin(const BoxDev& b, const Part<T>& q, T L, const double* tab, Walk<T>& k) {
  const int nm = (int)b.mesh;
  const int i0 = walk_axis<T>(b, tab, nm, k.j0, q.p[0], q.u[0], q.inv[0], k.j0, k.tn0);
  const int i1 = walk_axis<T>(b, tab, nm, k.j1, q.p[1], q.u[1], q.inv[1], k.j1, k.tn1);
  const int i2 = walk_axis<T>(b, tab, nm, k.j2, q.p[2], q.u[2], q.inv[2], k.j2, k.tn2);
  k.slot = (uint32_t)((i2 * nm + i1) * nm + i0);  // mesh <= 1024: below 2^30
  k.t = T(0);
  k.L = L;
}

// One piece of the walk: its track length into the voxel (t to the next
// plane or to L), then across the plane.  The next crossing on an axis is
// computed from the segment start directly, t = (plane - p) / u, so every
// piece has the length the clipping definition gives it.  Returns true when
// the walk has ended (L reached, or the mesh left).  base: this history's
// [mesh^3] slot row.
template <typename T>
__device__ __forceinline__ bool walk_step(const BoxDev& b, const Part<T>& q, Walk<T>& k, unsigned long long* base,
                                          const double* tab, bool agg) {
  const bool y = ltn(k.tn1, k.tn0);
  const T t01 = y ? k.tn1 : k.tn0;
  const bool z = ltn(k.tn2, t01);
  const T ta = z ? k.tn2 : t01;
  const bool inside = ltn(ta, k.L);
  const T tend = inside ? ta : k.L;
  const unsigned long long v = (unsigned long long)fix_of(q.w * (tend - k.t));
  if (ltn(k.t, tend)) {
    if (agg) mcd::warp_agg_add(base + k.slot, v);
    else atomicAdd(base + k.slot, v);
    k.t = tend;
  }
  if (!inside) return true;
  const uint32_t nm = b.mesh;
  const T p = z ? q.p[2] : (y ? q.p[1] : q.p[0]), inv = z ? q.inv[2] : (y ? q.inv[1] : q.inv[0]);
  const int s = lt0(inv) ? -1 : 1;
  const int j = (z ? k.j2 : (y ? k.j1 : k.j0)) + s;
  k.slot += (uint32_t)s * (z ? nm * nm : (y ? nm : 1u));
  if ((uint32_t)j > nm) return true;  // the plane crossed was the mesh's face
  const T tn = (plane<T>(b, tab, j) - p) * inv;
  if (z) { k.j2 = j; k.tn2 = tn; }
  else if (y) { k.j1 = j; k.tn1 = tn; }
  else { k.j0 = j; k.tn0 = tn; }
  return false;
}

// The source up to its direction (three draws): position, weight, group.
template <int M, typename T>
__device__ __forceinline__ void source_position(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q) {
  const T side = sel<T>(b.side, b.side_f);
#pragma unroll
  for (int a = 0; a < 3; ++a) q.p[a] = side * from_n<T>(r.next_n(l));
  q.w = T(1);
  q.g = 0u;
}

template <int M, typename T>
__device__ __forceinline__ void box_source(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q) {
  source_position<M, T>(b, r, l, q);
  iso_dir<M, T>(r, l, q.u);
  set_inv(q);
  q.region = region_of<T>(b, q.p, q.u);
}

// The fp32 path's decision near the surface, made again in fp64 from the
// flight's uniform: bit 0 collide, the upper bits the surface's kind.  Out
// of line: about one flight in 2^15 takes it.
static __device__ __noinline__ int decide_f64(const BoxDev* b, float p0, float p1, float p2, float u0, float u1,
                                              float u2, uint32_t region, uint64_t n) {
  Part<double> q;
  q.p[0] = p0;
  q.p[1] = p1;
  q.p[2] = p2;
  q.u[0] = u0;
  q.u[1] = u1;
  q.u[2] = u2;
  for (int a = 0; a < 3; ++a) q.inv[a] = q.u[a] != 0.0 ? mcx::recip_rn(q.u[a]) : 0.0;
  q.region = region;
  int kind = 0;
  const double ds = surface_of<double>(*b, q, kind);
  const double d = mclog::neglog1m_n(n) * b->inv_st[region];
  return (d < ds ? 1 : 0) | (kind << 1);
}

// The length of the next flight and how it ends (kBoxCollide, kBoxCross or
// kBoxLeak): the sampled distance against the region surface.
template <int M, typename T>
__device__ __forceinline__ int flight_length(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, const Part<T>& q,
                                             T& len) {
  int kind = 0;
  const T ds = surface<T>(b, q, kind);
  bool collide;
  T d;
  if constexpr (sizeof(T) == 8) {
    d = mclog::neglog1m_n(r.next_n(l)) * b.inv_st[q.region];
    collide = lt(d, ds);
  } else {
    const uint64_t n = r.next_n(l);
    d = mcs::flight_f32(n) * b.inv_st_f[q.region];
    collide = d < ds;
    if (fabsf(d - ds) <= 0x1p-16f * fmaxf(d, ds)) {  // near the surface: decide in fp64
      const int k = decide_f64(&b, q.p[0], q.p[1], q.p[2], q.u[0], q.u[1], q.u[2], q.region, n);
      collide = (k & 1) != 0;
      kind = k >> 1;
    }
  }
  len = collide ? d : ds;
  return collide ? kBoxCollide : (kind == 2 ? kBoxLeak : kBoxCross);
}

// The end of a flight of length len: the particle at its end point, in the
// region it crossed into.
template <typename T>
__device__ __forceinline__ void arrive(Part<T>& q, T len, int outcome) {
#pragma unroll
  for (int a = 0; a < 3; ++a) q.p[a] = q.p[a] + len * q.u[a];
  if (outcome == kBoxCross) q.region ^= 1u;
}

// One flight: collide (position moved to the site), cross into the other
// region (moved to the surface), or leak out of the box.
template <int M, typename T>
__device__ __forceinline__ int box_flight(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q,
                                          unsigned long long* base, const double* tab, bool agg) {
  T len;
  const int o = flight_length<M, T>(b, r, l, q, len);
  Walk<T> k;
  walk_locate<T>(b, q, k);
  walk_begin<T>(b, q, len, tab, k);
  while (!walk_step<T>(b, q, k, base, tab, agg)) {}
  arrive<T>(q, len, o);
  return o;
}

// The integer form of u < v over u = n 2^-53, n < 2^53: n < threshold.  The
// comparison is that of the bit patterns read as signed integers (a value
// with its sign bit set is below every uniform, one of 1 or more, or a NaN,
// above).
__device__ __forceinline__ uint64_t cdf_threshold(double v) {
  const long long bits = __double_as_longlong(v);
  if (bits < 0) return 0ull;
  if (bits >= 0x3ff0000000000000ll) return 1ull << 53;
  return (uint64_t)ceil(v * 0x1p53);
}

// A collision up to the new direction: implicit capture and the group.
template <int M, typename T>
__device__ __forceinline__ void collide_group(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q) {
  const uint32_t rg = q.region;
  q.w = q.w * sel<T>(b.c[rg], b.c_f[rg]);
  const uint64_t ug = r.next_n(l);
  uint32_t g2 = q.g;
  for (uint32_t k = q.g; k < b.ng; ++k) {
    if (ug < b.cdf_n[rg][q.g][k]) {
      g2 = k;
      break;
    }
  }
  q.g = g2;
}

// The weight window after a collision's new direction: kBoxContinue,
// kBoxKilled (roulette), or kSplitBase + n for a split into n >= 2 (the
// parent keeps weight w/n; the caller creates the n-1 children from the
// parent's state after this call).
constexpr int kSplitBase = 8;
template <int M, typename T>
__device__ __forceinline__ int weight_window(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q) {
  const uint32_t rg = q.region;
  const T wl = sel<T>(b.wl[rg], b.wl_f[rg]), wh = sel<T>(b.wh[rg], b.wh_f[rg]);
  if (lt(q.w, wl)) {
    const T ws = sel<T>(b.ws[rg], b.ws_f[rg]);
    const uint64_t n = r.next_n(l);
    bool survives;
    if constexpr (sizeof(T) == 8) {
      // u < w / ws, decided in fp32 (each side off by less than a relative
      // 2^-21) unless the two are within a relative 2^-20
      const float u = mcs::u53_to_float(n), v = mcx::f32_trunc(q.w) * b.inv_ws_f[rg];
      survives = u < v * (1.0f - 0x1p-20f);
      if (!b.f32_ok || !mcx::f32_range(q.w) || (!survives && !(u > v * (1.0f + 0x1p-20f))))
        survives = lt(from_n<T>(n), q.w / ws);
    } else {
      survives = from_n<T>(n) < q.w / ws;
    }
    if (survives) {
      q.w = ws;
      return kBoxContinue;
    }
    return kBoxKilled;
  }
  if (lt(wh, q.w)) {
    const T nd = ceil(q.w / wh);
    const uint32_t ns = nd > (T)b.max_split ? b.max_split : (uint32_t)nd;
    if (ns > 1u) {
      q.w = q.w / (T)ns;
      return kSplitBase + (int)ns;  // (> every other outcome)
    }
  }
  return kBoxContinue;
}

// One collision: implicit capture, group, direction, weight window.
template <int M, typename T>
__device__ __forceinline__ int box_collide(const BoxDev& b, mcs::Rng<M>& r, const mcd::Lcg& l, Part<T>& q) {
  collide_group<M, T>(b, r, l, q);
  iso_dir<M, T>(r, l, q.u);
  set_inv(q);
  return weight_window<M, T>(b, r, l, q);
}

// Per-lane counters of one problem, flushed with atomics (lane by lane, or
// summed over a converged warp first: a problem's counters share a cache line).
struct BoxCounts {
  int prob;
  uint32_t src, flights, coll, leaks, kills, splits, children, capped, exh;
  uint64_t draws, exd, maxd;
  __device__ void clear() {
    src = flights = coll = leaks = kills = splits = children = capped = exh = 0u;
    draws = exd = maxd = 0ull;
  }
  __device__ void flush(unsigned long long* counts) {
    if (prob < 0) return;
    unsigned long long* c = counts + (size_t)prob * MC_NCOUNT;
    if (src) atomicAdd(c + MC_C_SOURCE, (unsigned long long)src);
    if (flights) atomicAdd(c + MC_C_FLIGHTS, (unsigned long long)flights);
    if (coll) {
      atomicAdd(c + MC_C_COLLISIONS, (unsigned long long)coll);
      atomicAdd(c + MC_C_SCATTERS, (unsigned long long)coll);
    }
    if (leaks) atomicAdd(c + MC_C_LEAK_HI, (unsigned long long)leaks);
    if (kills) atomicAdd(c + MC_C_ROULETTE_KILLS, (unsigned long long)kills);
    if (splits) atomicAdd(c + MC_C_SPLITS, (unsigned long long)splits);
    if (children) atomicAdd(c + MC_C_CHILDREN, (unsigned long long)children);
    if (capped) atomicAdd(c + MC_C_CAPPED, (unsigned long long)capped);
    if (exh) atomicAdd(c + MC_C_EXCEED_HIST, (unsigned long long)exh);
    if (draws) atomicAdd(c + MC_C_DRAWS, (unsigned long long)draws);
    if (exd) atomicAdd(c + MC_C_EXCEED_DRAWS, (unsigned long long)exd);
    if (maxd) atomicMax(c + MC_C_MAX_DRAWS, (unsigned long long)maxd);
    clear();
  }
  // The same for a whole converged warp: sums first, then one lane's atomics
  // (a problem's counters share a cache line).
  __device__ void flush_warp(unsigned long long* counts) {
    const int p = mcd::warp_common_prob(prob);
    if (p == -2) { flush(counts); return; }
    if (p < 0) return;
    const unsigned long long so = mcd::warp_sum64(src), fl = mcd::warp_sum64(flights), co = mcd::warp_sum64(coll),
                             le = mcd::warp_sum64(leaks), ki = mcd::warp_sum64(kills), sp = mcd::warp_sum64(splits),
                             ch = mcd::warp_sum64(children), cp = mcd::warp_sum64(capped), ex = mcd::warp_sum64(exh),
                             dr = mcd::warp_sum64(draws), ed = mcd::warp_sum64(exd), mx = mcd::warp_max64(maxd);
    if ((threadIdx.x & 31u) == 0u) {
      unsigned long long* c = counts + (size_t)p * MC_NCOUNT;
      if (so) atomicAdd(c + MC_C_SOURCE, so);
      if (fl) atomicAdd(c + MC_C_FLIGHTS, fl);
      if (co) {
        atomicAdd(c + MC_C_COLLISIONS, co);
        atomicAdd(c + MC_C_SCATTERS, co);
      }
      if (le) atomicAdd(c + MC_C_LEAK_HI, le);
      if (ki) atomicAdd(c + MC_C_ROULETTE_KILLS, ki);
      if (sp) atomicAdd(c + MC_C_SPLITS, sp);
      if (ch) atomicAdd(c + MC_C_CHILDREN, ch);
      if (cp) atomicAdd(c + MC_C_CAPPED, cp);
      if (ex) atomicAdd(c + MC_C_EXCEED_HIST, ex);
      if (dr) atomicAdd(c + MC_C_DRAWS, dr);
      if (ed) atomicAdd(c + MC_C_EXCEED_DRAWS, ed);
      if (mx) atomicMax(c + MC_C_MAX_DRAWS, mx);
    }
    clear();
  }
};

// Child k of a split: Eq. (5), S_c = hash(k, S_p) mod 2^m.
__device__ __forceinline__ uint64_t child_seed(uint32_t k, uint64_t parent_state, uint64_t mask) {
  return mcd::hash64((uint64_t)k, parent_state & mask) & mask;
}

template <typename T>
__device__ __forceinline__ void store_child(ChildRec& c, const Part<T>& q, uint64_t seed, uint32_t prob,
                                            uint64_t tbase) {
  for (int a = 0; a < 3; ++a) {
    c.p[a] = (double)q.p[a];
    c.u[a] = (double)q.u[a];
  }
  c.w = (double)q.w;
  c.rng = seed;
  c.tbase = tbase;
  c.g = q.g;
  c.region = q.region;
  c.prob = prob;
  c.pad = 0;
}

// A child's record but for the inverse of its direction (child_state), and
// the whole of it.
template <typename T>
__device__ __forceinline__ void child_state(const ChildRec& c, Part<T>& q) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    q.p[a] = (T)c.p[a];
    q.u[a] = (T)c.u[a];
  }
  q.w = (T)c.w;
  q.g = c.g;
  q.region = c.region;
}

template <typename T>
__device__ __forceinline__ void load_child(const ChildRec& c, Part<T>& q) {
  child_state(c, q);
  set_inv(q);
}

}  // namespace mcb
