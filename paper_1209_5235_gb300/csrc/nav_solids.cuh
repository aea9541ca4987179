// nav_solids.cuh -- the solids in FP64: frames, Inside, DistanceToIn, DistanceToOut and safety of boxes, orbs, tube
// segments and cones (included by nav_device.cuh; arithmetic only, no tables).
#pragma once

#include <cstdint>

#include "g4n_internal.h"

namespace g4n {
namespace dev {

constexpr double kInf = __builtin_huge_val();

struct V3 {
  double x, y, z;
};

__device__ __forceinline__ double comp(const V3 &v, int a) { return a == 0 ? v.x : (a == 1 ? v.y : v.z); }

// key(x): a double's bits as a signed integer with the negative half reflected, so that
// x < y <=> key(x) < key(y) for all non-NaN doubles (-0 < +0).
__device__ __forceinline__ long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
}

// ---------------------------------------------------------------- sums of products
// Written with their fused operations: the full formulas and the evaluation of one chosen surface (surf_ratio), each in several
// kernels, have to give the same bits, and the compiler fuses a plain sum of products by the uses of its terms.

// a b + c d and a b - c d.
__device__ __forceinline__ double dot2(double a, double b, double c, double d) { return fma(a, b, c * d); }
__device__ __forceinline__ double cross2(double a, double b, double c, double d) { return fma(a, b, -(c * d)); }
__device__ __forceinline__ double dot3(const V3 &p, const V3 &v) { return fma(p.z, v.z, dot2(p.x, v.x, p.y, v.y)); }
__device__ __forceinline__ double dot3_yx(const V3 &p, const V3 &v) { return fma(p.z, v.z, dot2(p.y, v.y, p.x, v.x)); }

// ---------------------------------------------------------------- frames

__device__ __forceinline__ void to_local(const DVol &v, const V3 &pm, const V3 &vm, V3 &pl, V3 &vl) {
  const double dx = pm.x - v.tx, dy = pm.y - v.ty;
  if (v.flags & kPlacedAligned) {
    pl = V3{dx, dy, pm.z - v.tz};
    vl = vm;
    return;
  }
  pl.x = dot2(v.c, dx, v.s, dy);
  pl.y = cross2(v.c, dy, v.s, dx);
  pl.z = pm.z - v.tz;
  vl.x = dot2(v.c, vm.x, v.s, vm.y);
  vl.y = cross2(v.c, vm.y, v.s, vm.x);
  vl.z = vm.z;
}

// World -> local frame of a volume; world-aligned volumes need only the translation.
__device__ __forceinline__ void world_to_local(const DWorld &w, bool aligned, const V3 &p, const V3 &u, V3 &pl,
                                               V3 &vl) {
  const double dx = p.x - w.tx, dy = p.y - w.ty;
  if (aligned) {
    pl = V3{dx, dy, p.z - w.tz};
    vl = u;
    return;
  }
  pl.x = dot2(w.c, dx, w.s, dy);
  pl.y = cross2(w.c, dy, w.s, dx);
  pl.z = p.z - w.tz;
  vl.x = dot2(w.c, u.x, w.s, u.y);
  vl.y = cross2(w.c, u.y, w.s, u.x);
  vl.z = u.z;
}

// World -> local frame of a point alone.
__device__ __forceinline__ V3 world_to_local_point(const DWorld &w, bool aligned, const V3 &p) {
  const double dx = p.x - w.tx, dy = p.y - w.ty;
  if (aligned) return V3{dx, dy, p.z - w.tz};
  return V3{dot2(w.c, dx, w.s, dy), cross2(w.c, dy, w.s, dx), p.z - w.tz};
}

// Reciprocal direction components (0 where the component is 0: never used there).
struct Inv3 {
  double x, y, z;
};

__device__ __forceinline__ Inv3 inv_dir(const V3 &v) {
  return Inv3{v.x != 0.0 ? 1.0 / v.x : 0.0, v.y != 0.0 ? 1.0 / v.y : 0.0, v.z != 0.0 ? 1.0 / v.z : 0.0};
}

__device__ __forceinline__ double icomp(const Inv3 &v, int a) { return a == 0 ? v.x : (a == 1 ? v.y : v.z); }

// ---------------------------------------------------------------- box

__device__ __forceinline__ bool box_inside(const double *h, const V3 &p, const V3 &v, double half) {
  const double ax = fabs(p.x) - h[0], ay = fabs(p.y) - h[1], az = fabs(p.z) - h[2];
  const double m = fmax(ax, fmax(ay, az));
  if (m > half) return false;
  if (m < -half) return true;
  if (ax >= -half && p.x * v.x >= 0.0) return false;
  if (ay >= -half && p.y * v.y >= 0.0) return false;
  if (az >= -half && p.z * v.z >= 0.0) return false;
  return true;
}

__device__ __forceinline__ double box_dist_in(const double *h, const V3 &p, const V3 &v, double half) {
  if ((fabs(p.x) - h[0] >= -half && p.x * v.x >= 0.0) || (fabs(p.y) - h[1] >= -half && p.y * v.y >= 0.0) ||
      (fabs(p.z) - h[2] >= -half && p.z * v.z >= 0.0))
    return kInf;
  double tin = -kInf, tout = kInf;
  const double pp[3] = {p.x, p.y, p.z}, vv[3] = {v.x, v.y, v.z};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (vv[i] != 0.0) {
      const double a = (-h[i] - pp[i]) / vv[i], b = (h[i] - pp[i]) / vv[i];
      tin = fmax(tin, fmin(a, b));
      tout = fmin(tout, fmax(a, b));
    }
  }
  if (!(tout > tin + half)) return kInf;
  return fmax(tin, 0.0);
}

// DistanceToOut with the reciprocal direction of the same frame; *face = the exit face
// (2 axis + (v_axis > 0)) of the first axis attaining the minimum.  The zero tests of
// v, the minimum and the clamp at 0 are integer operations on the bit patterns (the
// order-preserving keys of doubles), which give the same value as fmin/fmax.
__device__ __forceinline__ bool nonzero_bits(double x) { return (__double_as_longlong(x) << 1) != 0; }

__device__ __forceinline__ double box_dist_out(const double *h, const V3 &p, const V3 &v, const Inv3 &iv, int *face) {
  constexpr long long kKeyInf = 0x7FF0000000000000ll;  // key of +inf; NaN keys lie outside [key(-inf), key(+inf)]
  double t = kInf;
  long long kt = kKeyInf;
  int f = -1;
  const double pp[3] = {p.x, p.y, p.z}, vv[3] = {v.x, v.y, v.z}, ii[3] = {iv.x, iv.y, iv.z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!nonzero_bits(vv[a])) continue;
    const double ta = (copysign(h[a], vv[a]) - pp[a]) * ii[a];
    const long long k = dkey(ta);
    if (k < kt && k >= -kKeyInf - 1) {
      kt = k;
      t = ta;
      f = 2 * a + (vv[a] > 0.0 ? 1 : 0);
    }
  }
  *face = f;
  return kt < 0 ? 0.0 : t;
}

__device__ __forceinline__ double box_safety_in(const double *h, const V3 &p) {
  return fmax(fmax(fabs(p.x) - h[0], fmax(fabs(p.y) - h[1], fabs(p.z) - h[2])), 0.0);
}

__device__ __forceinline__ double box_safety_out(const double *h, const V3 &p) {
  return fmax(fmin(h[0] - fabs(p.x), fmin(h[1] - fabs(p.y), h[2] - fabs(p.z))), 0.0);
}

// ---------------------------------------------------------------- orb

// Discriminant of a t^2 + 2 b t + c.
__device__ __forceinline__ double quad_disc(double a, double b, double c) { return fma(b, b, -(a * c)); }

// Roots of a t^2 + 2 b t + c = 0 without cancellation; false if the discriminant is not positive.
__device__ __forceinline__ bool quad_roots(double a, double b, double c, double &lo, double &hi) {
  const double disc = quad_disc(a, b, c);
  if (!(disc > 0.0)) return false;
  const double sq = sqrt(disc);
  const double q = -(b + copysign(sq, b));
  const double r1 = q / a, r2 = c / q;
  lo = fmin(r1, r2);
  hi = fmax(r1, r2);
  return true;
}

__device__ __forceinline__ bool orb_inside(double R, const V3 &p, const V3 &v, double half) {
  const double r2 = p.x * p.x + p.y * p.y + p.z * p.z;
  const double ro = R + half, ri = R - half;
  if (r2 > ro * ro) return false;
  if (r2 < ri * ri) return true;
  return p.x * v.x + p.y * v.y + p.z * v.z < 0.0;
}

__device__ __forceinline__ double orb_dist_in(double R, const V3 &p, const V3 &v, double half) {
  const double b = dot3(p, v), c = fma(-R, R, dot3(p, p));
  double lo, hi;
  if (!quad_roots(1.0, b, c, lo, hi)) return kInf;
  return lo > half ? lo : kInf;
}

__device__ __forceinline__ double orb_dist_out(double R, const V3 &p, const V3 &v) {
  const double b = dot3_yx(p, v), c = fma(-R, R, dot3_yx(p, p));
  double lo, hi;
  if (!quad_roots(1.0, b, c, lo, hi)) return 0.0;
  return fmax(hi, 0.0);
}

__device__ __forceinline__ double orb_safety_in(double R, const V3 &p) {
  return fmax(sqrt(p.x * p.x + p.y * p.y + p.z * p.z) - R, 0.0);
}

__device__ __forceinline__ double orb_safety_out(double R, const V3 &p) {
  return fmax(R - sqrt(p.x * p.x + p.y * p.y + p.z * p.z), 0.0);
}

// ---------------------------------------------------------------- tube segment
// q[0..6] = rmin, rmax, hz, cos(sphi), sin(sphi), cos(ephi), sin(ephi).
// ps = cross(u_start, p) and pe = cross(p, u_end) are the signed distances to the
// lines of the two phi half-planes, positive on the solid's side.

__device__ __forceinline__ bool tube_phi_ok(const double *q, int flags, double x, double y, double tol) {
  if (!(flags & kSeg)) return true;
  const double ps = q[3] * y - q[4] * x, pe = q[6] * x - q[5] * y;
  return (flags & kWide) ? (ps >= -tol || pe >= -tol) : (ps >= -tol && pe >= -tol);
}

__device__ __forceinline__ bool tube_r_ok(const double *q, int flags, double x, double y, double half) {
  const double r2 = x * x + y * y, ro = q[1] + half;
  if (r2 > ro * ro) return false;
  if (flags & kHasRmin) {
    const double ri = q[0] - half;
    if (r2 < ri * ri) return false;
  }
  return true;
}

__device__ __noinline__ bool tube_inside(const double *q, int flags, const V3 &p, const V3 &v, double half) {
  const double sz = fabs(p.z) - q[2];
  if (sz > half) return false;
  const double r2 = p.x * p.x + p.y * p.y;
  const double ro = q[1] + half;
  if (r2 > ro * ro) return false;
  bool nz = sz >= -half;
  const double rmi = q[1] - half;
  bool nrmax = r2 >= rmi * rmi;
  bool nrmin = false;
  if (flags & kHasRmin) {
    const double ri = q[0] - half, rio = q[0] + half;
    if (r2 < ri * ri) return false;
    nrmin = r2 <= rio * rio;
  }
  bool ns = false, ne = false;
  if (flags & kSeg) {
    const double ps = q[3] * p.y - q[4] * p.x, pe = q[6] * p.x - q[5] * p.y;
    if (!(flags & kWide)) {
      if (ps < -half || pe < -half) return false;
      ns = ps <= half;
      ne = pe <= half;
    } else {
      const double m = fmax(ps, pe);
      if (m < -half) return false;
      if (m <= half) {
        if (ps >= pe) ns = true;
        else ne = true;
      }
    }
  }
  if (!(nz || nrmax || nrmin || ns || ne)) return true;
  const double vr = p.x * v.x + p.y * v.y;
  if (nz && !(p.z * v.z < 0.0)) return false;
  if (nrmax && !(vr < 0.0)) return false;
  if (nrmin && !(vr > 0.0)) return false;
  if (ns && !(q[4] * v.x - q[3] * v.y < 0.0)) return false;
  if (ne && !(q[5] * v.y - q[6] * v.x < 0.0)) return false;
  return true;
}

// The crossings tube_cross takes the first of, one helper per surface: each returns its crossing
// parameter t when t lies in (tmin, best) and the crossing passes the surface's range tests, else
// +inf.
// z plane the ray enters (enter) or leaves (exit) through
__device__ __forceinline__ double tube_z_cand(const double *q, int flags, const V3 &p, const V3 &v, double half,
                                              bool enter, double tmin) {
  if (v.z == 0.0) return kInf;
  const double sg = ((v.z < 0.0) == enter) ? 1.0 : -1.0;
  const double t = (sg * q[2] - p.z) / v.z;
  if (!(t > tmin)) return kInf;
  const double qx = p.x + t * v.x, qy = p.y + t * v.y;
  return (tube_r_ok(q, flags, qx, qy, half) && tube_phi_ok(q, flags, qx, qy, half)) ? t : kInf;
}

// cylinder of radius R (outer: the root that enters / leaves the solid through rmax; inner: through rmin)
__device__ __forceinline__ double tube_cyl_cand(const double *q, int flags, const V3 &p, const V3 &v, double half,
                                                bool enter, double tmin, double best, bool outer) {
  const double a = dot2(v.x, v.x, v.y, v.y);
  if (!(a > 0.0)) return kInf;
  const double b = dot2(p.x, v.x, p.y, v.y);
  const double R = outer ? q[1] : q[0];
  double lo, hi;
  if (!quad_roots(a, b, fma(-R, R, dot2(p.y, p.y, p.x, p.x)), lo, hi)) return kInf;
  const double t = (enter == outer) ? lo : hi;
  if (t > tmin && t < best && fabs(p.z + t * v.z) <= q[2] + half &&
      tube_phi_ok(q, flags, p.x + t * v.x, p.y + t * v.y, half))
    return t;
  return kInf;
}

// phi half-plane at the start (start = true) or end of the segment
__device__ __forceinline__ double tube_phi_cand(const double *q, int flags, const V3 &p, const V3 &v, double half,
                                                bool enter, double tmin, double best, bool start) {
  // v . outward normal of the plane, the signed distance to its line (positive on the solid's side)
  const double dn = start ? cross2(q[4], v.x, q[3], v.y) : cross2(q[5], v.y, q[6], v.x);
  if (!(dn != 0.0 && ((dn < 0.0) == enter))) return kInf;
  const double t = (start ? cross2(q[3], p.y, q[4], p.x) : cross2(q[6], p.x, q[5], p.y)) / dn;
  if (!(t > tmin && t < best)) return kInf;
  const double qx = p.x + t * v.x, qy = p.y + t * v.y;
  const double along = start ? q[3] * qx + q[4] * qy : q[5] * qx + q[6] * qy;
  return (along >= -half && tube_r_ok(q, flags, qx, qy, half) && fabs(p.z + t * v.z) <= q[2] + half) ? t : kInf;
}

// enter = true: first entering crossing with t > half (DistanceToIn);
// enter = false: first exiting crossing with t > -half (DistanceToOut, clamped by the caller).
__device__ __noinline__ double tube_cross(const double *q, int flags, const V3 &p, const V3 &v, double half, bool enter) {
  const double tmin = enter ? half : -half;
  double best = tube_z_cand(q, flags, p, v, half, enter, tmin);
  best = fmin(best, tube_cyl_cand(q, flags, p, v, half, enter, tmin, best, true));
  if (flags & kHasRmin) best = fmin(best, tube_cyl_cand(q, flags, p, v, half, enter, tmin, best, false));
  if (flags & kSeg) {
    best = fmin(best, tube_phi_cand(q, flags, p, v, half, enter, tmin, best, true));
    best = fmin(best, tube_phi_cand(q, flags, p, v, half, enter, tmin, best, false));
  }
  return best;
}

__device__ __forceinline__ double tube_safety_in(const double *q, int flags, const V3 &p) {
  const double r = sqrt(p.x * p.x + p.y * p.y);
  double m = fmax(r - q[1], fabs(p.z) - q[2]);
  if (flags & kHasRmin) m = fmax(m, q[0] - r);
  if (flags & kSeg) {
    const double a = q[4] * p.x - q[3] * p.y, b = q[5] * p.y - q[6] * p.x;
    m = fmax(m, (flags & kWide) ? fmin(a, b) : fmax(a, b));
  }
  return fmax(m, 0.0);
}

__device__ __forceinline__ double tube_safety_out(const double *q, int flags, const V3 &p) {
  const double r = sqrt(p.x * p.x + p.y * p.y);
  double m = fmin(q[1] - r, q[2] - fabs(p.z));
  if (flags & kHasRmin) m = fmin(m, r - q[0]);
  if (flags & kSeg) m = fmin(m, fmin(fabs(q[3] * p.y - q[4] * p.x), fabs(q[6] * p.x - q[5] * p.y)));
  return fmax(m, 0.0);
}

// ---------------------------------------------------------------- cone (full in phi)
// q[0..6] = ki, ci, ko, co, hz, cos(inner half-angle), cos(outer half-angle): between
// z = -hz and +hz the solid is Rin(z) <= r <= Rout(z), Rout = ko z + co, Rin = ki z + ci
// (flag kHasRmin: inner surface present).  Bands along r at the point's z; outward normal of
// the outer surface along (x / r, y / r, -ko), of the inner one along (-x / r, -y / r, ki).

__device__ __noinline__ bool cone_inside(const double *q, int flags, const V3 &p, const V3 &v, double half) {
  const double sz = fabs(p.z) - q[4];
  if (sz > half) return false;
  const double r2 = p.x * p.x + p.y * p.y;
  const double ro = q[2] * p.z + q[3];
  const double rop = ro + half, rom = ro - half;
  if (r2 > rop * rop) return false;
  const bool nz = sz >= -half;
  const bool nrmax = r2 >= rom * rom;
  bool nrmin = false;
  if (flags & kHasRmin) {
    const double ri = q[0] * p.z + q[1];
    const double rim = ri - half, rip = ri + half;
    if (r2 < rim * rim) return false;
    nrmin = r2 <= rip * rip;
  }
  if (!(nz || nrmax || nrmin)) return true;
  const double r = sqrt(r2);
  const double vr = p.x * v.x + p.y * v.y;
  if (nz && !(p.z * v.z < 0.0)) return false;
  if (nrmax && !(vr - q[2] * r * v.z < 0.0)) return false;
  if (nrmin && !(vr - q[0] * r * v.z > 0.0)) return false;
  return true;
}

// enter = true: first entering crossing with t > half; enter = false: first exiting crossing
// with t > -half.  Conical surfaces: a t^2 + 2 b t + cc = 0 with d = a t + b half the rate of
// change of r^2 - R^2 along the ray (entering the solid: d < 0 at the outer surface, d > 0 at
// the inner one); roots on the other half of the double cone (R < 0) are not surface points.
__device__ __noinline__ double cone_cross(const double *q, int flags, const V3 &p, const V3 &v, double half, bool enter) {
  const double tmin = enter ? half : -half;
  const double hz = q[4];
  double best = kInf;
  if (v.z != 0.0) {
    const double sg = ((v.z < 0.0) == enter) ? 1.0 : -1.0;
    const double t = (sg * hz - p.z) / v.z;
    if (t > tmin) {
      const double qx = p.x + t * v.x, qy = p.y + t * v.y;
      const double r2 = qx * qx + qy * qy;
      const double ro = q[2] * (sg * hz) + q[3] + half;
      bool ok = r2 <= ro * ro;
      if (flags & kHasRmin) {
        const double ri = q[0] * (sg * hz) + q[1] - half;
        ok = ok && !(r2 < ri * ri);
      }
      if (ok) best = t;
    }
  }
  const int nw = (flags & kHasRmin) ? 2 : 1;
#pragma unroll 1
  for (int w = 0; w < nw; ++w) {
    const double k = w == 0 ? q[2] : q[0], c = w == 0 ? q[3] : q[1];
    const double rz = k * p.z + c;
    const double a = v.x * v.x + v.y * v.y - k * k * v.z * v.z;
    const double b = p.x * v.x + p.y * v.y - k * v.z * rz;
    const double cc = p.x * p.x + p.y * p.y - rz * rz;
    double t0 = kInf, t1 = kInf;
    if (a != 0.0) {
      const double disc = b * b - a * cc;
      if (disc > 0.0) {
        const double sq = sqrt(disc);
        const double qq = -(b + copysign(sq, b));
        t0 = qq / a;
        t1 = cc / qq;
      }
    } else if (b != 0.0) {
      t0 = -cc / (2.0 * b);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const double t = i == 0 ? t0 : t1;
      if (!(t > tmin && t < best)) continue;
      const double d = a * t + b;
      const bool into = w == 0 ? d < 0.0 : d > 0.0;
      if (into != enter) continue;
      const double qz = p.z + t * v.z;
      if (fabs(qz) > hz + half) continue;
      if (!(k * qz + c >= 0.0)) continue;
      best = t;
    }
  }
  return best;
}

__device__ __forceinline__ double cone_safety_in(const double *q, int flags, const V3 &p) {
  const double r = sqrt(p.x * p.x + p.y * p.y);
  double m = fmax(fabs(p.z) - q[4], (r - (q[2] * p.z + q[3])) * q[6]);
  if (flags & kHasRmin) m = fmax(m, ((q[0] * p.z + q[1]) - r) * q[5]);
  return fmax(m, 0.0);
}

__device__ __forceinline__ double cone_safety_out(const double *q, int flags, const V3 &p) {
  const double r = sqrt(p.x * p.x + p.y * p.y);
  double m = fmin(q[4] - fabs(p.z), ((q[2] * p.z + q[3]) - r) * q[6]);
  if (flags & kHasRmin) m = fmin(m, (r - (q[0] * p.z + q[1])) * q[5]);
  return fmax(m, 0.0);
}

}  // namespace dev
}  // namespace g4n
