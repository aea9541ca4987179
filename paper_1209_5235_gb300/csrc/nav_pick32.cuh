// nav_pick32.cuh -- which surface of a solid a ray crosses, decided in FP32 (included by nav_device.cuh).
//
// An FP64 instruction of a warp holds GB300's FP64 pipe for 16 cycles of the whole SM, whatever the number of its
// lanes; an FP32 one for half a cycle.  A tube segment's DistanceToIn or DistanceToOut in FP64 evaluates five surfaces
// with their range tests (seven divisions, two square roots, ~160 FP64 instructions), of which one surface's crossing
// parameter is the answer.  Here FP32 arithmetic with error bounds finds that surface, and only its parameter is
// evaluated in FP64 (one division, at most one square root): the full formulas' value, because the bounds prove that
// every other one is later, earlier than the start, or not on the solid.  Where they do not prove it the caller takes the
// full FP64 formulas.
//
// A solid along the ray is the interval between its last entry into and its first exit from the half-spaces and the
// cylinder whose intersection is its convex hull (the Hull below), less the interval inside its bore.  Each crossing
// parameter is kept as [t - e, t + e].
//
// The tolerance band is part of the bounds.  The FP64 formulas accept a crossing up to half a band outside the solid's other
// surfaces and refuse a start in a band, so a comparison of two crossings has to hold wherever each surface lies within its
// band: pick_solid adds the band to the bound of the point's error.  At the default tolerance that changes nothing for solids of a millimetre and
// more (2e-7 of their size in FP32 rounding against 1e-9 mm); solids of 1e-4 mm, or tolerances of 1e-5 of a solid's size,
// are decided in the full formulas more often.
//
// Error bounds.  u = 2^-23.  The FP32 point differs from the exact one by at most ep in each coordinate (the caller's
// bound: conversions, and the rotation into the solid's frame), sizes and plane normals are within u/2 relative, the
// direction's components within 4u of its length in the plane they are rotated in.  The helpers add their own roundings
// (approximate reciprocal and root: within u).  Derivations stand at each helper.
#pragma once

#include "nav_solids.cuh"

namespace g4n {
namespace dev {

// Approximate reciprocal and square root, relative error below u (MUFU; the host side of the tests has its own).
#ifdef __CUDACC__
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#endif

constexpr float kU = 1.1920929e-7f;
constexpr float kPickInf = __builtin_huge_valf();

// Surfaces: boxes 2 axis + (direction component > 0); tubes as below; orbs 0.
enum PickSurf : int { kPickMiss = -1, kPickUnsure = -2, kPickLeaving = -3, kPickZ = 0, kPickOuter = 1, kPickInner = 2, kPickStart = 3, kPickEnd = 4 };

struct Pick {
  int surf;       // the surface, kPickMiss (no crossing), kPickUnsure (the bounds do not decide) or kPickLeaving (a box
                  // DistanceToIn from inside, or from where it is left: zero or none)
  float lo, hi;   // enclosure of the crossing parameter; unsure: a lower bound in lo
};

// A double truncated to float by integer instructions (a conversion instruction costs as much as an FP64 add): |error|
// < u |x|; below 2^-126 zero, above FLT_MAX the largest float.
__device__ __forceinline__ float trunc_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sg = hi & 0x80000000u;
  const unsigned t = (hi & 0x7fffffffu) - 0x38000000u;   // exponent rebased to float's
  if ((int)t < 0x00100000) return __uint_as_float(sg);
  if (t >= 0x0ff00000u) return __uint_as_float(sg | 0x7f7fffffu);
  return __uint_as_float(sg | (t << 3) | (lo >> 29));
}

// Entries into and exits from the convex constraints: the latest entry a and the earliest exit b, with bounds.
struct Hull {
  float at, alo, ahi, a2hi;   // entry with the largest t; alo: bound from below of the latest entry; its own upper bound;
  int aid;                    //   the largest upper bound of the other entries; its surface
  float bt, bhi, blo, b2lo;   // exit with the smallest t; upper bound of the earliest exit; its own lower bound; the
  int bid;                    //   smallest lower bound of the other exits; its surface
};

__device__ __forceinline__ Hull hull_all() {
  return Hull{-kPickInf, -kPickInf, -kPickInf, -kPickInf, kPickMiss, kPickInf, kPickInf, kPickInf, kPickInf, kPickMiss};
}

__device__ __forceinline__ void hull_entry(Hull &H, float t, float e, int id) {
  if (t > H.at) {
    H.a2hi = fmaxf(H.a2hi, H.ahi);
    H.at = t;
    H.ahi = t + e;
    H.aid = id;
  } else {
    H.a2hi = fmaxf(H.a2hi, t + e);
  }
  H.alo = fmaxf(H.alo, t - e);
}

__device__ __forceinline__ void hull_exit(Hull &H, float t, float e, int id) {
  if (t < H.bt) {
    H.b2lo = fminf(H.b2lo, H.blo);
    H.bt = t;
    H.blo = t - e;
    H.bid = id;
  } else {
    H.b2lo = fminf(H.b2lo, t - e);
  }
  H.bhi = fminf(H.bhi, t + e);
}

// A constraint that the ray enters not before t = g, if at all / leaves not before t = g, if at all / anything.
__device__ __forceinline__ void hull_enter_after(Hull &H, float g) {
  H.alo = fmaxf(H.alo, g);
  H.a2hi = kPickInf;
}
__device__ __forceinline__ void hull_leave_after(Hull &H, float g) { H.b2lo = fminf(H.b2lo, g); }
__device__ __forceinline__ void hull_unsure(Hull &H) {
  H.a2hi = kPickInf;
  H.b2lo = -kPickInf;
}

// Error of a plane's rate of change v . n: the direction's component (4u, after a rotation) and the normal's (u/2 of
// its two components), with the rounding of the two products: below 10u.
constexpr float kDn = 10.0f * kU;

// Half-space d + t dn >= 0; ed bounds the error of d.  t = -d / dn; with |dn| > 4 kDn the quotient's error is at most
// (ed + |t| kDn) / (|dn| - kDn) <= 4/3 (ed + |t| kDn) / |dn|, plus the roundings of reciprocal and product, 2u |t|.
// A smaller |dn| has no certain sign: the plane is crossed beyond (|d| - ed) / (5 kDn), if at all.
__device__ __forceinline__ void hull_plane(Hull &H, float d, float dn, float ed, int id) {
  const float m = fabsf(dn);
  if (m > 4.0f * kDn) {
    const float r = rcp_approx(dn), t = -d * r;
    const float e = 1.4f * (ed + fabsf(t) * kDn) * fabsf(r) + 4.0f * kU * fabsf(t);
    if (dn > 0.0f) hull_entry(H, t, e, id);
    else hull_exit(H, t, e, id);
  } else if (fabsf(d) <= ed) {
    hull_unsure(H);
  } else {
    const float g = (fabsf(d) - ed) * (0.2f / kDn);
    if (d > 0.0f) hull_leave_after(H, g);
    else {
      hull_enter_after(H, g);
      hull_leave_after(H, g);
    }
  }
}

// Slab |x| <= h (both planes of hull_plane; one reciprocal).
__device__ __forceinline__ void hull_slab(Hull &H, float x, float v, float h, float ed, int id) {
  const float m = fabsf(v);
  if (m > 4.0f * kDn) {
    const float r = rcp_approx(m), xs = v > 0.0f ? x : -x;
    const float t0 = (-h - xs) * r, t1 = (h - xs) * r;
    hull_entry(H, t0, 1.4f * (ed + fabsf(t0) * kDn) * r + 4.0f * kU * fabsf(t0), id);
    hull_exit(H, t1, 1.4f * (ed + fabsf(t1) * kDn) * r + 4.0f * kU * fabsf(t1), id);
  } else {
    const float d = h - fabsf(x);
    if (fabsf(d) <= ed) {
      hull_unsure(H);
    } else {
      const float g = (fabsf(d) - ed) * (0.2f / kDn);
      if (d < 0.0f) hull_enter_after(H, g);
      hull_leave_after(H, g);
    }
  }
}

// Crossings of a circle (or sphere) of radius R by the line: a t^2 + 2 b t + c = 0 with a = |w|^2, b = q . w, c = |q|^2 -
// R^2, q the point and w the direction in its plane; s >= |q|_1 + R bounds the lengths.
//  * Coefficient errors: da <= 14u a, db <= sqrt(a) (2 ep + 7u s), dc <= 4 s ep + 4u s^2 (three coordinates included).
//  * At a root t the quadratic's error is da t^2 + 2 |t| db + dc <= n = k (14u k + 4 ep) with k = sqrt(a) |t| + s, and the
//    root's error n / (2 sqrt(disc)) to first order; the second order is covered by the factor 2 where disc >= 8 a n.
//  * disc's error is below E = a (12 s ep + 60u s^2): a disc below -E means that the line misses the circle.
// Roots that fail the test of n have only the bound of the gap: the radius is reached after (|r - R| - errors) / sqrt(a).
enum RootState : int { kRootsMiss, kRootsOk, kRootsGapIn, kRootsGapOut, kRootsUnsure };
struct Roots {
  int state;                // GapIn / GapOut: only the bound g, the point inside / outside the circle
  float t0, e0, t1, e1, g;
};

__device__ __forceinline__ Roots circle_roots(float a, float sa, float b, float r2, float R, float s, float ep) {
  Roots Q;
  const float c = r2 - R * R, disc = b * b - a * c;
  Q.state = kRootsMiss;
  if (disc < -a * s * (12.0f * ep + 60.0f * kU * s)) return Q;
  const float sq = sqrt_approx(fmaxf(disc, 0.0f)), rs = rcp_approx(sq);
  const float q = -(b + copysignf(sq, b));
  const float r1 = q * rcp_approx(a), r2_ = c * rcp_approx(q);
  Q.t0 = fminf(r1, r2_);
  Q.t1 = fmaxf(r1, r2_);
  const float k0 = sa * fabsf(Q.t0) + s, k1 = sa * fabsf(Q.t1) + s;
  const float n0 = k0 * (14.0f * kU * k0 + 4.0f * ep), n1 = k1 * (14.0f * kU * k1 + 4.0f * ep);
  Q.e0 = n0 * rs + 4.0f * kU * fabsf(Q.t0);
  Q.e1 = n1 * rs + 4.0f * kU * fabsf(Q.t1);
  if (a > 1e-20f && disc >= 8.0f * a * fmaxf(n0, n1)) {   // false for NaN as well
    Q.state = kRootsOk;
    return Q;
  }
  const float gap = sqrt_approx(r2) - R, far = fabsf(gap) - 3.0f * ep - 6.0f * kU * s;
  Q.state = !(far > 0.0f) ? kRootsUnsure : gap < 0.0f ? kRootsGapIn : kRootsGapOut;
  Q.g = far * rcp_approx(fmaxf(sa, 1e-30f)) * (1.0f - 16.0f * kU);
  return Q;
}

__device__ __forceinline__ void hull_circle(Hull &H, const Roots &Q, int id) {
  if (Q.state == kRootsOk) {
    hull_entry(H, Q.t0, Q.e0, id);
    hull_exit(H, Q.t1, Q.e1, id);
  } else if (Q.state == kRootsMiss) {
    H.alo = kPickInf;
    H.bhi = -kPickInf;
  } else if (Q.state == kRootsUnsure) {
    hull_unsure(H);
  } else {
    if (Q.state == kRootsGapOut) hull_enter_after(H, Q.g);
    hull_leave_after(H, Q.g);
  }
}

// The interval of the ray inside the bore: [h0, h1], each with bounds; +inf where the ray never enters it.
struct Bore {
  float h0lo, h0hi, h1lo, h1hi;
};
__device__ __forceinline__ Bore bore_of(const Roots &Q) {
  if (Q.state == kRootsOk) return Bore{Q.t0 - Q.e0, Q.t0 + Q.e0, Q.t1 - Q.e1, Q.t1 + Q.e1};
  if (Q.state == kRootsMiss) return Bore{kPickInf, kPickInf, kPickInf, kPickInf};
  if (Q.state == kRootsGapOut) return Bore{Q.g, kPickInf, Q.g, kPickInf};
  if (Q.state == kRootsGapIn) return Bore{-kPickInf, -kPickInf, Q.g, kPickInf};
  return Bore{-kPickInf, kPickInf, -kPickInf, kPickInf};
}

// DistanceToIn from the hull and the bore: the first entering crossing beyond the band.  Entering the hull counts unless
// the entry lies in the bore; leaving the bore inside the hull counts (in the bore at the hull's entry or start).
// A start in the band of the entry surface is unsure (its crossing is at t = 0 within the errors).
__device__ __forceinline__ Pick pick_enter(const Hull &H, const Bore &B, float band) {
  const float ahigh = fmaxf(H.ahi, H.a2hi), blow = fminf(H.blo, H.b2lo);
  if (H.alo > H.bhi || H.bhi < 0.0f) return Pick{kPickMiss, 0.f, 0.f};
  if (H.a2hi < H.alo && H.alo > band && ahigh + band < blow && (ahigh < B.h0lo || H.alo > B.h1hi))
    return Pick{H.aid, H.alo, H.ahi};
  if (ahigh < 0.0f || (H.alo > B.h0hi && ahigh < B.h1lo)) {   // no entry into the hull, or one in the bore
    if (B.h1hi < 0.0f || B.h1lo >= H.bhi) return Pick{kPickMiss, 0.f, 0.f};
    if (B.h1lo > band && B.h1lo > ahigh && B.h1hi + band < blow) return Pick{kPickInner, B.h1lo, B.h1hi};
  }
  return Pick{kPickUnsure, fmaxf(H.alo, 0.0f), kPickInf};
}

// DistanceToOut from inside: the first exit from the hull or entry into the bore.  A point that is not inside within the
// errors, or deep in the bore, is unsure.
__device__ __forceinline__ Pick pick_exit(const Hull &H, const Bore &B) {
  const bool bore = !(B.h0hi < 0.0f);   // the bore's entry is still ahead
  if (H.alo > 0.0f || H.bhi < 0.0f || (!bore && B.h1lo > 0.0f)) return Pick{kPickUnsure, 0.f, kPickInf};
  if (H.b2lo > H.bhi && (!bore || B.h0lo > H.bhi)) return Pick{H.bid, H.blo, H.bhi};
  if (bore && B.h0hi < fminf(H.blo, H.b2lo)) return Pick{kPickInner, B.h0lo, B.h0hi};
  return Pick{kPickUnsure, 0.f, kPickInf};
}

// The solids' hulls.  (x, y, z), (vx, vy, vz): point and direction in the solid's frame; q: the solid's sizes as in DVol.

template <bool ENTER>
__device__ __forceinline__ Pick pick_box(const float *q, float x, float y, float z, float vx, float vy, float vz, float ep,
                                         float band) {
  Hull H = hull_all();
  const float ed = 2.0f * ep;
  hull_slab(H, x, vx, q[0], ed, 0 + (vx > 0.0f));
  hull_slab(H, y, vy, q[1], ed, 2 + (vy > 0.0f));
  hull_slab(H, z, vz, q[2], ed, 4 + (vz > 0.0f));
  const Bore none{kPickInf, kPickInf, kPickInf, kPickInf};
  if (ENTER && fmaxf(H.ahi, H.a2hi) < 0.0f && H.bhi >= 0.0f) return Pick{kPickLeaving, 0.f, kPickInf};
  return ENTER ? pick_enter(H, none, band) : pick_exit(H, none);
}

template <bool ENTER>
__device__ __forceinline__ Pick pick_orb(float R, float x, float y, float z, float vx, float vy, float vz, float ep,
                                         float band) {
  Hull H = hull_all();
  // the FP64 formulas take |v|^2 = 1
  const Roots Q = circle_roots(1.0f, 1.0f, x * vx + y * vy + z * vz, x * x + y * y + z * z, R,
                               fabsf(x) + fabsf(y) + fabsf(z) + R, ep);
  hull_circle(H, Q, 0);
  const Bore none{kPickInf, kPickInf, kPickInf, kPickInf};
  return ENTER ? pick_enter(H, none, band) : pick_exit(H, none);
}

// Segments wider than pi are not convex in phi: unsure.
template <bool ENTER>
__device__ __forceinline__ Pick pick_tube(const float *q, int flags, float x, float y, float z, float vx, float vy, float vz,
                                          float ep, float band) {
  if ((flags & (kSeg | kWide)) == (kSeg | kWide)) return Pick{kPickUnsure, 0.f, kPickInf};
  Hull H = hull_all();
  const float ed = 2.0f * ep;
  hull_slab(H, z, vz, q[2], ed, kPickZ);
  if (flags & kSeg) {
    hull_plane(H, q[3] * y - q[4] * x, q[3] * vy - q[4] * vx, ed, kPickStart);
    hull_plane(H, q[6] * x - q[5] * y, q[6] * vx - q[5] * vy, ed, kPickEnd);
  }
  const float a = vx * vx + vy * vy, sa = sqrt_approx(a), b = x * vx + y * vy, r2 = x * x + y * y;
  const float l1 = fabsf(x) + fabsf(y);
  hull_circle(H, circle_roots(a, sa, b, r2, q[1], l1 + q[1], ep), kPickOuter);
  Bore B{kPickInf, kPickInf, kPickInf, kPickInf};
  if (flags & kHasRmin) B = bore_of(circle_roots(a, sa, b, r2, q[0], l1 + q[0], ep));
  return ENTER ? pick_enter(H, B, band) : pick_exit(H, B);
}

template <bool ENTER>
__device__ __forceinline__ Pick pick_solid(int kind, const float *q, int flags, float x, float y, float z, float vx,
                                           float vy, float vz, float ep, float band) {
  ep += band;   // every surface may lie half a band further in or out
  if (kind == kBox) return pick_box<ENTER>(q, x, y, z, vx, vy, vz, ep, band);
  if (kind == kOrb) return pick_orb<ENTER>(q[0], x, y, z, vx, vy, vz, ep, band);
  if (kind == kTube) return pick_tube<ENTER>(q, flags, x, y, z, vx, vy, vz, ep, band);
  return Pick{kPickUnsure, 0.f, kPickInf};   // cones
}

// The crossing parameter of one surface in FP64 as a quotient num / den, by the formulas of the full tests and with their
// operations in their order, for the same bits (nav_solids.cuh's fused sums; a box's exit takes the reciprocal): planes, and
// circles through the quadratic's root without cancellation (lo: q / a where q < 0, else c / q; hi the other one).  The
// caller divides: one division for all lanes of a warp whatever their surfaces.  NaN where the quadratic has no root.
__device__ __forceinline__ void surf_ratio(int kind, const double *p, int surf, bool enter, const V3 &x, const V3 &v,
                                           double &num, double &den) {
  if (kind == kBox) {
    const int a = surf >> 1;
    const double va = comp(v, a), h = copysign(a == 0 ? p[0] : (a == 1 ? p[1] : p[2]), va);
    num = (enter ? -h : h) - comp(x, a);
    den = va;
  } else if (kind == kTube && surf == kPickZ) {
    num = (((v.z < 0.0) == enter) ? p[2] : -p[2]) - x.z;
    den = v.z;
  } else if (kind == kTube && surf >= kPickStart) {
    const bool st = surf == kPickStart;
    num = cross2(st ? p[3] : p[6], st ? x.y : x.x, st ? p[4] : p[5], st ? x.x : x.y);
    den = cross2(st ? p[4] : p[5], st ? v.x : v.y, st ? p[3] : p[6], st ? v.y : v.x);
  } else {
    const bool orb = kind != kTube;
    const double a = orb ? 1.0 : dot2(v.x, v.x, v.y, v.y), R = !orb && surf == kPickOuter ? p[1] : p[0];
    // the terms in the order of orb_dist_in, orb_dist_out and tube_cyl_cand
    const bool by = orb && !enter, cy = !orb || !enter;
    double b = dot2(by ? x.y : x.x, by ? v.y : v.x, by ? x.x : x.y, by ? v.x : v.y);
    const double c0 = cy ? x.y : x.x, c1 = cy ? x.x : x.y;
    double c = dot2(c0, c0, c1, c1);
    if (orb) {
      b = fma(x.z, v.z, b);
      c = fma(x.z, x.z, c);
    }
    c = fma(-R, R, c);
    const double sq = sqrt(quad_disc(a, b, c)), q = -(b + copysign(sq, b));
    const bool lo = enter == (orb || surf == kPickOuter);
    const bool direct = lo == (__double2hiint(b) >= 0);   // by q's sign: b may be -0 (a ray from the axis)
    num = direct ? q : c;
    den = direct ? a : q;
  }
}

// A double as the sum of two floats: hi truncated, lo the next 24 of the 29 bits left (integer instructions and one
// conversion); hi + lo within 2^-46 |x|.
__device__ __forceinline__ void split_float(double x, float &hi, float &lo) {
  hi = trunc_float(x);
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  const float unit = e > 948u && e < 1151u ? __uint_as_float((e - 948u) << 23) : 0.0f;   // 2^(exponent - 52)
  lo = copysignf((float)((unsigned)__double2loint(x) & 0x1fffffffu) * unit, hi);
}

// A ray in a frame: the point as two floats, the direction truncated.
struct PickRay {
  float ph[3], pl[3], v[3];
};

__device__ __forceinline__ PickRay pick_ray(const V3 &p, const V3 &v) {
  PickRay r;
  split_float(p.x, r.ph[0], r.pl[0]);
  split_float(p.y, r.ph[1], r.pl[1]);
  split_float(p.z, r.ph[2], r.pl[2]);
  r.v[0] = trunc_float(v.x);
  r.v[1] = trunc_float(v.y);
  r.v[2] = trunc_float(v.z);
  return r;
}

// DistanceToOut of the volume whose frame the ray is given in.  The point is within u of its coordinates, the sizes
// within u / 2.
__device__ __forceinline__ Pick pick_leaf(const DPick32 &D, const PickRay &r, float band) {
  const int kind = D.kind_flags & 3;
  const float ext = kind == kOrb ? D.q[0] : D.q[0] + D.q[1] + D.q[2];
  const float ep = 2.0f * kU * (fabsf(r.ph[0]) + fabsf(r.ph[1]) + fabsf(r.ph[2]) + ext) + 1e-30f;
  return pick_solid<false>(kind, D.q, D.kind_flags >> 2, r.ph[0], r.ph[1], r.ph[2], r.v[0], r.v[1], r.v[2], ep, band);
}

// Point and direction in daughter D's frame, from its mother's.  The difference of the two-float point and translation
// is within u of its value (rounding of the high parts' difference, and of the sum with the low parts'), plus 2^-45 of
// the coordinates; the rotation adds 2u (|dx| + |dy|).  Returns the bound ep of a coordinate's error, the sizes' u / 2
// included: below 6u (|dx| + |dy| + |dz| + sizes).
__device__ __forceinline__ float pick_to_daughter(const DPick32 &D, const PickRay &r, float *x, float *v) {
  const float dx = (r.ph[0] - D.th[0]) + (r.pl[0] - D.tl[0]), dy = (r.ph[1] - D.th[1]) + (r.pl[1] - D.tl[1]);
  x[2] = (r.ph[2] - D.th[2]) + (r.pl[2] - D.tl[2]);
  v[2] = r.v[2];
  const int flags = D.kind_flags >> 2;
  if (flags & kPlacedAligned) {
    x[0] = dx;
    x[1] = dy;
    v[0] = r.v[0];
    v[1] = r.v[1];
  } else {
    x[0] = D.c * dx + D.s * dy;
    x[1] = D.c * dy - D.s * dx;
    v[0] = D.c * r.v[0] + D.s * r.v[1];
    v[1] = D.c * r.v[1] - D.s * r.v[0];
  }
  const float ext = (D.kind_flags & 3) == kOrb ? D.q[0] : D.q[0] + D.q[1] + D.q[2];
  const float far = fabsf(r.ph[0]) + fabsf(r.ph[1]) + fabsf(r.ph[2]) + fabsf(D.th[0]) + fabsf(D.th[1]) + fabsf(D.th[2]);
  return 6.0f * kU * (fabsf(dx) + fabsf(dy) + fabsf(x[2]) + ext) + 3e-14f * far + 1e-30f;
}

// Position of the point against the solid: 1 inside and -1 outside by more than the band, 0 undecided (cones: always).  Each
// distance is within 4 ep of the exact one: the coordinates' errors (up to sqrt 3 ep), the sizes', the radius's roundings.
__device__ __forceinline__ int classify_point(int kind, const float *q, int flags, float x, float y, float z, float ep,
                                              float band) {
  float d;
  if (kind == kBox) {
    d = fminf(q[0] - fabsf(x), fminf(q[1] - fabsf(y), q[2] - fabsf(z)));
  } else if (kind == kOrb) {
    d = q[0] - sqrt_approx(x * x + y * y + z * z);
  } else if (kind == kTube) {
    const float r = sqrt_approx(x * x + y * y);
    d = fminf(q[2] - fabsf(z), q[1] - r);
    if (flags & kHasRmin) d = fminf(d, r - q[0]);
    if (flags & kSeg) {
      const float ds = q[3] * y - q[4] * x, de = q[6] * x - q[5] * y;
      d = fminf(d, (flags & kWide) ? fmaxf(ds, de) : fminf(ds, de));
    }
  } else {
    return 0;
  }
  const float m = 4.0f * ep + band;
  return d > m ? 1 : (d < -m ? -1 : 0);
}

// The same for daughter D of the volume whose frame the point is given in.
__device__ __forceinline__ int classify_daughter(const DPick32 &D, const PickRay &r, float band) {
  float x[3], v[3];
  const float ep = pick_to_daughter(D, r, x, v);
  return classify_point(D.kind_flags & 3, D.q, D.kind_flags >> 2, x[0], x[1], x[2], ep, band);
}
// Is the ray, from inside box D or from where it leaves it, certainly leaving: does some axis's coordinate lie in or beyond
// the band of the face that the ray moves to?  Then DistanceToIn is none, else zero.  A track that has just left the
// box stands 1e-13 from that face, where hull_slab's bounds (7e-7 of the sizes) see no difference to a point inside; the
// distance from the face as a sum of floats does (the sizes' low parts are q[3 .. 5]): an FP64 test there instead cost the
// stack of plates 4 %.
__device__ __forceinline__ bool box_left(const DPick32 &D, const PickRay &r, float band) {
  bool left = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // x = p - t as two floats: the difference of the high parts with its rounding, and the low parts' (within 2^-45 of the coordinates)
    const float h = r.ph[a] - D.th[a], bb = h - r.ph[a];
    const float l = ((r.ph[a] - (h - bb)) - (D.th[a] + bb)) + (r.pl[a] - D.tl[a]);
    const bool neg = h < 0.0f;
    const float gap = (D.q[a] - fabsf(h)) + (D.q[3 + a] - (neg ? -l : l));   // to the face on the point's side
    const float err = 1e-13f * (fabsf(r.ph[a]) + fabsf(D.th[a]) + D.q[a]) + 4.0f * kU * fabsf(gap);
    left = left || (gap + err < 0.5f * band * (1.0f - 2.0f * kU) && (neg ? r.v[a] < 0.0f : r.v[a] > 0.0f));
  }
  return left;
}

// DistanceToIn of daughter D of the volume whose frame the ray is given in.
__device__ __forceinline__ Pick pick_daughter(const DPick32 &D, const PickRay &r, float band) {
  float x[3], v[3];
  const float ep = pick_to_daughter(D, r, x, v);
  Pick k = pick_solid<true>(D.kind_flags & 3, D.q, D.kind_flags >> 2, x[0], x[1], x[2], v[0], v[1], v[2], ep, band);
  if (k.surf == kPickLeaving) k.surf = (D.kind_flags >> 2 & kPlacedAligned) && box_left(D, r, band) ? kPickMiss : kPickUnsure;
  return k;
}

}  // namespace dev
}  // namespace g4n
