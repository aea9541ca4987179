// nav_device.cuh -- device-side navigation (sm_103a): solids, locate, the voxel
// walk of compute_step, relocation, attenuation tables, Philox and the step hash.
//
// Navigation problems (Sec. 3.2): (1) which volumes contain a point; (2) the
// distance to the next boundary along a direction.  Conventions shared with the
// host side of the library:
//  * tolerance band +-half around every surface (half = 0.5e-9 mm x scale);
//  * Inside is direction aware: a point in the band of a surface belongs to the
//    solid iff the direction points strictly inward through every surface
//    whose band holds the point;
//  * DistanceToIn from a point that is not inside only reports crossings
//    beyond the band; ties in compute_step go to the daughter over the mother
//    and to the lower daughter id.
//
// Precision modes.  kFP64: every distance in FP64.  kFP32: rigorous FP32
// interval bounds (directed rounding) on the padded bounding boxes decide which
// candidates can still matter and whether the physics step wins; only those
// candidates and the winning surface are evaluated in FP64, so every result is
// the FP64 one.  GB300's FP64 rate is ~1/72 of its FP32 rate, which is why the
// bounds are worth their extra FP32 work.
#pragma once

#include <cstdint>

#include "g4n_internal.h"
#include "mlp_device.cuh"
#include "nav_pick32.cuh"
#include "nav_solids.cuh"

namespace g4n {
namespace dev {

constexpr float kInfF = __builtin_huge_valf();
enum Mode : int { kFP64 = 0, kFP32 = 1, kLearned = 2 };  // kLearned: FP32 bounds + proposal first

// Per-thread event counters (registers; constant indices only), flushed once per warp.
struct Counters {
  uint32_t c[G4N_N_COUNTERS];
};

template <bool COUNT>
__device__ __forceinline__ void diag(Counters &c, int k) {
  if (COUNT) c.c[k]++;
}

template <bool COUNT>
__device__ __forceinline__ void diag_kind(Counters &c, int kind) {
  if (COUNT) {
    if (kind == kBox) c.c[G4N_C_CAND_BOX]++;
    else if (kind == kTube) c.c[G4N_C_CAND_TUBE]++;
    else if (kind == kCone) c.c[G4N_C_CAND_CONE]++;
    else c.c[G4N_C_CAND_ORB]++;
  }
}

// An FP64 DistanceToOut or Inside test of solid `kind`: tubes and cones are also counted apart (their
// formulas have several times the box's arithmetic).
template <bool COUNT>
__device__ __forceinline__ void diag_test(Counters &c, int which, int curved_which, int kind) {
  if (COUNT) {
    c.c[which]++;
    if (kind == kTube || kind == kCone) c.c[curved_which]++;
  }
}

// ---------------------------------------------------------------- dispatch on the solid kind

__device__ __forceinline__ bool vol_inside(const DVol &d, const V3 &p, const V3 &v, double half) {
  if (d.kind == kBox) return box_inside(d.p, p, v, half);
  if (d.kind == kOrb) return orb_inside(d.p[0], p, v, half);
  if (d.kind == kCone) return cone_inside(d.p, d.flags, p, v, half);
  return tube_inside(d.p, d.flags, p, v, half);
}

// The full FP64 formulas (every surface), for cones and where the FP32 bounds of pick_solid do not decide.
__device__ __noinline__ double vol_dist_in_full(const DVol &d, const V3 &p, const V3 &v, double half) {
  if (d.kind == kBox) return box_dist_in(d.p, p, v, half);
  if (d.kind == kOrb) return orb_dist_in(d.p[0], p, v, half);
  if (d.kind == kCone) return cone_cross(d.p, d.flags, p, v, half, true);
  return tube_cross(d.p, d.flags, p, v, half, true);
}

__device__ __noinline__ double vol_dist_out_full(const DVol &d, const V3 &p, const V3 &v, double half) {
  if (d.kind == kBox) {
    int face;
    return box_dist_out(d.p, p, v, inv_dir(v), &face);
  }
  if (d.kind == kOrb) return orb_dist_out(d.p[0], p, v);
  const double t = d.kind == kCone ? cone_cross(d.p, d.flags, p, v, half, false) : tube_cross(d.p, d.flags, p, v, half, false);
  return t == kInf ? 0.0 : fmax(t, 0.0);
}

// DistanceToIn, DistanceToOut: FP32 bounds choose the surface (or prove a miss), FP64 evaluates its crossing parameter.
// Out of line: one copy serves the kernel's call sites (inlined, the calorimeter batch and the persistent barrel were
// 1.4 and 2 % slower than with the full formulas out of line; so, level and 4 % faster).
// *surf: the surface where the bounds chose it, else -1.
__device__ __noinline__ double vol_dist_in(const DVol &d, const DPick32 &k32, const V3 &p, const V3 &v, double half,
                                           float band, int *surf) {
  const PickRay r = pick_ray(p, v);
  const int kind = d.kind;
  const float ext = kind == kOrb ? k32.q[0] : k32.q[0] + k32.q[1] + k32.q[2];
  const float ep = 2.0f * kU * (fabsf(r.ph[0]) + fabsf(r.ph[1]) + fabsf(r.ph[2]) + ext) + 1e-30f;
  const Pick k = pick_solid<true>(kind, k32.q, d.flags, r.ph[0], r.ph[1], r.ph[2], r.v[0], r.v[1], r.v[2], ep, band);
  *surf = k.surf;
  if (k.surf == kPickMiss) return kInf;
  if (k.surf >= 0) {
    double num, den;
    surf_ratio(kind, d.p, k.surf, true, p, v, num, den);
    const double t = num / den;
    if (t > half) return t;
  }
  *surf = -1;
  return vol_dist_in_full(d, p, v, half);
}

__device__ __noinline__ double vol_dist_out_curved(const DVol &d, const DPick32 &k32, const V3 &p, const V3 &v, double half,
                                                   float band, int *surf) {
  const Pick k = pick_leaf(k32, pick_ray(p, v), band);
  if (k.surf >= 0) {
    double num, den;
    surf_ratio(d.kind, d.p, k.surf, false, p, v, num, den);
    const double t = num / den;
    *surf = k.surf;
    if (t > -half) return fmax(t, 0.0);
  }
  *surf = -1;
  return vol_dist_out_full(d, p, v, half);
}

__device__ __forceinline__ double vol_dist_out(const DVol &d, const DPick32 &k32, const V3 &p, const V3 &v, const Inv3 &iv,
                                               double half, float band, int *face) {
  *face = -1;
  if (d.kind == kBox) return box_dist_out(d.p, p, v, iv, face);
  return vol_dist_out_curved(d, k32, p, v, half, band, face);
}

__device__ __forceinline__ double vol_safety_in(const DVol &d, const V3 &p) {
  if (d.kind == kBox) return box_safety_in(d.p, p);
  if (d.kind == kOrb) return orb_safety_in(d.p[0], p);
  if (d.kind == kCone) return cone_safety_in(d.p, d.flags, p);
  return tube_safety_in(d.p, d.flags, p);
}

__device__ __forceinline__ double vol_safety_out(const DVol &d, const V3 &p) {
  if (d.kind == kBox) return box_safety_out(d.p, p);
  if (d.kind == kOrb) return orb_safety_out(d.p[0], p);
  if (d.kind == kCone) return cone_safety_out(d.p, d.flags, p);
  return tube_safety_out(d.p, d.flags, p);
}

__device__ __forceinline__ float sel3(float a, float b, float c, int i) { return i == 0 ? a : (i == 1 ? b : c); }

// ---------------------------------------------------------------- FP32 interval bounds
// A point p (FP64) is enclosed by [lo, hi] = the float neighbours of (float)p; a
// direction component by its float neighbours, whose reciprocals, rounded
// outward, enclose 1/v.  All products and differences below are rounded in the
// direction that keeps each bound valid, so every lower bound is <= the exact
// FP64 quantity it bounds (and every upper bound >=).

struct Ray32 {
  float plo[3], phi[3];
  float ilo[3], ihi[3];  // enclosure of 1/|v_a|
  int sgn[3];            // sign of v_a (0 if |v_a| < 1e-30)
};

// The float neighbours of (float)x, below and above, by integer instructions (a conversion holds the FP64 pipe):
// truncation, rounding to nearest even, a step of one unit either way.  Doubles below 2^-126 take the conversion.
__device__ __forceinline__ void enclose(double x, float &lo, float &hi) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned t = (h & 0x7fffffffu) - 0x38000000u;
  if ((int)t < 0x00100000 || t >= 0x0fe00000u) {
    const float f = (float)x;
    lo = nextafterf(f, -kInfF);
    hi = nextafterf(f, kInfF);
    return;
  }
  unsigned m = (t << 3) | (l >> 29);
  const unsigned rest = l & 0x1fffffffu;
  m += (rest > 0x10000000u || (rest == 0x10000000u && (m & 1u))) ? 1u : 0u;
  const float in = __uint_as_float(m - 1u), out = __uint_as_float(m + 1u);
  const bool neg = (int)h < 0;
  lo = neg ? -out : in;
  hi = neg ? -in : out;
}

__device__ __forceinline__ Ray32 make_ray32(const V3 &p, const V3 &v) {
  Ray32 r;
  const double pp[3] = {p.x, p.y, p.z}, vv[3] = {v.x, v.y, v.z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    enclose(pp[a], r.plo[a], r.phi[a]);
    const long long wb = __double_as_longlong(vv[a]) & 0x7FFFFFFFFFFFFFFFll;
    if (wb < 0x39B4484BFEEBC2A0ll) {  // |v_a| < 1e-30
      r.sgn[a] = 0;
      r.ilo[a] = r.ihi[a] = 0.f;
      continue;
    }
    r.sgn[a] = __double_as_longlong(vv[a]) > 0 ? 1 : -1;
    float wlo, whi;
    enclose(__longlong_as_double(wb), wlo, whi);
    // the approximate reciprocal is within u of the reciprocal
    r.ilo[a] = __fmul_rd(rcp_approx(whi), 1.0f - 2.0f * kU);
    r.ihi[a] = __fmul_ru(rcp_approx(wlo), 1.0f + 2.0f * kU);
  }
  return r;
}

// Lower/upper bound of num / |v_a| given num in [nlo, nhi] (scalar num bounds).
__device__ __forceinline__ float div_lo(float n, const Ray32 &r, int a) {
  return n >= 0.f ? __fmul_rd(n, r.ilo[a]) : __fmul_rd(n, r.ihi[a]);
}
__device__ __forceinline__ float div_hi(float n, const Ray32 &r, int a) {
  return n >= 0.f ? __fmul_ru(n, r.ihi[a]) : __fmul_ru(n, r.ilo[a]);
}

// Rigorous lower bound of the parameter at which the ray enters box [lo, hi]
// (same frame), +inf when the ray certainly misses it.  Also the exit upper bound.
__device__ __forceinline__ float box_entry_lb(const float *lo, const float *hi, const Ray32 &r, float *exit_ub) {
  float tlo = 0.f, thi = kInfF;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (r.sgn[a] == 0) {
      if (r.phi[a] < lo[a] || r.plo[a] > hi[a]) return kInfF;
      continue;
    }
    float en, ex;
    if (r.sgn[a] > 0) {
      en = div_lo(__fsub_rd(lo[a], r.phi[a]), r, a);
      ex = div_hi(__fsub_ru(hi[a], r.plo[a]), r, a);
    } else {
      en = div_lo(__fsub_rd(r.plo[a], hi[a]), r, a);
      ex = div_hi(__fsub_ru(r.phi[a], lo[a]), r, a);
    }
    tlo = fmaxf(tlo, en);
    thi = fminf(thi, ex);
  }
  if (exit_ub) *exit_ub = thi;
  return tlo > thi ? kInfF : tlo;
}

// Lower bound of the Euclidean distance from the point to box [lo, hi].
__device__ __forceinline__ float box_gap_lb(const float *lo, const float *hi, const Ray32 &r) {
  float d = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) d = fmaxf(d, fmaxf(__fsub_rd(lo[a], r.phi[a]), __fsub_rd(r.plo[a], hi[a])));
  return d;
}

__device__ __forceinline__ float absmax(float lo, float hi) { return fmaxf(fabsf(lo), fabsf(hi)); }
__device__ __forceinline__ float absmin(float lo, float hi) { return (lo <= 0.f && hi >= 0.f) ? 0.f : fminf(fabsf(lo), fabsf(hi)); }

// __double2float_rd / _ru of a double that is not negative, by integer instructions where it is of normal float size.
__device__ __forceinline__ float float_rd(double x) {
  const unsigned t = (unsigned)__double2hiint(x) - 0x38000000u;
  if ((int)t < 0x00100000 || t >= 0x0fe00000u) return __double2float_rd(x);
  return __uint_as_float((t << 3) | ((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ float float_ru(double x) {
  const unsigned t = (unsigned)__double2hiint(x) - 0x38000000u, l = (unsigned)__double2loint(x);
  if ((int)t < 0x00100000 || t >= 0x0fe00000u) return __double2float_ru(x);
  return __uint_as_float(((t << 3) | (l >> 29)) + ((l & 0x1fffffffu) ? 1u : 0u));
}

// Lower bound of the isotropic safety of the leaf, point in its own frame (cones: 0).
__device__ __forceinline__ float leaf_safety32(const DVol &V, const Ray32 &r, const V3 &p) {
  float s;
  if (V.kind == kBox) {
    s = kInfF;
#pragma unroll
    for (int a = 0; a < 3; ++a) s = fminf(s, __fsub_rd(float_rd(V.p[a]), absmax(r.plo[a], r.phi[a])));
    return fmaxf(s, 0.f);
  }
  if (V.kind == kCone) return 0.f;
  const float ax = absmax(r.plo[0], r.phi[0]), ay = absmax(r.plo[1], r.phi[1]), az = absmax(r.plo[2], r.phi[2]);
  if (V.kind == kOrb) {
    const float rr = __fsqrt_ru(__fadd_ru(__fadd_ru(__fmul_ru(ax, ax), __fmul_ru(ay, ay)), __fmul_ru(az, az)));
    s = __fsub_rd(float_rd(V.p[0]), rr);
  } else {
    const float rup = __fsqrt_ru(__fadd_ru(__fmul_ru(ax, ax), __fmul_ru(ay, ay)));
    s = fminf(__fsub_rd(float_rd(V.p[1]), rup), __fsub_rd(float_rd(V.p[2]), az));
    if (V.flags & kHasRmin) {
      const float mx = absmin(r.plo[0], r.phi[0]), my = absmin(r.plo[1], r.phi[1]);
      const float rdn = __fsqrt_rd(__fadd_rd(__fmul_rd(mx, mx), __fmul_rd(my, my)));
      s = fminf(s, __fsub_rd(rdn, float_ru(V.p[0])));
    }
    if (V.flags & kSeg) {
      // phi planes: exact FP64 distances to the two lines, rounded down
      const double ds = fabs(V.p[3] * p.y - V.p[4] * p.x), de = fabs(V.p[6] * p.x - V.p[5] * p.y);
      s = fminf(s, fminf(float_rd(ds), float_rd(de)));
    }
  }
  return fmaxf(s, 0.f);
}

// Is the point inside the solid by more than the tolerance band whatever the direction?
// (conservative: false when undecided).
__device__ __forceinline__ bool certainly_inside32(const DVol &V, const Ray32 &r, float band) {
  if (V.kind == kBox) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (!(absmax(r.plo[a], r.phi[a]) < __fsub_rd(float_rd(V.p[a]), band))) return false;
    return true;
  }
  if (V.kind == kCone) return false;
  const float ax = absmax(r.plo[0], r.phi[0]), ay = absmax(r.plo[1], r.phi[1]), az = absmax(r.plo[2], r.phi[2]);
  if (V.kind == kOrb) {
    const float R = __fsub_rd(float_rd(V.p[0]), band);
    return R > 0.f && __fadd_ru(__fadd_ru(__fmul_ru(ax, ax), __fmul_ru(ay, ay)), __fmul_ru(az, az)) < __fmul_rd(R, R);
  }
  if (V.flags & kSeg) return false;
  const float rmax = __fsub_rd(float_rd(V.p[1]), band);
  if (!(az < __fsub_rd(float_rd(V.p[2]), band))) return false;
  if (!(__fadd_ru(__fmul_ru(ax, ax), __fmul_ru(ay, ay)) < __fmul_rd(rmax, rmax))) return false;
  if (V.flags & kHasRmin) {
    const float rmin = __fadd_ru(float_ru(V.p[0]), band);
    const float mx = absmin(r.plo[0], r.phi[0]), my = absmin(r.plo[1], r.phi[1]);
    if (!(__fadd_rd(__fmul_rd(mx, mx), __fmul_rd(my, my)) > __fmul_ru(rmin, rmin))) return false;
  }
  return true;
}

// Lower bound of the Euclidean distance from mother-frame point (x, y, z) to daughter D's
// solid, from FP32 copies of its placement and size: the FP32 local point is within
// `e` of the exact one (a generous allowance: 2^-20 of the magnitudes involved).
// Negative when the point may be inside.
__device__ __forceinline__ float iso_lb32(const DVol32 &D, float x, float y, float z) {
  const float dx = x - D.tx, dy = y - D.ty, lz = z - D.tz;
  float lx = dx, ly = dy;
  if (!(D.flags & kPlacedAligned)) {
    lx = D.c * dx + D.s * dy;
    ly = D.c * dy - D.s * dx;
  }
  const float e = 9.5367432e-7f * (fabsf(x) + fabsf(y) + fabsf(z) + D.scale) + 1e-30f;
  float d;
  if (D.kind == kBox) {
    d = fmaxf(fabsf(lx) - D.q0, fmaxf(fabsf(ly) - D.q1, fabsf(lz) - D.q2));
  } else if (D.kind == kOrb) {
    d = sqrtf(lx * lx + ly * ly + lz * lz) - D.q0;
  } else {
    const float r = sqrtf(lx * lx + ly * ly);
    d = fmaxf(r - D.q1, fabsf(lz) - D.q2);
    if (D.flags & kHasRmin) d = fmaxf(d, D.q0 - r);
  }
  return d - e;
}

// Conservative FP32 test: can the mother-frame point claim daughter box b?
__device__ __forceinline__ bool box32_contains(const DBox32 &b, float x, float y, float z) {
  return x >= b.lo[0] && x <= b.hi[0] && y >= b.lo[1] && y <= b.hi[1] && z >= b.lo[2] && z <= b.hi[2];
}

// ---------------------------------------------------------------- voxels

__device__ __forceinline__ int slice_of(const DVoxHdr &H, double coord) {
  double f = floor((coord - H.lo) * H.inv_width);
  f = fmin(fmax(f, 0.0), (double)(H.nslices - 1));
  return (int)f;
}

// ---------------------------------------------------------------- FP32 voxel walk
// The FP32 modes walk the voxel nodes with interval arithmetic on the headers' outward
// rounded FP32 copies (lo_dn/lo_up, w_dn/w_up, iw_dn/iw_up) and on the ray's enclosure
// (Ray32).  Every interval encloses the value the FP64 walk computes (each FP64 result
// is a double between two directed-rounded floats of the same operation), so a
// decision taken where the intervals do not overlap is the FP64 walk's decision; an
// overlapping case returns "undecided" and the FP64 code takes that node step.

__device__ __forceinline__ int sel3i(int a, int b, int c, int i) { return i == 0 ? a : (i == 1 ? b : c); }

// Slice index of every FP64 coordinate in [qlo, qhi] under slice_of, or -1 if they differ.
__device__ __forceinline__ int slice_of32(const DVoxHdr32 &H, float qlo, float qhi) {
  const float dlo = __fsub_rd(qlo, H.lo_up), dhi = __fsub_ru(qhi, H.lo_dn);
  const float slo = dlo >= 0.f ? __fmul_rd(dlo, H.iw_dn) : __fmul_rd(dlo, H.iw_up);
  const float shi = dhi >= 0.f ? __fmul_ru(dhi, H.iw_up) : __fmul_ru(dhi, H.iw_dn);
  const float top = (float)((H.n_axis >> 2) - 1);
  const float klo = fminf(fmaxf(floorf(slo), 0.f), top), khi = fminf(fmaxf(floorf(shi), 0.f), top);
  return klo == khi ? (int)klo : -1;
}

// Enclosure of the FP64 slab boundaries lo + k0 w and lo + (k1 + 1) w of a merged node.
__device__ __forceinline__ void slab32(const DVoxHdr32 &H, int k0, int k1, float &blo_dn, float &blo_up, float &bhi_dn,
                                       float &bhi_up) {
  const float a = (float)k0, b = (float)(k1 + 1);
  blo_dn = __fadd_rd(H.lo_dn, __fmul_rd(a, H.w_dn));
  blo_up = __fadd_ru(H.lo_up, __fmul_ru(a, H.w_up));
  bhi_dn = __fadd_rd(H.lo_dn, __fmul_rd(b, H.w_dn));
  bhi_up = __fadd_ru(H.lo_up, __fmul_ru(b, H.w_up));
}

// Enclosure [qlo, qhi] of the FP64 coordinate p_a + t v_a for t in [tl, th] (axis a of the ray).
// False when v_a is tiny but not zero (the FP32 enclosure does not hold it).
__device__ __forceinline__ bool advance32(const Ray32 &r, const V3 &v, int a, float tl, float th, float &qlo,
                                          float &qhi) {
  const float plo = sel3(r.plo[0], r.plo[1], r.plo[2], a), phi = sel3(r.phi[0], r.phi[1], r.phi[2], a);
  const int sg = sel3i(r.sgn[0], r.sgn[1], r.sgn[2], a);
  if (sg == 0) {
    qlo = plo;
    qhi = phi;
    return !nonzero_bits(comp(v, a));
  }
  // |v_a| lies in [1 / ihi, 1 / ilo]
  const float ilo = sel3(r.ilo[0], r.ilo[1], r.ilo[2], a), ihi = sel3(r.ihi[0], r.ihi[1], r.ihi[2], a);
  const float vlo = __fmul_rd(rcp_approx(ihi), 1.0f - 2.0f * kU), vhi = __fmul_ru(rcp_approx(ilo), 1.0f + 2.0f * kU);
  const float mlo = tl >= 0.f ? __fmul_rd(tl, vlo) : __fmul_rd(tl, vhi);
  const float mhi = th >= 0.f ? __fmul_ru(th, vhi) : __fmul_ru(th, vlo);
  if (sg > 0) {
    qlo = __fadd_rd(plo, mlo);
    qhi = __fadd_ru(phi, mhi);
  } else {
    qlo = __fsub_rd(plo, mhi);
    qhi = __fsub_ru(phi, mlo);
  }
  return true;
}

// Candidate list of the voxel node holding p (mother frame).
__device__ __forceinline__ int vox_lookup(const DGeom &G, int h, const V3 &p) {
#pragma unroll 1
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    const DVoxHdr H = G.hdr[h];
    const DVoxSlice S = G.slice[H.slice_base + slice_of(H, comp(p, H.axis))];
    if (S.child >= 0) return S.child;
    h = -S.child - 1;
  }
  return 0;
}

// The same decided in FP32 on the point's enclosure (slice_of32), FP64 where a slice boundary lies within it.
__device__ __forceinline__ int vox_lookup32(const DGeom &G, int h, const V3 &p) {
  const int root = h;
  float lo[3], hi[3];
  enclose(p.x, lo[0], hi[0]);
  enclose(p.y, lo[1], hi[1]);
  enclose(p.z, lo[2], hi[2]);
#pragma unroll 1
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    const DVoxHdr32 H = G.hdr32[h];
    const int a = H.n_axis & 3;
    const int k = slice_of32(H, sel3(lo[0], lo[1], lo[2], a), sel3(hi[0], hi[1], hi[2], a));
    if (k < 0) return vox_lookup(G, root, p);
    const DVoxSlice S = G.slice[H.slice_base + k];
    if (S.child >= 0) return S.child;
    h = -S.child - 1;
  }
  return 0;
}

// ---------------------------------------------------------------- exact coordinate keys
// key(x): a double's bits as a signed integer with the negative half reflected,
// so that x < y <=> key(x) < key(y).  The geometry carries, for world-aligned
// boxes and for the voxel slices of world-aligned mothers, the keys at which the
// FP64 predicates (Inside bands, slice index) change value; comparing keys then
// gives the FP64 answer with integer instructions only.


// A float near x built from the high word of its bits (truncated; no FP64 instruction).
__device__ __forceinline__ float approx_float(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned sg = hi & 0x80000000u;
  if (e < 897) return __uint_as_float(sg);
  if (e > 1150) return __uint_as_float(sg | 0x7f7fffffu);
  return __uint_as_float(sg | ((unsigned)(e - 896) << 23) | ((hi & 0xfffffu) << 3));
}

// A world point and direction with the keys of the point and a float guess of it.
struct WPos {
  V3 x, u;
  long long k[3];
  float f[3];
};

__device__ __forceinline__ WPos make_wpos(const V3 &x, const V3 &u) {
  WPos W;
  W.x = x;
  W.u = u;
  W.k[0] = dkey(x.x);
  W.k[1] = dkey(x.y);
  W.k[2] = dkey(x.z);
  W.f[0] = approx_float(x.x);
  W.f[1] = approx_float(x.y);
  W.f[2] = approx_float(x.z);
  return W;
}

__device__ __forceinline__ long long kcomp(const long long *k, int a) { return a == 0 ? k[0] : (a == 1 ? k[1] : k[2]); }
__device__ __forceinline__ float fcomp(const float *f, int a) { return a == 0 ? f[0] : (a == 1 ? f[1] : f[2]); }

// box_inside on p = x - t of a kKeyBox volume d (the same answer, by its keys).
// In the surface band of axis a the sign of p_a is known (the side of the band),
// so p_a v_a >= 0 reduces to a sign test; only a subnormal v_a needs the product.
__device__ __forceinline__ bool keybox_inside(const DGeom &G, int d, const WPos &W) {
  const DKeyBox &K = G.kbox[d];
  int near = 0;  // bit a: axis a in the band; bit a + 3: on its high side
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const long long k = W.k[a];
    if (k <= K.k[a][0] || k >= K.k[a][3]) return false;
    if (k <= K.k[a][1]) near |= 1 << a;
    else if (k >= K.k[a][2]) near |= 9 << a;
  }
  if (!near) return true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!(near & (1 << a))) continue;
    const double va = comp(W.u, a);
    const long long vb = __double_as_longlong(va);
    const long long mag = vb & 0x7FFFFFFFFFFFFFFFll;
    if (mag == 0) return false;                      // p_a v_a = 0
    if (mag < 0x0010000000000000ll) {                // subnormal v_a: the product decides
      const DWorld &w = G.wxf[d];
      const double pa = comp(W.x, a) - (a == 0 ? w.tx : (a == 1 ? w.ty : w.tz));
      if (pa * va >= 0.0) return false;
    } else if ((vb < 0) != ((near >> (a + 3)) & 1)) {
      return false;                                  // v_a points outward
    }
  }
  return true;
}

// vox_lookup for a keyed header tree (world-aligned mother), from the world point.
__device__ __forceinline__ int vox_lookup_keys(const DGeom &G, int h, const WPos &W) {
#pragma unroll 1
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    const DVoxHdr H = G.hdr[h];
    const int n = H.nslices;
    const long long kx = kcomp(W.k, H.axis);
    const long long *S = reinterpret_cast<const long long *>(G.skey) + H.slice_base;
    int k = __float2int_rd((fcomp(W.f, H.axis) - H.lo_wf) * H.inv_wf);
    k = max(0, min(k, n - 1));
#pragma unroll 1
    while (k > 0 && kx < __ldg(&S[k])) --k;
#pragma unroll 1
    while (k + 1 < n && kx >= __ldg(&S[k + 1])) ++k;
    const DVoxSlice Sl = G.slice[H.slice_base + k];
    if (Sl.child >= 0) return Sl.child;
    h = -Sl.child - 1;
  }
  return 0;
}

// Warp-collective navigation.  Every lane of the warp must call these functions
// together (they synchronise with __syncwarp / __any_sync over the full warp);
// lanes with `active` false only take part in the synchronisation.  The point is
// SIMT efficiency: each round every searching lane first scans its candidate list
// in cheap FP32/integer code to the next candidate that needs FP64 work, then the
// warp meets and all those lanes run the FP64 test together.
constexpr unsigned kFull = 0xffffffffu;

// Descend from volume m into the first daughter, in id order, that contains the
// point; repeat.  CLASSIFY: the daughters are first classified in FP32 (nav_pick32.cuh) and the voxel slices
// looked up in FP32, so that only a point within the FP32 errors of a daughter's surface takes an FP64 test.  10^7
// barrel queries of k_locate: 3.52 -> 2.20 ms (each candidate that passed its box in FP64 kept the FP64 pipe 78 %
// busy); where the tracks of a nested barrel start, a batch of 10^6 17.9 -> 17.2 ms.  Relocations go without: with the
// portals they are few, and the added code cost the barrel and the batched worlds 1 %, the default barrel 4 %.
// (p, v) is the point in m's frame when have_p is set; otherwise it
// is derived from the world point when an FP64 test needs it.  kKeyBox daughters
// and keyed voxel trees are answered from the world point's keys.  `blocked` is a
// daughter of m already known not to contain the point (the volume just left).
// Returns the deepest volume.
// KEYED: every volume is a kKeyBox; nothing but keys.
template <bool COUNT, bool CLASSIFY, bool KEYED = false>
__device__ __forceinline__ int descend_body(const DGeom &G, bool active, int m, V3 p, V3 v, bool have_p,
                                            const WPos &W, int blocked, Counters &cnt) {
#pragma unroll 1
  for (int lev = 0; lev < kDMax; ++lev) {
    const bool want = active && G.vol[m].vox >= 0;
    if (!__any_sync(kFull, want)) break;
    DCandList L{0, 0};
    if (want) {
      const int h = G.vol[m].vox;
      if (KEYED || G.hdr[h].keyed) {
        L = G.clist[vox_lookup_keys(G, h, W)];
      } else {
        if (!have_p) {
          if (CLASSIFY) p = world_to_local_point(G.wxf[m], G.vol[m].flags & kWorldAligned, W.x);
          else world_to_local(G.wxf[m], G.vol[m].flags & kWorldAligned, W.x, W.u, p, v);
          have_p = true;
        }
        L = G.clist[CLASSIFY ? vox_lookup32(G, h, p) : vox_lookup(G, h, p)];
      }
    }
    PickRay q;
    bool have_q = false;
    int i = 0, found = -1;
    bool searching = want, via_fp64 = false;
    V3 fp = p, fv = v;
#pragma unroll 1
    while (__any_sync(kFull, searching)) {
      int d = -1;
      if (searching) {
#pragma unroll 1
        while (i < L.count) {
          const int c = __ldg(&G.cand[L.offset + i]);
          ++i;
          if (c == blocked) continue;
          const DBox32 &B = G.box[c];
          if (KEYED || B.keyed) {
            diag<COUNT>(cnt, G4N_C_KEY_INSIDE);
            if (keybox_inside(G, c, W)) {
              found = c;
              searching = false;
              break;
            }
            continue;
          }
          if (!have_p) {
            if (CLASSIFY) p = world_to_local_point(G.wxf[m], G.vol[m].flags & kWorldAligned, W.x);
            else world_to_local(G.wxf[m], G.vol[m].flags & kWorldAligned, W.x, W.u, p, v);
            have_p = true;
          }
          if (!have_q) {
            if (CLASSIFY) {
              q = pick_ray(p, V3{0.0, 0.0, 0.0});
            } else {
              q.ph[0] = (float)p.x;
              q.ph[1] = (float)p.y;
              q.ph[2] = (float)p.z;
            }
            have_q = true;
          }
          if (!box32_contains(B, q.ph[0], q.ph[1], q.ph[2])) continue;
          const int in = CLASSIFY ? classify_daughter(G.pick[c], q, G.band32)
                                  : iso_lb32(G.v32[c], q.ph[0], q.ph[1], q.ph[2]) > G.band32 ? -1 : 0;
          if (in < 0) continue;
          if (in > 0) {
            found = c;
            searching = false;
          } else {
            d = c;
          }
          break;
        }
        if (d < 0) searching = false;
      }
      __syncwarp();
      if (!KEYED && d >= 0) {
        const DVol &D = G.vol[d];
        V3 dp, dv;
        if (CLASSIFY) world_to_local(G.wxf[m], G.vol[m].flags & kWorldAligned, W.x, W.u, p, v);
        to_local(D, p, v, dp, dv);
        diag_test<COUNT>(cnt, G4N_C_INSIDE, G4N_C_INSIDE_CURVED, D.kind);
        if (vol_inside(D, dp, dv, G.half)) {
          found = d;
          fp = dp;
          fv = dv;
          via_fp64 = true;
          searching = false;
        }
      }
    }
    if (want && found >= 0) {
      m = found;
      have_p = via_fp64;
      p = fp;
      v = fv;
      blocked = -1;
    } else {
      active = false;
    }
  }
  return m;
}

// The descent out of line: one copy of its code serves every call site of a kernel.  The
// FP32 modes use it (their kernels are larger and stall on instruction fetch, which the
// shared copy relieves: measured 8 % on the barrel scene); the FP64 navigator inlines it
// (measured 2 % faster on the calorimeter, whose relocations are mostly face records).
// Counters are passed by pointer (null without diagnostics) so that they stay in registers.
template <bool COUNT, bool CLASSIFY>
__device__ __noinline__ int descend_ool(const DGeom &G, bool active, int m, V3 p, V3 v, bool have_p, const WPos &W,
                                        int blocked, Counters *cntp) {
  Counters none;
  return descend_body<COUNT, CLASSIFY>(G, active, m, p, v, have_p, W, blocked, COUNT ? *cntp : none);
}

template <bool COUNT, bool OOL, bool CLASSIFY>
__device__ __forceinline__ int descend_warp(const DGeom &G, bool active, int m, V3 p, V3 v, bool have_p,
                                            const WPos &W, int blocked, Counters &cnt) {
  if (OOL) return descend_ool<COUNT, CLASSIFY>(G, active, m, p, v, have_p, W, blocked, COUNT ? &cnt : nullptr);
  return descend_body<COUNT, CLASSIFY>(G, active, m, p, v, have_p, W, blocked, cnt);
}

// Locate from the world (warp-collective): the leaf, or -1 outside the world.
template <bool COUNT, bool OOL, bool CLASSIFY, bool KEYED = false>
__device__ __forceinline__ int locate_world_warp(const DGeom &G, bool active, const V3 &x, const V3 &u, Counters &cnt) {
  V3 p{0, 0, 0}, v{0, 0, 1};
  bool in = false, have_p = false;
  const WPos W = make_wpos(x, u);
  if (active) {
    if (KEYED || (G.vol[0].flags & kKeyBox)) {
      diag<COUNT>(cnt, G4N_C_KEY_INSIDE);
      in = keybox_inside(G, 0, W);
    } else {
      world_to_local(G.wxf[0], G.vol[0].flags & kWorldAligned, x, u, p, v);
      have_p = true;
      diag_test<COUNT>(cnt, G4N_C_INSIDE, G4N_C_INSIDE_CURVED, G.vol[0].kind);
      in = vol_inside(G.vol[0], p, v, G.half);
    }
  }
  const int leaf = KEYED ? descend_body<COUNT, false, true>(G, in, 0, p, v, have_p, W, -1, cnt)
                         : descend_warp<COUNT, OOL, CLASSIFY>(G, in, 0, p, v, have_p, W, -1, cnt);
  return in ? leaf : -1;
}

// After a move (warp-collective): leave every volume that no longer contains the
// point, then descend.  A step that ended on the leaf's own exit surface (limiter
// mother, positive length) leaves the leaf for certain: the point is on that
// surface moving outward, so the leaf's Inside test is false and is skipped.  A
// volume left on the way up is blocked in the descent below its mother (its
// Inside is already known to be false).  Returns the new leaf or -1 (left the world).
template <int MODE, bool COUNT>
__device__ __forceinline__ int relocate_warp(const DGeom &G, bool active, int leaf, const V3 &x, const V3 &u,
                                             bool left_leaf, Counters &cnt) {
  if (!__any_sync(kFull, active)) return -1;  // no lane relocates: skip the warp's whole search
  int blocked = -1;
  if (active && left_leaf) {
    blocked = leaf;
    leaf = G.vol[leaf].mother;
  }
  bool up = active && leaf >= 0;
  bool in = false, have_p = false;
  V3 p{0, 0, 0}, v{0, 0, 1};
  const WPos W = make_wpos(x, u);
#pragma unroll 1
  while (__any_sync(kFull, up)) {
    if (up) {
      const DVol &L = G.vol[leaf];
      bool ok = false;
      if (L.flags & kKeyBox) {
        diag<COUNT>(cnt, G4N_C_KEY_INSIDE);
        ok = keybox_inside(G, leaf, W);
        have_p = false;
      } else {
        world_to_local(G.wxf[leaf], L.flags & kWorldAligned, x, u, p, v);
        have_p = true;
        if (MODE != kFP64) ok = certainly_inside32(L, make_ray32(p, v), 2.0f * G.band32 + 1e-30f);
        if (!ok) {
          diag_test<COUNT>(cnt, G4N_C_INSIDE, G4N_C_INSIDE_CURVED, L.kind);
          ok = vol_inside(L, p, v, G.half);
        }
      }
      if (ok) {
        in = true;
        up = false;
      } else {
        blocked = leaf;
        leaf = L.mother;
        if (leaf < 0) up = false;
      }
    }
  }
  const int out = descend_warp<COUNT, MODE != kFP64, false>(G, in, in ? leaf : 0, p, v, have_p, W, blocked, cnt);
  return in ? out : -1;
}

// Relocation after a step that left kKeyBox volume `leaf` through `face` (limiter mother,
// positive length), from the volume's precomputed face record: true, and the new leaf
// (-1: left the world) in *out, when x lies in the record's region and the direction's
// normal component is not subnormal; the answer is then the one relocate_warp gives.
__device__ __forceinline__ bool face_relocate(const DGeom &G, int leaf, int face, const V3 &x, const V3 &u, int *out) {
  const int base = G.vol[leaf].face;
  if (base < 0 || face < 0) return false;
  const DFace &F = G.face[base + face];
  if (!F.ok) return false;
  if ((__double_as_longlong(comp(u, face >> 1)) & 0x7FF0000000000000ll) == 0) return false;
  const long long kx = dkey(x.x), ky = dkey(x.y), kz = dkey(x.z);
  if (kx < F.k[0][0] || kx > F.k[0][1] || ky < F.k[1][0] || ky > F.k[1][1] || kz < F.k[2][0] || kz > F.k[2][1])
    return false;
  *out = F.leaf;
  return true;
}

// Relocation after a step of length t > 0 (p + t v the crossing point, in the frame of `leaf`) that left `leaf` (lim
// mother) or entered its daughter lim, through surface surf, from the portal of the crossed face: true, and the new leaf
// (-1: left the world) in *out, when the face has a portal, the crossing point is away from the solid's other faces and the
// direction is not along the face; the answer is then the one relocate_warp gives.  FP32 throughout: what has to be proved
// is a distance of more than the band (1e-9 mm) and a clear sign, and a margin above the FP32 errors proves it.
// Identical histories; barrel batch of 10^7 tracks 101.3 -> 82.5 ms, default barrel of 3 10^5 17.8 -> 14.6 ms, nested
// barrel of 10^6 23.0 -> 20.2 ms, 48 batched worlds 28.1 -> 25.6 ms, stack of plates 24.2 -> 19.9 ms.
__device__ __forceinline__ bool portal_relocate(const DGeom &G, int leaf, int lim, int surf, const V3 &p, const V3 &v,
                                                double t, int *out) {
  const bool enter = lim >= 0;
  const int vol = enter ? lim : leaf;
  const DPick32 &D = G.pick[vol];
  const int kind = D.kind_flags & 3, flags = D.kind_flags >> 2;
  const PickRay r = pick_ray(p, v);
  float x[3] = {r.ph[0], r.ph[1], r.ph[2]}, w[3] = {r.v[0], r.v[1], r.v[2]};
  const float ext = kind == kOrb ? D.q[0] : D.q[0] + D.q[1] + D.q[2];
  float ep = 2.0f * kU * (fabsf(x[0]) + fabsf(x[1]) + fabsf(x[2]) + ext);
  if (enter) ep = pick_to_daughter(D, r, x, w);
  int face = surf;
  if (kind == kBox) {
    if (enter) face ^= 1;
  } else if (kind == kTube && surf == kPickZ) {
    face = (w[2] > 0.f) != enter ? 1 : 0;
  } else if (kind == kTube) {
    face = surf + 1;
  }
  const int to = __ldg(&G.portal[12 * vol + (enter ? 6 : 0) + face]);
  if (to == kPortalNone) return false;
  const float s = trunc_float(t);
  const float del = 2.0f * (ep + 12.0f * kU * (s + fabsf(x[0]) + fabsf(x[1]) + fabsf(x[2]) + ext)) + 1e-6f + 2.0f * G.band32;
#pragma unroll
  for (int a = 0; a < 3; ++a) x[a] += s * w[a];
  constexpr float kSlope = 1e-3f;   // least |v . n|
  bool ok;
  if (kind == kBox) {
    const int a = face >> 1;
    ok = (a == 0 || D.q[0] - fabsf(x[0]) > del) && (a == 1 || D.q[1] - fabsf(x[1]) > del) &&
         (a == 2 || D.q[2] - fabsf(x[2]) > del) && fabsf(sel3(w[0], w[1], w[2], a)) > kSlope;
  } else if (kind == kOrb) {
    ok = fabsf(x[0] * w[0] + x[1] * w[1] + x[2] * w[2]) > kSlope * D.q[0];
  } else {
    const float rr = sqrt_approx(x[0] * x[0] + x[1] * x[1]);
    ok = (face < 2 || D.q[2] - fabsf(x[2]) > del) && (face == 2 || D.q[1] - rr > del) &&
         (face == 3 || !(flags & kHasRmin) || rr - D.q[0] > del);
    float slope = fabsf(w[2]);
    if (face == 2 || face == 3) slope = fabsf(x[0] * w[0] + x[1] * w[1]) * rcp_approx(rr);
    if (flags & kSeg) {
      const float ds = D.q[3] * x[1] - D.q[4] * x[0], de = D.q[6] * x[0] - D.q[5] * x[1];
      if (face < 4) {
        ok = ok && ((flags & kWide) ? fmaxf(ds, de) : fminf(ds, de)) > del;
      } else {
        const float c = face == 4 ? D.q[3] : D.q[5], sn = face == 4 ? D.q[4] : D.q[6];
        ok = ok && c * x[0] + sn * x[1] > del && ((flags & kWide) || (face == 4 ? de : ds) > del);
        slope = fabsf(c * w[1] - sn * w[0]);
      }
    }
    ok = ok && slope > kSlope;
  }
  *out = to;
  return ok;
}

// Voxel walk state: per level the header, the merged node's slice range.
struct Chain {
  int h[kMaxLevels];
  int k0[kMaxLevels], k1[kMaxLevels];
  int nlev;
  int list;
};

__device__ __forceinline__ void chain_fill(const DGeom &G, Chain &ch, int lev, int h, const V3 &p) {
#pragma unroll 1
  for (; lev < kMaxLevels; ++lev) {
    const DVoxHdr H = G.hdr[h];
    const DVoxSlice S = G.slice[H.slice_base + slice_of(H, comp(p, H.axis))];
    ch.h[lev] = h;
    ch.k0[lev] = S.k0;
    ch.k1[lev] = S.k1;
    if (S.child >= 0) {
      ch.nlev = lev + 1;
      ch.list = S.child;
      return;
    }
    h = -S.child - 1;
  }
  ch.nlev = kMaxLevels;
  ch.list = 0;
}

// One node step of the plain FP64 voxel walk: the exit texit of the current node along the
// ray (the first level whose slab the ray leaves), the end test texit >= bound, the
// neighbouring node across that face and the lookup of its deeper levels at p + texit v.
// Returns 0: the walk ends; 1: ch holds the next node.  With `saf` the distances from the
// point to the node's slab faces lower *saf.
__device__ __forceinline__ int walk_step64(const DGeom &G, Chain &ch, const V3 &p, const V3 &v, const Inv3 &iv,
                                           double bound, bool saf, double *saf64, int *it, int cap, bool *timeout) {
  double texit = kInf;
  int lstar = -1;
#pragma unroll 1
  for (int l = 0; l < ch.nlev; ++l) {
    const DVoxHdr H = G.hdr[ch.h[l]];
    const double pa = comp(p, H.axis), va = comp(v, H.axis);
    const double blo = H.lo + ch.k0[l] * H.width, bhi = H.lo + (ch.k1[l] + 1) * H.width;
    if (saf) *saf64 = fmin(*saf64, fmax(fmin(pa - blo, bhi - pa), 0.0));
    double t = kInf;
    if (va > 0.0) t = (bhi - pa) * icomp(iv, H.axis);
    else if (va < 0.0) t = (blo - pa) * icomp(iv, H.axis);
    if (t < texit) {
      texit = t;
      lstar = l;
    }
  }
  if (!(texit < bound)) return 0;
  const DVoxHdr H = G.hdr[ch.h[lstar]];
  const int nk = comp(v, H.axis) > 0.0 ? ch.k1[lstar] + 1 : ch.k0[lstar] - 1;
  if (nk < 0 || nk >= H.nslices || ++*it >= cap) {
    if (*it >= cap) *timeout = true;
    return 0;
  }
  const DVoxSlice S = G.slice[H.slice_base + nk];
  ch.k0[lstar] = S.k0;
  ch.k1[lstar] = S.k1;
  if (S.child >= 0) {
    ch.nlev = lstar + 1;
    ch.list = S.child;
  } else {
    const V3 qpt{p.x + texit * v.x, p.y + texit * v.y, p.z + texit * v.z};
    chain_fill(G, ch, lstar + 1, -S.child - 1, qpt);
  }
  return 1;
}

// The same, out of line: the FP32 modes take it only when their intervals do not decide.
__device__ __noinline__ int walk_step64_ool(const DGeom &G, Chain &ch, const V3 &p, const V3 &v, const Inv3 &iv,
                                            double bound, bool saf, double *saf64, int *it, int cap, bool *timeout) {
  return walk_step64(G, ch, p, v, iv, bound, saf, saf64, it, cap, timeout);
}

// chain_fill from the root header h0 for every FP64 point in the ray's enclosure (FP32
// modes); false if a level's slice index is undecided (the caller then fills in FP64).
__device__ __forceinline__ bool chain_fill32(const DGeom &G, Chain &ch, int h, const Ray32 &r) {
#pragma unroll 1
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    const DVoxHdr32 H = G.hdr32[h];
    const int a = H.n_axis & 3;
    const int k = slice_of32(H, sel3(r.plo[0], r.plo[1], r.plo[2], a), sel3(r.phi[0], r.phi[1], r.phi[2], a));
    if (k < 0) return false;
    const DVoxSlice S = G.slice[H.slice_base + k];
    ch.h[lev] = h;
    ch.k0[lev] = S.k0;
    ch.k1[lev] = S.k1;
    if (S.child >= 0) {
      ch.nlev = lev + 1;
      ch.list = S.child;
      return true;
    }
    h = -S.child - 1;
  }
  ch.nlev = kMaxLevels;
  ch.list = 0;
  return true;
}

// Lower / upper bound of num / |v_a| for a runtime axis a.
__device__ __forceinline__ float div_lo_a(float n, const Ray32 &r, int a) {
  return n >= 0.f ? __fmul_rd(n, sel3(r.ilo[0], r.ilo[1], r.ilo[2], a)) : __fmul_rd(n, sel3(r.ihi[0], r.ihi[1], r.ihi[2], a));
}
__device__ __forceinline__ float div_hi_a(float n, const Ray32 &r, int a) {
  return n >= 0.f ? __fmul_ru(n, sel3(r.ihi[0], r.ihi[1], r.ihi[2], a)) : __fmul_ru(n, sel3(r.ilo[0], r.ilo[1], r.ilo[2], a));
}

// One node step of the voxel walk in FP32 interval arithmetic (FP32 modes): the exit of
// the current node along the ray (the level whose slab the ray leaves first), the end
// test against bound_f (an upper bound of the FP64 walk's bound min(best, stop)), the
// neighbouring node and the lookup of its deeper levels at the entry point.  Returns 0:
// the walk ends; 1: ch holds the next node; 2: undecided (ch unchanged), the FP64 code
// takes this node step.  With `saf` the distances from the point to the node's slab
// faces lower the isotropic safety *saf_f.
__device__ __forceinline__ int walk_step32(const DGeom &G, Chain &ch, const Ray32 &r, const V3 &v, float bound_f,
                                           bool saf, float *saf_f, int *it, int cap, bool *timeout) {
  float tl[kMaxLevels], th[kMaxLevels];
  const int nlev = ch.nlev;
  int lstar = -1;
  float ts_lo = kInfF, ts_hi = kInfF;
  bool tiny = false;
#pragma unroll
  for (int l = 0; l < kMaxLevels; ++l) {
    tl[l] = th[l] = kInfF;
    if (l < nlev) {
      const DVoxHdr32 H = G.hdr32[ch.h[l]];
      const int a = H.n_axis & 3;
      float blo_dn, blo_up, bhi_dn, bhi_up;
      slab32(H, ch.k0[l], ch.k1[l], blo_dn, blo_up, bhi_dn, bhi_up);
      const float plo = sel3(r.plo[0], r.plo[1], r.plo[2], a), phi = sel3(r.phi[0], r.phi[1], r.phi[2], a);
      if (saf) *saf_f = fminf(*saf_f, fmaxf(fminf(__fsub_rd(plo, blo_up), __fsub_rd(bhi_dn, phi)), 0.f));
      const int sg = sel3i(r.sgn[0], r.sgn[1], r.sgn[2], a);
      if (sg > 0) {
        tl[l] = div_lo_a(__fsub_rd(bhi_dn, phi), r, a);
        th[l] = div_hi_a(__fsub_ru(bhi_up, plo), r, a);
      } else if (sg < 0) {
        tl[l] = div_lo_a(__fsub_rd(plo, blo_up), r, a);
        th[l] = div_hi_a(__fsub_ru(phi, blo_dn), r, a);
      } else {
        tiny |= nonzero_bits(comp(v, a));  // a direction component too small for the enclosure
      }
      if (th[l] < ts_hi) {
        ts_hi = th[l];
        ts_lo = tl[l];
        lstar = l;
      }
    }
  }
  if (tiny) return 2;
  if (lstar < 0) return 0;  // the ray leaves no slab: the FP64 exit is +inf
  // the FP64 minimum is taken by lstar alone (the first level attaining it wins ties)
#pragma unroll
  for (int l = 0; l < kMaxLevels; ++l)
    if (l != lstar && !(tl[l] > ts_hi)) return 2;
  if (ts_lo >= bound_f) return 0;  // texit >= bound_f >= min(best, stop)
  const DVoxHdr32 H = G.hdr32[ch.h[lstar]];
  const int nk = sel3i(r.sgn[0], r.sgn[1], r.sgn[2], H.n_axis & 3) > 0 ? ch.k1[lstar] + 1 : ch.k0[lstar] - 1;
  if (nk < 0 || nk >= (H.n_axis >> 2) || ++*it >= cap) {
    if (*it >= cap) *timeout = true;
    return 0;
  }
  const DVoxSlice S = G.slice[H.slice_base + nk];
  int list = S.child;
  int dh[kMaxLevels - 1], dk0[kMaxLevels - 1], dk1[kMaxLevels - 1];
  int nd = 0;
  if (list < 0) {
    // deeper levels: slices of the entry point p + texit v, texit in [ts_lo, ts_hi]
    int hh = -S.child - 1;
#pragma unroll
    for (int j = 0; j < kMaxLevels - 1; ++j) {
      if (list < 0 && lstar + 1 + j < kMaxLevels) {
        const DVoxHdr32 D = G.hdr32[hh];
        float qlo, qhi;
        if (!advance32(r, v, D.n_axis & 3, ts_lo, ts_hi, qlo, qhi)) return 2;
        const int k = slice_of32(D, qlo, qhi);
        if (k < 0) return 2;
        const DVoxSlice Sd = G.slice[D.slice_base + k];
        dh[j] = hh;
        dk0[j] = Sd.k0;
        dk1[j] = Sd.k1;
        nd = j + 1;
        if (Sd.child >= 0) list = Sd.child;
        else hh = -Sd.child - 1;
      }
    }
  }
  ch.k0[lstar] = S.k0;
  ch.k1[lstar] = S.k1;
#pragma unroll
  for (int j = 0; j < kMaxLevels - 1; ++j) {
    if (j < nd) {
      ch.h[lstar + 1 + j] = dh[j];
      ch.k0[lstar + 1 + j] = dk0[j];
      ch.k1[lstar + 1 + j] = dk1[j];
    }
  }
  if (list >= 0) {
    ch.nlev = lstar + 1 + nd;
    ch.list = list;
  } else {
    ch.nlev = kMaxLevels;
    ch.list = 0;
  }
  return 1;
}

// Training-sample log written by the plain navigator (features, label = list slot of the
// daughter entered, candidate count); `count` may exceed `capacity` (extra samples dropped).
struct MlpLog {
  float *feat;
  int32_t *label;
  int32_t *ncand;
  unsigned long long *count;
  int64_t capacity;
};

// What geom_step needs for the proposal: the weights and this warp's scratch (learned
// mode), the sample log (plain mode, optional) and the track's log-energy feature.
struct MlpCtx {
  const mlp::SmemWeights *w;
  mlp::SmemWarp *scratch;
  const MlpLog *log;
  float loge;
};

// Proposal features of the node holding p (leaf frame): the point in the node's own
// coordinates (axes the node does not slice use the leaf's half extent), the direction,
// log E, n / 32 and 1.
__device__ __forceinline__ void node_features(const DGeom &G, const DVol &V, const Chain &ch, const V3 &p, const V3 &v,
                                              float loge, int n, float *f) {
  double c[3] = {0.0, 0.0, 0.0};
  double h[3];
  if (V.kind == kBox) {
    h[0] = V.p[0];
    h[1] = V.p[1];
    h[2] = V.p[2];
  } else if (V.kind == kOrb) {
    h[0] = h[1] = h[2] = V.p[0];
  } else if (V.kind == kCone) {
    h[0] = h[1] = fmax(V.p[3] - V.p[2] * V.p[4], V.p[3] + V.p[2] * V.p[4]);
    h[2] = V.p[4];
  } else {
    h[0] = h[1] = V.p[1];
    h[2] = V.p[2];
  }
  for (int l = 0; l < ch.nlev; ++l) {
    const DVoxHdr H = G.hdr[ch.h[l]];
    const double lo = H.lo + ch.k0[l] * H.width, hi = H.lo + (ch.k1[l] + 1) * H.width;
    c[H.axis] = 0.5 * (lo + hi);
    h[H.axis] = 0.5 * (hi - lo);
  }
  f[0] = fminf(fmaxf((float)((p.x - c[0]) / h[0]), -2.f), 2.f);
  f[1] = fminf(fmaxf((float)((p.y - c[1]) / h[1]), -2.f), 2.f);
  f[2] = fminf(fmaxf((float)((p.z - c[2]) / h[2]), -2.f), 2.f);
  f[3] = (float)v.x;
  f[4] = (float)v.y;
  f[5] = (float)v.z;
  f[6] = loge;
  f[7] = (float)n * (1.0f / 32.0f);
  f[8] = 1.0f;
}

// A boundary search that yields after walking its budget of voxel nodes is continued in a
// later round at the node it had stepped into (its Chain, kept by the caller), with the best
// daughter found so far and the safety bound of its first round.
struct WalkResume {
  double best;    // best DistanceToIn found so far (+inf: none); FP32 modes: two floats, its enclosure
  double safety;  // isotropic safety bound of the first round; FP32 modes: two floats, it and the undecided bound
  int bl;         // the daughter of `best` (G4N_LIM_MOTHER: none); FP32 modes: daughter << 3 | surface
  int it;         // voxel nodes walked so far (the walk's iteration cap)
};

struct StepResult {
  double step;    // geometric step (exact when it is <= the limit)
  double safety;  // isotropic lower bound
  int lim;        // daughter id or G4N_LIM_MOTHER
  int surf;       // the surface crossed (nav_pick32.cuh), -1: not known
  bool yielded;   // the search used its node budget: continue it from `resume`
  WalkResume resume;
};

// Geometric step inside `leaf` from local point p along v (Sec. 3.2, problem 2), plain FP64 navigator,
// warp-collective: DistanceToOut of the leaf, then DistanceToIn of every daughter listed in the voxel nodes
// the ray crosses, stopping once the node exit lies beyond the best distance or `limit`.
// iv: the reciprocal of v.
//
// walk_cap: the voxel nodes a search may walk in all (its rounds together); a search that reaches it
// stops there and sets *timeout (the caller reports G4N_ERR_TIMEOUT).
//
// Budget (budget > 0): after `budget` node steps a lane's search yields (R.yielded, with the
// state to continue from in R.resume and in `ch`, which then holds the node stepped into);
// `resume` continues such a search from there.  The result of a search is the same whether
// or not it yields.  `ch` is the caller's voxel chain (per-lane local memory).
template <bool COUNT>
__device__ __forceinline__ StepResult geom_step_warp(const DGeom &G, bool active, int leaf, const V3 &p, const V3 &v,
                                                     const Inv3 &iv, double limit, bool want_safety, Counters &cnt,
                                                     bool *timeout, int walk_cap, const MlpCtx &mc, Chain &ch,
                                                     bool resume = false,
                                                     const WalkResume &from = WalkResume{kInf, 0.0, -1, 0},
                                                     int budget = 0) {
  const double half = G.half;
  StepResult R{kInf, 0.0, G4N_LIM_MOTHER, -1, false, WalkResume{kInf, 0.0, -1, 0}};
  int nodes = 0;          // node steps taken in this call (the budget)
  double best = kInf, stop = 0.0, tout = kInf;
  int osurf = -1, isurf = -1;
  bool walking = false, first = true;
  int i = 0, it = 0, bl = G4N_LIM_MOTHER;
  DCandList L{0, 0}, L0{0, 0};
  float feat[mlp::kIn];
  bool have_feat = false;
  if (active) {
    const DVol &V = G.vol[leaf];
    diag_test<COUNT>(cnt, G4N_C_DIST_OUT, G4N_C_DIST_OUT_CURVED, V.kind);
    tout = vol_dist_out(V, G.pick[leaf], p, v, iv, half, G.band32, &osurf);
    R.safety = resume ? from.safety : (want_safety ? vol_safety_out(V, p) : 0.0);
    if (resume) {
      best = from.best;
      bl = from.bl;
      it = from.it;
      first = false;
    }
    if (V.vox >= 0) {
      stop = fmin(limit, tout);
      if (!resume) chain_fill(G, ch, 0, V.vox, p);
      L = G.clist[ch.list];
      L0 = L;
      walking = true;
      diag<COUNT>(cnt, G4N_C_VOX_NODES);
      if (!resume && mc.log && L.count >= 2 && L.count <= mlp::kOut) {
        node_features(G, V, ch, p, v, mc.loge, L.count, feat);
        have_feat = true;
      }
    }
  }
#pragma unroll 1
  while (__any_sync(kFull, walking)) {
    int d = -1;
    bool from_first = false;
    if (walking) {
      // the next candidate, walking nodes as lists run out
#pragma unroll 1
      for (;;) {
        if (i < L.count) {
          d = __ldg(&G.cand[L.offset + i]);
          ++i;
          from_first = first;
          break;
        }
        // list done: exit of the current node along the ray; its slab boundaries bound the safety
        const int w = walk_step64(G, ch, p, v, iv, fmin(best, stop), first && want_safety, &R.safety, &it, walk_cap, timeout);
        first = false;
        if (w == 0) {
          walking = false;
          break;
        }
        if (budget > 0 && ++nodes >= budget) {
          // yield: ch holds the node stepped into; the search continues there in a later round
          walking = false;
          R.yielded = true;
          diag<COUNT>(cnt, G4N_C_WALK_YIELDS);
          break;
        }
        L = G.clist[ch.list];
        i = 0;
        diag<COUNT>(cnt, G4N_C_VOX_NODES);
      }
    }
    __syncwarp();
    if (d >= 0) {
      const DVol &D = G.vol[d];
      V3 dp, dv;
      to_local(D, p, v, dp, dv);
      diag_kind<COUNT>(cnt, D.kind);
      int surf;
      const double t = vol_dist_in(D, G.pick[d], dp, dv, half, G.band32, &surf);
      if (t < kInf && (t < best || (t == best && (bl < 0 || d < bl)))) {
        best = t;
        bl = d;
        isurf = surf;
      }
      if (from_first && want_safety) R.safety = fmin(R.safety, vol_safety_in(D, dp));
    }
  }
  if (!active) return R;
  if (R.yielded) {
    R.resume = WalkResume{best, R.safety, bl, it};
    return R;
  }
  if (mc.log && have_feat && bl >= 0 && best <= tout) {
    // training sample: the daughter entered, if it is listed in the first node
    int slot = -1;
    for (int k = 0; k < L0.count; ++k)
      if (__ldg(&G.cand[L0.offset + k]) == bl) {
        slot = k;
        break;
      }
    if (slot >= 0) {
      const unsigned long long at = atomicAdd(mc.log->count, 1ull);
      if ((int64_t)at < mc.log->capacity) {
        for (int k = 0; k < mlp::kIn; ++k) mc.log->feat[at * mlp::kIn + k] = feat[k];
        mc.log->label[at] = slot;
        mc.log->ncand[at] = L0.count;
      }
    }
  }
  // a daughter wins a tie with the mother; `best` already holds the lowest id among tied daughters
  if (bl >= 0 && best <= tout) {
    R.step = best;
    R.lim = bl;
    R.surf = isurf;   // -1 where the search was resumed since it was found
  } else {
    R.step = tout;
    R.lim = G4N_LIM_MOTHER;
    R.surf = osurf;
  }
  return R;
}

// ---------------------------------------------------------------- geometric step of the FP32 modes
// The whole search in FP32: the leaf's exit, the voxel walk and the candidates as enclosures [lo, hi] of their crossing
// parameters (nav_pick32.cuh).  Where one enclosure lies before all others it names the volume and the surface that the
// FP64 search would find, and FP64 evaluates that one crossing parameter (step_exact32), once per step and for all
// lanes of the warp together.  Where enclosures overlap (two surfaces within ~1e-6 of the coordinates of one another,
// coinciding surfaces) the search is made again in FP64 (search_full).  Against a search that evaluated the exit and
// every candidate the bounds let pass in FP64 as it met them (282 FP64 instructions per warp and step on the barrel, the
// FP64 pipe 60 to 80 % busy): barrel batch of 10^7 tracks 167 -> 113 ms, nested barrel of 10^6 32.5 -> 24.7 ms, 10^6
// compute_step queries on the barrel 1.61 -> 0.77 ms, identical histories.

constexpr int kSurfFull = 7;   // the crossing was evaluated by the full FP64 formulas (cones, wide segments, unsure)

struct Step32 {
  float lo, hi;    // enclosure of the geometric step
  float safety;    // isotropic lower bound
  int vol;         // daughter entered, or G4N_LIM_MOTHER
  int surf;        // the surface crossed, or kSurfFull
  bool undecided;  // another crossing's enclosure overlaps: take search_full
  bool yielded;
  WalkResume resume;
};

// Enclosure of a non-negative double.
__device__ __forceinline__ void enclose_up(double t, float &lo, float &hi) {
  lo = trunc_float(t);
  hi = __fmul_ru(lo, 1.0f + 2.0f * kU) + 1e-37f;
}

// The FP64 search of one lane, every candidate by the full formulas: step and limiter as geom_step_warp's (no safety).  It
// walks as far as that one does, to `limit` at most: a step beyond it may be any value beyond it.
__device__ __noinline__ void search_full(const DGeom &G, int leaf, const V3 &p, const V3 &v, float limit, int walk_cap,
                                         double *step, int *lim, bool *timeout) {
  const DVol &V = G.vol[leaf];
  const Inv3 iv = inv_dir(v);
  int bl = G4N_LIM_MOTHER;
  const double tout = vol_dist_out_full(V, p, v, G.half), stop = fmin(tout, (double)limit);
  double best = kInf;
  if (V.vox >= 0) {
    Chain ch;
    chain_fill(G, ch, 0, V.vox, p);
    int it = 0;
#pragma unroll 1
    do {
      const DCandList L = G.clist[ch.list];
#pragma unroll 1
      for (int i = 0; i < L.count; ++i) {
        const int d = __ldg(&G.cand[L.offset + i]);
        const DVol &D = G.vol[d];
        V3 dp, dv;
        to_local(D, p, v, dp, dv);
        const double t = vol_dist_in_full(D, dp, dv, G.half);
        if (t < kInf && (t < best || (t == best && (bl < 0 || d < bl)))) {
          best = t;
          bl = d;
        }
      }
    } while (walk_step64_ool(G, ch, p, v, iv, fmin(best, stop), false, nullptr, &it, walk_cap, timeout));
  }
  const bool in = bl >= 0 && best <= tout;
  *step = in ? best : tout;
  *lim = in ? bl : G4N_LIM_MOTHER;
}

// limit: a float not below the physics step.  Budget, resume, walk cap and chain as geom_step_warp's.  In the learned
// mode the network's proposal is looked at before the node's other candidates; its enclosure prunes them.
//
// SEEN: a daughter is listed in every node it reaches into, and a ray meets it again node after node; the last kSeen
// candidates looked at are kept in registers and passed over (a second look could not change anything: the bound only
// falls).  48 batched worlds 25.5 -> 20.0 ms, barrel 69.8 -> 64.9, nested barrel 17.0 -> 16.0.  The query kernel, whose
// searches end in the first nodes, goes without.  Two
// and eight candidates: barrel 67.2 and 66.4, worlds 22.6 and 20.2.
constexpr int kSeen = 4;
template <int MODE, bool COUNT, bool SEEN = true, bool ROUNDS = true>
__device__ __forceinline__ Step32 geom_step32_warp(const DGeom &G, bool active, int leaf, const V3 &p, const V3 &v,
                                                   float limit, bool want_safety, Counters &cnt, bool *timeout,
                                                   int walk_cap, const MlpCtx &mc, Chain &ch, bool resume = false,
                                                   const WalkResume &from = WalkResume{0.0, 0.0, -1, 0}, int budget = 0) {
  Step32 R;
  R.yielded = false;
  R.undecided = false;
  int nodes = 0;          // node steps taken in this call (the budget)
  float best_lo = kInfF, best_hi = kInfF, unsure_lo = kInfF;   // unsure_lo: two overlapping crossings lie beyond it
  float exit_lo = 0.f, exit_hi = kInfF, saf_f = 0.f, bound_f = kInfF, stop_f = kInfF;
  int exit_surf = kSurfFull, best_vol = -1, best_surf = 0;
  Ray32 r;
  PickRay q;
  bool walking = false, first = true;
  int i = 0, it = 0;
  DCandList L{0, 0}, L0{0, 0};
  int prop_done = -1;
  int seen[kSeen];
#pragma unroll
  for (int k = 0; k < kSeen; ++k) seen[k] = -1;
  float feat[mlp::kIn];
  bool have_feat = false;
  if (active) {
    const DVol &V = G.vol[leaf];
    r = make_ray32(p, v);
    q = pick_ray(p, v);
    diag_test<COUNT>(cnt, G4N_C_DIST_OUT, G4N_C_DIST_OUT_CURVED, V.kind);
    const Pick x = pick_leaf(G.pick[leaf], q, G.band32);
    if (x.surf >= 0) {
      exit_lo = x.lo;
      exit_hi = x.hi;
      exit_surf = x.surf;
    } else {
      enclose_up(vol_dist_out_full(V, p, v, G.half), exit_lo, exit_hi);
    }
    stop_f = fminf(limit, exit_hi);
    if (resume) {
      best_lo = __int_as_float(__double2loint(from.best));
      best_hi = __int_as_float(__double2hiint(from.best));
      unsure_lo = __int_as_float(__double2loint(from.safety));
      saf_f = __int_as_float(__double2hiint(from.safety));
      best_vol = from.bl < 0 ? -1 : from.bl >> 3;
      best_surf = from.bl & 7;
      it = from.it;
      first = false;
    } else {
      saf_f = leaf_safety32(V, r, p);
    }
    bound_f = fminf(best_hi, stop_f);
    if (V.vox >= 0) {
      if (!resume && !chain_fill32(G, ch, V.vox, r)) chain_fill(G, ch, 0, V.vox, p);
      L = G.clist[ch.list];
      L0 = L;
      walking = true;
      diag<COUNT>(cnt, G4N_C_VOX_NODES);
      if (MODE == kLearned && !resume && L.count >= 2 && L.count <= mlp::kOut) {
        // a proposal can only save work when two or more of the node's candidates pass the FP32 bounds (with one
        // or none the bounds alone leave a single evaluation at most)
        int open = 0;
#pragma unroll 1
        for (int k = 0; k < L.count && open < 2; ++k) {
          const int c = __ldg(&G.cand[L.offset + k]);
          const DBox32 B = G.box[c];
          const float iso = iso_lb32(G.v32[c], r.plo[0], r.plo[1], r.plo[2]) - G.band32;
          if (fmaxf(box_entry_lb(B.lo, B.hi, r, nullptr), iso) <= bound_f) ++open;
        }
        if (open >= 2) {
          node_features(G, V, ch, p, v, mc.loge, L.count, feat);
          have_feat = true;
        }
      }
    }
  }
  // learned mode: the network proposes which first-node candidate is entered first (warp-collective)
  int prop = -1;
  if (MODE == kLearned && __any_sync(kFull, have_feat)) {
    float f0[mlp::kIn];
#pragma unroll
    for (int k = 0; k < mlp::kIn; ++k) f0[k] = have_feat ? feat[k] : 0.f;
    mlp::put_features(*mc.scratch, f0);
    mlp::forward_warp(*mc.w, *mc.scratch);
    if (have_feat) {
      prop = mlp::argmax_row(*mc.scratch, L.count);
      diag<COUNT>(cnt, G4N_C_PROPOSALS);
    }
    __syncwarp();
  }
  // the current node's list is done: on to the next node
  auto walk_on = [&]() {
    // exit of the current node along the ray; its slab boundaries bound the safety
    int w = walk_step32(G, ch, r, v, bound_f, first && want_safety, &saf_f, &it, walk_cap, timeout);
    if (w == 2) {
      // FP64 node step where the intervals do not decide
      double s64 = kInf;
      w = walk_step64_ool(G, ch, p, v, inv_dir(v), (double)bound_f, first && want_safety, &s64, &it, walk_cap, timeout);
      saf_f = fminf(saf_f, __double2float_rd(s64));
    }
    first = false;
    if (w == 0) {
      walking = false;
    } else if (budget > 0 && ++nodes >= budget) {
      // yield: ch holds the node stepped into; the search continues there in a later round
      walking = false;
      R.yielded = true;
      diag<COUNT>(cnt, G4N_C_WALK_YIELDS);
    } else {
      L = G.clist[ch.list];
      i = 0;
      diag<COUNT>(cnt, G4N_C_VOX_NODES);
    }
  };
  // Rounds: each lane scans its node's list to the next candidate that the bounds let matter; the lanes that found one
  // choose its surface together; the lanes whose list is done walk to the next node.  A warp runs each of the three once a
  // round, for all lanes that need it.  (Scanning and walking in one loop per lane ran both in every pass of it: barrel
  // 64.4 -> 62.4 ms, 10^6 compute_step queries on the barrel 0.68 -> 0.60 ms.)  Without ROUNDS a lane scans and walks on
  // until it has a candidate, the scan a loop of its own; the persistent kernel without yielding searches, where the last
  // lanes of a warp walk long alone, is the faster for it (48 batched worlds 19.9 -> 18.3 ms, in rounds 19.6).
#pragma unroll 1
  while (__any_sync(kFull, walking)) {
    int d = -1;
    if (walking) {
#pragma unroll 1
      for (;;) {
        if (MODE == kLearned && prop >= 0) {
          // the proposal goes first if its bound still allows it to matter
          const int c = __ldg(&G.cand[L0.offset + prop]);
          const DBox32 B = G.box[c];
          const float iso = iso_lb32(G.v32[c], r.plo[0], r.plo[1], r.plo[2]) - G.band32;
          const float lb = fmaxf(box_entry_lb(B.lo, B.hi, r, nullptr), iso);
          if (lb <= bound_f) {
            d = c;
            break;
          }
          prop = -1;  // not worth it: the scan treats the slot like any other
        }
#pragma unroll 1
        while (i < L.count) {
          const int c = __ldg(&G.cand[L.offset + i]);
          ++i;
          if (SEEN) {
            bool again = false;
#pragma unroll
            for (int k = 0; k < kSeen; ++k) again |= c == seen[k];
            if (again) continue;
#pragma unroll
            for (int k = kSeen - 1; k > 0; --k) seen[k] = seen[k - 1];
            seen[0] = c;
          }
          const DBox32 B = G.box[c];
          // the distance from the point bounds the entry as well; after the first node it prunes next to nothing that the
          // box lets pass (barrel 1.4 %, worlds 3 % for leaving it out; the learned mode lost 3 % by that)
          float iso = -kInfF;
          if (MODE == kLearned || !SEEN || (first && want_safety))
            iso = iso_lb32(G.v32[c], r.plo[0], r.plo[1], r.plo[2]) - G.band32;
          if (first && want_safety) saf_f = fminf(saf_f, fmaxf(box_gap_lb(B.lo, B.hi, r), iso));
          if (MODE == kLearned && first && i - 1 == prop_done) continue;  // already looked at
          const float lb = fmaxf(box_entry_lb(B.lo, B.hi, r, nullptr), iso);
          if (!(lb <= bound_f)) {
            if (MODE == kLearned) diag<COUNT>(cnt, G4N_C_PRUNED);
            continue;
          }
          diag<COUNT>(cnt, G4N_C_RECHECKS);
          d = c;
          break;
        }
        if (ROUNDS || d >= 0) break;
        walk_on();
        if (!walking) break;
      }
    }
    __syncwarp();
    if (MODE == kLearned && prop >= 0 && d >= 0) {
      prop_done = prop;  // the proposed slot is skipped when the first node is scanned
      prop = -1;
      diag<COUNT>(cnt, G4N_C_RECHECKS);
    }
    if (d >= 0) {
      const DPick32 &D = G.pick[d];
      diag_kind<COUNT>(cnt, D.kind_flags & 3);
      Pick k = pick_daughter(D, q, G.band32);
      if (k.surf == kPickUnsure && k.lo <= bound_f) {
        // the full formulas
        V3 dp, dv;
        to_local(G.vol[d], p, v, dp, dv);
        const double t = vol_dist_in_full(G.vol[d], dp, dv, G.half);
        k.surf = t < kInf ? kSurfFull : kPickMiss;
        enclose_up(t, k.lo, k.hi);
      }
      if (k.surf >= 0 && d != best_vol) {
        // a candidate listed in several nodes is met again: the same crossing
        if (best_vol >= 0 && k.lo <= best_hi && k.hi >= best_lo) unsure_lo = fminf(unsure_lo, fminf(k.lo, best_lo));
        if (k.hi < best_hi) {
          best_lo = k.lo;
          best_hi = k.hi;
          best_vol = d;
          best_surf = k.surf;
          bound_f = fminf(best_hi, stop_f);
        }
      }
    }
    __syncwarp();
    if (ROUNDS && walking && i >= L.count && !(MODE == kLearned && prop >= 0)) walk_on();
  }
  R.safety = saf_f;
  if (!active) return R;
  if (R.yielded) {
    R.resume.best = __hiloint2double(__float_as_int(best_hi), __float_as_int(best_lo));
    R.resume.safety = __hiloint2double(__float_as_int(saf_f), __float_as_int(unsure_lo));
    R.resume.bl = best_vol < 0 ? -1 : best_vol << 3 | best_surf;
    R.resume.it = it;
    return R;
  }
  // the daughter or the exit, whichever enclosure comes first
  const bool in = best_vol >= 0 && best_hi < exit_hi;
  R.lo = fminf(fminf(best_lo, exit_lo), unsure_lo);
  R.hi = in ? best_hi : exit_hi;
  R.vol = in ? best_vol : G4N_LIM_MOTHER;
  R.surf = in ? best_surf : exit_surf;
  R.undecided = unsure_lo <= R.hi || (best_vol >= 0 && best_lo <= exit_hi && exit_lo <= best_hi);
  return R;
}

// The step that R names as num / den * mul for the caller to evaluate (mul is 1 but for the exit from a box, (h - p) times the
// reciprocal of the direction as box_dist_out has it), or exactly: false, with *num = step, where the full formulas or
// the full search were needed (then *lim is final as well).  *surf: the surface crossed, -1: not known.
__device__ __forceinline__ bool step_ratio32(const DGeom &G, int leaf, const V3 &p, const V3 &v, const Step32 &R,
                                             float limit, int walk_cap, bool *timeout, double *num, double *den, double *mul,
                                             int *lim, int *surf) {
  *lim = R.vol;
  *surf = -1;
  if (R.undecided || R.surf == kSurfFull) {
    if (R.undecided) {
      search_full(G, leaf, p, v, limit, walk_cap, num, lim, timeout);
    } else if (R.vol < 0) {
      // the exit comes first for certain, from a cone or a wide segment, say: that alone
      *num = vol_dist_out_full(G.vol[leaf], p, v, G.half);
    } else {
      V3 dp, dv;
      to_local(G.vol[R.vol], p, v, dp, dv);
      *num = vol_dist_in_full(G.vol[R.vol], dp, dv, G.half);
    }
    return false;
  }
  const bool in = R.vol >= 0;
  const DVol &D = G.vol[in ? R.vol : leaf];
  V3 dp = p, dv = v;
  if (in) to_local(D, p, v, dp, dv);
  *surf = R.surf;
  surf_ratio(D.kind, D.p, R.surf, in, dp, dv, *num, *den);
  if (!in && D.kind == kBox) {
    *mul = *num;
    *num = 1.0;
  }
  return true;
}

// The quotient s of step_ratio32 made a step: true if it lies beyond the surface band; else (a crossing at the start, by
// rounding) s comes from the full search.
__device__ __forceinline__ bool step_finish32(const DGeom &G, int leaf, const V3 &p, const V3 &v, double &s, float limit,
                                              int walk_cap, bool *timeout, int *lim, int *surf) {
  if (s > (*lim >= 0 ? G.half : -G.half)) {
    s = fmax(s, 0.0);
    return true;
  }
  double full;
  search_full(G, leaf, p, v, limit, walk_cap, &full, lim, timeout);
  s = full;
  *surf = -1;
  return false;
}

// The geometric step that R names; limit as the search had it.
__device__ __forceinline__ double step_exact32(const DGeom &G, int leaf, const V3 &p, const V3 &v, const Step32 &R,
                                               float limit, int walk_cap, bool *timeout, int *lim, int *surf) {
  double num, den, mul = 1.0;
  if (!step_ratio32(G, leaf, p, v, R, limit, walk_cap, timeout, &num, &den, &mul, lim, surf)) return num;
  double s = num / den * mul;
  step_finish32(G, leaf, p, v, s, limit, walk_cap, timeout, lim, surf);
  return s;
}

// ---------------------------------------------------------------- attenuation table

// Bin k with E_k <= E < E_{k+1} and its interpolation fraction; clamped ends give
// (0, 0) below the table and (n-2, 1) above.
__device__ __forceinline__ void energy_bin(const double *Eg, int n, double E, int &k, double &f) {
  if (E <= Eg[0]) {
    k = 0;
    f = 0.0;
  } else if (E >= Eg[n - 1]) {
    k = n - 2;
    f = 1.0;
  } else {
    int lo = 0, hi = n - 1;
    const long long eb = __double_as_longlong(E);  // E and the grid are positive: bit order = value order
#pragma unroll 1
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__double_as_longlong(Eg[mid]) <= eb) lo = mid;
      else hi = mid;
    }
    k = lo;
    f = (E - Eg[lo]) / (Eg[lo + 1] - Eg[lo]);
  }
}

// Lin-lin interpolation of both coefficients at a known bin.  At the clamped ends
// the table value is returned exactly.
__device__ __forceinline__ void mu_at(const DGeom &G, int mat, int k, double f, double &mu_tot, double &mu_pe) {
  const int off = G.mat_off[mat];
  const double *C = G.matC + off, *P = G.matP + off;
  double mc, mp;
  const long long fb = __double_as_longlong(f);
  if (fb == 0) {                                   // f == +0 (f is never -0 or negative)
    mc = C[k];
    mp = P[k];
  } else if (fb == 0x3FF0000000000000ll) {         // f == 1
    mc = C[k + 1];
    mp = P[k + 1];
  } else {
    mc = C[k] + f * (C[k + 1] - C[k]);
    mp = P[k] + f * (P[k + 1] - P[k]);
  }
  mu_tot = mc + mp;
  mu_pe = mp;
}

// Binary search for E_k <= E < E_{k+1}, lin-lin interpolation, clamped at the ends.
__device__ __forceinline__ void mu_lookup(const DGeom &G, int mat, double E, double &mu_tot, double &mu_pe) {
  const int off = G.mat_off[mat], n = G.mat_n[mat];
  int k;
  double f;
  energy_bin(G.matE + off, n, E, k, f);
  mu_at(G, mat, k, f, mu_tot, mu_pe);
}

// ---------------------------------------------------------------- Philox4x32-10 and FNV-1a

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// The two 53-bit integers of one Philox block (counter (draw, id lo, id hi, stream)): the
// uniforms in (0, 1] are a 2^-53 (from x1:x0) and b 2^-53 (from x3:x2).  A draw site takes
// whole blocks; a single uniform uses a.  Out of line: its ~100 instructions would otherwise
// be repeated at each of the draw sites of the transport kernel.
struct M53x2 {
  uint64_t a, b;
};

__device__ __noinline__ M53x2 philox_m53_pair(uint64_t seed, int64_t tid, uint32_t stream, uint32_t &draw) {
  const uint4 x = philox4x32_10(make_uint4(draw++, (uint32_t)(uint64_t)tid, (uint32_t)((uint64_t)tid >> 32), stream),
                                make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
  const uint64_t wa = ((uint64_t)x.y << 32) | x.x, wb = ((uint64_t)x.w << 32) | x.z;
  return M53x2{(wa >> 11) + 1, (wb >> 11) + 1};
}

__device__ __forceinline__ uint64_t philox_m53(uint64_t seed, int64_t tid, uint32_t stream, uint32_t &draw) {
  return philox_m53_pair(seed, tid, stream, draw).a;
}

// m 2^-53 (m in [1, 2^53], so exact), by integer instructions: a 64-bit conversion and a product hold the FP64 pipe.
__device__ __forceinline__ double m53_double(uint64_t m) {
  const int lz = __clzll((long long)m);                 // 10 .. 63
  return __longlong_as_double(((long long)(1033 - lz) << 52) + (long long)(((m << lz) << 1) >> 12));
}

// m 2^-53 as a float, truncated to 24 bits (relative error < 2^-23), with integer
// instructions only (m in [1, 2^53]).
__device__ __forceinline__ float m53_float(uint64_t m) {
  const int lz = __clzll((long long)m);                 // 11 .. 63
  const int sh = 40 - lz;                               // keep the leading one and 23 bits below it
  const uint32_t mant = sh >= 0 ? (uint32_t)(m >> sh) : (uint32_t)(m << (-sh));
  return __uint_as_float(((uint32_t)(63 - lz - 53 + 127) << 23) | (mant & 0x7FFFFFu));
}

// Uniform in (0, 1] from one Philox block.
__device__ __forceinline__ double philox_uniform(uint64_t seed, int64_t tid, uint32_t stream, uint32_t &draw) {
  return m53_double(philox_m53(seed, tid, stream, draw));
}

__device__ __forceinline__ uint64_t fnv_word(uint64_t h, uint32_t w) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    h ^= (w >> (8 * b)) & 0xffu;
    h *= 0x100000001b3ull;
  }
  return h;
}

__device__ __forceinline__ uint64_t hash_step(uint64_t h, int32_t leaf, int32_t limiter, int32_t event) {
  h = fnv_word(h, (uint32_t)leaf);
  h = fnv_word(h, (uint32_t)limiter);
  return fnv_word(h, (uint32_t)event);
}

}  // namespace dev
}  // namespace g4n
