// The FP32 surface choice (csrc/nav_pick32.cuh) against the full FP64 formulas (csrc/nav_solids.cuh), compiled for the
// host: CUDA's qualifiers and the few intrinsics the two headers use are given here, the approximate reciprocal and root
// with an error of up to one unit in the last place.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>

#define __device__
#define __forceinline__ inline
#define __noinline__
using std::copysign;
using std::copysignf;
using std::fabs;
using std::fmax;
using std::fmin;
static inline long long __double_as_longlong(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static inline int __double2loint(double x) { return (int)__double_as_longlong(x); }
static inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static std::mt19937_64 rng(1);
static inline float jitter(float f) {
  const int k = (int)(rng() % 3) - 1;
  return k == 0 || !std::isfinite(f) ? f : std::nextafterf(f, k > 0 ? INFINITY : -INFINITY);
}

#include "nav_solids.cuh"
namespace g4n {
namespace dev {
static inline float rcp_approx(float x) { return jitter(1.0f / x); }
static inline float sqrt_approx(float x) { return jitter(std::sqrt(x)); }
}  // namespace dev
}  // namespace g4n
#include "nav_pick32.cuh"

using namespace g4n;
using namespace g4n::dev;

static double uni(double a, double b) { return a + (b - a) * ((double)(rng() >> 11) * 0x1.0p-53); }

// `mode` 0: a point anywhere around the solid; 1: the point of a crossing (in a surface's band), moved along the ray by
// at most 1e-9; 2: a point on the solid's axis.  `rotated`: the solid is a daughter, rotated about z and moved by up to 2000
// in its mother's frame, in which the ray is given.
// out: 0 cases, 1 chosen, 2 misses proved, 3 unsure (chosen, but the quotient lies in the band, among them), 4 wrong, 5 crossing outside its enclosure; *worst: relative error.
extern "C" void pick_check(int kind, int seg, int bore, int mode, int rotated, double scale, long long n, uint64_t seed,
                           long long *out, double *worst) {
  rng.seed(seed);
  const double half = 0.5e-9;
  const float band = 2.0f * trunc_float(half);
  for (int k = 0; k < 6; ++k) out[k] = 0;
  *worst = 0.0;
  for (long long i = 0; i < n; ++i) {
    double p[7] = {0, 0, 0, 0, 0, 0, 0};
    int flags = 0;
    double ext;
    if (kind == kBox) {
      for (int k = 0; k < 3; ++k) p[k] = scale * std::exp(uni(-3.0, 0.0));
      ext = scale;
    } else if (kind == kOrb) {
      p[0] = scale * std::exp(uni(-3.0, 0.0));
      ext = p[0];
    } else {
      p[1] = scale * std::exp(uni(-2.0, 0.0));
      p[0] = bore ? p[1] * uni(0.05, 0.98) : 0.0;
      p[2] = scale * std::exp(uni(-2.0, 1.0));
      flags = bore ? kHasRmin : 0;
      if (seg) {
        const double s = uni(0.0, 6.28), d = seg == 1 ? uni(0.05, 3.14) : uni(3.15, 6.2);
        p[3] = std::cos(s); p[4] = std::sin(s); p[5] = std::cos(s + d); p[6] = std::sin(s + d);
        flags |= kSeg | (seg == 2 ? kWide : 0);
      }
      ext = std::fmax(p[1], p[2]);
    }
    V3 x{uni(-2, 2) * ext, uni(-2, 2) * ext, uni(-2, 2) * ext}, v;
    const double ct = uni(-1, 1), ph = uni(0, 6.283185307), st = std::sqrt(1 - ct * ct);
    v = V3{st * std::cos(ph), st * std::sin(ph), ct};
    if (rng() % 16 == 0) {  // along an axis
      const int a = (int)(rng() % 3);
      v = V3{a == 0 ? 1.0 : 0.0, a == 1 ? 1.0 : 0.0, a == 2 ? 1.0 : 0.0};
    }
    DVol d;
    std::memset(&d, 0, sizeof d);
    for (int k = 0; k < 7; ++k) d.p[k] = p[k];
    d.kind = kind;
    d.flags = flags;
    auto inside = [&](const V3 &q) {
      return kind == kBox ? box_inside(p, q, v, half) : kind == kOrb ? orb_inside(p[0], q, v, half) : tube_inside(p, flags, q, v, half);
    };
    auto dist_in = [&](const V3 &q) {
      return kind == kBox ? box_dist_in(p, q, v, half) : kind == kOrb ? orb_dist_in(p[0], q, v, half) : tube_cross(p, flags, q, v, half, true);
    };
    auto dist_out = [&](const V3 &q) {
      if (kind == kOrb) return orb_dist_out(p[0], q, v);
      if (kind == kTube) {
        const double t = tube_cross(p, flags, q, v, half, false);
        return t == kInf ? 0.0 : std::fmax(t, 0.0);
      }
      int face;
      const Inv3 iv{v.x != 0 ? 1 / v.x : 0, v.y != 0 ? 1 / v.y : 0, v.z != 0 ? 1 / v.z : 0};
      return box_dist_out(p, q, v, iv, &face);
    };
    if (mode == 2) {  // on the axis, as from a beam line: b = x . v is a signed zero
      x.x = x.y = 0.0;
    }
    if (mode == 1) {  // to a surface of the solid, entering or leaving
      double t = inside(x) ? dist_out(x) : dist_in(x);
      if (!(t < kInf)) continue;
      t += uni(-1e-9, 1e-9);
      x = V3{x.x + t * v.x, x.y + t * v.y, x.z + t * v.z};
    }
    const bool in = inside(x);
    if (rotated && in) continue;
    ++out[0];
    DPick32 D;
    std::memset(&D, 0, sizeof D);
    for (int k = 0; k < 7; ++k) D.q[k] = (float)p[k];
    Pick k;
    if (!rotated) {
      D.c = 1.0f;
      D.kind_flags = (flags | kPlacedAligned) << 2 | kind;
      const PickRay r = pick_ray(x, v);
      k = in ? pick_leaf(D, r, band) : pick_daughter(D, r, band);
    } else {  // the solid as a daughter, rotated and moved in its mother's frame
      const double a = uni(0, 6.283185307), c = std::cos(a), s = std::sin(a);
      const double t[3] = {uni(-2000, 2000), uni(-2000, 2000), uni(-2000, 2000)};
      for (int j = 0; j < 3; ++j) {
        D.th[j] = (float)t[j];
        D.tl[j] = (float)(t[j] - (double)D.th[j]);
      }
      D.c = (float)c;
      D.s = (float)s;
      D.kind_flags = flags << 2 | kind;
      const V3 m{c * x.x - s * x.y + t[0], s * x.x + c * x.y + t[1], x.z + t[2]}, mv{c * v.x - s * v.y, s * v.x + c * v.y, v.z};
      k = pick_daughter(D, pick_ray(m, mv), band);
    }
    const double full = in ? dist_out(x) : dist_in(x);
    if (k.surf == kPickUnsure) {
      ++out[3];
      if (full < (double)k.lo) ++out[4];
      continue;
    }
    if (k.surf == kPickMiss) {
      ++out[2];
      if (in || full < kInf) ++out[4];
      continue;
    }
    ++out[1];
    double num, den;
    surf_ratio(kind, p, k.surf, !in, x, v, num, den);
    double t = num / den;
    if (!(t > (in ? -half : half))) {   // the caller then takes the full formulas
      ++out[3];
      continue;
    }
    t = std::fmax(t, 0.0);
    if (!(full < kInf) || std::fabs(t - full) > 1e-11 * std::fmax(1.0, std::fmax(scale, full))) ++out[4];
    else *worst = std::fmax(*worst, std::fabs(t - full) / std::fmax(1.0, full));
    if (!((double)k.lo <= full && full <= (double)k.hi) && full > 0.0) ++out[5];
  }
}
