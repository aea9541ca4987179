// DistanceToIn from points inside the solid (a query whose path names the mother): the FP32 choice (csrc/nav_pick32.cuh)
// against the full FP64 formulas.  Builds on the shims of pick_host.cpp.
#include "pick_host.cpp"

// out: 0 points inside the solid, 1 of them with a DistanceToIn, 2 undecided by the bounds, 3 wrong.
extern "C" void pick_inside_check(int kind, int seg, int bore, double scale, int near, long long n, uint64_t seed, long long *out) {
  rng.seed(seed);
  const double half = 0.5e-9;
  const float band = 2.0f * trunc_float(half);
  for (int k = 0; k < 4; ++k) out[k] = 0;
  for (long long i = 0; i < n; ++i) {
    double p[7] = {scale, scale, scale, 0, 0, 0, 0};
    int flags = 0;
    if (kind == kBox) {
      for (int k = 0; k < 3; ++k) p[k] = scale * std::exp(uni(-2.0, 0.0));
    } else if (kind == kTube) {
      p[1] = scale * uni(0.3, 1.0);
      p[0] = bore ? p[1] * uni(0.05, 0.9) : 0.0;
      p[2] = scale * uni(0.3, 1.0);
      flags = bore ? kHasRmin : 0;
      if (seg) {
        const double s = uni(0.0, 6.28), d = seg == 1 ? uni(0.05, 3.14) : uni(3.15, 6.2);
        p[3] = std::cos(s); p[4] = std::sin(s); p[5] = std::cos(s + d); p[6] = std::sin(s + d);
        flags |= kSeg | (seg == 2 ? kWide : 0);
      }
    }
    V3 x{uni(-1, 1) * scale, uni(-1, 1) * scale, uni(-1, 1) * scale};
    const double ct = uni(-1, 1), ph = uni(0, 6.283185307), st = std::sqrt(1 - ct * ct);
    const V3 v{st * std::cos(ph), st * std::sin(ph), ct};
    const bool in = kind == kBox ? box_inside(p, x, v, half) : kind == kOrb ? orb_inside(p[0], x, v, half) : tube_inside(p, flags, x, v, half);
    if (!in) continue;
    if (kind == kBox && near) {   // along the ray to the face it leaves by, and there within 10^near bands of it, still inside or just out
      int face;
      const Inv3 iv{1 / v.x, 1 / v.y, 1 / v.z};
      const double t = box_dist_out(p, x, v, iv, &face) + uni(-1, 1) * std::pow(10.0, near) * half;
      x = V3{x.x + t * v.x, x.y + t * v.y, x.z + t * v.z};
    }
    ++out[0];
    const double full = kind == kBox ? box_dist_in(p, x, v, half) : kind == kOrb ? orb_dist_in(p[0], x, v, half) : tube_cross(p, flags, x, v, half, true);
    if (full < kInf) ++out[1];
    const double t0[3] = {near ? uni(-900, 900) : 0.0, near ? uni(-900, 900) : 0.0, near ? uni(-900, 900) : 0.0};
    DPick32 D;
    std::memset(&D, 0, sizeof D);
    for (int k = 0; k < 7; ++k) D.q[k] = (float)p[k];
    if (kind == kBox)
      for (int k = 0; k < 3; ++k) D.q[3 + k] = (float)(p[k] - (double)D.q[k]);
    for (int k = 0; k < 3; ++k) {   // placed in its mother
      D.th[k] = (float)t0[k];
      D.tl[k] = (float)(t0[k] - (double)D.th[k]);
    }
    D.c = 1.0f;
    D.kind_flags = (flags | kPlacedAligned) << 2 | kind;
    const Pick k = pick_daughter(D, pick_ray(V3{x.x + t0[0], x.y + t0[1], x.z + t0[2]}, v), band);
    if (k.surf == kPickUnsure) {
      ++out[2];
      if (full < (double)k.lo) ++out[3];
    } else if (k.surf == kPickMiss) {
      if (full < kInf) ++out[3];
    } else {
      double num, den;
      surf_ratio(kind, p, k.surf, true, x, v, num, den);
      if (!(std::fabs(num / den - full) <= 1e-11 * std::fmax(1.0, scale))) ++out[3];
    }
  }
}
