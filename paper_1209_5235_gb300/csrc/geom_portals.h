// geom_portals.h -- relocation across the faces of any box, tube segment or orb, decided once on the host (included by
// geom_host.cpp).
//
// After a step that crosses a face of volume V -- leaving V, or entering V from its mother -- the navigator searches for
// the new leaf: up through the mothers, then down through the daughters in id order, with an Inside test each.  For most
// faces the search ends in the same volume wherever on the face the ray crosses (the next segment behind a phi plane, the
// mother around a lone orb).  A portal is that volume, found here by running the search for the whole face at once.
//
// All rotations are about z, so every surface is a z plane, a vertical plane, or a vertical cylinder, or a sphere, and a
// face is a point set in xy times a z interval.  Each Inside test of the search is decided for the whole face by the
// signed distances of the tested volume's surfaces over it:
//   * a surface that coincides with the crossed face (within tol / 16) holds every crossing point in its band, where the
//     direction decides: crossed inward, it is passed; outward, the volume is left;
//   * a surface that coincides with another face of V lies farther than the band from the crossing points for which the
//     portal is used (the device takes it only for points that far from V's other faces), on a known side;
//   * any other surface's distance is bounded over the face; it must keep one sign by a margin.
// If some test is not decided the face has no portal.  kPortalNone: none; -1: the ray leaves the world.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

#include "g4n_internal.h"

namespace g4n {

constexpr double kPi = 3.14159265358979323846;

enum PortalSurf : int { kZPlane, kLine, kCircle, kSphere };

// d(x, y, z), positive inside the volume: z plane n z + o; line nx x + ny y + o; circle and sphere sign (R - distance to
// the centre).  World frame.
struct PSurf {
  int type = kZPlane;
  double nx = 0, ny = 0, o = 0, cx = 0, cy = 0, cz = 0, R = 0;
  int sign = 1, face = 0;
};

// A face in xy (points, an arc, an annular sector or a disc's bounding circle for an orb) and z.
struct PPatch {
  enum Kind { kPoints, kArc, kSector, kBall } kind = kPoints;
  int n = 0;                       // points of a segment (2) or convex polygon (4, in order)
  double px[4], py[4];
  double cx = 0, cy = 0, r0 = 0, r1 = 0, a0 = 0, a1 = 0;
  double c[2] = {0, 0}, s[2] = {0, 0};   // cosines and sines of a0, a1
  double zlo = 0, zhi = 0;
};

// Is the direction (dx, dy) in the patch's angles a0 .. a1 (<= 2 pi), or within 1e-12 of them?  (In is the safe answer: it
// widens the ranges below.)
inline bool direction_in(const PPatch &P, double dx, double dy) {
  const double span = P.a1 - P.a0, tol = 1e-12 * (std::fabs(dx) + std::fabs(dy));
  if (span > 2.0 * kPi - 1e-9) return true;
  const bool after = P.c[0] * dy - P.s[0] * dx >= -tol, before = dx * P.s[1] - dy * P.c[1] >= -tol;
  return span <= kPi ? after && before : after || before;
}

inline double length(double x, double y) { return std::sqrt(x * x + y * y); }   // (hypot's care for overflow costs 20 ns)

struct PRange {
  double lo = INFINITY, hi = -INFINITY;
  void add(double x) {
    lo = std::min(lo, x);
    hi = std::max(hi, x);
  }
};

// nx x + ny y + o over the patch.
inline PRange range_linear(const PPatch &P, double nx, double ny, double o) {
  PRange r;
  if (P.kind == PPatch::kPoints) {
    for (int i = 0; i < P.n; ++i) r.add(nx * P.px[i] + ny * P.py[i] + o);
    return r;
  }
  const double c = nx * P.cx + ny * P.cy + o, len = length(nx, ny);
  if (P.kind == PPatch::kBall) {
    r.add(c - len * P.r1);
    r.add(c + len * P.r1);
    return r;
  }
  const bool most = direction_in(P, nx, ny), least = direction_in(P, -nx, -ny);
  for (int k = P.kind == PPatch::kArc ? 1 : 0; k < 2; ++k) {
    const double R = k ? P.r1 : P.r0;
    for (int a = 0; a < 2; ++a) r.add(c + R * (nx * P.c[a] + ny * P.s[a]));
    if (most) r.add(c + R * len);
    if (least) r.add(c - R * len);
  }
  return r;
}

inline double segment_distance(double x, double y, double ax, double ay, double bx, double by) {
  const double dx = bx - ax, dy = by - ay, l2 = dx * dx + dy * dy;
  const double t = l2 > 0.0 ? std::min(1.0, std::max(0.0, ((x - ax) * dx + (y - ay) * dy) / l2)) : 0.0;
  return length(ax + t * dx - x, ay + t * dy - y);
}

// Distance from (x, y) over the patch.
inline PRange range_distance(const PPatch &P, double x, double y) {
  PRange r;
  if (P.kind == PPatch::kPoints) {
    for (int i = 0; i < P.n; ++i) r.add(length(P.px[i] - x, P.py[i] - y));
    bool in = P.n > 2, pos = false, neg = false;
    for (int i = 0; i < P.n; ++i) {
      const int j = (i + 1) % P.n;
      r.add(segment_distance(x, y, P.px[i], P.py[i], P.px[j], P.py[j]));
      const double s = (P.px[j] - P.px[i]) * (y - P.py[i]) - (P.py[j] - P.py[i]) * (x - P.px[i]);
      pos |= s > 0;
      neg |= s < 0;
    }
    if (in && !(pos && neg)) r.add(0.0);
    return r;
  }
  const double D = length(x - P.cx, y - P.cy);
  if (P.kind == PPatch::kBall) {
    r.add(std::max(0.0, D - P.r1));
    r.add(D + P.r1);
    return r;
  }
  const bool near = direction_in(P, x - P.cx, y - P.cy), far = direction_in(P, P.cx - x, P.cy - y);
  for (int k = P.kind == PPatch::kArc ? 1 : 0; k < 2; ++k) {
    const double R = k ? P.r1 : P.r0;
    for (int a = 0; a < 2; ++a) r.add(length(P.cx + R * P.c[a] - x, P.cy + R * P.s[a] - y));
    if (near) r.add(std::fabs(R - D));
    if (far) r.add(R + D);
    if (D < 1e-9 * (1.0 + R)) {   // about the centre: the angle of (x, y) means nothing
      r.add(std::max(0.0, R - D));
      r.add(R + D);
    }
  }
  if (P.kind == PPatch::kSector) {
    for (int a = 0; a < 2; ++a)
      r.add(segment_distance(x, y, P.cx + P.r0 * P.c[a], P.cy + P.r0 * P.s[a], P.cx + P.r1 * P.c[a], P.cy + P.r1 * P.s[a]));
    if (D >= P.r0 && D <= P.r1 && (near || D < 1e-9)) r.add(0.0);
  }
  return r;
}

class PortalBuilder {
 public:
  PortalBuilder(const HGeom &geom, double tolerance) : g(geom), tol(tolerance), eps(tolerance / 16.0) {
    const int n = (int)g.vol.size();
    surfs.resize(n);
    daughters.resize(n);
    cand_seen.resize(n);
    list_seen.resize(g.clist.size());
    double size = 0.0;
    for (int i = 0; i < n; ++i) {
      volume_surfaces(i);
      const DVol &v = g.vol[i];
      if (v.mother >= 0) daughters[v.mother].push_back(i);
      const DWorld &w = g.wxf[i];
      size = std::max(size, std::fabs(w.tx) + std::fabs(w.ty) + std::fabs(w.tz) + extent(v));
    }
    margin = 1e-6 + 1e-9 * size + 2.0 * tol;   // clear of the band, half a tolerance, at any tolerance scale
    // the band has to be far above the rounding of coordinates of this size (2e-16 each, through a move and a transform)
    // for "in the band" to be certain
    usable = 0.5 * tol >= 4e-14 * size;
    scale = size;
  }

  // Portals of volume V: [f] leaving through face f, [6 + f] entering through it.
  void build(int V, int32_t *out) {
    for (int k = 0; k < 12; ++k) out[k] = kPortalNone;
    const DVol &v = g.vol[V];
    if (!usable || v.kind == kCone) return;
    for (const PSurf &s : surfs[V]) {
      PPatch P;
      if (!patch_of(V, s.face, P)) continue;
      int leaf;
      if (search(V, s, P, +1, leaf)) out[s.face] = leaf;
      if (v.mother >= 0 && search(V, s, P, -1, leaf)) out[6 + s.face] = leaf;
    }
  }

 private:
  const HGeom &g;
  double tol, eps, margin = 0.0, scale = 0.0;
  bool usable = false;
  std::vector<std::vector<PSurf>> surfs;
  std::vector<std::vector<int32_t>> daughters;        // in id order
  std::vector<int32_t> lists, cands;
  std::vector<uint32_t> list_seen, cand_seen;         // the search that last met a list, a candidate
  uint32_t searches = 0;

  static double extent(const DVol &v) {
    if (v.kind == kBox) return v.p[0] + v.p[1] + v.p[2];
    if (v.kind == kOrb) return v.p[0];
    if (v.kind == kCone) return std::fabs(v.p[3]) + std::fabs(v.p[2]) * v.p[4] + v.p[4];
    return v.p[1] + v.p[2];
  }

  // The plane d = a lx + b ly + k of volume i's local coordinates, in the world.
  PSurf line(int i, double a, double b, double k, int face) const {
    const DWorld &w = g.wxf[i];
    PSurf s;
    s.type = kLine;
    s.nx = a * w.c - b * w.s;
    s.ny = a * w.s + b * w.c;
    s.o = k - s.nx * w.tx - s.ny * w.ty;
    s.face = face;
    return s;
  }

  void volume_surfaces(int i) {
    const DVol &v = g.vol[i];
    const DWorld &w = g.wxf[i];
    std::vector<PSurf> &S = surfs[i];
    auto zplane = [&](double n, double hz, int face) {
      PSurf s;
      s.nx = n;
      s.o = hz - n * w.tz;
      s.face = face;
      S.push_back(s);
    };
    auto round = [&](int type, double R, int sign, int face) {
      PSurf s;
      s.type = type;
      s.cx = w.tx;
      s.cy = w.ty;
      s.cz = w.tz;
      s.R = R;
      s.sign = sign;
      s.face = face;
      S.push_back(s);
    };
    if (v.kind == kBox) {
      S.push_back(line(i, 1.0, 0.0, v.p[0], 0));
      S.push_back(line(i, -1.0, 0.0, v.p[0], 1));
      S.push_back(line(i, 0.0, 1.0, v.p[1], 2));
      S.push_back(line(i, 0.0, -1.0, v.p[1], 3));
      zplane(1.0, v.p[2], 4);
      zplane(-1.0, v.p[2], 5);
    } else if (v.kind == kOrb) {
      round(kSphere, v.p[0], 1, 0);
    } else if (v.kind == kTube) {
      zplane(1.0, v.p[2], 0);
      zplane(-1.0, v.p[2], 1);
      round(kCircle, v.p[1], 1, 2);
      if (v.flags & kHasRmin) round(kCircle, v.p[0], -1, 3);
      if (v.flags & kSeg) {
        S.push_back(line(i, -v.p[4], v.p[3], 0.0, 4));
        S.push_back(line(i, v.p[6], -v.p[5], 0.0, 5));
      }
    } else {   // a cone: its bounding tube, only ever used to be outside of
      zplane(1.0, v.p[4], 0);
      zplane(-1.0, v.p[4], 1);
      round(kCircle, std::max(v.p[3] - v.p[2] * v.p[4], v.p[3] + v.p[2] * v.p[4]), 1, 2);
    }
  }

  bool patch_of(int V, int face, PPatch &P) const {
    const DVol &v = g.vol[V];
    const DWorld &w = g.wxf[V];
    auto point = [&](double lx, double ly) {
      P.px[P.n] = w.tx + w.c * lx - w.s * ly;
      P.py[P.n] = w.ty + w.s * lx + w.c * ly;
      ++P.n;
    };
    if (v.kind == kBox) {
      const double x = v.p[0], y = v.p[1];
      if (face == 0 || face == 1) {
        point(face ? x : -x, -y);
        point(face ? x : -x, y);
      } else if (face == 2 || face == 3) {
        point(-x, face == 3 ? y : -y);
        point(x, face == 3 ? y : -y);
      } else {
        point(-x, -y);
        point(x, -y);
        point(x, y);
        point(-x, y);
      }
      P.zlo = w.tz + (face == 5 ? v.p[2] : -v.p[2]);
      P.zhi = w.tz + (face == 4 ? -v.p[2] : v.p[2]);
      return true;
    }
    P.cx = w.tx;
    P.cy = w.ty;
    if (v.kind == kOrb) {
      P.kind = PPatch::kBall;
      P.r1 = v.p[0];
      P.zlo = w.tz - v.p[0];
      P.zhi = w.tz + v.p[0];
      return true;
    }
    const double turn = std::atan2(w.s, w.c);
    P.a0 = turn;
    P.a1 = turn + 2.0 * kPi;
    if (v.flags & kSeg) {
      const double a = std::atan2(v.p[4], v.p[3]);
      double d = std::atan2(v.p[6], v.p[5]) - a;
      while (d <= 0.0) d += 2.0 * kPi;
      P.a0 = turn + a;
      P.a1 = P.a0 + d;
    }
    for (int a = 0; a < 2; ++a) {
      P.c[a] = std::cos(a ? P.a1 : P.a0);
      P.s[a] = std::sin(a ? P.a1 : P.a0);
    }
    P.r0 = (v.flags & kHasRmin) ? v.p[0] : 0.0;
    P.r1 = v.p[1];
    P.zlo = w.tz - v.p[2];
    P.zhi = w.tz + v.p[2];
    if (face < 2) {
      P.kind = PPatch::kSector;
      P.zlo = P.zhi = w.tz + (face ? v.p[2] : -v.p[2]);
    } else if (face < 4) {
      P.kind = PPatch::kArc;
      if (face == 3) P.r1 = P.r0;
    } else {
      const double a = face == 4 ? std::atan2(v.p[4], v.p[3]) : std::atan2(v.p[6], v.p[5]);
      point(P.r0 * std::cos(a), P.r0 * std::sin(a));
      point(P.r1 * std::cos(a), P.r1 * std::sin(a));
    }
    return true;
  }

  // +1: the same surface with the same inside, -1: with the opposite inside, 0: not the same surface (within eps).
  int coincide(const PSurf &a, const PSurf &b) const {
    if (a.type != b.type) return 0;
    if (a.type == kZPlane) {
      if (std::fabs(a.o * a.nx - b.o * b.nx) > eps) return 0;
      return a.nx * b.nx > 0.0 ? 1 : -1;
    }
    if (a.type == kLine) {
      for (int s : {1, -1})
        if ((std::fabs(a.nx - s * b.nx) + std::fabs(a.ny - s * b.ny)) * scale + std::fabs(a.o - s * b.o) <= eps) return s;
      return 0;
    }
    if (std::fabs(a.cx - b.cx) + std::fabs(a.cy - b.cy) + std::fabs(a.R - b.R) > eps) return 0;
    if (a.type == kSphere && std::fabs(a.cz - b.cz) > eps) return 0;
    return a.sign == b.sign ? 1 : -1;
  }

  PRange range(const PSurf &s, const PPatch &P) const {
    PRange r;
    if (s.type == kZPlane) {
      r.add(s.nx * P.zlo + s.o);
      r.add(s.nx * P.zhi + s.o);
      return r;
    }
    if (s.type == kLine) return range_linear(P, s.nx, s.ny, s.o);
    PRange d = range_distance(P, s.cx, s.cy);
    if (s.type == kSphere) {
      const double zmin = std::max(0.0, std::max(P.zlo - s.cz, s.cz - P.zhi));
      const double zmax = std::max(std::fabs(P.zlo - s.cz), std::fabs(P.zhi - s.cz));
      d.lo = length(d.lo, zmin);
      d.hi = length(d.hi, zmax);
    }
    r.add(s.sign * (s.R - d.lo));
    r.add(s.sign * (s.R - d.hi));
    return r;
  }

  // Inside of volume W over V's face (surface f, patch P) for rays crossing it outward (dir +1) or inward (-1): 1, 0, or
  // -1 if not decided.
  int inside(int W, int V, const PSurf &f, const PPatch &P, int dir) const {
    if (W == V) return dir < 0 ? 1 : 0;   // the crossing points lie on its face, away from its other surfaces
    const DVol &w = g.vol[W];
    const bool wide = w.kind == kTube && (w.flags & kWide), v_wide = g.vol[V].kind == kTube && (g.vol[V].flags & kWide);
    // most volumes lie beyond a plane of theirs (that no face of V coincides with: outside all the same if one does)
    for (const PSurf &s : surfs[W])
      if ((s.type == kZPlane || (s.type == kLine && !wide)) && range(s, P).hi < -margin) return 0;
    bool all = w.kind != kCone;
    int phi_in = 0, phi_out = 0;
    for (const PSurf &s : surfs[W]) {
      int in = -1;
      const int same = coincide(s, f);
      if (same) {
        in = same == dir ? 0 : 1;   // crossed outward (leaving W) or inward
      } else {
        for (const PSurf &h : surfs[V]) {
          if (h.face == f.face) continue;
          // beside a wide segment's face only one of its phi planes is certain to be away
          if (v_wide && h.type == kLine) continue;
          const int rel = coincide(s, h);
          if (rel) {
            in = rel > 0 ? 1 : 0;
            break;
          }
        }
        if (in < 0) {
          const PRange r = range(s, P);
          if (r.lo > margin) in = 1;
          else if (r.hi < -margin) in = 0;
        }
      }
      if (wide && s.type == kLine) {   // the union of the two half-planes
        phi_in += in == 1 && !same;
        phi_out += in == 0 && !same;
      } else {
        if (in == 0) return 0;
        if (in < 0) all = false;
      }
    }
    if (wide) {
      if (phi_out == 2) return 0;
      if (phi_in == 0) all = false;
    }
    return all ? 1 : -1;
  }

  // The candidate lists of the nodes of header h that the box lo .. hi reaches, while they list fewer than `most` in all.
  void collect(int32_t h, const double *lo, const double *hi, size_t most, size_t &listed) {
    const DVoxHdr &H = g.hdr[h];
    const int n = H.nslices;
    const long k0 = std::max(0L, std::min((long)n - 1, (long)std::floor((lo[H.axis] - H.lo) * H.inv_width - 1e-6)));
    const long k1 = std::max(0L, std::min((long)n - 1, (long)std::floor((hi[H.axis] - H.lo) * H.inv_width + 1e-6)));
    for (long k = k0; k <= k1 && listed < most; ++k) {
      const DVoxSlice &S = g.slice[H.slice_base + k];
      if (k > k0 && S.k0 < k) continue;   // a merged node, already taken
      if (S.child < 0) {
        collect(-S.child - 1, lo, hi, most, listed);
      } else if (list_seen[S.child] != searches) {
        list_seen[S.child] = searches;
        lists.push_back(S.child);
        listed += g.clist[S.child].count;
      }
    }
  }

  bool search(int V, const PSurf &f, const PPatch &P, int dir, int &leaf) {
    int blocked = dir > 0 ? V : -1, cur = g.vol[V].mother;
    while (cur >= 0) {
      const int in = inside(cur, V, f, P, dir);
      if (in < 0) return false;
      if (in == 1) break;
      blocked = cur;
      cur = g.vol[cur].mother;
    }
    if (cur < 0) {
      leaf = -1;
      return true;
    }
    for (int lev = 0; lev < kDMax && g.vol[cur].vox >= 0; ++lev) {
      // the daughters whose voxel nodes and boxes the face can reach, in id order
      const DWorld &w = g.wxf[cur];
      const PRange x = range_linear(P, w.c, w.s, -w.c * w.tx - w.s * w.ty), y = range_linear(P, -w.s, w.c, w.s * w.tx - w.c * w.ty);
      const double sl = margin;
      const double lo[3] = {x.lo - sl, y.lo - sl, P.zlo - w.tz - sl}, hi[3] = {x.hi + sl, y.hi + sl, P.zhi - w.tz + sl};
      auto reached = [&](int32_t d) {
        const DBox32 &B = g.box[d];
        for (int b = 0; b < 3; ++b)
          if ((double)B.hi[b] < lo[b] || (double)B.lo[b] > hi[b]) return false;
        return d != blocked;
      };
      lists.clear();
      cands.clear();
      ++searches;
      size_t listed = 0;
      collect(g.vol[cur].vox, lo, hi, daughters[cur].size(), listed);
      if (listed >= daughters[cur].size()) {
        // a face that large meets daughters again node after node: each once, then (600 shells about one axis: 7.5 s of finalize -> .5)
        for (int32_t d : daughters[cur])
          if (reached(d)) cands.push_back(d);
      } else {
        for (int32_t l : lists) {
          const DCandList &cl = g.clist[l];
          for (int32_t q = 0; q < cl.count; ++q) {
            const int32_t d = g.cand[cl.offset + q];
            if (cand_seen[d] == searches) continue;
            cand_seen[d] = searches;
            if (reached(d)) cands.push_back(d);
          }
        }
        std::sort(cands.begin(), cands.end());
      }
      int found = -1;
      for (int32_t d : cands) {
        const int in = inside(d, V, f, P, dir);
        if (in < 0) return false;
        if (in == 1) {
          found = d;
          break;
        }
      }
      if (found < 0) break;
      cur = found;
      blocked = -1;
    }
    leaf = cur;
    return true;
  }
};

}  // namespace g4n
