// Host-side check of the free directions' bounds (st_horizon.cuh), compiled and called by test_free_directions_bounds.py:
// pairs of a face and a neighbour, the cells that the neighbour marks, and rays from points of the face to points of the
// neighbour or anywhere above the face. A ray answered free that the watertight test hits is counted.
#include "../paper_2012_03939_gb300/csrc/st_horizon.cuh"

namespace {

struct Rng {   // SplitMix64
  unsigned long long s;
  unsigned long long next() {
    unsigned long long z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
  }
  double u() { return (double)(next() >> 11) * 0x1p-53; }
  double u(double a, double b) { return a + (b - a) * u(); }
  double loga(double a, double b) { return a * std::pow(b / a, u()); }
  int n(int k) { return (int)(next() % (unsigned)k); }
};

struct D3 { double x, y, z; };
using st::operator-;
using st::operator*;
D3 operator+(D3 a, D3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
D3 operator-(D3 a, D3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
D3 operator*(D3 a, double s) { return {a.x * s, a.y * s, a.z * s}; }
double dot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
D3 cross(D3 a, D3 b) { return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x}; }
D3 unit(D3 a) { return a * (1.0 / std::sqrt(dot(a, a))); }
D3 dir(Rng& r) {
  for (;;) {
    D3 d{r.u(-1, 1), r.u(-1, 1), r.u(-1, 1)};
    const double l = dot(d, d);
    if (l > 1e-3 && l <= 1.0) return unit(d);
  }
}
D3 wide(float3 a) { return {a.x, a.y, a.z}; }
float3 narrow(D3 a) { return make_float3((float)a.x, (float)a.y, (float)a.z); }

// the cells a neighbour marks on an unmarked face, as k_horizon takes a leaf
st::HzCells marks(const st::HzFace& f, const float* ln, const float3 (&x)[3]) {
  float3 v;
  float r, hb;
  const bool finer = st::hz_leaf(f, x[0], x[1], x[2], v, r, hb);
  const float slack = st::hz_slack(f, v, r);
  hb += slack;
  if (!(hb > 0.0f)) return {{0u, 0u, 0u, 0u}};
  bool far;
  st::HzCells c = st::hz_sphere(f, v, (r + f.r) * 1.00001f + slack, hb, far);
  int marked = 0;
  for (unsigned w : c.w)
    for (; w; w &= w - 1) ++marked;
  return marked > st::HZ_FEW && !far && finer ? st::hz_fine(f, ln, x[0], x[1], x[2]) : c;
}

double longest(const float3 (&a)[3]) {
  double l = 0.0;
  for (int k = 0; k < 3; ++k) {
    D3 e = wide(a[(k + 1) % 3]) - wide(a[k]);
    l = std::fmax(l, std::sqrt(dot(e, e)));
  }
  return l;
}

// what a traversal finds of the neighbour: its box, then the watertight test
bool hit(float3 p, float3 d, const float3 (&x)[3]) {
  const float3 inv = st::safe_inv(d);
  auto lo = [](float a, float b, float c) { return fminf(a, fminf(b, c)); };
  auto hi = [](float a, float b, float c) { return fmaxf(a, fmaxf(b, c)); };
  if (st::box_hit(lo(x[0].x, x[1].x, x[2].x), hi(x[0].x, x[1].x, x[2].x), lo(x[0].y, x[1].y, x[2].y),
                  hi(x[0].y, x[1].y, x[2].y), lo(x[0].z, x[1].z, x[2].z), hi(x[0].z, x[1].z, x[2].z), p, inv,
                  INFINITY) == INFINITY)
    return false;
  return st::tri_test(st::ray_pre(p, d), x[0], x[1], x[2], INFINITY) > 0.0f;
}

}  // namespace

// kind 0: the neighbour shares an edge, 1: a vertex, 2: it has a vertex on an edge of the face, 3: it stands near.
// Coordinates about `where` in magnitude, faces about `size`. out = (rays asked, rays answered free); returns the free rays
// that hit the neighbour.
extern "C" long long hz_check(unsigned long long seed, long long pairs, int rays, double where, double size, int kind,
                              long long* out) {
  Rng r{seed};
  long long wrong = 0;
  out[0] = out[1] = 0;
  for (long long i = 0; i < pairs; ++i) {
    const D3 at{r.u(-where, where), r.u(-where, where), r.u(-where, where)};
    const D3 n0 = dir(r), t0 = unit(cross(n0, dir(r))), b0 = cross(n0, t0);
    // a face of aspect 1 to 100 and a neighbour that rises little, or by any slope
    const double thin = r.n(2) ? 1.0 : r.loga(0.01, 1.0);
    auto plane = [&](double a, double b, double h) { return narrow(at + t0 * (a * size) + b0 * (b * size) + n0 * (h * size)); };
    float3 F[3] = {plane(0, 0, 0), plane(r.u(0.5, 1), r.u(-0.2, 0.2), 0), plane(r.u(-0.2, 1), thin * r.u(0.5, 1), 0)};
    const int turn = r.n(3);
    float3 f[3];
    for (int k = 0; k < 3; ++k) f[k] = F[(k + turn) % 3];
    const float side = r.n(2) ? 1.0f : -1.0f;
    const double rise = r.n(4) == 0 ? 0.0 : (r.n(8) ? 1.0 : -1.0) * r.loga(1e-8, 1.0), reach = r.loga(1e-3, 2.0);
    const double a0 = r.u(-1.5, 2.0);
    float3 x[3];
    // the edge F[0] F[1] lies along t0; the neighbour is on its other side
    const float3 apex = plane(a0, -reach, side * rise);
    if (kind == 0) { x[0] = F[1]; x[1] = F[0]; x[2] = apex; }
    if (kind == 1) { x[0] = F[0]; x[1] = plane(a0 - r.loga(1e-3, 1.0), -reach * r.u(0.0, 1.0), side * rise * r.u()); x[2] = apex; }
    if (kind == 2) {
      const double w = r.u();
      x[0] = narrow(wide(F[0]) * (1.0 - w) + wide(F[1]) * w);
      x[1] = r.n(2) ? F[0] : plane(a0 - r.loga(1e-3, 1.0), -reach * r.u(0.0, 1.0), side * rise * r.u());
      x[2] = apex;
    }
    if (kind == 3) {
      x[0] = plane(a0 + r.u(-0.3, 0.3), -reach, side * rise);
      x[1] = plane(a0 + r.u(-0.3, 0.3), -reach - r.loga(1e-3, 1.0), side * rise * r.u(0.0, 2.0));
      x[2] = plane(a0 + r.u(-0.3, 0.3), -reach * r.u(0.1, 1.0), side * rise * r.u());
    }
    st::HzFace face;
    if (!st::hz_face(f[0], f[1], f[2], side, face)) continue;
    float ln[18];
    for (int k = 0; k < 3; ++k) st::hz_border(face, side, k, ln);
    const st::HzCells c = marks(face, ln, x);
    const float eta = 1e-6f * (float)std::fmax(longest(f), longest(x));
    const float3 n = st::norm3(st::cross3(f[1] - f[0], f[2] - f[0])) * side;
    for (int k = 0; k < rays; ++k) {
      // from anywhere in the face or from near its edges, to anywhere in the neighbour or near its vertices
      auto weights = [&](double (&w)[3]) {
        const int mode = r.n(3);
        for (double& v : w) v = mode == 0 ? r.u() : r.loga(1e-7, 1.0);
        if (mode == 2) w[r.n(3)] = 1.0;
        const double s = w[0] + w[1] + w[2];
        for (double& v : w) v /= s;
      };
      double a[3], b[3];
      weights(a);
      weights(b);
      const float3 p = narrow(wide(f[0]) * a[0] + wide(f[1]) * a[1] + wide(f[2]) * a[2]);
      const D3 q = wide(x[0]) * b[0] + wide(x[1]) * b[1] + wide(x[2]) * b[2] - wide(p);
      if (!(dot(q, q) > 0.0)) continue;
      const float3 d = narrow(k & 1 ? unit(wide(n) + dir(r)) : unit(q));   // every other one anywhere above the face
      ++out[0];
      const st::HzPoint z = st::hz_point(eta, make_uint4(c.w[0], c.w[1], c.w[2], c.w[3]), p, f[0], f[1], f[2], n);
      if (!st::hz_free(z, d)) continue;
      ++out[1];
      if (hit(p, d, x)) ++wrong;
    }
  }
  return wrong;
}
