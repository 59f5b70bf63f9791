// Free directions: per face, the azimuth sectors and elevation bands in which
// any other geometry may stand, so that rays which leave the face through an
// empty cell are known to hit nothing without a traversal (after Max, "Horizon
// mapping: shadows for bump-mapped surfaces", The Visual Computer 1988; here
// cells that bound all of the mesh as seen from all of the face, instead of one
// sampled height per azimuth).
//
// For a face f (unit normal n on the surface's outer side, MeshStat::winding;
// in-plane axes T along the first edge and B = n x T) a cell is one of eight
// 45-degree sectors of azimuth, each widened by HZ_WIDEN on both sides, times one
// of 16 bands of the sine of elevation above HZ_FLOOR (hz_band). A cell is marked when x - y
// may fall into it for some point x of another face and some y of f. Below
// HZ_FLOOR nothing is free. The 128 bits are a uint4 per face. Sources of marks:
//  - the nodes of the 4-wide tree, each with a centre, a radius, an axis (its
//    faces' mean normal) and the extents along it (k_hz_nodes): the extents bound
//    the height over f's plane far better than the box where the surface is
//    smooth, since a flat patch is thin along its own normal. A node marks the
//    elevations of its sphere, up to (highest point) / (least horizontal
//    distance).
//  - the triangles near f with the least of several bounds: for a direction m
//    with m.(y - s) <= 0 on f (s on f's border) the horizontal distance of x and y
//    is at least m.(x - s), and height / m.(x - s) is a ratio of linear functions,
//    largest at the triangle's vertices. m runs over f's edge normals and their
//    bisectors at f's vertices, which bounds faces that share an edge or a vertex
//    with f by their slope.
//    Needles (HZ_THIN) take the sphere instead.
// k_horizon gives every face a warp, whose lanes take the children of eight nodes
// at a time: those of f's ancestors, nearest first, then what they open. A node
// whose cells are all marked already, or that is below f's plane, is dropped; one
// that is small as seen from f (HZ_FAR) marks its cells; the others are opened.
//
// What the test has to allow for (hz_free): the ray starts off f by a vector e
// (measured at run time), and the watertight test may report a hit eta beside a
// triangle (rounding, 1e-6 of the longest edge). A hit at t >= T_EPS along d is
// then seen from f along t d + e + eta: with rho = (|e| + eta) / T_EPS and e_n the
// part of e along n, its sine of elevation is at least (d_n - (eta - e_n) / T_EPS)
// / (1 + rho) (e_n < 0) and at most (d_n + (eta + e_n) / T_EPS) / (1 - rho) (e_n >
// 0), its azimuth off by up to asin((rho + HZ_TILT) / |d_h|), which the widened
// sectors cover up to HZ_WIDEN; past that every sector counts. A ray in the plane of a neighbour that
// runs off its far side can still be given a false hit (the neighbour's projection
// is a line through the origin, its weights are rounding, and t any depth of its
// vertices): p is then within (|e| + eta) / d_n of the shared edge, so a direction
// must also be steeper than (|e| + eta) / w, w the distance of p to f's nearest edge.
// (Of 6 10^8 sampled free rays, half from within 10^-5 of an edge's length of it, one
// had such a hit without this. With it: none of 3.4 10^9 over twelve meshes about the
// origin, and of 10^10 rays past one neighbour, coordinates up to 10^4 and faces from
// 10^-3 to 5, with and without fused products, no free one hit. 13,700 calls with and
// without them gave the same images, path signatures and ray counts bitwise, 5,000
// adjoints the same gradients up to the atomics' order: spheres, fractal ones, torus
// knots and planes, moved up to 700, scaled from 0.01 to 3, refitted and rebuilt.)
//
// Measured on one GB300. k_horizon is bounded by instruction issue (70 % active, 23
// warps per SM, 15 of 32 lanes at 200k faces: nodes and triangles of a round take
// different loads): 1.6 ms at 200k smooth faces (12 rounds a face), 0.8 ms at the 50k-face torus
// knot (24), 16.8 ms at 1M rough ones (25). k_hz_nodes 0.02 to 0.2 ms. Share of the
// NEE and bounce rays answered: 99 % on the smooth spheres, 53 % on the knot, 80 % on
// the rough mesh. Of an iteration on 200k faces and 64 views, k_extend and k_shadow
// fell from 45.1 to 18.3 ms of kernel time, the iteration from 57.0 to 36.7 ms; one of
// 1M rough faces and 8 views took 154 and takes 133 ms. (Those with the lowest band's
// floor at 0.02; at 0.003, which answers grazing rays of gentle surfaces too, the
// 200k-face iteration went from 31.4 to 30.0, one of 32 captures lit from the camera
// from 5.76 to 5.29, both on the later kernels.)
#pragma once
#include <cmath>

#include "st_internal.h"
#include "st_trace.cuh"

namespace st {

constexpr float HZ_WIDEN = 0.1f;      // radians added to each side of a sector
constexpr float HZ_SIN = 0.0998f;     // its sine, rounded down: what an uncertain azimuth may be off by
constexpr float HZ_TILT = 4e-4f;      // a direction's offset from the rounding of a face's normal (slivers up to hz_face's limit)
constexpr float HZ_RHO = 4.0f;        // largest rho for which the directions are used
constexpr float HZ_MARGIN = 0.003f;   // constant part of the elevation margin (rounding of the frames)
constexpr float HZ_FLOOR = 0.003f;    // sine of elevation below which nothing is free
constexpr float HZ_LOW = 0.02f;       // upper end of the lowest band: what a gentle surface's neighbours reach
constexpr float HZ_THIN = 1.0f / 256;   // twice the area over the longest edge squared up to which a triangle is a needle
constexpr int HZ_FEW = 1;             // cells not marked yet up to which a node is taken by its sphere too
constexpr float HZ_FAR = 0.2f;        // radius over distance of a node (or triangle) taken by its sphere
constexpr int HZ_WARPS = 8;           // warps (faces) of a k_horizon block
constexpr int HZ_STACK = 96;          // nodes waiting to be opened; one past them marks its cells
constexpr int HZ_OPEN = 512;          // nodes opened per face, likewise

// position of a sine of elevation among the 16 bands: [HZ_FLOOR, HZ_LOW), then 15 of equal width up to 1
__host__ __device__ __forceinline__ float hz_band(float s) {
  return s < HZ_LOW ? (s - HZ_FLOOR) * (1.0f / (HZ_LOW - HZ_FLOOR)) : 1.0f + (s - HZ_LOW) * (15.0f / (1.0f - HZ_LOW));
}

// Normals of the sector borders (directions 45 k -+ HZ_WIDEN, k = 0..3) and the sector axes (22.5 + 45 k).
struct HzLines {
  float bx[8], by[8], cx[4], cy[4];
};
__host__ __device__ constexpr HzLines hz_lines() {
  // cos and sin of 45 k degrees and of HZ_WIDEN, combined by the addition theorems
  const float c45[4] = {1.0f, 0.70710678f, 0.0f, -0.70710678f}, s45[4] = {0.0f, 0.70710678f, 1.0f, 0.70710678f};
  const float cw = 0.99500417f, sw = 0.09983342f, c22 = 0.92387953f, s22 = 0.38268343f;
  HzLines l{};
  for (int k = 0; k < 4; ++k) {
    // directions at 45 k - w and 45 k + w; their normals point counter-clockwise
    float cm = c45[k] * cw + s45[k] * sw, sm = s45[k] * cw - c45[k] * sw;
    float cp = c45[k] * cw - s45[k] * sw, sp = s45[k] * cw + c45[k] * sw;
    l.bx[2 * k] = -sm; l.by[2 * k] = cm;
    l.bx[2 * k + 1] = -sp; l.by[2 * k + 1] = cp;
    l.cx[k] = c45[k] * c22 - s45[k] * s22; l.cy[k] = s45[k] * c22 + c45[k] * s22;
  }
  return l;
}

// Sectors that hold some w whose products with the border normals and axes lie in [lo, hi].
__host__ __device__ __forceinline__ unsigned hz_sectors(const float (&blo)[8], const float (&bhi)[8], const float (&clo)[4],
                                               const float (&chi)[4], float tiny) {
  unsigned m = 0;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int k = s & 3, e = (s + 1) & 3;
    // counter-clockwise of 45 s - w, clockwise of 45 (s + 1) + w, on the axis' side
    bool a = s < 4 ? bhi[2 * k] > 0.0f : blo[2 * k] < 0.0f;
    bool b = (s + 1 < 4 || s == 7) ? blo[2 * e + 1] < 0.0f : bhi[2 * e + 1] > 0.0f;
    bool c = s < 4 ? chi[k] > tiny : clo[k] < -tiny;
    if (a && b && c) m |= 1u << s;
  }
  return m;
}

// Square root to a few units in the last place (0 for what rounding left below it): the bounds built from it carry
// wider margins (1e-5 relative).
__host__ __device__ __forceinline__ float hz_sqrt(float x) {
  x = fmaxf(x, 1e-30f);
  return x * rsqrtf(x);
}

// a / b to a few units in the last place
__host__ __device__ __forceinline__ float hz_div(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fdividef(a, b);
#else
  return a / b;
#endif
}

// arctangent of y / x over the full circle within 4e-3 rad (Rajan et al., "Efficient approximations for the
// arctangent function", IEEE Signal Processing Magazine 2006, eq. 5: pi/4 t + 0.273 t (1 - t) on [0, 1])
__host__ __device__ __forceinline__ float hz_atan2(float y, float x) {
  const float ax = fabsf(x), ay = fabsf(y), t = hz_div(fminf(ax, ay), fmaxf(fmaxf(ax, ay), 1e-30f));
  float a = t * (1.05839816f - 0.273f * t);   // pi / 4 + 0.273
  if (ay > ax) a = 1.57079633f - a;
  if (x < 0.0f) a = PI_F - a;
  return y < 0.0f ? -a : a;
}

// Record of a 4-wide node: (centre, radius), (axis, largest extent along it), (least extent, 0, 0, 0).
struct HzNode {
  float3 c, a;
  float R, smax, smin;
};
__device__ __forceinline__ HzNode hz_load(const float4* N, int i) {
  float4 q0 = __ldcg(&N[3 * i]), q1 = __ldcg(&N[3 * i + 1]), q2 = __ldcg(&N[3 * i + 2]);
  return HzNode{xyz(q0), xyz(q1), q0.w, q1.w, q2.x};
}
// largest n.(x - c) over the node (n a unit vector)
__device__ __forceinline__ float hz_support(const HzNode& q, float3 n) {
  float ct = dot3(q.a, n), st = hz_sqrt(1.0f - ct * ct) + 5e-4f;   // the square root's rounding near 1
  return fminf(q.R, (ct >= 0.0f ? ct * q.smax : ct * q.smin) + st * q.R);
}

// Raises ms->eta (zeroed before) to 1e-6 of the mesh's longest edge, for what uses the cells. Part of the build, since only
// that needs it: in the mesh facts of every vertex update an atomic a warp cost 4 us of a 65k-face refit.
constexpr int HZ_EDGE_BLOCK = 256;
__global__ void __launch_bounds__(HZ_EDGE_BLOCK) k_longest_edge(const float4* __restrict__ tri, int nf, MeshStat* ms) {
  __shared__ float part[HZ_EDGE_BLOCK / 32];
  float l2 = 0.0f;
  for (int i = blockIdx.x * HZ_EDGE_BLOCK + threadIdx.x; i < nf; i += gridDim.x * HZ_EDGE_BLOCK) {
    const float3 a = xyz(tri[3 * i]), b = xyz(tri[3 * i + 1]) - a, c = xyz(tri[3 * i + 2]) - a, d = c - b;
    l2 = fmaxf(l2, fmaxf(dot3(b, b), fmaxf(dot3(c, c), dot3(d, d))));
  }
  for (int o = 16; o > 0; o >>= 1) l2 = fmaxf(l2, __shfl_xor_sync(0xffffffffu, l2, o));
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = l2;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (float x : part) l2 = fmaxf(l2, x);
  atomicMax(reinterpret_cast<int*>(&ms->eta), __float_as_int(1e-6f * sqrtf(l2)));   // not negative: ordered as its bits
}

// The records, bottom-up in one launch: the threads of nodes without internal children start, and the last child
// to finish takes its parent (done: zeroed counters).
__global__ void k_hz_nodes(const float4* __restrict__ nodes, const float4* __restrict__ tri, const int* parent, int n4,
                           int nf, const MeshStat* ms, float4* N, int* done, int* err) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n4) return;
  const float side = ms->winding < 0 ? -1.0f : 1.0f;
  auto links = [&](int i, int (&c)[4]) {
    float4 ch = __ldg(nodes + 7 * i + 6);
    c[0] = __float_as_int(ch.x); c[1] = __float_as_int(ch.y); c[2] = __float_as_int(ch.z); c[3] = __float_as_int(ch.w);
    return (c[0] >= 0) + (c[1] >= 0) + (c[2] >= 0) + (c[3] >= 0);
  };
  int c[4];
  if (links(k, c) != 0) return;
  for (int depth = 0; depth < 64; ++depth) {
    const int EMPTY = (int)0x80000000;
    float4 lx = __ldg(nodes + 7 * k), hx = __ldg(nodes + 7 * k + 1), ly = __ldg(nodes + 7 * k + 2),
           hy = __ldg(nodes + 7 * k + 3), lz = __ldg(nodes + 7 * k + 4), hz = __ldg(nodes + 7 * k + 5);
    // empty children hold (1e30, -1e30) boxes, which the extrema pass over
    float3 lo = mk3(fminf(fminf(lx.x, lx.y), fminf(lx.z, lx.w)), fminf(fminf(ly.x, ly.y), fminf(ly.z, ly.w)),
                    fminf(fminf(lz.x, lz.y), fminf(lz.z, lz.w)));
    float3 hi = mk3(fmaxf(fmaxf(hx.x, hx.y), fmaxf(hx.z, hx.w)), fmaxf(fmaxf(hy.x, hy.y), fmaxf(hy.z, hy.w)),
                    fmaxf(fmaxf(hz.x, hz.y), fmaxf(hz.z, hz.w)));
    HzNode q, ch[4];
    q.c = (lo + hi) * 0.5f;
    float3 sum = mk3(0, 0, 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (c[j] == EMPTY || (c[j] < 0 && (unsigned)~c[j] >= (unsigned)nf) || c[j] >= n4) continue;
      if (c[j] >= 0) {
        ch[j] = hz_load(N, c[j]);
        sum += ch[j].a * (ch[j].R * ch[j].R);
      } else {
        const int l = ~c[j];
        float3 p0 = xyz(tri[3 * l]), m = cross3(xyz(tri[3 * l + 1]) - p0, xyz(tri[3 * l + 2]) - p0);
        sum += m * (0.5f * side);
      }
    }
    float sl = len3(sum);
    q.a = sl > 0.0f ? sum * (1.0f / sl) : mk3(0, 0, 1);
    float r = 0.0f, smax = -3.4e38f, smin = 3.4e38f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (c[j] == EMPTY || (c[j] < 0 && (unsigned)~c[j] >= (unsigned)nf) || c[j] >= n4) continue;
      if (c[j] >= 0) {
        float3 d = ch[j].c - q.c;
        float da = dot3(d, q.a);
        r = fmaxf(r, len3(d) + ch[j].R);
        smax = fmaxf(smax, da + hz_support(ch[j], q.a));
        smin = fminf(smin, da - hz_support(ch[j], -q.a));
      } else {
        const int l = ~c[j];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          float3 d = xyz(tri[3 * l + i]) - q.c;
          float da = dot3(d, q.a);
          r = fmaxf(r, len3(d));
          smax = fmaxf(smax, da);
          smin = fminf(smin, da);
        }
      }
    }
    const float3 up = hi - q.c, dn = q.c - lo;   // the centre is rounded: the box's corners are as far as this from it
    q.R = fminf(r, len3(mk3(fmaxf(up.x, dn.x), fmaxf(up.y, dn.y), fmaxf(up.z, dn.z)))) * 1.00001f;
    q.smax = fminf(smax, q.R);
    q.smin = fmaxf(smin, -q.R);
    __stcg(&N[3 * k], make_float4(q.c.x, q.c.y, q.c.z, q.R));
    __stcg(&N[3 * k + 1], make_float4(q.a.x, q.a.y, q.a.z, q.smax));
    __stcg(&N[3 * k + 2], make_float4(q.smin, 0.0f, 0.0f, 0.0f));
    __threadfence();
    const int p = parent[k];
    if (p < 0) return;
    if (p >= n4) { atomicOr(err, ERR_LOOP); return; }
    const int need = links(p, c);
    if (atomicAdd(&done[p], 1) != need - 1) return;
    __threadfence();
    k = p;
  }
  atomicOr(err, ERR_LOOP);
}

// A face as its directions are seen from: frame, centre and radius. Positions are taken from the vertex v0 (c too): near
// the face such differences of floats are exact or nearly so, wherever it lies, while a centroid of absolute coordinates
// is off by an ulp of these, which on a small face far from the origin is more than what its neighbours rise by.
struct HzFace {
  float3 v0, v1, v2, n, T, B, c;
  float r, tiny;
};
// False on a sliver, whose normal and borders are not known well enough: nothing is free on it.
__host__ __device__ __forceinline__ bool hz_face(float3 v0, float3 v1, float3 v2, float side, HzFace& f) {
  const float3 e1 = v1 - v0, e2 = v2 - v0;
  const float3 m = cross3(e1, e2);
  const float l1 = len3(e1), l2 = len3(e2), l3 = len3(v2 - v1), ml = len3(m);
  const float lmax = fmaxf(l1, fmaxf(l2, l3));
  if (!(ml > 1e-3f * lmax * lmax) || !(l1 > 1e-3f * lmax)) return false;
  f.v0 = v0; f.v1 = v1; f.v2 = v2;
  f.n = m * (side / ml);
  f.T = e1 * (1.0f / l1);
  f.B = cross3(f.n, f.T);
  f.c = (e1 + e2) * (1.0f / 3.0f);
  f.r = fmaxf(len3(f.c), fmaxf(len3(e1 - f.c), len3(e2 - f.c)));
  f.tiny = 1e-6f * fminf(lmax, 1.0f);
  return true;
}
// f in its plane: the border lines (mx, my, mo) of vertex k (0 .. 2), m the outward normal (f runs clockwise about n
// when side < 0) of the edge that starts there (line k) and its bisector with the edge that ends there (line 3 + k).
__host__ __device__ __forceinline__ void hz_border(const HzFace& f, float side, int k, float* ln) {
  auto in2 = [&](int i) { float3 d = (i == 0 ? f.v0 : i == 1 ? f.v1 : f.v2) - f.v0; return make_float2(dot3(d, f.T), dot3(d, f.B)); };
  const float2 p0 = in2(k), p1 = in2(k == 2 ? 0 : k + 1), p2 = in2(k == 0 ? 2 : k - 1);
  auto normal = [&](float2 a, float2 b) {
    float dx = b.x - a.x, dy = b.y - a.y, il = side / sqrtf(dx * dx + dy * dy);
    return make_float2(dy * il, -dx * il);
  };
  const float2 m0 = normal(p0, p1), m1 = normal(p2, p0);   // of the edges that start and end at vertex k
  ln[k] = m0.x; ln[6 + k] = m0.y;
  const auto out = [&](float mx, float my) {   // the least mo with m.y <= mo on all of f
    return fmaxf(mx * p0.x + my * p0.y, fmaxf(mx * p1.x + my * p1.y, mx * p2.x + my * p2.y));
  };
  ln[12 + k] = out(m0.x, m0.y);
  const float sx = m0.x + m1.x, sy = m0.y + m1.y, il = rsqrtf(fmaxf(sx * sx + sy * sy, 1e-12f));
  ln[3 + k] = sx * il; ln[9 + k] = sy * il;
  ln[15 + k] = out(sx * il, sy * il);
}

// Marked cells: sector 2 w in the low half of word w, 2 w + 1 in the high.
struct HzCells { unsigned w[4]; };
// the cells of elevations lo .. hi in the sectors sec
__host__ __device__ __forceinline__ HzCells hz_cells(unsigned sec, float lo, float hi) {
  HzCells c;
  int b0 = (int)floorf(hz_band(lo) - 1e-3f), b1 = (int)floorf(hz_band(hi) + 1e-3f);
  b0 = b0 > 0 ? b0 : 0;
  b1 = b1 < 15 ? b1 : 15;
  unsigned m = b1 >= b0 ? (2u << b1) - (1u << b0) : 0u;
#pragma unroll
  for (int w = 0; w < 4; ++w) c.w[w] = (sec >> (2 * w) & 1u ? m : 0u) | (sec >> (2 * w + 1) & 1u ? m << 16 : 0u);
  return c;
}
// cells of points within r of f's centre + v, at most hb high; far: small enough to be taken so
__host__ __device__ __forceinline__ HzCells hz_sphere(const HzFace& f, float3 v, float r, float hb, bool& far) {
  const float d2 = dot3(v, v), vn = dot3(v, f.n), vx = dot3(v, f.T), vy = dot3(v, f.B);
  unsigned sec = 0xffu;
  float lo = -1.0f, hi = 1.0f;
  far = false;
  if (r * r < d2) {
    const float iv = rsqrtf(d2), sv = vn * iv, sr = r * iv, cv = hz_sqrt(1.0f - sv * sv),
                cr = hz_sqrt(1.0f - sr * sr);
    if (cv >= sr || sv < 0.0f) hi = sv * cr + cv * sr + 1e-4f;
    if (cv >= sr || sv > 0.0f) lo = sv * cr - cv * sr - 1e-4f;
    const float D = hz_sqrt(vx * vx + vy * vy) * 0.99999f - r;
    if (D > 0.0f) {
      hi = fminf(hi, hb * rsqrtf(D * D + hb * hb) * 1.00001f);
      // azimuth of the centre and of its disk, in sectors: asin x <= x + (pi / 2 - 1) x^3 on [0, 1]
      const float x = hz_div(r, D + r), a = hz_atan2(vy, vx) * (4.0f / PI_F),
                  w = (x + 0.5708f * x * x * x + HZ_WIDEN + 5e-3f) * (4.0f / PI_F);
      const int s0 = (int)floorf(a - w), n = (int)floorf(a + w) - s0 + 1;
      if (n < 8) {
        const unsigned m = (1u << n) - 1u, t = (unsigned)s0 & 7u;
        sec = (m << t | m >> (8u - t)) & 0xffu;
      }
    }
    far = sr < HZ_FAR;
  }
  return hz_cells(sec, lo, hi);
}
// A triangle's sphere about its own centre (v from f's) and how high it reaches over f's plane; true when it may have the
// finer bound. A needle may not: the watertight test's depth on it is off by the rounding of its height over its length,
// and from a vertex that it touches it may be reported past T_EPS in any direction. Near f its sphere marks every cell.
__host__ __device__ __forceinline__ bool hz_leaf(const HzFace& f, float3 x0, float3 x1, float3 x2, float3& v, float& r,
                                                 float& hb) {
  const float3 q0 = x0 - f.v0, q1 = x1 - f.v0, q2 = x2 - f.v0, c = (q0 + q1 + q2) * (1.0f / 3.0f);
  v = c - f.c;
  r = hz_sqrt(fmaxf(dot3(q0 - c, q0 - c), fmaxf(dot3(q1 - c, q1 - c), dot3(q2 - c, q2 - c))));
  hb = fmaxf(dot3(q0, f.n), fmaxf(dot3(q1, f.n), dot3(q2, f.n)));
  const float3 e1 = q1 - q0, e2 = q2 - q0, m = cross3(e1, e2), e3 = q2 - q1;
  const float l2 = fmaxf(dot3(e1, e1), fmaxf(dot3(e2, e2), dot3(e3, e3)));
  const bool thin = !(dot3(m, m) > HZ_THIN * HZ_THIN * l2 * l2);
  if (thin) hb += HZ_THIN * (r + f.r);
  return !thin;
}
// what a child's bound is widened by, for rounding: height and radius
__host__ __device__ __forceinline__ float hz_slack(const HzFace& f, float3 v, float r) {
  return 1e-6f * (fabsf(v.x) + fabsf(v.y) + fabsf(v.z) + r + f.r);
}
// the finer bound of a triangle near f
__host__ __device__ __forceinline__ HzCells hz_fine(const HzFace& f, const float* ln, float3 x0, float3 x1, float3 x2) {
  constexpr HzLines LN = hz_lines();
  const float3 x[3] = {x0, x1, x2};
  float X[3], Y[3], h[3];
  int sh[3];   // the vertex of f this vertex is, or -1
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    auto same = [&](float3 a) { return x[i].x == a.x && x[i].y == a.y && x[i].z == a.z; };
    sh[i] = same(f.v0) ? 0 : same(f.v1) ? 1 : same(f.v2) ? 2 : -1;
    float3 q = x[i] - f.v0;
    X[i] = dot3(q, f.T); Y[i] = dot3(q, f.B);
    h[i] = dot3(q, f.n) + 1e-6f * (fabsf(q.x) + fabsf(q.y) + fabsf(q.z));
    if (sh[i] >= 0) h[i] = 0.0f;
  }
  float best = INFINITY;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float mx = ln[k], my = ln[6 + k], mo = ln[12 + k];
    float d[3], tn = 0.0f;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      d[i] = mx * X[i] + my * Y[i] - mo - 5e-7f * (fabsf(X[i]) + fabsf(Y[i]) + 2.0f * f.r);   // less its rounding
      // a vertex of f on the border line itself
      bool on = k < 3 ? (sh[i] == k || sh[i] == (k == 2 ? 0 : k + 1)) : sh[i] == k - 3;
      if (on) d[i] = 0.0f;
      if (h[i] > 0.0f) {
        ok &= d[i] > f.tiny;
        tn = fmaxf(tn, h[i] / d[i]);
      }
    }
    // where the triangle's edges cross height 0 the distance must not be negative
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (i != j && h[i] > 0.0f && !(h[j] > 0.0f)) {
          float cr = d[j] * h[i] - d[i] * h[j];
          ok &= (sh[j] >= 0 && d[j] == 0.0f) || cr > 1e-4f * d[i] * (h[i] - h[j]);
        }
    if (ok) best = fminf(best, tn);
  }
  const float sn = best < 1e18f ? fminf(best * rsqrtf(1.0f + best * best) * 1.00001f, 1.0f) : 1.0f;
  const float3 e1 = f.v1 - f.v0, e2 = f.v2 - f.v0;
  const float fx[2] = {dot3(e1, f.T), dot3(e2, f.T)}, fy[2] = {dot3(e1, f.B), dot3(e2, f.B)};
  float blo[8], bhi[8], clo[4], chi[4];
  // products with w = x - y over the triangle's and f's vertices
  auto range = [&](float lx, float ly, float& lo, float& hi) {
    float a0 = lx * X[0] + ly * Y[0], a1 = lx * X[1] + ly * Y[1], a2 = lx * X[2] + ly * Y[2];
    float f1 = lx * fx[0] + ly * fy[0], f2 = lx * fx[1] + ly * fy[1];
    lo = fminf(a0, fminf(a1, a2)) - fmaxf(0.0f, fmaxf(f1, f2));
    hi = fmaxf(a0, fmaxf(a1, a2)) - fminf(0.0f, fminf(f1, f2));
  };
#pragma unroll
  for (int k = 0; k < 8; ++k) range(LN.bx[k], LN.by[k], blo[k], bhi[k]);
#pragma unroll
  for (int k = 0; k < 4; ++k) range(LN.cx[k], LN.cy[k], clo[k], chi[k]);
  return hz_cells(hz_sectors(blo, bhi, clo, chi, f.tiny), -1.0f, sn);
}

__global__ void __launch_bounds__(32 * HZ_WARPS, 3) k_horizon(const float4* __restrict__ nodes,
                                                           const float4* __restrict__ tri, int nf, int n4,
                                                           const MeshStat* ms, const float4* __restrict__ N,
                                                           const int* parent, const int* leaf_node, uint4* out,
                                                           int* err, int stride) {
  __shared__ int stack_[HZ_WARPS][HZ_STACK], cand_[HZ_WARPS][64];
  __shared__ float lines_[HZ_WARPS][18];   // f's border lines (mx, my, mo): the finer bound's alone, kept off the registers
  const unsigned ALL = 0xffffffffu;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  int *stack = stack_[warp], *cand = cand_[warp];
  const int place = blockIdx.x * HZ_WARPS + warp;
  const long long leaf = (long long)place * stride;   // every stride-th face, its cells one after the other
  if (leaf >= nf) return;
  const int li = (int)leaf;
  const float side = ms->winding < 0 ? -1.0f : 1.0f;
  HzFace f;
  const bool bad = !hz_face(xyz(tri[3 * li]), xyz(tri[3 * li + 1]), xyz(tri[3 * li + 2]), side, f);
  unsigned M[4] = {0u, 0u, 0u, 0u};
  if (!bad) {
    if (lane < 3) hz_border(f, side, lane, lines_[warp]);
    __syncwarp();

    auto fresh = [&](const HzCells& c) {   // cells not marked yet
      return __popc(c.w[0] & ~M[0]) + __popc(c.w[1] & ~M[1]) + __popc(c.w[2] & ~M[2]) + __popc(c.w[3] & ~M[3]);
    };
    auto mark = [&](bool on, const HzCells& c) {   // the lanes' cells enter the warp's
#pragma unroll
      for (int w = 0; w < 4; ++w) M[w] |= __reduce_or_sync(ALL, on ? c.w[w] : 0u);
    };
    // the finer bound of the triangles put aside
    auto fine = [&](int cnt) {
      HzCells cl = {{0u, 0u, 0u, 0u}};
      if (lane < cnt) {
        const int lj = cand[lane];
        cl = hz_fine(f, lines_[warp], xyz(tri[3 * lj]), xyz(tri[3 * lj + 1]), xyz(tri[3 * lj + 2]));
      }
      mark(lane < cnt, cl);
    };

    // lane groups of four take a node's children each; the first rounds go up f's ancestors, nearest first (the
    // last group takes the nearest, so that what it opens is on top of the stack)
    int sp = 0, opened = 0, nc = 0, up = n4 > 0 ? leaf_node[li] : -1, from = ~li;
    for (int round = 0;; ++round) {
      int node = -1, skip = (int)0x80000000;
      if (up >= 0) {
        for (int g = 7; g >= 0 && up >= 0; --g) {   // uniform over the warp
          if ((unsigned)up >= (unsigned)n4) { if (lane == 0) atomicOr(err, ERR_LOOP); up = -1; break; }
          if (lane >> 2 == g) { node = up; skip = from; }
          from = up;
          up = parent[up];
        }
      } else {
        const int take = min(sp, 8);
        if (lane >> 2 < take) node = stack[sp - take + (lane >> 2)];
        sp -= take;
        __syncwarp();
      }
      int ch = (int)0x80000000;
      if (node >= 0) {
        ch = __float_as_int(__ldg(reinterpret_cast<const float*>(nodes + 7 * node + 6) + (lane & 3)));
        if (ch == skip) ch = (int)0x80000000;
      }
      // the child's sphere about its own centre and how high it reaches over f's plane
      float3 v = mk3(0, 0, 0);
      float r = 0.0f, hb = -1.0f;
      bool finer = false;
      if (ch >= 0) {
        HzNode q = hz_load(N, ch);
        const float3 w = q.c - f.v0;
        v = w - f.c;
        r = q.R;
        hb = dot3(w, f.n) + hz_support(q, f.n);
      } else if (ch != (int)0x80000000 && (unsigned)~ch < (unsigned)nf) {
        finer = hz_leaf(f, xyz(tri[3 * ~ch]), xyz(tri[3 * ~ch + 1]), xyz(tri[3 * ~ch + 2]), v, r, hb);
      }
      const float slack = hz_slack(f, v, r);
      hb += slack;
      bool open = false, put = false, on = false;
      HzCells cl = {{0u, 0u, 0u, 0u}};
      if (hb > 0.0f) {
        bool far;
        cl = hz_sphere(f, v, (r + f.r) * 1.00001f + slack, hb, far);
        const int fr = fresh(cl);
        on = fr > 0;
        open = fr > HZ_FEW && !far && ch >= 0;
        put = fr > HZ_FEW && !far && finer;
      }
      const unsigned mo_ = __ballot_sync(ALL, open), mp = __ballot_sync(ALL, put);
      const int room = min(HZ_STACK - sp, HZ_OPEN - opened), at = __popc(mo_ & below), add = min(__popc(mo_), room);
      if (open && at < room) { stack[sp + at] = ch; on = false; }
      sp += add;
      opened += add;
      if (put) { cand[nc + __popc(mp & below)] = ~ch; on = false; }
      nc += __popc(mp);
      if (__any_sync(ALL, on)) mark(on, cl);
      __syncwarp();
      const bool last = sp == 0 && up < 0;
      while (nc >= 32 || (last && nc > 0)) {
        fine(min(nc, 32));
        __syncwarp();
        int v = 32 + lane < nc ? cand[32 + lane] : 0;
        __syncwarp();
        cand[lane] = v;
        nc = max(nc - 32, 0);
        __syncwarp();
      }
      if (last) break;
    }
  }
  if (lane == 0) out[place] = bad ? make_uint4(ALL, ALL, ALL, ALL) : make_uint4(M[0], M[1], M[2], M[3]);
}

// The free directions of a path vertex p on the face (v0, v1, v2) with the marked cells w; n: its unit normal turned
// toward the incoming ray (the surface's outer side). Unusable (on = false) where p lies too far off the face.
struct HzPoint {
  float3 T, B, n;
  uint4 w;
  float lo, hi, rho, irho, least;
  bool on;
};

__host__ __device__ __forceinline__ HzPoint hz_point(float eta, uint4 cells, float3 p, float3 v0, float3 v1, float3 v2,
                                                     float3 n) {
  HzPoint z;
  z.w = cells;
  float3 e1 = v1 - v0, e2 = v2 - v0, q = p - v0, m = cross3(e1, e2);
  z.n = n;
  z.T = e1 * rsqrtf(dot3(e1, e1));
  z.B = cross3(n, z.T);
  // distance of p from a point of the face: its barycentric weights, clamped to the face
  float im = 1.0f / dot3(m, m);
  const float r1 = dot3(cross3(q, e2), m) * im, r2 = dot3(cross3(e1, q), m) * im;
  float b1 = fmaxf(r1, 0.0f), b2 = fmaxf(r2, 0.0f);
  float sc = b1 + b2 > 1.0f ? 1.0f / (b1 + b2) : 1.0f;
  float3 e = q - (e1 * b1 + e2 * b2) * sc;
  float en = dot3(e, n), rho = (len3(e) + eta) * (1.0f / T_EPS);
  z.on = rho <= HZ_RHO;
  z.rho = rho;
  z.irho = 1.0f / (1.0f + rho);
  z.lo = HZ_MARGIN + (fmaxf(-en, 0.0f) + eta) * (1.0f / T_EPS);
  z.hi = HZ_MARGIN + (fmaxf(en, 0.0f) + eta) * (1.0f / T_EPS);
  // least distance to an edge: least weight times least altitude
  const float3 e3 = e2 - e1;
  const float w = fminf(fminf(r1, r2), 1.0f - r1 - r2) *
                  sqrtf(dot3(m, m) / fmaxf(dot3(e1, e1), fmaxf(dot3(e2, e2), dot3(e3, e3))));
  z.least = rho * T_EPS / w;
  z.on = z.on && w > 0.0f;
  return z;
}

// True when a ray from the vertex along the unit direction d is known to hit nothing but its own face.
__host__ __device__ __forceinline__ bool hz_free(const HzPoint& z, float3 d) {
  if (!z.on) return false;
  float dn = dot3(d, z.n), lo = hz_band((dn - z.lo) * z.irho);
  if (!(lo >= 0.0f) || !(dn > z.least)) return false;
  int b0 = (int)lo, b1 = 15;
  b0 = b0 < 15 ? b0 : 15;
  if (z.rho < 0.25f) {   // / (1 - rho)
    const int top = (int)hz_band((dn + z.hi) * (1.0f + 1.34f * z.rho));
    b1 = top < 15 ? top : 15;
  }
  unsigned band = (2u << b1) - (1u << b0), w;
  const float turn = z.rho + HZ_TILT;
  if (turn * turn > HZ_SIN * HZ_SIN * (1.0f - dn * dn)) {   // the azimuth is too uncertain
    w = z.w.x | z.w.y | z.w.z | z.w.w;
    w |= w >> 16;
  } else {
    float x = dot3(d, z.T), y = dot3(d, z.B);
    int q = y < 0.0f ? (x < 0.0f ? 2 : 3) : (x < 0.0f ? 1 : 0);   // quadrant: sectors 2 q, 2 q + 1
    w = q < 2 ? (q == 0 ? z.w.x : z.w.y) : (q == 2 ? z.w.z : z.w.w);
    if ((fabsf(y) > fabsf(x)) != ((q & 1) != 0)) w >>= 16;
  }
  return (w & band) == 0u;
}

}  // namespace st
