// typed.cuh -- the typed FP64 distance of a stencil at the cost of one formula.
//
// The exact routine of geometry.cuh decides a stencil's type in FP64: a face
// or line-line test, then three or four point-segment distances, some 200 to
// 270 FP64 operations.  Away from ties FP32 knows the outcome.  Each FP64
// comparison of that routine compares one of a few polynomials of the local
// coordinates with zero; certain_type evaluates the same polynomials in FP32
// and answers only if each is further from zero than its FP32 error bound, so
// that the FP64 comparison (whose error is 2^-29 of that) falls the same way.
// The distance then takes the one formula of the type: the same operations on
// the same operands, so the same bits.
//
// Bounds, with u = 2^-24, R the largest local coordinate, M the longest edge:
// coordinates are rounded by u R, differences by 4 u R a component, so a
// vector by at most 7 u R.  Hence a dot product e . w errs by less than
// 32 u R (|e| + |w|), the triangle's barycentric numerators by 256 u M R^3
// and the segments' parameter numerators by 512 u M^2 R^2.  A type that wins
// by those amounts also wins the FP64 minimum over the segments: the next
// candidate's squared distance is larger by at least (32 u R)^2 = 3.6e-12 R^2,
// while with no edge below R / 20 the FP64 values err by less than 3e-13 R^2.
// 97 % of a pleated sheet's active pairs are certain (regular meshes hold many
// parallel edges), 99.9 % of a weave's and of stacked layers'.  The additive-CCD
// iteration runs the rule at every step: 9,600 active pairs in layers 264 ->
// 106 us, 64 rod scenes with up to 236 steps 2.03 -> 0.98 ms (one lane a pair;
// 68 us and 0.5 ms with half a warp, accd16.cuh).
#pragma once
#include "bound32.cuh"
#include "geometry.cuh"

namespace cbt {

// the type (as in geometry.cuh) of a stencil with local points 0, P1, P2, P3, or -1
__device__ __forceinline__ int certain_type(bool ee, cbb::f3 P1, cbb::f3 P2, cbb::f3 P3) {
  using namespace cbb;
  const float u = 5.9604645e-8f;  // 2^-24
  const float R = fmaxf(fmaxabs3(P1), fmaxf(fmaxabs3(P2), fmaxabs3(P3)));
  const float k = 32.f * u * R, s2 = 2.5e-3f * R * R;
  bool ok = R > 1e-7f && R < 1e7f;  // R^4 within FP32's range
  int type = -1;
  if (!ee) {
    // triangle a b c, the point at the origin
    const f3 a = P1, b = P2, c = P3, ab = fsub3(b, a), ac = fsub3(c, a), bc = fsub3(c, b);
    const float lab = fdot3(ab, ab), lac = fdot3(ac, ac), lbc = fdot3(bc, bc);
    const float M = sqrtf(fmaxf(lab, fmaxf(lac, lbc)));
    ok = ok && fminf(lab, fminf(lac, lbc)) > s2;
    const float tol = k * (M + 1.75f * R), E = 8.f * k * M * R * R;
    const float d1 = -fdot3(ab, a), d2 = -fdot3(ac, a), d3 = -fdot3(ab, b), d4 = -fdot3(ac, b), d5 = -fdot3(ab, c),
                d6 = -fdot3(ac, c), e1 = fdot3(bc, b), e2 = -fdot3(bc, c);
    const float vc = d1 * d4 - d3 * d2, vb = d5 * d2 - d1 * d6, va = d3 * d6 - d5 * d4;
    // a vertex: both edges there lead away from the point, whose projection is outside
    if (-d1 > tol && -d2 > tol && fminf(vb, vc) < -E) type = 0;
    if (d3 > tol && e1 > tol && fminf(va, vc) < -E) type = 1;
    if (d6 > tol && e2 > tol && fminf(va, vb) < -E) type = 2;
    // an edge: the foot lies inside it and the projection beyond it
    if (d1 > tol && -d3 > tol && vc < -E) type = 3;
    if (-e1 > tol && -e2 > tol && va < -E) type = 4;
    if (d2 > tol && -d6 > tol && vb < -E) type = 5;
    if (va > E && vb > E && vc > E) type = 6;
  } else {
    const f3 d1 = P1, d2 = fsub3(P3, P2), A1B0 = fsub3(P1, P2), B1A1 = fsub3(P3, P1);
    const float a = fdot3(d1, d1), e = fdot3(d2, d2), b = fdot3(d1, d2), M2 = fmaxf(a, e);
    ok = ok && fminf(a, e) > s2;
    const float tol = k * (sqrtf(M2) + 3.5f * R), E = 16.f * k * R * M2;
    // (A_i - B0) . d2, (B1 - A_i) . d2, (B_j - A0) . d1, (A1 - B_j) . d1: positive when the end's foot lies inside
    const float la0 = -fdot3(P2, d2), ha0 = fdot3(P3, d2), la1 = fdot3(A1B0, d2), ha1 = fdot3(B1A1, d2);
    const float lb0 = fdot3(P2, d1), hb0 = fdot3(A1B0, d1), lb1 = fdot3(P3, d1), hb1 = -fdot3(B1A1, d1);
    const float sn = b * la0 + lb0 * e, tn = a * la0 + b * lb0, den = a * e - b * b;
    const bool s_lo = sn < -E, s_hi = sn > den + E, t_lo = tn < -E, t_hi = tn > den + E;
    if (s_lo || s_hi || t_lo || t_hi) {  // the lines' closest points are not both inside
      if (la0 < -tol && lb0 < -tol) type = 0;
      if (ha0 < -tol && lb1 < -tol) type = 1;
      if (la1 < -tol && hb0 < -tol) type = 2;
      if (ha1 < -tol && hb1 < -tol) type = 3;
      if (s_lo && la0 > tol && ha0 > tol) type = 4;
      if (s_hi && la1 > tol && ha1 > tol) type = 5;
      if (t_lo && lb0 > tol && hb0 > tol) type = 6;
      if (t_hi && lb1 > tol && hb1 > tol) type = 7;
    } else if (sn > E && den - sn > E && tn > E && den - tn > E) {
      type = 8;
    }
  }
  return ok ? type : -1;
}

// Points of the difference vectors A = p[1] - p[0], B = p[3] - p[2], E = p[5] - p[4] of each type, two bits a
// point: point-edge A = w, B = u (squared distance |A x B|^2 / |B|^2); face and line-line A = u, B = v, E = w
// ((E . (A x B))^2 / |A x B|^2); point-point A = B = b - a (|B|^2).
constexpr uint32_t pick6(int a0, int a1, int b0, int b1, int e0, int e1) {
  return (uint32_t)(a0 | a1 << 2 | b0 << 4 | b1 << 6 | e0 << 8 | e1 << 10);
}
__constant__ uint32_t c_pick_pt[7] = {pick6(0, 1, 0, 1, 0, 0), pick6(0, 2, 0, 2, 0, 0), pick6(0, 3, 0, 3, 0, 0),
                                      pick6(1, 0, 1, 2, 0, 0), pick6(2, 0, 2, 3, 0, 0), pick6(3, 0, 3, 1, 0, 0),
                                      pick6(1, 2, 1, 3, 1, 0)};
__constant__ uint32_t c_pick_ee[9] = {pick6(0, 2, 0, 2, 0, 0), pick6(0, 3, 0, 3, 0, 0), pick6(1, 2, 1, 2, 0, 0),
                                      pick6(1, 3, 1, 3, 0, 0), pick6(2, 0, 2, 3, 0, 0), pick6(2, 1, 2, 3, 0, 0),
                                      pick6(0, 2, 0, 1, 0, 0), pick6(0, 3, 0, 1, 0, 0), pick6(0, 1, 2, 3, 0, 2)};

__device__ __forceinline__ d3 pick(const cbg::Local& L, uint32_t i) {
  i &= 3u;
  const d3 a = i & 1u ? L.P1 : L.P0, b = i & 1u ? L.P3 : L.P2;
  return i & 2u ? b : a;
}

// squared distance of a known type, one instruction stream for all types
__device__ __forceinline__ double typed_d2(bool ee, const cbg::Local& L, int type) {
  const uint32_t k = ee ? c_pick_ee[type] : c_pick_pt[type];
  const bool plane = type == (ee ? 8 : 6), pp = ee ? type < 4 : type < 3;
  const d3 A = sub3(pick(L, k >> 2), pick(L, k)), B = sub3(pick(L, k >> 6), pick(L, k >> 4)),
           E = sub3(pick(L, k >> 10), pick(L, k >> 8));
  const d3 C = cross3(A, B);
  const double cc = dot3(C, C), bb = dot3(B, B), g = dot3(E, C);
  const double num = plane ? xmul(g, g) : (pp ? bb : cc), den = plane ? cc : (pp ? 1.0 : bb);
  return xdiv(num, den);
}

__device__ __forceinline__ cbb::f3 to_f3(d3 a) { return cbb::f3{(float)a.x, (float)a.y, (float)a.z}; }

// distance and type of a stencil given its 4 global points, as cbg::stencil_distance
__device__ __forceinline__ int stencil_distance(bool is_ee, d3 x0, d3 x1, d3 x2, d3 x3, double& d) {
  const cbg::Local L = cbg::make_local(x0, x1, x2, x3);
  int t = certain_type(is_ee, to_f3(L.P1), to_f3(L.P2), to_f3(L.P3));
  double d2 = 0.0;
  if (t >= 0) d2 = typed_d2(is_ee, L, t);
  else t = is_ee ? cbg::ee_type(L, d2) : cbg::pt_type(L, d2);  // only the undecided lanes' warps
  d = __dsqrt_rn(d2);
  return t;
}

}  // namespace cbt
