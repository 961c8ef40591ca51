// accd32.cuh -- rigorous FP32 bounds of a pair's additive-CCD time.
//
// Additive CCD (ccd.cu) runs T_1 = (1-s) g0 / l, T_{k+1} = T_k + c f(T_k) / l
// with f(T) the gap (distance minus offset) after the step T, g0 = f(0), l a
// bound on f's slope; from k = 2 on it stops at the first k with f(T_k) < s g0
// and returns T_{k-1}, or 1 once an accepted T_k exceeds 1.  Since |f'| <= l
// and c < 1, T + c f(T) / l grows with T, so an interval [l_k, u_k] holding
// T_k maps to one holding T_{k+1} by evaluating bounds of f at its two ends.
// In FP32, with every step rounded outwards, that brackets the FP64
// iteration's own T_k (whose rounding, at most a few thousand ulp of FP64, is
// far inside the FP32 margins) until its stopping test is surely met (t_p lies
// in the last interval), surely passed beyond T = 1 (t_p is 1), or cannot be
// told at FP32 accuracy (t_p is at least the last accepted lower end).
//
// The step bound needs only the smallest t_p: after this pass, on the FP32
// pipe (64 times the FP64 rate), the FP64 iteration is left with the pairs
// whose lower bound is not above the smallest upper bound -- a handful instead
// of every pair within a ceiling of the smallest first step.  On GB300, from
// rounds of FP64 iterations under a growing ceiling (selected, scanned and
// counted on the host each round) to one bracket pass and one FP64 pass: step
// bound of a 200k-triangle graded disk 5.48 -> 3.61 ms (FP64 iterations 1.50 ->
// 0.04 ms, brackets 0.26), of 64 rod scenes 7.03 -> 4.65, of a woven patch of
// 4,112 vertices 0.83 -> 0.40 (five rounds); a list of 650k stencils 1.22 ->
// 0.26 ms.
#pragma once
#include "bound32.cuh"

namespace cbb {

constexpr int REFINE_ITERS = 64;

struct Motion32 {
  bool ee;
  f3 Y[4], Q[4];         // positions relative to the first vertex, displacements relative to their mean
  float X;               // bound on the rounding scale of Y + T Q
  float off_dn, off_up;  // the offset, rounded down and up
  float lp_dn, lp_up;    // the slope bound l, rounded down and up
};

// bounds of the gap after the step T
__device__ __forceinline__ void gap_bounds(const Motion32& M, float T, float& lo, float& hi) {
  f3 W[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    W[k] = f3{fmaf(T, M.Q[k].x, M.Y[k].x), fmaf(T, M.Q[k].y, M.Y[k].y), fmaf(T, M.Q[k].z, M.Y[k].z)};
  float ub;
  const float lb = distance_bounds(M.ee, W[0], W[1], W[2], W[3], M.X, ub);
  lo = __fsub_rd(lb, M.off_up);
  hi = __fsub_ru(ub, M.off_dn);
}

// l_p from the relative displacements; false if FP32 cannot hold the pair
// (not finite, out of range, or no motion to speak of)
__device__ __forceinline__ bool motion_slopes(Motion32& M) {
  const float n0 = sqrtf(fdot3(M.Q[0], M.Q[0])), n1 = sqrtf(fdot3(M.Q[1], M.Q[1])), n2 = sqrtf(fdot3(M.Q[2], M.Q[2])),
              n3 = sqrtf(fdot3(M.Q[3], M.Q[3]));
  const float l = M.ee ? fmaxf(n0, n1) + fmaxf(n2, n3) : n0 + fmaxf(fmaxf(n1, n2), n3);
  // sum, not maximum: a NaN must not pass
  const float R = fmaxabs3(M.Y[1]) + fmaxabs3(M.Y[2]) + fmaxabs3(M.Y[3]);
  const float P = n0 + n1 + n2 + n3;
  const float s = fabsf(M.Y[1].x) + fabsf(M.Y[1].y) + fabsf(M.Y[1].z) + fabsf(M.Y[2].x) + fabsf(M.Y[2].y) +
                  fabsf(M.Y[2].z) + fabsf(M.Y[3].x) + fabsf(M.Y[3].y) + fabsf(M.Y[3].z) + P;
  M.X = 2.f * (R + 4.f * P);  // T stays below 4
  M.lp_dn = l * (1.f - 64.f * 5.9604645e-8f);
  M.lp_up = l * (1.f + 64.f * 5.9604645e-8f);
  return s < 1e15f && l > 1e-15f;
}

// Bounds [lo, hi] of t_p; cap() is an upper bound of the smallest t_p known so
// far (the pair is dropped once its lower bound is above it).  Returns 1 if
// t_p is exactly 1, 0 if lo <= t_p <= hi, -1 if FP32 cannot tell the gap at
// T = 0 from zero (no bounds).
template <typename Cap>
__device__ __forceinline__ int accd_bounds32(const Motion32& M, Cap cap, float& lo, float& hi) {
  constexpr float C_DN = 0.9f, C_UP = 0.90000004f;   // c = 1 - s = 0.9 between them
  constexpr float S_DN = 0.099999994f, S_UP = 0.1f;  // s = 0.1 between them
  float g0l, g0u;
  gap_bounds(M, 0.f, g0l, g0u);
  if (!(g0l > 0.f)) return -1;
  float l = __fdiv_rd(__fmul_rd(C_DN, g0l), M.lp_up), u = __fdiv_ru(__fmul_ru(C_UP, g0u), M.lp_dn);
  if (l > 1.f) return 1;
  lo = l;
  hi = 1.f;
  if (!(u <= 1.f)) return 0;
  const float gl = __fmul_rd(S_DN, g0l), gu = __fmul_ru(S_UP, g0u);
  float al, au, bl, bu;  // bounds of f at l and at u
  gap_bounds(M, l, al, au);
  gap_bounds(M, u, bl, bu);
  for (int it = 0; it < REFINE_ITERS; ++it) {
    if (lo > cap() || !(bu < 1e30f)) return 0;  // dropped, or no upper bound (a degenerate stencil)
    const float l2 = __fadd_rd(l, __fdiv_rd(__fmul_rd(C_DN, fmaxf(al, 0.f)), M.lp_up));
    const float u2 = __fadd_ru(u, __fdiv_ru(__fmul_ru(C_UP, fmaxf(bu, 0.f)), M.lp_dn));
    if (!(u2 < 4.f)) return 0;  // far past 1: nothing more to learn at FP32 accuracy
    gap_bounds(M, l2, al, au);
    gap_bounds(M, u2, bl, bu);
    const float w = __fmul_ru(M.lp_up, __fsub_ru(u2, l2));
    const float fmin = __fmul_rd(0.5f, __fsub_rd(__fadd_rd(al, bl), w));
    const float fmax = __fmul_ru(0.5f, __fadd_ru(__fadd_ru(au, bu), w));
    if (fmin >= gu) {  // surely goes on: T_k is accepted
      l = l2;
      u = u2;
      if (l > 1.f) return 1;
      lo = l;
      if (!(u <= 1.f)) return 0;
    } else {
      if (fmax < gl) hi = u;  // surely stops: t_p = T_{k-1}
      return 0;
    }
  }
  return 0;
}

}  // namespace cbb
