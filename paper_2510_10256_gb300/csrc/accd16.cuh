// accd16.cuh -- the FP64 additive-CCD iteration of one pair by half a warp.
//
// A short list of pairs is bound by the longest chain of dependent FP64
// instructions: a warp issues one in 64 cycles whether one lane or 32 use it,
// and a step of a pair on one lane takes about 110 of them.  Here lane 4 v + c
// of a half-warp holds component c of vertex v (the fourth lane of a quad
// repeats the third), so the four position updates, the differences, the cross
// product and the dot products each are one instruction for all their
// components: about 50 a step.  Every operation and its order are those of the
// one-lane iteration, so the results are the same bits.  The formula of the
// last step's distance type runs while FP32 decides the type (typed.cuh); it is
// run again when the type has changed.  A step takes about 4,000 cycles (half of
// it the two divisions and the square root).  Measured against one lane per
// pair, lists of 10 to 4,000 pairs: stacked layers (21 steps) 106 -> 70 us, a
// woven patch (28) 132 -> 89, 64 rod scenes (236) 984 -> 507, 649k caller's
// stencils 70 -> 47.
#pragma once
#include "typed.cuh"

namespace cba {

constexpr unsigned FULL = 0xffffffffu;
__device__ __forceinline__ unsigned half_mask() { return 0xffffu << (threadIdx.x & 16u); }
__device__ __forceinline__ int quad_vertex() { return (int)(threadIdx.x & 15u) >> 2; }
__device__ __forceinline__ int quad_component() { return min((int)(threadIdx.x & 3u), 2); }
__device__ __forceinline__ bool half_leader() { return (threadIdx.x & 15u) == 0; }
// A value read by one lane of the half for all 16.  Other warps lower the
// bounds of the smallest t_p while they are read, so lanes that read them for
// themselves could see different values and part before a shuffle that names
// them all; every branch on such a bound takes it from here.
template <class Read>
__device__ __forceinline__ auto half_read(Read read) -> decltype(read()) {
  decltype(read()) v{};
  if (half_leader()) v = read();
  return __shfl_sync(half_mask(), v, 0, 16);
}

// One pair on its half-warp: component c of vertex v on each lane, the rest alike on all 16.
struct Pair16 {
  double y, q;  // local position, displacement without its mean
  double off, lp, g, t, tl, hi, cap;
  int it, type;
  bool ee, first;
};

// sum over a quad's components, (x + y) + z
__device__ __forceinline__ double quad_sum(double a, unsigned mask) {
  const int b = (int)(threadIdx.x & 12u);
  const double x = __shfl_sync(mask, a, b, 16), y = __shfl_sync(mask, a, b + 1, 16), z = __shfl_sync(mask, a, b + 2, 16);
  return xadd(xadd(x, y), z);
}

// squared distance of a known type (typed_d2 of typed.cuh); P: local positions, both halves of the warp take part
__device__ __forceinline__ double formula16(double P, bool ee, int type) {
  const int v = quad_vertex(), c = quad_component(), c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
  const uint32_t k = (ee ? cbt::c_pick_ee[type] : cbt::c_pick_pt[type]) >> (4 * v);
  // quads 0, 1, 2: the difference vectors A, B, E
  const double to = __shfl_sync(FULL, P, (int)(4 * (k >> 2 & 3u)) + c, 16), from = __shfl_sync(FULL, P, (int)(4 * (k & 3u)) + c, 16);
  const double D = xsub(to, from);
  const double a1 = __shfl_sync(FULL, D, c1, 16), a2 = __shfl_sync(FULL, D, c2, 16);
  const double b1 = __shfl_sync(FULL, D, 4 + c1, 16), b2 = __shfl_sync(FULL, D, 4 + c2, 16);
  const double C = xsub(xmul(a1, b2), xmul(a2, b1));
  // quads 0, 1, 2: C . C, B . B, E . C
  const double s = quad_sum(xmul(v == 0 ? C : D, v == 1 ? D : C), FULL);
  const double cc = __shfl_sync(FULL, s, 0, 16), bb = __shfl_sync(FULL, s, 4, 16), g = __shfl_sync(FULL, s, 8, 16);
  const bool plane = type == (ee ? 8 : 6), pp = ee ? type < 4 : type < 3;
  return xdiv(plane ? xmul(g, g) : (pp ? bb : cc), plane ? cc : (pp ? 1.0 : bb));
}

// distance of the pair with local positions S.y; S.type: the last step's type, in and out
__device__ __forceinline__ double distance16(Pair16& S, bool live) {
  const double P = xsub(S.y, __shfl_sync(FULL, S.y, quad_component(), 16));
  const float f = (float)P;
  float F[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) F[k] = __shfl_sync(FULL, f, 4 + 4 * (k / 3) + k % 3, 16);
  double d2 = formula16(P, S.ee, S.type);
  const int type =
      cbt::certain_type(S.ee, cbb::f3{F[0], F[1], F[2]}, cbb::f3{F[3], F[4], F[5]}, cbb::f3{F[6], F[7], F[8]});
  if (__any_sync(FULL, live && type >= 0 && type != S.type)) {
    if (type >= 0) S.type = type;
    d2 = formula16(P, S.ee, S.type);
  }
  if (live && type < 0) {  // undecided: the full routine, on every lane of the half alike
    double X[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) X[k] = __shfl_sync(half_mask(), P, 4 + 4 * (k / 3) + k % 3, 16);
    const cbg::Local L{mk3(0.0, 0.0, 0.0), mk3(X[0], X[1], X[2]), mk3(X[3], X[4], X[5]), mk3(X[6], X[7], X[8])};
    S.type = S.ee ? cbg::ee_type(L, d2) : cbg::pt_type(L, d2);
  }
  return __dsqrt_rn(d2);
}

// Local position, displacement without its mean and relative speed bound of
// the pair whose vertex v this lane's quad holds (one half of the warp);
// false if a displacement's norm is not finite.
__device__ __forceinline__ bool load16(const double* __restrict__ x, const double* __restrict__ p, int n, int v, bool ee,
                                       Pair16& S) {
  const unsigned hm = half_mask();
  S.ee = ee;
  S.type = 0;  // a type of either kind
  const int c = quad_component();
  const double X = x[(size_t)c * n + v], Q = p[(size_t)c * n + v];
  S.y = xsub(X, __shfl_sync(hm, X, c, 16));
  const double p0 = __shfl_sync(hm, Q, c, 16), p1 = __shfl_sync(hm, Q, 4 + c, 16), p2 = __shfl_sync(hm, Q, 8 + c, 16),
               p3 = __shfl_sync(hm, Q, 12 + c, 16);
  S.q = xsub(Q, xmul(xadd(xadd(xadd(p0, p1), p2), p3), 0.25));
  const double nv = __dsqrt_rn(quad_sum(xmul(S.q, S.q), hm));
  const double n0 = __shfl_sync(hm, nv, 0, 16), n1 = __shfl_sync(hm, nv, 4, 16), n2 = __shfl_sync(hm, nv, 8, 16),
               n3 = __shfl_sync(hm, nv, 12, 16);
  S.lp = S.ee ? xadd(fmax(n0, n1), fmax(n2, n3)) : xadd(n0, fmax(fmax(n1, n2), n3));
  S.first = true;
  return isfinite(n0) && isfinite(n1) && isfinite(n2) && isfinite(n3);
}

// FP64 values as integers of the same order, for comparisons off the FP64 pipe: t, the bounds and g are not
// negative, and a negative gap compares below them as it should.  NaN has no place in that order (its sign may be
// set): a comparison that must be false for it asks number() as well.
__device__ __forceinline__ long long bits(double a) { return __double_as_longlong(a); }
__device__ __forceinline__ bool number(double a) { return (bits(a) & 0x7fffffffffffffffll) <= 0x7ff0000000000000ll; }

// The iteration over pairs [0, m), split evenly over the half-warps of `warps`
// warps.  J.wanted(w) compares pair w's lower bound with the bounds found so
// far (1: not above them), J.load(w, S) loads it (false: nothing to iterate),
// J.begin(S, d) takes its first distance (false: finished), J.cap() reads the
// smallest t_p found, J.done(S, t, how) ends a pair.  wanted and cap read values that other warps write: half_read takes the leader's answer; the
// rest of a pair is the same arithmetic on all 16 lanes.  Returns the most
// steps of a pair.
enum Done { REACHED, STOPPED, LIMIT };
template <class Job>
__device__ __forceinline__ int iterate16(Job& J, int64_t m, int warps, int warp, double c_step, int max_iter) {
  Pair16 S;
  S.y = S.q = S.off = S.lp = S.g = S.t = S.tl = S.hi = S.cap = 0.0;
  S.it = S.type = 0;
  S.ee = false;
  S.first = true;
  int64_t w = (threadIdx.x & 16u ? warps : 0) + warp;
  bool have = false;
  int most = 0;
  for (;;) {
    for (; !have && w < m; w += 2 * warps) have = half_read([&] { return J.wanted(w); }) && J.load(w, S);
    if (!__any_sync(FULL, have)) break;
    if (!S.first) S.y = xadd(S.y, xmul(S.tl, S.q));
    const double d = distance16(S, have);
    if (have && S.first) {
      S.first = false;
      S.t = 0.0;
      S.it = 0;
      have = J.begin(S, d);
      if (have) S.cap = half_read([&] { return J.cap(); });
    } else if (have) {
      const int it = S.it++;
      const double gap = xsub(d, S.off);
      if (bits(S.t) > 0 && bits(gap) < bits(S.g) && number(gap)) {
        J.done(S, S.t, REACHED);
        have = false;
      } else {
        S.t = xadd(S.t, S.tl);
        const bool some = number(S.t);
        if (some && bits(S.t) > bits(1.0)) {
          J.done(S, 1.0, REACHED);
          have = false;
        } else {
          if ((it & 7) == 7) S.cap = half_read([&] { return J.cap(); });
          if (some && ((bits(S.cap) < bits(1.0) && bits(S.t) >= bits(S.cap)) || bits(S.t) > bits(S.hi))) {  // t_p >= t: this pair cannot lower the minimum
            J.done(S, S.t, STOPPED);
            have = false;
          } else if (it + 1 >= max_iter) {
            J.done(S, S.t, LIMIT);
            have = false;
          } else {
            S.tl = xdiv(xmul(c_step, gap), S.lp);
          }
        }
      }
      if (!have) most = max(most, it + 1);
    }
    __syncwarp();
  }
  return most;
}

}  // namespace cba
