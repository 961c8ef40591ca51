// ccd.cu -- stage (e): conservative step bound for the line search (Sec. 3.3).
//
// Candidates: pairs whose swept boxes (x and x + p) inflated by xi/2 overlap.
// Class of a pair at x: F if filtered (Sec. 3.2), C if unfiltered and already
// within the offset (Sec. 3.4), U otherwise.  Offset: U -> xi (0 in the
// single-phase mode), F and C -> 0 (the filtered pairs are single-phase, Eq. 4).
// Each pair is bounded by additive CCD (C-IPC): in the pair's local frame with
// the mean displacement removed, l_p bounds the relative speed of the closest
// points; the first step (1-s) g0 / l_p and every later step c (d - offset)/l_p
// cannot close the gap, and the iteration stops before the gap would drop
// below s g0.  alpha = min(1, min_p t_p).
//
// Only the minimum is needed, so the step bound is computed exactly without
// iterating every pair in FP64.  The additive-CCD iterate t only grows, and
// t_p >= min(1, (1-s) g0 / l_p).  Pass 1 bounds that first step per pair (FP32
// bounds; one FP64 distance where they cannot decide) and lists the pairs it
// leaves below 1.  Pass 2 brackets each listed pair's t_p in FP32
// (accd32.cuh), keeping the smallest upper bound per member, and lists the
// pairs whose lower bound is not above it.  Pass 3 runs the FP64 iteration on
// those, dropping a pair once its iterate is above that bound or reaches the
// smallest exact t_p found: every pair dropped has t_p no smaller, so alpha is
// the minimum over all pairs of the full iteration's t_p, bit for bit.  Every
// list length stays on the device: no host wait after the broad phase.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "accd16.cuh"
#include "accd32.cuh"
#include "geometry.cuh"
#include "prims.cuh"
#include "scene.cuh"
#include "typed.cuh"

namespace {

constexpr double ACCD_S = 0.1;
constexpr double ACCD_C = 0.9;
constexpr int ACCD_MAX_ITER = 10000;
constexpr uint8_t EXACT = CB_CCD_EXACT, ONE = CB_CCD_ONE;  // class byte flags (scene.cuh)

struct CcdArgs {
  int64_t np;
  const uint64_t* __restrict__ keys;
  const int32_t* __restrict__ ev0;
  const int32_t* __restrict__ ev1;
  const int32_t* __restrict__ tv;
  int T, n;
  const int32_t* __restrict__ vsc;           // member of each vertex
  const MemberParams* __restrict__ mp;
  const double* __restrict__ cx;             // per member: centre[3], X
  const double* __restrict__ x;
  const double* __restrict__ p;
  double* __restrict__ t_out;
  uint8_t* __restrict__ cls_out;             // in: 1 filtered, 3 culled, else 0 (Sec. 3.2); out: class | flags
  unsigned long long* __restrict__ macc;     // per member: alpha bits, status, smallest upper bound
  int members;
  unsigned long long* __restrict__ status;
  unsigned long long* __restrict__ max_iters;
  const float4* __restrict__ xf;  // FP32 (x - member centre), one float4 per vertex
  const float4* __restrict__ pf;  // FP32 p, one float4 per vertex
  uint32_t* __restrict__ ulist;   // pairs left unresolved by the first step (t_out, a lower bound, below 1)
  unsigned int* __restrict__ nu;
  // pairs left for the FP64 iteration: point-triangle from the front (nlist[0] of them), edge-edge from the back
  // (nlist[1]) of np entries: the distance routine branches on the kind, and a warp that mixes them runs both
  uint32_t* __restrict__ list;
  unsigned int* __restrict__ nlist;
};

__device__ __forceinline__ unsigned long long* macc_of(const CcdArgs& A, int m, int slot) {
  return &A.macc[(size_t)m * MACC_STRIDE + slot];
}

__device__ __forceinline__ d3 ld(const double* __restrict__ a, int n, int v) {
  return mk3(a[v], a[(size_t)n + v], a[2 * (size_t)n + v]);
}
__device__ __forceinline__ double norm3(d3 a) { return __dsqrt_rn(dot3(a, a)); }
__device__ __forceinline__ d3 axpy3(d3 x, double t, d3 p) {
  return mk3(xadd(x.x, xmul(t, p.x)), xadd(x.y, xmul(t, p.y)), xadd(x.z, xmul(t, p.z)));
}

// Everything additive CCD needs before its first step.
struct AccdStart {
  bool ee;
  int cls, mem;
  double off, lp, g0;
  d3 Y0, Y1, Y2, Y3, Q0, Q1, Q2, Q3;
};

__device__ __forceinline__ AccdStart accd_start(const CcdArgs& A, int64_t q) {
  AccdStart S;
  const uint64_t key = A.keys[q];
  const uint32_t ty = cb_key_type(key), ki = cb_key_i(key), kj = cb_key_j(key);
  int v[4];
  if (ty == CB_KEY_PT) {
    v[0] = (int)ki;
    v[1] = A.tv[kj];
    v[2] = A.tv[A.T + kj];
    v[3] = A.tv[2 * A.T + kj];
    S.ee = false;
  } else {
    v[0] = A.ev0[ki];
    v[1] = A.ev1[ki];
    v[2] = A.ev0[kj];
    v[3] = A.ev1[kj];
    S.ee = true;
  }
  S.mem = A.vsc[v[0]];
  const MemberParams& M = A.mp[S.mem];
  const bool filt = (A.cls_out[q] & 3u) == 1u;
  const d3 X0 = ld(A.x, A.n, v[0]), X1 = ld(A.x, A.n, v[1]), X2 = ld(A.x, A.n, v[2]), X3 = ld(A.x, A.n, v[3]);
  const d3 P0 = ld(A.p, A.n, v[0]), P1 = ld(A.p, A.n, v[1]), P2 = ld(A.p, A.n, v[2]), P3 = ld(A.p, A.n, v[3]);
  double d;
  cbt::stencil_distance(S.ee, X0, X1, X2, X3, d);
  S.cls = filt ? 1 : 0;
  if (!filt && M.core_temp && !M.single && d <= M.xi) S.cls = 2;
  S.off = (S.cls == 0 && !M.single) ? M.xi : 0.0;
  const d3 pb = mk3(xmul(xadd(xadd(xadd(P0.x, P1.x), P2.x), P3.x), 0.25),
                    xmul(xadd(xadd(xadd(P0.y, P1.y), P2.y), P3.y), 0.25),
                    xmul(xadd(xadd(xadd(P0.z, P1.z), P2.z), P3.z), 0.25));
  S.Y0 = sub3(X0, X0);
  S.Y1 = sub3(X1, X0);
  S.Y2 = sub3(X2, X0);
  S.Y3 = sub3(X3, X0);
  S.Q0 = sub3(P0, pb);
  S.Q1 = sub3(P1, pb);
  S.Q2 = sub3(P2, pb);
  S.Q3 = sub3(P3, pb);
  const double n0 = norm3(S.Q0), n1 = norm3(S.Q1), n2 = norm3(S.Q2), n3 = norm3(S.Q3);
  S.lp = S.ee ? xadd(fmax(n0, n1), fmax(n2, n3)) : xadd(n0, fmax(fmax(n1, n2), n3));
  // The distance of the local-frame copy Y (Y0 = 0) equals d bit for bit: the
  // distance routine itself works relative to the first vertex, and
  // (x_i - x_0) - 0 = x_i - x_0 exactly.
  S.g0 = (S.lp != 0.0) ? xsub(d, S.off) : 0.0;
  return S;
}

__device__ __forceinline__ cbb::f3 ldf(const float4* __restrict__ a, int n, int v) {
  const float4 q = a[v];
  return cbb::f3{q.x, q.y, q.z};
}

// FP32 motion of a stencil in its local frame: positions relative to the
// first vertex, displacements relative to their mean, subtracted in FP64
__device__ __forceinline__ void pair_motion32(const double* __restrict__ x, const double* __restrict__ p, int n,
                                              const int (&v)[4], cbb::Motion32& M) {
  const d3 X0 = ld(x, n, v[0]);
  d3 P[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const d3 Y = sub3(ld(x, n, v[k]), X0);
    M.Y[k] = cbb::f3{(float)Y.x, (float)Y.y, (float)Y.z};
    P[k] = ld(p, n, v[k]);
  }
  const d3 pb = mk3(xmul(xadd(xadd(xadd(P[0].x, P[1].x), P[2].x), P[3].x), 0.25),
                    xmul(xadd(xadd(xadd(P[0].y, P[1].y), P[2].y), P[3].y), 0.25),
                    xmul(xadd(xadd(xadd(P[0].z, P[1].z), P[2].z), P[3].z), 0.25));
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const d3 Q = sub3(P[k], pb);
    M.Q[k] = cbb::f3{(float)Q.x, (float)Q.y, (float)Q.z};
  }
}

__device__ __forceinline__ void warp_append(bool flag, uint32_t value, uint32_t* __restrict__ list,
                                            unsigned int* __restrict__ count) {
  const unsigned m = __ballot_sync(0xffffffffu, flag);
  if (!m) return;
  const unsigned lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if ((int)lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (flag) list[base + __popc(m & ((1u << lane) - 1u))] = value;
}
// ... from the end of a list of cap entries backwards
__device__ __forceinline__ void warp_append_back(bool flag, uint32_t value, uint32_t* __restrict__ list, int64_t cap,
                                                 unsigned int* __restrict__ count) {
  const unsigned m = __ballot_sync(0xffffffffu, flag);
  if (!m) return;
  const unsigned lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if ((int)lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (flag) list[cap - 1 - (int64_t)(base + __popc(m & ((1u << lane) - 1u)))] = value;
}

// pass 1a: an FP32 lower bound of the distance and an FP32 upper bound of
// l_p give a lower bound of the first step.  A pair whose class is certain and
// whose bound exceeds 1 is resolved (t_p = 1); a smaller bound is kept as its
// lower bound.  Pairs the FP32 bounds cannot settle are queued for pass 1b.
// The bound is formed in FP32 with every operation rounded towards the safe
// side (__f*_rd for lower bounds, __f*_ru for upper ones) and a final factor
// 1 - 2^-23, so it stays below the first step as FP64 evaluates it; the
// thresholds are the members' FP32 copies rounded up.  (FP64 would put ~25
// operations per candidate on the FP64 pipe, which issues 1/64 as fast.)
__global__ void __launch_bounds__(128) k_ccd_screen(CcdArgs A, uint32_t* __restrict__ list,
                                                    unsigned int* __restrict__ nlist) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool need = false, unres = false;
  if (q < A.np) {
    const uint64_t key = A.keys[q];
    const uint32_t ty = cb_key_type(key), ki = cb_key_i(key), kj = cb_key_j(key);
    int v[4];
    bool ee;
    if (ty == CB_KEY_PT) {
      v[0] = (int)ki;
      v[1] = A.tv[kj];
      v[2] = A.tv[A.T + kj];
      v[3] = A.tv[2 * A.T + kj];
      ee = false;
    } else {
      v[0] = A.ev0[ki];
      v[1] = A.ev1[ki];
      v[2] = A.ev0[kj];
      v[3] = A.ev1[kj];
      ee = true;
    }
    const int mem = A.vsc[v[0]];
    const MemberParams& M = A.mp[mem];
    const uint8_t cls0 = A.cls_out[q];
    const bool filt = cls0 == 1;
    need = true;
    if (cls0 == 3) {  // culled (Kaldor mode): the pair does not constrain the step
      A.cls_out[q] = (uint8_t)3 | EXACT | ONE;
      need = false;
    } else {
      const double Xd = A.cx[4 * mem + 3];
      const float lb = cbb::lower_bound(ee, ldf(A.xf, A.n, v[0]), ldf(A.xf, A.n, v[1]), ldf(A.xf, A.n, v[2]),
                                        ldf(A.xf, A.n, v[3]), (float)Xd);
      if (filt || lb >= M.thrC32) {  // surely not class C at or above thrC32
        const int cls = filt ? 1 : 0;
        const float off = (cls == 0 && !M.single) ? M.xi32 : 0.f;
        const cbb::f3 p0 = ldf(A.pf, A.n, v[0]), p1 = ldf(A.pf, A.n, v[1]), p2 = ldf(A.pf, A.n, v[2]),
                      p3 = ldf(A.pf, A.n, v[3]);
        const cbb::f3 pm = cbb::fscale3(cbb::fadd3(cbb::fadd3(p0, p1), cbb::fadd3(p2, p3)), 0.25f);
        const cbb::f3 r0 = cbb::fsub3(p0, pm), r1 = cbb::fsub3(p1, pm), r2 = cbb::fsub3(p2, pm), r3 = cbb::fsub3(p3, pm);
        const float m0 = cbb::fdot3(r0, r0), m1 = cbb::fdot3(r1, r1), m2 = cbb::fdot3(r2, r2), m3 = cbb::fdot3(r3, r3);
        // (the root of the larger square is the larger root)
        const float lp32 = ee ? cbb::qsqrt(fmaxf(m0, m1)) + cbb::qsqrt(fmaxf(m2, m3))
                              : cbb::qsqrt(m0) + cbb::qsqrt(fmaxf(fmaxf(m1, m2), m3));
        const float Pm = fmaxf(fmaxf(cbb::fmaxabs3(p0), cbb::fmaxabs3(p1)), fmaxf(cbb::fmaxabs3(p2), cbb::fmaxabs3(p3)));
        const float u64 = 3.8146973e-6f;  // 64 u, u = 2^-24: exact
        const float lp_ub = __fadd_ru(__fmul_ru(lp32, 1.f + u64), __fmul_ru(u64, Pm));
        const float slack = __fmul_ru(1e-12f, __fadd_ru(1.f, __double2float_ru(Xd)));
        const float g_lb = __fsub_rd(__fsub_rd(lb, off), slack);
        if (lp32 > 1e-30f && g_lb > 0.f) {
          // (1 - s) g / l_p; 0.9f rounds below 0.9 = 1 - s
          const float tl_lb = __fmul_rd(__fdiv_rd(__fmul_rd(0.9f, g_lb), lp_ub), 0.99999988f);
          unres = !(tl_lb > 1.f);
          if (unres) A.t_out[q] = (double)tl_lb;
          A.cls_out[q] = (uint8_t)cls | (unres ? 0 : EXACT | ONE);
          need = false;
        }
      }
    }
  }
  warp_append(need, (uint32_t)q, list, nlist);
  warp_append(unres, (uint32_t)q, A.ulist, A.nu);
}

// pass 1b: exact FP64 first step of the queued pairs
__global__ void __launch_bounds__(128) k_ccd_bound(CcdArgs A, const uint32_t* __restrict__ list,
                                                   const unsigned int* __restrict__ nlist) {
  const unsigned m = *nlist;
  // uniform trip count per block so that every lane reaches the append
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x; w0 < m; w0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = w0 + threadIdx.x;
    bool unres = false;
    uint32_t qq = 0;
    if (w < m) {
      const int64_t q = list[w];
      const AccdStart S = accd_start(A, q);
      const double tl = S.lp == 0.0 ? 2.0 : xdiv(xmul(xsub(1.0, ACCD_S), S.g0), S.lp);
      uint8_t flags = EXACT | ONE;  // no motion, or the first step already passes t_c = 1
      if (S.lp != 0.0 && S.g0 <= 0.0) {
        flags = EXACT;
        A.t_out[q] = 0.0;
        atomicOr(A.status, (unsigned long long)CB_DEV_PENETRATION);
        atomicOr(macc_of(A, S.mem, MACC_STATUS), (unsigned long long)CB_DEV_PENETRATION);
        atomicMin(macc_of(A, S.mem, MACC_ALPHA), 0ull);
      } else if (!(tl > 1.0)) {
        flags = 0;
        A.t_out[q] = tl;
        unres = true;
      }
      A.cls_out[q] = (uint8_t)S.cls | flags;
      qq = (uint32_t)q;
    }
    warp_append(unres, qq, A.ulist, A.nu);
  }
}

// an upper bound of the member's smallest t_p: FP32 brackets and exact values so far (rounded up)
__device__ __forceinline__ float member_cap(const CcdArgs& A, int mem) {
  const double a = __longlong_as_double(*(volatile unsigned long long*)macc_of(A, mem, MACC_ALPHA));
  const double h = __longlong_as_double(*(volatile unsigned long long*)macc_of(A, mem, MACC_HI));
  return __double2float_ru(fmin(a, h));
}

// pass 2: FP32 brackets of the unresolved pairs (grid-stride; the trip count
// is uniform over a warp so that every lane reaches the appends).  Bound by the
// latency of each pair's chain of steps: 80 registers let six blocks share an SM
// instead of five (pleated 256x256 174 -> 150 us; at eight the spills cost more)
__global__ void __launch_bounds__(128, 6) k_ccd_refine(CcdArgs A) {
  const int64_t nu = min((int64_t)*A.nu, A.np);
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x; w0 < nu; w0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = w0 + threadIdx.x;
    bool keep = false, ee = false;
    uint32_t q = 0;
    if (w < nu) {
      q = A.ulist[w];
      const uint64_t key = A.keys[q];
      const uint32_t ki = cb_key_i(key), kj = cb_key_j(key);
      ee = cb_key_type(key) != CB_KEY_PT;
      const int v0 = ee ? A.ev0[ki] : (int)ki;
      const int mem = A.members > 1 ? A.vsc[v0] : 0;
      const double lb = A.t_out[q];
      if (__double2float_rd(lb) <= member_cap(A, mem)) {
        int v[4] = {v0, 0, 0, 0};
        if (ee) {
          v[1] = A.ev1[ki];
          v[2] = A.ev0[kj];
          v[3] = A.ev1[kj];
        } else {
#pragma unroll
          for (int k = 0; k < 3; ++k) v[1 + k] = A.tv[(size_t)k * A.T + kj];
        }
        cbb::Motion32 M;
        M.ee = ee;
        const uint8_t cls = A.cls_out[q];
        const MemberParams& MP = A.mp[mem];
        const double off = (cls == 0 && !MP.single) ? MP.xi : 0.0;
        M.off_dn = __double2float_rd(off);
        M.off_up = __double2float_ru(off);
        pair_motion32(A.x, A.p, A.n, v, M);
        float lo = 0.f, hi = 1.f;
        const int r = cbb::motion_slopes(M) ? cbb::accd_bounds32(M, [&] { return member_cap(A, mem); }, lo, hi) : -1;
        if (r == 1) {
          A.cls_out[q] = cls | EXACT | ONE;
        } else {
          if (r == 0 && (double)lo > lb) A.t_out[q] = (double)lo;
          if (r == 0 && hi < 1.f) atomicMin(macc_of(A, mem, MACC_HI), (unsigned long long)__double_as_longlong((double)hi));
          keep = r < 0 || lo <= member_cap(A, mem);
        }
      }
    }
    warp_append(keep && !ee, q, A.list, &A.nlist[0]);
    warp_append_back(keep && ee, q, A.list, A.np, &A.nlist[1]);
  }
}

// pass 3: additive CCD of the pairs left by pass 2 whose lower bound is still
// not above the member's bound.
// Pairs need very different numbers of steps, and an FP64 warp instruction
// costs a warp the same whether one lane or 32 use it, so the warps are
// persistent and hand idle lanes new pairs -- but only once EXACT_REFILL of
// them are idle (or all are): the set-up of a pair (its first distance) then
// runs once for a group of lanes instead of once per lane that finishes.
// A pair's arithmetic is the same whichever lane runs it.
constexpr int EXACT_REFILL = 8;
// Pairs per 128-thread block (one per SM) up to which a half-warp takes each (accd16.cuh).  A half-warp's step costs
// its warp 25 FP64 instructions a pair, 32 single lanes' 3.5 -- but they wait for the longest of 32 pairs, at twice the
// time a step.  With every pair alike (a tie, three steps each; the worst case for half-warps) the two are even at
// 2,000 pairs and 5,000 take 110 against 76 us; with 2,500 pairs of 6 steps and one of 236 half-warps take 507 us
// against 984.  The line lies at 4,864 pairs on 152 SMs: at most 0.03 ms lost, half a millisecond won.
constexpr int FEW_PER_BLOCK = 32;

struct ExactLane {
  AccdStart S;
  int64_t q;
  double t, tl, g, hi, cap;
  int it;
};

// finish a pair: exact t_p, or (stopped) a lower bound
__device__ __forceinline__ void exact_finish(const CcdArgs& A, int64_t q, int mem, int cls, bool stopped, double t) {
  A.t_out[q] = t;
  A.cls_out[q] = (uint8_t)cls | (stopped ? 0 : EXACT);
  if (!stopped) atomicMin(macc_of(A, mem, MACC_ALPHA), (unsigned long long)__double_as_longlong(t));
}
__device__ __forceinline__ void exact_finish(const CcdArgs& A, const ExactLane& L, bool stopped, double t) {
  exact_finish(A, L.q, L.S.mem, L.S.cls, stopped, t);
}

// a short list: half a warp per pair (accd16.cuh)
struct ExactJob {
  const CcdArgs& A;
  int64_t mf;  // point-triangle pairs, from the list's front
  int64_t q;
  int mem, cls;

  __device__ __forceinline__ int64_t pair(int64_t w) const { return w < mf ? A.list[w] : A.list[A.np - 1 - (w - mf)]; }
  __device__ __forceinline__ int member(uint64_t key) const {
    const uint32_t ki = cb_key_i(key);
    return A.members > 1 ? A.vsc[cb_key_type(key) != CB_KEY_PT ? A.ev0[ki] : (int)ki] : 0;
  }
  __device__ __forceinline__ int wanted(int64_t w) const {
    const int64_t k = pair(w);
    return __double2float_rd(A.t_out[k]) <= member_cap(A, member(A.keys[k]));
  }
  __device__ __forceinline__ bool load(int64_t w, cba::Pair16& S) {
    q = pair(w);
    const uint64_t key = A.keys[q];
    const uint32_t ki = cb_key_i(key), kj = cb_key_j(key);
    const bool ee = cb_key_type(key) != CB_KEY_PT;
    const int k = cba::quad_vertex();
    mem = member(key);
    const int v0 = ee ? A.ev0[ki] : (int)ki;
    const uint32_t e = k < 2 ? ki : kj;
    const int v = ee ? (k & 1 ? A.ev1[e] : A.ev0[e]) : (k == 0 ? v0 : A.tv[(size_t)(k - 1) * A.T + kj]);
    cba::load16(A.x, A.p, A.n, v, ee, S);
    return true;
  }
  __device__ __forceinline__ bool begin(cba::Pair16& S, double d) {
    const MemberParams& M = A.mp[mem];
    cls = (A.cls_out[q] & 3u) == 1u ? 1 : 0;
    if (cls == 0 && M.core_temp && !M.single && d <= M.xi) cls = 2;
    S.off = (cls == 0 && !M.single) ? M.xi : 0.0;
    const double g0 = S.lp != 0.0 ? xsub(d, S.off) : 0.0;
    if (S.lp == 0.0 || g0 <= 0.0) {
      if (S.lp != 0.0 && cba::half_leader()) {
        atomicOr(A.status, (unsigned long long)CB_DEV_PENETRATION);
        atomicOr(macc_of(A, mem, MACC_STATUS), (unsigned long long)CB_DEV_PENETRATION);
      }
      done(S, S.lp == 0.0 ? 1.0 : 0.0, cba::REACHED);
      return false;
    }
    S.hi = __longlong_as_double(*macc_of(A, mem, MACC_HI));  // no longer moves
    S.g = xmul(ACCD_S, g0);
    S.tl = xdiv(xmul(xsub(1.0, ACCD_S), g0), S.lp);
    return true;
  }
  __device__ __forceinline__ double cap() const {
    return __longlong_as_double(*(volatile unsigned long long*)macc_of(A, mem, MACC_ALPHA));
  }
  __device__ __forceinline__ void done(const cba::Pair16&, double t, cba::Done how) const {
    if (!cba::half_leader()) return;
    if (how == cba::LIMIT) atomicOr(A.status, (unsigned long long)CB_DEV_ITER_LIMIT);
    exact_finish(A, q, mem, cls, how == cba::STOPPED, t);
  }
};

// fetch: a zeroed counter of the pairs handed out
__global__ void __launch_bounds__(128) k_ccd_exact(CcdArgs A, unsigned long long* __restrict__ fetch, int sms) {
  const int64_t mf = min((int64_t)A.nlist[0], A.np), m = min(mf + (int64_t)A.nlist[1], A.np);
  const unsigned lane = threadIdx.x & 31u;
  const int blocks = min((int)gridDim.x, sms);  // of the short form: one FP64 warp per SM quarter
  if (m <= (int64_t)blocks * FEW_PER_BLOCK) {
    if (blockIdx.x >= blocks) return;
    ExactJob J{A, mf, 0, 0, 0};
    const int most = cba::iterate16(J, m, 4 * blocks, (int)(threadIdx.x >> 5) * blocks + (int)blockIdx.x, ACCD_C, ACCD_MAX_ITER);
    const int wm = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0 && wm > 0) atomicMax(A.max_iters, (unsigned long long)wm);
    return;
  }
  const unsigned below = (1u << lane) - 1u;
  ExactLane L;
  bool have = false, drained = false;
  int max_it = 0;
  for (;;) {
    const unsigned idle = __ballot_sync(0xffffffffu, !have);
    const int nidle = __popc(idle);
    if (!drained && (nidle >= EXACT_REFILL || nidle == 32)) {
      // the group of idle lanes takes the next pairs of the list
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(fetch, (unsigned long long)nidle);
      b = __shfl_sync(0xffffffffu, b, 0);
      if ((int64_t)b + nidle >= m) drained = true;  // nothing left after this group
      const int64_t w = (int64_t)b + __popc(idle & below);
      bool take = !have && w < m;
      if (take) {
        L.q = w < mf ? A.list[w] : A.list[A.np - 1 - (w - mf)];
        const uint64_t key = A.keys[L.q];
        const int v0 = cb_key_type(key) == CB_KEY_PT ? (int)cb_key_i(key) : A.ev0[cb_key_i(key)];
        take = __double2float_rd(A.t_out[L.q]) <= member_cap(A, A.members > 1 ? A.vsc[v0] : 0);
      }
      if (take) {
        L.S = accd_start(A, L.q);
        if (L.S.lp == 0.0 || L.S.g0 <= 0.0) {  // only reachable through an FP32 bound below 1
          if (L.S.lp != 0.0) {
            atomicOr(A.status, (unsigned long long)CB_DEV_PENETRATION);
            atomicOr(macc_of(A, L.S.mem, MACC_STATUS), (unsigned long long)CB_DEV_PENETRATION);
          }
          exact_finish(A, L, false, L.S.lp == 0.0 ? 1.0 : 0.0);
        } else {
          // dropped above the member's bound (pass 2 is over: it no longer moves), or on reaching its minimum so far
          L.hi = __longlong_as_double(*macc_of(A, L.S.mem, MACC_HI));
          L.cap = __longlong_as_double(*(volatile unsigned long long*)macc_of(A, L.S.mem, MACC_ALPHA));
          L.g = xmul(ACCD_S, L.S.g0);
          L.t = 0.0;
          L.tl = xdiv(xmul(xsub(1.0, ACCD_S), L.S.g0), L.S.lp);
          L.it = 0;
          have = true;
        }
      }
    }
    if (!__any_sync(0xffffffffu, have)) {
      if (drained) break;
      continue;  // every pair of the group finished at its set-up: fetch again
    }
    if (have) {
      // one additive-CCD step
      AccdStart& S = L.S;
      S.Y0 = axpy3(S.Y0, L.tl, S.Q0);
      S.Y1 = axpy3(S.Y1, L.tl, S.Q1);
      S.Y2 = axpy3(S.Y2, L.tl, S.Q2);
      S.Y3 = axpy3(S.Y3, L.tl, S.Q3);
      double d;
      cbt::stencil_distance(S.ee, S.Y0, S.Y1, S.Y2, S.Y3, d);
      const int it = L.it++;
      if (L.t > 0.0 && xsub(d, S.off) < L.g) {
        exact_finish(A, L, false, L.t);
        have = false;
      } else {
        L.t = xadd(L.t, L.tl);
        if (L.t > 1.0) {
          exact_finish(A, L, false, 1.0);
          have = false;
        } else {
          if ((it & 7) == 7)
            L.cap = __longlong_as_double(*(volatile unsigned long long*)macc_of(A, S.mem, MACC_ALPHA));
          if ((L.cap < 1.0 && L.t >= L.cap) || L.t > L.hi) {  // t_p >= t: this pair cannot lower the minimum
            exact_finish(A, L, true, L.t);
            have = false;
          } else if (it + 1 >= ACCD_MAX_ITER) {
            atomicOr(A.status, (unsigned long long)CB_DEV_ITER_LIMIT);
            exact_finish(A, L, false, L.t);
            have = false;
          } else {
            L.tl = xdiv(xmul(ACCD_C, xsub(d, S.off)), S.lp);
          }
        }
      }
      if (!have) max_it = max(max_it, it + 1);
    }
  }
  const int wm = __reduce_max_sync(0xffffffffu, max_it);
  if (lane == 0 && wm > 0) atomicMax(A.max_iters, (unsigned long long)wm);
}

__global__ void k_alpha_final(int count, const unsigned long long* __restrict__ macc, double* __restrict__ out) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < count) out[m] = __longlong_as_double(macc[(size_t)m * MACC_STRIDE + MACC_ALPHA]);
}
// One launch for the resets at the start of a step bound: its counters and
// every member's minimum, bound and status.
__global__ void k_ccd_reset(unsigned long long* __restrict__ sc, int count, unsigned long long* __restrict__ macc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) sc[SC_ITERS] = sc[SC_NLIST] = sc[SC_NU] = sc[SC_NX] = sc[SC_FETCH] = 0ull;
  if (i < count) {
    unsigned long long* m = macc + (size_t)i * MACC_STRIDE;
    m[MACC_ALPHA] = m[MACC_HI] = 0x3ff0000000000000ull;  // 1.0
    m[MACC_STATUS] = 0ull;
  }
}

}  // namespace

cb_status ccd_run(cb_scene* s, const double* x, const double* p, double* alpha, cudaStream_t st) {
  CB_TRY(broad_phase(s, s->bwc, x, p, true, false, s->ccd_keys, &s->ccd_cls, &s->n_ccd, st));
  uint64_t* sc = scalars(s);
  const int M = s->count;
  unsigned long long* macc = bp<unsigned long long>(s->macc);
  unsigned long long* mi = (unsigned long long*)(sc + SC_ITERS);
  k_ccd_reset<<<cb_grid(M), CB_THREADS, 0, cb_count(st)>>>((unsigned long long*)sc, M, macc);
  const int64_t np = s->n_ccd;
  if (np > 0) {
    CB_TRY(buf_ensure(s->ccd_t, sizeof(double) * (size_t)np, st));
    CB_TRY(buf_ensure(s->ccd_list, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(s->ccd_ulist, sizeof(uint32_t) * (size_t)np, st));
    CB_TRY(buf_ensure(s->dlist, sizeof(uint32_t) * (size_t)np, st));
    CcdArgs A;
    A.np = np;
    A.keys = bp<uint64_t>(s->ccd_keys);
    A.ev0 = bp<int32_t>(s->ev0);
    A.ev1 = bp<int32_t>(s->ev1);
    A.tv = bp<int32_t>(s->tv);
    A.T = s->T;
    A.n = s->n;
    A.vsc = bp<int32_t>(s->vsc);
    A.mp = bp<MemberParams>(s->mp);
    A.cx = bp<double>(s->bwc.cx);
    A.x = x;
    A.p = p;
    A.t_out = bp<double>(s->ccd_t);
    A.cls_out = bp<uint8_t>(s->ccd_cls);
    A.macc = macc;
    A.members = M;
    A.status = (unsigned long long*)(sc + SC_STATUS);
    A.max_iters = mi;
    CB_TRY(to_f32(s, x, bp<double>(s->bwc.cx), s->xf, st));
    CB_TRY(to_f32(s, p, nullptr, s->pf, st));
    A.xf = bp<float4>(s->xf);
    A.pf = bp<float4>(s->pf);
    unsigned int* nl = (unsigned int*)(sc + SC_NLIST);
    A.ulist = bp<uint32_t>(s->ccd_ulist);
    A.nu = (unsigned int*)(sc + SC_NU);
    A.list = bp<uint32_t>(s->ccd_list);
    A.nlist = (unsigned int*)(sc + SC_NX);
    k_ccd_screen<<<cb_grid(np, 128), 128, 0, cb_count(st)>>>(A, bp<uint32_t>(s->dlist), nl);
    k_ccd_bound<<<std::min<int64_t>(cb_grid(np, 128), (int64_t)s->n_sms * 16), 128, 0, cb_count(st)>>>(
        A, bp<uint32_t>(s->dlist), nl);
    k_ccd_refine<<<std::min<int64_t>(cb_grid(np, 128), (int64_t)s->n_sms * 16), 128, 0, cb_count(st)>>>(A);
    // persistent warps: at most three 128-thread blocks per SM (the kernel's registers); a block has eight half-warps
    k_ccd_exact<<<std::min<int64_t>(cb_grid(np, 8), (int64_t)s->n_sms * 3), 128, 0, cb_count(st)>>>(
        A, (unsigned long long*)(sc + SC_FETCH), s->n_sms);
    CB_CUDA(cudaGetLastError());
  }
  if (alpha) k_alpha_final<<<cb_grid(M), CB_THREADS, 0, cb_count(st)>>>(M, macc, alpha);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}

// ---------------------------------------------------------------------------
// ccd_step_noalloc: the same additive-CCD step bound over a caller-given list
// of stencils, with no device allocation at all.
//
// Some callers cannot allocate device memory while they run the step bound: a
// solver that has handed a fixed budget of the device to a memory pool, or a
// time-critical loop where an allocation or a free could stall the device.
// For them every buffer this call needs is the one array below, allocated when
// the library's code is loaded onto a device.  The first call on each device
// looks up its address (and may make the CUDA runtime load this code onto that
// device), so it should come before any stream capture.  The array is shared
// by every call on a device: calls that overlap in time on one device (two
// streams, two host threads) race and give wrong results.
//
// Layout: NA_SLOTS 64-bit accumulator words (alpha bits, smallest upper bound
// bits, condition flags, list lengths), then per stencil an FP32 lower bound
// and a list entry (the stencils left for the FP64 iteration: point-triangle
// from the front, edge-edge from the back).

namespace {
constexpr int NA_SLOTS = 32;  // 256 bytes: keeps the per-stencil part 256-byte aligned
constexpr int NA_ALPHA = 0, NA_HI = 1, NA_FLAGS = 2, NA_COUNT = 3;  // NA_COUNT: two uint32
constexpr unsigned long long NA_ONE = 0x3ff0000000000000ull;  // 1.0
}  // namespace

static __device__ __align__(256) unsigned long long g_noalloc_scratch[NA_SLOTS + CB_NOALLOC_MAX_STENCILS];

namespace {

struct NaArgs {
  int64_t ns;
  int n;
  const int32_t* __restrict__ st;   // [ns][4] vertex ids
  const uint8_t* __restrict__ ee;   // [ns] 1 edge-edge, 0 point-triangle
  const double* __restrict__ off;   // [ns] offset
  const double* __restrict__ x;
  const double* __restrict__ p;
  unsigned long long* scr;
};

__device__ __forceinline__ float* na_lb(const NaArgs& A) { return (float*)(A.scr + NA_SLOTS); }
__device__ __forceinline__ uint32_t* na_list(const NaArgs& A) {
  return (uint32_t*)(A.scr + NA_SLOTS) + CB_NOALLOC_MAX_STENCILS;
}
// an upper bound of the smallest t_p: FP32 brackets and exact values so far (rounded up)
__device__ __forceinline__ float na_cap(const NaArgs& A) {
  const volatile unsigned long long* s = A.scr;
  return __double2float_ru(fmin(__longlong_as_double(s[NA_ALPHA]), __longlong_as_double(s[NA_HI])));
}

struct NaStart {
  bool ee;
  double off, lp, g0;
  d3 Y0, Y1, Y2, Y3, Q0, Q1, Q2, Q3;
};

// first-step data of stencil q (the same arithmetic as accd_start); false for
// a stencil with a vertex id outside [0, n), an offset that is negative or
// not finite, or positions / displacements that make its distance or motion
// bound non-finite (such a stencil is reported, never silently passed)
__device__ __forceinline__ bool na_start(const NaArgs& A, int64_t q, NaStart& S) {
  int v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = A.st[4 * q + k];
    if (v[k] < 0 || v[k] >= A.n) return false;
  }
  S.ee = A.ee[q] != 0;
  S.off = A.off[q];
  if (!(S.off >= 0.0) || !isfinite(S.off)) return false;
  const d3 X0 = ld(A.x, A.n, v[0]), X1 = ld(A.x, A.n, v[1]), X2 = ld(A.x, A.n, v[2]), X3 = ld(A.x, A.n, v[3]);
  const d3 P0 = ld(A.p, A.n, v[0]), P1 = ld(A.p, A.n, v[1]), P2 = ld(A.p, A.n, v[2]), P3 = ld(A.p, A.n, v[3]);
  double d;
  cbt::stencil_distance(S.ee, X0, X1, X2, X3, d);
  const d3 pb = mk3(xmul(xadd(xadd(xadd(P0.x, P1.x), P2.x), P3.x), 0.25),
                    xmul(xadd(xadd(xadd(P0.y, P1.y), P2.y), P3.y), 0.25),
                    xmul(xadd(xadd(xadd(P0.z, P1.z), P2.z), P3.z), 0.25));
  S.Y0 = sub3(X0, X0);
  S.Y1 = sub3(X1, X0);
  S.Y2 = sub3(X2, X0);
  S.Y3 = sub3(X3, X0);
  S.Q0 = sub3(P0, pb);
  S.Q1 = sub3(P1, pb);
  S.Q2 = sub3(P2, pb);
  S.Q3 = sub3(P3, pb);
  const double n0 = norm3(S.Q0), n1 = norm3(S.Q1), n2 = norm3(S.Q2), n3 = norm3(S.Q3);
  // fmax drops a NaN operand, so a non-finite displacement is caught from the norms themselves
  if (!isfinite(n0) || !isfinite(n1) || !isfinite(n2) || !isfinite(n3) || !isfinite(d)) return false;
  S.lp = S.ee ? xadd(fmax(n0, n1), fmax(n2, n3)) : xadd(n0, fmax(fmax(n1, n2), n3));
  S.g0 = (S.lp != 0.0) ? xsub(d, S.off) : 0.0;
  return isfinite(S.lp) && isfinite(S.g0);
}

__global__ void k_na_init(unsigned long long* __restrict__ scr) {
  if (threadIdx.x == 0) {
    scr[NA_ALPHA] = scr[NA_HI] = NA_ONE;
    scr[NA_FLAGS] = scr[NA_COUNT] = 0ull;
  }
}

// FP32 brackets of the stencils' t_p (accd32.cuh), in two launches: every
// NA_SAMPLE-th stencil first, so that the rest meet an upper bound that already
// drops most of them after their first step.  The stencils still below it are
// listed.  Grid-stride; the trip count is uniform over a warp so that every
// lane reaches the appends.
constexpr int NA_SAMPLE = 16;

__global__ void __launch_bounds__(128) k_na_refine(NaArgs A, int part) {
  const int64_t ns = A.ns, head = (ns + NA_SAMPLE - 1) / NA_SAMPLE, m = part == 0 ? head : ns - head;
  unsigned int* cnt = (unsigned int*)&A.scr[NA_COUNT];
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x; w0 < m; w0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = w0 + threadIdx.x;
    bool keep = false, ee = false;
    // part 1: the w-th stencil that is not a multiple of NA_SAMPLE
    const int64_t q = part == 0 ? w * NA_SAMPLE : w + w / (NA_SAMPLE - 1) + 1;
    if (w < m) {
      int v[4];
      bool ok = true;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = A.st[4 * q + k];
        ok = ok && v[k] >= 0 && v[k] < A.n;
      }
      const double off = A.off[q];
      if (!ok || !(off >= 0.0) || !isfinite(off)) {
        atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_NOALLOC_BAD_STENCIL);
      } else {
        ee = A.ee[q] != 0;
        cbb::Motion32 M;
        M.ee = ee;
        M.off_dn = __double2float_rd(off);
        M.off_up = __double2float_ru(off);
        pair_motion32(A.x, A.p, A.n, v, M);
        float lo = 0.f, hi = 1.f;
        const int r = cbb::motion_slopes(M) ? cbb::accd_bounds32(M, [&] { return na_cap(A); }, lo, hi) : -1;
        if (r == 0 && hi < 1.f) atomicMin(&A.scr[NA_HI], (unsigned long long)__double_as_longlong((double)hi));
        keep = r < 0 || (r == 0 && lo <= na_cap(A));
        if (keep) na_lb(A)[q] = r < 0 ? 0.f : lo;
      }
    }
    warp_append(keep && !ee, (uint32_t)q, na_list(A), &cnt[0]);
    warp_append_back(keep && ee, (uint32_t)q, na_list(A), ns, &cnt[1]);
  }
}

// full additive CCD of stencil q (the iteration of k_ccd_exact), dropped once
// t is above the smallest upper bound or reaches the smallest exact t_p
__device__ double na_iterate(const NaArgs& A, int64_t q) {
  NaStart S;
  if (!na_start(A, q, S)) {
    atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_NOALLOC_BAD_STENCIL);
    return 1.0;
  }
  if (S.lp == 0.0) return 1.0;
  if (S.g0 <= 0.0) {
    atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_DEV_PENETRATION);
    return 0.0;
  }
  const volatile unsigned long long* scr = A.scr;
  const double top = __longlong_as_double(scr[NA_HI]);  // no longer moves
  const double g = xmul(ACCD_S, S.g0);
  double t = 0.0, d, cap = __longlong_as_double(scr[NA_ALPHA]);
  double tl = xdiv(xmul(xsub(1.0, ACCD_S), S.g0), S.lp);
  for (int it = 0; it < ACCD_MAX_ITER; ++it) {
    S.Y0 = axpy3(S.Y0, tl, S.Q0);
    S.Y1 = axpy3(S.Y1, tl, S.Q1);
    S.Y2 = axpy3(S.Y2, tl, S.Q2);
    S.Y3 = axpy3(S.Y3, tl, S.Q3);
    cbt::stencil_distance(S.ee, S.Y0, S.Y1, S.Y2, S.Y3, d);
    if (t > 0.0 && xsub(d, S.off) < g) return t;
    t = xadd(t, tl);
    if (t > 1.0) return 1.0;
    if ((it & 7) == 7) cap = __longlong_as_double(scr[NA_ALPHA]);
    if (t > top || (cap < 1.0 && t >= cap)) return 1.0;  // t_p >= t: cannot lower the minimum
    tl = xdiv(xmul(ACCD_C, xsub(d, S.off)), S.lp);
  }
  atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_DEV_ITER_LIMIT);
  return t;
}

// a short list: half a warp per stencil (accd16.cuh)
struct NaJob {
  const NaArgs& A;
  int64_t mf;
  int64_t q;

  __device__ __forceinline__ int64_t pair(int64_t w) const { return w < mf ? na_list(A)[w] : na_list(A)[A.ns - 1 - (w - mf)]; }
  __device__ __forceinline__ bool bad() const {
    if (cba::half_leader()) atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_NOALLOC_BAD_STENCIL);
    return false;
  }
  __device__ __forceinline__ int wanted(int64_t w) const { return na_lb(A)[pair(w)] <= na_cap(A); }
  __device__ __forceinline__ bool load(int64_t w, cba::Pair16& S) {
    q = pair(w);
    // (listed: its vertex ids and offset are in order)
    const int v = A.st[4 * q + cba::quad_vertex()];
    S.off = A.off[q];
    return cba::load16(A.x, A.p, A.n, v, A.ee[q] != 0, S) || bad();
  }
  __device__ __forceinline__ bool begin(cba::Pair16& S, double d) {
    const double g0 = S.lp != 0.0 ? xsub(d, S.off) : 0.0;
    if (!isfinite(d) || !isfinite(S.lp) || !isfinite(g0)) return bad();
    if (S.lp == 0.0) return false;
    if (g0 <= 0.0) {
      if (cba::half_leader()) atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_DEV_PENETRATION);
      done(S, 0.0, cba::REACHED);
      return false;
    }
    S.hi = __longlong_as_double(A.scr[NA_HI]);  // no longer moves
    S.g = xmul(ACCD_S, g0);
    S.tl = xdiv(xmul(xsub(1.0, ACCD_S), g0), S.lp);
    return true;
  }
  __device__ __forceinline__ double cap() const {
    return __longlong_as_double(*(const volatile unsigned long long*)&A.scr[NA_ALPHA]);
  }
  __device__ __forceinline__ void done(const cba::Pair16&, double t, cba::Done how) const {
    if (!cba::half_leader()) return;
    if (how == cba::LIMIT) atomicOr(&A.scr[NA_FLAGS], (unsigned long long)CB_DEV_ITER_LIMIT);
    if (how != cba::STOPPED && t < 1.0) atomicMin(&A.scr[NA_ALPHA], (unsigned long long)__double_as_longlong(t));
  }
};

// the listed stencils whose lower bound is still not above the bound; every
// other stencil has t_p above it, so alpha = min(1, m) exactly
__global__ void __launch_bounds__(128) k_na_exact(NaArgs A, int sms) {
  const unsigned int* cnt = (const unsigned int*)&A.scr[NA_COUNT];
  const int64_t mf = min((int64_t)cnt[0], A.ns), m = min(mf + (int64_t)cnt[1], A.ns);
  const int blocks = min((int)gridDim.x, sms);
  if (m <= (int64_t)blocks * FEW_PER_BLOCK) {
    if (blockIdx.x >= blocks) return;
    NaJob J{A, mf, 0};
    cba::iterate16(J, m, 4 * blocks, (int)(threadIdx.x >> 5) * blocks + (int)blockIdx.x, ACCD_C, ACCD_MAX_ITER);
    return;
  }
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < m; w += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t q = w < mf ? na_list(A)[w] : na_list(A)[A.ns - 1 - (w - mf)];
    if (!(na_lb(A)[q] <= na_cap(A))) continue;
    const double t = na_iterate(A, q);
    if (t < 1.0) atomicMin(&A.scr[NA_ALPHA], (unsigned long long)__double_as_longlong(t));
  }
}

__global__ void k_na_final(const unsigned long long* __restrict__ scr, double* __restrict__ alpha,
                           uint32_t* __restrict__ flags) {
  if (threadIdx.x == 0) {
    *alpha = __longlong_as_double(scr[NA_ALPHA]);
    *flags = (uint32_t)scr[NA_FLAGS];
  }
}

constexpr int NA_MAX_DEVICES = 256;
std::mutex g_na_mutex;
unsigned long long* g_na_ptr[NA_MAX_DEVICES];
int g_na_sms[NA_MAX_DEVICES];

// address of the scratch array on the current device and the device's SM
// count, looked up once per device (valid until the device is reset)
cb_status na_scratch(int* dev_out, unsigned long long** out, int* sms) {
  int dev = -1;
  CB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= NA_MAX_DEVICES) return CB_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_na_mutex);
  if (!g_na_ptr[dev]) {
    void* ptr = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr) {
      fprintf(stderr, "contact: ccd_step_noalloc: scratch address lookup failed on device %d: %s\n", dev,
              cudaGetErrorString(e));
      return CB_ERR_CUDA;
    }
    int nsm = 0;
    CB_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    g_na_sms[dev] = nsm > 0 ? nsm : 1;
    g_na_ptr[dev] = (unsigned long long*)ptr;
  }
  *dev_out = dev;
  *out = g_na_ptr[dev];
  *sms = g_na_sms[dev];
  return CB_OK;
}

// true if p is device memory of `dev` or managed memory; a host pointer or
// memory of another device is rejected before any kernel dereferences it
bool na_on_device(const void* p, int dev) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();  // clear the sticky-free error of an unknown pointer
    return false;
  }
  if (at.type == cudaMemoryTypeManaged) return true;
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

}  // namespace

cb_status ccd_step_noalloc(const double* x_dev, const double* p_dev, int32_t n_verts, const int32_t* stencils_dev,
                           const uint8_t* is_ee_dev, const double* offset_dev, int64_t n_stencils,
                           double* alpha_dev, uint32_t* flags_dev, void* stream) {
  if (!alpha_dev || !flags_dev || n_verts < 0 || n_stencils < 0) return CB_ERR_ARG;
  if (n_stencils > CB_NOALLOC_MAX_STENCILS) {
    fprintf(stderr, "contact: ccd_step_noalloc: %lld stencils exceed the fixed maximum of %d per call\n",
            (long long)n_stencils, (int)CB_NOALLOC_MAX_STENCILS);
    return CB_ERR_TOO_LARGE;
  }
  if (n_stencils > 0 && (n_verts < 1 || !x_dev || !p_dev || !stencils_dev || !is_ee_dev || !offset_dev))
    return CB_ERR_ARG;
  unsigned long long* scr = nullptr;
  int dev = -1, nsm = 1;
  CB_TRY(na_scratch(&dev, &scr, &nsm));
  if (!na_on_device(alpha_dev, dev) || !na_on_device(flags_dev, dev)) return CB_ERR_ARG;
  if (n_stencils > 0 && (!na_on_device(x_dev, dev) || !na_on_device(p_dev, dev) ||
                         !na_on_device(stencils_dev, dev) || !na_on_device(is_ee_dev, dev) ||
                         !na_on_device(offset_dev, dev)))
    return CB_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  k_na_init<<<1, 32, 0, cb_count(st)>>>(scr);
  if (n_stencils > 0) {
    NaArgs A;
    A.ns = n_stencils;
    A.n = n_verts;
    A.st = stencils_dev;
    A.ee = is_ee_dev;
    A.off = offset_dev;
    A.x = x_dev;
    A.p = p_dev;
    A.scr = scr;
    // grid-stride over the list: up to 8 (FP32) and 4 (FP64) resident blocks of 128 threads per SM
    const int64_t g = cb_grid(n_stencils, 128);
    const int g32 = (int)std::min<int64_t>(g, (int64_t)nsm * 8);
    k_na_refine<<<g32, 128, 0, cb_count(st)>>>(A, 0);
    k_na_refine<<<g32, 128, 0, cb_count(st)>>>(A, 1);
    k_na_exact<<<(int)std::min<int64_t>(cb_grid(n_stencils, 8), (int64_t)nsm * 4), 128, 0, cb_count(st)>>>(A, nsm);
  }
  k_na_final<<<1, 32, 0, cb_count(st)>>>(scr, alpha_dev, flags_dev);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}
