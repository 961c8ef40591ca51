// narrow.cu -- stages (b), (c), (d): barrier filter, distances, barrier energy,
// gradient and PSD-projected Hessian, assembly into a global gradient and BSR.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "bound32.cuh"
#include "geometry.cuh"
#include "pairhess.cuh"
#include "pairs.cuh"
#include "prims.cuh"
#include "scene.cuh"
#include "typed.cuh"

namespace {


// ------------------------------------------------------------------ (b) ----

// rods: arc length S at every vertex, summed sequentially along each polyline
__global__ void k_arclength(int n_rods, const int32_t* __restrict__ rod_ptr, const double* __restrict__ rest, int n,
                            double* __restrict__ S) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rods) return;
  const int s = rod_ptr[r], e = rod_ptr[r + 1];
  if (e <= s) return;
  S[s] = 0.0;
  for (int v = s + 1; v < e; ++v) {
    double dx = xsub(rest[v], rest[v - 1]);
    double dy = xsub(rest[(size_t)n + v], rest[(size_t)n + v - 1]);
    double dz = xsub(rest[2 * (size_t)n + v], rest[2 * (size_t)n + v - 1]);
    S[v] = xadd(S[v - 1], __dsqrt_rn(xadd(xadd(xmul(dx, dx), xmul(dy, dy)), xmul(dz, dz))));
  }
}

// rods: for edge k the last edge l of the same polyline with arc-length gap
// s0(l) - s1(k) < a (the reference distance between the edges; it grows with
// l), win[k]; on a closed loop also the first edge l past that window whose
// gap the other way round, (L - s1(l)) + s0(k), is below a (it shrinks as l
// grows), wst[k] (-1 if none).  An edge spans arc lengths s0 = S[v0] to s1 =
// S[v1], the closing edge of a loop from S at the last vertex to the loop
// length L.  The reference distance of a pair is the smaller gap; incident
// pairs (a shared vertex) are skipped.
__device__ __forceinline__ double edge_len(const double* __restrict__ rest, int n, int a, int b) {
  const double dx = xsub(rest[b], rest[a]);
  const double dy = xsub(rest[(size_t)n + b], rest[(size_t)n + a]);
  const double dz = xsub(rest[2 * (size_t)n + b], rest[2 * (size_t)n + a]);
  return __dsqrt_rn(xadd(xadd(xmul(dx, dx), xmul(dy, dy)), xmul(dz, dz)));
}

__global__ void k_rod_window(int E, const int32_t* __restrict__ ev0, const int32_t* __restrict__ ev1,
                             const int32_t* __restrict__ comp, const double* __restrict__ S,
                             const double* __restrict__ rest, int n, const int32_t* __restrict__ rlast, double a,
                             int32_t* __restrict__ win, int32_t* __restrict__ wst,
                             unsigned long long* __restrict__ dmin_bits, unsigned long long* __restrict__ nfilt,
                             unsigned long long* __restrict__ dmin_comp) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= E) return;
  const int k0 = ev0[k], k1 = ev1[k];
  const int rl = rlast[k];
  const double s0k = S[k0];
  const double s1k = k1 > k0 ? S[k1] : xadd(S[k0], edge_len(rest, n, k0, k1));
  // closed loop: its length, and the gap the other way round to edge l
  const bool loop = rl >= 0 && k < rl;
  const double L = loop ? xadd(S[ev0[rl]], edge_len(rest, n, ev0[rl], ev1[rl])) : 0.0;
  auto back_gap = [&](int l) {
    const double s1l = l == rl ? L : S[ev1[l]];
    return xadd(xsub(L, s1l), s0k);
  };
  auto incident = [&](int l) {
    const int l0 = ev0[l], l1 = ev1[l];
    return l0 == k0 || l0 == k1 || l1 == k0 || l1 == k1;
  };
  int last = k + 1;
  double mn = INFINITY;
  unsigned long long cnt = 0;
  for (int l = k + 1; l < E; ++l) {
    const int l0 = ev0[l];
    if (comp[l0] != comp[k1]) break;
    if (incident(l)) continue;
    const double dbar = xsub(S[l0], s1k);
    if (!(dbar < a)) break;
    last = l;
    mn = fmin(mn, loop ? fmin(dbar, back_gap(l)) : dbar);
    ++cnt;
  }
  win[k] = last;
  int first = -1;
  if (loop) {
    for (int l = rl; l > last && l > k; --l) {
      if (incident(l)) continue;
      const double g = back_gap(l);
      if (!(g < a)) break;
      first = l;
      mn = fmin(mn, g);
      ++cnt;
    }
  }
  wst[k] = first;
  if (cnt) {
    atomicMin(dmin_bits, (unsigned long long)__double_as_longlong(mn));
    atomicMin(&dmin_comp[comp[k1]], (unsigned long long)__double_as_longlong(mn));
    atomicAdd(nfilt, cnt);
  }
}

// shells: rest candidates of one component whose rest distance is below a
__global__ void k_rest_filter(int64_t nc, const uint64_t* __restrict__ keys, const int32_t* __restrict__ ev0,
                              const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv, int T,
                              const int32_t* __restrict__ comp, const double* __restrict__ rest, int n, double a,
                              uint32_t* __restrict__ flag, double* __restrict__ dbar,
                              unsigned long long* __restrict__ dmin_bits,
                              unsigned long long* __restrict__ dmin_comp) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long mb = 0x7ff0000000000000ull;  // +inf: no filtered pair in this lane
  if (c < nc) {
    Stencil s = stencil_of(keys[c], ev0, ev1, tv, T);
    uint32_t f = 0;
    double d = 0.0;
    if (comp[s.v[0]] == comp[s.v[2]]) {
      cbg::stencil_distance(s.ee, load3(rest, n, s.v[0]), load3(rest, n, s.v[1]), load3(rest, n, s.v[2]),
                            load3(rest, n, s.v[3]), d);
      if (d < a) {
        f = 1;
        mb = (unsigned long long)__double_as_longlong(d);
        atomicMin(&dmin_comp[comp[s.v[0]]], mb);
      }
    }
    flag[c] = f;
    dbar[c] = d;
  }
  // one atomicMin per warp
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = u < mb ? u : mb;
  }
  if ((threadIdx.x & 31) == 0 && mb != 0x7ff0000000000000ull) atomicMin(dmin_bits, mb);
}

// Per-stencil activation: whether the FP64 boxes of a pair's two primitives
// (uninflated boxes of the static broad phase), each inflated by half the
// pair's own width fw, overlap on all three axes (closed intervals).
__device__ __forceinline__ bool within_own_width(const double* __restrict__ box_raw, int64_t prim1, int64_t prim2,
                                                 double fw) {
  const double h = xmul(0.5, fw);
  const double* b1 = box_raw + prim1 * 6;
  const double* b2 = box_raw + prim2 * 6;
  bool ov = true;
#pragma unroll
  for (int k = 0; k < 3; ++k) ov = ov && xsub(b1[k], h) <= xadd(b2[3 + k], h) && xsub(b2[k], h) <= xadd(b1[3 + k], h);
  return ov;
}

// class-F width of a pair whose first stencil vertex is v0 (per member:
// dbar_min, or its component's with CB_DBAR_PER_COMPONENT)
__device__ __forceinline__ double member_f_width(const MemberParams& M, const unsigned long long* __restrict__ dbar_comp,
                                                 const int32_t* __restrict__ comp, int v0) {
  return M.per_comp ? __longlong_as_double((long long)dbar_comp[comp[v0]]) : M.dbar_min;
}

// class byte of a filtered candidate dropped by the per-stencil activation
constexpr uint8_t KL_DROPPED = 0xFE;

// Per-stencil activation: the class-F candidates outside their own width take
// class KL_DROPPED (counted in ndrop); the rest are counted in nfilt.
__global__ void k_own_width(int64_t nc, const uint64_t* __restrict__ cand, const double* __restrict__ box_raw,
                            const int32_t* __restrict__ ev0, const int32_t* __restrict__ vsc,
                            const MemberParams* __restrict__ mp, const unsigned long long* __restrict__ dbar_comp,
                            const int32_t* __restrict__ comp, bool rod, int n, int T, uint8_t* __restrict__ klass,
                            unsigned long long* __restrict__ nfilt, unsigned long long* __restrict__ ndrop) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool f = false, dropped = false;
  if (c < nc && klass[c] == 1) {
    const uint64_t key = cand[c];
    const bool pt = cb_key_type(key) == CB_KEY_PT;
    const int64_t i = cb_key_i(key), j = cb_key_j(key);
    const int v0 = pt ? (int)i : ev0[i];
    const MemberParams& M = mp[vsc[v0]];
    // broad-phase primitive ids: vertices, then triangles, then edges (rods: edges)
    const int64_t p1 = pt || rod ? i : (int64_t)n + T + i, p2 = rod ? j : (pt ? (int64_t)n + j : (int64_t)n + T + j);
    dropped = M.per_stencil && !within_own_width(box_raw, p1, p2, member_f_width(M, dbar_comp, comp, v0));
    f = !dropped;
    if (dropped) klass[c] = KL_DROPPED;
  }
  uint32_t b = __ballot_sync(0xffffffffu, f);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd(nfilt, (unsigned long long)__popc(b));
  b = __ballot_sync(0xffffffffu, dropped);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd(ndrop, (unsigned long long)__popc(b));
}

// per-stencil activation: keep flags of the candidates, then the kept ones
// (keys and classes) in their order
__global__ void k_keep_flag(int64_t nc, const uint8_t* __restrict__ klass, uint32_t* __restrict__ flag) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nc) flag[c] = klass[c] != KL_DROPPED ? 1u : 0u;
}
__global__ void k_keep_write(int64_t nc, const uint64_t* __restrict__ cand, const uint8_t* __restrict__ klass,
                             const uint32_t* __restrict__ flag, const uint32_t* __restrict__ pos,
                             uint64_t* __restrict__ cand_out, uint8_t* __restrict__ klass_out) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < nc && flag[c]) {
    cand_out[pos[c]] = cand[c];
    klass_out[pos[c]] = klass[c];
  }
}

// ------------------------------------------------------------------ (c) ----

// Per-member sum of lane values: one atomic per warp when the warp holds one
// member (lanes without a value pass mem < 0), one per lane otherwise.  Every
// lane of the warp must call it.
__device__ __forceinline__ void member_energy_add(unsigned long long* __restrict__ macc, int mem, double e) {
  const int m0 = __shfl_sync(0xffffffffu, mem, 0);
  if (__all_sync(0xffffffffu, mem == m0 || mem < 0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0 && e != 0.0 && m0 >= 0)
      atomicAdd((double*)&macc[(size_t)m0 * MACC_STRIDE + MACC_E], e);
  } else if (mem >= 0 && e != 0.0) {
    atomicAdd((double*)&macc[(size_t)mem * MACC_STRIDE + MACC_E], e);
  }
}

// Warp-aggregated append of flagged lanes' values to a list.
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

// Warp-aggregated append from the end of a list of cap entries backwards.
__device__ __forceinline__ void warp_append_back(bool flag, uint32_t value, uint32_t* __restrict__ list,
                                                 int64_t cap, unsigned int* __restrict__ count) {
  const unsigned m = __ballot_sync(0xffffffffu, flag);
  if (!m) return;
  const unsigned lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  unsigned base = 0;
  if ((int)lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (flag) list[cap - 1 - (int64_t)(base + __popc(m & ((1u << lane) - 1u)))] = value;
}

// Per candidate, phase 1: an FP32 lower bound of the distance.  Candidates it
// places beyond every threshold of their class (U: a, which is above xi; F:
// dbar_min) are inactive and not class C, and nothing is written for them.
// The rest are queued for the exact
// FP64 phase, so that no warp pays for FP64 on behalf of a few lanes:
// point-triangle pairs from the start of the list (count nlist[0]), edge-edge
// pairs from its end backwards (count nlist[1]), so that the exact kernel's
// warps run one of the two distance routines.
__global__ void k_distance_screen(int64_t nc, const uint64_t* __restrict__ cand,
                                  const uint8_t* __restrict__ klass_in, const int32_t* __restrict__ ev0,
                                  const int32_t* __restrict__ ev1, const int32_t* __restrict__ tv, int T,
                                  const float4* __restrict__ xf, const double* __restrict__ cx,
                                  const int32_t* __restrict__ vsc, const MemberParams* __restrict__ mp, int n,
                                  uint32_t* __restrict__ list, unsigned int* __restrict__ nlist) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool exact = false, ee = false;
  if (c < nc) {
    Stencil s = stencil_of(cand[c], ev0, ev1, tv, T);
    ee = s.ee;
    const int k = klass_in[c];
    const int mem = vsc[s.v[0]];
    const MemberParams& M = mp[mem];
    if (k != 3) {  // (3: culled in Kaldor mode, no barrier)
      // thresholds beyond which a pair is surely inactive and not class C (the
      // 1e-9 margins cover the rounding of the FP64 decision; FP32 copies
      // rounded up, so the FP32 comparison is as safe)
      const float thr = k == 1 ? M.thrF32 : M.thrU32;
      const float X = (float)cx[4 * mem + 3];
      const float4 q0 = xf[s.v[0]], q1 = xf[s.v[1]], q2 = xf[s.v[2]], q3 = xf[s.v[3]];
      const float lb = cbb::lower_bound(s.ee, cbb::f3{q0.x, q0.y, q0.z}, cbb::f3{q1.x, q1.y, q1.z},
                                        cbb::f3{q2.x, q2.y, q2.z}, cbb::f3{q3.x, q3.y, q3.z}, X);
      exact = !(lb >= thr);
    }
  }
  warp_append(exact && !ee, (uint32_t)c, list, &nlist[0]);
  warp_append_back(exact && ee, (uint32_t)c, list, nc, &nlist[1]);
}

// phase 2: exact FP64 distance, class C and activity of the queued candidates
// (list entries [0, nlist[0]) and [cap - nlist[1], cap)).  Class-C candidates
// are listed in clist.  With ENERGY (the energy-only pass) every active pair
// adds kappa b(y) to its member's energy; otherwise the active candidates are
// listed in aidx: face / line-line pairs (the branch of k_pair_hess with the
// most FP64 work) from the front, the others from the back, so that a warp of
// that kernel runs one branch.  Appends are warp-aggregated, so the lists keep
// the candidates' order but for the arrival of warps.  (Flags, a scan and a
// compaction over all candidates made these lists before: 0.35 ms of a
// pleated 256x256 pass, 14 bytes written per candidate.)
//
// Bound by the FP64 pipe.  Each pair whose type FP32 is sure of takes one
// formula (typed.cuh); the undecided few wait in shared memory until a block's
// worth, or the rest, runs the full routine in full warps.  862k pairs of a
// pleated sheet 458 -> 292 us, of 64 rod scenes 736 -> 326, the energy-only
// pass of a 181x181 sheet 212 -> 113.  One wave of resident blocks (three per SM,
// 80 registers) instead of several of two per SM: each block ends with its
// undecided pairs' long chain only once; 292 -> 170 us and 326 -> 278.
template <bool ENERGY>
__global__ void __launch_bounds__(CB_THREADS, 3) k_distance_exact(const uint32_t* __restrict__ list, int64_t cap, const unsigned int* __restrict__ nlist,
                                 const uint64_t* __restrict__ cand, const uint8_t* __restrict__ klass_in,
                                 const int32_t* __restrict__ ev0, const int32_t* __restrict__ ev1,
                                 const int32_t* __restrict__ tv, int T, const double* __restrict__ x, int n,
                                 const int32_t* __restrict__ vsc, const MemberParams* __restrict__ mp,
                                 double* __restrict__ dout, int8_t* __restrict__ tout,
                                 uint8_t* __restrict__ cls, uint32_t* __restrict__ clist, uint32_t* __restrict__ aidx,
                                 unsigned* __restrict__ nsplit, uint32_t* __restrict__ mlist,
                                 unsigned* __restrict__ nmoll,
                                 unsigned long long* __restrict__ status, unsigned long long* __restrict__ ncore,
                                 unsigned long long* __restrict__ macc, const int32_t* __restrict__ comp,
                                 const unsigned long long* __restrict__ dbar_comp, const double* __restrict__ elen2) {
  constexpr bool energy = ENERGY;  // energy only (barrier_energy): add kappa b per active pair
  const unsigned m0 = nlist[0], m = m0 + nlist[1];
  __shared__ uint32_t unsure[2 * CB_THREADS];
  __shared__ unsigned n_unsure;
  if (threadIdx.x == 0) n_unsure = 0;
  __syncthreads();
  // block-uniform: the next CB_THREADS queued pairs, or as many of the undecided ones once enough wait (or no others are left)
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x;;) {  // (64 bits: the last step of a list near 2^32 pairs passes it)
    const unsigned nu = n_unsure;
    const bool more = w0 < m, typed = more && nu < CB_THREADS;
    if (!more && nu == 0) break;
    __syncthreads();
    bool is_core = false, active = false, plane = false, moll = false;
    uint32_t c = 0;
    double e_local = 0.0;
    int e_mem = -1;
    bool live;
    if (typed) {
      const int64_t w = w0 + threadIdx.x;
      live = w < m;
      if (live) c = w < m0 ? list[w] : list[cap - 1 - (w - m0)];
      w0 += gridDim.x * blockDim.x;
    } else {
      const unsigned take = min(nu, (unsigned)CB_THREADS);
      live = threadIdx.x < take;
      if (live) c = unsure[nu - 1 - threadIdx.x];
      __syncthreads();
      if (threadIdx.x == 0) n_unsure = nu - take;
    }
    Stencil s;
    double d = 0.0;
    int ty = -1;
    if (live) {
      s = stencil_of(cand[c], ev0, ev1, tv, T);
      const cbg::Local L = cbg::make_local(load3(x, n, s.v[0]), load3(x, n, s.v[1]), load3(x, n, s.v[2]), load3(x, n, s.v[3]));
      double d2 = 0.0;
      if (typed) {
        ty = cbt::certain_type(s.ee, cbt::to_f3(L.P1), cbt::to_f3(L.P2), cbt::to_f3(L.P3));
        if (ty >= 0) d2 = cbt::typed_d2(s.ee, L, ty);
      } else {
        ty = s.ee ? cbg::ee_type(L, d2) : cbg::pt_type(L, d2);
      }
      d = __dsqrt_rn(d2);
    }
    if (typed) {
      warp_append(live && ty < 0, c, unsure, &n_unsure);  // fewer than CB_THREADS waited: room for all
      live = live && ty >= 0;
    }
    if (live) {
      int k = klass_in[c];
      const int mem = vsc[s.v[0]];
      const PassParams P = member_pass(mp[mem]);
      if (k == 0 && P.core_temp && !P.single && d <= P.xi) k = 2;
      double xi_p, dh_p;
      pair_params(P, k, f_width(P, dbar_comp, comp, s.v[0]), xi_p, dh_p);
      const double y = xsub(d, xi_p);
      const bool act = y < dh_p;
      if (act && y <= 0.0) {
        atomicOr(status, (unsigned long long)CB_DEV_PENETRATION);
        atomicOr(&macc[(size_t)mem * MACC_STRIDE + MACC_STATUS], (unsigned long long)CB_DEV_PENETRATION);
      }
      is_core = (k == 2);
      if (!energy && act) {
        active = true;
        plane = ty == (s.ee ? 8 : 6);
        // an edge-edge pair below its mollifier's threshold: its energy, gradient and 9x9 matrix come from
        // k_moll_hess instead of k_pair_hess
        if (P.mollify && s.ee) {
          const double c2 = ee_cross2(load3(x, n, s.v[0]), load3(x, n, s.v[1]), load3(x, n, s.v[2]), load3(x, n, s.v[3]));
          moll = c2 < 1e-3 * elen2[cb_key_i(cand[c])] * elen2[cb_key_j(cand[c])];
        }
        dout[c] = d;
        tout[c] = (int8_t)ty;
        cls[c] = (uint8_t)k | (moll ? CB_CLS_MOLLIFIED : 0);
      }
      if (energy && act && y > 0.0) {
        double mf = 1.0;
        if (P.mollify && s.ee) {  // IPC's edge-edge mollifier
          const double eps = 1e-3 * elen2[cb_key_i(cand[c])] * elen2[cb_key_j(cand[c])];
          double m1, m2;
          ee_mollifier(ee_cross2(load3(x, n, s.v[0]), load3(x, n, s.v[1]), load3(x, n, s.v[2]),
                                 load3(x, n, s.v[3])),
                       eps, mf, m1, m2);
        }
        e_local = P.kappa * mf * barrier_b(y, dh_p);
        e_mem = mem;
      }
    }
    warp_append(is_core, c, clist, (unsigned*)ncore);
    if (energy) {
      member_energy_add(macc, e_mem, e_local);
    } else {
      warp_append(active && plane, c, aidx, &nsplit[0]);
      warp_append_back(active && !plane, c, aidx, cap, &nsplit[1]);
      if (mlist) warp_append(moll, c, mlist, nmoll);
    }
    __syncthreads();
  }
}

// FP32 copy of a [3][n] FP64 vector, minus the member centre when cx is
// given, one float4 (x, y, z, 0) per vertex: the screens gather a vertex's
// three components in one 16-byte load
__global__ void k_to_f32(int n, const double* __restrict__ v, const double* __restrict__ cx,
                         const int32_t* __restrict__ vsc, float4* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* c = cx ? cx + 4 * vsc[i] : nullptr;
  out[i] = make_float4((float)(v[i] - (c ? c[0] : 0.0)), (float)(v[(size_t)n + i] - (c ? c[1] : 0.0)),
                       (float)(v[2 * (size_t)n + i] - (c ? c[2] : 0.0)), 0.f);
}

// ------------------------------------------------------------------ (d) ----

// The BSR pattern: the distinct (row, column) of the 16 blocks of every active
// stencil, columns ascending in each row, without sorting the keys: each run of
// BK_PAIRS active pairs makes its blocks distinct in shared memory
// (k_block_keys), the survivors are bucketed by row (counts, scan, k_row_fill),
// and each row's short bucket is made distinct and sorted by a warp
// (k_row_unique; a block for buckets past ROW_MAX, k_row_unique_long; those past
// ROW_BLOCK_MAX go through a radix sort together, huge_rows).  On a
// pleated 256x256 pass (862k active pairs, 1.7M blocks) the keys take 0.11 ms,
// fill, unique and write 0.16; a set of 4,096 keys per run and a radix sort of
// the survivors (five digits) with its flags and scans took 0.18 and 0.75.
//
// A run of active pairs (in candidate order, i.e. tile by tile) shares most of
// its vertices, so its 4 x BK_PAIRS vertices become few local numbers through
// an open-addressing set (linear probing, at most half full) and the blocks
// bits of a local adjacency matrix.  A run with more than BK_VERTS vertices
// appends all its blocks as they are: the rows' unique pass removes the rest.
constexpr int BK_PAIRS = 256;
constexpr int BK_SLOTS = 2048;  // 2 x 4 vertices x BK_PAIRS
constexpr int BK_VERTS = 512;
constexpr int BK_WORDS = BK_VERTS / 32;
constexpr int BK_SMEM = (BK_SLOTS + BK_VERTS + BK_VERTS * BK_WORDS) * 4 + BK_SLOTS * 2;

__global__ void __launch_bounds__(BK_PAIRS) k_block_keys(ActiveList act, const uint64_t* __restrict__ cand,
                                                         const int32_t* __restrict__ ev0,
                                                         const int32_t* __restrict__ ev1,
                                                         const int32_t* __restrict__ tv, int T,
                                                         uint2* __restrict__ bkey, unsigned int* __restrict__ m_out,
                                                         uint32_t* __restrict__ row_cnt) {
  extern __shared__ int bk_smem[];
  int* key = bk_smem;                               // [BK_SLOTS] vertex (-1: empty)
  int* vert = key + BK_SLOTS;                       // [BK_VERTS] vertex of each local number
  uint32_t* adj = (uint32_t*)(vert + BK_VERTS);     // [BK_VERTS][BK_WORDS]
  uint16_t* loc = (uint16_t*)(adj + BK_VERTS * BK_WORDS);  // [BK_SLOTS] local number
  __shared__ unsigned nv_s, wsum[BK_PAIRS / 32], base_s;
  const int tid = threadIdx.x;
  const int64_t a = (int64_t)blockIdx.x * BK_PAIRS + tid;
  for (int k = tid; k < BK_SLOTS; k += BK_PAIRS) key[k] = -1;
  if (tid == 0) nv_s = 0;
  __syncthreads();
  Stencil s;
  int slot[4];
  if (a < act.n) {
    s = stencil_of(cand[act.at(a)], ev0, ev1, tv, T);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // Fibonacci hashing (multiplicative, Knuth): the top bits of v x 2^32/phi
      unsigned h = ((unsigned)s.v[i] * 0x9E3779B1u) >> 21;
      for (int probe = 0; probe < BK_SLOTS; ++probe) {
        const int prev = atomicCAS(&key[h], -1, s.v[i]);
        if (prev == -1 || prev == s.v[i]) break;
        h = (h + 1) & (BK_SLOTS - 1);
      }
      slot[i] = (int)h;
    }
  }
  __syncthreads();
  for (int k = tid; k < BK_SLOTS; k += BK_PAIRS)
    if (key[k] >= 0) {
      const unsigned id = atomicAdd(&nv_s, 1u);
      loc[k] = (uint16_t)id;
      if (id < BK_VERTS) vert[id] = key[k];
    }
  __syncthreads();
  const unsigned nv = nv_s;
  const unsigned lane = tid & 31, wid = tid >> 5;
  const bool raw = nv > BK_VERTS;
  const unsigned words = (nv + 31) / 32;
  if (!raw) {
    for (unsigned k = tid; k < nv * BK_WORDS; k += BK_PAIRS) adj[k] = 0u;
    __syncthreads();
    if (a < act.n) {
      unsigned l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) l[i] = loc[slot[i]];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicOr(&adj[l[i] * BK_WORDS + (l[j] >> 5)], 1u << (l[j] & 31));
    }
    __syncthreads();
  }
  // this thread's blocks: local rows 2 tid and 2 tid + 1, or its stencil's 16
  unsigned c = raw ? (a < act.n ? 16u : 0u) : 0u, cr[2] = {0u, 0u};
  if (!raw)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const unsigned r = 2 * tid + q;
      if (r >= nv) continue;
      for (unsigned w = 0; w < words; ++w) cr[q] += (unsigned)__popc(adj[r * BK_WORDS + w]);
      c += cr[q];
    }
  unsigned incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
    if ((int)lane >= o) incl += v;
  }
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  unsigned woff = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < BK_PAIRS / 32; ++w) {
    woff += (w < (int)wid) ? wsum[w] : 0u;
    tot += wsum[w];
  }
  if (tid == 0) base_s = tot ? atomicAdd(m_out, tot) : 0u;
  __syncthreads();
  size_t pos = (size_t)base_s + woff + incl - c;
  if (raw) {
    if (a < act.n) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        atomicAdd(&row_cnt[s.v[i]], 4u);
#pragma unroll
        for (int j = 0; j < 4; ++j) bkey[pos++] = make_uint2((uint32_t)s.v[i], (uint32_t)s.v[j]);
      }
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const unsigned r = 2 * tid + q;
    if (r >= nv) continue;
    const uint32_t row = (uint32_t)vert[r];
    atomicAdd(&row_cnt[row], cr[q]);
    for (unsigned w = 0; w < words; ++w)
      for (uint32_t bits = adj[r * BK_WORDS + w]; bits; bits &= bits - 1u)
        bkey[pos++] = make_uint2(row, (uint32_t)vert[32 * w + __ffs((int)bits) - 1]);
  }
}

// The columns of the keys into their rows' buckets.  A run's keys of one row
// are neighbours, so one lane reserves the places of all of a row's keys in its
// warp: an atomic with a returned value per key, to places scattered over the
// buckets, had bound the kernel (pleated 256x256 124 -> 64 us, 64 rod scenes
// 96 -> 50, two stacked layers 25 -> 7).
__global__ void k_row_fill(const uint2* __restrict__ bkey, const unsigned int* __restrict__ m_in,
                           const uint32_t* __restrict__ off, uint32_t* __restrict__ cursor, uint32_t* __restrict__ rcol) {
  const unsigned full = 0xffffffffu;
  const int64_t m = *m_in;
  const int lane = threadIdx.x & 31;
  for (int64_t w0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; w0 < m; w0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = w0 + lane;
    const uint2 k = i < m ? bkey[i] : make_uint2(full, 0u);
    const uint32_t before = __shfl_up_sync(full, k.x, 1);
    const unsigned heads = __ballot_sync(full, lane == 0 || before != k.x);
    const int head = 31 - __clz((int)(heads & (full >> (31 - lane))));
    const unsigned rest = heads & ~(full >> (31 - lane));
    uint32_t at = 0;
    if (head == lane && i < m) at = off[k.x] + atomicAdd(&cursor[k.x], (unsigned)((rest ? __ffs((int)rest) - 1 : 32) - lane));
    at = __shfl_sync(full, at, head);
    if (i < m) rcol[at + (uint32_t)(lane - head)] = k.y;
  }
}

// Ascending bitonic sort of len values at p by `threads` threads of one warp or
// block (sync() between steps): each merge starts by comparing mirrored pairs,
// so every exchange puts the smaller value first and values past the end (as
// if infinite) never move.
template <typename Sync>
__device__ __forceinline__ void sort_segment(uint32_t* p, unsigned len, unsigned tid, unsigned threads, Sync sync) {
  unsigned size = 2;
  for (;; size <<= 1) {
    for (unsigned half = size >> 1, first = 1; half > 0; half >>= 1, first = 0) {
      // pair t of this step: the t-th index whose bit `half` is clear, and its partner
      const unsigned pairs = (len + 2 * half - 1) / (2 * half) * half;
      for (unsigned t = tid; t < pairs; t += threads) {
        const unsigned lo = (t / half) * 2 * half + (t & (half - 1));
        const unsigned hi = first ? (lo ^ (size - 1)) : lo + half;
        if (hi < len) {
          const uint32_t x = p[lo], y = p[hi];
          if (x > y) {
            p[lo] = y;
            p[hi] = x;
          }
        }
      }
      sync();
    }
    if (size >= len) break;
  }
}

constexpr unsigned ROW_MAX = 512;  // bucket entries a warp takes in shared memory
constexpr int ROW_WARPS = 4;

// distinct values of 32 lanes (~0: none), ascending, to out; returns their number
__device__ __forceinline__ unsigned row_sort32(uint32_t v, int lane, uint32_t* __restrict__ out) {
  const unsigned full = 0xffffffffu;
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
    for (int half = size >> 1; half > 0; half >>= 1) {
      const int o = half == size >> 1 ? size - 1 : half;
      const uint32_t u = __shfl_xor_sync(full, v, o);
      v = (lane & half) ? max(u, v) : min(u, v);
    }
  const uint32_t before = __shfl_up_sync(full, v, 1);
  const bool keep = v != full && (lane == 0 || v != before);
  const unsigned m = __ballot_sync(full, keep);
  if (keep) out[__popc(m & ((1u << lane) - 1u))] = v;
  return (unsigned)__popc(m);
}

// A warp per row, or per 8 rows where that still fills the chip (rows may be
// mostly empty): the bucket made distinct and sorted in place, the count to
// uniq; longer buckets are listed for k_row_unique_long.  Bound by instruction
// issue, so the many duplicates (a bucket holds its row's columns two to three
// times over) go first, through an open-addressing set at most half full, and
// only the distinct columns are sorted -- in registers where 32 lanes hold
// them.  A pleated 256x256 pass 235 -> 84 us (a warp sorting each whole bucket in
// shared memory before), two stacked layers 31 -> 15, 64 rod scenes 193 -> 145.
__global__ void __launch_bounds__(32 * ROW_WARPS) k_row_unique(int n, int per, const uint32_t* __restrict__ off,
                                                               uint32_t* __restrict__ rcol, uint32_t* __restrict__ uniq,
                                                               uint32_t* __restrict__ longs,
                                                               unsigned int* __restrict__ nlong) {
  __shared__ uint4 set4[ROW_WARPS][2 * ROW_MAX / 4];
  __shared__ uint32_t buf[ROW_WARPS][ROW_MAX];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint32_t* set = (uint32_t*)set4[threadIdx.x >> 5];
  uint32_t* p = buf[threadIdx.x >> 5];
  const int64_t r0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
  const uint32_t first = off[min(r0 + lane, (int64_t)n)];
  const uint32_t mine = __shfl_down_sync(full, first, 1) - first;
  if (lane < per && r0 + lane < n && mine == 0) uniq[r0 + lane] = 0;
  for (unsigned todo = __ballot_sync(full, lane < per && r0 + lane < n && mine > 0); todo; todo &= todo - 1u) {
    const int q = __ffs((int)todo) - 1;
    const int64_t r = r0 + q;
    const uint32_t b = __shfl_sync(full, first, q), len = __shfl_sync(full, mine, q);
    if (len > ROW_MAX) {
      if (lane == 0) longs[atomicAdd(nlong, 1u)] = (uint32_t)r;
      continue;
    }
    if (len <= 32) {
      const unsigned m = row_sort32(lane < (int)len ? rcol[b + lane] : full, lane, rcol + b);
      if (lane == 0) uniq[r] = m;
      continue;
    }
    __syncwarp();  // the last row's reads are over
    const int bits = 33 - __clz(len - 1);  // 2^bits >= 2 len
    for (int i = lane; i < 1 << (bits - 2); i += 32) set4[threadIdx.x >> 5][i] = make_uint4(full, full, full, full);
    __syncwarp();
    unsigned nu = 0;
    for (unsigned i0 = 0; i0 < len; i0 += 32) {
      const unsigned i = i0 + lane;
      bool fresh = false;
      uint32_t v = full;
      if (i < len) {
        v = rcol[b + i];
        for (unsigned h = v * 2654435769u >> (32 - bits);; h = (h + 1) & ((1u << bits) - 1u)) {  // ends: half the slots are free
          const uint32_t u = atomicCAS(&set[h], full, v);
          fresh = u == full;
          if (fresh || u == v) break;
        }
      }
      const unsigned m = __ballot_sync(full, fresh);
      if (fresh) p[nu + __popc(m & ((1u << lane) - 1u))] = v;
      nu += (unsigned)__popc(m);
    }
    __syncwarp();
    if (nu <= 32) {
      row_sort32(lane < (int)nu ? p[lane] : full, lane, rcol + b);
    } else {
      sort_segment(p, nu, lane, 32, [] { __syncwarp(); });
      for (unsigned i = lane; i < nu; i += 32) rcol[b + i] = p[i];
    }
    if (lane == 0) uniq[r] = nu;
  }
}

// ... a block per long bucket of up to ROW_BLOCK_MAX entries: duplicates go through an open-addressing set at most half
// full, the distinct columns are sorted in shared memory.  Longer buckets are numbered in hrow, with the first of
// their entries among all such buckets' in hstart; `huge` counts both (buckets << 32 | entries).  Bound by the latency
// of the sort's steps, which a block's 1,024 threads and shared memory shorten and the set keeps to distinct columns
// (before, 256 threads sorted a whole bucket of any length in global memory): the barrier stage without its Hessian
// kernel with one edge across 700 needles 184 -> 144 us, across 4,000 525 -> 215.
constexpr unsigned ROW_BLOCK_MAX = 16384;
constexpr int ROW_LONG_T = 1024;
constexpr int ROW_LONG_SMEM = 3 * (int)ROW_BLOCK_MAX * 4;

__global__ void __launch_bounds__(ROW_LONG_T) k_row_unique_long(const uint32_t* __restrict__ off, uint32_t* rcol,
                                                            uint32_t* __restrict__ uniq,
                                                            const uint32_t* __restrict__ longs,
                                                            const unsigned int* __restrict__ nlong,
                                                            uint32_t* __restrict__ hrow, uint32_t* __restrict__ hstart,
                                                            unsigned long long* __restrict__ huge) {
  extern __shared__ uint32_t long_smem[];
  uint32_t *set = long_smem, *p = long_smem + 2 * ROW_BLOCK_MAX;
  __shared__ unsigned nu;
  for (unsigned q = blockIdx.x; q < *nlong; q += gridDim.x) {
    const uint32_t r = longs[q], b = off[r], len = off[r + 1] - b;
    if (len > ROW_BLOCK_MAX) {
      if (threadIdx.x == 0) {
        const unsigned long long at = atomicAdd(huge, 1ull << 32 | len);  // (the buckets hold fewer than 2^32 entries)
        hrow[at >> 32] = r;
        hstart[at >> 32] = (uint32_t)at;
      }
      continue;
    }
    const int bits = 33 - __clz(len - 1);  // 2^bits >= 2 len
    for (unsigned i = threadIdx.x; i < 1u << bits; i += ROW_LONG_T) set[i] = 0xffffffffu;
    if (threadIdx.x == 0) nu = 0;
    __syncthreads();
    for (unsigned i = threadIdx.x; i < len; i += ROW_LONG_T) {
      const uint32_t v = rcol[b + i];
      for (unsigned h = v * 2654435769u >> (32 - bits);; h = (h + 1) & ((1u << bits) - 1u)) {  // ends: half the slots are free
        const uint32_t u = atomicCAS(&set[h], 0xffffffffu, v);
        if (u == 0xffffffffu) p[atomicAdd(&nu, 1u)] = v;
        if (u == 0xffffffffu || u == v) break;
      }
    }
    __syncthreads();
    const unsigned m = nu;
    sort_segment(p, m, threadIdx.x, ROW_LONG_T, [] { __syncthreads(); });
    for (unsigned i = threadIdx.x; i < m; i += ROW_LONG_T) rcol[b + i] = p[i];
    if (threadIdx.x == 0) uniq[r] = m;
    __syncthreads();  // before the next bucket takes the set
  }
}

// ... the buckets past ROW_BLOCK_MAX together: their entries as (bucket, column) keys, radix sorted, made distinct and put
// back.  One bucket's time in a block grows with its length, and the pass waits for it; the sort spreads over the chip,
// for one more host wait.  Without the Hessian kernel, a sheet of 65k vertices on two triangles (four rows of 65k
// columns) 6.79 -> 0.35 ms, an edge across 100,000 needles 41.9 -> 0.56.  The line: 20 buckets of 8,000 entries take
// 291 us in blocks against 378 sorted, of 16,200 534 against 527 -- and a block's shared memory ends at 16,384.
struct HugeRows {
  unsigned n, entries;
  int cbits;  // bits of a column
  const uint32_t* __restrict__ row;
  const uint32_t* __restrict__ start;
  const uint32_t* __restrict__ off;
  __device__ __forceinline__ unsigned bucket_of(unsigned i) const {
    unsigned lo = 0, hi = n;  // the last bucket that starts at or before entry i
    while (hi - lo > 1) {
      const unsigned mid = (lo + hi) >> 1;
      if (start[mid] <= i) lo = mid;
      else hi = mid;
    }
    return lo;
  }
};

__global__ void k_huge_keys(HugeRows H, const uint32_t* __restrict__ rcol, uint64_t* __restrict__ key) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H.entries) return;
  const unsigned k = H.bucket_of((unsigned)i);
  key[i] = (uint64_t)k << H.cbits | rcol[H.off[H.row[k]] + ((unsigned)i - H.start[k])];
}
__global__ void k_huge_flag(unsigned entries, const uint64_t* __restrict__ key, uint32_t* __restrict__ flag) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i <= entries) flag[i] = i < entries && (i == 0 || key[i] != key[i - 1]) ? 1u : 0u;
}
__global__ void k_huge_write(HugeRows H, const uint64_t* __restrict__ key, const uint32_t* __restrict__ flag,
                             const uint32_t* __restrict__ pos, uint32_t* __restrict__ rcol, uint32_t* __restrict__ uniq) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H.entries || !flag[i]) return;
  const unsigned k = (unsigned)(key[i] >> H.cbits), first = H.start[k], end = k + 1 < H.n ? H.start[k + 1] : H.entries;
  const uint32_t r = H.row[k];
  rcol[H.off[r] + (pos[i] - pos[first])] = (uint32_t)(key[i] & ((1ull << H.cbits) - 1ull));
  if (i == first) uniq[r] = pos[end] - pos[first];
}

// the rows' distinct columns to their place, 8 lanes a row (a full warp left most lanes without work: 64 rod scenes
// with 1.1M rows 142 -> 46 us); rows past ROW_MAX columns take a block, those past ROW_BLOCK_MAX a thread per entry
__global__ void k_row_write(int n, const uint32_t* __restrict__ off, const uint32_t* __restrict__ rcol,
                            const int32_t* __restrict__ row_ptr, int32_t* __restrict__ col) {
  const int r = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3);
  if (r >= n) return;
  const int o = row_ptr[r], c = row_ptr[r + 1] - o;
  if (c == 0 || c > (int)ROW_MAX) return;
  const uint32_t b = off[r];
  for (int i = threadIdx.x & 7; i < c; i += 8) col[o + i] = (int32_t)rcol[b + i];
}
__global__ void __launch_bounds__(ROW_LONG_T) k_row_write_long(const uint32_t* __restrict__ longs, unsigned nlong,
                                                               const uint32_t* __restrict__ off,
                                                               const uint32_t* __restrict__ rcol,
                                                               const int32_t* __restrict__ row_ptr,
                                                               int32_t* __restrict__ col) {
  for (unsigned q = blockIdx.x; q < nlong; q += gridDim.x) {
    const uint32_t r = longs[q], b = off[r];
    const int o = row_ptr[r], c = row_ptr[r + 1] - o;
    if (c <= (int)ROW_MAX || c > (int)ROW_BLOCK_MAX) continue;
    for (int i = threadIdx.x; i < c; i += ROW_LONG_T) col[o + i] = (int32_t)rcol[b + i];
  }
}
__global__ void k_huge_cols(HugeRows H, const uint32_t* __restrict__ rcol, const int32_t* __restrict__ row_ptr,
                            int32_t* __restrict__ col) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= H.entries) return;
  const unsigned k = H.bucket_of((unsigned)i);
  const uint32_t r = H.row[k];
  const int o = row_ptr[r], c = row_ptr[r + 1] - o, q = (int)((unsigned)i - H.start[k]);
  if (c > (int)ROW_BLOCK_MAX && q < c) col[o + q] = (int32_t)rcol[H.off[r] + q];
}

// Distance types as difference vectors z_m = x_plus - x_minus:
//   point-point: z0 = b - a;  point-edge: z0 = w = q - e0, z1 = u = e1 - e0;
//   plane: z0 = w, z1 = u, z2 = v (point-triangle face: w = p - t0, u = t1 - t0,
//   v = t2 - t0; edge-edge interior: w = b0 - a0, u = a1 - a0, v = b1 - b0),
// up to a common sign; two bits a point: plus0, minus0, plus1, minus1, plus2, minus2.
constexpr int diff_code(int p0, int m0, int p1 = 0, int m1 = 0, int p2 = 0, int m2 = 0) {
  return p0 | m0 << 2 | p1 << 4 | m1 << 6 | p2 << 8 | m2 << 10;
}
__constant__ int c_pt_diff[7] = {diff_code(1, 0),       diff_code(2, 0),       diff_code(3, 0),      diff_code(0, 1, 2, 1),
                                 diff_code(0, 2, 3, 2), diff_code(0, 3, 1, 3), diff_code(0, 1, 2, 1, 3, 1)};
__constant__ int c_ee_diff[9] = {diff_code(2, 0),       diff_code(3, 0),       diff_code(2, 1),
                                 diff_code(3, 1),       diff_code(0, 2, 3, 2), diff_code(1, 2, 3, 2),
                                 diff_code(2, 0, 1, 0), diff_code(3, 0, 1, 0), diff_code(2, 0, 1, 0, 3, 2)};

// Orthonormal basis of the complement of rigid translations of four points
__constant__ double c_K4[4][3] = {{0.5, 0.5, 0.5}, {0.5, -0.5, -0.5}, {-0.5, 0.5, -0.5}, {-0.5, -0.5, 0.5}};

__host__ __device__ __forceinline__ int tri_idx(int i, int j, int D) {  // packed upper triangle, i <= j
  return i * D - (i * (i - 1)) / 2 + (j - i);
}

__device__ __forceinline__ int64_t find_block(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                              int r, int c) {
  int lo = row_ptr[r], hi = row_ptr[r + 1];
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (col[mid] < c) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

struct HessArgs {
  ActiveList act;
  const uint64_t* __restrict__ cand;
  const double* __restrict__ cd;
  const int8_t* __restrict__ ctype;
  const uint8_t* __restrict__ ccls;
  const int32_t* __restrict__ ev0;
  const int32_t* __restrict__ ev1;
  const int32_t* __restrict__ tv;
  int T;
  const double* __restrict__ x;
  int n;
  const int32_t* __restrict__ vsc;
  const MemberParams* __restrict__ mp;
  unsigned long long* __restrict__ macc;
  const int32_t* __restrict__ comp;                 // component label per vertex
  const unsigned long long* __restrict__ dbar_comp; // per-component dbar_min bits (CB_DBAR_PER_COMPONENT)
  const int32_t* __restrict__ row_ptr;
  const int32_t* __restrict__ col;
  double* __restrict__ val;
  double* __restrict__ grad;
  unsigned long long* __restrict__ status;
  unsigned int* __restrict__ n9;   // face / line-line pairs (and mollified ones)
  unsigned int* __restrict__ n6;   // point-edge pairs nearly on the edge's line (|w| |u| > 64 |u x w|)
  unsigned int* __restrict__ n4;   // the other point-edge pairs
  // CB_EE_MOLLIFIER: the queued 9x9 matrices of the mollified pairs, packed upper triangle, element-major
  // ([e * cap + slot], slot = the pair's place in mlist)
  double* __restrict__ B9;
  int64_t cap;
  // CB_EE_MOLLIFIER: candidates handled by k_moll_hess
  const uint32_t* __restrict__ mlist;
  const unsigned* __restrict__ nmoll;
  const double* __restrict__ elen2;
};


// entries c[0..NC) of row r: their block indices, -1 where the pattern has none
// (the searches advance together, so their loads overlap)
template <int NC>
__device__ __forceinline__ void find_blocks(const HessArgs& A, int r, const int (&c)[NC], int64_t (&out)[NC]) {
  const int b = A.row_ptr[r], e = A.row_ptr[r + 1];
  int lo[NC], hi[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    lo[k] = b;
    hi[k] = e;
  }
  for (int len = e - b; len > 0; len >>= 1) {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      if (lo[k] >= hi[k]) continue;
      const int mid = (lo[k] + hi[k]) >> 1;
      if (A.col[mid] < c[k]) lo[k] = mid + 1;
      else hi[k] = mid;
    }
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) out[k] = lo[k] < e && A.col[lo[k]] == c[k] ? (int64_t)lo[k] : -1;
}

// a 3x3 block into the BSR values (transposed if tr); a pattern miss is never expected
__device__ __forceinline__ void add_block(const HessArgs& A, int64_t bi, const double (&blk)[9], bool tr) {
  if (bi < 0) {
    atomicOr(A.status, (unsigned long long)CB_DEV_CAPACITY);
    return;
  }
  double* dst = A.val + 9 * bi;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) atomicAdd(&dst[3 * i + j], tr ? blk[3 * j + i] : blk[3 * i + j]);
}

// Stage (d), one thread per active pair: barrier value and derivatives,
// energy, gradient scatter, the PSD-projected Hessian in closed form
// (pairhess.cuh) and its scatter into the BSR values.  PAIR_T threads a block:
// the work is a few hundred to a thousand FP64 instructions per warp, of which
// an SM completes one per 16 cycles at best (full occupancy, independent chains)
// and one per 19 with four warps of dependent ones, so small blocks spread a
// short list over more SMs and cost a long one nothing.  It loads only the
// points its type needs and subtracts them once (a type's matrix of signs
// took 27 multiply-adds and nine conversions more, symmetric blocks their lower
// triangles): 666 -> 594 FP64 instructions a warp, pleated 97x97 189 -> 157 us.
constexpr int PAIR_T = 64;

// v[i] for an index known only at run time, without a local-memory array
__device__ __forceinline__ int pick(const int (&v)[4], int i) {
  i &= 3;
  return i == 0 ? v[0] : (i == 1 ? v[1] : (i == 2 ? v[2] : v[3]));
}

__global__ void __launch_bounds__(PAIR_T) k_pair_hess(HessArgs A) {
  const int64_t t = (int64_t)blockIdx.x * PAIR_T + threadIdx.x;
  const uint32_t c = t < A.act.n ? A.act.at(t) : 0u;
  const uint8_t cls = t < A.act.n ? A.ccls[c] : CB_CLS_MOLLIFIED;
  double e_local = 0.0;
  int mem = -1, counted = 0;  // 9, 6, 4: the statistics' kinds
  if (!(cls & CB_CLS_MOLLIFIED)) {  // (mollified: k_moll_hess)
    const Stencil s = stencil_of(A.cand[c], A.ev0, A.ev1, A.tv, A.T);
    const int ty = A.ctype[c];
    const int code = s.ee ? c_ee_diff[ty] : c_pt_diff[ty];
    const int kind = ty == (s.ee ? 8 : 6) ? 2 : (ty >= (s.ee ? 4 : 3) ? 1 : 0);
    const double d = A.cd[c];
    mem = A.vsc[s.v[0]];
    const PassParams P = member_pass(A.mp[mem]);
    double xi_p, dh_p;
    pair_params(P, cls, f_width(P, A.dbar_comp, A.comp, s.v[0]), xi_p, dh_p);
    const double y = d - xi_p;
    double b, b1, b2;
    barrier_b012(y, dh_p, b, b1, b2);
    e_local = P.kappa * b;
    const double g1 = P.kappa * b1, beta = P.kappa * b2;
    const bool out = y > 0.0;  // inside the offset the energy is +inf and the pair adds no Hessian
    // the difference vectors z_m = x_plus - x_minus (only the points a type needs are loaded)
    const int p0 = pick(s.v, code), m0 = pick(s.v, code >> 2);
    const d3 X0 = load3(A.x, A.n, p0), Y0 = load3(A.x, A.n, m0);
    double z[3][3] = {{X0.x - Y0.x, X0.y - Y0.y, X0.z - Y0.z}, {}, {}};
    auto diff = [&](int m, int shift) {
      const d3 X = load3(A.x, A.n, pick(s.v, code >> shift)), Y = load3(A.x, A.n, pick(s.v, code >> (shift + 2)));
      z[m][0] = X.x - Y.x;
      z[m][1] = X.y - Y.y;
      z[m][2] = X.z - Y.z;
    };
    if (kind >= 1) diff(1, 4);
    if (kind == 2) diff(2, 8);
    auto grad_add = [&](int v, double cw, const double (&n)[3]) {
#pragma unroll
      for (int al = 0; al < 3; ++al) atomicAdd(&A.grad[(size_t)al * A.n + v], g1 * cw * n[al]);
    };
    if (kind == 2) {
      counted = 9;
      cbh::PlaneBlocks Q;
      cbh::plane_blocks(s.ee, z[0], z[1], z[2], d, beta, -g1, Q);
      if (A.grad)
#pragma unroll
        for (int q = 0; q < 4; ++q) grad_add(s.v[q], Q.c[q], Q.n);
      if (out) {
        int64_t at[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) find_blocks<4>(A, s.v[q], s.v, at[q]);
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int r = p; r < 4; ++r) {
            double blk[9];
            cbh::plane_block(Q, p, r, blk);
            add_block(A, at[p][r], blk, false);
            if (r > p) add_block(A, at[r][p], blk, true);
          }
      }
    } else if (kind == 1) {
      // r = w - t u with one rounding per component, its part along u (t's rounding) then removed: n keeps full
      // accuracy however close the point lies to the edge
      const double(&w)[3] = z[0];
      const double(&u)[3] = z[1];
      const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2], iu = rsqrt(uu), iuu = iu * iu;
      double tp = (w[0] * u[0] + w[1] * u[1] + w[2] * u[2]) * iuu, r[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) r[k] = fma(-tp, u[k], w[k]);
      const double dt = (r[0] * u[0] + r[1] * u[1] + r[2] * u[2]) * iuu;
      tp += dt;
#pragma unroll
      for (int k = 0; k < 3; ++k) r[k] = fma(-dt, u[k], r[k]);
      const double rr = r[0] * r[0] + r[1] * r[1] + r[2] * r[2], ir = rsqrt(rr);
      const double ww = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
      counted = ww <= 4096.0 * rr ? 4 : 6;
      cbh::EdgeBlocks Q;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        Q.n[k] = r[k] * ir;
        Q.e[k] = u[k] * iu;
      }
      cbh::edge_blocks(tp, iu, d, beta, -g1, Q);
      // the stencil points q, e0, e1: w = q - e0, u = e1 - e0, up to the sign of both
      const int v3[3] = {p0, m0, pick(s.v, code >> 4)};
      if (A.grad)
#pragma unroll
        for (int q = 0; q < 3; ++q) grad_add(v3[q], Q.c[q], Q.n);
      if (out) {
        int64_t at[3][3];
#pragma unroll
        for (int q = 0; q < 3; ++q) find_blocks<3>(A, v3[q], v3, at[q]);
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
          for (int q = p; q < 3; ++q) {
            double blk[9];
            cbh::edge_block(Q, p, q, blk);
            add_block(A, at[p][q], blk, false);
            if (q > p) add_block(A, at[q][p], blk, true);
          }
      }
    } else {
      // point-point: kappa b'' n n^T + (kappa b'/d)(I - n n^T), each part clamped
      const double id = 1.0 / d;
      const double n[3] = {z[0][0] * id, z[0][1] * id, z[0][2] * id};
      const int v2[2] = {p0, m0};
      if (A.grad) {
        grad_add(v2[0], 1.0, n);
        grad_add(v2[1], -1.0, n);
      }
      if (out) {
        const double lam_n = fmax(beta, 0.0), lam_t = fmax(g1 * id, 0.0);
        double blk[9], neg[9];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            blk[3 * i + j] = lam_n * n[i] * n[j] + lam_t * ((i == j ? 1.0 : 0.0) - n[i] * n[j]);
            neg[3 * i + j] = -blk[3 * i + j];
          }
        int64_t at[2][2];
#pragma unroll
        for (int q = 0; q < 2; ++q) find_blocks<2>(A, v2[q], v2, at[q]);
        add_block(A, at[0][0], blk, false);
        add_block(A, at[1][1], blk, false);
        add_block(A, at[0][1], neg, false);
        add_block(A, at[1][0], neg, false);
      }
    }
  }
#pragma unroll
  for (int which = 0; which < 3; ++which) {
    const unsigned m = __ballot_sync(0xffffffffu, counted == (which == 0 ? 9 : (which == 1 ? 6 : 4)));
    if (m && (threadIdx.x & 31) == 0) atomicAdd(which == 0 ? A.n9 : (which == 1 ? A.n6 : A.n4), (unsigned)__popc(m));
  }
  member_energy_add(A.macc, mem, e_local);
}

// ---- IPC's edge-edge mollifier (CB_EE_MOLLIFIER) -------------------------
// A mollified pair's energy m(c) kappa b(d) depends on all four points
// whatever its distance type, so it leaves the closed forms of k_pair_hess.
// Its gradient and Hessian are formed here from analytic derivatives of the
// typed distance d and of c = |e0 x e1|^2, written in the difference vectors
// the distance is a function of and mapped to the four points:
//   point-point  r = q - p:              s = |r|^2
//   point-line   w = q - e0, u = e1 - e0: s = |w|^2 - (w.u)^2 / |u|^2
//     (then grad d = grad s / 2d, hess d = (hess s - 2 grad d grad d^T) / 2d)
//   line-line    w = b0 - a0, u = a1 - a0, v = b1 - b0, n = u x v:
//     d = |g| / sqrt(N), g = w.n, N = |n|^2, differentiated directly (no
//     squared distance, whose two large terms cancel for near-parallel edges)
//   c = N (the same u, v), grad and hess in closed form.
// The Hessian by the product rule,
//   H = kappa (m (b'' gd gd^T + b' Hd) + b' m' (gc gd^T + gd gc^T)
//              + b (m'' gc gc^T + m' Hc)),
// and the 9x9 matrix of the four-point translation-free basis
// (B = (K4 x I)^T H (K4 x I)) is queued for the 9x9 projection.
struct LocalDeriv {
  int nb;                  // difference vectors (blocks of 3)
  int plus[3], minus[3];   // block b = x[plus[b]] - x[minus[b]] (stencil points 0..3)
  double g[9];             // gradient in the blocks
  double H[9][9];          // Hessian in the blocks
};

// the gradient and Hessian of a function of the difference vectors, as
// functions of the 12 coordinates of the four stencil points
__device__ void local_to_points(const LocalDeriv& L, double (&g12)[12], double (&H12)[12][12]) {
  double cf[4][3];
  for (int P = 0; P < 4; ++P)
    for (int b = 0; b < 3; ++b) cf[P][b] = b < L.nb ? (L.plus[b] == P ? 1.0 : 0.0) - (L.minus[b] == P ? 1.0 : 0.0) : 0.0;
  for (int P = 0; P < 4; ++P)
    for (int i = 0; i < 3; ++i) {
      double v = 0.0;
      for (int b = 0; b < L.nb; ++b) v += cf[P][b] * L.g[3 * b + i];
      g12[3 * P + i] = v;
    }
  for (int P = 0; P < 4; ++P)
    for (int Q = 0; Q < 4; ++Q)
      for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
          double v = 0.0;
          for (int b = 0; b < L.nb; ++b) {
            if (cf[P][b] == 0.0) continue;
            for (int e = 0; e < L.nb; ++e) v += cf[P][b] * cf[Q][e] * L.H[3 * b + i][3 * e + j];
          }
          H12[3 * P + i][3 * Q + j] = v;
        }
}

// |u x v|^2 of u (block bu) and v (block bv): gradient and Hessian entries added with weight w
__device__ void add_cross2(LocalDeriv& L, int bu, int bv, const d3& u, const d3& v, double wg, double wh) {
  const double uu = dot3(u, u), vv = dot3(v, v), uv = dot3(u, v);
  const double U[3] = {u.x, u.y, u.z}, V[3] = {v.x, v.y, v.z};
  for (int i = 0; i < 3; ++i) {
    L.g[3 * bu + i] += wg * (2.0 * vv * U[i] - 2.0 * uv * V[i]);
    L.g[3 * bv + i] += wg * (2.0 * uu * V[i] - 2.0 * uv * U[i]);
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      const double dl = i == j ? 1.0 : 0.0;
      L.H[3 * bu + i][3 * bu + j] += wh * (2.0 * vv * dl - 2.0 * V[i] * V[j]);
      L.H[3 * bv + i][3 * bv + j] += wh * (2.0 * uu * dl - 2.0 * U[i] * U[j]);
      const double m = 4.0 * U[i] * V[j] - 2.0 * V[i] * U[j] - 2.0 * uv * dl;  // d2/du_i dv_j
      L.H[3 * bu + i][3 * bv + j] += wh * m;
      L.H[3 * bv + j][3 * bu + i] += wh * m;
    }
}

// gradient and Hessian of the typed edge-edge distance d (types as in
// geometry.cuh) in difference vectors of the stencil X (a0 a1 b0 b1)
__device__ void ee_distance_derivs(int ty, const d3 (&X)[4], double d, LocalDeriv& L) {
  for (int i = 0; i < 9; ++i) {
    L.g[i] = 0.0;
    for (int j = 0; j < 9; ++j) L.H[i][j] = 0.0;
  }
  if (ty <= 7) {
    // squared distance s in (r) or (w, u), then d
    if (ty <= 3) {
      const int p = ty <= 1 ? 0 : 1, q = (ty & 1) ? 3 : 2;
      L.nb = 1;
      L.plus[0] = q;
      L.minus[0] = p;
      const d3 r = sub3(X[q], X[p]);
      const double R[3] = {r.x, r.y, r.z};
      for (int i = 0; i < 3; ++i) {
        L.g[i] = 2.0 * R[i];
        L.H[i][i] = 2.0;
      }
    } else {
      // point q, line e0 e1: 4 PE(a0, b), 5 PE(a1, b), 6 PE(b0, a), 7 PE(b1, a)
      const int q = ty == 4 ? 0 : ty == 5 ? 1 : ty == 6 ? 2 : 3;
      const int e0 = ty <= 5 ? 2 : 0, e1 = ty <= 5 ? 3 : 1;
      L.nb = 2;
      L.plus[0] = q;
      L.minus[0] = e0;
      L.plus[1] = e1;
      L.minus[1] = e0;
      const d3 w = sub3(X[q], X[e0]), u = sub3(X[e1], X[e0]);
      const double a = dot3(w, u), gg = dot3(u, u), ig = 1.0 / gg;
      const double W[3] = {w.x, w.y, w.z}, U[3] = {u.x, u.y, u.z};
      for (int i = 0; i < 3; ++i) {
        L.g[i] = 2.0 * W[i] - 2.0 * a * U[i] * ig;
        L.g[3 + i] = -2.0 * a * W[i] * ig + 2.0 * a * a * U[i] * ig * ig;
      }
      for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
          const double dl = i == j ? 1.0 : 0.0;
          L.H[i][j] = 2.0 * dl - 2.0 * U[i] * U[j] * ig;
          const double wu = -2.0 * U[i] * W[j] * ig - 2.0 * a * dl * ig + 4.0 * a * U[i] * U[j] * ig * ig;
          L.H[i][3 + j] = wu;
          L.H[3 + j][i] = wu;
          L.H[3 + i][3 + j] = -2.0 * W[i] * W[j] * ig + 4.0 * a * (W[i] * U[j] + U[i] * W[j]) * ig * ig +
                              2.0 * a * a * dl * ig * ig - 8.0 * a * a * U[i] * U[j] * ig * ig * ig;
        }
    }
    // s -> d: grad d = grad s / 2d, hess d = (hess s - 2 grad d grad d^T) / 2d
    const double h = 0.5 / d;
    for (int i = 0; i < 3 * L.nb; ++i) L.g[i] *= h;
    for (int i = 0; i < 3 * L.nb; ++i)
      for (int j = 0; j < 3 * L.nb; ++j) L.H[i][j] = (L.H[i][j] - 2.0 * L.g[i] * L.g[j]) * h;
    return;
  }
  // line-line: d = |g| / sqrt(N), blocks w = b0 - a0, u = a1 - a0, v = b1 - b0
  L.nb = 3;
  L.plus[0] = 2;
  L.minus[0] = 0;
  L.plus[1] = 1;
  L.minus[1] = 0;
  L.plus[2] = 3;
  L.minus[2] = 2;
  const d3 w = sub3(X[2], X[0]), u = sub3(X[1], X[0]), v = sub3(X[3], X[2]);
  const d3 n = cross3(u, v), vw = cross3(v, w), wu = cross3(w, u);
  const double g = dot3(w, n), N = dot3(n, n);
  const double sg = g >= 0.0 ? 1.0 : -1.0, r = 1.0 / sqrt(N), r3 = r * r * r, r5 = r3 * r * r;
  // grad g = (n, v x w, w x u); hess g: the cross-product blocks
  const double Gg[9] = {n.x, n.y, n.z, vw.x, vw.y, vw.z, wu.x, wu.y, wu.z};
  // grad N and hess N (blocks u, v)
  LocalDeriv Nd;
  Nd.nb = 3;
  for (int i = 0; i < 9; ++i) {
    Nd.g[i] = 0.0;
    for (int j = 0; j < 9; ++j) Nd.H[i][j] = 0.0;
  }
  add_cross2(Nd, 1, 2, u, v, 1.0, 1.0);
  // hess g: d2g/dw du = -[v]x, d2g/dw dv = [u]x, d2g/du dv = -[w]x ([a]x b = a x b)
  auto crossm = [](const d3& a, double sgn, double (&M)[3][3]) {
    M[0][0] = 0.0;
    M[0][1] = -sgn * a.z;
    M[0][2] = sgn * a.y;
    M[1][0] = sgn * a.z;
    M[1][1] = 0.0;
    M[1][2] = -sgn * a.x;
    M[2][0] = -sgn * a.y;
    M[2][1] = sgn * a.x;
    M[2][2] = 0.0;
  };
  double Hg[9][9];
  for (int i = 0; i < 9; ++i)
    for (int j = 0; j < 9; ++j) Hg[i][j] = 0.0;
  {
    double M[3][3], T[3][3];
    crossm(v, -1.0, M);  // rows w, cols u
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Hg[i][3 + j] = M[i][j];
        Hg[3 + j][i] = M[i][j];
      }
    crossm(u, 1.0, T);  // rows w, cols v
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Hg[i][6 + j] = T[i][j];
        Hg[6 + j][i] = T[i][j];
      }
    crossm(w, -1.0, M);  // rows u, cols v
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Hg[3 + i][6 + j] = M[i][j];
        Hg[6 + j][3 + i] = M[i][j];
      }
  }
  for (int i = 0; i < 9; ++i) L.g[i] = sg * (r * Gg[i] - 0.5 * g * r3 * Nd.g[i]);
  for (int i = 0; i < 9; ++i)
    for (int j = 0; j < 9; ++j)
      L.H[i][j] = sg * (r * Hg[i][j] - 0.5 * r3 * (Gg[i] * Nd.g[j] + Nd.g[i] * Gg[j]) - 0.5 * g * r3 * Nd.H[i][j] +
                        0.75 * g * r5 * Nd.g[i] * Nd.g[j]);
}

// One thread per mollified pair (listed by k_distance_exact); bound by the latency of its chain, so blocks of one
// warp spread a short list over all SMs (10,231 pairs: 576 us in blocks of 128, 365 in blocks of 32)
__global__ void __launch_bounds__(32) k_moll_hess(HessArgs A) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double e_local = 0.0;
  int mem = -1;
  if (t < (int64_t)*A.nmoll) {
    const uint32_t c = A.mlist[t];
    const uint64_t key = A.cand[c];
    const Stencil s = stencil_of(key, A.ev0, A.ev1, A.tv, A.T);
    const int ty = A.ctype[c];
    mem = A.vsc[s.v[0]];
    const PassParams P = member_pass(A.mp[mem]);
    double xi_p, dh_p;
    pair_params(P, A.ccls[c] & ~CB_CLS_MOLLIFIED, f_width(P, A.dbar_comp, A.comp, s.v[0]), xi_p, dh_p);
    const double d = A.cd[c];
    double b, b1, b2;
    barrier_b012(d - xi_p, dh_p, b, b1, b2);
    // points relative to the first one (translation changes no derivative)
    const d3 X0 = load3(A.x, A.n, s.v[0]);
    d3 X[4];
    for (int q = 0; q < 4; ++q) X[q] = sub3(load3(A.x, A.n, s.v[q]), X0);
    double gd[12], gc[12], Hd[12][12], Hc[12][12];
    {
      LocalDeriv L;
      ee_distance_derivs(ty, X, d, L);
      local_to_points(L, gd, Hd);
    }
    double cval;
    {
      LocalDeriv L;
      L.nb = 2;
      L.plus[0] = 1;
      L.minus[0] = 0;
      L.plus[1] = 3;
      L.minus[1] = 2;
      for (int i = 0; i < 9; ++i) {
        L.g[i] = 0.0;
        for (int j = 0; j < 9; ++j) L.H[i][j] = 0.0;
      }
      const d3 u = sub3(X[1], X[0]), v = sub3(X[3], X[2]);
      const d3 n = cross3(u, v);
      cval = dot3(n, n);
      add_cross2(L, 0, 1, u, v, 1.0, 1.0);
      local_to_points(L, gc, Hc);
    }
    const double eps = 1e-3 * A.elen2[cb_key_i(key)] * A.elen2[cb_key_j(key)];
    double m, m1, m2;
    ee_mollifier(cval, eps, m, m1, m2);
    const double kap = P.kappa;
    e_local = kap * m * b;
    if (A.grad)
      for (int i = 0; i < 12; ++i) {
        const double g = kap * (m * b1 * gd[i] + b * m1 * gc[i]);
        if (g != 0.0) atomicAdd(&A.grad[(size_t)(i % 3) * A.n + s.v[i / 3]], g);
      }
    double Bf[81];
    for (int k = 0; k < 81; ++k) Bf[k] = 0.0;
    for (int i = 0; i < 12; ++i)
      for (int j = i; j < 12; ++j) {
        const double h = kap * (m * (b2 * gd[i] * gd[j] + b1 * Hd[i][j]) + b1 * m1 * (gc[i] * gd[j] + gd[i] * gc[j]) +
                                b * (m2 * gc[i] * gc[j] + m1 * Hc[i][j]));
        const int q1 = i / 3, al = i % 3, q2 = j / 3, be = j % 3;
        for (int p1 = 0; p1 < 3; ++p1)
          for (int p2 = 0; p2 < 3; ++p2) {
            const double w = c_K4[q1][p1] * c_K4[q2][p2] * h;
            Bf[(3 * p1 + al) * 9 + 3 * p2 + be] += w;
            if (i != j) Bf[(3 * p2 + be) * 9 + 3 * p1 + al] += w;
          }
      }
    for (int i = 0; i < 9; ++i)
      for (int j = i; j < 9; ++j) A.B9[(size_t)tri_idx(i, j, 9) * A.cap + t] = Bf[i * 9 + j];
  }
  const unsigned mm = __ballot_sync(0xffffffffu, mem >= 0);
  if (mm && (threadIdx.x & 31) == 0) atomicAdd(A.n9, (unsigned)__popc(mm));
  member_energy_add(A.macc, mem, e_local);
}

// Cyclic Jacobi with symmetric updates on a packed upper-triangular matrix
// held in shared memory (element e of this thread at Am[e * S]); rotations are
// accumulated into V (column-major: row i of column k at V[(k * D + i) * S]).
// Rotations with |a_pq| below
// 1e-16 of the norm are skipped; stops when off^2 <= tol2 * ||A||^2.
template <typename R, int D>
__device__ __forceinline__ void jacobi_packed(R* Am, R* V, const int S, const R tol2, const int max_sweeps) {
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    R off = 0, fro = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const R d = Am[tri_idx(i, i, D) * S];
      fro += d * d;
#pragma unroll
      for (int j = i + 1; j < D; ++j) {
        const R v = Am[tri_idx(i, j, D) * S];
        off += R(2) * v * v;
      }
    }
    fro += off;
    if (fro == R(0) || off <= tol2 * fro) break;
    const R skip = R(1e-16) * sqrt(fro);
    for (int p = 0; p < D - 1; ++p)
      for (int q = p + 1; q < D; ++q) {
        const R apq = Am[tri_idx(p, q, D) * S];
        if (fabs(apq) <= skip) continue;
        const R app = Am[tri_idx(p, p, D) * S], aqq = Am[tri_idx(q, q, D) * S];
        const R tau = (aqq - app) / (R(2) * apq);
        const R t = (tau >= R(0) ? R(1) : R(-1)) / (fabs(tau) + sqrt(R(1) + tau * tau));
        const R c = R(1) / sqrt(R(1) + t * t), s = t * c;
        Am[tri_idx(p, p, D) * S] = app - t * apq;
        Am[tri_idx(q, q, D) * S] = aqq + t * apq;
        Am[tri_idx(p, q, D) * S] = R(0);
        for (int k = 0; k < D; ++k) {
          if (k == p || k == q) continue;
          const int ikp = (k < p ? tri_idx(k, p, D) : tri_idx(p, k, D)) * S;
          const int ikq = (k < q ? tri_idx(k, q, D) : tri_idx(q, k, D)) * S;
          const R akp = Am[ikp], akq = Am[ikq];
          Am[ikp] = c * akp - s * akq;
          Am[ikq] = s * akp + c * akq;
        }
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const R vkp = V[(p * D + k) * S], vkq = V[(q * D + k) * S];
          V[(p * D + k) * S] = c * vkp - s * vkq;
          V[(q * D + k) * S] = s * vkp + c * vkq;
        }
      }
  }
}

// 1 / sqrt(u) for u >= 1 in FP64 without the FP64 square root and division:
// the FP32 estimate (relative error < 1e-7) refined by two Newton steps
// (error squared each time, so to FP64 rounding).
__device__ __forceinline__ double rsqrt_refined(double u) {
  double c = (double)rsqrtf((float)u);
  c = c * (1.5 - 0.5 * u * c * c);
  c = c * (1.5 - 0.5 * u * c * c);
  return c;
}

// The FP64 sweeps of the projection, after the FP32 eigenvectors: cyclic
// Jacobi where each rotation's tangent comes from FP32 arithmetic on values
// scaled by the matrix norm, and the rotation itself is exact: c = 1/sqrt(1+t^2)
// to FP64 rounding (rsqrt_refined), s = t c, and the 2x2 pivot block is
// transformed with the full similarity formulas.  A tangent off by a relative
// 1e-7 leaves a_pq at 1e-7 of its value -- quadratically small after the FP32
// phase -- for the next sweep, while A stays an exact similarity of the input
// and V stays orthonormal.  This avoids every FP64 division and square root
// in the rotations.  Stops when off^2 <= tol2 ||A||^2.
template <int D>
__device__ __forceinline__ void jacobi_refine64(double* Am, double* V, const int S, const double tol2,
                                                const int max_sweeps) {
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0, fro = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      const double d = Am[tri_idx(i, i, D) * S];
      fro += d * d;
#pragma unroll
      for (int j = i + 1; j < D; ++j) {
        const double v = Am[tri_idx(i, j, D) * S];
        off += 2.0 * v * v;
      }
    }
    fro += off;
    if (fro == 0.0 || off <= tol2 * fro) break;
    const double nrm = sqrt(fro);
    const double skip = 1e-16 * nrm;
    const double inv = 1.0 / nrm;
    for (int p = 0; p < D - 1; ++p)
      for (int q = p + 1; q < D; ++q) {
        const double apq = Am[tri_idx(p, q, D) * S];
        if (fabs(apq) <= skip) continue;
        const double app = Am[tri_idx(p, p, D) * S], aqq = Am[tri_idx(q, q, D) * S];
        // |apq| > 1e-16 ||A||, so the scaled FP32 values stay normal
        const float apq32 = (float)(apq * inv), dd32 = (float)((aqq - app) * inv);
        const float tau = dd32 / (2.f * apq32);
        const float t32 = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
        const double t = (double)t32;
        if (__all_sync(__activemask(), fabs(t) < 1e-8)) {
          // small angle in every lane (warp-uniform, so no lane runs both
          // paths): c = 1/sqrt(1+t^2) rounds to 1 in FP64, s = t; the residual
          // a_pq (a relative 1e-7 of a_pq, below 1e-15 ||A||) is dropped
          Am[tri_idx(p, p, D) * S] = app - t * apq;
          Am[tri_idx(q, q, D) * S] = aqq + t * apq;
          Am[tri_idx(p, q, D) * S] = 0.0;
          for (int k = 0; k < D; ++k) {
            if (k == p || k == q) continue;
            const int ikp = (k < p ? tri_idx(k, p, D) : tri_idx(p, k, D)) * S;
            const int ikq = (k < q ? tri_idx(k, q, D) : tri_idx(q, k, D)) * S;
            const double akp = Am[ikp], akq = Am[ikq];
            Am[ikp] = akp - t * akq;
            Am[ikq] = akq + t * akp;
          }
#pragma unroll
          for (int k = 0; k < D; ++k) {
            const double vkp = V[(p * D + k) * S], vkq = V[(q * D + k) * S];
            V[(p * D + k) * S] = vkp - t * vkq;
            V[(q * D + k) * S] = vkq + t * vkp;
          }
          continue;
        }
        const double c = rsqrt_refined(1.0 + t * t), s = t * c;
        const double cc = c * c, ss = s * s, cs = c * s;
        Am[tri_idx(p, p, D) * S] = cc * app - 2.0 * cs * apq + ss * aqq;
        Am[tri_idx(q, q, D) * S] = ss * app + 2.0 * cs * apq + cc * aqq;
        Am[tri_idx(p, q, D) * S] = cs * (app - aqq) + (cc - ss) * apq;
        for (int k = 0; k < D; ++k) {
          if (k == p || k == q) continue;
          const int ikp = (k < p ? tri_idx(k, p, D) : tri_idx(p, k, D)) * S;
          const int ikq = (k < q ? tri_idx(k, q, D) : tri_idx(q, k, D)) * S;
          const double akp = Am[ikp], akq = Am[ikq];
          Am[ikp] = c * akp - s * akq;
          Am[ikq] = s * akp + c * akq;
        }
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const double vkp = V[(p * D + k) * S], vkq = V[(q * D + k) * S];
          V[(p * D + k) * S] = c * vkp - s * vkq;
          V[(q * D + k) * S] = s * vkp + c * vkq;
        }
      }
  }
}

// Threads (= queued pairs) per block of the projection kernels.  One warp per
// block: each block's warp moves through the FP32 and FP64 phases on its
// own, so on every SM some warps keep the scarce FP64 pipe busy while others
// are in their FP32 phase (with larger blocks the phase barrier would hold all
// of an SM's warps in step).
#ifndef PROJ_THREADS
#define PROJ_THREADS 32
#endif
// squared relative off-diagonal norm at which the FP32 Jacobi phase stops
#ifndef PROJ_FP32_TOL2
#define PROJ_FP32_TOL2 1e-12f
#endif

// The 4-point transform behind K4 = H / 2 (H rows (1,1,1), (1,-1,-1),
// (-1,1,-1), (-1,-1,1)): h = H p in six additions.
__host__ __device__ __forceinline__ void had3(double p0, double p1, double p2, double (&h)[4]) {
  const double t = p1 + p2, d = p1 - p2;
  h[0] = p0 + t;
  h[1] = p0 - t;
  h[2] = d - p0;
  h[3] = -d - p0;
}

// Entries (i, j) of all sixteen 3x3 blocks of (K4 x I) B+ (K4 x I)^T: with
// P[a][b] = B+[3a+i][3b+j] / 4 (Bq holds B+ / 4), X = H P H^T, block
// (q1, q2) gets X[q1][q2] at (i, j) and, for i != j, X[q2][q1] at (j, i)
// (B+ is symmetric).  Additions only, instead of the products with K4.
__host__ __device__ __forceinline__ void hadamard_block_entries(const double* Bq, int S, int i, int j,
                                                                double (&X)[4][4]) {
  double Q[3][4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double p[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int r = 3 * a + i, cl = 3 * b + j;
      p[b] = Bq[(r <= cl ? tri_idx(r, cl, 9) : tri_idx(cl, r, 9)) * S];
    }
    had3(p[0], p[1], p[2], Q[a]);
  }
#pragma unroll
  for (int q2 = 0; q2 < 4; ++q2) {
    double h[4];
    had3(Q[0][q2], Q[1][q2], Q[2][q2], h);
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1) X[q1][q2] = h[q1];
  }
}

__device__ __forceinline__ void hadamard_scatter(const HessArgs& A, const Stencil& st, const double* Bq, int S) {
  int64_t off[4][4];
  bool miss = false;
#pragma unroll
  for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) {
      const int r = st.v[q1], cc = st.v[q2];
      const int64_t bi = find_block(A.row_ptr, A.col, r, cc);
      const bool hit = bi < A.row_ptr[r + 1] && A.col[bi] == cc;
      miss |= !hit;
      off[q1][q2] = hit ? 9 * bi : -1;
    }
  if (miss) atomicOr(A.status, (unsigned long long)CB_DEV_CAPACITY);  // pattern miss: never expected
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      double X[4][4];
      hadamard_block_entries(Bq, S, i, j, X);
#pragma unroll
      for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
          if (off[q1][q2] < 0) continue;
          double* dst = A.val + off[q1][q2];
          atomicAdd(&dst[3 * i + j], X[q1][q2]);
          if (i != j) atomicAdd(&dst[3 * j + i], X[q2][q1]);
        }
    }
}

// per thread: V (D*D doubles, column-major; the FP32 eigenvectors occupy its
// first D*D floats during the FP32 phase) | A (D(D+1)/2 doubles; the FP32 matrix
// in its first floats during the FP32 phase, then the FP64 matrix, then B+)
constexpr int PROJ_SMEM = (81 + 45) * 8;

// Mollified pairs, one thread per queued pair: PSD projection of the 9x9
// reduced matrix and the BSR scatter.  The input B stays in registers; the
// eigenvectors V and the working matrix A live in shared memory laid out
// element-major ([element][thread]), so a warp touches 32 consecutive words
// per access, 1008 B per thread for D = 9.  The eigen-decomposition is FP32
// first (Jacobi on the cheap pipe to ~1e-6), its arrays inside the V and A
// regions; then FP64: modified Gram-Schmidt on the eigenvectors, A = V^T B V,
// and symmetric Jacobi sweeps to an off-diagonal norm of 1e-14 ||A||.
// Projection onto the PSD cone is non-expansive in the Frobenius norm, so the
// projected matrix is exact to 1e-14 of ||B||.  B+ is mapped back to the
// involved points with K (x) I and scattered.
template <int S>
__global__ void __launch_bounds__(S) k_hess_proj(HessArgs A) {
  constexpr int D = 9, NP = D * (D + 1) / 2;
  extern __shared__ double smem[];
  const int tid = threadIdx.x;
  const int64_t m = (int64_t)*A.nmoll;
  // grid-stride over the queue, S pairs per step; the loop bound is the same
  // for every thread of a block, and a thread past the end leaves only in the
  // block's last step, after its last barrier
  for (int64_t base = (int64_t)blockIdx.x * S; base < m; base += (int64_t)gridDim.x * S) {
    // the previous step's B+ and V (double layout) overlap other threads' FP32
    // arrays of this step
    __syncthreads();
    const int64_t w = base + tid;
    double* Vs = smem + tid;                            // V: row i of column k at [(k * D + i) * S]
    double* Ad = smem + D * D * S + tid;                // A: element e at [e * S]
    float* V32 = (float*)smem + tid;                    // FP32 V, same indexing, inside the V region
    float* A32 = (float*)(smem + D * D * S) + tid;      // FP32 A, same indexing, inside the A region
    const bool act = w < m;                             // no early exit before the last barrier
    const uint32_t c = act ? A.mlist[w] : 0u;
    // B stays in registers until B+ is formed
    double Br[NP];
    double mx = 0.0;
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      Br[e] = act ? A.B9[(size_t)e * A.cap + w] : 0.0;
      mx = fmax(mx, fabs(Br[e]));
    }
    const bool work = act && mx != 0.0;
    if (work) {
      const double inv = 1.0 / mx;
#pragma unroll
      for (int e = 0; e < NP; ++e) A32[e * S] = (float)(Br[e] * inv);
      for (int k = 0; k < D; ++k)
        for (int i = 0; i < D; ++i) V32[(k * D + i) * S] = (i == k) ? 1.f : 0.f;
      jacobi_packed<float, D>(A32, V32, S, PROJ_FP32_TOL2, 12);
    }
    // FP64 re-orthonormalisation of the FP32 eigenvectors (modified Gram-Schmidt),
    // columns in descending order.  Double column k takes the bytes of float
    // columns 2k and 2k+1 (column 0: 0 and 1), all read before it is written:
    // higher columns in earlier steps, column k itself before the barrier.
    for (int k = D - 1; k >= 0; --k) {
      double v[D];
#pragma unroll
      for (int i = 0; i < D; ++i) v[i] = work ? (double)V32[(k * D + i) * S] : 0.0;
      __syncthreads();
      if (work) {
        for (int j = k + 1; j < D; ++j) {
          double dp = 0.0;
#pragma unroll
          for (int i = 0; i < D; ++i) dp += Vs[(j * D + i) * S] * v[i];
#pragma unroll
          for (int i = 0; i < D; ++i) v[i] -= dp * Vs[(j * D + i) * S];
        }
        double nn = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i) nn += v[i] * v[i];
        nn = rsqrt_refined(nn);  // nn is 1 to FP32 accuracy here
#pragma unroll
        for (int i = 0; i < D; ++i) Vs[(k * D + i) * S] = v[i] * nn;
      }
    }
    // from here on every thread touches only its own elements: no more barriers
    if (!act) continue;  // the block's last step
    // eigenvalues -> diagonal of Ad, eigenvectors -> Vs
    if (!work) {
      for (int e = 0; e < NP; ++e) Ad[e * S] = 0.0;
      for (int k = 0; k < D; ++k)
        for (int i = 0; i < D; ++i) Vs[(k * D + i) * S] = (i == k) ? 1.0 : 0.0;
    } else {
      // A = V^T B V, column by column (the FP32 A is dead: every thread passed
      // the Gram-Schmidt barriers after its FP32 phase)
      for (int l = 0; l < D; ++l) {
        double vl[D], t[D];
#pragma unroll
        for (int j = 0; j < D; ++j) vl[j] = Vs[(l * D + j) * S];
#pragma unroll
        for (int i = 0; i < D; ++i) {
          double v = 0.0;
#pragma unroll
          for (int j = 0; j < D; ++j) v += Br[i <= j ? tri_idx(i, j, D) : tri_idx(j, i, D)] * vl[j];
          t[i] = v;
        }
        for (int k = 0; k <= l; ++k) {
          double v = 0.0;
#pragma unroll
          for (int i = 0; i < D; ++i) v += Vs[(k * D + i) * S] * t[i];
          Ad[tri_idx(k, l, D) * S] = v;
        }
      }
      jacobi_refine64<D>(Ad, Vs, S, 1e-28, 12);
    }
    // B+ (into the A region) from the side with fewer terms: the sum over the
    // positive eigenpairs of lam v v^T, or B minus the sum over the negative
    // ones (B = V A V^T to the FP64 sweeps' tolerance).  The loop runs as many
    // terms as the warp's busiest lane needs; each lane adds its own j-th term.
    double lam[D];
    int npos = 0, nneg = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      lam[k] = Ad[tri_idx(k, k, D) * S];
      npos += lam[k] > 0.0;
      nneg += lam[k] < 0.0;
    }
    const bool from_b = nneg < npos;
    const int nterm = from_b ? nneg : npos;
    const int wterm = __reduce_max_sync(__activemask(), nterm);
    double* Bs = Ad;  // B+ replaces A (scaled by 1/4, the square of K4's entries)
    constexpr double bsc = 0.25;
#pragma unroll
    for (int e = 0; e < NP; ++e) Bs[e * S] = from_b ? Br[e] * bsc : 0.0;
    for (int j = 0; j < wterm; ++j) {
      int k = -1, cnt = 0;
      double wk = 0.0;
#pragma unroll
      for (int kk = 0; kk < D; ++kk) {
        const bool sel = from_b ? lam[kk] < 0.0 : lam[kk] > 0.0;
        if (sel && cnt == j) {
          k = kk;
          wk = (from_b ? -lam[kk] : lam[kk]) * bsc;
        }
        cnt += sel;
      }
      if (k < 0) continue;
      double v[D];
#pragma unroll
      for (int i = 0; i < D; ++i) v[i] = Vs[(k * D + i) * S];
#pragma unroll
      for (int i = 0; i < D; ++i) {
        const double wi = wk * v[i];
#pragma unroll
        for (int jj = i; jj < D; ++jj) Bs[tri_idx(i, jj, D) * S] += wi * v[jj];
      }
    }
    const Stencil st = stencil_of(A.cand[c], A.ev0, A.ev1, A.tv, A.T);
    hadamard_scatter(A, st, Bs, S);
  }
}

// ---- the 9x9 projection for short queues: a warp per pair ----------------
// One thread per pair runs some 8,500 dependent FP64 instructions, and an FP64
// warp instruction occupies a warp for 64 cycles however many of its lanes
// are active (measured on GB300: 64 cycles per dependent or independent DFMA
// of a lone warp; 76 with one warp per SM sub-partition, one per 19 cycles and
// SM, near the unit's rate of one per 16), so a short queue (a
// small scene) waits for that chain however idle the device is.  This form
// spreads one pair over a warp, the three lanes (r, t) = (l / 3, l % 3) of
// row r (lanes 0..26) owning entries t, t + 3, t + 6 of row and column r,
// and orders the Jacobi rotations round robin: in round k of a sweep row r
// pairs with (2k - r) mod 9 (row k rests), the four disjoint rotations of a
// round are applied at once (X = A J by columns, then J^T X by rows, V J by
// columns), so a sweep is 9 rounds of 18 FP64 instructions per lane
// instead of 36 rotations in sequence.  Each lane computes its own row's
// rotation, the same bits in every lane of the pair's two rows.  The arithmetic is
// otherwise that of k_hess_proj: FP32 Jacobi on the scaled matrix to
// the same tolerance, FP64 modified Gram-Schmidt, A = V^T B V, FP64 sweeps
// with FP32 tangents and FP64-normalised rotations to an off-diagonal norm
// of 1e-14 ||A||, B+ from the positive eigenpairs, the Hadamard scatter.
constexpr int PL_PAIRS = 4;                 // pairs per block
constexpr int PL_THREADS = 32 * PL_PAIRS;   // one warp per pair: three lanes per row
// doubles per pair: A, X (A J; later the Hadamard staging, 108), V, and the
// FP32 phase's A, X, V (3 x 81 floats)
constexpr int PL_SMEM = 81 + 108 + 81 + 122;
// Queues of at most this many (mollified) pairs take the lane-parallel form.  Stage (d) with n such pairs, lane-parallel
// against one thread a pair: 100 pairs 374 / 713 us, 2,000 486 / 722, 4,000 629 / 724, 5,000 708 / 730, 6,000 819 / 733;
// a pleated 97x97 sheet with 1,296 of 47,510 active pairs mollified 627 / 1,180.
constexpr int64_t PL_MAX_PAIRS = 4096;

// sum over the warp: a butterfly, so every lane gets the same bits
template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// one round of simultaneous rotations on a 9x9 matrix As and vectors Vs held
// in shared memory ([9 i + j]); the three lanes (r, t) of row r apply its
// pair's rotation (c, sg: sg = -s for the lower index of the pair, +s for the
// upper, 0 and c = 1 for a resting row or a skipped pair) to entries
// t, t + 3, t + 6 of column r, then of row r
template <typename R>
__device__ __forceinline__ void rr_apply3(R* As, R* Xs, R* Vs, int r, int t, int pr, R c, R sg, bool row) {
  R vr[3], vp[3];
  if (row) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int i = t + 3 * m;
      Xs[9 * i + r] = c * As[9 * i + r] + sg * As[9 * i + pr];
      vr[m] = Vs[9 * i + r];
      vp[m] = Vs[9 * i + pr];
    }
  }
  __syncwarp();  // X complete; every lane holds the V entries it needs
  if (row) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int i = t + 3 * m;
      Vs[9 * i + r] = c * vr[m] + sg * vp[m];
      As[9 * r + i] = c * Xs[9 * r + i] + sg * Xs[9 * pr + i];
    }
  }
  __syncwarp();
}

// the rotation of row r's pair (r, pr) in a round: c and sg as rr_apply3 takes
// them; every lane of the pair's two rows computes the same bits
template <typename R>
__device__ __forceinline__ void pl_rotation(const R* As, int r, int pr, bool row, R skip, double inv, R& c, R& sg);

template <>
__device__ __forceinline__ void pl_rotation<float>(const float* As, int r, int pr, bool row, float skip, double,
                                                   float& c, float& sg) {
  c = 1.f;
  sg = 0.f;
  if (!row || pr == r) return;
  const int p = min(r, pr), q = max(r, pr);
  const float apq = As[9 * p + q];
  if (!(fabsf(apq) > skip)) return;
  const float app = As[9 * p + p], aqq = As[9 * q + q];
  const float tau = (aqq - app) / (2.f * apq);
  const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
  c = 1.f / sqrtf(1.f + t * t);
  sg = r == p ? -t * c : t * c;
}

// FP64: the tangent from FP32 arithmetic on the values scaled by the norm,
// c = 1/sqrt(1 + t^2) to FP64 rounding
template <>
__device__ __forceinline__ void pl_rotation<double>(const double* As, int r, int pr, bool row, double skip,
                                                    double inv, double& c, double& sg) {
  c = 1.0;
  sg = 0.0;
  if (!row || pr == r) return;
  const int p = min(r, pr), q = max(r, pr);
  const double apq = As[9 * p + q];
  if (!(fabs(apq) > skip)) return;
  const double app = As[9 * p + p], aqq = As[9 * q + q];
  const float apq32 = (float)(apq * inv), dd32 = (float)((aqq - app) * inv);
  const float tau = dd32 / (2.f * apq32);
  const float t32 = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
  const double t = (double)t32;
  c = rsqrt_refined(1.0 + t * t);
  sg = r == p ? -t * c : t * c;
}

__global__ void __launch_bounds__(PL_THREADS) k_hess_proj_lanes(HessArgs A) {
  extern __shared__ double pl_smem[];
  const int seg = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane / 3, t = lane - 3 * r;  // row r (< 9 for lanes 0..26), third t
  const bool row = lane < 27;
  const int64_t w = (int64_t)blockIdx.x * PL_PAIRS + seg;
  if (w >= (int64_t)*A.nmoll) return;  // the whole warp leaves together
  double* As = pl_smem + (size_t)seg * PL_SMEM;  // A[i][j] at [9 i + j]
  double* Xs = As + 81;                          // A J; later the Hadamard staging
  double* Vs = Xs + 108;                         // V[i][k]: component i of eigenvector k
  float* A32 = (float*)(Vs + 81);
  float* X32 = A32 + 81;
  float* V32 = X32 + 81;
  const uint32_t ci = A.mlist[w];
  double Br[9];  // row r of B
  double mx = 0.0;
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    Br[j] = row ? A.B9[(size_t)(r <= j ? tri_idx(r, j, 9) : tri_idx(j, r, 9)) * A.cap + w] : 0.0;
    mx = fmax(mx, fabs(Br[j]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (mx == 0.0) return;  // B+ = 0: nothing to add
  // FP32 phase on B / max|B|
  {
    const double inv = 1.0 / mx;
    if (row)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int j = t + 3 * m;
        A32[9 * r + j] = (float)(Br[j] * inv);
        V32[9 * r + j] = r == j ? 1.f : 0.f;
      }
    __syncwarp();
    for (int sweep = 0; sweep < 12; ++sweep) {
      float off = 0.f, fro = 0.f;
      if (row)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          const int j = t + 3 * m;
          const float v = A32[9 * r + j];
          if (j == r) fro += v * v;
          else off += v * v;
        }
      off = warp_sum(off);
      fro = warp_sum(fro) + off;
      if (fro == 0.f || off <= PROJ_FP32_TOL2 * fro) break;
      const float skip = 1e-16f * sqrtf(fro);
      for (int k = 0; k < 9; ++k) {
        const int pr = row ? (2 * k - r + 18) % 9 : r;
        float c, sg;
        pl_rotation<float>(A32, r, pr, row, skip, 0.0, c, sg);
        rr_apply3<float>(A32, X32, V32, r, t, pr, c, sg, row);
      }
    }
  }
  // FP64 modified Gram-Schmidt on the FP32 eigenvectors, columns in
  // descending order; the three lanes of row r hold component r (the same
  // bits), and only lane t = 0 of each row enters the sums
  for (int k = 8; k >= 0; --k) {
    double v = row ? (double)V32[9 * r + k] : 0.0;
    for (int j = k + 1; j < 9; ++j) {
      const double vj = row ? Vs[9 * r + j] : 0.0;
      const double dp = warp_sum(t == 0 ? vj * v : 0.0);
      v -= dp * vj;
    }
    const double nn = rsqrt_refined(warp_sum(t == 0 ? v * v : 0.0));  // 1 to FP32 accuracy here
    if (row) Vs[9 * r + k] = v * nn;  // each lane of the row writes the same bits, then reads its own
  }
  __syncwarp();
  // A = V^T (B V): entries t, t + 3, t + 6 of row r of W = B V into X, then
  // those of the upper triangle of row r of A from the columns of V and W, mirrored
  if (row)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int l = t + 3 * m;
      double s = 0.0;
#pragma unroll
      for (int j = 0; j < 9; ++j) s += Br[j] * Vs[9 * j + l];
      Xs[9 * r + l] = s;
    }
  __syncwarp();
  if (row)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int l = t + 3 * m;
      if (l < r) continue;
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < 9; ++i) s += Vs[9 * i + r] * Xs[9 * i + l];
      As[9 * r + l] = s;
      As[9 * l + r] = s;
    }
  __syncwarp();
  // FP64 sweeps to an off-diagonal norm of 1e-14 ||A||
  for (int sweep = 0; sweep < 12; ++sweep) {
    double off = 0.0, fro = 0.0;
    if (row)
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int j = t + 3 * m;
        const double v = As[9 * r + j];
        if (j == r) fro += v * v;
        else off += v * v;
      }
    off = warp_sum(off);
    fro = warp_sum(fro) + off;
    if (fro == 0.0 || off <= 1e-28 * fro) break;
    const double nrm = sqrt(fro);
    const double skip = 1e-16 * nrm, inv = 1.0 / nrm;
    for (int k = 0; k < 9; ++k) {
      const int pr = row ? (2 * k - r + 18) % 9 : r;
      double c, sg;
      pl_rotation<double>(As, r, pr, row, skip, inv, c, sg);
      rr_apply3<double>(As, Xs, Vs, r, t, pr, c, sg, row);
    }
  }
  // B+ / 4 (the square of K4's entries), entries j = t, t + 3, t + 6 of row
  // r: sum over the positive eigenpairs of lam v v^T (the product v_r v_j is
  // formed first, so rows r and j get the same bits); then the point
  // transform over those three column points (axis t) into the staging rows
  double P[3] = {0.0, 0.0, 0.0};
  if (row)
    for (int k = 0; k < 9; ++k) {
      const double lam = As[9 * k + k];
      if (!(lam > 0.0)) continue;
      const double l4 = 0.25 * lam, vr = Vs[9 * r + k];
#pragma unroll
      for (int m = 0; m < 3; ++m) P[m] = fma(vr * Vs[9 * (t + 3 * m) + k], l4, P[m]);
    }
  __syncwarp();  // every lane is done with X
  if (row) {
    double h[4];
    had3(P[0], P[1], P[2], h);
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) Xs[12 * r + 3 * q2 + t] = h[q2];
  }
  __syncwarp();
  // lane l < 12 takes block row q1 = l / 3, axis i = l % 3: the transform
  // over the row points, and the sixteen blocks' entries of that row
  if (lane < 12) {
    const int q1 = lane / 3, i = lane % 3;
    const Stencil st = stencil_of(A.cand[ci], A.ev0, A.ev1, A.tv, A.T);
    const int rv = st.v[q1];
#pragma unroll
    for (int q2 = 0; q2 < 4; ++q2) {
      const int cv = st.v[q2];
      const int64_t bi = find_block(A.row_ptr, A.col, rv, cv);
      if (!(bi < A.row_ptr[rv + 1] && A.col[bi] == cv)) {
        atomicOr(A.status, (unsigned long long)CB_DEV_CAPACITY);  // pattern miss: never expected
        continue;
      }
      double* dst = A.val + 9 * bi + 3 * i;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        double h[4];
        had3(Xs[12 * i + 3 * q2 + j], Xs[12 * (3 + i) + 3 * q2 + j], Xs[12 * (6 + i) + 3 * q2 + j], h);
        atomicAdd(&dst[j], h[q1]);
      }
    }
  }
}

// k_hess_proj over at most one resident wave of blocks (the occupancy looked
// up once per scene)
cb_status launch_proj(cb_scene* s, const HessArgs& A, int64_t cap, cudaStream_t st) {
  const int smem = PROJ_SMEM * PROJ_THREADS;
  int& occ = s->proj_occ;
  CB_CUDA(cudaFuncSetAttribute(k_hess_proj<PROJ_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  if (occ <= 0) {
    CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_hess_proj<PROJ_THREADS>, PROJ_THREADS, smem));
    occ = std::max(1, occ);
  }
  const int64_t g = std::min<int64_t>(cb_grid(cap, PROJ_THREADS), (int64_t)s->n_sms * occ);
  k_hess_proj<PROJ_THREADS><<<(int)std::max<int64_t>(1, g), PROJ_THREADS, smem, cb_count(st)>>>(A);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}

__global__ void k_energy_final(int count, const unsigned long long* __restrict__ macc, double* __restrict__ out) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= count) return;
  double e = __longlong_as_double(macc[(size_t)m * MACC_STRIDE + MACC_E]);
  if (macc[(size_t)m * MACC_STRIDE + MACC_STATUS] & CB_DEV_PENETRATION) e = __longlong_as_double(0x7ff0000000000000LL);
  out[m] = e;
}

__global__ void k_set_u64(unsigned long long* p, unsigned long long v) { *p = v; }

// One launch for the resets at the start of a barrier pass: the scalar slots
// in sc_mask and, for every member, the accumulator slots in macc_mask.
__global__ void k_pass_reset(unsigned long long* __restrict__ sc, uint32_t sc_mask, int count,
                             unsigned long long* __restrict__ macc, uint32_t macc_mask) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < SC_N && ((sc_mask >> i) & 1u)) sc[i] = 0ull;
  if (i < count)
    for (int k = 0; k < MACC_STRIDE; ++k)
      if ((macc_mask >> k) & 1u) macc[(size_t)i * MACC_STRIDE + k] = 0ull;
}

}  // namespace

// the distinct columns of the buckets past ROW_BLOCK_MAX (counted in `huge`)
static cb_status huge_rows(cb_scene* s, const HugeRows& H, uint32_t* uniq, cudaStream_t st) {
  int bits = H.cbits;
  while ((uint64_t)(H.n - 1) >> (bits - H.cbits)) ++bits;
  const int64_t L = H.entries;
  CB_TRY(buf_ensure(s->hkey, sizeof(uint64_t) * (size_t)L, st));
  CB_TRY(buf_ensure(s->hflag, sizeof(uint32_t) * 2 * (size_t)(L + 1), st));
  CB_TRY(buf_ensure(s->hhist, sizeof(uint32_t) * (size_t)cbp::radix_hist_elems(L), st));
  CB_TRY(buf_ensure(s->scan_tmp, sizeof(uint64_t) * (size_t)(std::max(cbp::scan_tmp_elems(cbp::radix_hist_elems(L)),
                                                                      cbp::scan_tmp_elems(L + 1)) + 8), st));
  // the blocks' keys are in their buckets by now: their memory (16 an active pair) holds these
  uint64_t *k0 = bp<uint64_t>(s->bkey), *k1 = bp<uint64_t>(s->hkey);
  uint32_t *flag = bp<uint32_t>(s->hflag), *pos = flag + (L + 1);
  k_huge_keys<<<cb_grid(L), CB_THREADS, 0, cb_count(st)>>>(H, bp<uint32_t>(s->rcol), k0);
  const uint64_t* key = cbp::radix_sort<uint64_t, uint32_t, false>(k0, nullptr, k1, nullptr, L, 0, bits,
                                                                   bp<uint32_t>(s->hhist), bp<uint32_t>(s->scan_tmp), st)
                            ? k1
                            : k0;
  k_huge_flag<<<cb_grid(L + 1), CB_THREADS, 0, cb_count(st)>>>((unsigned)L, key, flag);
  cbp::exclusive_scan<uint32_t, uint32_t>(flag, pos, L + 1, bp<uint32_t>(s->scan_tmp), (uint32_t*)nullptr, st);
  k_huge_write<<<cb_grid(L), CB_THREADS, 0, cb_count(st)>>>(H, key, flag, pos, bp<uint32_t>(s->rcol), uniq);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}

__global__ void k_fill_u64(int64_t n, unsigned long long* __restrict__ p, unsigned long long v) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

cb_status filter_precompute(cb_scene* s, cudaStream_t st) {
  uint64_t* sc = scalars(s);
  unsigned long long* dmin = (unsigned long long*)(sc + SC_DBAR_MIN_BITS);
  unsigned long long* nf = (unsigned long long*)(sc + SC_NFILT);
  k_set_u64<<<1, 1, 0, cb_count(st)>>>(dmin, 0x7ff0000000000000ull);
  k_set_u64<<<1, 1, 0, cb_count(st)>>>(nf, 0ull);
  // per-component minima, by component label (rods: polyline index; shells: a vertex id)
  CB_TRY(buf_ensure(s->dbar_comp, sizeof(unsigned long long) * (size_t)std::max(1, s->n), st));
  unsigned long long* dcomp = bp<unsigned long long>(s->dbar_comp);
  k_fill_u64<<<cb_grid(std::max(1, s->n)), CB_THREADS, 0, cb_count(st)>>>(std::max(1, s->n), dcomp,
                                                                          0x7ff0000000000000ull);
  if (s->kind == CB_ROD) {
    CB_TRY(buf_ensure(s->S, sizeof(double) * (size_t)s->n, st));
    CB_TRY(buf_ensure(s->win, sizeof(int32_t) * (size_t)std::max(1, s->E), st));
    CB_TRY(buf_ensure(s->wst, sizeof(int32_t) * (size_t)std::max(1, s->E), st));
    k_arclength<<<cb_grid(s->n_rods), CB_THREADS, 0, cb_count(st)>>>(s->n_rods, bp<int32_t>(s->rod_ptr), bp<double>(s->rest),
                                                           s->n, bp<double>(s->S));
    if (s->E > 0)
      k_rod_window<<<cb_grid(s->E), CB_THREADS, 0, cb_count(st)>>>(
          s->E, bp<int32_t>(s->ev0), bp<int32_t>(s->ev1), bp<int32_t>(s->comp), bp<double>(s->S),
          bp<double>(s->rest), s->n, bp<int32_t>(s->rlast), s->a, bp<int32_t>(s->win), bp<int32_t>(s->wst), dmin,
          nf, dcomp);
    CB_CUDA(cudaGetLastError());
    uint64_t h[2];
    CB_TRY(read_scalars(s, SC_DBAR_MIN_BITS, 1, &h[0], st));
    CB_TRY(read_scalars(s, SC_NFILT, 1, &h[1], st));
    memcpy(&s->dbar_min, &h[0], 8);
    s->n_frest = (int64_t)h[1];
  } else {
    // rest broad phase at the full activation, then rest distances below a (a
    // geodesic distance is at least the 3D one, so the same candidates serve it)
    int64_t nr = 0;
    ScopedBuf rcs(st);
    DevBuf& rc = rcs.b;
    // positions of the reference distances: the flat pattern when given, else the rest shape
    const double* rf = s->ruv.p ? bp<double>(s->ruv) : bp<double>(s->rest);
    CB_TRY(broad_phase(s, s->bw, rf, nullptr, false, true, rc, nullptr, &nr, st));
    if (nr > 0) {
      ScopedBuf flags(st), poss(st), dbars(st);
      DevBuf &flag = flags.b, &pos = poss.b, &dbar = dbars.b;
      CB_TRY(buf_ensure(flag, sizeof(uint32_t) * (size_t)nr, st));
      CB_TRY(buf_ensure(pos, sizeof(uint32_t) * ((size_t)nr + 1), st));
      CB_TRY(buf_ensure(dbar, sizeof(double) * (size_t)nr, st));
      CB_TRY(buf_ensure(s->scan_tmp, sizeof(uint64_t) * (size_t)(cbp::scan_tmp_elems(nr) + 8), st));
      if (s->geodesic) {
        CB_TRY(geo_rest_dbar(s, bp<uint64_t>(rc), nr, bp<uint32_t>(flag), bp<double>(dbar), dmin, dcomp, st));
      } else {
        k_rest_filter<<<cb_grid(nr), CB_THREADS, 0, cb_count(st)>>>(nr, bp<uint64_t>(rc), bp<int32_t>(s->ev0),
                                                          bp<int32_t>(s->ev1), bp<int32_t>(s->tv), s->T,
                                                          bp<int32_t>(s->comp), rf, s->n, s->a,
                                                          bp<uint32_t>(flag), bp<double>(dbar), dmin, dcomp);
      }
      uint32_t* tot = (uint32_t*)(sc + SC_COUNT1);
      cbp::exclusive_scan<uint32_t, uint32_t>(bp<uint32_t>(flag), bp<uint32_t>(pos), nr, bp<uint32_t>(s->scan_tmp),
                                              tot, st);
      uint64_t h[2];
      CB_CUDA(cudaGetLastError());
      CB_TRY(read_scalars(s, SC_COUNT1, 1, &h[0], st));
      const int64_t nf_ = (int64_t)(uint32_t)h[0];
      CB_TRY(buf_ensure(s->frest, sizeof(uint64_t) * (size_t)std::max<int64_t>(1, nf_), st));
      CB_TRY(buf_ensure(s->frest_dbar, sizeof(double) * (size_t)std::max<int64_t>(1, nf_), st));
      cbp::k_compact<uint64_t, uint32_t><<<cb_grid(nr), CB_THREADS, 0, cb_count(st)>>>(bp<uint64_t>(rc), bp<uint32_t>(flag),
                                                                         bp<uint32_t>(pos), nr, bp<uint64_t>(s->frest));
      cbp::k_compact<double, uint32_t><<<cb_grid(nr), CB_THREADS, 0, cb_count(st)>>>(bp<double>(dbar), bp<uint32_t>(flag),
                                                                       bp<uint32_t>(pos), nr,
                                                                       bp<double>(s->frest_dbar));
      CB_CUDA(cudaGetLastError());
      CB_TRY(read_scalars(s, SC_DBAR_MIN_BITS, 1, &h[1], st));
      memcpy(&s->dbar_min, &h[1], 8);
      s->n_frest = nf_;
    } else {
      s->dbar_min = INFINITY;
      s->n_frest = 0;
    }
  }
  if (s->n_frest > 0 && !(s->dbar_min > 0.0)) return CB_ERR_DEGENERATE;
  s->dbar_fmax = s->dbar_min;
  if (s->hmp.size() == 1 && s->hmp[0].per_comp) {
    std::vector<unsigned long long> h((size_t)std::max(1, s->n));
    CB_CUDA(cudaMemcpyAsync(h.data(), dcomp, sizeof(unsigned long long) * h.size(), cudaMemcpyDeviceToHost, st));
    CB_CUDA(cudaStreamSynchronize(st));
    double mx = -INFINITY;
    for (unsigned long long b : h) {
      double v;
      memcpy(&v, &b, 8);
      if (std::isfinite(v)) mx = std::max(mx, v);
    }
    if (std::isfinite(mx)) s->dbar_fmax = mx;
  }
  return CB_OK;
}

// The candidates' classes come with them from contact_build (broad.cu); what
// is left here is their count and the per-stencil activation.
cb_status filter_apply(cb_scene* s, cudaStream_t st) {
  const int64_t nc = s->n_cand;
  uint64_t* sc = scalars(s);
  unsigned long long* nf = (unsigned long long*)(sc + SC_NFILT);
  s->n_dropped = 0;
  const bool ps = s->per_stencil();
  if (nc == 0 || ps) {
    CB_CUDA(cudaMemsetAsync(nf, 0, sizeof(unsigned long long), st));
    if (nc == 0) return CB_OK;
  } else {
    CB_CUDA(cudaMemcpyAsync(nf, sc + SC_NFB, sizeof(unsigned long long), cudaMemcpyDeviceToDevice, st));
    return CB_OK;
  }
  if (!s->bw.box_raw.p) return CB_ERR_ARG;  // the candidates came from before the mode was set
  unsigned long long* ndrop = (unsigned long long*)(sc + SC_COUNT1);
  k_set_u64<<<1, 1, 0, cb_count(st)>>>(ndrop, 0ull);
  k_own_width<<<cb_grid(nc), CB_THREADS, 0, cb_count(st)>>>(
      nc, bp<uint64_t>(s->cand), bp<double>(s->bw.box_raw), bp<int32_t>(s->ev0), bp<int32_t>(s->vsc),
      bp<MemberParams>(s->mp), bp<unsigned long long>(s->dbar_comp), bp<int32_t>(s->comp), s->kind == CB_ROD, s->n,
      s->T, bp<uint8_t>(s->klass), nf, ndrop);
  CB_CUDA(cudaGetLastError());
  // per-stencil activation: drop the class-F candidates outside their own width
  uint64_t hd;
  CB_TRY(read_scalars(s, SC_COUNT1, 1, &hd, st));
  s->n_dropped = (int64_t)hd;
  if (hd == 0) return CB_OK;
  CB_TRY(buf_ensure(s->cflag, sizeof(uint32_t) * (size_t)nc, st));
  CB_TRY(buf_ensure(s->cpos, sizeof(uint32_t) * ((size_t)nc + 1), st));
  CB_TRY(buf_ensure(s->scan_tmp, sizeof(uint64_t) * (size_t)(cbp::scan_tmp_elems(nc) + 8), st));
  CB_TRY(buf_ensure(s->cand_alt, sizeof(uint64_t) * (size_t)nc, st));
  CB_TRY(buf_ensure(s->klass_alt, (size_t)nc, st));
  k_keep_flag<<<cb_grid(nc), CB_THREADS, 0, cb_count(st)>>>(nc, bp<uint8_t>(s->klass), bp<uint32_t>(s->cflag));
  cbp::exclusive_scan<uint32_t, uint32_t>(bp<uint32_t>(s->cflag), bp<uint32_t>(s->cpos), nc,
                                          bp<uint32_t>(s->scan_tmp), (uint32_t*)nullptr, st);
  k_keep_write<<<cb_grid(nc), CB_THREADS, 0, cb_count(st)>>>(nc, bp<uint64_t>(s->cand), bp<uint8_t>(s->klass),
                                                            bp<uint32_t>(s->cflag), bp<uint32_t>(s->cpos),
                                                            bp<uint64_t>(s->cand_alt), bp<uint8_t>(s->klass_alt));
  CB_CUDA(cudaGetLastError());
  std::swap(s->cand, s->cand_alt);
  std::swap(s->klass, s->klass_alt);
  s->n_cand = nc - s->n_dropped;
  return CB_OK;
}

cb_status to_f32(cb_scene* s, const double* v, const double* cx, DevBuf& out, cudaStream_t st) {
  CB_TRY(buf_ensure(out, sizeof(float4) * (size_t)std::max(1, s->n), st));
  k_to_f32<<<cb_grid(s->n), CB_THREADS, 0, cb_count(st)>>>(s->n, v, cx, bp<int32_t>(s->vsc), bp<float4>(out));
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}

cb_status barrier_run(cb_scene* s, const double* x, double* energy, double* grad, bool energy_only,
                      cudaStream_t st) {
  const int64_t nc = s->n_cand;
  uint64_t* sc = scalars(s);
  unsigned long long* status = (unsigned long long*)(sc + SC_STATUS);
  unsigned long long* ncore = (unsigned long long*)(sc + SC_NCORE);
  unsigned long long* macc = bp<unsigned long long>(s->macc);
  const int M = s->count;
  bool mollify = false;
  for (const MemberParams& m : s->hmp) mollify |= m.mollify != 0;
  s->cd_split = false;
  s->core_valid = true;
  // the pass's counters (the queue lengths stay readable until the next pass)
  {
    const uint32_t scm = (1u << SC_NCORE) | (1u << SC_NLIST) | (1u << SC_KSPLIT) | (1u << SC_NMOLL) |
                         (1u << SC_N9) | (1u << SC_N6) | (1u << SC_N4) | (1u << SC_NBK) | (1u << SC_NLONG) |
                         (1u << SC_HUGE);
    k_pass_reset<<<cb_grid(std::max(M, (int)SC_N)), CB_THREADS, 0, cb_count(st)>>>(
        (unsigned long long*)sc, scm, M, macc, (1u << MACC_E) | (1u << MACC_STATUS));
  }
  if (grad) CB_CUDA(cudaMemsetAsync(grad, 0, sizeof(double) * 3 * (size_t)s->n, st));
  s->n_active = s->n_plane = 0;
  int64_t nmoll = 0;
  s->nnzb = 0;
  CB_TRY(buf_ensure(s->bsr_row, sizeof(int32_t) * ((size_t)s->n + 1), st));
  CB_CUDA(cudaMemsetAsync(s->bsr_row.p, 0, sizeof(int32_t) * ((size_t)s->n + 1), st));
  if (nc > 0) {
    CB_TRY(buf_ensure(s->cd, sizeof(double) * (size_t)nc, st));
    CB_TRY(buf_ensure(s->ctype, (size_t)nc, st));
    CB_TRY(buf_ensure(s->ccls, (size_t)nc, st));
    CB_TRY(buf_ensure(s->clist, sizeof(uint32_t) * (size_t)nc, st));
    CB_TRY(buf_ensure(s->aidx, sizeof(uint32_t) * (size_t)nc, st));
    if (mollify) CB_TRY(buf_ensure(s->mlist, sizeof(uint32_t) * (size_t)nc, st));
    CB_TRY(to_f32(s, x, bp<double>(s->bw.cx), s->xf, st));
    CB_TRY(buf_ensure(s->dlist, sizeof(uint32_t) * (size_t)nc, st));
    unsigned int* nl = (unsigned int*)(sc + SC_NLIST);
    k_distance_screen<<<cb_grid(nc), CB_THREADS, 0, cb_count(st)>>>(
        nc, bp<uint64_t>(s->cand), bp<uint8_t>(s->klass), bp<int32_t>(s->ev0), bp<int32_t>(s->ev1),
        bp<int32_t>(s->tv), s->T, bp<float4>(s->xf), bp<double>(s->bw.cx), bp<int32_t>(s->vsc),
        bp<MemberParams>(s->mp), s->n, bp<uint32_t>(s->dlist), nl);
    (energy_only ? k_distance_exact<true> : k_distance_exact<false>)<<<std::min<int64_t>(cb_grid(nc), (int64_t)s->n_sms * 3), CB_THREADS, 0, cb_count(st)>>>(
        bp<uint32_t>(s->dlist), nc, nl, bp<uint64_t>(s->cand), bp<uint8_t>(s->klass), bp<int32_t>(s->ev0),
        bp<int32_t>(s->ev1), bp<int32_t>(s->tv), s->T, x, s->n, bp<int32_t>(s->vsc), bp<MemberParams>(s->mp),
        bp<double>(s->cd), bp<int8_t>(s->ctype), bp<uint8_t>(s->ccls), bp<uint32_t>(s->clist), bp<uint32_t>(s->aidx),
        (unsigned*)(sc + SC_KSPLIT), mollify ? bp<uint32_t>(s->mlist) : nullptr, (unsigned*)(sc + SC_NMOLL), status, ncore,
        macc, bp<int32_t>(s->comp), bp<unsigned long long>(s->dbar_comp), bp<double>(s->elen2));
    if (energy_only) {
      if (energy) k_energy_final<<<cb_grid(M), CB_THREADS, 0, cb_count(st)>>>(M, macc, energy);
      CB_CUDA(cudaGetLastError());
      return CB_OK;
    }
    CB_CUDA(cudaGetLastError());
    uint64_t h[SC_NMOLL - SC_KSPLIT + 1];
    CB_TRY(read_scalars(s, SC_KSPLIT, SC_NMOLL - SC_KSPLIT + 1, h, st));
    s->n_plane = (int64_t)(uint32_t)h[0];
    s->n_active = s->n_plane + (int64_t)(h[0] >> 32);
    nmoll = (int64_t)(uint32_t)h[SC_NMOLL - SC_KSPLIT];
    s->act_cap = nc;
    // end of stage (c): distances, classes and the active set
    if (s->timing) cudaEventRecord(s->ev[12], st);
    s->cd_split = true;
  }
  const int64_t na = s->n_active;
  if (na > 0) {
    const ActiveList act = active_list(s);
    // BSR pattern: distinct (row, col) of the 16 blocks of every active stencil
    const int n = s->n;
    const size_t m = 16 * (size_t)na;  // capacity; the keys are counted by k_block_keys
    CB_TRY(buf_ensure(s->bkey, sizeof(uint2) * m, st));
    CB_TRY(buf_ensure(s->rcol, sizeof(uint32_t) * m, st));
    // row counts, fill cursors, distinct counts (cleared together), bucket offsets, long buckets
    CB_TRY(buf_ensure(s->row_cnt, sizeof(uint32_t) * 5 * ((size_t)n + 1), st));
    CB_TRY(buf_ensure(s->scan_tmp, sizeof(uint64_t) * (size_t)(cbp::scan_tmp_elems(n + 1) + 8), st));
    uint32_t* cnt = bp<uint32_t>(s->row_cnt);
    uint32_t *cursor = cnt + (n + 1), *uniq = cursor + (n + 1), *off = uniq + (n + 1), *longs = off + (n + 1);
    CB_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * 3 * ((size_t)n + 1), st));
    unsigned int* nbk = (unsigned int*)(sc + SC_NBK);
    unsigned int* nlong = (unsigned int*)(sc + SC_NLONG);
    CB_CUDA(cudaFuncSetAttribute(k_block_keys, cudaFuncAttributeMaxDynamicSharedMemorySize, BK_SMEM));
    k_block_keys<<<(int)((na + BK_PAIRS - 1) / BK_PAIRS), BK_PAIRS, BK_SMEM, cb_count(st)>>>(
        act, bp<uint64_t>(s->cand), bp<int32_t>(s->ev0), bp<int32_t>(s->ev1), bp<int32_t>(s->tv), s->T,
        bp<uint2>(s->bkey), nbk, cnt);
    cbp::exclusive_scan<uint32_t, uint32_t>(cnt, off, (int64_t)n + 1, bp<uint32_t>(s->scan_tmp), (uint32_t*)nullptr, st);
    k_row_fill<<<(int)std::min<int64_t>(cb_grid((int64_t)m), (int64_t)s->n_sms * 16), CB_THREADS, 0, cb_count(st)>>>(
        bp<uint2>(s->bkey), nbk, off, cursor, bp<uint32_t>(s->rcol));
    const int per = n >= s->n_sms * 64 * 8 ? 8 : 1;
    k_row_unique<<<cb_grid(((int64_t)n + per - 1) / per * 32, 32 * ROW_WARPS), 32 * ROW_WARPS, 0, cb_count(st)>>>(
        n, per, off, bp<uint32_t>(s->rcol), uniq, longs, nlong);
    // rows, and the first entries, of the buckets past ROW_BLOCK_MAX: the counts and cursors are of no more use
    uint32_t *hrow = cnt, *hstart = cursor;
    CB_CUDA(cudaFuncSetAttribute(k_row_unique_long, cudaFuncAttributeMaxDynamicSharedMemorySize, ROW_LONG_SMEM));
    k_row_unique_long<<<s->n_sms, ROW_LONG_T, ROW_LONG_SMEM, cb_count(st)>>>(off, bp<uint32_t>(s->rcol), uniq, longs, nlong, hrow,
                                                                     hstart, (unsigned long long*)(sc + SC_HUGE));
    uint64_t h[SC_HUGE - SC_COUNT1 + 1];
    auto row_pointers = [&]() -> cb_status {
      // uniq[n] = 0: the scan's last entry is the block count
      uint32_t* tot = (uint32_t*)(sc + SC_COUNT1);
      cbp::exclusive_scan<uint32_t, int32_t>(uniq, bp<int32_t>(s->bsr_row), (int64_t)n + 1,
                                             (int32_t*)bp<uint32_t>(s->scan_tmp), (int32_t*)tot, st);
      CB_CUDA(cudaGetLastError());
      return read_scalars(s, SC_COUNT1, SC_HUGE - SC_COUNT1 + 1, h, st);
    };
    CB_TRY(row_pointers());
    const uint64_t huge = h[SC_HUGE - SC_COUNT1];
    HugeRows H{(unsigned)(huge >> 32), (unsigned)huge, 1, hrow, hstart, off};
    while ((int64_t)(n - 1) >> H.cbits) ++H.cbits;
    if (H.n > 0) {
      CB_TRY(huge_rows(s, H, uniq, st));
      CB_TRY(row_pointers());
    }
    s->nnzb = (int64_t)(uint32_t)h[0];
    CB_TRY(buf_ensure(s->bsr_col, sizeof(int32_t) * (size_t)s->nnzb, st));
    CB_TRY(buf_ensure(s->bsr_val, sizeof(double) * 9 * (size_t)s->nnzb, st));
    CB_CUDA(cudaMemsetAsync(s->bsr_val.p, 0, sizeof(double) * 9 * (size_t)s->nnzb, st));
    k_row_write<<<cb_grid((int64_t)n * 8), CB_THREADS, 0, cb_count(st)>>>(n, off, bp<uint32_t>(s->rcol),
                                                                          bp<int32_t>(s->bsr_row),
                                                                          bp<int32_t>(s->bsr_col));
    if (const unsigned rows = (unsigned)h[SC_NLONG - SC_COUNT1])
      k_row_write_long<<<(int)std::min<int64_t>(rows, (int64_t)s->n_sms * 2), ROW_LONG_T, 0, cb_count(st)>>>(
          longs, rows, off, bp<uint32_t>(s->rcol), bp<int32_t>(s->bsr_row), bp<int32_t>(s->bsr_col));
    if (H.n > 0)
      k_huge_cols<<<cb_grid(H.entries), CB_THREADS, 0, cb_count(st)>>>(H, bp<uint32_t>(s->rcol), bp<int32_t>(s->bsr_row),
                                                                      bp<int32_t>(s->bsr_col));
    HessArgs A;
    A.act = act;
    A.cand = bp<uint64_t>(s->cand);
    A.cd = bp<double>(s->cd);
    A.ctype = bp<int8_t>(s->ctype);
    A.ccls = bp<uint8_t>(s->ccls);
    A.ev0 = bp<int32_t>(s->ev0);
    A.ev1 = bp<int32_t>(s->ev1);
    A.tv = bp<int32_t>(s->tv);
    A.T = s->T;
    A.x = x;
    A.n = s->n;
    A.vsc = bp<int32_t>(s->vsc);
    A.mp = bp<MemberParams>(s->mp);
    A.macc = macc;
    A.comp = bp<int32_t>(s->comp);
    A.dbar_comp = bp<unsigned long long>(s->dbar_comp);
    A.row_ptr = bp<int32_t>(s->bsr_row);
    A.col = bp<int32_t>(s->bsr_col);
    A.val = bp<double>(s->bsr_val);
    A.grad = grad;
    A.status = status;
    if (nmoll > 0) CB_TRY(buf_ensure(s->hB9, sizeof(double) * 45 * (size_t)nmoll, st));
    A.B9 = bp<double>(s->hB9);
    A.n9 = (unsigned int*)(sc + SC_N9);
    A.n6 = (unsigned int*)(sc + SC_N6);
    A.n4 = (unsigned int*)(sc + SC_N4);
    A.cap = nmoll;
    A.mlist = bp<uint32_t>(s->mlist);
    A.nmoll = (const unsigned*)(sc + SC_NMOLL);
    A.elen2 = bp<double>(s->elen2);
    if (s->timing) cudaEventRecord(s->ev[10], st);
    k_pair_hess<<<cb_grid(na, PAIR_T), PAIR_T, 0, cb_count(st)>>>(A);
    CB_CUDA(cudaGetLastError());
    if (nmoll > 0) {
      k_moll_hess<<<cb_grid(nmoll, 32), 32, 0, cb_count(st)>>>(A);
      if (nmoll <= PL_MAX_PAIRS) {
        const int smem = PL_SMEM * (int)sizeof(double) * PL_PAIRS;
        k_hess_proj_lanes<<<(int)((nmoll + PL_PAIRS - 1) / PL_PAIRS), PL_THREADS, smem, cb_count(st)>>>(A);
      } else {
        CB_TRY(launch_proj(s, A, nmoll, st));
      }
      CB_CUDA(cudaGetLastError());
    }
    if (s->timing) cudaEventRecord(s->ev[11], st);
    CB_CUDA(cudaGetLastError());
  }
  if (energy) k_energy_final<<<cb_grid(M), CB_THREADS, 0, cb_count(st)>>>(M, macc, energy);
  CB_CUDA(cudaGetLastError());
  return CB_OK;
}
